"""The one-system CG as a resident kernel (csrc/cg_resident.cu): every number
of lanes per site, precision and link form against the oracle's residual, and
the lattices next to the sizes at which the form changes."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import gauge

pytestmark = pytest.mark.gpu


def _unitary_field(sq, dims, seed):
    """A gauge field of random SU(3) links built on the device."""
    import torch
    g = torch.Generator(device='cuda')
    g.manual_seed(seed)
    vol = int(np.prod(dims))
    q, _ = torch.linalg.qr(torch.randn((vol, 4, 3, 3), generator=g, device='cuda', dtype=torch.complex128))
    u = (q / torch.linalg.det(q)[..., None, None] ** (1 / 3)).contiguous()
    fat, lng = torch.empty_like(u), torch.empty_like(u)
    sq.gauge_fatten(dims, u, fat, lng)
    torch.cuda.synchronize()
    return sq.gauge_load(dims, fat, lng)


def _residual(sq, gid, b, x, mass):
    """|b - A x| / |b| by the library's FP64 operator."""
    import torch
    nbytes, _ = sq.spinor_bytes(gid, 'f64')
    v, w = (torch.zeros(nbytes, dtype=torch.uint8, device='cuda') for _ in range(2))
    ax = torch.empty_like(b)
    sq.pack_spinor(gid, 'f64', x, v)
    sq.mdagm_apply(gid, 'f64', 18, mass, v, w)
    sq.unpack_spinor(gid, 'f64', w, ax)
    return float((b - ax).norm() / b.norm())


@pytest.mark.parametrize('prec,recon', [('f32', 18), ('f32', 12), ('i16', 18), ('i16', 12),
                                        ('f64', 18), ('f64', 12)])
@pytest.mark.parametrize('dims', [(2, 2, 2, 2), (2, 4, 2, 6), (6, 4, 4, 4), (4, 6, 8, 10)])
def test_small_lattices_match_the_oracle(sq, dims, prec, recon):
    fat, lng = gauge(dims, 0.25, 0)
    vh = oracle.volume(dims) // 2
    b = synth.gaussian_source(vh, 1)
    gid = sq.gauge_load(dims, fat, lng, antiperiodic_t=True)
    try:
        x, st = sq.cg_solve(gid, b, 0.1, 1e-9, precision=prec, long_recon=recon)
        assert st['status'] == 0 and st['true_residual'] <= 1e-9
        assert oracle.true_residual(dims, fat, lng, 0.1, b, x, t_sign=-1) <= 1e-9
        again, _ = sq.cg_solve(gid, b, 0.1, 1e-9, precision=prec, long_recon=recon, graph=False)
        assert np.array_equal(x, again)
    finally:
        sq.gauge_free(gid)


# around 512 threads per SM with four, two and one lanes per site (152 SMs):
# 19456, 38912 and 77824 sites per parity
@pytest.mark.parametrize('dims', [(16, 16, 16, 8), (16, 16, 10, 14), (16, 16, 16, 10),
                                  (16, 16, 16, 18), (16, 16, 16, 20), (16, 16, 16, 38),
                                  (16, 16, 16, 40), (14, 18, 22, 28)])
@pytest.mark.parametrize('prec,recon', [('f32', 18), ('i16', 12), ('f64', 18)])
def test_sizes_at_which_the_form_changes(sq, dims, prec, recon):
    import torch
    gid = _unitary_field(sq, dims, 3)
    try:
        b = torch.view_as_complex(torch.randn((int(np.prod(dims)) // 2, 3, 2), device='cuda',
                                              dtype=torch.float64))
        x, st = sq.cg_solve(gid, b, 0.3, 1e-10, precision=prec, long_recon=recon)
        assert st['status'] == 0
        assert _residual(sq, gid, b, x, 0.3) <= 1e-10 * 1.001
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('prec', ['f32', 'i16', 'f64'])
def test_guess_limits_and_long_solves(sq, prec):
    """More iterations than one launch runs, an iteration limit inside a
    launch, a guess, a zero and a non-finite source."""
    from paper_1411_2223_gb300 import sq as sqm
    dims = (8, 8, 8, 16)
    fat, lng = gauge(dims, 0.3, 0)
    b = synth.gaussian_source(oracle.volume(dims) // 2, 2)
    gid = sq.gauge_load(dims, fat, lng)
    try:
        x, st = sq.cg_solve(gid, b, 0.01, 1e-9, precision=prec)
        assert st['status'] == 0 and st['iterations'] > 128
        assert oracle.true_residual(dims, fat, lng, 0.01, b, x) <= 1e-9
        y, s2 = sq.cg_solve(gid, b, 0.01, 1e-9, precision=prec, x0=x)
        assert s2['iterations'] == 0 and np.array_equal(x, y)
        y, s2 = sq.cg_solve(gid, b, 0.01, 1e-12, precision=prec, max_iter=37, check=False)
        assert s2['status'] == sqm.NOT_CONVERGED and s2['iterations'] == 37
        y, s2 = sq.cg_solve(gid, 0 * b, 0.01, 1e-9, precision=prec)
        assert s2['status'] == 0 and np.all(y == 0)
        bad = b.copy()
        bad[5, 1] = np.nan
        with pytest.raises(sqm.SqError) as e:
            sq.cg_solve(gid, bad, 0.01, 1e-9, precision=prec)
        assert e.value.status == sqm.ERR_NONFINITE
        z, _ = sq.cg_solve(gid, b, 0.01, 1e-9, precision=prec)  # nothing is left behind
        assert np.array_equal(x, z)
    finally:
        sq.gauge_free(gid)


def test_a_launch_ends_within_milliseconds(sq):
    """FP64 at 65536 sites per parity, some 80 us an iteration: other streams get
    the device after 4 ms, that is 64 iterations or fewer, and the solve is a
    chain of such launches, each with the pair of an update after it (three more
    kernels pack, start and unpack)."""
    dims = (16, 16, 16, 32)
    fat, lng = gauge(dims, 0.25, 0)
    b = synth.gaussian_source(oracle.volume(dims) // 2, 4)
    gid = sq.gauge_load(dims, fat, lng)
    try:
        sq.cg_solve(gid, b, 0.5, 1e-2, precision='f64')  # tunes
        n = sq.kernel_launches()
        x, st = sq.cg_solve(gid, b, 0.01, 1e-9, precision='f64')
        n = sq.kernel_launches() - n
        assert oracle.true_residual(dims, fat, lng, 0.01, b, x) <= 1e-9
        assert st['iterations'] > 256 and (n - 3) // 3 * 64 >= st['iterations'], (n, st['iterations'])
    finally:
        sq.gauge_free(gid)
