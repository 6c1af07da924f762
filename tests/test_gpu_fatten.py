"""Fat and long links built on the GPU from thin links (gauge_fatten,
gauge_load_thin) vs the FP64 oracle's construction of the same recipe."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import rel

pytestmark = pytest.mark.gpu


def _fatten_gpu(sq, dims, thin, **kw):
    import torch
    u = torch.from_numpy(np.ascontiguousarray(thin)).cuda()
    fat = torch.zeros_like(u)
    lng = torch.zeros_like(u)
    sq.gauge_fatten(dims, u, fat, lng, **kw)
    torch.cuda.synchronize()
    return fat.cpu().numpy(), lng.cpu().numpy()


@pytest.mark.parametrize('dims', [(4, 6, 8, 10), (2, 4, 6, 4), (4, 4, 4, 4)])
def test_fatten_matches_oracle(sq, dims):
    thin = synth.thin_links(dims, 0.8, seed=2)
    fat, lng = _fatten_gpu(sq, dims, thin)
    f0, l0 = oracle.fat_long(dims, thin)
    assert np.abs(fat - f0).max() <= 1e-14
    assert np.abs(lng - l0).max() <= 1e-15
    # other coefficients reach the kernel
    fat2, lng2 = _fatten_gpu(sq, dims, thin, c1=1.0, c3=0.5, staple_weight=0.25)
    f2, l2 = oracle.fat_long(dims, thin, c1=1.0, c3=0.5, w=0.25)
    assert np.abs(fat2 - f2).max() <= 1e-14 and np.abs(lng2 - l2).max() <= 1e-14


def test_load_thin_then_dslash_and_solve(sq):
    dims = (4, 6, 8, 10)
    thin = synth.thin_links(dims, 0.25, seed=0)
    fat, lng = oracle.fat_long(dims, thin)
    gid = sq.gauge_load_thin(dims, thin)
    try:
        from gpu_helpers import gpu_dslash
        vh = oracle.volume(dims) // 2
        v = synth.gaussian_source(vh, 1)
        got = gpu_dslash(sq, gid, 'f64', 18, v, 1, vh)
        want = oracle.dslash_half(dims, fat, lng, v, 1)
        assert rel(got, want) <= 1e-13
        x, st = sq.cg_solve(gid, v, 0.05, 1e-9, long_recon=12)
        assert st['status'] == 0
        assert oracle.true_residual(dims, fat, lng, 0.05, v, x) <= 1e-9
    finally:
        sq.gauge_free(gid)


def test_fatten_rejects_bad_arguments(sq):
    import torch
    from paper_1411_2223_gb300 import sq as sqm
    u = torch.zeros((16 * 4, 4, 3, 3), dtype=torch.complex128, device='cuda')
    with pytest.raises(sqm.SqError):
        sq.gauge_fatten((4, 4, 4, 3), u, u.clone(), u.clone())   # odd extent
    with pytest.raises(sqm.SqError):
        sq.gauge_fatten((4, 4, 2, 2), u, u.clone(), u.clone(), staple_weight=float('inf'))
    thin = np.full((16 * 4, 4, 3, 3), np.nan, dtype=np.complex128)
    with pytest.raises(sqm.SqError) as e:
        sq.gauge_load_thin((4, 4, 2, 2), thin)
    assert e.value.status == sqm.ERR_NONFINITE


def test_fatten_full_size_20x64(sq):
    """The benchmark lattice 20^3 x 64 (eps 0.25): every link against the oracle."""
    dims = (20, 20, 20, 64)
    thin = synth.thin_links(dims, 0.25, seed=0)
    fat, lng = _fatten_gpu(sq, dims, thin)
    f0, l0 = oracle.fat_long(dims, thin)
    assert np.abs(fat - f0).max() <= 1e-14
    assert np.abs(lng - l0).max() <= 1e-15


def _asqtad_gpu(sq, dims, thin):
    import torch
    u = torch.from_numpy(np.ascontiguousarray(thin)).cuda()
    fat = torch.zeros_like(u)
    lng = torch.zeros_like(u)
    sq.gauge_fatten_asqtad(dims, u, fat, lng)
    torch.cuda.synchronize()
    return fat, lng


@pytest.mark.parametrize('dims', [(4, 6, 8, 10), (2, 4, 6, 4)])
def test_asqtad_links_match_oracle(sq, dims):
    thin = synth.thin_links(dims, 0.6, seed=4)
    fat, lng = _asqtad_gpu(sq, dims, thin)
    f0, l0 = oracle.asqtad_links(dims, thin)
    assert np.abs(fat.cpu().numpy() - f0).max() <= 1e-14
    assert np.abs(lng.cpu().numpy() - l0).max() <= 1e-15


def test_asqtad_links_solve(sq):
    """A CG solve on the GPU-built asqtad links (12-real Naik links) meets the
    oracle's residual computed on the oracle's own asqtad links."""
    dims = (4, 6, 8, 10)
    thin = synth.thin_links(dims, 0.25, seed=0)
    fat_d, lng_d = _asqtad_gpu(sq, dims, thin)
    f0, l0 = oracle.asqtad_links(dims, thin)
    gid = sq.gauge_load(dims, fat_d, lng_d)
    try:
        b = synth.gaussian_source(oracle.volume(dims) // 2, 2)
        for prec, recon in (('f32', 12), ('i16', 12), ('f64', 18)):
            x, st = sq.cg_solve(gid, b, 0.03, 1e-9, precision=prec, long_recon=recon)
            assert st['status'] == 0
            assert oracle.true_residual(dims, f0, l0, 0.03, b, x) <= 1e-9
    finally:
        sq.gauge_free(gid)


def test_asqtad_full_size_20x64(sq):
    """The benchmark lattice 20^3 x 64: every asqtad link against the oracle."""
    dims = (20, 20, 20, 64)
    thin = synth.thin_links(dims, 0.25, seed=0)
    fat, lng = _asqtad_gpu(sq, dims, thin)
    f0, l0 = oracle.asqtad_links(dims, thin)
    assert np.abs(fat.cpu().numpy() - f0).max() <= 1e-14
    assert np.abs(lng.cpu().numpy() - l0).max() <= 1e-15


def _asqtad_ref(dims, u, coeffs):
    """The path set as nested staples, on the CPU in complex128."""
    one, three, five, seven, lepage, naik = coeffs
    dag = lambda m: np.conj(np.swapaxes(m, -1, -2))  # noqa: E731
    sh = lambda a, mu, d: synth.shift_field(a, dims, mu, d)  # noqa: E731

    def staple(w, mu, nu, s):
        un = u[:, nu]
        if s > 0:
            return un @ sh(w, nu, 1) @ dag(sh(un, mu, 1))
        return sh(dag(un) @ w @ sh(un, mu, 1), nu, -1)

    fat, lng = np.empty_like(u), np.empty_like(u)
    for mu in range(4):
        um = u[:, mu]
        acc = one * um
        for nu in range(4):
            if nu == mu:
                continue
            for s in (-1, 1):
                s3 = staple(um, mu, nu, s)
                acc = acc + three * s3 + lepage * staple(s3, mu, nu, s)
                for rho in range(4):
                    if rho in (mu, nu):
                        continue
                    for t in (-1, 1):
                        s5 = staple(s3, mu, rho, t)
                        sg = 6 - mu - nu - rho
                        acc = acc + five * s5 + seven * (staple(s5, mu, sg, -1) + staple(s5, mu, sg, 1))
        fat[:, mu] = acc
        lng[:, mu] = naik * (um @ sh(um, mu, 1) @ sh(um, mu, 2))
    return fat, lng


@pytest.mark.parametrize('what', ['su3', 'one', 'three', 'five', 'seven', 'lepage', 'naik', 'none',
                                  'mixed', 'scaled', 'small', 'uneven', 'general', 'zero'])
def test_asqtad_forms(sq, what):
    """Each kind of path alone, coefficients of very different size, and
    links that take the fixed-point kernels (even in size) or the FP64 ones.
    60 products of 3 x 3 matrices nested 6 deep: errors of a few ulp of the
    largest link."""
    import torch
    dims = (4, 2, 6, 4)
    u = synth.thin_links(dims, 0.7, 3)
    c = [5 / 8, 1 / 16, 1 / 64, 1 / 384, -1 / 16, -1 / 24]
    kinds = ['one', 'three', 'five', 'seven', 'lepage', 'naik']
    if what in kinds:
        c = [1.5 if k == what else 0.0 for k in kinds]
    elif what == 'none':
        c = [0.0] * 6
    elif what == 'mixed':
        c = [1e-3, -1e5, 1e-8, 3.0, 1e2, 1e-30]
    elif what == 'scaled':
        u = u * 7.0
    elif what == 'small':
        u = u * 1e-25
    elif what == 'uneven':
        u = u * np.exp(np.random.default_rng(1).uniform(-6, 0, u.shape[:2]))[..., None, None]
    elif what == 'general':
        r = np.random.default_rng(2)
        u = r.standard_normal(u.shape) + 1j * r.standard_normal(u.shape)
    elif what == 'zero':
        u = np.zeros_like(u)
    t = torch.from_numpy(u).cuda()
    fat, lng = torch.full_like(t, float('nan')), torch.full_like(t, float('nan'))
    sq.gauge_fatten_asqtad(dims, t, fat, lng, c)
    f0, l0 = _asqtad_ref(dims, u, c)
    for got, want in ((fat.cpu().numpy(), f0), (lng.cpu().numpy(), l0)):
        assert np.isfinite(got).all()
        if np.abs(want).max() == 0:
            assert np.all(got == 0)
            continue
        assert rel(got, want) <= 2e-15
        assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()


@pytest.mark.parametrize('bad', [np.nan, np.inf])
def test_asqtad_non_finite_links(sq, bad):
    """Only links near the bad one are lost."""
    import torch
    dims = (10, 8, 8, 8)
    u = synth.thin_links(dims, 0.25, 4)
    f0, l0 = _asqtad_ref(dims, u, sq.ASQTAD_COEFFS)
    u[0, 0, 1, 1] = bad
    t = torch.from_numpy(u).cuda()
    fat, lng = torch.empty_like(t), torch.empty_like(t)
    sq.gauge_fatten_asqtad(dims, t, fat, lng)
    got = fat.cpu().numpy()
    c = np.stack(np.unravel_index(np.arange(u.shape[0]), dims, order='F'), 1)
    d = np.minimum(c, np.array(dims) - c)
    far = (d.max(axis=1) > 3)
    assert not np.isfinite(got[0, 0]).all()
    assert np.abs(got[far] - f0[far]).max() <= 1e-14
    assert np.abs(lng.cpu().numpy()[far] - l0[far]).max() <= 1e-15


@pytest.mark.parametrize('what', ['ones', 'phases', 'phases_at_random', 'one_link', 'edge', 'past_edge'])
def test_asqtad_links_with_unit_rows_that_are_not_unitary(sq, what):
    """Unit rows and columns do not bound a link's matrix norm (all elements
    1/sqrt(3): norm sqrt(3)), so such links take the FP64 kernels; multiples of
    unitary links just inside and outside the line between the forms, with
    constant links, where every staple adds up.  Tolerances as in
    test_asqtad_forms."""
    import torch
    dims = (4, 2, 6, 4)
    vol = oracle.volume(dims)
    u = np.empty((vol, 4, 3, 3), dtype=np.complex128)
    rng = np.random.default_rng(5)
    if what == 'ones':
        u[:] = 1 / np.sqrt(3)
    elif what == 'phases':
        u[:] = np.array([[1, 1, -1], [1, 1j, 1], [-1j, 1, 1]]) / np.sqrt(3)
    elif what == 'phases_at_random':
        u[:] = np.exp(2j * np.pi * rng.uniform(size=u.shape)) / np.sqrt(3)
    elif what == 'one_link':
        u[:] = synth.thin_links(dims, 0.7, 3)
        u[vol // 2, 1] = 1 / np.sqrt(3)
    else:
        u[:] = np.eye(3) * np.sqrt(1 + (0.9 if what == 'edge' else 1.1) / 512)
    t = torch.from_numpy(u).cuda()
    fat, lng = torch.full_like(t, float('nan')), torch.full_like(t, float('nan'))
    sq.gauge_fatten_asqtad(dims, t, fat, lng)
    f0, l0 = _asqtad_ref(dims, u, sq.ASQTAD_COEFFS)
    for got, want in ((fat.cpu().numpy(), f0), (lng.cpu().numpy(), l0)):
        assert rel(got, want) <= 2e-15
        assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()


@pytest.mark.parametrize('unitary', [True, False])
@pytest.mark.parametrize('dims', [(4, 2, 4, 16), (4, 2, 14, 4), (2, 12, 4, 12), (10, 4, 2, 4), (2, 2, 2, 8),
                                  (6, 4, 2, 6)])
def test_asqtad_slabs_give_the_bits_of_the_whole_lattice(sq, dims, unitary):
    """Where the scratch is more than is left of the budget the lattice is done in
    slabs across its longest direction: of one slice, of two, of as many as leave
    a part of one at the end, of all but the halo's worth; the first and the last
    wrap around.  The same sums, so the same bits."""
    import torch
    from paper_1411_2223_gb300 import sq as sqm
    u = synth.thin_links(dims, 0.7, 6)
    if not unitary:
        u = u * np.random.default_rng(3).uniform(0.5, 2, u.shape[:2])[..., None, None]
    t = torch.from_numpy(u).cuda()
    want = [torch.empty_like(t) for _ in range(2)]
    sq.gauge_fatten_asqtad(dims, t, *want)
    assert rel(want[0].cpu().numpy(), _asqtad_ref(dims, u, sq.ASQTAD_COEFFS)[0]) <= 2e-15
    longest = max(dims)
    slice_bytes = 2736 * (oracle.volume(dims) // longest)
    for nt in sorted({1, 2, 3, longest - 7}):
        if nt < 1 or nt > max(longest - 7, 1):
            continue
        with sqm.Context(0, hbm_budget=slice_bytes * (nt + 6) + slice_bytes // 2) as ctx:
            got = [torch.full_like(t, float('nan')) for _ in range(2)]
            torch.cuda.synchronize()
            n = ctx.kernel_launches()
            ctx.gauge_fatten_asqtad(dims, t, *got)
            torch.cuda.synchronize()
            slabs = 1 if longest <= 7 else -(-longest // nt)
            assert ctx.kernel_launches() - n == 1 + 27 * slabs
        assert all(torch.equal(g, w) for g, w in zip(got, want))
