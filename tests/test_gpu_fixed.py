"""The FP64 operator on fixed-point links (csrc/sq_fixed.cuh).

A 55-bit fixed-point mat-vec drops at most 2^-54 of the product of the two
operands' scales per real product and rounds the sum of an output component
to FP64 once (2^-53 relative).  For Gaussian vectors the largest of the 96
neighbour components is about 4 times their RMS and the links' elements are
at most 1.2, so an output component (RMS about 2 in those units) is off by
at most about 10 * 2^-54 * 5 / 2 of its RMS in the dropped terms (random
signs over 96 products): the 2-norm error stays below 2^-51.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import gauge, gpu_dslash, rel, site_rel, to_dev

pytestmark = pytest.mark.gpu

DIMS = [(2, 4, 2, 6), (4, 6, 8, 10), (6, 4, 10, 4)]


def _reference(dims, fat, lng, v_half, out_parity, t_sign=1):
    """D v in long double (64 or more mantissa bits)."""
    lx, ly, lz, lt = dims
    vol = lx * ly * lz * lt
    ld = np.clongdouble
    full = np.zeros((vol, 3), dtype=ld)
    full[oracle.half_sites(dims, 1 - out_parity)] = v_half
    lex = np.arange(vol)
    c = np.stack([lex % lx, (lex // lx) % ly, (lex // (lx * ly)) % lz, lex // (lx * ly * lz)], 1)
    st = np.array([1, lx, lx * ly, lx * ly * lz])
    out = np.zeros((vol, 3), dtype=ld)

    def at(mu, d):
        n = (c[:, mu] + d) % dims[mu]
        wraps = np.floor_divide(c[:, mu] + d, dims[mu])
        s = np.where((mu == 3) & (wraps % 2 != 0), t_sign, 1)
        return lex + (n - c[:, mu]) * st[mu], s[:, None]

    for mu in range(4):
        eta = (1 - 2 * (c[:, :mu].sum(1) & 1))[:, None] * np.longdouble(0.5)
        for u, d in ((fat, 1), (lng, 3)):
            u = u[:, mu].astype(ld)
            n, s = at(mu, d)
            out += eta * s * (u * full[n][:, None, :]).sum(-1)
            n, s = at(mu, -d)
            out -= eta * s * (np.conj(np.swapaxes(u[n], 1, 2)) * full[n][:, None, :]).sum(-1)
    return out[oracle.half_sites(dims, out_parity)]


@pytest.mark.parametrize('dims', DIMS)
@pytest.mark.parametrize('spread', [0, 8])
def test_fixed_point_dslash_error(sq, dims, spread):
    """Even fields, and sites whose magnitudes differ by up to e^16."""
    fat, lng = gauge(dims)
    vh = oracle.volume(dims) // 2
    rng = np.random.default_rng(4)
    gid = sq.gauge_load(dims, fat, lng, antiperiodic_t=True)
    try:
        for p in (0, 1):
            v = synth.gaussian_source(vh, 5 + p) * np.exp(rng.uniform(-spread, spread, (vh, 1)))
            got = gpu_dslash(sq, gid, 'f64', 18, v, p, vh)
            want = _reference(dims, fat, lng, v, p, t_sign=-1)
            assert rel(got, want.astype(np.complex128)) <= 2.0 ** -51
            assert site_rel(got, want.astype(np.complex128)) <= 2.0 ** -48
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('scale', [1e-300, 1e-30, 1e250, 1e300])
def test_magnitudes_at_the_ends_of_fp64(sq, scale):
    """Inside and outside the fixed-point exponents; also a single non-zero
    site (all other neighbours zero)."""
    dims = (4, 6, 8, 10)
    fat, lng = gauge(dims)
    vh = oracle.volume(dims) // 2
    v = synth.gaussian_source(vh, 6)
    point = np.zeros_like(v)
    point[17] = v[17]
    gid = sq.gauge_load(dims, fat, lng)
    try:
        for w in (v, point):
            got = gpu_dslash(sq, gid, 'f64', 18, w * scale, 1, vh) / scale
            assert rel(got, oracle.dslash_half(dims, fat, lng, w, 1)) <= 1e-15
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('bad', [np.nan, np.inf, -np.inf])
def test_non_finite_neighbours(sq, bad):
    """A site is non-finite exactly where one of its neighbours is; the
    others are untouched."""
    dims = (4, 6, 8, 10)
    fat, lng = gauge(dims)
    vh = oracle.volume(dims) // 2
    v = synth.gaussian_source(vh, 7)
    mark = np.zeros_like(v)
    mark[31] = 1.0
    hit = np.abs(oracle.dslash_half(dims, fat, lng, mark, 1)).sum(1) > 0
    want = oracle.dslash_half(dims, fat, lng, v, 1)
    v[31, 1] = bad
    gid = sq.gauge_load(dims, fat, lng)
    try:
        got = gpu_dslash(sq, gid, 'f64', 18, v, 1, vh)
        assert not np.isfinite(got[hit]).all(axis=1).any()
        assert rel(got[~hit], want[~hit]) <= 1e-15
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('least', [1.0, 2.0 ** -3, 2.0 ** -6, 0.0])
def test_links_of_uneven_size(sq, least):
    """Links much smaller than the field's largest keep FP64 FMAs: every
    output site is accurate on its own scale either way."""
    dims = (4, 4, 4, 6)
    fat, lng = (a.copy() for a in gauge(dims))
    s = np.ones(oracle.volume(dims))
    s[::2] = least
    fat *= s[:, None, None, None]
    lng *= s[:, None, None, None]
    vh = oracle.volume(dims) // 2
    v = synth.gaussian_source(vh, 8)
    gid = sq.gauge_load(dims, fat, lng)
    try:
        for p in (0, 1):
            got = gpu_dslash(sq, gid, 'f64', 18, v, p, vh)
            want = oracle.dslash_half(dims, fat, lng, v, p)
            assert rel(got, want) <= 1e-15
            x = sq.cg_solve(gid, v, 0.3, 1e-10, precision='f64')[0]
            assert oracle.true_residual(dims, fat, lng, 0.3, v, x) <= 1e-10
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('nrhs', [2, 3, 4, 7])
def test_tiles_give_the_bits_of_one_system(sq, nrhs):
    """Every tile of systems computes what the one-system kernel does."""
    import torch
    dims = (4, 6, 8, 10)
    fat, lng = gauge(dims)
    vh = oracle.volume(dims) // 2
    gid = sq.gauge_load(dims, fat, lng)
    try:
        nbytes, _ = sq.spinor_bytes(gid, 'f64')
        src = torch.zeros((nrhs, nbytes), dtype=torch.uint8, device='cuda')
        out, one = torch.zeros_like(src), torch.zeros_like(src)
        for j in range(nrhs):
            v = torch.from_numpy(synth.gaussian_source(vh, j)).cuda()
            sq.pack_spinor(gid, 'f64', v, src[j])
            sq.dslash_apply(gid, 0, 'f64', 18, src[j], one[j])
        sq.dslash_apply_multi(gid, 0, 'f64', 18, nrhs, src, out)
        torch.cuda.synchronize()
        assert torch.equal(out, one)
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('dims', [(2, 2, 2, 2), (4, 6, 8, 10), (6, 2, 10, 4)])
@pytest.mark.parametrize('antiperiodic', [False, True])
def test_dirac_apply_gathers_from_the_whole_lattice(sq, dims, antiperiodic):
    """Against the Dslash of the halves, on a side stream; with a site that
    takes the FP64 form (its neighbours are infinite) and links that do."""
    import torch
    fat, lng = gauge(dims)
    vol = oracle.volume(dims)
    even, odd = oracle.half_sites(dims, 0), oracle.half_sites(dims, 1)
    for scale in (1.0, 0.01):  # uneven links keep FP64 FMAs
        f, l = fat.copy(), lng.copy()
        f[0] *= scale
        l[0] *= scale
        gid = sq.gauge_load(dims, f, l, antiperiodic_t=antiperiodic)
        try:
            v = synth.gaussian_source(vol, 9)
            want = np.empty_like(v)
            for p, (a, b) in enumerate(((even, odd), (odd, even))):
                want[a] = 0.07 * v[a] + gpu_dslash(sq, gid, 'f64', 18, v[b], p, vol // 2)
            st = torch.cuda.Stream()
            x = to_dev(v)
            out = torch.full_like(x, float('nan'))
            torch.cuda.synchronize()
            sq.dirac_apply(gid, 0.07, x, out, stream=st)
            assert rel(out.cpu().numpy(), want) <= 1e-15
            v[even[0]] = np.inf
            sq.dirac_apply(gid, 0.07, to_dev(v), out)
            got = out.cpu().numpy()
            bad = ~np.isfinite(got).all(axis=1)
            assert bad[even[0]] and bad[odd].any() and not bad[even[1:]].any()
            assert rel(got[~bad], want[~bad]) <= 1e-15
        finally:
            sq.gauge_free(gid)


# around the size up to which a site's directions go to four warps (29184
# sites per parity on 152 SMs), whole and part warps of sites
@pytest.mark.parametrize('prec', ['f32', 'i16'])
@pytest.mark.parametrize('dims', [(2, 2, 2, 2), (6, 2, 10, 4), (12, 14, 14, 24), (16, 16, 16, 16)])
def test_reliable_updates_of_one_system(sq, dims, prec):
    """The residual a solve reports is its last reliable update's: it is the
    oracle's, to the FP64 rounding of A x (|x| <= 4 |b|, |A| of order 10: some
    1e-14, with room 1e-12), also from a guess outside the fixed-point range."""
    fat, lng = gauge(dims)
    vh = oracle.volume(dims) // 2
    b = synth.gaussian_source(vh, 11)
    tiny = np.zeros_like(b)
    tiny[::7] = 1e-300
    gid = sq.gauge_load(dims, fat, lng)
    try:
        for x0 in (None, tiny):
            x, st = sq.cg_solve(gid, b, 0.5, 1e-9, precision=prec, x0=x0)
            assert st['status'] == 0
            true = oracle.true_residual(dims, fat, lng, 0.5, b, x)
            assert true <= 1e-9
            assert abs(st['true_residual'] - true) <= 1e-12
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('shift', [3, -3])
def test_dirac_apply_on_overlapping_vectors(sq, shift):
    """The result is that of separate vectors, as it is written last."""
    import torch
    dims = (6, 2, 10, 4)
    fat, lng = gauge(dims)
    vol = oracle.volume(dims)
    v = to_dev(synth.gaussian_source(vol, 9))
    gid = sq.gauge_load(dims, fat, lng)
    try:
        want = torch.empty_like(v)
        sq.dirac_apply(gid, 0.07, v, want)
        both = torch.zeros((vol + abs(shift), 3), dtype=torch.complex128, device='cuda')
        src, dst = both[max(shift, 0):][:vol], both[max(-shift, 0):][:vol]
        src.copy_(v)
        torch.cuda.synchronize()
        sq.dirac_apply(gid, 0.07, src, dst)
        assert rel(dst.cpu().numpy(), want.cpu().numpy()) <= 1e-15
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('long_scale', [1.0, 2.0 ** -2, 2.0 ** -14, 2.0 ** -30, 2.0 ** 5, 'half', 0.0])
def test_point_source_site_by_site(sq, long_scale):
    """Every site that a point source reaches, relative to itself: on 8^4 each
    is reached by one hop.  A fat link's elements are off by 2^-55 (the fields'
    largest is 1.1 to 1.4), that is 3 sqrt(2) 2^-55 of the result at most, and the
    result by 2^-53; long links of 1/96 to 4/3 are held to 2^-60, or 2^-53 of
    3 sqrt(2) times themselves, and FP64 FMAs add 3 2^-53: below 2^-51.  Long links
    of zero ('half': of half the sites) are exact."""
    dims = (8, 8, 8, 8)
    fat, lng = (a.copy() for a in gauge(dims))
    if long_scale == 'half':
        lng[::2] = 0.0
    else:
        lng *= long_scale
    vol = oracle.volume(dims)
    vh = vol // 2
    gid = sq.gauge_load(dims, fat, lng)
    try:
        for p in (0, 1):
            v = np.zeros((vh, 3), dtype=np.complex128)
            v[901] = synth.gaussian_source(vh, 3)[901]
            want = _reference(dims, fat, lng, v, p).astype(np.complex128)
            size = np.linalg.norm(want, axis=1)
            got = gpu_dslash(sq, gid, 'f64', 18, v, p, vh)
            assert np.all(np.linalg.norm(got - want, axis=1) <= 2.0 ** -51 * size)
            full = np.zeros((vol, 3), dtype=np.complex128)
            full[oracle.half_sites(dims, 1 - p)] = v
            out = to_dev(np.full_like(full, np.nan))
            sq.dirac_apply(gid, 0.0, to_dev(full), out)
            got = out.cpu().numpy()[oracle.half_sites(dims, p)]
            assert np.all(np.linalg.norm(got - want, axis=1) <= 2.0 ** -51 * size)
    finally:
        sq.gauge_free(gid)


@pytest.mark.parametrize('decay', [0.0, 0.7, 1.5, 3.0])
def test_steep_decays_site_by_site(sq, decay):
    """Neighbours by long hops exp(2 decay) times larger than those by fat hops:
    a fat-hop neighbour at most 8 times smaller is cut at 2^-53 of the larger
    one's size, uniformly, and six parts enter a component, which is
    sqrt(6 / 3) 8 2^-54 = 2^-50.5 of it (rms); past 8 both kinds keep an exponent
    of their own.  The rms over the sites of the error relative to the site stays
    below 2^-50."""
    dims = (8, 8, 8, 16)
    fat, lng = gauge(dims)
    vh = oracle.volume(dims) // 2
    gid = sq.gauge_load(dims, fat, lng)
    try:
        for p in (0, 1):
            t = oracle.half_sites(dims, 1 - p) // 512
            v = synth.gaussian_source(vh, 5) * np.exp(-decay * np.minimum(t, 16 - t))[:, None]
            want = _reference(dims, fat, lng, v, p)
            got = gpu_dslash(sq, gid, 'f64', 18, v, p, vh)
            err = np.linalg.norm((got - want).astype(np.complex128), axis=1)
            err /= np.linalg.norm(want.astype(np.complex128), axis=1)
            assert np.sqrt(np.mean(err ** 2)) <= 2.0 ** -50
    finally:
        sq.gauge_free(gid)


# sites per parity that the resident kernel takes with four, two and one lane
@pytest.mark.parametrize('dims', [(4, 4, 4, 8), (12, 14, 14, 24), (16, 16, 16, 32)])
def test_point_source_solves(sq, dims):
    """A point source sends its surroundings through the site-by-site form in the
    operator's tiles, the resident kernel and the reliable updates: tiles give
    the bits of one system, and solves the residual they report (as
    test_reliable_updates_of_one_system)."""
    import torch
    fat, lng = gauge(dims)
    vh = oracle.volume(dims) // 2
    b = np.zeros((vh, 3), dtype=np.complex128)
    b[vh // 3] = synth.gaussian_source(vh, 3)[vh // 3]
    gid = sq.gauge_load(dims, fat, lng)
    try:
        nbytes, _ = sq.spinor_bytes(gid, 'f64')
        src = torch.zeros((5, nbytes), dtype=torch.uint8, device='cuda')
        out, one = torch.zeros_like(src), torch.zeros_like(src)
        for j in range(5):
            sq.pack_spinor(gid, 'f64', to_dev(np.roll(b, 7 * j, axis=0)), src[j])
            sq.dslash_apply(gid, 1, 'f64', 18, src[j], one[j])
        sq.dslash_apply_multi(gid, 1, 'f64', 18, 5, src, out)
        torch.cuda.synchronize()
        assert torch.equal(out, one)
        for prec in ('f64', 'f32', 'i16'):
            x, st = sq.cg_solve(gid, b, 0.5, 1e-9, precision=prec)
            assert st['status'] == 0
            true = oracle.true_residual(dims, fat, lng, 0.5, b, x)
            assert true <= 1e-9 and abs(st['true_residual'] - true) <= 1e-12
    finally:
        sq.gauge_free(gid)
