"""The NPR one-colour four-fermion operator (Eq. 1) on the GPU vs the FP64
oracle, hypercube by hypercube.

Tolerance: both sides are FP64.  One output is a sum of 256 products of two
sandwiches, each a sum of 9 products with averaged links (sums of up to 24
path products), so the rounding differs by a few hundred ulps of the terms'
size at most; the tests allow 1e-12 of the largest output of the tensor.
"""
import numpy as np
import pytest

import oracle
import synth
from synth import npr as snpr

pytestmark = pytest.mark.gpu

TOL = 1e-12
OPS16 = snpr.bk_ops() + [(0, 0, 0, 0), (15, 15, 15, 15), (3, 5, 12, 9), (1, 3, 12, 9),
                         (6, 0, 0, 10), (9, 9, 6, 6), (7, 8, 11, 4), (14, 1, 2, 13)]


def _inputs(dims, eps=0.5, seed=3):
    return synth.thin_links(dims, eps, seed), snpr.propagators(dims, seed + 10)


def _gpu(sq, dims, links, props, ops, per_hc=True):
    import torch
    u = torch.from_numpy(np.ascontiguousarray(links)).cuda()
    ps = [torch.from_numpy(np.ascontiguousarray(p)).cuda() for p in props]
    nops = len(ops)
    out = torch.full((max(nops, 1), 3, 3, 3, 3), float('nan'), dtype=torch.complex128,
                     device='cuda')
    hc = None
    if per_hc:
        hc = torch.full((oracle.hypercube_count(dims), max(nops, 1), 3, 3, 3, 3), float('nan'),
                        dtype=torch.complex128, device='cuda')
    sq.npr_four_fermion(dims, u, ps, ops, out, hc)
    torch.cuda.synchronize()
    return out.cpu().numpy()[:nops], None if hc is None else hc.cpu().numpy()[:, :nops]


def _close(got, want, tol=TOL):
    scale = np.abs(want).max()
    assert scale > 0
    err = np.abs(got - want).max()
    assert err <= tol * scale, (err, scale)


@pytest.mark.parametrize('dims,nops', [((4, 4, 4, 4), 16), ((6, 2, 10, 4), 1),
                                       ((2, 2, 2, 2), 3), ((4, 6, 4, 8), 8)])
def test_npr_matches_oracle(sq, dims, nops):
    links, props = _inputs(dims)
    ops = OPS16[:nops]
    out, hc = _gpu(sq, dims, links, props, ops)
    want = oracle.npr_four_fermion(dims, links, props, ops)
    _close(hc, want)
    _close(out, want.sum(axis=0))


def test_npr_ragged_grid(sq):
    # 384 hypercubes: more than one resident CTA per hypercube slot, some
    # CTAs take two hypercubes and the rest one
    dims = (8, 8, 8, 12)
    links, props = _inputs(dims, 0.25, 7)
    ops = snpr.bk_ops()
    out, hc = _gpu(sq, dims, links, props, ops)
    want = oracle.npr_four_fermion(dims, links, props, ops)
    _close(hc, want)
    _close(out, want.sum(axis=0))
    # without the per-hypercube output (the kernel's other form: running
    # sums across hypercubes), the same sums to rounding
    out2, _ = _gpu(sq, dims, links, props, ops, per_hc=False)
    _close(out2, want.sum(axis=0))


def test_npr_full_size_sampled(sq):
    """The 20^3 x 64 workload of the benchmark: sampled hypercubes against the
    oracle, and the sum over all 32000 against the per-hypercube outputs."""
    dims = (20, 20, 20, 64)
    links, props = synth.thin_links(dims, 0.25, 0), snpr.propagators(dims, 1)
    ops = snpr.bk_ops()
    out, hc = _gpu(sq, dims, links, props, ops)
    nhc = oracle.hypercube_count(dims)
    pick = [0, 1, 9, 10, 99, 100, nhc // 2, nhc - 101, nhc - 1]
    pick += list(np.random.default_rng(5).choice(nhc, 16, replace=False))
    want = oracle.npr_four_fermion(dims, links, props, ops, hypercubes=pick)
    _close(hc[pick], want)
    _close(out, hc.sum(axis=0), 1e-12)


def test_npr_gauge_invariant_on_gpu(sq):
    dims = (8, 8, 8, 8)
    links, props = _inputs(dims, 0.4, 2)
    ops = snpr.bk_ops()[:4]
    g = synth.random_su3(oracle.volume(dims), 2.0, np.random.default_rng(21))
    out, hc = _gpu(sq, dims, links, props, ops)
    outg, hcg = _gpu(sq, dims, synth.gauge_transform_links(links, g, dims),
                     [g @ p for p in props], ops)
    _close(hcg, hc)
    _close(outg, out)


def test_npr_more_operators_than_one_launch(sq):
    # 37 operators: three groups of at most 16, each a launch pair; outputs
    # land at their operator's place in both tensors
    dims = (4, 4, 6, 4)
    links, props = _inputs(dims, 0.4, 9)
    rng = np.random.default_rng(3)
    ops = [tuple(int(v) for v in rng.integers(0, 16, 4)) for _ in range(37)]
    out, hc = _gpu(sq, dims, links, props, ops)
    want = oracle.npr_four_fermion(dims, links, props, ops)
    _close(hc, want)
    _close(out, want.sum(axis=0))


@pytest.mark.parametrize('nops', [16, 8, 5])
def test_npr_deterministic(sq, nops):
    dims = (8, 8, 8, 12)
    links, props = _inputs(dims, 0.3, 4)
    a, _ = _gpu(sq, dims, links, props, OPS16[:nops], per_hc=False)
    b, _ = _gpu(sq, dims, links, props, OPS16[:nops], per_hc=False)
    assert np.array_equal(a, b)
    want = oracle.npr_four_fermion(dims, links, props, OPS16[:nops]).sum(axis=0)
    _close(a, want)


def test_npr_arguments(sq):
    import torch
    from paper_1411_2223_gb300.sq import SqError
    dims = (4, 4, 4, 4)
    links, props = _inputs(dims)
    u = torch.from_numpy(links).cuda()
    ps = [torch.from_numpy(p).cuda() for p in props]
    out = torch.zeros((SQ_MAX + 1, 3, 3, 3, 3), dtype=torch.complex128, device='cuda')
    # no operators: nothing to do, nothing written
    sq.npr_four_fermion(dims, u, ps, [], out)
    torch.cuda.synchronize()
    assert torch.count_nonzero(out).item() == 0
    with pytest.raises(SqError):
        sq.npr_four_fermion(dims, u, ps, [(16, 0, 0, 0)], out)          # mask out of range
    with pytest.raises(SqError):
        sq.npr_four_fermion((4, 4, 4, 5), u, ps, [(0, 0, 0, 0)], out)   # odd extent
    with pytest.raises(SqError):                                        # misaligned output
        sq.npr_four_fermion(dims, u, ps, [(0, 0, 0, 0)], out.data_ptr() + 8)


SQ_MAX = 16


@pytest.mark.parametrize('nops', [1, 2, 3, 4, 5, 8, 9, 16, 17])
def test_every_slicing_of_the_contraction(sq, nops):
    """The number of operators picks how the sum over corners is split."""
    dims = (4, 4, 6, 4)
    links, props = _inputs(dims, seed=5)
    ops = (OPS16 + [(2, 7, 1, 8)])[:nops]
    out, hc = _gpu(sq, dims, links, props, ops)
    want = oracle.npr_four_fermion(dims, links, props, ops)
    _close(hc, want)
    _close(out, want.sum(axis=0))


@pytest.mark.parametrize('what', ['links3', 'links0.1', 'small', 'large', 'tiny', 'huge', 'spread',
                                  'zero', 'equal'])
def test_inputs_inside_and_outside_the_fixed_point_form(sq, what):
    """Hypercubes that do not fit the two-word form go through FP64; either
    way every hypercube holds the tolerance on its own scale.  'equal': all
    terms of every sum equal, the largest sums the form can meet."""
    dims = (4, 4, 6, 4)
    links, props = _inputs(dims, seed=6)
    if what == 'links3':
        links = links * 3.0
    elif what == 'links0.1':
        links = links * 0.1
    elif what in ('small', 'large', 'tiny', 'huge'):
        s = {'small': 1e-40, 'large': 1e40, 'tiny': 1e-70, 'huge': 1e70}[what]
        props = [p * s for p in props]
    elif what == 'spread':  # hypercubes of very different size
        s = np.exp(np.random.default_rng(2).uniform(-30, 30, props[0].shape[0]))[:, None, None]
        props = [p * s for p in props]
    elif what == 'zero':
        props[2] = np.zeros_like(props[2])
    elif what == 'equal':
        links = snpr.unit_links(dims)
        props = [np.full_like(p, 0.9999999 + 0.9999999j) for p in props]
    ops = OPS16[:5] + [(0, 0, 0, 0)]
    out, hc = _gpu(sq, dims, links, props, ops)
    want = oracle.npr_four_fermion(dims, links, props, ops)
    if what == 'zero':
        assert np.all(hc == 0) and np.all(out == 0)
        return
    scale = np.abs(want).max(axis=tuple(range(1, want.ndim)), keepdims=True)
    assert np.all(np.abs(hc - want) <= TOL * scale)
    _close(out, want.sum(axis=0))


@pytest.mark.parametrize('bad', [np.nan, np.inf])
def test_non_finite_inputs_stay_in_their_hypercube(sq, bad):
    dims = (4, 4, 6, 4)
    links, props = _inputs(dims, seed=7)
    want = oracle.npr_four_fermion(dims, links, props, OPS16[:3])
    props[1] = props[1].copy()
    props[1][0, 1, 2] = bad  # site 0: hypercube 0
    _, hc = _gpu(sq, dims, links, props, OPS16[:3])
    assert not np.isfinite(hc[0]).all()
    _close(hc[1:], want[1:])


@pytest.mark.parametrize('seed', [0, 1])
def test_operators_in_any_order(sq, seed):
    """Q's digits go from one operator's order and signs to the next one's in
    place: every change of t1, t2 and the signs between neighbours."""
    dims = (2, 2, 2, 2)
    links, props = _inputs(dims)
    rng = np.random.default_rng(seed)
    ops = [tuple(int(v) for v in rng.integers(0, 16, 4)) for _ in range(64)]
    ops += [(0, d, 0, t) for d in range(2) for t in (0, 1, 0, 2, 0, 4, 0, 8, 0, 15, 15, 0, 7)]
    out, hc = _gpu(sq, dims, links, props, ops)
    want = oracle.npr_four_fermion(dims, links, props, ops)
    for k in range(len(ops)):
        _close(hc[:, k], want[:, k])
        _close(out[k], want[:, k].sum(axis=0))


def _averaged_links(dims, links):
    """U[hypercube][A][D], the means over the shortest paths, in long double."""
    lx, ly, lz, lt = dims
    z = np.indices([d // 2 for d in dims][::-1]).reshape(4, -1)[::-1]
    st = np.array([1, lx, lx * ly, lx * ly * lz])
    base = 2 * (z * st[:, None]).sum(0)
    site = np.stack([base + sum(st[m] for m in range(4) if a >> m & 1) for a in range(16)], 1)
    u = np.zeros((len(base), 16, 16, 3, 3), dtype=np.clongdouble)
    u[:, range(16), range(16)] = np.eye(3)
    l = links.astype(np.clongdouble)
    for n in range(1, 5):
        for a in range(16):
            for x in (x for x in range(16) if bin(x).count('1') == n):
                for m in (m for m in range(4) if x >> m & 1):
                    b = a ^ (1 << m)
                    s = l[site[:, a], m] if b > a else np.conj(np.swapaxes(l[site[:, b], m], 1, 2))
                    u[:, a, a ^ x] += s @ u[:, b, a ^ x] / np.longdouble(n)
    return site, u


def _sandwiches(dims, links, props):
    site, u = _averaged_links(dims, links)
    g = [p.astype(np.clongdouble)[site] for p in props]
    p = np.einsum('hxca,hxycd,hydb->hxyab', np.conj(g[0]), u, g[3], optimize=True)
    q = np.einsum('hxca,hxycd,hydb->hxyab', np.conj(g[2]), u, g[1], optimize=True)
    return p, q


@pytest.mark.parametrize('what', ['gauss', 'opposite2', 'opposite8', 'opposite64', 'opposite1024',
                                  'corners', 'columns', 'disjoint', 'zero_corner', 'tiny_column',
                                  'one_column'])
def test_every_output_on_the_scale_of_its_own_products(sq, what):
    """Flavours that peak at different corners or source colours.  An output
    sums 256 products of P and Q: with R the root of the sum of their squared
    magnitudes, FP64 rounding leaves some 2e-15 R at most (P and Q a few ulp
    each, sums of 64 terms); 64 ulp of R = 7.1e-15 is allowed, against long
    double."""
    dims = (4, 4, 2, 4)
    links, props = _inputs(dims, seed=8)
    vol = oracle.volume(dims)
    rng = np.random.default_rng(9)
    lx, ly, lz, lt = dims
    lex = np.arange(vol)
    corner = (lex % lx & 1) + 2 * (lex // lx % ly & 1) + 4 * (lex // (lx * ly) % lz & 1) + \
        8 * (lex // (lx * ly * lz) & 1)
    s = [np.ones((vol, 1, 3)) for _ in range(4)]
    if what.startswith('opposite'):
        for f, c in ((0, 0), (3, 0), (1, 15), (2, 15)):
            s[f][corner == c] = float(what[8:])
    elif what == 'corners':
        s = [np.exp(rng.uniform(-3, 3, (vol, 1, 1))) * np.ones((1, 1, 3)) for _ in range(4)]
    elif what == 'columns':
        s = [np.exp(rng.uniform(-2, 2, (1, 1, 3))) * np.ones((vol, 1, 1)) for _ in range(4)]
    elif what == 'disjoint':  # no operator has all its products zero, most have few
        for f, c in ((0, 3), (1, 3), (2, 5), (3, 6)):
            s[f][(corner & c) != 0] = 0.0
    elif what == 'zero_corner':
        s[1][corner == 6] = 0.0
    elif what == 'tiny_column':
        s[2][:, :, 1] = 1e-20
    elif what == 'one_column':
        for f in range(4):
            s[f][:, :, 1:] = 0.0
    props = [p * w for p, w in zip(props, s)]
    ops = OPS16[:4] + OPS16[8:]
    _, hc = _gpu(sq, dims, links, props, ops)
    p, q = _sandwiches(dims, links, props)
    a = np.arange(16)
    for k, (s1, f1, s2, f2) in enumerate(ops):
        sign = [oracle.spin_taste(x, y)[a, a ^ x ^ y].real for x, y in ((s1, f1), (s2, f2))]
        pk = p[:, :, a ^ s2 ^ f2] * (sign[0][:, None] * sign[1][None, :])[None, :, :, None, None]
        qk = q[:, :, a ^ s1 ^ f1].transpose(0, 2, 1, 3, 4)  # [A][C]
        want = np.einsum('hacxw,haczy->hxyzw', pk, qk)
        r = np.sqrt(np.einsum('hacxw,haczy->hxyzw', np.abs(pk) ** 2, np.abs(qk) ** 2))
        assert np.all(np.abs(hc[:, k] - want) <= 64 * 2.0 ** -53 * r)
