"""The work a user of this library has it do, as cases that can be timed.

A case is one call (or one short stream of calls) of the public Python
binding on a lattice from the range the tests, the benchmark and the serving
configuration cover: 8^4 up to 32^3 x 64, cubic and ragged, FP64, FP32 and
16-bit storage, 18- and 12-real long links, one right-hand side, batches and
shifted systems.  ``listed`` names the fixed cases, ``draw`` gives others of
the same ranges, ``exact`` the same results in plain torch complex128.

Solves run to a relative residual of 1e-12, the tolerance the tests solve
their reference solutions to, at masses 0.02 to 0.1.  A program solves many
sources on one gauge field, so ``prepare`` leaves the field loaded and the
solver's workspace made by a first short solve.
"""

import math

import numpy as np
import torch

from paper_1411_2223_gb300 import sq

C1, C3, STAPLE_WEIGHT = 9.0 / 8.0, -1.0 / 24.0, 0.1
ASQTAD = (5.0 / 8.0, 1.0 / 16.0, 1.0 / 64.0, 1.0 / 384.0, -1.0 / 16.0, -1.0 / 24.0)
TOL = 1e-12

# --------------------------------------------------------------------- cases


def listed():
    return [
        # the smallest served volume: one mixed-precision solve, where launches
        # and the latency of each dependent step count
        dict(name='solve_8', kind='solve', lx=8, ly=8, lz=8, lt=8, nrhs=1, prec='f32', recon=18,
             mass=0.05),
        # the paper's lattice: one mixed-precision solve of one source
        dict(name='solve_20x64', kind='solve', lx=20, ly=20, lz=20, lt=64, nrhs=1, prec='f32',
             recon=18, mass=0.02),
        # 16-bit storage with 12-real long links at the largest lattice
        dict(name='solve_i16_32x64', kind='solve', lx=32, ly=32, lz=32, lt=64, nrhs=1, prec='i16',
             recon=12, mass=0.02),
        # a propagator: 12 right-hand sides in one batched solve
        dict(name='solve_24x64_12rhs', kind='solve', lx=24, ly=24, lz=24, lt=64, nrhs=12,
             prec='f32', recon=18, mass=0.02),
        # 8 quark masses from one source
        dict(name='multishift_24x64_8', kind='multishift', lx=24, ly=24, lz=24, lt=64, nshift=8,
             prec='f32', recon=18, mass=0.02, mass_hi=0.1),
        # both parities, FP64 throughout, at a middle served volume
        dict(name='full_f64_16x32', kind='full', lx=16, ly=16, lz=16, lt=32, prec='f64', recon=18,
             mass=0.05),
        # the operator alone on the paper's lattice, FP32
        dict(name='dslash_f32_20x64', kind='dslash', lx=20, ly=20, lz=20, lt=64, nrhs=1,
             prec='f32', recon=18, parity=1),
        # the operator on a batch of 12 vectors
        dict(name='dslash_f32_24x64_12rhs', kind='dslash', lx=24, ly=24, lz=24, lt=64, nrhs=12,
             prec='f32', recon=18, parity=0),
        # the FP64 whole-lattice operator on a ragged lattice (residual checks)
        dict(name='dirac_f64_ragged', kind='dirac', lx=14, ly=18, lz=22, lt=54, mass=0.02),
        # fat and Naik links of a new configuration (MILC's asqtad path set)
        dict(name='asqtad_20x64', kind='asqtad', lx=20, ly=20, lz=20, lt=64),
        # the four-fermion operators of the B_K basis, summed over the lattice
        dict(name='npr_20x64_8ops', kind='npr', lx=20, ly=20, lz=20, lt=64, nops=8, per_cube=False),
        # a burst of requests on four resident fields, as a serving process sees it
        dict(name='serve_mix', kind='serve', requests=24, mass=0.02, mass_hi=0.05, fields=4),
    ]


def _even(rng, lo, hi):
    """An even extent, spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)))


def _draw_dims(rng, most_sites, lo=8, hi=32, lt_hi=64):
    while True:
        d = [_even(rng, lo, hi) for _ in range(3)] + [_even(rng, lo, lt_hi)]
        if d[0] * d[1] * d[2] * d[3] <= most_sites:
            return dict(lx=d[0], ly=d[1], lz=d[2], lt=d[3])


def draw(rng):
    kind = rng.choice(['solve', 'solve', 'batch', 'multishift', 'full', 'dslash', 'dslash',
                       'dirac', 'asqtad', 'npr', 'serve'])
    mass = round(math.exp(rng.uniform(math.log(0.02), math.log(0.1))), 4)
    if kind == 'solve':
        prec = rng.choice(['f32', 'f32', 'i16'])
        return dict(kind='solve', nrhs=1, prec=prec, recon=rng.choice([18, 12]), mass=mass,
                    **_draw_dims(rng, 1 << 20))
    if kind == 'batch':
        return dict(kind='solve', nrhs=rng.randint(2, 12), prec='f32', recon=18, mass=mass,
                    **_draw_dims(rng, 24 ** 3 * 48))
    if kind == 'multishift':
        return dict(kind='multishift', nshift=rng.randint(2, 8), prec='f32', recon=18, mass=0.02,
                    mass_hi=max(0.03, mass), **_draw_dims(rng, 24 ** 3 * 48))
    if kind == 'full':
        return dict(kind='full', prec=rng.choice(['f64', 'f32']), recon=18, mass=mass,
                    **_draw_dims(rng, 16 ** 3 * 48))
    if kind == 'dslash':
        prec = rng.choice(['f32', 'f32', 'f64'])
        return dict(kind='dslash', nrhs=rng.choice([1, 1, rng.randint(2, 16)]), prec=prec,
                    recon=rng.choice([18, 12]), parity=rng.randint(0, 1),
                    **_draw_dims(rng, 24 ** 3 * 64))
    if kind == 'dirac':
        return dict(kind='dirac', mass=mass, **_draw_dims(rng, 24 ** 3 * 64))
    if kind == 'asqtad':
        return dict(kind='asqtad', **_draw_dims(rng, 20 ** 3 * 64, lo=6))
    if kind == 'npr':
        per_cube = rng.random() < 0.3
        return dict(kind='npr', nops=rng.randint(1, 20), per_cube=per_cube,
                    **_draw_dims(rng, 1 << (15 if per_cube else 18), lo=4))
    return dict(kind='serve', requests=rng.randint(4, 24), mass=0.02, mass_hi=0.05,
                fields=rng.randint(1, 4))


SERVE_DIMS = [(8, 8, 8, 8), (16, 16, 16, 32), (20, 20, 20, 64), (24, 24, 24, 48)]


def _dims(case):
    return (case['lx'], case['ly'], case['lz'], case['lt'])


def _vol(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


# ------------------------------------------------------------------ synthesis


def _gen(seed, *salt):
    g = torch.Generator(device='cuda')
    g.manual_seed((seed * 1000003 + sum((k + 1) * 7919 * s for k, s in enumerate(salt))) % (1 << 62))
    return g


def _thin(dims, eps, gen):
    """Near-identity SU(3) links (V, 4, 3, 3): the unitary part of
    1 + i eps H - (eps H)^2 / 2 with H = sum_a omega_a lambda_a / 2."""
    n = 4 * _vol(dims)
    w = torch.randn(8, n, generator=gen, device='cuda', dtype=torch.float64) * (0.5 * eps)
    h = torch.empty((3, 3, n), device='cuda', dtype=torch.complex128)
    h[0, 0] = w[2] + w[7] / math.sqrt(3)
    h[1, 1] = -w[2] + w[7] / math.sqrt(3)
    h[2, 2] = -2 * w[7] / math.sqrt(3)
    for (i, j), (a, b) in {(0, 1): (0, 1), (0, 2): (3, 4), (1, 2): (5, 6)}.items():
        h[i, j] = torch.complex(w[a], -w[b])
        h[j, i] = torch.complex(w[a], w[b])
    rows = []
    for i in range(2):
        r = [1j * h[i, j] - 0.5 * (h[i, 0] * h[0, j] + h[i, 1] * h[1, j] + h[i, 2] * h[2, j])
             for j in range(3)]
        r[i] = r[i] + 1
        rows.append(r)
    a, b = rows
    norm = torch.sqrt(sum(x.real ** 2 + x.imag ** 2 for x in a))
    a = [x / norm for x in a]
    dot = sum(x.conj() * y for x, y in zip(a, b))
    b = [y - dot * x for x, y in zip(a, b)]
    norm = torch.sqrt(sum(x.real ** 2 + x.imag ** 2 for x in b))
    b = [x / norm for x in b]
    c = [(a[(k + 1) % 3] * b[(k + 2) % 3] - a[(k + 2) % 3] * b[(k + 1) % 3]).conj()
         for k in range(3)]
    return torch.stack(a + b + c, dim=1).reshape(_vol(dims), 4, 3, 3).contiguous()


def _gauss(shape, gen):
    x = torch.randn(tuple(shape) + (2,), generator=gen, device='cuda', dtype=torch.float64)
    return torch.view_as_complex(x)


EPS = 0.25
_CTX = None


def _context():
    """The process's one context, as a program keeps it."""
    global _CTX
    if _CTX is None:
        _CTX = sq.Context(0)
    return _CTX


class _Field:
    """A gauge field resident in the context, released with the state."""

    def __init__(self, dims, gen):
        self.ctx = _context()
        u = _thin(dims, EPS, gen)
        fat, lng = torch.empty_like(u), torch.empty_like(u)
        self.ctx.gauge_fatten(dims, u, fat, lng, C1, C3, STAPLE_WEIGHT)
        torch.cuda.synchronize()
        self.gid = self.ctx.gauge_load(dims, fat, lng)
        self.vh = _vol(dims) // 2

    def __del__(self):
        try:
            self.ctx.gauge_free(self.gid)
        except Exception:  # the process may be ending
            pass


def _bk_ops(n, gen):
    """n operators: the eight of the B_K basis, then others."""
    ops = [(1 << m, 15, 1 << m, 15) for m in range(4)]
    ops += [(15 ^ (1 << m), 15, 15 ^ (1 << m), 15) for m in range(4)]
    more = torch.randint(0, 16, (max(0, n - 8), 4), generator=gen, device='cuda').tolist()
    return (ops + [tuple(o) for o in more])[:n]


def _masses(case, n):
    lo, hi = case['mass'], case['mass_hi']
    return [lo * (hi / lo) ** (k / max(1, n - 1)) for k in range(n)]


def _requests(case, seed):
    """(field, mass) of each request of a burst."""
    r = np.random.default_rng(seed)
    n = case['requests']
    which = [k % case['fields'] for k in range(n)]
    return [(f, float(m)) for f, m in zip(which, r.uniform(case['mass'], case['mass_hi'], n))]


def _inputs(case, seed):
    """What prepare() and exact() both start from: thin links and vectors."""
    k = case['kind']
    if k == 'serve':
        reqs = _requests(case, seed)
        out = {'reqs': reqs, 'b': []}
        for j, (f, _) in enumerate(reqs):
            out['b'].append(_gauss((_vol(SERVE_DIMS[f]) // 2, 3), _gen(seed, 11, j)))
        return out
    dims = _dims(case)
    vol = _vol(dims)
    if k == 'solve':
        return {'b': _gauss((case['nrhs'], vol // 2, 3), _gen(seed, 3))}
    if k == 'multishift':
        return {'b': _gauss((vol // 2, 3), _gen(seed, 3))}
    if k in ('full', 'dirac'):
        return {'b': _gauss((vol, 3), _gen(seed, 3))}
    if k == 'dslash':
        return {'b': _gauss((case['nrhs'], vol // 2, 3), _gen(seed, 3))}
    if k == 'asqtad':
        return {'thin': _thin(dims, EPS, _gen(seed, 1))}
    return {'thin': _thin(dims, EPS, _gen(seed, 1)),
            'props': [_gauss((vol, 3, 3), _gen(seed, 5, f)) for f in range(4)],
            'ops': _bk_ops(case['nops'], _gen(seed, 9))}


# ------------------------------------------------------------- prepare and run


def prepare(case, seed):
    s = {'case': case, **_inputs(case, seed)}
    k = case['kind']
    ctx = s['ctx'] = _context()
    if k == 'serve':
        s['fields'] = [_Field(SERVE_DIMS[f], _gen(seed, 1, f)) for f in range(case['fields'])]
        s['b'] = [b.cpu().numpy() for b in s['b']]  # requests arrive in host memory
        for f in range(min(case['fields'], len(s['b']))):  # the fields' batches exist
            ctx.serve_poll(ctx.serve_submit(s['fields'][f].gid, s['b'][f], 0.1, 0.5), want_x=False)
        return s
    dims = _dims(case)
    if k == 'asqtad':
        s['fat'], s['lng'] = torch.empty_like(s['thin']), torch.empty_like(s['thin'])
        return s
    if k == 'npr':
        n, hc = case['nops'], _vol(dims) // 16
        s['out'] = torch.empty((n, 3, 3, 3, 3), dtype=torch.complex128, device='cuda')
        if case['per_cube']:
            s['hc'] = torch.empty((hc, n, 3, 3, 3, 3), dtype=torch.complex128, device='cuda')
        return s
    f = s['field'] = _Field(dims, _gen(seed, 1))
    if k == 'dslash':
        nbytes, _ = ctx.spinor_bytes(f.gid, case['prec'])
        s['in'] = torch.zeros((case['nrhs'], nbytes), dtype=torch.uint8, device='cuda')
        s['out'] = torch.zeros_like(s['in'])
        for j in range(case['nrhs']):
            ctx.pack_spinor(f.gid, case['prec'], s['b'][j], s['in'][j])
    elif k == 'dirac':
        s['out'] = torch.empty_like(s['b'])
    elif k == 'solve':
        ctx.cg_solve_multi(f.gid, s['b'], [0.1] * case['nrhs'], 0.5, precision=case['prec'],
                           long_recon=case['recon'], check=False)
    elif k == 'multishift':
        ctx.cg_solve_multishift(f.gid, s['b'], _masses(case, case['nshift']), 0.5,
                                precision=case['prec'], long_recon=case['recon'], check=False)
    elif k == 'full':
        ctx.cg_solve_full(f.gid, s['b'], 0.1, 0.5, precision=case['prec'],
                          long_recon=case['recon'], check=False)
    return s


def run(s):
    case, ctx, k = s['case'], s['ctx'], s['case']['kind']
    if k == 'solve':
        gid = s['field'].gid
        if case['nrhs'] == 1:
            return ctx.cg_solve(gid, s['b'][0], case['mass'], TOL, precision=case['prec'],
                                long_recon=case['recon'])[0]
        return ctx.cg_solve_multi(gid, s['b'], [case['mass']] * case['nrhs'], TOL,
                                  precision=case['prec'], long_recon=case['recon'])[0]
    if k == 'multishift':
        return ctx.cg_solve_multishift(s['field'].gid, s['b'], _masses(case, case['nshift']), TOL,
                                       precision=case['prec'], long_recon=case['recon'])[0]
    if k == 'full':
        return ctx.cg_solve_full(s['field'].gid, s['b'], case['mass'], TOL,
                                 precision=case['prec'], long_recon=case['recon'])[0]
    if k == 'dslash':
        gid, real = s['field'].gid, torch.float64 if case['prec'] == 'f64' else torch.float32
        if case['nrhs'] == 1:
            ctx.dslash_apply(gid, case['parity'], case['prec'], case['recon'], s['in'], s['out'])
        else:
            ctx.dslash_apply_multi(gid, case['parity'], case['prec'], case['recon'], case['nrhs'],
                                   s['in'], s['out'])
        return s['out'].view(real)
    if k == 'dirac':
        ctx.dirac_apply(s['field'].gid, case['mass'], s['b'], s['out'])
        return s['out']
    if k == 'asqtad':
        ctx.gauge_fatten_asqtad(_dims(case), s['thin'], s['fat'], s['lng'], ASQTAD)
        return s['fat'], s['lng']
    if k == 'npr':
        ctx.npr_four_fermion(_dims(case), s['thin'], s['props'], s['ops'], s['out'], s.get('hc'))
        return (s['out'], s['hc']) if 'hc' in s else s['out']
    tickets = [ctx.serve_submit(s['fields'][f].gid, b, m, TOL)
               for (f, m), b in zip(s['reqs'], s['b'])]
    return [ctx.serve_poll(t, vh=s['fields'][f].vh)[1] for t, (f, _) in zip(tickets, s['reqs'])]


# ------------------------------------------------------------------------ work

FLOPS_PER_SITE = 1146  # of the operator, per output site


def _iterations(mass, tol=TOL):
    """About the CG iterations a solve takes on these fields."""
    return math.log(1 / tol) / (0.038 + 1.07 * mass)


def _link_bytes(prec, recon):
    """Bytes of the 16 hop matrices of one output site."""
    real = {'f64': 8, 'f32': 4, 'i16': 2}[prec]
    return 8 * (18 + recon) * real


def _vec_bytes(prec):
    return {'f64': 48, 'f32': 24, 'i16': 16}[prec]


def _cg_work(vh, nrhs, prec, recon, mass):
    """Per iteration: the links of both parities once, and per system the
    gathered fields, t out and in, and p, r, x of the update."""
    v, x = _vec_bytes(prec), _vec_bytes('f64' if prec == 'f64' else 'f32')
    it = _iterations(mass)
    per_site = 2 * _link_bytes(prec, recon) + nrhs * (9 * v + 2 * x)
    return {'bytes': it * vh * per_site, 'flops': it * vh * nrhs * (2 * FLOPS_PER_SITE + 72)}


def work(case):
    k = case['kind']
    if k == 'serve':
        b = f = 0.0
        m = math.sqrt(case['mass'] * case['mass_hi'])
        for j in range(case['fields']):
            n = len(range(j, case['requests'], case['fields']))
            w = _cg_work(_vol(SERVE_DIMS[j]) // 2, n, 'f32', 18, m)
            b, f = b + w['bytes'], f + w['flops']
        return {'bytes': b, 'flops': f}
    dims = _dims(case)
    vol, vh = _vol(dims), _vol(dims) // 2
    if k in ('solve', 'full'):
        return _cg_work(vh, case.get('nrhs', 1), case['prec'], case['recon'], case['mass'])
    if k == 'multishift':
        w = _cg_work(vh, 1, case['prec'], case['recon'], case['mass'])
        it, ns = _iterations(case['mass']), case['nshift']
        return {'bytes': w['bytes'] + it * vh * (ns - 1) * 96.0,
                'flops': w['flops'] + it * vh * (ns - 1) * 48.0}
    if k == 'dslash':
        n = case['nrhs']
        return {'bytes': vh * (_link_bytes(case['prec'], case['recon'])
                               + 2.0 * n * _vec_bytes(case['prec'])),
                'flops': vh * n * float(FLOPS_PER_SITE)}
    if k == 'dirac':
        return {'bytes': vol * (_link_bytes('f64', 18) + 96.0), 'flops': vol * 1158.0}
    if k == 'asqtad':
        # 170 SU(3) products and 85 scaled additions per link, as nested staples
        return {'bytes': vol * 4 * 144 * 3.0, 'flops': vol * 4 * 39330.0}
    hc, n = vol // 16, case['nops']
    groups = -(-n // 16)
    out = 81 * 16.0 * n * (hc if case['per_cube'] else 1)
    # per hypercube: 224 products of the averaged links and 1024 of the
    # sandwiches (216 each) per group of operators; 256 x 81 terms per operator
    flops = hc * (groups * (224 + 1024) * 216.0 + n * 256 * 81 * 8.0)
    return {'bytes': vol * (4 * 144.0 + 2 * 144.0) + out, 'flops': flops}


# ------------------------------------------------- the same in 64 bits, in torch


def _grid(a, dims):
    return a.reshape((dims[3], dims[2], dims[1], dims[0]) + tuple(a.shape[1:]))


def _shift(a, dims, mu, d):
    """a(x + d mu), a of shape (V, ...)."""
    return torch.roll(_grid(a, dims), -d, dims=3 - mu).reshape(a.shape)


def _dag(m):
    return m.conj().transpose(-1, -2)


def _mm(a, b):
    """3 x 3 products of (V, 3, 3) fields."""
    return sum(a[:, :, k, None] * b[:, None, k, :] for k in range(3))


def _fat_long(u, dims):
    fat, lng = torch.empty_like(u), torch.empty_like(u)
    for mu in range(4):
        um = u[:, mu]
        st = torch.zeros_like(um)
        for nu in range(4):
            if nu == mu:
                continue
            un = u[:, nu]
            st += _mm(_mm(un, _shift(um, dims, nu, 1)), _dag(_shift(un, dims, mu, 1)))
            st += _shift(_mm(_mm(_dag(un), um), _shift(un, dims, mu, 1)), dims, nu, -1)
        fat[:, mu] = C1 * (um + STAPLE_WEIGHT * st) / (1 + 6 * STAPLE_WEIGHT)
        lng[:, mu] = C3 * _mm(_mm(um, _shift(um, dims, mu, 1)), _shift(um, dims, mu, 2))
    return fat, lng


class _Operator:
    """D between the parities as one (Vh, 3, 48) matrix per output site."""

    def __init__(self, dims, gen):
        self.dims = dims
        fat, lng = _fat_long(_thin(dims, EPS, gen), dims)
        vol = _vol(dims)
        i = torch.arange(vol, device='cuda')
        c, r = [], i
        for L in dims:
            c.append(r % L)
            r = r // L
        par = (c[0] + c[1] + c[2] + c[3]) & 1
        self.sites = [i[par == p] for p in (0, 1)]
        rank = torch.div(i, 2, rounding_mode='floor')  # index within its parity
        self.mat, self.nbr = [], []
        eta = [torch.ones_like(i), 1 - 2 * (c[0] & 1), 1 - 2 * ((c[0] + c[1]) & 1),
               1 - 2 * ((c[0] + c[1] + c[2]) & 1)]
        blocks, nbrs = [], []
        for mu in range(4):
            for links, d in ((fat, 1), (lng, 3)):
                e = 0.5 * eta[mu].to(torch.float64)[:, None, None]
                blocks.append(e * links[:, mu])
                nbrs.append(rank[_shift(i, dims, mu, d)])
                blocks.append(-e * _dag(_shift(links[:, mu].contiguous(), dims, mu, -d)))
                nbrs.append(rank[_shift(i, dims, mu, -d)])
        for p in (0, 1):
            s = self.sites[p]
            self.mat.append(torch.cat([b[s] for b in blocks], dim=2))
            self.nbr.append(torch.stack([n[s] for n in nbrs], dim=1))

    def apply(self, p, v):
        """D_{p,1-p} v for v (Vh, 3, n)."""
        out = torch.empty_like(v)
        step = max(1, (1 << 26) // (48 * v.shape[2]))
        for a in range(0, v.shape[0], step):
            nb = self.nbr[p][a:a + step]
            g = v[nb].reshape(nb.shape[0], 48, v.shape[2])
            out[a:a + step] = torch.bmm(self.mat[p][a:a + step], g)
        return out

    def solve(self, b, masses):
        """(m_j^2 - D_eo D_oe) x_j = b_j by CG, b (Vh, 3, n)."""
        m2 = torch.tensor([m * m for m in masses], device='cuda', dtype=torch.float64)
        x, r = torch.zeros_like(b), b.clone()
        p = r.clone()
        dot = lambda y: (y.real ** 2 + y.imag ** 2).sum(dim=(0, 1))  # noqa: E731
        rr = dot(r)
        stop = rr * 1e-26
        for _ in range(4000):
            t = self.apply(1, p)
            pap = m2 * dot(p) + dot(t)
            ap = m2 * p - self.apply(0, t)
            al = torch.where(rr > stop, rr / pap, torch.zeros_like(rr))
            x += al * p
            r -= al * ap
            new = dot(r)
            if bool((new <= stop).all()):
                break
            p = r + torch.where(rr > stop, new / rr, torch.zeros_like(rr)) * p
            rr = new
        return x


def _exact_asqtad(u, dims):
    one, three, five, seven, lepage, naik = ASQTAD
    fat, lng = torch.empty_like(u), torch.empty_like(u)

    def staple(w, mu, nu, s):
        un = u[:, nu].contiguous()
        if s > 0:
            return _mm(_mm(un, _shift(w, dims, nu, 1)), _dag(_shift(un, dims, mu, 1)))
        return _shift(_mm(_mm(_dag(un), w), _shift(un, dims, mu, 1)), dims, nu, -1)

    for mu in range(4):
        um = u[:, mu].contiguous()
        acc = one * um
        for nu in range(4):
            if nu == mu:
                continue
            for s in (-1, 1):
                s3 = staple(um, mu, nu, s)
                acc += three * s3 + lepage * staple(s3, mu, nu, s)
                for rho in range(4):
                    if rho in (mu, nu):
                        continue
                    for t in (-1, 1):
                        s5 = staple(s3, mu, rho, t)
                        sg = 6 - mu - nu - rho
                        acc += five * s5
                        acc += seven * (staple(s5, mu, sg, -1) + staple(s5, mu, sg, 1))
        fat[:, mu] = acc
        lng[:, mu] = naik * _mm(_mm(um, _shift(um, dims, mu, 1)), _shift(um, dims, mu, 2))
    return fat, lng


def _spin_taste(s, f):
    """(partner, sign) of the rows of (gamma_S x xi_F), from gamma matrices."""
    sx, sy, sz, i2 = (np.array(m, dtype=complex) for m in (
        [[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]], [[1, 0], [0, 1]]))
    g = [np.kron(sy, sx), np.kron(sy, sy), np.kron(sy, sz), np.kron(sx, i2)]

    def gam(m):
        out = np.eye(4, dtype=complex)
        for mu in range(4):
            if (m >> mu) & 1:
                out = out @ g[mu]
        return out

    part, sign = [], []
    for a in range(16):
        b = a ^ s ^ f
        t = np.trace(gam(a).conj().T @ gam(s) @ gam(b) @ gam(f).conj().T) / 4
        part.append(b)
        sign.append(float(round(t.real)))
    return part, sign


def _exact_npr(case, inp):
    dims = _dims(case)
    hc = [d // 2 for d in dims]
    ncube = hc[0] * hc[1] * hc[2] * hc[3]
    z = torch.arange(ncube, device='cuda')
    base, r, st = torch.zeros_like(z), z, 1
    for mu in range(4):
        base, r = base + 2 * (r % hc[mu]) * st, r // hc[mu]
        st *= dims[mu]
    strides = [1, dims[0], dims[0] * dims[1], dims[0] * dims[1] * dims[2]]
    off = [sum(strides[mu] for mu in range(4) if (a >> mu) & 1) for a in range(16)]
    nops = case['nops']
    total = torch.zeros((nops, 81), dtype=torch.complex128, device='cuda')
    cubes = [] if case['per_cube'] else None
    for z0 in range(0, ncube, 4096):
        b = base[z0:z0 + 4096]
        n = b.shape[0]
        link = {}
        eye = torch.eye(3, dtype=torch.complex128, device='cuda').expand(n, 3, 3)
        for a in range(16):
            link[a, a] = eye
            for mu in range(4):
                if not (a >> mu) & 1:
                    u = inp['thin'][b + off[a], mu]
                    link[a, a | (1 << mu)], link[a | (1 << mu), a] = u, _dag(u)
        for dist in (2, 3, 4):
            for a in range(16):
                for d in range(16):
                    if bin(a ^ d).count('1') == dist:
                        mid = [a ^ (1 << mu) for mu in range(4) if ((a ^ d) >> mu) & 1]
                        link[a, d] = sum(_mm(link[a, m], link[m, d]) for m in mid) / dist
        g = [torch.stack([p[b + off[a]] for a in range(16)], 1) for p in inp['props']]
        uu = torch.stack([torch.stack([link[a, d] for d in range(16)], 1) for a in range(16)], 1)
        P = torch.einsum('zaci,zadck,zdkj->zadij', g[0].conj(), uu, g[3])
        Q = torch.einsum('zaci,zadck,zdkj->zadij', g[2].conj(), uu, g[1])
        outs = []
        for s1, f1, s2, f2 in inp['ops']:
            p1, g1 = _spin_taste(s1, f1)
            p2, g2 = _spin_taste(s2, f2)
            sg = torch.tensor(np.outer(g1, g2), device='cuda')
            pp = P[:, :, p2] * sg[None, :, :, None, None]      # [z, A, C, a1, a4]
            qq = Q[:, :, p1].transpose(1, 2)                   # [z, A, C, a3, a2]
            o = torch.bmm(pp.reshape(n, 256, 9).transpose(1, 2), qq.reshape(n, 256, 9))
            o = o.reshape(n, 3, 3, 3, 3).permute(0, 1, 4, 3, 2)  # a1 a4 a3 a2 -> a1 a2 a3 a4
            outs.append(o.reshape(n, 81))
        o = torch.stack(outs, 1)
        total += o.sum(0)
        if cubes is not None:
            cubes.append(o.reshape(n, nops, 3, 3, 3, 3))
    total = total.reshape(nops, 3, 3, 3, 3)
    return total if cubes is None else (total, torch.cat(cubes))


def _packed(v, prec, dims):
    """Canonical (n, Vh, 3) complex128 as the packed planes, in 64-bit reals."""
    n, vh, _ = v.shape
    stride = (vh + 63) // 64 * 64
    r = torch.view_as_real(v)  # n, vh, 3, 2
    if prec == 'f64':
        out = torch.zeros((n, 3, stride, 2), dtype=torch.float64, device=v.device)
        out[:, :, :vh] = r.transpose(1, 2)
        return out.reshape(n, -1)
    a = torch.zeros((n, stride, 4), dtype=torch.float64, device=v.device)
    c = torch.zeros((n, stride, 2), dtype=torch.float64, device=v.device)
    a[:, :vh] = r[:, :, :2].reshape(n, vh, 4)
    c[:, :vh] = r[:, :, 2]
    return torch.cat([a.reshape(n, -1), c.reshape(n, -1)], 1)


def exact(case, seed):
    inp, k = _inputs(case, seed), case['kind']
    if k == 'serve':
        out = [None] * len(inp['reqs'])
        for f in range(case['fields']):
            op = _Operator(SERVE_DIMS[f], _gen(seed, 1, f))
            mine = [j for j, (g, _) in enumerate(inp['reqs']) if g == f]
            if mine:
                x = op.solve(torch.stack([inp['b'][j] for j in mine], -1),
                             [inp['reqs'][j][1] for j in mine])
                for n, j in enumerate(mine):
                    out[j] = x[..., n].contiguous().cpu().numpy()
        return out
    dims = _dims(case)
    if k == 'asqtad':
        return _exact_asqtad(inp['thin'], dims)
    if k == 'npr':
        return _exact_npr(case, inp)
    op = _Operator(dims, _gen(seed, 1))
    b = inp['b']
    if k == 'solve':
        x = op.solve(b.permute(1, 2, 0).contiguous(), [case['mass']] * case['nrhs'])
        x = x.permute(2, 0, 1).contiguous()
        return x[0] if case['nrhs'] == 1 else x
    if k == 'multishift':
        ms = _masses(case, case['nshift'])
        x = op.solve(b[..., None].repeat(1, 1, len(ms)), ms)
        return x.permute(2, 0, 1).contiguous()
    if k == 'dslash':
        v = op.apply(case['parity'], b.permute(1, 2, 0).contiguous()).permute(2, 0, 1).contiguous()
        return _packed(v, case['prec'], dims)
    even, odd = (b[s][..., None] for s in op.sites)
    out = torch.empty_like(b)
    if k == 'dirac':
        out[op.sites[0]] = (case['mass'] * even + op.apply(0, odd))[..., 0]
        out[op.sites[1]] = (case['mass'] * odd + op.apply(1, even))[..., 0]
        return out
    m = case['mass']
    xe = op.solve(m * even - op.apply(0, odd), [m])
    out[op.sites[0]] = xe[..., 0]
    out[op.sites[1]] = ((odd - op.apply(1, xe)) / m)[..., 0]
    return out
