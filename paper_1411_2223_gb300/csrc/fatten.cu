// Fat and long links from thin links on the GPU, in FP64.
//
// The paper's lattices are MILC asqtad ensembles (Sec. 2, Fig. 1), whose fat
// and Naik links come from the thin gauge links by path sums.  This file
// builds the benchmark workloads' recipe of them from thin links U:
//   F_mu(x) = c1 [ U_mu(x) + w sum_{nu != mu} ( U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
//                + U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu) ) ] / (1 + 6w),
//   L_mu(x) = c3 U_mu(x) U_mu(x+mu) U_mu(x+2mu),
// one thread per (site, direction), periodic neighbours, links in the
// canonical host layout [site_lex][mu][row][col] complex128.  The work is
// FP64 arithmetic (about 2800 flops per link against 432 bytes of traffic),
// so it is bound by the FP64 units, not by HBM.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sq_fixed.cuh"
#include "sq_host.h"

namespace sq {
namespace {

struct M3 {
  double2 e[9];
};

__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }

// c = op(a) op(b), op = identity or dagger; each complex term is four FMAs
// into the accumulator (the FP64 units bound these kernels).
template <bool DA, bool DB>
__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b) {
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double2 t = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double2 x = DA ? cconj(a.e[3 * k + i]) : a.e[3 * i + k];
        const double2 y = DB ? cconj(b.e[3 * j + k]) : b.e[3 * k + j];
        t.x = fma(x.x, y.x, t.x);
        t.x = fma(-x.y, y.y, t.x);
        t.y = fma(x.x, y.y, t.y);
        t.y = fma(x.y, y.x, t.y);
      }
      c.e[3 * i + j] = t;
    }
  }
  return c;
}

struct FatGeom {
  int L[4];
  long st[4];
  long vol;
};

__device__ __forceinline__ M3 load_link(const double2 *u, long s, int mu) {
  M3 m;
  const double2 *p = u + (s * 4 + mu) * 9;
#pragma unroll
  for (int e = 0; e < 9; ++e) m.e[e] = __ldg(p + e);
  return m;
}

// site of x + d * mu_hat, periodic (|d| <= 2)
__device__ __forceinline__ long shift(const FatGeom &g, long s, const int c[4], int mu, int d) {
  int v = c[mu] + d;
  while (v < 0) v += g.L[mu];
  while (v >= g.L[mu]) v -= g.L[mu];
  return s + (long)(v - c[mu]) * g.st[mu];
}

__global__ void __launch_bounds__(128) fatten_kernel(FatGeom g, const double2 *u, double c1,
                                                     double c3, double w, double2 *fat,
                                                     double2 *lng) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4 * g.vol) return;
  const long s = idx >> 2;
  const int mu = (int)(idx & 3);
  int c[4];
  {
    long r = s;
    c[0] = (int)(r % g.L[0]); r /= g.L[0];
    c[1] = (int)(r % g.L[1]); r /= g.L[1];
    c[2] = (int)(r % g.L[2]);
    c[3] = (int)(r / g.L[2]);
  }
  const long xpm = shift(g, s, c, mu, 1);
  const M3 umu = load_link(u, s, mu);
  M3 st;
#pragma unroll
  for (int e = 0; e < 9; ++e) st.e[e] = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    // up staple U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
    const long xpn = shift(g, s, c, nu, 1);
    M3 t = mul<false, false>(load_link(u, s, nu), load_link(u, xpn, mu));
    M3 up = mul<false, true>(t, load_link(u, xpm, nu));
    // down staple U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)
    const long xmn = shift(g, s, c, nu, -1);
    int cm[4] = {c[0], c[1], c[2], c[3]};
    cm[nu] = (c[nu] == 0) ? g.L[nu] - 1 : c[nu] - 1;
    const long xmnpm = shift(g, xmn, cm, mu, 1);
    t = mul<true, false>(load_link(u, xmn, nu), load_link(u, xmn, mu));
    M3 dn = mul<false, false>(t, load_link(u, xmnpm, nu));
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      st.e[e].x += up.e[e].x + dn.e[e].x;
      st.e[e].y += up.e[e].y + dn.e[e].y;
    }
  }
  const double k = c1 / (1.0 + 6.0 * w);
  double2 *f = fat + idx * 9;
#pragma unroll
  for (int e = 0; e < 9; ++e)
    f[e] = make_double2(k * fma(w, st.e[e].x, umu.e[e].x), k * fma(w, st.e[e].y, umu.e[e].y));
  const long xp2m = shift(g, s, c, mu, 2);
  const M3 n = mul<false, false>(mul<false, false>(umu, load_link(u, xpm, mu)),
                                 load_link(u, xp2m, mu));
  double2 *l = lng + idx * 9;
#pragma unroll
  for (int e = 0; e < 9; ++e) l[e] = make_double2(c3 * n.e[e].x, c3 * n.e[e].y);
}

// ---------------------------------------------------------------- asqtad
// The asqtad action's fat link (MILC's path set): the one-link term, the 6
// three-link staples, 24 five-link and 48 seven-link staples and 6 Lepage
// terms, each a product of links along its path, weighted by its
// coefficient; the Naik link is c_N U U U.  Paths, for direction mu, with
// nu, rho, sigma distinct and != mu and every sign s, r, q = +-1:
//   3-staple  (s nu) mu (-s nu)
//   5-staple  (r rho)(s nu) mu (-s nu)(-r rho)
//   7-staple  (q sg)(r rho)(s nu) mu (-s nu)(-r rho)(-q sg)
//   Lepage    (s nu)(s nu) mu (-s nu)(-s nu)
// A hop +d at y multiplies by U_d(y), a hop -d by U_d(y - d)^dag.
//
// Every longer path is a staple around a shorter one,
//   St_{s nu}[W](x) = h(x) W(x + s nu) h(x + mu)^dag,
//   h(y) = U_nu(y) (s = +1) or U_nu(y - nu)^dag (s = -1),
// and St is linear in W, so the paths are summed from the inside out before
// the next staple is put around them, as fields over the lattice:
//   S_{s nu} = St_{s nu}[U_mu],               A_nu = S_{+nu} + S_{-nu}
//   X_sg = c3 U_mu + c5 (A_nu + A_rho) + c7 sum_r (St_{r rho}[A_nu] + St_{r nu}[A_rho])
//   fat = c1 U_mu + sum_{sg, q} St_{q sg}[X_sg + c_L S_{q sg}]
// (nu, rho the two directions besides mu and sg): 24 staples of two SU(3)
// products per link, 48 products, where a staple per path prefix takes 168
// and every path multiplied out 422.
//
// The products run on the integer multiply-add units in the fixed-point form
// of sq_fixed.cuh when every link is unitary to 2^-9, in each element of
// U U^dag - 1.  That matrix's norm is then at most 3 sqrt(2) 2^-9, and every
// field is bounded, as a matrix norm and so in its elements: |U| <= 1.0042,
// |S| <= 1.013, |A| <= 2.03, |Y| <= 8.17 for Y = the sum in X, and
// |X + c_L S| <= 1.022 (|c3| + 4 |c5| + 8 |c7| + |c_L|) < 2^E, so each is kept
// at its own fixed unit (55 bits where it is an operand) and no sum overflows
// (rows and columns of norm 1 would not do: a 3 x 3 matrix of them can have norm
// sqrt(3), and Y then passes the 2^58 units that fat_times takes):
//   U 2^-55, S 2^-55, A 2^-53, Y 2^-55, X 2^(E-60), W = X + c_L S 2^(E-55),
//   T = U W 2^-1 and S = T U 2^-2 of W's unit, |T| <= 2^57, |S| <= 2^59.6 for six.
// Other links go through the same kernels in FP64; the flag is on the device
// and the kernels of the other form return at once.
//
// A thread computes one row of one site's staples (threadIdx.y), so that only
// that row's sums, one row of W and one of U_nu are in registers at a time;
// the rows' loads of the same matrices meet in L1.
//
// 20^3 x 64, tree-level coefficients: 76.9 ms with a staple kernel per path
// prefix in FP64 (FP64 units 96 % busy), 8.8 ms here (9.5 ms before the
// products were written as mad.wide.s32, 16.4 ms with a thread per site, which
// spilled).  The integer multiply-adds alone are 3.2 ms, the fields' traffic
// 1.9 ms of HBM time; the level-2 kernel issues 3830 instructions per warp for
// 930 of them and keeps that pipe 58 % busy.  Error against long double 7.6e-17
// (before: 2.8e-16), with only the seven-link paths 7.8e-17 (1.5e-16).

struct FatScale {
  unsigned uneven;             // a link is not unitary
};

// Slices of the lattice across direction `ax` in scratch: slot (t - t0) mod L for
// the slice at coordinate t, slots 0 .. nslots - 1; in a slice the other three
// directions in their order.
struct Slab {
  FatGeom g;
  int ax, od[3];               // the slices' direction, and the others
  long st[4];                  // scratch strides of the others
  int t0, nslots;
  int first, count;            // slots a kernel writes
  long v3;                     // sites of a slice
  long n;                      // scratch sites: nslots * v3
};

// A coefficient as c = (h, l) 2^(ec - FX_BITS), and the shift that takes its
// product with a field (see fat_times) to X's unit.
struct FatCoef {
  int h, l, down;
};

struct AsqtadArgs {
  Slab sl;
  const FatScale *sc;
  const int4 *u;               // links [mu][e][scratch site]
  int4 *s;                     // S [direction slot 0..2][+, -][e][scratch site]
  int4 *sa;                    // A [direction slot 0..2][e][scratch site]
  int4 *w;                     // W [direction slot 0..2][+, -][e][scratch site]
  double2 *fat;                // [site][mu][9]
  int mu;
  double c1, c3, c5, c7, cl;
  FatCoef f3, f5, f7, fl;
  double w_unit;               // 2^(E - FX_BITS - 2), the unit of level 3's sums
};

constexpr int FAT_SITES = 64;  // sites per block; 3 threads (rows) each

struct SlabSite {
  int c[4];
  long s;      // scratch site
  long lex;    // lattice site
};

__device__ __forceinline__ bool slab_site(const Slab &sl, SlabSite &p) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= sl.count * sl.v3) return false;
  const int dt = (int)(idx / sl.v3);
  const int r3 = (int)(idx - dt * sl.v3);
  const int slot = sl.first + dt;
  int t = sl.t0 + slot;
  if (t >= sl.g.L[sl.ax]) t -= sl.g.L[sl.ax];
  const int l0 = sl.g.L[sl.od[0]], l1 = sl.g.L[sl.od[1]];
  const int c0 = r3 % l0, q = r3 / l0, c1 = q % l1, c2 = q / l1;
  p.lex = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    p.c[k] = k == sl.ax ? t : k == sl.od[0] ? c0 : k == sl.od[1] ? c1 : c2;
    p.lex += p.c[k] * sl.g.st[k];
  }
  p.s = slot * sl.v3 + r3;
  return true;
}

// y + d mu_hat (d = +-1) in scratch; the slabs hold every site asked for
__device__ __forceinline__ SlabSite slab_step(const Slab &sl, const SlabSite &y, int mu, int d) {
  SlabSite z = y;
  const int L = sl.g.L[mu];
  const int cy = mu == 0 ? y.c[0] : mu == 1 ? y.c[1] : mu == 2 ? y.c[2] : y.c[3];
  int v = cy + d;
  if (v < 0) v += L;
  if (v >= L) v -= L;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (k == mu) z.c[k] = v;
  if (mu != sl.ax) {
    z.s = y.s + (long)(v - cy) * sl.st[mu];
  } else {  // whole lattice in scratch: the wrap; else the next slot
    long s = y.s + d * sl.v3;
    if (s < 0) s += sl.n;
    if (s >= sl.n) s -= sl.n;
    z.s = s;
  }
  return z;
}

// ---- fixed-point rows
struct FxWide { long long hr, mr, hi, mi; };

__device__ __forceinline__ void fat_mac(FxWide &w, const int4 a, const int4 b) {  // a b
  const Fx ar = {a.y, a.x}, ai = {a.w, a.z}, br = {b.y, b.x}, bi = {b.w, b.z}, nb = {-b.w, -b.z};
  fx_mac(w.hr, w.mr, ar, br);
  fx_mac(w.hi, w.mi, ar, bi);
  fx_mac(w.hr, w.mr, ai, nb);
  fx_mac(w.hi, w.mi, ai, br);
}
__device__ __forceinline__ int4 fat_conj(const int4 a) { return make_int4(a.x, a.y, -a.z, -a.w); }
__device__ __forceinline__ int2 fat_split(long long v) {
  const long long h = (v + (1ll << (FX_LOW - 1))) >> FX_LOW;
  return make_int2((int)(v - (h << FX_LOW)), (int)h);
}
__device__ __forceinline__ int4 fat_word(long long re, long long im) {
  const int2 r = fat_split(re), i = fat_split(im);
  return make_int4(r.x, r.y, i.x, i.y);
}
__device__ __forceinline__ long long fat_join(int l, int h) { return ((long long)h << FX_LOW) + l; }
// hi 2^FX_LOW + mid without its last FX_LOW bits
__device__ __forceinline__ long long fat_round(long long hi, long long mid) {
  return hi + ((mid + (1ll << (FX_LOW - 1))) >> FX_LOW);
}
__device__ __forceinline__ long long fat_shift(long long v, int s) {
  return s > 0 ? (v + (1ll << (s - 1))) >> s : v;
}
// c v in X's unit (v up to 58 bits)
__device__ __forceinline__ long long fat_times(const FatCoef &c, long long v) {
  const int2 q = fat_split(v);
  long long hi = 0, mid = 0;
  fx_mac(hi, mid, Fx{c.h, c.l}, Fx{q.y, q.x});
  return fat_shift((hi << 4) + (mid >> (FX_LOW - 4)), c.down);
}

struct Row { static constexpr bool fixed = true; long long v[6]; };  // re, im of three elements

// Row i of L W R added to acc; L and R are U_nu or its dagger (DL, DR) at the
// scratch sites ls and rs, W the field w at ws.
template <bool DL, bool DR>
__device__ __forceinline__ void fx_row_staple(const AsqtadArgs &a, int nu, int i, long ls,
                                              const int4 *w, long ws, long rs, Row &acc) {
  const long n = a.sl.n;
  const int4 *u = a.u + (size_t)(9 * nu) * n;
  FxWide z[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) z[j] = {0, 0, 0, 0};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int4 l = __ldg(u + (size_t)(DL ? 3 * k + i : 3 * i + k) * n + ls);
    if (DL) l = fat_conj(l);
#pragma unroll
    for (int j = 0; j < 3; ++j) fat_mac(z[j], l, __ldg(w + (size_t)(3 * k + j) * n + ws));
  }
  int4 t[3];
#pragma unroll
  for (int j = 0; j < 3; ++j)
    t[j] = fat_word(fat_round(z[j].hr, z[j].mr), fat_round(z[j].hi, z[j].mi));
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    FxWide y = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int4 r = __ldg(u + (size_t)(DR ? 3 * j + k : 3 * k + j) * n + rs);
      fat_mac(y, t[k], DR ? fat_conj(r) : r);
    }
    acc.v[2 * j] += fat_round(y.hr, y.mr);
    acc.v[2 * j + 1] += fat_round(y.hi, y.mi);
  }
}

struct RowF { static constexpr bool fixed = false; double v[6]; };

template <bool DL, bool DR>
__device__ __forceinline__ void f64_row_staple(const AsqtadArgs &a, int nu, int i, long ls,
                                               const int4 *w, long ws, long rs, RowF &acc) {
  const long n = a.sl.n;
  const double2 *u = reinterpret_cast<const double2 *>(a.u) + (size_t)(9 * nu) * n;
  const double2 *wd = reinterpret_cast<const double2 *>(w);
  auto mac = [](double2 &z, double2 x, double2 y) {
    z.x = fma(x.x, y.x, z.x);
    z.x = fma(-x.y, y.y, z.x);
    z.y = fma(x.x, y.y, z.y);
    z.y = fma(x.y, y.x, z.y);
  };
  double2 t[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) t[j] = make_double2(0.0, 0.0);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double2 l = __ldg(u + (size_t)(DL ? 3 * k + i : 3 * i + k) * n + ls);
    if (DL) l = cconj(l);
#pragma unroll
    for (int j = 0; j < 3; ++j) mac(t[j], l, __ldg(wd + (size_t)(3 * k + j) * n + ws));
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    double2 y = make_double2(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double2 r = __ldg(u + (size_t)(DR ? 3 * j + k : 3 * k + j) * n + rs);
      mac(y, t[k], DR ? cconj(r) : r);
    }
    acc.v[2 * j] += y.x;
    acc.v[2 * j + 1] += y.y;
  }
}

// Row i of St_{s nu}[w](x) added to acc (Row: fixed point, RowF: FP64).
template <typename R>
__device__ __forceinline__ void row_staple(const AsqtadArgs &a, const SlabSite &x, int nu, int s, int i,
                                           const int4 *w, R &acc) {
  constexpr bool fixed = R::fixed;
  if (s > 0) {  // U_nu(x) W(x + nu) U_nu(x + mu)^dag
    const long ws = slab_step(a.sl, x, nu, 1).s, rs = slab_step(a.sl, x, a.mu, 1).s;
    if constexpr (fixed) fx_row_staple<false, true>(a, nu, i, x.s, w, ws, rs, acc);
    else f64_row_staple<false, true>(a, nu, i, x.s, w, ws, rs, acc);
  } else {      // U_nu(x - nu)^dag W(x - nu) U_nu(x - nu + mu)
    const SlabSite y = slab_step(a.sl, x, nu, -1);
    const long rs = slab_step(a.sl, y, a.mu, 1).s;
    if constexpr (fixed) fx_row_staple<true, false>(a, nu, i, y.s, w, y.s, rs, acc);
    else f64_row_staple<true, false>(a, nu, i, y.s, w, y.s, rs, acc);
  }
}

// The k-th (0..2) direction besides mu.
__device__ __forceinline__ int other_dir(int mu, int k) { return k < mu ? k : k + 1; }

// Are all links unitary?  |U U^dag - 1| < 2^-9 in the parts of every element,
// which NaN and infinities fail.  Bound by the links' loads (76 MB at 16^3 x 32 in
// 22.5 us, 1 % of a call).
__global__ void __launch_bounds__(256) fat_scale_kernel(const double2 *u, long nlinks, FatScale *sc) {
  bool even = true;
  for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < nlinks;
       k += (long)gridDim.x * blockDim.x) {
    float2 m[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const double2 v = __ldg(u + k * 9 + e);
      m[e] = make_float2((float)v.x, (float)v.y);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j <= i; ++j) {
        float re = i == j ? -1.f : 0.f, im = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 x = m[3 * i + c], y = m[3 * j + c];
          re = fmaf(x.x, y.x, fmaf(x.y, y.y, re));
          im = fmaf(x.y, y.x, fmaf(-x.x, y.y, im));
        }
        even = even && fabsf(re) < 1.f / 512 && fabsf(im) < 1.f / 512;
      }
  }
  if (!__all_sync(0xffffffffu, even) && (threadIdx.x & 31) == 0) sc->uneven = 1;
}

// The links of a slab's slots into scratch planes.
__global__ void __launch_bounds__(128) fat_links_kernel(AsqtadArgs a, const double2 *thin, int4 *u) {
  SlabSite p;
  if (!slab_site(a.sl, p)) return;
  const bool fixed = a.sc->uneven == 0;
  const int mu = blockIdx.y;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const double2 v = __ldg(thin + (p.lex * 4 + mu) * 9 + e);
    int4 q;
    if (fixed) {  // |v| <= 1.0042: the units of 2^-55 times elements that may reach 2^1
      const Fx r = fx_from_double(v.x, 1023, 1), i = fx_from_double(v.y, 1023, 1);
      q = fat_word(fat_join(r.l, r.h) * 2, fat_join(i.l, i.h) * 2);
    } else {
      q = make_int4(__double2loint(v.x), __double2hiint(v.x), __double2loint(v.y), __double2hiint(v.y));
    }
    u[(size_t)(9 * mu + e) * a.sl.n + p.s] = q;
  }
}

// lng = c_N U_mu(x) U_mu(x+mu) U_mu(x+2mu), every direction of the slots
template <typename R>
__global__ void __launch_bounds__(3 * FAT_SITES) naik_kernel(AsqtadArgs a, double c_naik, double2 *lng) {
  if ((a.sc->uneven == 0) != R::fixed) return;
  SlabSite x;
  if (!slab_site(a.sl, x)) return;
  const int mu = blockIdx.y, i = threadIdx.y;
  const SlabSite y = slab_step(a.sl, x, mu, 1), z = slab_step(a.sl, y, mu, 1);
  const int4 *w = a.u + (size_t)(9 * mu) * a.sl.n;
  double2 *o = lng + (x.lex * 4 + mu) * 9 + 3 * i;
  R acc{};
  if constexpr (R::fixed) fx_row_staple<false, false>(a, mu, i, x.s, w, y.s, z.s, acc);
  else f64_row_staple<false, false>(a, mu, i, x.s, w, y.s, z.s, acc);
  const double unit = R::fixed ? c_naik * ldexp(1.0, 4 * FX_LOW - 3 * FX_BITS) : c_naik;
#pragma unroll
  for (int j = 0; j < 3; ++j)
    o[j] = make_double2(unit * (double)acc.v[2 * j], unit * (double)acc.v[2 * j + 1]);
}

// Level 1: S_{+nu}, S_{-nu} and their sum A for the direction slot blockIdx.y.
template <typename R>
__global__ void __launch_bounds__(3 * FAT_SITES) staple1_kernel(const __grid_constant__ AsqtadArgs a) {
  if ((a.sc->uneven == 0) != R::fixed) return;
  SlabSite x;
  if (!slab_site(a.sl, x)) return;
  const int mu = a.mu, k = blockIdx.y, i = threadIdx.y, nu = other_dir(mu, k);
  const long n = a.sl.n;
  const int4 *w = a.u + (size_t)(9 * mu) * n;
  R sum[2];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    sum[b] = R{};
    row_staple(a, x, nu, b ? -1 : 1, i, w, sum[b]);
    int4 *dst = a.s + (size_t)((2 * k + b) * 9 + 3 * i) * n + x.s;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if constexpr (R::fixed)  // 2^-57 -> 2^-55
        dst[(size_t)j * n] = fat_word(fat_shift(sum[b].v[2 * j], 2), fat_shift(sum[b].v[2 * j + 1], 2));
      else
        reinterpret_cast<double2 *>(dst)[(size_t)j * n] = make_double2(sum[b].v[2 * j], sum[b].v[2 * j + 1]);
    }
  }
  int4 *dst = a.sa + (size_t)(k * 9 + 3 * i) * n + x.s;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const auto re = sum[0].v[2 * j] + sum[1].v[2 * j], im = sum[0].v[2 * j + 1] + sum[1].v[2 * j + 1];
    if constexpr (R::fixed) dst[(size_t)j * n] = fat_word(fat_shift(re, 4), fat_shift(im, 4));  // -> 2^-53
    else reinterpret_cast<double2 *>(dst)[(size_t)j * n] = make_double2(re, im);
  }
}

// Level 2: W = X + c_L S_{+-sg} of the direction slot blockIdx.y.
template <typename R>
__global__ void __launch_bounds__(3 * FAT_SITES) staple2_kernel(const __grid_constant__ AsqtadArgs a) {
  if ((a.sc->uneven == 0) != R::fixed) return;
  SlabSite x;
  if (!slab_site(a.sl, x)) return;
  const int mu = a.mu, k = blockIdx.y, i = threadIdx.y;
  const long n = a.sl.n;
  const int ka = (k + 1) % 3, kb = (k + 2) % 3;  // slots of nu and rho
  R acc{};
#pragma unroll 1
  for (int b = 0; b < 2; ++b) {  // inner A_nu, outer rho, and the other way round
    const int4 *w = a.sa + (size_t)((b ? kb : ka) * 9) * n;
    const int nu = other_dir(mu, b ? ka : kb);
    row_staple(a, x, nu, 1, i, w, acc);
    row_staple(a, x, nu, -1, i, w, acc);
  }
  const int4 *pu = a.u + (size_t)(9 * mu + 3 * i) * n + x.s;
  const int4 *pa = a.sa + (size_t)(ka * 9 + 3 * i) * n + x.s, *pb = a.sa + (size_t)(kb * 9 + 3 * i) * n + x.s;
  const size_t o = (size_t)(2 * k * 9 + 3 * i) * n + x.s;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int4 u = __ldg(pu + (size_t)j * n), v = __ldg(pa + (size_t)j * n), w = __ldg(pb + (size_t)j * n);
    const int4 sp = __ldg(a.s + o + (size_t)j * n), sm = __ldg(a.s + o + (size_t)(9 + j) * n);
    int4 *dp = a.w + o + (size_t)j * n, *dm = a.w + o + (size_t)(9 + j) * n;
    if constexpr (R::fixed) {
      const long long xr = fat_times(a.f3, fat_join(u.x, u.y)) +
                           fat_times(a.f5, fat_join(v.x, v.y) + fat_join(w.x, w.y)) +
                           fat_times(a.f7, fat_shift(acc.v[2 * j], 1));
      const long long xi = fat_times(a.f3, fat_join(u.z, u.w)) +
                           fat_times(a.f5, fat_join(v.z, v.w) + fat_join(w.z, w.w)) +
                           fat_times(a.f7, fat_shift(acc.v[2 * j + 1], 1));
      *dp = fat_word(fat_shift(xr + fat_times(a.fl, fat_join(sp.x, sp.y)), 5),
                     fat_shift(xi + fat_times(a.fl, fat_join(sp.z, sp.w)), 5));
      *dm = fat_word(fat_shift(xr + fat_times(a.fl, fat_join(sm.x, sm.y)), 5),
                     fat_shift(xi + fat_times(a.fl, fat_join(sm.z, sm.w)), 5));
    } else {
      auto re = [](int4 q) { return __hiloint2double(q.y, q.x); };
      auto im = [](int4 q) { return __hiloint2double(q.w, q.z); };
      const double xr = fma(a.c7, acc.v[2 * j], fma(a.c5, re(v) + re(w), a.c3 * re(u)));
      const double xi = fma(a.c7, acc.v[2 * j + 1], fma(a.c5, im(v) + im(w), a.c3 * im(u)));
      *reinterpret_cast<double2 *>(dp) = make_double2(fma(a.cl, re(sp), xr), fma(a.cl, im(sp), xi));
      *reinterpret_cast<double2 *>(dm) = make_double2(fma(a.cl, re(sm), xr), fma(a.cl, im(sm), xi));
    }
  }
}

// Level 3: the fat link.
template <typename R>
__global__ void __launch_bounds__(3 * FAT_SITES) staple3_kernel(const __grid_constant__ AsqtadArgs a,
                                                                const double2 *thin) {
  if ((a.sc->uneven == 0) != R::fixed) return;
  SlabSite x;
  if (!slab_site(a.sl, x)) return;
  const int mu = a.mu, i = threadIdx.y;
  R acc{};
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    const int4 *w = a.w + (size_t)(2 * k * 9) * a.sl.n;
    const int nu = other_dir(mu, k);
    row_staple(a, x, nu, 1, i, w, acc);
    row_staple(a, x, nu, -1, i, w + (size_t)9 * a.sl.n, acc);
  }
  const double2 *l = thin + (x.lex * 4 + mu) * 9 + 3 * i;
  double2 *o = a.fat + (x.lex * 4 + mu) * 9 + 3 * i;
  const double unit = R::fixed ? a.w_unit : 1.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double2 v = __ldg(l + j);
    o[j] = make_double2(fma(unit, (double)acc.v[2 * j], a.c1 * v.x),
                        fma(unit, (double)acc.v[2 * j + 1], a.c1 * v.y));
  }
}

// c = (h, l) 2^(ec - FX_BITS), |c| < 2^ec; `unit` the exponent of the field's
// unit: fat_times' product is in 2^(ec + unit + 2 FX_LOW - FX_BITS - 4), X in
// 2^(E - 60).
FatCoef fat_coef(double c, int unit, int E) {
  FatCoef f{0, 0, 0};
  if (c == 0.0) return f;
  const int ec = std::ilogb(c) + 1;
  const long long q = std::llrint(std::ldexp(c, FX_BITS - ec));
  const long long h = (q + (1ll << (FX_LOW - 1))) >> FX_LOW;
  const int down = E - 60 - (ec + unit + 2 * FX_LOW - FX_BITS - 4);
  if (down > 62) return f;  // below X's last bit
  f.h = (int)h;
  f.l = (int)(q - (h << FX_LOW));
  f.down = down;
  return f;
}

struct AsqtadCoeffs {
  double one, three, five, seven, lepage, naik;
};

int launch_fatten(const int dims[4], long vol, const double *thin, double c1, double c3, double w,
                  double *fat, double *lng, cudaStream_t st) {
  FatGeom g;
  for (int mu = 0; mu < 4; ++mu) g.L[mu] = dims[mu];
  g.st[0] = 1;
  g.st[1] = dims[0];
  g.st[2] = (long)dims[0] * dims[1];
  g.st[3] = (long)dims[0] * dims[1] * dims[2];
  g.vol = vol;
  const long n = 4 * vol;
  fatten_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(
      g, reinterpret_cast<const double2 *>(thin), c1, c3, w, reinterpret_cast<double2 *>(fat),
      reinterpret_cast<double2 *>(lng));
  SQ_CUDA_TRY(cudaGetLastError());
  return SQ_OK;
}

FatGeom make_fat_geom(const int dims[4], long vol) {
  FatGeom g;
  for (int mu = 0; mu < 4; ++mu) g.L[mu] = dims[mu];
  g.st[0] = 1;
  g.st[1] = dims[0];
  g.st[2] = (long)dims[0] * dims[1];
  g.st[3] = (long)dims[0] * dims[1] * dims[2];
  g.vol = vol;
  return g;
}

}  // namespace

int check_lattice_dims(const int dims[4], long *vol) {
  long v = 1;
  for (int mu = 0; mu < 4; ++mu) {
    if (dims[mu] < 2 || (dims[mu] & 1)) return SQ_ERR_ARG;
    v *= dims[mu];
    if (v > (1L << 30)) return SQ_ERR_ARG;
  }
  *vol = v;
  return SQ_OK;
}

}  // namespace sq

using namespace sq;

extern "C" int gauge_fatten_asqtad(sq_ctx *ctx, const int dims[4], const double *thin_dev,
                                   const double coeffs[6], double *fat_dev, double *lng_dev,
                                   void *stream) {
  if (!ctx || !dims || !thin_dev || !coeffs || !fat_dev || !lng_dev) return SQ_ERR_ARG;
  for (int k = 0; k < 6; ++k)
    if (!std::isfinite(coeffs[k])) return SQ_ERR_ARG;
  long vol;
  int rc = check_lattice_dims(dims, &vol);
  if (rc) return rc;
  cudaSetDevice(ctx->device);
  cudaStream_t st = stream ? (cudaStream_t)stream : cudaStreamLegacy;  // NULL: default stream
  const AsqtadCoeffs k{coeffs[0], coeffs[1], coeffs[2], coeffs[3], coeffs[4], coeffs[5]};
  const double2 *u = reinterpret_cast<const double2 *>(thin_dev);
  AsqtadArgs a{};
  a.sl.g = make_fat_geom(dims, vol);
  auto slices = [&](int ax) {
    a.sl.ax = ax;
    a.sl.v3 = vol / dims[ax];
    long s = 1;
    for (int k = 0, j = 0; k < 4; ++k)
      if (k != ax) {
        a.sl.od[j++] = k;
        a.sl.st[k] = s;
        s *= dims[k];
      }
  };
  a.fat = reinterpret_cast<double2 *>(fat_dev);
  a.c1 = k.one;
  a.c3 = k.three;
  a.c5 = k.five;
  a.c7 = k.seven;
  a.cl = k.lepage;
  // X + c_L S is below 2^E (see above); kept in range for extreme coefficients
  const double most = 1.03 * (std::abs(k.three) + 4 * std::abs(k.five) + 8 * std::abs(k.seven) +
                              std::abs(k.lepage));
  const bool extreme = !(most < 1e270) || (most > 0 && most < 1e-270);  // FP64 then
  const int E = most > 0 && !extreme ? std::ilogb(most) + 1 : 0;
  a.f3 = fat_coef(k.three, -FX_BITS, E);
  a.f5 = fat_coef(k.five, 2 - FX_BITS, E);
  a.f7 = fat_coef(k.seven, 1 - FX_BITS, E);
  a.fl = fat_coef(k.lepage, -FX_BITS, E);
  a.w_unit = std::ldexp(1.0, E - FX_BITS - 2);
  // Scratch of a site: 36 link planes, 6 S, 3 A and 6 W fields of 9 planes, 16
  // bytes each.  The whole lattice at once where that is within what is left of
  // the context's budget and can be had; else slabs of nt slices across the
  // longest direction, with the slices their staples reach: links to 3, S and A
  // to 2, W to 1 slices beyond (the Naik link reaches 2).  The smallest slab, of
  // one slice and 7 slots, is taken whatever is left, and lattices with no
  // direction longer than 7 (1296 sites at most) are done whole.
  const size_t site_b = 16 * (36 + 54 + 27 + 54), head = 256;
  size_t left;
  {
    std::lock_guard<std::mutex> lk(ctx->mu);
    left = ctx->budget > ctx->in_use ? ctx->budget - ctx->in_use : 0;
  }
  int longest = 3;
  for (int k = 2; k >= 0; --k)
    if (dims[k] > dims[longest]) longest = k;
  bool whole = dims[longest] <= 7 || head + site_b * vol <= left;
  void *scratch = nullptr;
  int nt = 0;
  for (;;) {
    slices(whole ? 3 : longest);
    const size_t slice_b = site_b * a.sl.v3;
    if (whole) nt = dims[3];
    else if (nt == 0) nt = (int)std::min<size_t>(std::max<size_t>(left / slice_b, 7) - 6, dims[longest] - 7);
    a.sl.nslots = whole ? nt : nt + 6;
    const cudaError_t me = cudaMallocAsync(&scratch, head + slice_b * a.sl.nslots, st);
    if (me == cudaSuccess) break;
    if (me != cudaErrorMemoryAllocation) SQ_CUDA_TRY(me);
    cudaGetLastError();
    nt = whole ? 0 : nt / 2;
    if ((whole && dims[longest] <= 7) || (!whole && nt < 1)) SQ_CUDA_TRY(me);
    whole = false;
  }
  a.sl.n = a.sl.nslots * a.sl.v3;
  FatScale *sc = static_cast<FatScale *>(scratch);
  a.sc = sc;
  int4 *planes = reinterpret_cast<int4 *>(static_cast<char *>(scratch) + head);
  a.u = planes;
  a.s = planes + (size_t)36 * a.sl.n;
  a.sa = planes + (size_t)90 * a.sl.n;
  a.w = planes + (size_t)117 * a.sl.n;
  cudaError_t e = cudaMemsetAsync(sc, extreme ? 0xff : 0, sizeof(FatScale), st);
  if (e == cudaSuccess) {
    fat_scale_kernel<<<8 * ctx->sms, 256, 0, st>>>(u, 4 * vol, sc);
    ctx->launches++;
  }
  const int Lt = dims[a.sl.ax];
  for (int t = 0; t < Lt && e == cudaSuccess; t += nt) {
    const int m = std::min(nt, Lt - t);       // slices finished by this slab
    const int halo = whole ? 0 : 3;
    a.sl.t0 = (t - halo + Lt) % Lt;
    auto range = [&](int reach, int sites = FAT_SITES) {  // slots of the slab and `reach` beyond
      a.sl.first = whole ? 0 : halo - reach;
      a.sl.count = whole ? Lt : m + 2 * reach;
      return (unsigned)((a.sl.count * a.sl.v3 + sites - 1) / sites);
    };
    const dim3 blk(FAT_SITES, 3);
    fat_links_kernel<<<dim3(range(3, 128), 4), 128, 0, st>>>(a, u, planes);
    const dim3 gn(range(0), 4);
    double2 *lng = reinterpret_cast<double2 *>(lng_dev);
    naik_kernel<Row><<<gn, blk, 0, st>>>(a, k.naik, lng);
    naik_kernel<RowF><<<gn, blk, 0, st>>>(a, k.naik, lng);
    ctx->launches += 3;
    for (a.mu = 0; a.mu < 4; ++a.mu) {
      const dim3 g1(range(2), 3);
      staple1_kernel<Row><<<g1, blk, 0, st>>>(a);
      staple1_kernel<RowF><<<g1, blk, 0, st>>>(a);
      const dim3 g2(range(1), 3);
      staple2_kernel<Row><<<g2, blk, 0, st>>>(a);
      staple2_kernel<RowF><<<g2, blk, 0, st>>>(a);
      const unsigned g3 = range(0);
      staple3_kernel<Row><<<g3, blk, 0, st>>>(a, u);
      staple3_kernel<RowF><<<g3, blk, 0, st>>>(a, u);
      ctx->launches += 6;
    }
    e = cudaGetLastError();
  }
  cudaFreeAsync(scratch, st);
  if (e != cudaSuccess) {
    set_last_cuda_error(e, "asqtad staple kernels", __FILE__, __LINE__);
    return SQ_ERR_CUDA;
  }
  return SQ_OK;
}

extern "C" int gauge_fatten(sq_ctx *ctx, const int dims[4], const double *thin_dev, double c1,
                            double c3, double staple_weight, double *fat_dev, double *lng_dev,
                            void *stream) {
  if (!ctx || !dims || !thin_dev || !fat_dev || !lng_dev) return SQ_ERR_ARG;
  if (!std::isfinite(c1) || !std::isfinite(c3) || !std::isfinite(staple_weight) ||
      1.0 + 6.0 * staple_weight == 0.0)
    return SQ_ERR_ARG;
  long vol;
  int rc = check_lattice_dims(dims, &vol);
  if (rc) return rc;
  cudaSetDevice(ctx->device);
  cudaStream_t st = stream ? (cudaStream_t)stream : cudaStreamLegacy;  // NULL: default stream
  rc = launch_fatten(dims, vol, thin_dev, c1, c3, staple_weight, fat_dev, lng_dev, st);
  if (rc == SQ_OK) ctx->launches++;
  return rc;
}

extern "C" int gauge_load_thin(sq_ctx *ctx, const int dims[4], const double *thin, double c1,
                               double c3, double staple_weight, unsigned flags, int *gauge_id) {
  if (!ctx || !dims || !thin || !gauge_id) return SQ_ERR_ARG;
  long vol;
  int rc = check_lattice_dims(dims, &vol);
  if (rc) return rc;
  const size_t nbytes = (size_t)vol * 4 * 9 * 16;
  cudaSetDevice(ctx->device);
  cudaStream_t st = ctx->stream;
  // staging of thin, fat and long links, freed before return: outside the budget
  void *buf = nullptr;
  cudaError_t e = cudaMalloc(&buf, 3 * nbytes);
  if (e != cudaSuccess) {
    set_last_cuda_error(e, "cudaMalloc(link staging)", __FILE__, __LINE__);
    return SQ_ERR_OOM;
  }
  double *du = static_cast<double *>(buf);
  double *df = du + (size_t)vol * 72, *dl = df + (size_t)vol * 72;
  const double *src = thin;
  if (!(flags & SQ_GAUGE_DEVICE_PTRS)) {
    for (size_t k = 0; k < (size_t)vol * 72; ++k)
      if (!std::isfinite(thin[k])) {
        cudaFree(buf);
        return SQ_ERR_NONFINITE;
      }
    e = cudaMemcpyAsync(du, thin, nbytes, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) {
      cudaFree(buf);
      set_last_cuda_error(e, "cudaMemcpyAsync(thin links)", __FILE__, __LINE__);
      return SQ_ERR_CUDA;
    }
    src = du;
  }
  rc = gauge_fatten(ctx, dims, src, c1, c3, staple_weight, df, dl, st);
  if (rc == SQ_OK) {
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
      set_last_cuda_error(e, "gauge_fatten", __FILE__, __LINE__);
      rc = SQ_ERR_CUDA;
    }
  }
  if (rc == SQ_OK) rc = gauge_load(ctx, dims, df, dl, flags | SQ_GAUGE_DEVICE_PTRS, gauge_id);
  cudaFree(buf);
  return rc;
}
