// The one-colour four-fermion operator of the NPR code in Sec. 2 (Eq. 1,
// Fig. 2, Table 3), in FP64 on the GPU.
//
// For every hypercube z of the lattice (corner sites z_A = 2z + A, A in
// {0,1}^4, A = A_x + 2 A_y + 4 A_z + 8 A_t) and every operator
// (S1, F1, S2, F2):
//   O[a1][a2][a3][a4](z) = sum_{A,C} M1[A][B] M2[C][D]
//       (G1(z_A)^dag U_AD G4(z_D))[a1][a4] (G3(z_C)^dag U_CB G2(z_B))[a3][a2]
// with B = A ^ S1 ^ F1 and D = C ^ S2 ^ F2: the hypercube spin-taste matrix
// (gamma_S x xi_F)_{AB} = Tr(gamma_A^dag gamma_S gamma_B gamma_F^dag) / 4 has
// one entry, +1 or -1, per row, at B = A ^ S ^ F (spin_taste_sign below).
// U_AD(z) is the mean of the link products over the shortest paths from z_A
// to z_D.  The propagators G^f are [site][colour][source colour]; flavours 1
// and 3 enter conjugated, as the antiquark fields of Eq. 1.
//
// One CTA works on one hypercube at a time (persistent grid), in shared
// memory:
//   1. the 16 corners' propagators and the 32 links inside the hypercube
//      arrive by cp.async, prefetched while the previous hypercube's
//      contraction runs;
//   2. U_AD for A < D, level by level in the distance n = |A ^ D|, from
//      U_AD = (1/n) sum_{mu in A ^ D} U_{A, A^mu} U_{A^mu, D}: a shortest
//      path starts with any of the n differing directions, each first in
//      (n-1)! of the n! paths.  U_DA = U_AD^dag is read, not stored;
//   3. P[A][D] = G1(A)^dag U_AD G4(D) and Q[C][B] = G3(C)^dag U_CB G2(B) for
//      all 256 corner pairs, shared by every operator;
//   4. per operator and output, the 256-term sum over (A, C) of
//      +-P[A][C ^ t2][a1][a4] Q[C][A ^ t1][a3][a2], t = S ^ F.
// The arithmetic (about 1.6 MFLOP per hypercube for 8 operators, against
// 14 KB of input) runs on the integer multiply-add units in the two-word
// fixed-point form of sq_fixed.cuh, 54 bits relative to block scales: one per
// hypercube for the links, for each flavour's propagators, for P and for Q
// (npr_kernel).  A hypercube whose inputs or averaged links do not fit that
// form (infinities, NaN, elements near the ends of FP64, links far from
// unitary) is marked there and computed by npr_fp64_kernel in FP64.
// Per-hypercube results are written when asked for; the sums over hypercubes
// go through per-CTA partials and a fixed-order second pass, so they do not
// depend on scheduling.
#include <cmath>
#include <cstdint>

#include "sq_fixed.cuh"
#include "sq_host.h"

namespace sq {
namespace {

int spin_taste_sign(int s, int f, int a) {
  // gamma_X gamma_Y = sigma(X, Y) gamma_{X^Y}: each gamma_j of Y moves left
  // past the gamma_i of X with i > j.  gamma_X^dag = (-1)^(n(n-1)/2) gamma_X
  // for |X| = n.  With B = A ^ S ^ F,
  //   gamma_A^dag gamma_S gamma_B gamma_F^dag
  //     = r(A) r(F) sigma(A, S) sigma(A^S, B) sigma(F, F) * 1
  // and sigma(F, F) = r(F).
  auto sigma = [](int x, int y) {
    int n = 0;
    for (int i = 0; i < 4; ++i)
      if ((x >> i) & 1)
        for (int j = 0; j < i; ++j) n += (y >> j) & 1;
    return (n & 1) ? -1 : 1;
  };
  auto rev = [](int x) {
    const int n = __builtin_popcount(x);
    return ((n * (n - 1) / 2) & 1) ? -1 : 1;
  };
  const int b = a ^ s ^ f;
  return rev(a) * sigma(a, s) * sigma(a ^ s, b);
}

constexpr int kThreads = 512;    // npr_fp64_kernel
constexpr int kFxThreads = 288;  // npr_kernel
constexpr int kMaxOps = SQ_NPR_MAX_OPS;
constexpr int kItemsPerThread = (kMaxOps * 81 + kThreads - 1) / kThreads;
constexpr int kTri = 136;                  // corner pairs A <= D
constexpr int kLoadChunks = 4 * 16 * 9 + 32 * 9;
constexpr size_t kSmemBytes =
    sizeof(double2) * (kTri * 9 + 4 * 16 * 9 + 2 * 256 * 9) + sizeof(double) * 2 * 256 * 9;

struct NprOp {
  uint16_t neg1, neg2;  // bit A (C): the entry of row A (C) is -1
  uint8_t t1, t2;       // S1 ^ F1, S2 ^ F2
};

struct NprArgs {
  const double2 *links;    // [site][mu][3][3]
  const double2 *prop[4];  // [site][3][3]
  double2 *out_hc;         // this group's first op of [hypercube][op][81], or null
  long hc_stride;          // elements per hypercube of out_hc (all ops x 81)
  double2 *partial;        // [cta][op][81]
  unsigned char *marked;   // [hypercube]: left to npr_fp64_kernel
  int *any_marked;         // set when one is
  int H[4];                // hypercubes per direction
  long st[4];              // site strides
  int nhc;
  int nops;
  NprOp ops[kMaxOps];
};

__device__ __forceinline__ int tri(int a, int d) {  // a <= d
  return 16 * a - (a * (a - 1)) / 2 + (d - a);
}

__device__ __forceinline__ double flip(double v, unsigned neg) {
  return __longlong_as_double(__double_as_longlong(v) ^ ((unsigned long long)neg << 63));
}

// element (i, j) of U_XY for any corners X, Y
__device__ __forceinline__ double2 u_elem(const double2 *ut, int x, int y, int i, int j) {
  const bool sw = x > y;
  const int lo = sw ? y : x, hi = sw ? x : y;
  const double2 v = ut[tri(lo, hi) * 9 + (sw ? 3 * j + i : 3 * i + j)];
  return make_double2(v.x, flip(v.y, sw));
}

__device__ __forceinline__ void cmac(double2 &c, double2 a, double2 b) {
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(-a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(a.y, b.x, c.y);
}

__device__ __forceinline__ void cmac_conj(double2 &c, double2 a, double2 b) {  // conj(a) b
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(-a.y, b.x, c.y);
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

// Step 1: propagators of the 16 corners and links inside hypercube h.
template <int THREADS>
__device__ void issue_loads(const NprArgs &a, int h, double2 *gs, double2 *ut) {
  int r = h;
  long s0 = 0;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    s0 += 2L * (r % a.H[mu]) * a.st[mu];
    r /= a.H[mu];
  }
  for (int i = threadIdx.x; i < kLoadChunks; i += THREADS) {
    const double2 *src;
    double2 *dst;
    if (i < 4 * 16 * 9) {
      const int f = i / 144, c = (i / 9) % 16, e = i % 9;
      const long site = s0 + (c & 1) * a.st[0] + ((c >> 1) & 1) * a.st[1] +
                        ((c >> 2) & 1) * a.st[2] + (c >> 3) * a.st[3];
      src = a.prop[f] + site * 9 + e;
      dst = gs + (f * 16 + c) * 9 + e;
    } else {
      const int j = i - 4 * 16 * 9;
      const int mu = j / 72, k = (j / 9) % 8, e = j % 9;
      const int c = ((k >> mu) << (mu + 1)) | (k & ((1 << mu) - 1));  // corner with bit mu = 0
      const long site = s0 + (c & 1) * a.st[0] + ((c >> 1) & 1) * a.st[1] +
                        ((c >> 2) & 1) * a.st[2] + (c >> 3) * a.st[3];
      src = a.links + (site * 4 + mu) * 9 + e;
      dst = ut + tri(c, c | (1 << mu)) * 9 + e;
    }
    cp_async16(dst, src);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// Step 2, distance n: U_AD for the 8 C(4, n) pairs A < D with |A ^ D| = n.
__device__ void path_level(double2 *ut, int n) {
  const int npairs = n == 2 ? 48 : (n == 3 ? 32 : 8);
  const double inv = n == 2 ? 0.5 : (n == 3 ? 1.0 / 3.0 : 0.25);
  for (int it = threadIdx.x; it < npairs * 9; it += kThreads) {
    const int k = it / 9, e = it % 9, i = e / 3, j = e % 3;
    int x = 0;  // the (k/8)-th difference mask with n bits
    for (int m = 1, seen = 0; m < 16; ++m)
      if (__popc(m) == n && seen++ == (k >> 3)) {
        x = m;
        break;
      }
    const int top = 31 - __clz(x);
    const int lo = k & 7;
    const int A = ((lo >> top) << (top + 1)) | (lo & ((1 << top) - 1));  // bit top = 0
    const int D = A ^ x;
    double2 s = make_double2(0.0, 0.0);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      if (!((x >> mu) & 1)) continue;
      const int m = A ^ (1 << mu);
#pragma unroll
      for (int kk = 0; kk < 3; ++kk) cmac(s, u_elem(ut, A, m, i, kk), u_elem(ut, m, D, kk, j));
    }
    ut[tri(A, D) * 9 + e] = make_double2(s.x * inv, s.y * inv);
  }
}

// Step 3: P[X][Y] = G1(X)^dag U_XY G4(Y) and Q[X][Y] = G3(X)^dag U_XY G2(Y),
// one column of one pair per item.
__device__ void sandwiches(const double2 *ut, const double2 *gs, double2 *ps, double2 *qs,
                           double *pss, double *qss) {
  for (int it = threadIdx.x; it < 2 * 256 * 3; it += kThreads) {
    const int which = it >= 768;
    const int rem = it - which * 768;
    const int pair = rem / 3, col = rem % 3;
    const int x = pair >> 4, y = pair & 15;
    const double2 *gl = gs + ((which ? 2 : 0) * 16 + x) * 9;
    const double2 *gr = gs + ((which ? 1 : 3) * 16 + y) * 9;
    double2 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      h[c] = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < 3; ++k) cmac(h[c], u_elem(ut, x, y, c, k), gr[3 * k + col]);
    }
    double2 *dst = (which ? qs : ps) + pair * 9;
    double *dsum = (which ? qss : pss) + pair * 9;
#pragma unroll
    for (int a1 = 0; a1 < 3; ++a1) {
      double2 v = make_double2(0.0, 0.0);
#pragma unroll
      for (int c = 0; c < 3; ++c) cmac_conj(v, gl[3 * c + a1], h[c]);
      dst[3 * a1 + col] = v;
      dsum[3 * a1 + col] = v.x + v.y;
    }
  }
}

// Step 4: output o = 27 a1 + 9 a2 + 3 a3 + a4 of one operator.  The complex
// products go by the 3M method (Higham, "Stability of a method for
// multiplying complex matrices with three real matrix multiplications",
// SIMAX 1992): with re + im of P and Q stored beside them,
//   sum p q = (T1 - T2) + i (T3 - T1 - T2),
//   T1 = sum p.re q.re,  T2 = sum p.im q.im,  T3 = sum (p.re + p.im)(q.re + q.im),
// three real multiply-adds per term instead of four.
__device__ __forceinline__ double2 contract(const double2 *ps, const double2 *qs,
                                            const double *pss, const double *qss, NprOp op,
                                            int o) {
  const int a1 = o / 27, a2 = (o / 9) % 3, a3 = (o / 3) % 3, a4 = o % 3;
  const int pe = 3 * a1 + a4, qe = 3 * a3 + a2;
  double t1[4], t2[4], t3[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) t1[k] = t2[k] = t3[k] = 0.0;
#pragma unroll 2
  for (int A = 0; A < 16; ++A) {
    const int qo = (A ^ op.t1) * 9 + qe;  // Q[C][A ^ t1] at qo + C * 16 * 9
    const int po = A * 16 * 9 + pe;       // P[A][D] at po + D * 9
    const unsigned sa = (op.neg1 >> A) & 1;
#pragma unroll
    for (int C = 0; C < 16; ++C) {
      const int pi = po + (C ^ op.t2) * 9, qi = qo + C * 16 * 9;
      const double2 p = ps[pi], q = qs[qi];
      const double sp = pss[pi], sq = qss[qi];
      const unsigned neg = sa ^ ((op.neg2 >> C) & 1);
      t1[C & 3] = fma(flip(p.x, neg), q.x, t1[C & 3]);
      t2[C & 3] = fma(flip(p.y, neg), q.y, t2[C & 3]);
      t3[C & 3] = fma(flip(sp, neg), sq, t3[C & 3]);
    }
  }
  const double T1 = (t1[0] + t1[1]) + (t1[2] + t1[3]);
  const double T2 = (t2[0] + t2[1]) + (t2[2] + t2[3]);
  const double T3 = (t3[0] + t3[1]) + (t3[2] + t3[3]);
  return make_double2(T1 - T2, (T3 - T1) - T2);
}

// ------------------------------------------------------------- FP64 kernel
// The hypercubes npr_kernel marked, added to its partials.
__global__ void __launch_bounds__(kThreads, 1) npr_fp64_kernel(const NprArgs a) {
  if (*a.any_marked == 0) return;
  extern __shared__ double2 smem[];
  double2 *ut = smem;              // [pair A <= D][3][3]
  double2 *gs = ut + kTri * 9;     // [flavour][corner][3][3]
  double2 *ps = gs + 4 * 16 * 9;   // [A][D][a1][a4]
  double2 *qs = ps + 256 * 9;      // [C][B][a3][a2]
  double *pss = reinterpret_cast<double *>(qs + 256 * 9);  // re + im of ps
  double *qss = pss + 256 * 9;                             // re + im of qs
  const int tid = threadIdx.x;
  for (int i = tid; i < 16 * 9; i += kThreads) {
    const int c = i / 9, e = i % 9;
    ut[tri(c, c) * 9 + e] = make_double2(e % 4 == 0 ? 1.0 : 0.0, 0.0);
  }
  const int nitems = a.nops * 81;
  double2 tot[kItemsPerThread];
#pragma unroll
  for (int r = 0; r < kItemsPerThread; ++r) tot[r] = make_double2(0.0, 0.0);
  bool any = false;
  for (int h = blockIdx.x; h < a.nhc; h += gridDim.x) {
    if (!a.marked[h]) continue;  // the same in every thread
    any = true;
    __syncthreads();
    issue_loads<kThreads>(a, h, gs, ut);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    for (int n = 2; n <= 4; ++n) {
      path_level(ut, n);
      __syncthreads();
    }
    sandwiches(ut, gs, ps, qs, pss, qss);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kItemsPerThread; ++r) {
      const int it = tid + r * kThreads;
      if (it < nitems) {
        const double2 v = contract(ps, qs, pss, qss, a.ops[it / 81], it % 81);
        if (a.out_hc) a.out_hc[(long)h * a.hc_stride + it] = v;
        tot[r].x += v.x;
        tot[r].y += v.y;
      }
    }
  }
  if (!any) return;
#pragma unroll
  for (int r = 0; r < kItemsPerThread; ++r) {
    const int it = tid + r * kThreads;
    if (it < nitems) {
      double2 *p = a.partial + (long)blockIdx.x * nitems + it;
      *p = make_double2(p->x + tot[r].x, p->y + tot[r].y);
    }
  }
}

// ------------------------------------------------------ fixed-point kernel
// Elements in shared memory are int4 (re.l, re.h, im.l, im.h) with balanced
// low words of 27 bits.  Bits at a block's scale: 55 for the propagators, 56
// for the links and their averages, 54 (53 with 2 slices) and 55 for P and Q,
// whose products are added 512 at a time: over a thread's slice
//   |hi| <= (512 / slices) 2^27 2^28 < 2^63,
//   |mid| <= (512 / slices) (2^27 2^26 + 2^26 2^28) < 2^63.
// The dropped products of two low words are below 2^-57 of the blocks' scales.
//
// The contraction takes most of the time.  A thread owns the outputs (a4, a2)
// of one (operator, a1, a3), 9 complex sums, over one slice of A: two groups
// of 3 elements are loaded for 9 complex terms of 12 multiply-adds each, so
// the shared-memory reads stay below the multiply-add time.  The slices (2 to
// 16, as many as fill 288 threads for the number of operators) are added by
// shuffles; integer sums do not depend on the order.  Two CTAs of 9 warps per
// SM (96 registers, a few spilled) and one of 164 registers measured the same.
//
// 8 operators at 20^3 x 64: 37.2 ms with FP64 FMAs (their pipe 93 % busy),
// 15.6 ms here, the multiply-add pipe 61 % busy (mad.wide.s32 issues 32 lanes
// per clock and SM).  Error of a hypercube against long double 2.0e-16 to
// 2.3e-16, with FP64 FMAs (three per complex term) 4.6e-16.
struct FxC { Fx re, im; };
struct Wide { long long hr, mr, hi, mi; };

__device__ __forceinline__ FxC fx_load(const int4 *p) {
  const int4 q = *p;
  return {{q.y, q.x}, {q.w, q.z}};
}

__device__ __forceinline__ Fx fx_neg(Fx a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Fx fx_flip(Fx a, int s) { return {(a.h ^ s) - s, (a.l ^ s) - s}; }  // s: 0, -1

__device__ __forceinline__ void wide_mac(Wide &w, FxC a, FxC b) {
  const Fx nb = fx_neg(b.im);
  fx_mac(w.hr, w.mr, a.re, b.re);
  fx_mac(w.hi, w.mi, a.re, b.im);
  fx_mac(w.hr, w.mr, a.im, nb);
  fx_mac(w.hi, w.mi, a.im, b.re);
}

// A value as a balanced two-word number.
__device__ __forceinline__ Fx fx_split(long long v) {
  const long long h = (v + (1ll << (FX_LOW - 1))) >> FX_LOW;
  return {(int)h, (int)(v - (h << FX_LOW))};
}
__device__ __forceinline__ int4 fx_word(long long re, long long im) {
  const Fx r = fx_split(re), i = fx_split(im);
  return make_int4(r.l, r.h, i.l, i.h);
}
// hi 2^27 + mid, less its last FX_LOW - UP bits
template <int UP>
__device__ __forceinline__ long long wide_round(long long hi, long long mid) {
  constexpr int d = FX_LOW - UP;
  return (hi << UP) + ((mid + (1ll << (d - 1))) >> d);
}
__device__ __forceinline__ long long abs64(long long v) { return v < 0 ? -v : v; }

// element (i, j) of U_XY for any corners X, Y
__device__ __forceinline__ FxC fx_u(const int4 *ut, int x, int y, int i, int j) {
  const bool sw = x > y;
  const int lo = sw ? y : x, hi = sw ? x : y;
  FxC u = fx_load(ut + tri(lo, hi) * 9 + (sw ? 3 * j + i : 3 * i + j));
  u.im = fx_flip(u.im, sw ? -1 : 0);
  return u;
}

constexpr int kFxRow = 16 * 9 + 2;      // padded row of P: slices of A fall on different banks
constexpr int kFxP = 16 * kFxRow, kFxQ = 256 * 9;
constexpr size_t kFxSmem = sizeof(int4) * (kTri * 9 + 4 * 16 * 9 + kFxP + kFxQ);
constexpr long long kFxMost = 1ll << (FX_LOW + 30);  // two words hold values below this
constexpr int kPropBits = FX_BITS, kLinkBits = 56;   // bits at the blocks' scales
constexpr int kMidBits = 55;                         // ... of U G4 and U G2
template <int SLICES> struct PQBits { static constexpr int p = SLICES >= 4 ? 54 : 53, q = 55; };

struct FxShared {
  int e[5];                    // largest biased exponents: 4 flavours, links
  int bad;                     // the hypercube does not fit
  unsigned long long most[2];  // largest |v| of P and Q before scaling
};

__device__ __forceinline__ int fx_biased(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v 2^(FX_BITS - e) for a largest biased exponent e + 1022
__device__ __forceinline__ long long fx_scaled(double v, int biased_top) {
  const Fx a = fx_from_double(v, biased_top, 1);
  return ((long long)a.h << FX_LOW) + a.l;
}

template <int SLICES>
__device__ __forceinline__ void fx_contract(const int4 *ps, const int4 *qs, NprOp op, int a1, int a3,
                                            int slice, Wide (&w)[9]) {
#pragma unroll 1
  for (int A = slice; A < 16; A += SLICES) {
    const int4 *pa = ps + A * kFxRow + 3 * a1;
    const int4 *qa = qs + (A ^ op.t1) * 9 + 3 * a3;
    const unsigned sa = ((op.neg1 >> A) & 1) ? 0xffffu : 0u;
    const unsigned neg = op.neg2 ^ sa;
#pragma unroll 1
    for (int C = 0; C < 16; ++C) {
      const int s = -(int)((neg >> C) & 1);
      FxC p[3], q[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        p[k] = fx_load(pa + (C ^ op.t2) * 9 + k);
        q[k] = fx_load(qa + C * 144 + k);
        q[k].re = fx_flip(q[k].re, s);
        q[k].im = fx_flip(q[k].im, s);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int m = 0; m < 3; ++m) wide_mac(w[3 * k + m], p[k], q[m]);
    }
  }
}

template <int SLICES>
__global__ void __launch_bounds__(kFxThreads, 2) npr_kernel(const __grid_constant__ NprArgs a) {
  extern __shared__ int4 fsm[];
  __shared__ FxShared sh;
  int4 *ut = fsm;              // [pair A <= D][3][3]
  int4 *gs = ut + kTri * 9;    // [flavour][corner][3][3]
  int4 *ps = gs + 4 * 16 * 9;  // [A][D][a1][a4], rows of kFxRow
  int4 *qs = ps + kFxP;        // [C][B][a3][a2]
  const int tid = threadIdx.x;
  const int slice = tid % SLICES, tile = (tid / SLICES) % 9, iop = tid / (9 * SLICES);
  const bool mine = iop < a.nops;
  const NprOp op = a.ops[mine ? iop : 0];
  const int a1 = tile / 3, a3 = tile % 3;
  constexpr int kOwn = (9 + SLICES - 1) / SLICES;  // outputs a thread finishes
  double2 tot[kOwn];
#pragma unroll
  for (int r = 0; r < kOwn; ++r) tot[r] = make_double2(0.0, 0.0);
  if (tid == 0) {
    for (int k = 0; k < 5; ++k) sh.e[k] = 0;
    sh.bad = 0;
    sh.most[0] = sh.most[1] = 0;
  }
  int h = blockIdx.x;
  if (h < a.nhc)
    issue_loads<kFxThreads>(a, h, reinterpret_cast<double2 *>(gs), reinterpret_cast<double2 *>(ut));
  for (; h < a.nhc; h += gridDim.x) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    // block scales of the inputs: 864 elements, 3 per thread, 2 of the
    // propagators' and 1 of the links' (a warp's 32 span two flavours at most)
    int4 *own[3];
    double2 raw[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int i = tid + k * kFxThreads;
      if (k < 2) {
        own[k] = gs + i;
      } else {
        const int j = tid, mu = j / 72, m = (j / 9) % 8, e = j % 9;
        const int c = ((m >> mu) << (mu + 1)) | (m & ((1 << mu) - 1));
        own[k] = ut + tri(c, c | (1 << mu)) * 9 + e;
      }
      raw[k] = *reinterpret_cast<const double2 *>(own[k]);
      const int b = max(fx_biased(raw[k].x), fx_biased(raw[k].y));
      const int f = k < 2 ? i / 144 : 4;
      const int f0 = __shfl_sync(0xffffffffu, f, 0), f1 = __shfl_sync(0xffffffffu, f, 31);
      const int b0 = __reduce_max_sync(0xffffffffu, f == f0 ? b : 0);
      const int b1 = __reduce_max_sync(0xffffffffu, f == f1 ? b : 0);
      if ((tid & 31) == 0) {
        atomicMax(&sh.e[f0], b0);
        if (f1 != f0) atomicMax(&sh.e[f1], b1);
      }
    }
    __syncthreads();
    int e[5];
    bool fits = true;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      e[k] = sh.e[k];
      if (e[k] == 0) e[k] = 1022;  // all zero (or denormal: see below)
      else fits &= k == 4 ? (e[k] >= 1022 - 1 && e[k] <= 1022 + 2) : (e[k] >= 1022 - 200 && e[k] <= 1022 + 200);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int i = tid + k * kFxThreads;
      const int top = k < 2 ? e[i / 144] : e[4];
      const int up = k < 2 ? 0 : kLinkBits - FX_BITS;
      *own[k] = fx_word(fx_scaled(raw[k].x, top) << up, fx_scaled(raw[k].y, top) << up);
      if (fx_biased(raw[k].x) == 0) fits &= raw[k].x == 0.0;  // no denormals
      if (fx_biased(raw[k].y) == 0) fits &= raw[k].y == 0.0;
    }
    const int eu = e[4] - 1022;  // |link element| < 2^eu
    const int one = min(kLinkBits - eu, kLinkBits + 1);  // U_AA = 1 in the links' units
    if (tid < 144) {
      const int c = tid / 9, el = tid % 9;
      ut[tri(c, c) * 9 + el] = fx_word(el % 4 == 0 ? 1ll << one : 0ll, 0);
    }
    if (!fits) sh.bad = 1;
    __syncthreads();
#pragma unroll 1
    for (int n = 2; n <= 4; ++n) {  // distance n: U_AD for the 8 C(4, n) pairs A < D
      const int npairs = n == 2 ? 48 : (n == 3 ? 32 : 8);
      for (int it = tid; it < npairs * 9; it += kFxThreads) {
        const int k = it / 9, el = it % 9, i = el / 3, j = el % 3;
        int x = 0;  // the (k/8)-th difference mask with n bits
        for (int m = 1, seen = 0; m < 16; ++m)
          if (__popc(m) == n && seen++ == (k >> 3)) {
            x = m;
            break;
          }
        const int top = 31 - __clz(x);
        const int lo = k & 7;
        const int A = ((lo >> top) << (top + 1)) | (lo & ((1 << top) - 1));  // bit top = 0
        const int D = A ^ x;
        Wide w = {0, 0, 0, 0};
#pragma unroll 1
        for (int mu = 0; mu < 4; ++mu) {
          if (!((x >> mu) & 1)) continue;
          const int m = A ^ (1 << mu);
#pragma unroll
          for (int kk = 0; kk < 3; ++kk) wide_mac(w, fx_u(ut, A, m, i, kk), fx_u(ut, m, D, kk, j));
        }
        // sums below 24 2^(2 (kLinkBits - FX_LOW)) in units of
        // 2^(2 (eu - kLinkBits) + 2 FX_LOW)
        long long re = wide_round<0>(w.hr, w.mr), im = wide_round<0>(w.hi, w.mi);
        if (n == 3) {
          re /= 3;
          im /= 3;
        }
        const int dn = kLinkBits - 2 * FX_LOW - eu + (n == 2 ? 1 : n == 4 ? 2 : 0);  // 0 to 5
        const long long half = dn > 0 ? 1ll << (dn - 1) : 0;
        re = (re + half) >> dn;
        im = (im + half) >> dn;
        // the elements' bound: 2^eu, as for unitary links
        if (max(abs64(re), abs64(im)) > 1ll << kLinkBits) sh.bad = 1;
        ut[tri(A, D) * 9 + el] = fx_word(re, im);
      }
      __syncthreads();
    }
    // sandwiches: one column of one pair per item, P then Q, as 64-bit values
    unsigned long long most[2] = {0, 0};
    bool big = false;
#pragma unroll 1
    for (int it = tid; it < 2 * 256 * 3; it += kFxThreads) {
      const int which = it >= 768;
      const int rem = it - which * 768;
      const int pair = rem / 3, col = rem % 3;
      const int x = pair >> 4, y = pair & 15;
      const int4 *gl = gs + ((which ? 2 : 0) * 16 + x) * 9;
      const int4 *gr = gs + ((which ? 1 : 3) * 16 + y) * 9;
      FxC hcol[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        Wide w = {0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < 3; ++k) wide_mac(w, fx_u(ut, x, y, c, k), fx_load(gr + 3 * k + col));
        // kPropBits + kLinkBits - 2 FX_LOW -> kMidBits
        constexpr int dn = kPropBits + kLinkBits - 2 * FX_LOW - kMidBits;
        const long long re = (wide_round<0>(w.hr, w.mr) + (1 << (dn - 1))) >> dn;
        const long long im = (wide_round<0>(w.hi, w.mi) + (1 << (dn - 1))) >> dn;
        big |= max(abs64(re), abs64(im)) >= kFxMost;
        hcol[c] = {fx_split(re), fx_split(im)};
      }
      longlong2 *dst = reinterpret_cast<longlong2 *>(which ? qs + pair * 9 : ps + x * kFxRow + y * 9) + col;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        Wide w = {0, 0, 0, 0};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          FxC g = fx_load(gl + 3 * c + r);
          g.im = fx_neg(g.im);
          wide_mac(w, g, hcol[c]);
        }
        const long long re = wide_round<2>(w.hr, w.mr), im = wide_round<2>(w.hi, w.mi);
        dst[3 * r] = make_longlong2(re, im);
        const unsigned long long v = (unsigned long long)(abs64(re) | abs64(im));
        if (which) most[1] |= v;
        else most[0] |= v;
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(most[k] >> 32));
      const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)most[k]);
      if ((tid & 31) == 0) atomicOr(&sh.most[k], ((unsigned long long)hi << 32) | lo);
    }
    if (big) sh.bad = 1;
    __syncthreads();
    const bool bad = sh.bad != 0;
    // P and Q at their own scales
    int sc[2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
      sc[k] = max(0, 64 - __clzll((long long)sh.most[k]) - (k ? PQBits<SLICES>::q : PQBits<SLICES>::p));
    __syncthreads();
    if (tid == 0) {
      for (int k = 0; k < 5; ++k) sh.e[k] = 0;
      sh.bad = 0;
      sh.most[0] = sh.most[1] = 0;
      a.marked[h] = bad;
      if (bad) *a.any_marked = 1;
    }
    if (h + (int)gridDim.x < a.nhc)
      issue_loads<kFxThreads>(a, h + gridDim.x, reinterpret_cast<double2 *>(gs),
                              reinterpret_cast<double2 *>(ut));
    if (bad) continue;  // the same in every thread
#pragma unroll 1
    for (int i = tid; i < 2 * 2304; i += kFxThreads) {
      const int k = i >= 2304, j = i - k * 2304;
      int4 *p = k ? qs + j : ps + (j / 144) * kFxRow + j % 144;
      const longlong2 v = *reinterpret_cast<const longlong2 *>(p);
      const int s = k ? sc[1] : sc[0];
      const long long half = s > 0 ? 1ll << (s - 1) : 0;
      *p = fx_word((v.x + half) >> s, (v.y + half) >> s);
    }
    __syncthreads();
    Wide w[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = {0, 0, 0, 0};
    if (mine) fx_contract<SLICES>(ps, qs, op, a1, a3, slice, w);
    // add the slices; afterwards every lane of a group holds the sums, as
    // 4 (re + rl 2^-FX_LOW): the sum of all slices may need 65 bits
    long long re[9], im[9];
    unsigned rl[9], il[9];
    constexpr int mask = (1 << FX_LOW) - 1;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const long long vr = w[k].hr + (w[k].mr >> FX_LOW), vi = w[k].hi + (w[k].mi >> FX_LOW);
      re[k] = vr >> 2;
      rl[k] = (((unsigned)vr & 3) << (FX_LOW - 2)) | (((unsigned)w[k].mr & mask) >> 2);
      im[k] = vi >> 2;
      il[k] = (((unsigned)vi & 3) << (FX_LOW - 2)) | (((unsigned)w[k].mi & mask) >> 2);
#pragma unroll
      for (int d = 1; d < SLICES; d <<= 1) {
        re[k] += __shfl_xor_sync(0xffffffffu, re[k], d);
        im[k] += __shfl_xor_sync(0xffffffffu, im[k], d);
        rl[k] += __shfl_xor_sync(0xffffffffu, rl[k], d);
        il[k] += __shfl_xor_sync(0xffffffffu, il[k], d);
      }
    }
    if (mine) {
      // units: P 2^(eu + e4 + e1 - kLinkBits - 2 kPropBits + ... + s), Q the
      // same with flavours 2, 3; the sums are in 2^(2 FX_LOW) of their product
      constexpr int vb = kMidBits + kPropBits - 2 * FX_LOW + 2;  // bits of |v| at scale 1
      const int ex = 2 * eu + (e[0] + e[1] + e[2] + e[3] - 4 * 1022) + sc[0] + sc[1] - 2 * vb +
                     2 * FX_LOW + 2;
      const double unit = __hiloint2double((ex + 1023) << 20, 0);
#pragma unroll
      for (int r = 0; r < kOwn; ++r) {
        const int k = r * SLICES + slice;
        long long vr = re[0], vi = im[0];
        unsigned lr = rl[0], li = il[0];
#pragma unroll
        for (int j = r * SLICES; j < (r + 1) * SLICES && j < 9; ++j)
          if (j == k) {
            vr = re[j];
            vi = im[j];
            lr = rl[j];
            li = il[j];
          }
        if (k < 9) {
          // low part through the bits of 2^52 + l: subtract its 2^52 / 2^27 from the high part
          const double dr = fma(__hiloint2double(0x43300000, (int)lr), 1.0 / (1 << FX_LOW),
                                (double)(vr - (1ll << (52 - FX_LOW))));
          const double di = fma(__hiloint2double(0x43300000, (int)li), 1.0 / (1 << FX_LOW),
                                (double)(vi - (1ll << (52 - FX_LOW))));
          if (a.out_hc)
            a.out_hc[(long)h * a.hc_stride + iop * 81 + 27 * a1 + 9 * (k % 3) + 3 * a3 + k / 3] =
                make_double2(dr * unit, di * unit);
          tot[r].x = fma(dr, unit, tot[r].x);
          tot[r].y = fma(di, unit, tot[r].y);
        }
      }
    }
  }
  if (mine) {
#pragma unroll
    for (int r = 0; r < kOwn; ++r) {
      const int k = r * SLICES + slice;
      if (k < 9)
        a.partial[((long)blockIdx.x * a.nops + iop) * 81 + 27 * a1 + 9 * (k % 3) + 3 * a3 + k / 3] = tot[r];
    }
  }
}

// Sum of the per-CTA partials, CTA 0 first.
__global__ void npr_sum_kernel(const double2 *partial, int nparts, int n, double2 *out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double2 s = make_double2(0.0, 0.0);
  for (int b = 0; b < nparts; ++b) {
    const double2 v = partial[(long)b * n + i];
    s.x += v.x;
    s.y += v.y;
  }
  out[i] = s;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace
}  // namespace sq

using namespace sq;

extern "C" int sq_spin_taste(int s, int f, int partner[16], int sign[16]) {
  if (s < 0 || s > 15 || f < 0 || f > 15 || !partner || !sign) return SQ_ERR_ARG;
  for (int a = 0; a < 16; ++a) {
    partner[a] = a ^ s ^ f;
    sign[a] = spin_taste_sign(s, f, a);
  }
  return SQ_OK;
}

extern "C" int npr_four_fermion(sq_ctx *ctx, const int dims[4], const double *links_dev,
                                const double *const props_dev[4], int nops, const int *ops,
                                double *out_dev, double *out_hc_dev, void *stream) {
  if (!ctx || !dims || !links_dev || !props_dev || nops < 0 || nops > (1 << 20))
    return SQ_ERR_ARG;
  if (nops > 0 && (!ops || !out_dev)) return SQ_ERR_ARG;
  long vol;
  int rc = check_lattice_dims(dims, &vol);
  if (rc) return rc;
  if (!aligned16(links_dev) || !aligned16(out_dev) || !aligned16(out_hc_dev)) return SQ_ERR_ARG;
  for (int f = 0; f < 4; ++f)
    if (!props_dev[f] || !aligned16(props_dev[f])) return SQ_ERR_ARG;
  for (long k = 0; k < 4L * nops; ++k)
    if (ops[k] < 0 || ops[k] > 15) return SQ_ERR_ARG;
  if (nops == 0) return SQ_OK;

  NprArgs a{};
  a.links = reinterpret_cast<const double2 *>(links_dev);
  for (int f = 0; f < 4; ++f) a.prop[f] = reinterpret_cast<const double2 *>(props_dev[f]);
  a.nhc = (int)(vol / 16);
  for (int mu = 0; mu < 4; ++mu) a.H[mu] = dims[mu] / 2;
  a.st[0] = 1;
  for (int mu = 1; mu < 4; ++mu) a.st[mu] = a.st[mu - 1] * dims[mu - 1];
  a.hc_stride = 81L * nops;

  cudaSetDevice(ctx->device);
  cudaStream_t st = stream ? (cudaStream_t)stream : cudaStreamLegacy;  // NULL: default stream
  // 2 to 16 slices of the sum over A per output tile: as many as the 288
  // threads hold for the operators of a group (9 tiles each)
  auto kernel_for = [](int n) {
    return n <= 2 ? npr_kernel<16> : n <= 4 ? npr_kernel<8> : n <= 8 ? npr_kernel<4> : npr_kernel<2>;
  };
  SQ_CUDA_TRY(cudaFuncSetAttribute(npr_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kSmemBytes));
  const int first = std::min(kMaxOps, nops), rest = nops % kMaxOps;
  for (int n : {first, rest})
    if (n > 0)
      SQ_CUDA_TRY(cudaFuncSetAttribute(kernel_for(n), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kFxSmem));
  int per_sm = 0;
  SQ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel_for(first), kFxThreads,
                                                            kFxSmem));
  if (per_sm < 1) per_sm = 1;
  const int grid = (int)std::min<long>(a.nhc, (long)per_sm * ctx->sms);
  void *partial = nullptr;
  const size_t partial_b = sizeof(double2) * (size_t)grid * kMaxOps * 81;
  SQ_CUDA_TRY(cudaMallocAsync(&partial, partial_b + 16 + (size_t)a.nhc, st));
  a.partial = static_cast<double2 *>(partial);
  a.any_marked = reinterpret_cast<int *>(static_cast<char *>(partial) + partial_b);
  a.marked = reinterpret_cast<unsigned char *>(a.any_marked + 4);
  cudaError_t e = cudaMemsetAsync(a.any_marked, 0, sizeof(int), st);
  // kMaxOps operators per launch group; each group recomputes the averaged
  // links and the sandwiches P, Q of every hypercube
  for (int g0 = 0; g0 < nops && e == cudaSuccess; g0 += kMaxOps) {
    a.nops = std::min(kMaxOps, nops - g0);
    for (int k = 0; k < a.nops; ++k) {
      const int *o = ops + 4 * (g0 + k);
      NprOp &p = a.ops[k];
      p.t1 = (uint8_t)(o[0] ^ o[1]);
      p.t2 = (uint8_t)(o[2] ^ o[3]);
      p.neg1 = p.neg2 = 0;
      for (int c = 0; c < 16; ++c) {
        if (spin_taste_sign(o[0], o[1], c) < 0) p.neg1 |= (uint16_t)(1u << c);
        if (spin_taste_sign(o[2], o[3], c) < 0) p.neg2 |= (uint16_t)(1u << c);
      }
    }
    a.out_hc = out_hc_dev ? reinterpret_cast<double2 *>(out_hc_dev) + 81L * g0 : nullptr;
    const int nitems = a.nops * 81;
    kernel_for(a.nops)<<<grid, kFxThreads, kFxSmem, st>>>(a);
    npr_fp64_kernel<<<std::min(grid, ctx->sms), kThreads, kSmemBytes, st>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess) {
      npr_sum_kernel<<<(nitems + 255) / 256, 256, 0, st>>>(
          a.partial, grid, nitems, reinterpret_cast<double2 *>(out_dev) + 81L * g0);
      e = cudaGetLastError();
      ctx->launches += 3;
    }
  }
  cudaFreeAsync(partial, st);
  if (e != cudaSuccess) {
    set_last_cuda_error(e, "npr kernels", __FILE__, __LINE__);
    return SQ_ERR_CUDA;
  }
  return SQ_OK;
}
