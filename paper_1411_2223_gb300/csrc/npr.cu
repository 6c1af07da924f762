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
// 14 KB of input) is FP64 in its results but not in its units, which GB300
// has few of (npr_kernel):
//   - steps 2 and 3 run on the integer multiply-add units in the two-word
//     fixed-point form of sq_fixed.cuh, 54 to 57 bits relative to block
//     scales: one per hypercube for the links and for each flavour's
//     propagators;
//   - step 4, four fifths of the work, on the tensor cores: P and Q, at one
//     scale each, are cut into six signed 9-bit digits, which FP16 holds
//     exactly, and the digits' products are summed over the 256 (A, C) by
//     tcgen05.mma into FP32 accumulators in TMEM, exactly (256 256 256 = 2^24):
//     the error-free splitting of Ozaki, Ogita, Oishi and Rump ("Error-free
//     transformations of matrix multiplication by using fast routines of matrix
//     multiplication and its applications", Numer. Algorithms 59 (2012) 95).
// A hypercube whose inputs or averaged links do not fit that form (infinities,
// NaN, elements near the ends of FP64, links far from unitary), or of which an
// output is so much smaller than the largest products of its P and Q that the
// form's one scale would cost it digits (kRough below), is marked there and
// computed by npr_fp64_kernel in FP64.
// Per-hypercube results are written when asked for; the sums over hypercubes
// go through per-CTA partials and a fixed-order second pass, so they do not
// depend on scheduling.
#include <cmath>
#include <cstdint>

#include <cuda_fp16.h>

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
constexpr int kFxThreads = 512;  // npr_kernel
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
// for the links and their averages.
//
// Contraction.  With i, j = 0 .. 5 the digits of P and Q from the top,
//   P = sum_i p_i 512^(5-i), |p_i| <= 256,
// row 18 i + 2 (3 a1 + a4) + (0 re, 1 im) of the [108] x [256] matrix of p
// digits and column 18 j + 2 (3 a3 + a2) + (0, 1) of the [256] x [108] matrix
// of q digits give C = one 108 x 108 product per operator, of which the blocks
// i + j <= 6 are needed (the others are below 2^-59 of the scales' product).
// It is 16 tcgen05.mma of M 128, N 112, K 16 by one thread, one per A: P's
// digits stay as they were cut, in rows (A, D); Q's, in rows (B, C), are
// brought from the last operator's order of C and signs to this one's in place
// (an XOR of the row within 16, so pairs of rows swap), and B = A ^ t1 is in
// the descriptors.  While the tensor cores work, the last operator's C is
// added: the sums of digit pairs of one i + j as integers, the seven of them
// to two 64-bit words, and these converted once.  The wait for the products is
// bounded; a block in which one runs out returns NaN.
//
// 8 operators at 20^3 x 64: 37.2 ms with FP64 FMAs (their pipe 93 % busy),
// 15.2 ms with the contraction on the integer units too (three mad.wide.s32
// per real product, 32 lanes a clock and SM), 9.8 ms with mma.sync (7 thousand
// cycles per operator, of which ldmatrix reads of the permuted rows 3.7),
// 8.1 ms on tcgen05, 8.3 ms with the comparison below.  About 40 thousand cycles per hypercube go to the steps up to
// the digits (the integer multiply-adds alone are 10), 5 thousand to each
// operator: reordering Q, and C from TMEM through shared memory.  Error of a
// hypercube against long double 3.2e-16 to 3.6e-16, with FP64 FMAs (three per
// complex term) 4.6e-16.
//
// One scale for all of P and Q: an output is a sum of P[A][D] Q[C][B] over
// pairs of corners that the operator picks, and where the flavours peak at
// different corners (or source colours) it has only products of large P with
// small Q and the other way round, while P and Q are rounded to 2^-54 of their
// largest elements.  With g_f(c, a) the norm of flavour f's column a at corner c,
// an output's FP64 rounding goes with R, its rounding here with M,
//   R^2 = sum_A g1(A, a1)^2 g2(A ^ t1, a2)^2  sum_C g3(C, a3)^2 g4(C ^ t2, a4)^2,
//   M^2 = |P|max^2 sum g3^2 sum g2^2 + |Q|max^2 sum g1^2 sum g4^2.
// A hypercube with M > 12 R in any output and for any t1, t2 (so that it does not
// depend on the other operators of the call) goes to npr_fp64_kernel.  The
// largest error of a hypercube's outputs, each over the root of the sum of its
// |P|^2 |Q|^2, is 0.9e-15 at M / R = 5, 1.1e-15 at 7, 1.6e-15 at 12, 2.3e-15 at 20
// and 1e-14 at 100, and 1.7e-15 with FP64 FMAs (medians, the steps in long
// double).  Gaussian propagators have M / R of 5, above 8 in 1 % of the
// hypercubes and above 11 in none of 20000; with peaks of 2 at opposite corners
// it is 9 to 16, of 8 200 to 400.  The norms and the comparison cost 2.6 % of the
// call (16^3 x 32, 8 operators: 2.11 to 2.165 ms).
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

constexpr long long kFxMost = 1ll << (FX_LOW + 30);  // two words hold values below this
constexpr int kPropBits = FX_BITS, kLinkBits = 56;   // bits at the blocks' scales
constexpr int kMidBits = 55;                         // ... of U G4 and U G2
constexpr int kDigits = 6, kDigitBits = 9;
constexpr float kRough = 144.f;                      // largest M^2 / R^2 of an output
constexpr int kPQBits = kDigits * kDigitBits - 1;    // P and Q: |v| <= 2^53
// Digits of P, Q in core matrices of 8 rows (k) of 8 columns, 128 bytes; the 14
// of a row of cores follow each other.
constexpr int kCores = 14, kCols = 8 * kCores;
constexpr int kCoreRow = kCores * 128;               // bytes of 8 rows
constexpr size_t kDigitBytes = 32 * kCoreRow;
constexpr int kFxUG = kTri * 9 + 4 * 16 * 9;  // int4 of the links and propagators
constexpr size_t kFxSmem = sizeof(int4) * (kFxUG + 2 * 2304) + 2 * kDigitBytes;

struct FxShared {
  int e[5];                    // largest biased exponents: 4 flavours, links
  int bad;                     // the hypercube does not fit
  int fail;                    // a wait for the tensor cores ran out
  unsigned tmem;               // first column of the accumulator
  unsigned long long done;     // mbarrier: an operator's products are complete
  unsigned long long most[2];  // largest |v| of P and Q before scaling
  unsigned seen;               // bit 3 f + a: column a of flavour f has a nonzero element
  float g2[4][16][3];          // squared norms of the propagators' columns, at the scales
  float g2_sum[4][3];          // ... summed over the corners
  float pair[18];              // the sums of R^2: least over t1 of 3 a1 + a2, then over t2 of 3 a3 + a4
};

__device__ __forceinline__ int fx_biased(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v 2^(FX_BITS - e) for a largest biased exponent e + 1022
__device__ __forceinline__ long long fx_scaled(double v, int biased_top) {
  const Fx a = fx_from_double(v, biased_top, 1);
  return ((long long)a.h << FX_LOW) + a.l;
}

constexpr int kCRow = 108;                           // floats of a row of C
static_assert(108 * kCRow * sizeof(float) <= 2 * 2304 * sizeof(longlong2), "C fits where P and Q were");
constexpr int kTmemCols = 128;
constexpr unsigned kWaitLimit = 1u << 22;            // polls of an mbarrier: under a second
constexpr int kIssuer = kFxThreads - 32;             // the thread that issues the products

// byte of (row k, column c) of a digit matrix
__device__ __forceinline__ unsigned digit_at(int k, int c) {
  return (k >> 3) * kCoreRow + (c >> 3) * 128 + (k & 7) * 16 + (c & 7) * 2;
}

// Shared-memory descriptor: no swizzle, columns (M, N) contiguous; cores 128
// bytes apart along the columns, kCoreRow along k.
__device__ __forceinline__ unsigned long long digit_desc(unsigned addr) {
  return (unsigned long long)((addr & 0x3ffff) >> 4) | ((unsigned long long)(kCoreRow >> 4) << 16) |
         ((unsigned long long)(128 >> 4) << 32) | (1ull << 46);
}

// C = the digit products of one operator, 128 x 112 x 256, by one thread.
__device__ __forceinline__ void issue_products(unsigned pd, unsigned qd, int t1, unsigned tmem, unsigned done) {
  // FP32 sums of FP16 products, both operands contiguous in their columns
  constexpr unsigned idesc = (1u << 4) | (1u << 15) | (1u << 16) | ((unsigned)(kCols >> 3) << 17) | ((128u >> 4) << 24);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
  for (int A = 0; A < 16; ++A) {
    const unsigned long long da = digit_desc(pd + A * 2 * kCoreRow), db = digit_desc(qd + (A ^ t1) * 2 * kCoreRow);
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
        ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(A) : "memory");
  }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(done) : "memory");
}

__device__ __forceinline__ bool wait_products(unsigned done, unsigned parity) {
  for (unsigned k = 0; k < kWaitLimit; ++k) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok) : "r"(done), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}

// The accumulator to C in shared memory: warp w its quarter w % 4 of the rows,
// 32 columns from 32 (w / 4).
__device__ __forceinline__ void store_products(unsigned tmem, float *c) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = (warp & 3) * 32 + lane, col = (warp >> 2) * 32;
  unsigned v[32];
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(tmem + ((unsigned)((warp & 3) * 32) << 16) + col));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (row < 108) {
#pragma unroll
    for (int u = 0; u < 32; u += 4)
      if (col + u < 108)
        *reinterpret_cast<uint4 *>(c + row * kCRow + col + u) = make_uint4(v[u], v[u + 1], v[u + 2], v[u + 3]);
  }
}

// Signs and order of C of the digits of Q, from operator `was` (no permutation,
// no sign if null) to `op`: row (B, c) holds +-Q[B][c ^ t2], of sign
// neg1[B ^ t1] neg2[c ^ t2], where the rows of P meet it in their own order.
__device__ __forceinline__ void arrange_q(char *qd, NprOp was, NprOp op) {
  const int d = was.t2 ^ op.t2;
  const int bit = d ? 31 - __clz(d) : 3;
  const int lo = threadIdx.x & 7, B = (threadIdx.x >> 3) & 15;
  int x = ((lo >> bit) << (bit + 1)) | (lo & ((1 << bit) - 1));
  // the eight lanes of a 128-byte access on different rows of the two cores
  if (bit < 3 && (x & 8)) x |= 1 << bit;
  const int y = d ? x ^ d : x | 8;  // x's partner
  const unsigned b = ((was.neg1 >> (B ^ was.t1)) ^ (op.neg1 >> (B ^ op.t1))) & 1;
  auto sign = [&](int c) {  // of the value now at row c, which goes to row c ^ d
    const unsigned f = b ^ ((was.neg2 >> (c ^ was.t2)) & 1) ^ ((op.neg2 >> (c ^ d ^ op.t2)) & 1);
    return f ? 0x80008000u : 0u;
  };
  const unsigned sx = sign(x), sy = sign(y);
  for (int n = threadIdx.x >> 7; n < kCores; n += kFxThreads / 128) {
    uint4 *px = reinterpret_cast<uint4 *>(qd + digit_at(B * 16 + x, n * 8));
    uint4 *py = reinterpret_cast<uint4 *>(qd + digit_at(B * 16 + y, n * 8));
    const uint4 vx = *px, vy = *py;
    *(d ? py : px) = make_uint4(vx.x ^ sx, vx.y ^ sx, vx.z ^ sx, vx.w ^ sx);
    *(d ? px : py) = make_uint4(vy.x ^ sy, vy.y ^ sy, vy.z ^ sy, vy.w ^ sy);
  }
}

// Sums over (A, C) of p q for the real parts (ra, rb) of output elements
// pe, qe: hi + lo 2^-27 in units of 512^7.
__device__ __forceinline__ void digit_sum(const float *c, int ra, int rb, long long &hi, long long &lo) {
  int level[7];
#pragma unroll
  for (int s = 0; s < 7; ++s) level[s] = 0;
#pragma unroll
  for (int i = 0; i < kDigits; ++i)
#pragma unroll
    for (int j = 0; j < kDigits; ++j)
      if (i + j <= 6)
        level[i + j] += __float2int_rn(c[(18 * i + ra) * kCRow + 18 * j + rb]);
  hi = ((((long long)level[0] * 512 + level[1]) * 512 + level[2]) * 512) + level[3];
  lo = (((long long)level[4] * 512 + level[5]) * 512) + level[6];
}

__global__ void __launch_bounds__(kFxThreads, 1) npr_kernel(const __grid_constant__ NprArgs a) {
  extern __shared__ int4 fsm[];
  __shared__ FxShared sh;
  int4 *ut = fsm;                       // [pair A <= D][3][3]
  int4 *gs = ut + kTri * 9;             // [flavour][corner][3][3]
  longlong2 *pq = reinterpret_cast<longlong2 *>(gs + 4 * 16 * 9);  // P [A][D][9], Q [B][C][9]
  float *cm = reinterpret_cast<float *>(pq);                       // C, once these are cut
  char *pd = reinterpret_cast<char *>(pq + 2 * 2304);              // digits of P, then of Q
  const unsigned pd_s = (unsigned)__cvta_generic_to_shared(pd), qd_s = pd_s + (unsigned)kDigitBytes;
  const unsigned done = (unsigned)__cvta_generic_to_shared(&sh.done);
  const int tid = threadIdx.x;
  if (tid == 0) {
    for (int k = 0; k < 5; ++k) sh.e[k] = 0;
    sh.bad = 0;
    sh.fail = 0;
    sh.seen = 0;
    sh.most[0] = sh.most[1] = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"((unsigned)__cvta_generic_to_shared(&sh.tmem)), "n"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  unsigned phase = 0;
  // columns 108 .. 111 of the digits meet no output, but are multiplied
  for (int i = tid; i < 2 * 256; i += kFxThreads)
    *reinterpret_cast<uint2 *>(pd + (i >> 8) * kDigitBytes + digit_at(i & 255, 108)) = make_uint2(0, 0);
  // this thread's part of an operator's outputs: output o = tid / 4, and the
  // real (0) or imaginary (1) parts of P and Q
  const int o = tid >> 2, part = tid & 3;
  const bool mine = o < 81;
  const int oe = mine ? o : 0;
  const int ra = 2 * (3 * (oe / 27) + oe % 3) + (part >> 1);            // P[a1][a4]
  const int rb = 2 * (3 * ((oe / 3) % 3) + (oe / 9) % 3) + (part & 1);  // Q[a3][a2]
  double *sum = reinterpret_cast<double *>(a.partial + (long)blockIdx.x * a.nops * 81);
  if (mine && part < 2)
    for (int op = 0; op < a.nops; ++op) sum[2 * (op * 81 + o) + part] = 0.0;
  int h = blockIdx.x;
  if (h < a.nhc)
    issue_loads<kFxThreads>(a, h, reinterpret_cast<double2 *>(gs), reinterpret_cast<double2 *>(ut));
  for (; h < a.nhc; h += gridDim.x) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    // block scales of the inputs: 576 elements of the propagators, then 288 of
    // the links (a warp's 32 span two blocks at most)
    int4 *own[2];
    double2 raw[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = tid + k * kFxThreads;
      if (i < 576) {
        own[k] = gs + i;
      } else {
        const int j = min(i - 576, 287), mu = j / 72, m = (j / 9) % 8, e = j % 9;
        const int c = ((m >> mu) << (mu + 1)) | (m & ((1 << mu) - 1));
        own[k] = ut + tri(c, c | (1 << mu)) * 9 + e;
      }
      raw[k] = *reinterpret_cast<const double2 *>(own[k]);
      const int b = max(fx_biased(raw[k].x), fx_biased(raw[k].y));
      const int f = min(i / 144, 4);
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
    unsigned seen = 0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = tid + k * kFxThreads;
      if (i >= 864) break;
      int top = e[4];
#pragma unroll
      for (int f = 0; f < 4; ++f)
        if (i / 144 == f) top = e[f];
      const int up = i < 576 ? 0 : kLinkBits - FX_BITS;
      *own[k] = fx_word(fx_scaled(raw[k].x, top) << up, fx_scaled(raw[k].y, top) << up);
      if (fx_biased(raw[k].x) == 0) fits &= raw[k].x == 0.0;  // no denormals
      if (fx_biased(raw[k].y) == 0) fits &= raw[k].y == 0.0;
      if (i < 576 && (raw[k].x != 0.0 || raw[k].y != 0.0)) seen |= 1u << (3 * (i / 144) + i % 3);
    }
    seen = __reduce_or_sync(0xffffffffu, seen);
    if ((tid & 31) == 0) atomicOr(&sh.seen, seen);
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
      if (tid < npairs * 9) {
        const int k = tid / 9, el = tid % 9, i = el / 3, j = el % 3;
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
      } else if (n == 3 && tid >= 320) {  // threads without a pair: M and R's norms
        const int k = tid - 320;
        const int4 *g = gs + (k / 3) * 9 + k % 3;
        float q = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int4 v = g[3 * c];
          const float re = fmaf((float)v.y, 0x1p-28f, (float)v.x * 0x1p-55f);
          const float im = fmaf((float)v.w, 0x1p-28f, (float)v.z * 0x1p-55f);
          q = fmaf(re, re, fmaf(im, im, q));
        }
        sh.g2[k / 48][(k / 3) % 16][k % 3] = q;
      } else if (n == 4 && tid >= 96 && tid < 384) {  // t in the 16 lanes, the sum's columns
        const int k = (tid - 96) >> 4, t = tid & 15;
        const int f = k < 9 ? 0 : 2, a = (k % 9) / 3, b = k % 3;
        float q = 0.f;
#pragma unroll
        for (int c = 0; c < 16; ++c) q = fmaf(sh.g2[f][c][a], sh.g2[f + 1][c ^ t][b], q);
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) q = fminf(q, __shfl_xor_sync(0xffffffffu, q, d));
        if (t == 0) sh.pair[k] = q;
      } else if (n == 4 && tid >= 384 && tid < 396) {
        const int f = (tid - 384) / 3, a = tid % 3;
        float q = 0.f;
        for (int c = 0; c < 16; ++c) q += sh.g2[f][c][a];
        sh.g2_sum[f][a] = q;
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
      // P[A][D] in rows (A, D); Q[C][B] in rows (B, C)
      const int x = which ? pair & 15 : pair >> 4, y = which ? pair >> 4 : pair & 15;
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
      longlong2 *dst = pq + which * 2304 + pair * 9 + col;
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
    constexpr int vb = kMidBits + kPropBits - 2 * FX_LOW + 2;  // bits of |v| at scale 1
    // P and Q at their own scales
    int sc[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) sc[k] = max(0, 64 - __clzll((long long)sh.most[k]) - kPQBits);
    bool rough = false;  // output tid: M^2 > kRough R^2, of columns that are not all zero
    if (tid < 81) {
      const int a1 = tid / 27, a2 = (tid / 9) % 3, a3 = (tid / 3) % 3, a4 = tid % 3;
      // |P|max, |Q|max as powers of two; the steps before P and Q round to the
      // propagators' scales, which counts as 1/2 of their product
      const float p = __int_as_float((max(sc[0] + kPQBits + eu - vb, -1) + 127) << 23);
      const float q = __int_as_float((max(sc[1] + kPQBits + eu - vb, -1) + 127) << 23);
      const float m2 = fmaf(p * p, sh.g2_sum[2][a3] * sh.g2_sum[1][a2], q * q * (sh.g2_sum[0][a1] * sh.g2_sum[3][a4]));
      const unsigned cols = 1u << a1 | 8u << a2 | 64u << a3 | 512u << a4;
      rough = (sh.seen & cols) == cols && !(m2 <= kRough * sh.pair[3 * a1 + a2] * sh.pair[9 + 3 * a3 + a4]);
    }
    const bool bad = __syncthreads_or(rough || sh.bad != 0);
    if (tid == 0) {
      for (int k = 0; k < 5; ++k) sh.e[k] = 0;
      sh.bad = 0;
      sh.seen = 0;
      sh.most[0] = sh.most[1] = 0;
      a.marked[h] = bad;
      if (bad) *a.any_marked = 1;
    }
    if (h + (int)gridDim.x < a.nhc)
      issue_loads<kFxThreads>(a, h + gridDim.x, reinterpret_cast<double2 *>(gs),
                              reinterpret_cast<double2 *>(ut));
    if (bad) continue;  // the same in every thread
    // cut into digits: with 256 (1 + 512 + ... + 512^5) added, the digits are
    // the value's 9-bit fields less 256; 1024 + field is an FP16 bit pattern
#pragma unroll 1
    for (int i = tid; i < 2 * 2304; i += kFxThreads) {
      const int k = i >= 2304;
      const longlong2 v = pq[i];
      const int s = k ? sc[1] : sc[0];
      const long long half = s > 0 ? 1ll << (s - 1) : 0;
      constexpr long long bias = 256ll * (1ll + 512 + (1ll << 18) + (1ll << 27) + (1ll << 36) + (1ll << 45));
      const unsigned long long re = (unsigned long long)(((v.x + half) >> s) + bias);
      const unsigned long long im = (unsigned long long)(((v.y + half) >> s) + bias);
      const int j = i - k * 2304;
      char *dst = pd + k * kDigitBytes;
#pragma unroll
      for (int d = 0; d < kDigits; ++d) {  // from the top
        const int at = kDigitBits * (kDigits - 1 - d);
        const unsigned mr = d ? 511u : 1023u;  // the top field may reach 512
        const unsigned w = ((unsigned)(re >> at) & mr) | (((unsigned)(im >> at) & mr) << 16) | 0x64006400u;
        *reinterpret_cast<__half2 *>(dst + digit_at(j / 9, 18 * d + 2 * (j % 9))) = __hsub2(*reinterpret_cast<const __half2 *>(&w), __floats2half2_rn(1280.f, 1280.f));
      }
    }
    // units: P 2^(eu + e4 + e1 - vb + s), Q the same with flavours 2, 3; the
    // sums are in 512^7 of their product
    const int ex = 2 * eu + (e[0] + e[1] + e[2] + e[3] - 4 * 1022) + sc[0] + sc[1] - 2 * vb + 7 * kDigitBits;
    const double unit = __hiloint2double((ex + 1023) << 20, 0);
    __syncthreads();
    auto add = [&](int op) {  // operator op's outputs from C
      if (tid >= 352) return;  // whole warps with outputs
      long long hi, lo;
      digit_sum(cm, ra, rb, hi, lo);
      // parts 0..3: re re, re im, im re, im im; part 0 becomes re re - im im,
      // part 1 re im + im re
      const long long hx = __shfl_xor_sync(0xffffffffu, hi, 3), lx = __shfl_xor_sync(0xffffffffu, lo, 3);
      hi += part == 0 ? -hx : hx;
      lo += part == 0 ? -lx : lx;
      if (mine && part < 2) {
        const double d = fma((double)lo, 1.0 / (1 << 27), (double)hi);
        const int at = op * 81 + o;
        if (a.out_hc) reinterpret_cast<double *>(a.out_hc + (long)h * a.hc_stride + at)[part] = d * unit;
        sum[2 * at + part] = fma(d, unit, sum[2 * at + part]);
      }
    };
    // operator op's products while op - 1's are added
    NprOp was = {0, 0, 0, 0};
#pragma unroll 1
    for (int op = 0; op < a.nops; ++op) {
      arrange_q(pd + kDigitBytes, was, a.ops[op]);
      was = a.ops[op];
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (tid == kIssuer) issue_products(pd_s, qd_s, was.t1, sh.tmem, done);
      if (op > 0) add(op - 1);
      __syncwarp();
      const bool ok = wait_products(done, phase);
      phase ^= 1;
      if (!ok) sh.fail = 1;
      __syncthreads();
      if (sh.fail) break;
      store_products(sh.tmem, cm);
    }
    if (sh.fail) break;
    __syncthreads();
    add(a.nops - 1);
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  if (sh.fail) {  // the same in every thread: NaN, once the products in flight are
    // complete or have had eight times the limit more
    for (int k = 0; k < 8 && !wait_products(done, phase ^ 1); ++k) {}
    if (mine && part < 2)
      for (int op = 0; op < a.nops; ++op) sum[2 * (op * 81 + o) + part] = __longlong_as_double(-1ll);
    for (; h < a.nhc; h += gridDim.x) {
      if (tid == 0) a.marked[h] = 0;
      for (int i = tid; a.out_hc && i < a.nops * 162; i += kFxThreads)
        reinterpret_cast<double *>(a.out_hc + (long)h * a.hc_stride)[i] = __longlong_as_double(-1ll);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid < 32) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh.tmem), "n"(kTmemCols));
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
  SQ_CUDA_TRY(cudaFuncSetAttribute(npr_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kSmemBytes));
  SQ_CUDA_TRY(cudaFuncSetAttribute(npr_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kFxSmem));
  const int grid = (int)std::min<long>(a.nhc, ctx->sms);  // one CTA per SM
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
    npr_kernel<<<grid, kFxThreads, kFxSmem, st>>>(a);
    npr_fp64_kernel<<<grid, kThreads, kSmemBytes, st>>>(a);
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
