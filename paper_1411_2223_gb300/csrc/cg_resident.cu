// One-system CG as a kernel that stays on the device.
//
// A CG iteration of the launched form is five dependent kernels (two Dslash,
// their finish kernels, p = r + beta p), and on lattices of up to some 10^4
// sites per parity the launches and each thread's serial walk over the four
// directions, not the links, take its time: 21.7 us an iteration at 8^4.
// Here one cooperative launch, one block per SM, runs iterations until the
// system needs the host's sequence again (a reliable update, the end).
//   - Every site has its own lanes for the whole solve: its p, r and x stay in
//     registers, and what is left of an iteration are the gathers between grid
//     barriers, three of them (t = D_oe p with <p, A p>; the update with
//     |r|^2; p), or two where the neighbours form p as they gather (FP32 on
//     the smallest lattices: 13.2 -> 11.9 us).
//   - Up to four lanes share a site, a direction each (8^4: 17.7 -> 13.2 us).
//   - A barrier carries the blocks' sums; every block adds them in the same
//     order and takes the scalar step on its own copy of the system's state.
//     Arrival is one red.release and waiting one ld.acquire loop: separate
//     fences around them cost 0.9 us per iteration each way, and publishing
//     the sums as tagged words that every block polls was slower (a barrier
//     of 3.9 against 2.1 us at 6144 sites).
//   - The next phase's links are loaded before a barrier is waited for.
// Every wait is bounded: after kSpinLimit polls (seconds) a block sets the
// fault flag, and all blocks leave.
#include <algorithm>

#include "sq_host.h"

namespace sq {
namespace {

constexpr unsigned kSpinLimit = 1u << 24;

struct ResidentArgs {
  DslashArgs norm, update;
  char *p2;            // second buffer of p (merged form)
  unsigned *count;     // arrivals at the barrier, zero on entry
  double *sums;        // [2][grid]: what the blocks publish
  int *fault;          // set when a wait ran out
  int max_steps;       // iterations of this launch
};

// Grid barrier: arrive publishes the block's writes and a number of the block
// (v, thread 0's), wait makes every block's visible (to coherent loads) and
// returns the sum of the numbers, added in a fixed order (to warp 0).  Two sets
// of sums alternate: a block that writes the set of barrier n + 2 has passed
// n + 1, which every block enters after reading n.
struct GridBarrier {
  unsigned *count;
  double *sums;
  int *fault;
  int *ok;             // shared
  unsigned n, target;
  __device__ __forceinline__ void arrive(double v) {
    ++n;
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
      sums[(n & 1) * gridDim.x + blockIdx.x] = v;
      // releases the block's writes too: they are before the barrier above
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    }
  }
  // false when a wait ran out (in every thread)
  template <bool SUM>
  __device__ __forceinline__ bool wait(double &sum) {
    if (threadIdx.x == 0) {
      unsigned v = 0, polls = 0;
      *ok = 1;
      for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
        if (v >= target) break;
        if (++polls >= kSpinLimit || ((polls & 1023) == 0 && *(volatile int *)fault != 0)) {
          *(volatile int *)fault = 1;
          *ok = 0;
          break;
        }
      }
    }
    __syncthreads();
    if (SUM && threadIdx.x < 32) {
      double s = 0.0;
      for (int k = threadIdx.x; k < (int)gridDim.x; k += 32)
        s += __ldcg(sums + (n & 1) * gridDim.x + k);
      sum = warp_sum(s);
    }
    return *ok != 0;
  }
};

// Links of one direction, loaded before a barrier is waited for.
template <int PREC, int RECON> struct DirLinks {
  Mat3<float> m[4];
  __device__ __forceinline__ void load(const DslashArgs &a, int i, int mu) {
    LinkIO<PREC_F32, RECON>::load(a.links, a.g.stride, i, mu, a.ls, m);
  }
};
template <int RECON> struct DirLinks<PREC_I16, RECON> {
  I16Words<RECON> w;
  __device__ __forceinline__ void load(const DslashArgs &a, int i, int mu) {
    i16_load_words<RECON>(a.links, a.g.stride, i, mu, w, a.ls);
  }
};
template <int RECON> struct DirLinks<PREC_F64, RECON> {
  __device__ __forceinline__ void load(const DslashArgs &, int, int) {}
};

// p = a r + beta p
template <typename R>
__device__ __forceinline__ void xpay(Vec3<R> &p, const Vec3<R> &r, R are, R aim, R beta) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const R px = fma(are, r.c[c].x, fma(-aim, r.c[c].y, beta * p.c[c].x));
    const R py = fma(are, r.c[c].y, fma(aim, r.c[c].x, beta * p.c[c].y));
    p.c[c].x = px;
    p.c[c].y = py;
  }
}

// D in at site i by SPLIT neighbouring lanes, lane `sub` taking directions
// sub, sub + SPLIT, ...; the sum in every lane.  All lanes of the warp call
// it.  With a state s (FP32) the input is a r + beta p, r and p gathered.
template <int PREC, int RECON, int SPLIT, typename R>
__device__ __forceinline__ Vec3<R> split_dslash(const DslashArgs &a, bool valid, int i, int sub,
                                                DirLinks<PREC, RECON> &links, const char *r = nullptr,
                                                const char *pold = nullptr,
                                                const SlotState *s = nullptr) {
  const Geom &g = a.g;
  const bool active[1] = {true};
  Vec3<R> acc[1];
  zero(acc[0]);
  FxForm form = {0, 0, false};
  if (valid) {
    const SiteCoords sc = site_coords(g, a.out_parity, i);
    if constexpr (PREC == PREC_F64) {
      fixed_hops<1, MODE_PLAIN, IN_CO>(a, a.ls, sc, i, 0, active, acc, sub, SPLIT, &form);
    } else {
#pragma unroll 1
      for (int mu = sub; mu < 4; mu += SPLIT) {
        if (mu != sub) links.load(a, i, mu);
        if constexpr (PREC == PREC_I16) {
          i16_dir<RECON, 1, true>(a, a.ls, sc, mu, links.w.w, 0, active, acc);
        } else {
          int nb[4];
          float f[4];
          nb[0] = hop<+1>(g, sc, mu, f[0]);
          nb[1] = hop<-1>(g, sc, mu, f[1]);
          nb[2] = hop<+3>(g, sc, mu, f[2]);
          nb[3] = hop<-3>(g, sc, mu, f[3]);
          const float eta = eta_sign(sc, mu);
          Vec3<float> v[4];
#pragma unroll
          for (int h = 0; h < 4; ++h)
            v[h] = SpinorIO<PREC_F32>::template load<true>(s ? pold : a.in, g.stride, nb[h]);
          if (s) {
            const float are = (float)s->a_re, aim = (float)s->a_im, beta = (float)s->beta;
            Vec3<float> w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) w[h] = SpinorIO<PREC_F32>::template load<true>(r, g.stride, nb[h]);
#pragma unroll
            for (int h = 0; h < 4; ++h) xpay(v[h], w[h], are, aim, beta);
          }
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const float s = (h & 1) ? -eta * f[h] : eta * f[h];
#pragma unroll
            for (int c = 0; c < 3; ++c) { v[h].c[c].x *= s; v[h].c[c].y *= s; }
            mat_vec_acc(acc[0], links.m[h], v[h]);
          }
        }
      }
    }
  }
  if constexpr (PREC == PREC_F64) {
    // of all directions: the exponents' maxima and whether a neighbour was odd
    const bool odd_here = form.odd;
#pragma unroll
    for (int d = 1; d < SPLIT; d <<= 1) {
      form.e = max(form.e, __shfl_xor_sync(0xffffffffu, form.e, d));
      form.fat = max(form.fat, __shfl_xor_sync(0xffffffffu, form.fat, d));
    }
    const unsigned who = __ballot_sync(0xffffffffu, odd_here);
    form.odd = (who & (((1u << SPLIT) - 1) << ((threadIdx.x & 31) / SPLIT * SPLIT))) != 0;
    if (!form.odd && form.apart()) {  // each lane its directions, as before
      double o[6];
      fixed_site_apart<IN_CO>(a, i, 0, form, sub, SPLIT, o);
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[0].c[c] = make_double2(o[2 * c], o[2 * c + 1]);
    }
  }
#pragma unroll
  for (int d = 1; d < SPLIT; d <<= 1)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[0].c[c].x += __shfl_xor_sync(0xffffffffu, acc[0].c[c].x, d);
      acc[0].c[c].y += __shfl_xor_sync(0xffffffffu, acc[0].c[c].y, d);
    }
  if constexpr (PREC == PREC_F64) {
    if (form.odd) {
      double o[6];
      fixed_site_fp64<MODE_PLAIN, IN_CO>(a, i, 0, o);
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[0].c[c] = make_double2(o[2 * c], o[2 * c + 1]);
    }
  }
  return acc[0];
}

template <int PREC, int RECON, int SPLIT, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) cg_resident_kernel(const __grid_constant__ ResidentArgs a) {
  using R = typename SpinorIO<PREC>::R;
  constexpr int XP = (PREC == PREC_F64) ? PREC_F64 : PREC_F32;
  using RX = typename SpinorIO<XP>::R;
  // Merged form: the neighbours' new p is formed from r and the old p as they
  // are gathered, so that an iteration needs two barriers; p alternates
  // between two buffers.  FP32 only: in FP64 the FMAs at the gathers cost what
  // the barrier does, and a 16-bit p has to be the one that was stored.
  constexpr bool kMerged = PREC == PREC_F32 && SPLIT == 4;
  __shared__ SlotState s;
  __shared__ double red[THREADS / 32];
  __shared__ int ok;
  const Geom &g = a.norm.g;
  const int S = g.stride;
  const int tid = threadIdx.x;
  const int i = (blockIdx.x * blockDim.x + tid) / SPLIT, sub = tid % SPLIT;
  const bool valid = i < g.vh, mine = valid && sub == 0;  // the site's own-site work
  if (tid == 0) s = *a.norm.slots;
  __syncthreads();
  if (s.status != SLOT_RUNNING) return;  // the same in every block
  GridBarrier bar{a.count, a.sums, a.fault, &ok, 0, 0};
  auto block_sum = [&](R val) {  // in thread 0
    const R sv = warp_sum(val);
    if ((tid & 31) == 0) red[tid >> 5] = (double)sv;
    __syncthreads();
    double v = 0.0;
    if (tid == 0)
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
    return v;
  };
  DirLinks<PREC, RECON> links;
  Vec3<R> p, r;
  Vec3<RX> x;
  zero(p);
  zero(r);
  zero(x);
  char *const rm = a.update.out, *const pm = const_cast<char *>(a.update.p);
  if (mine) {
    p = SpinorIO<PREC>::template load<true>(pm, S, i);
    r = SpinorIO<PREC>::template load<true>(rm, S, i);
    x = SpinorIO<XP>::template load<true>(a.update.xs, S, i);
  }
  const R m2 = (R)s.m2;
  double sum = 0.0;
  for (int step = 0;; ++step) {
    // p = a r + beta p (after the start a = 1, beta = 0, or of a guess's residual)
    char *const pnew = kMerged && (step & 1) == 0 ? a.p2 : pm;
    if (mine) {
      xpay(p, r, (R)s.a_re, (R)s.a_im, (R)s.beta);
      SpinorIO<PREC>::store(pnew, S, i, p);
      if constexpr (PREC == PREC_I16) p = SpinorIO<PREC>::template load<true>(pnew, S, i);
    }
    if constexpr (!kMerged) {
      bar.arrive(0.0);
      if (valid) links.load(a.norm, i, sub);
      if (!bar.template wait<false>(sum)) break;
    } else if (step == 0) {
      if (valid) links.load(a.norm, i, sub);
    }
    // t = D_oe p, sum of |t|^2 + m^2 |p|^2
    {
      const Vec3<R> d = kMerged ? split_dslash<PREC, RECON, SPLIT, R>(a.norm, valid, i, sub, links, rm,
                                                                      (step & 1) ? a.p2 : pm, &s)
                                : split_dslash<PREC, RECON, SPLIT, R>(a.norm, valid, i, sub, links);
      R val = 0;
      if (mine) {
        Vec3<R> o;
        R no = 0, np = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          o.c[c].x = R(0.5) * d.c[c].x;
          o.c[c].y = R(0.5) * d.c[c].y;
          no = fma(o.c[c].x, o.c[c].x, fma(o.c[c].y, o.c[c].y, no));
          np = fma(p.c[c].x, p.c[c].x, fma(p.c[c].y, p.c[c].y, np));
        }
        SpinorIO<PREC>::store(a.norm.out, S, i, o);
        val = fma(m2, np, no);
      }
      bar.arrive(block_sum(val));
    }
    if (valid) links.load(a.update, i, sub);
    if (!bar.template wait<true>(sum)) break;
    if (tid == 0) finish_alpha(&s, sum);
    // xs += alpha p, r -= alpha (m^2 p - D_eo t), sum of |r|^2
    {
      const Vec3<R> d = split_dslash<PREC, RECON, SPLIT, R>(a.update, valid, i, sub, links);
      __syncthreads();  // alpha
      const R al = (R)s.alpha;
      R val = 0;
      if (mine && s.status == SLOT_RUNNING) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const R apx = fma(m2, p.c[c].x, R(-0.5) * d.c[c].x);
          const R apy = fma(m2, p.c[c].y, R(-0.5) * d.c[c].y);
          x.c[c].x = fma((RX)al, (RX)p.c[c].x, x.c[c].x);
          x.c[c].y = fma((RX)al, (RX)p.c[c].y, x.c[c].y);
          r.c[c].x = fma(-al, apx, r.c[c].x);
          r.c[c].y = fma(-al, apy, r.c[c].y);
          val = fma(r.c[c].x, r.c[c].x, fma(r.c[c].y, r.c[c].y, val));
        }
        if constexpr (kMerged) SpinorIO<PREC>::store(rm, S, i, r);
      }
      bar.arrive(block_sum(val));
    }
    if (kMerged && valid) links.load(a.norm, i, sub);
    if (!bar.template wait<true>(sum)) break;
    if (tid == 0 && s.status == SLOT_RUNNING) finish_update(&s, sum, 1);
    __syncthreads();
    if (s.status != SLOT_RUNNING || s.ru_pending || step + 1 >= a.max_steps) break;
  }
  if (mine) {  // the rest of the solver reads them from memory
    SpinorIO<PREC>::store(rm, S, i, r);
    SpinorIO<XP>::store(a.update.xs, S, i, x);
    if constexpr (kMerged) SpinorIO<PREC>::store(pm, S, i, p);
  }
  if (blockIdx.x == 0 && tid == 0) *a.norm.slots = s;
}

// Iterations of one launch: about 4 ms of them at most, as the kernel holds every
// SM and other streams' kernels (a served batch's) get in between launches only.
// 128 whatever the size, as it was first, were 10 ms in FP64 at 65536 sites; a new
// launch and the empty update pair before it cost some 20 us.
inline int resident_steps(int prec, int vh) {
  const double us = 10.0 + vh * (prec == PREC_F64 ? 1.1e-3 : 0.45e-3);  // see the table below
  return std::min(128, (int)(4000.0 / us));
}

// Lanes per site, and threads per block with the sites spread over the SMs in
// whole warps: four lanes while a block stays within 512 threads.
inline int lanes_per_site(int vh, int sms) {
  return 4 * vh <= 512 * sms ? 4 : 2 * vh <= 512 * sms ? 2 : 1;
}
inline int block_for(int vh, int sms) {
  const int threads = (vh * lanes_per_site(vh, sms) + sms - 1) / sms;
  return std::max(32, (threads + 31) / 32 * 32);
}

template <int PREC, int RECON, int SPLIT>
int launch(const ResidentArgs &a, int block, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.norm.g.vh * SPLIT + block - 1) / block);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto kern = block <= 256 ? cg_resident_kernel<PREC, RECON, SPLIT, 256>
                           : cg_resident_kernel<PREC, RECON, SPLIT, 512>;
  return cudaLaunchKernelEx(&cfg, kern, a) == cudaSuccess ? 0 : -1;
}

template <int PREC, int RECON>
int launch_split(const ResidentArgs &a, int block, int lanes, cudaStream_t st) {
  return lanes == 4 ? launch<PREC, RECON, 4>(a, block, st)
       : lanes == 2 ? launch<PREC, RECON, 2>(a, block, st)
                    : launch<PREC, RECON, 1>(a, block, st);
}

}  // namespace

// A workspace's fault flag, barrier count and sums, and second p.
static size_t barrier_bytes(const sq_ctx *ctx) {
  return (256 + sizeof(double) * 2 * ctx->sms + 255) / 256 * 256;
}

// One site per thread of one block per SM (77824 sites per parity on 152 SMs)
// is as far as the resident form goes; it is the faster one up to there, in
// us per iteration against the launched form (12-real long links for 16-bit):
//   sites per parity     2048       6144      20736      35840      65536
//   FP32           21.7  10.1  23.1  10.4  28.5  19.4  32.2  26.0  42.1  34.8
//   16-bit         22.1  14.4  24.6  14.2  27.1  18.6  29.0  22.1  36.9  32.3
//   FP64           41.5  20.1  54.1  26.7  65.4  43.0  68.2  54.2  86.4  78.0
// (whole solves over their iterations, reliable updates included, at one
// thread per site then: with a site's directions on four warps, 2048 sites
// take 9.5 in FP32 and 12.6 in 16-bit, 20736 take 19.2 and 18.0; FP64 takes 4 %
// more at 65536 since it compares the neighbours' exponents).  With two
// rounds per thread it loses: 50.5 against 42.1 at 65536 sites, 170 against
// 114 at 256000, as the SMs' last round is part empty.
size_t cg_resident_bytes(const sq_ctx *ctx, int vh, int nrhs, int prec, size_t fb) {
  if (nrhs != 1 || vh > 512 * ctx->sms) return 0;
  const bool merged = prec == PREC_F32 && lanes_per_site(vh, ctx->sms) == 4;
  return barrier_bytes(ctx) + (merged ? fb : 0);
}

int cg_resident_block(const CGWork *w) {
  const sq_ctx *ctx = w->ctx;
  const int vh = w->gf->g.vh;
  if (w->resident == nullptr) return 0;  // too large, or no memory for it
  if (w->prec == PREC_F64 && !w->gf->scales(PREC_F64, w->recon).fixed) return 0;
  int coop = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) != cudaSuccess || !coop)
    return 0;
  return block_for(vh, ctx->sms);
}

int cg_enqueue_resident(CGWork *w, const DslashArgs &norm, const DslashArgs &update,
                        cudaStream_t st) {
  ResidentArgs a;
  a.norm = norm;
  a.update = update;
  char *base = static_cast<char *>(w->resident);
  a.fault = reinterpret_cast<int *>(base);
  a.count = reinterpret_cast<unsigned *>(base + 128);
  a.sums = reinterpret_cast<double *>(base + 256);
  a.p2 = base + barrier_bytes(w->ctx);
  a.max_steps = resident_steps(w->prec, norm.g.vh);
  SQ_CUDA_TRY(cudaMemsetAsync(a.count, 0, sizeof(unsigned), st));
  int rc = -1;
  const int block = w->resident_block, lanes = lanes_per_site(norm.g.vh, w->ctx->sms);
  if (w->prec == PREC_F32)
    rc = w->recon == 12 ? launch_split<PREC_F32, 12>(a, block, lanes, st)
                        : launch_split<PREC_F32, 18>(a, block, lanes, st);
  else if (w->prec == PREC_I16)
    rc = w->recon == 12 ? launch_split<PREC_I16, 12>(a, block, lanes, st)
                        : launch_split<PREC_I16, 18>(a, block, lanes, st);
  else
    rc = launch_split<PREC_F64, RECON_FIXED>(a, block, lanes, st);
  if (rc) {
    const cudaError_t e = cudaGetLastError();
    set_last_cuda_error(e, "resident CG launch", __FILE__, __LINE__);
    return SQ_ERR_CUDA;
  }
  w->ctx->launches++;
  return SQ_OK;
}

}  // namespace sq
