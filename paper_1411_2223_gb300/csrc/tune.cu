// Run-time autotuner of the Dslash launch shape: threads per block and the
// number of right-hand sides each thread applies a loaded link to.  The
// paper's QUDA path picks launch parameters "dynamically and automatically"
// (Sec. 3); this tuner times every candidate with CUDA events on the first
// use of a (lattice, precision, link format, batch size) key and caches the
// winner for the context.  SQ_TUNE_CACHE=<file> persists the cache across
// processes; lines that a user puts there force their shapes.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <utility>
#include <vector>

#include "sq_host.h"

namespace sq {

struct Tuner {
  std::mutex mu;
  std::map<std::string, DslashConfig> cache;
  std::map<std::string, DslashConfig> forced;  // the user's lines of the file
  std::string path;
};

// A user's line of the file and a choice of the tuner have different names, so
// that what the library has written there itself forces nothing on a later
// process.  The FP64 kernels of fields with fixed-point links (:x) and with
// doubles (:d) are different ones.
constexpr char FORCED[] = "dslash_v4:", CHOSEN[] = "dslash_v5:";
static std::string shape_key(const Geom &g, int prec, int recon, int nrhs, int mode) {
  std::ostringstream s;
  s << g.L[0] << "x" << g.L[1] << "x" << g.L[2] << "x" << g.L[3] << ":p" << prec << ":r" << recon
    << ":n" << nrhs << ":m" << mode;
  return s.str();
}
static std::string forced_key(const GaugeField &gf, int prec, int recon, int nrhs, int mode) {
  return FORCED + shape_key(gf.g, prec, recon, nrhs, mode);
}
static std::string chosen_key(const GaugeField &gf, int prec, int recon, int nrhs, int mode) {
  const char *form = prec != PREC_F64 ? "" : gf.scales(prec, recon).fixed ? ":x" : ":d";
  return CHOSEN + shape_key(gf.g, prec, recon, nrhs, mode) + form;
}

Tuner *tuner_create() {
  Tuner *t = new Tuner();
  const char *p = std::getenv("SQ_TUNE_CACHE");
  if (p && *p) {
    t->path = p;
    std::ifstream in(t->path);
    std::string key;
    DslashConfig c;
    while (in >> key >> c.block >> c.nr)
      (key.rfind(FORCED, 0) == 0 ? t->forced : t->cache)[key] = c;
  }
  return t;
}

void tuner_destroy(Tuner *t) { delete t; }

bool tuned_forced(sq_ctx *ctx, const GaugeField &gf, int prec, int recon, int nrhs, int mode) {
  Tuner *t = ctx->tuner;  // `forced` does not change after the start
  return t && t->forced.count(forced_key(gf, prec, recon, nrhs, mode)) != 0;
}

static void tuner_save(Tuner *t) {
  if (t->path.empty()) return;
  std::ofstream out(t->path);
  for (auto *m : {&t->forced, &t->cache})
    for (auto &kv : *m) out << kv.first << " " << kv.second.block << " " << kv.second.nr << "\n";
}

// Device buffers and arguments of one Dslash kernel on synthetic inputs, for
// timing it alone: the gauge field's own links, zero-filled vector fields
// with a finite non-zero input, and, for the reducing epilogues, running
// systems that the timed launches cannot stop (no convergence, no max_iter,
// no reliable update).
struct KernelBench {
  void *in = nullptr, *out = nullptr, *aux = nullptr;
  DslashArgs a;
  ~KernelBench() {
    if (in) cudaFree(in);
    if (out) cudaFree(out);
    if (aux) cudaFree(aux);
  }
  bool setup(const GaugeField &gf, int prec, int recon, int nrhs, int mode, cudaStream_t st) {
    const bool reduces = mode != MODE_PLAIN;
    const Geom &g = gf.g;
    const size_t fb = spinor_bytes(prec, g.stride);
    // aux: the p field, slot states, partial sums, the ticket counters and
    // the solution increment xs, each 256-byte aligned
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t xs_b = spinor_bytes(xs_prec(prec), g.stride) * nrhs;
    const size_t o_slots = al(fb * nrhs);
    const size_t o_part = o_slots + al(sizeof(SlotState) * nrhs);
    const size_t o_cnt = o_part + al(sizeof(double) * 3 * nrhs * red_stride(g));
    const size_t o_xs = o_cnt + al(sizeof(unsigned) * nrhs * ticket_stride(g));
    const size_t aux_b = o_xs + al(xs_b);
    if (cudaMalloc(&in, fb * nrhs) != cudaSuccess || cudaMalloc(&out, fb * nrhs) != cudaSuccess ||
        cudaMalloc(&aux, aux_b) != cudaSuccess)
      return false;
    // input: a finite non-zero byte pattern (about 0.01 in FP32)
    cudaMemsetAsync(in, 0x3c, fb * nrhs, st);
    cudaMemsetAsync(out, 0, fb * nrhs, st);
    cudaMemsetAsync(aux, 0, aux_b, st);
    char *auxc = static_cast<char *>(aux);
    SlotState *slots = reinterpret_cast<SlotState *>(auxc + o_slots);
    if (reduces) {
      std::vector<SlotState> hs(nrhs);
      for (auto &s : hs) {
        std::memset(&s, 0, sizeof(s));
        s.status = SLOT_RUNNING;
        s.m2 = 1e-4;
        s.rr = 1.0;
        s.tol2b2 = -1.0;
        s.max_iter = 1 << 30;
      }
      if (cudaMemcpyAsync(slots, hs.data(), sizeof(SlotState) * nrhs, cudaMemcpyHostToDevice,
                          st) != cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess)
        return false;
    }
    std::memset(&a, 0, sizeof(a));
    a.g = g;
    a.out_parity = 1;
    a.links = gf.link_ptr(prec, recon, 1);
    a.ls = gf.scales(prec, recon);
    a.in = static_cast<const char *>(in);
    a.out = static_cast<char *>(out);
    a.in_fb = a.out_fb = fb;
    a.nrhs = nrhs;
    a.gate = GATE_NONE;
    if (reduces) {
      a.slots = slots;
      a.partial = reinterpret_cast<double *>(auxc + o_part);
      a.counter = reinterpret_cast<unsigned *>(auxc + o_cnt);
      a.gate = GATE_RUNNING;
    }
    if (mode == MODE_MDAGM || mode == MODE_UPDATE) {
      a.out_parity = 0;
      a.links = gf.link_ptr(prec, recon, 0);
      a.p = auxc;
      a.p_fb = fb;
    }
    if (mode == MODE_UPDATE) {
      a.xs = auxc + o_xs;
      a.xs_fb = spinor_bytes(xs_prec(prec), g.stride);
      a.xs_prec = xs_prec(prec);
    }
    return true;
  }
};

// Milliseconds per launch of `reps` back-to-back launches (CUDA events on
// `st`) after one untimed launch; negative if the shape cannot launch.
static float time_launches(KernelBench &kb, int prec, int recon, int nr, int mode, int block,
                           int reps, cudaStream_t st, sq_ctx *ctx) {
  if (launch_dslash(prec, recon, nr, mode, prec, kb.a, block, st) != 0) return -1.f;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaEventRecord(e0, st);
  for (int k = 0; k < reps; ++k) launch_dslash(prec, recon, nr, mode, prec, kb.a, block, st);
  cudaEventRecord(e1, st);
  float ms = -1.f;
  if (cudaEventSynchronize(e1) == cudaSuccess) {
    cudaEventElapsedTime(&ms, e0, e1);
    ms /= reps;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  ctx->launches += reps + 1;
  if (cudaGetLastError() != cudaSuccess) return -1.f;
  return ms;
}

DslashConfig tuned_dslash(sq_ctx *ctx, const GaugeField &gf, int prec, int recon, int nrhs,
                          int mode, cudaStream_t st) {
  // PLAIN and the reduction epilogues (MDAGM, NORM, UPDATE) are tuned apart:
  // a reduction favours more, smaller blocks per SM.  RESID uses the PLAIN
  // shape.
  if (mode != MODE_MDAGM && mode != MODE_NORM && mode != MODE_UPDATE) mode = MODE_PLAIN;
  DslashConfig def;
  def.block = 256;
  def.nr = nrhs >= 4 ? 4 : nrhs >= 2 ? 2 : 1;
  Tuner *t = ctx->tuner;
  if (!t || !gf.has(prec, recon)) return def;
  const auto forced = t->forced.find(forced_key(gf, prec, recon, nrhs, mode));
  if (forced != t->forced.end()) return forced->second;
  const std::string key = chosen_key(gf, prec, recon, nrhs, mode);
  std::lock_guard<std::mutex> lk(t->mu);
  auto it = t->cache.find(key);
  if (it != t->cache.end()) return it->second;
  cudaStreamCaptureStatus cs;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone)
    return def;
  KernelBench kb;
  if (!kb.setup(gf, prec, recon, nrhs, mode, st)) return def;
  // RHS tiles (1, 2 or 4 systems per thread)
  std::vector<int> nrs = {1};
  for (int nr : {2, 4})
    if (nrhs >= nr) nrs.push_back(nr);
  float best = 1e30f;
  DslashConfig best_c = def;
  std::vector<std::pair<DslashConfig, float>> timed;
  for (int nr : nrs) {
    const int max_block = dslash_max_block(prec, nr);
    for (int block = 128; block <= max_block; block += 128) {
      const float ms = time_launches(kb, prec, recon, nr, mode, block, 5, st, ctx);
      if (ms < 0.f) continue;
      DslashConfig c;
      c.block = block;
      c.nr = nr;
      timed.push_back({c, ms});
      if (ms < best) {
        best = ms;
        best_c = c;
      }
    }
  }
  // The CG's reducing kernels run in a chain of dependent launches (each
  // waits for a finish kernel), where a launch cannot overlap the tail of
  // the previous one as back-to-back launches of one kernel do: there the
  // smallest block within 3 % of the best isolated time wins (20^3 x 64
  // solve, one box: 128/128 threads 43.5 ms, the isolated pick 256/128
  // 44.0 ms, 512/384 46.1 ms).  64-thread blocks are not candidates: forced,
  // they gave 42.7 against 43.1 ms on one box, but as the tuner's pick the
  // 20^3 x 64 solves lost 3 % (FP32) and 10 % (16-bit) on another.
  if (mode != MODE_PLAIN)
    for (const auto &ct : timed)
      if (ct.first.nr == best_c.nr && ct.first.block < best_c.block && ct.second <= 1.03f * best)
        best_c = ct.first;
  t->cache[key] = best_c;
  tuner_save(t);
  return best_c;
}

}  // namespace sq

using namespace sq;

extern "C" int sq_time_dslash(sq_ctx *ctx, int gauge_id, int prec, int long_recon, int nrhs,
                              int mode, int reps, void *stream, float *us_per_launch) {
  if (!ctx || !us_per_launch || prec < 0 || prec > 2 || reps < 1) return SQ_ERR_ARG;
  if (long_recon != 18 && long_recon != 12) return SQ_ERR_ARG;
  if (nrhs < 1 || nrhs > 64) return SQ_ERR_ARG;
  if (mode != MODE_PLAIN && mode != MODE_MDAGM && mode != MODE_NORM && mode != MODE_UPDATE)
    return SQ_ERR_ARG;
  GaugeField *gf = ctx->gauge(gauge_id);
  if (!gf) return SQ_ERR_NOTFOUND;
  if (!gf->has(prec, long_recon)) return SQ_ERR_UNSUPPORTED;
  SQ_CUDA_TRY(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  const DslashConfig cfg = tuned_dslash(ctx, *gf, prec, long_recon, nrhs, mode, st);
  KernelBench kb;
  if (!kb.setup(*gf, prec, long_recon, nrhs, mode, st)) return SQ_ERR_OOM;
  for (int k = 0; k < 4; ++k)  // warm-up
    if (launch_dslash(prec, long_recon, cfg.nr, mode, prec, kb.a, cfg.block, st)) return SQ_ERR_ARG;
  ctx->launches += 4;
  const float ms = time_launches(kb, prec, long_recon, cfg.nr, mode, cfg.block, reps, st, ctx);
  if (ms < 0.f) return SQ_ERR_CUDA;
  *us_per_launch = ms * 1e3f;
  return SQ_OK;
}
