// Host side of the C ABI declared in include/mls.h: argument validation,
// workspace planning, TMA tensor-map encoding and the launch sequences of the
// forward and backward passes.  Nothing here allocates device memory.
#include <cudaTypedefs.h>

#include <climits>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "mls.h"
#include "mls_kernels.h"

namespace mls {
namespace {

__device__ int g_status;  // MLS_STATUS_* bits raised by the kernels

constexpr int kMaxDevices = 64;

struct DeviceState {
  bool ready = false;
  int err = 0;
  int sms = 0;
  int gemm_pairs = 0;  // co-resident CTA pairs of the GEMM kernel
  int head_pairs = 0;  // co-resident CTA pairs of the head kernels
  int* status = nullptr;
};

std::mutex g_mu;
DeviceState g_dev[kMaxDevices];

// With MLS_DEBUG set in the environment, failures are described on stderr.
int fail(int code, const char* what, cudaError_t e = cudaSuccess) {
  static const bool verbose = std::getenv("MLS_DEBUG") != nullptr;
  if (verbose)
    std::fprintf(stderr, "[mls] %s failed: %s%s%s\n", what, e != cudaSuccess ? cudaGetErrorName(e) : "",
                 e != cudaSuccess ? " " : "", e != cudaSuccess ? cudaGetErrorString(e) : "");
  return code;
}
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

// Checks the current device once and prepares the kernels for it.
int device_state(DeviceState** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MLS_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return MLS_ERR_DEVICE;
  std::lock_guard<std::mutex> lk(g_mu);
  DeviceState& s = g_dev[dev];
  if (!s.ready) {
    s.ready = true;
    int major = 0, minor = 0;
    cudaError_t e;
    if ((e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&s.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "device query", e);
    } else if (major != 10 || minor != 3) {
      s.err = fail(MLS_ERR_DEVICE, "device check (need compute capability 10.3)");
    } else if ((e = cudaGetSymbolAddress(reinterpret_cast<void**>(&s.status), g_status)) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "cudaGetSymbolAddress(status)", e);
    } else if ((e = setup_head_kernels()) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "head kernel attributes", e);
    } else if ((e = setup_gemm_kernels()) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "gemm kernel attributes", e);
    } else if ((e = setup_eval_kernels()) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "eval kernel attributes", e);
    } else if ((e = setup_spec_kernels()) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "spec kernel attributes", e);
    } else if ((e = setup_logits_kernels()) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "logits kernel attributes", e);
    } else if ((e = setup_junction_kernels()) != cudaSuccess) {
      s.err = fail(MLS_ERR_CUDA, "junction kernel attributes", e);
    } else if ((s.gemm_pairs = gemm_max_active_pairs()) <= 0) {
      s.err = fail(MLS_ERR_CUDA, "gemm cluster occupancy");
    } else if ((s.head_pairs = head_max_active_pairs()) <= 0) {
      s.err = fail(MLS_ERR_CUDA, "head cluster occupancy");
    } else if (!g_encode) {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult q;
      if ((e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                cudaEnableDefault, &q)) != cudaSuccess ||
          q != cudaDriverEntryPointSuccess || !fn) {
        s.err = fail(MLS_ERR_CUDA, "cuTensorMapEncodeTiled entry point", e);
      } else {
        g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
      }
    }
  }
  *out = &s;
  return s.err;
}

// Co-resident CTA pairs of the head and GEMM kernels on the current device, for
// sizing a plan without launching (76 on a GB300 when no device can be queried).
void current_pairs(int& head, int& gemm) {
  DeviceState* dev = nullptr;
  head = gemm = 76;
  if (device_state(&dev) == MLS_OK && dev->head_pairs > 0) {
    head = dev->head_pairs;
    gemm = dev->gemm_pairs;
    return;
  }
  cudaGetLastError();
}

// ------------------------------------------------------------------ planning
constexpr size_t kAlign = 256;
size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }
long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }

struct Plan {
  int elt = 2;
  int ntt = 0, nvt = 0;
  int band = 1;      // token tiles per band of the forward and evaluation launch order
  int band_bwd = 1;  // the same for the backward head kernel
  // forward
  TileSplit split = {};      // forward
  int nparts = 0, merge_blocks = 0, eval_merge_blocks = 0;
  size_t off_part = 0, off_bsum = 0, off_bcnt = 0, fwd_bytes = 0;
  // backward
  long long group = 0, ngroups = 0;
  size_t off_invn = 0, off_G = 0, off_split = 0, bwd_bytes = 0;
  // pairwise evaluation
  TileSplit eval_split = {};
  int eval_nparts = 0;
  size_t off_epart = 0, off_eacc = 0, off_ecnt = 0, eval_bytes = 0;
  size_t total = 0;
};

// CTA pairs per token tile (vocabulary splits).  Each pair of a head kernel
// walks ceil(tiles / S) vocabulary tiles and `pairs` pairs are resident at a
// time, so the kernel lasts about waves * (tiles per pair + a fixed per-pair
// cost); S minimises that.
// cta_cost: what one CTA pair costs beyond its tiles, in vocabulary tiles
// (prologue, pipeline fill and drain, the exposed epilogue of its last tile).
constexpr double kHeadCtaCost = 0.25;
// The evaluation kernel's last tile exposes its whole epilogue (every pass) and
// the partial-state write.  Measured at the 3-level suite (T = 8192, 197
// vocabulary tiles): 33 splits (the head kernels' choice) 3.39 ms per call,
// 7 splits 3.24 ms, which puts its per-pair cost near 1.2 tiles.
constexpr double kEvalCtaCost = 1.25;
// Token tiles per band of the head kernels' launch order (band_unit): the
// pairs resident at one time re-read the hidden states of every sub-model for
// the band's tokens once per vocabulary tile, so a band's H is kept within a
// share of L2 that stays resident while W streams past it.  Fewer token tiles
// per band mean more passes over W (one per band); the bands are made equal.
// The backward streams its dL/dz stores through L2 as well, so its band's H
// gets a smaller share (measured on the 3-level suite: 48 MB gave the
// forward its least traffic at no cost in time; 32 MB, with the stores
// marked evict-first, cut the backward's DRAM reads from 4.8 to 3.3 GB).
constexpr long long kBandBytesFwd = 48ll << 20;
constexpr long long kBandBytesBwd = 32ll << 20;
int choose_band(int ntt, long long h_bytes_per_tile, long long budget) {
  if (ntt < 1) return 1;
  long long band = budget / (h_bytes_per_tile > 0 ? h_bytes_per_tile : 1);
  if (band < 1) band = 1;
  if (band >= ntt) return ntt;
  const long long nbands = (ntt + band - 1) / band;
  return static_cast<int>((ntt + nbands - 1) / nbands);
}

// The dH problems of a backward GEMM launch run in wide units
// (GemmProblem::wide) when each of them has a reduction of at least this many
// k-blocks of 128 bytes, an even number of column tiles (no single-tile
// units, which would only lose the epilogue overlap) and nothing to
// accumulate (the first vocabulary group): a wide unit's two accumulators are
// drained while no MMA runs, which costs a share inversely proportional to
// the reduction and doubles when dH is read back.  Measured on one GB300 in a
// seconds-long loop under the power cap: the 3-level suite at T = 8192 (786
// k-blocks) gains 2.6% on the GEMM, while the paper's 3B suite (9 and 17
// column tiles) lost 5% and the 4-level suite (504 k-blocks, four groups)
// 2% when they ran wide.
constexpr long long kWideMinBlocks = 512;

// Cost of a unit beyond its k-blocks, in k-blocks: draining its 256x256 accumulator.
constexpr long long kDrainBlocks = 8;

// Short units that a pair left one long unit short takes first (two-class schedule).
int catchup_units(int pairs, int n_long, long long cost_long, int n_short, long long cost_short) {
  const int r = n_long % pairs;
  if (r == 0) return 0;
  const int c = static_cast<int>((cost_long + cost_short / 2) / cost_short);
  const int most = n_short / (pairs - r);
  return c < most ? c : most;
}

// Two-class schedule of a persistent GEMM launch whose first n_long tiles take
// cost_long and the other n_short cost_short (K-blocks plus a per-tile
// allowance): see GemmParams.  The pairs that get one long tile fewer take
// `catchup` short tiles first, about the cost of that long tile.
void schedule_two_class(GemmParams& g, int pairs, int n_long, long long cost_long, int n_short,
                        long long cost_short) {
  g.two_class = 0;
  if (pairs < 1 || n_long <= 0 || n_short <= 0) return;
  g.two_class = 1;
  g.n_long = n_long;
  g.catchup = catchup_units(pairs, n_long, cost_long, n_short, cost_short);
}

// Time of that schedule in k-blocks: the busiest pair.
long long two_class_time(int pairs, int n_long, long long cost_long, int n_short, long long cost_short) {
  const int r = n_long % pairs, q = n_long / pairs;
  const int c = n_short > 0 ? catchup_units(pairs, n_long, cost_long, n_short, cost_short) : 0;
  const int rest = n_short - c * (pairs - r);
  auto share = [&](int first) { return static_cast<long long>(rest > first ? (rest - first + pairs - 1) / pairs : 0); };
  const long long extra = r > 0 ? (q + 1) * cost_long + share(0) * cost_short : 0;
  const long long plain = q * cost_long + (c + share(r)) * cost_short;
  return extra > plain ? extra : plain;
}

// How one vocabulary group's dW + dH launch is cut: which class has the longer
// reduction, whether dH runs in wide units, and into how many units the long
// reductions are split (GemmProblem::ksplit).
struct GemmCut {
  bool dh_long = true, wide = false;
  int ksplit = 1, kb_split = 0;
  long long cost_long = 0, cost_short = 0;
  long long part_floats = 0;  // workspace of the splits' copies
  bool chained = false;       // launched before its predecessor completes (chain_wait)
};

// With few output tiles the long reductions bound the launch.  Splitting each
// over several units (at least kSplitMinBlocks each) costs one more pass over
// the output per split and a launch to add them up: kSplitLaunch k-blocks (of
// about 0.33 us) and one per kSplitBytes written and read.  A split has to be
// estimated kSplitGain faster, so that large launches stay whole.  Measured,
// launch whole against split with its sum: 300 tokens, d = (96, 400), V = 30000
// in fp32 (6 dH tiles of 938 k-blocks) 261 against 73 us; 100 tokens, d =
// (512, 1024), V = 20000 (6 of 313) 117 against 50 us; 20000 tokens, d =
// (512, 1024), V = 600 (dW, 18 of 313) 117 against 78 us; 256 tokens, d = (128,
// 256), V = 1024 in fp32 (2 of 32): a step of 55.9 against 53.1 us.  Where whole
// reductions would run in wide units: 520 tokens, d = (320, 1008), V = 35000 317
// against 112 us, 2000 tokens, d = (512, 1024), V = 50304 504 against 387 us.  At
// the rule's far end, with 60 to 82 MB of copies: 7979 tokens, d = 416, V = 228345
// 2266 against 2120 us; 8088, d = 504, V = 73613 779 against 768; 37116, d = (168,
// 192), V = 49242 2480 against 2469; 7466 in fp32, d = 512, V = 192659 3974 against
// 3944 us.
constexpr int kSplitMinBlocks = 12, kSplitMost = 32;
constexpr long long kSplitLaunch = 8, kSplitBytes = 1700000;
constexpr double kSplitGain = 0.95;
// A launch estimated shorter than this (about 170 us) starts chained to its
// predecessor, which saves some 3 us of launch latency.  A long one is launched
// normally: chained, its CTAs take SMs in the order in which the head kernel's
// last ones leave them (8192 tokens of the 3-level suite 0.4 to 1.2% slower).
constexpr double kChainBlocks = 512;

GemmCut cut_gemm(int M, const int32_t* d, long long T, long long gc, bool first, int KE, int pairs) {
  GemmCut c;
  c.dh_long = gc >= T;
  int t_dh = 0, t_dw = 0;  // 256 x kGemmBN output tiles
  long long sum_d = 0;
  c.wide = first && ceil_div(gc, KE) >= kWideMinBlocks;
  for (int m = 0; m < M; ++m) {
    const int tn = static_cast<int>(ceil_div(d[m], kGemmBN));
    t_dh += static_cast<int>(ceil_div(T, 2 * kGemmBM)) * tn;
    t_dw += static_cast<int>(ceil_div(gc, 2 * kGemmBM)) * tn;
    sum_d += d[m];
    c.wide = c.wide && tn % 2 == 0;
  }
  const long long kb_dh = ceil_div(gc, KE), kb_dw = ceil_div(T, KE);
  const long long kb_long = c.dh_long ? kb_dh : kb_dw;
  const int n_long = c.dh_long ? t_dh : t_dw, n_short = c.dh_long ? t_dw : t_dh;
  c.cost_short = (c.dh_long ? kb_dw : kb_dh) + kDrainBlocks;
  c.cost_long = kb_long + kDrainBlocks;
  const int w_dh = c.wide ? 2 : 1;  // dH units of two tiles
  if (!c.dh_long) c.cost_short *= w_dh;
  else c.cost_long *= w_dh;
  const long long whole =
      two_class_time(pairs, c.dh_long ? n_long / w_dh : n_long, c.cost_long,
                     c.dh_long ? n_short : n_short / w_dh, c.cost_short);
  const long long rows = c.dh_long ? T : gc, out_bytes = 4 * rows * sum_d;
  double best = kSplitGain * static_cast<double>(whole), best_time = static_cast<double>(whole);
  for (int s = 2; s <= kSplitMost; ++s) {
    const long long per = ceil_div(kb_long, s);
    if (per < kSplitMinBlocks) break;
    if ((s - 1) * per >= kb_long) continue;
    const long long cost_short = (c.dh_long ? kb_dw : kb_dh) + kDrainBlocks;
    const long long t = two_class_time(pairs, n_long * s, per + kDrainBlocks, n_short, cost_short) +
                        kSplitLaunch + (s + 1) * out_bytes / kSplitBytes;
    if (static_cast<double>(t) < best) {
      best = best_time = static_cast<double>(t);
      c.ksplit = s;
      c.kb_split = static_cast<int>(per);
    }
  }
  if (c.ksplit > 1) {
    c.wide = false;
    c.cost_long = c.kb_split + kDrainBlocks;
    c.cost_short = (c.dh_long ? kb_dw : kb_dh) + kDrainBlocks;
    c.part_floats = c.ksplit * rows * sum_d;
  }
  c.chained = best_time < kChainBlocks;
  return c;
}

// Leaving some tiles to extra pairs (TileSplit) has to be estimated this much
// faster.  Measured, all tiles in one wave of regular pairs against this: head
// forward and backward of 1531 tokens, d = (520, 1032, 2056), V = 32003 (6 token
// tiles x 12 splits of 10 or 11 tiles; 10 each and 12 runs of 3) 300 + 333 -> 285
// + 318 us; evaluation of 2999 tokens, d = (1024, 3072), V = 49152 (12 x 6 of 32;
// 31 each and 12 runs of 6) 765 -> 738 us.
constexpr double kExtraGain = 0.985;
TileSplit choose_splits(int ntt, long long tiles, int pairs, int band, double cta_cost = kHeadCtaCost) {
  TileSplit sp = {};
  sp.S = 1;
  sp.band = band;
  sp.ntt = ntt;
  sp.main_end = sp.end = static_cast<int>(tiles);
  if (ntt < 1) ntt = 1;
  if (tiles < 1) return sp;
  long long best = 1;
  double best_cost = 1e300;
  // of the S with the same tiles per pair, the smallest (fewest waves); trying every
  // S cost a step of the 3-level suite some 10 us on the host
  for (long long S = 1, per = tiles; S <= tiles && S <= 512;
       S = per > 1 ? (tiles + per - 2) / (per - 1) : tiles + 1) {
    per = (tiles + S - 1) / S;
    const long long waves = (ntt * S + pairs - 1) / pairs;
    const double cost = waves * (per + cta_cost);
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = S;
    }
  }
  sp.S = static_cast<int>(best);
  if (band < ntt) return sp;  // several bands: pairs of one band share its hidden states in L2

  // One wave of ntt x S pairs leaves `spare` pairs' SMs idle and, where S does not
  // divide the tiles, makes some pairs take one tile more.  So the regular pairs
  // may stop after `cap` tiles each, and the rest runs as short extra pairs on
  // the spare SMs (TileSplit).
  best_cost *= kExtraGain;
  for (long long S = pairs / ntt; S >= 1 && S >= pairs / ntt - 1; --S) {
    const long long spare = pairs - ntt * S;
    if (spare < 1 || S > tiles) continue;
    const long long most = (tiles - 1) / S;  // tiles per pair that leave some over
    for (long long cap = most; cap >= 1 && cap >= most - 3; --cap) {
      const long long left = tiles - S * cap;
      for (long long E = 1; E <= 8 && E <= left; ++E) {
        const long long run = (left + E - 1) / E;
        if ((E - 1) * run >= left) continue;
        const double rounds = static_cast<double>((ntt * E + spare - 1) / spare) * (run + cta_cost);
        const double cost = cap + cta_cost > rounds ? cap + cta_cost : rounds;
        if (cost < best_cost - 1e-9) {
          best_cost = cost;
          sp.S = static_cast<int>(S);
          sp.main_end = static_cast<int>(S * cap);
          sp.extra = static_cast<int>(E);
          sp.run = static_cast<int>(run);
        }
      }
    }
  }
  return sp;
}

int validate(const mls_problem* p) {
  if (!p || p->M < 1 || p->M > MLS_MAX_MODELS || p->T < 0 || p->V < 1 || p->V > INT_MAX ||
      p->T > INT_MAX || !p->d)
    return MLS_ERR_ARG;
  if (p->teacher < 0 || p->teacher >= p->M) return MLS_ERR_ARG;
  if (!(p->tau > 0.f) || !std::isfinite(p->tau)) return MLS_ERR_ARG;
  if (!(p->alpha >= 0.f && p->alpha <= 1.f)) return MLS_ERR_ARG;
  if (p->in_dtype != MLS_BF16 && p->in_dtype != MLS_FP32) return MLS_ERR_ARG;
  if (p->vocab_group < 0 || p->vocab_group % kHeadBN != 0) return MLS_ERR_ARG;
  const int elt = p->in_dtype == MLS_BF16 ? 2 : 4;
  for (int m = 0; m < p->M; ++m) {
    if (p->d[m] < 1) return MLS_ERR_ARG;
    if ((static_cast<long long>(p->d[m]) * elt) % 16 != 0) return MLS_ERR_UNSUPPORTED;
  }
  if (p->w)
    for (int m = 0; m < p->M; ++m)
      if (!std::isfinite(p->w[m])) return MLS_ERR_ARG;
  return MLS_OK;
}

Plan make_plan(const mls_problem* p, int pairs, int gemm_pairs) {
  Plan pl;
  pl.elt = p->in_dtype == MLS_BF16 ? 2 : 4;
  const long long T = p->T, V = p->V, M = p->M;
  pl.ntt = static_cast<int>(ceil_div(T, 2 * kHeadBM));  // token tiles of a CTA pair
  pl.nvt = static_cast<int>(ceil_div(V, kHeadBN));
  long long sum_d = 0;
  for (int m = 0; m < p->M; ++m) sum_d += p->d[m];
  pl.band = choose_band(pl.ntt, 2LL * kHeadBM * sum_d * pl.elt, kBandBytesFwd);
  pl.band_bwd = choose_band(pl.ntt, 2LL * kHeadBM * sum_d * pl.elt, kBandBytesBwd);
  pl.split = choose_splits(pl.ntt, pl.nvt, pairs, pl.band);
  pl.nparts = pl.split.S + pl.split.extra;
  pl.merge_blocks = static_cast<int>(ceil_div(T, merge_tokens_per_block(pl.nparts)));
  pl.eval_merge_blocks = static_cast<int>(ceil_div(T, kEvalMergeTokens));
  size_t o = 0;
  pl.off_part = o;
  o = align_up(o + sizeof(float) * static_cast<size_t>(pl.nparts) * kPartFields * M * T);
  pl.off_bsum = o;
  o = align_up(o + sizeof(double) * static_cast<size_t>(pl.merge_blocks + 1));
  pl.off_bcnt = o;
  o = align_up(o + sizeof(long long) * static_cast<size_t>(pl.merge_blocks + 1));
  pl.fwd_bytes = o;

  // Backward vocabulary groups: the bf16 (fp32) gradient of the logits of one
  // group of columns for every sub-model stays within ~4 GiB unless the caller
  // chose the group width.
  const long long vpad = static_cast<long long>(pl.nvt) * kHeadBN;
  long long gmax = p->vocab_group;
  if (gmax == 0) {
    const long long budget = 4LL << 30;
    const long long per_col = M * (T > 0 ? T : 1) * pl.elt;
    gmax = budget / per_col / kHeadBN * kHeadBN;
    if (gmax < 2048) gmax = 2048;
  }
  if (gmax > vpad) gmax = vpad;
  pl.ngroups = ceil_div(vpad, gmax);
  pl.group = ceil_div(ceil_div(vpad, pl.ngroups), kHeadBN) * kHeadBN;
  pl.ngroups = ceil_div(vpad, pl.group);
  o = 0;
  pl.off_invn = o;
  o = align_up(o + sizeof(float));
  pl.off_G = o;
  o = align_up(o + static_cast<size_t>(pl.elt) * M * T * pl.group);
  // copies of a split reduction's output: the full groups' or the last one's
  pl.off_split = o;
  if (T > 0) {
    const long long last = V - (pl.ngroups - 1) * pl.group;
    long long most = 0;
    for (const long long g : {0LL, 1LL, pl.ngroups - 1}) {
      if (g >= pl.ngroups) continue;
      const GemmCut c = cut_gemm(p->M, p->d, T, g + 1 < pl.ngroups ? pl.group : last, g == 0,
                                 128 / pl.elt, gemm_pairs);
      if (c.part_floats > most) most = c.part_floats;
    }
    o = align_up(o + sizeof(float) * static_cast<size_t>(most));
  }
  pl.bwd_bytes = o;

  pl.eval_split = choose_splits(pl.ntt, ceil_div(V, eval_tile_cols(p->M)), pairs, pl.band, kEvalCtaCost);
  pl.eval_nparts = pl.eval_split.S + pl.eval_split.extra;
  o = 0;
  pl.off_epart = o;
  o = align_up(o + sizeof(float) * static_cast<size_t>(pl.eval_nparts) * kEvalFields * T);
  pl.off_eacc = o;
  o = align_up(o + sizeof(double) * 2 * kMaxModels * kMaxModels * static_cast<size_t>(pl.eval_merge_blocks + 1));
  pl.off_ecnt = o;
  o = align_up(o + sizeof(long long) * static_cast<size_t>(pl.eval_merge_blocks + 1));
  pl.eval_bytes = o;

  pl.total = pl.fwd_bytes > pl.bwd_bytes ? pl.fwd_bytes : pl.bwd_bytes;
  if (pl.eval_bytes > pl.total) pl.total = pl.eval_bytes;
  return pl;
}

// One vocabulary group of the backward: its columns and how its two launches are cut.
struct GroupPlan {
  long long c0 = 0, cols = 0;
  TileSplit split = {};  // the head kernel's vocabulary tiles
  GemmCut cut;
};

GroupPlan plan_group(const mls_problem* p, const Plan& pl, long long g, int pairs, int gemm_pairs) {
  GroupPlan gp;
  gp.c0 = g * pl.group;
  gp.cols = (p->V - gp.c0 < pl.group) ? p->V - gp.c0 : pl.group;
  const int vt0 = static_cast<int>(gp.c0 / kHeadBN);
  gp.split = choose_splits(pl.ntt, ceil_div(gp.c0 + gp.cols, kHeadBN) - vt0, pairs, pl.band_bwd);
  gp.split.begin += vt0;
  gp.split.main_end += vt0;
  gp.split.end += vt0;
  gp.cut = cut_gemm(p->M, p->d, p->T, gp.cols, g == 0, 128 / pl.elt, gemm_pairs);
  return gp;
}

bool aligned16(const void* ptr) { return (reinterpret_cast<uintptr_t>(ptr) & 15u) == 0; }

// 2-D row-major tensor [rows, cols] of `elt`-byte elements (128-byte swizzle
// unless told otherwise).
int encode(CUtensorMap* map, const void* ptr, int elt, long long cols, long long rows,
           long long pitch_elems, int box_cols, int box_rows,
           CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(pitch_elems) * elt};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(box_cols), static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = g_encode(
      map, elt == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
      const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
      swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    char what[160];
    std::snprintf(what, sizeof what, "cuTensorMapEncodeTiled (CUresult %d, %lld x %lld, box %d x %d)",
                  static_cast<int>(r), cols, rows, box_cols, box_rows);
    return fail(MLS_ERR_CUDA, what);
  }
  return MLS_OK;
}

// Row-major fp32 output [copies, rows, cols] of dense rows, `stride` floats
// between copies, as boxes of 32 x 32 for TMA stores.
int encode_out(CUtensorMap* map, float* ptr, long long cols, long long rows, int copies,
               long long stride) {
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows),
                              static_cast<cuuint64_t>(copies)};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(cols) * 4, static_cast<cuuint64_t>(stride) * 4};
  const cuuint32_t box[3] = {32, 32, 1}, estr[3] = {1, 1, 1};
  const CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, ptr, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MLS_OK : fail(MLS_ERR_CUDA, "cuTensorMapEncodeTiled (output)");
}

void fill_head_common(HeadParams& hp, const mls_problem* p, const Plan& pl, const int* y,
                      int* status) {
  const int KE = 128 / pl.elt;
  hp.M = p->M;
  hp.order[0] = p->teacher;
  for (int m = 0, j = 1; m < p->M; ++m)
    if (m != p->teacher) hp.order[j++] = m;
  for (int m = 0; m < p->M; ++m) hp.nk[m] = static_cast<int>(ceil_div(p->d[m], KE));
  hp.T = p->T;
  hp.V = p->V;
  hp.L1 = 1.4426950408889634f;
  hp.Ltau = static_cast<float>(1.4426950408889634 / static_cast<double>(p->tau));
  hp.y = y;
  hp.status = status;
  // Failure-detection test hook: with MLS_TEST_STALL_FIRST_STAGE set, the first
  // CTA pair of a head kernel skips its first stage so that a bounded pipeline
  // wait runs out and the call reports MLS_STATUS_TIMEOUT.
  hp.test_stall = std::getenv("MLS_TEST_STALL_FIRST_STAGE") != nullptr ? 1 : 0;
}

int encode_head_maps(HeadParams& hp, const mls_problem* p, const Plan& pl, const void* const* H,
                     const void* const* W) {
  const int KE = 128 / pl.elt;
  for (int m = 0; m < p->M; ++m) {
    if (encode(&hp.mapH[m], H[m], pl.elt, p->d[m], p->T, p->d[m], KE, kHeadBM) ||
        encode(&hp.mapW[m], W[m], pl.elt, p->d[m], p->V, p->d[m], KE, kHeadBHalf))
      return MLS_ERR_CUDA;
  }
  return MLS_OK;
}

int check_ws(const Plan& pl, void* ws, size_t ws_bytes, size_t need) {
  if (need == 0) return MLS_OK;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & (kAlign - 1)) != 0 || ws_bytes < need)
    return MLS_ERR_WORKSPACE;
  return MLS_OK;
}

int launch_ok(cudaError_t e) { return e == cudaSuccess ? MLS_OK : fail(MLS_ERR_CUDA, "launch", e); }

// ------------------------------------------------------------------ kernel timing
struct ProfRec {
  const char* name;
  cudaEvent_t a, b;
};
std::mutex g_prof_mu;
bool g_prof_on = false;
std::vector<ProfRec> g_prof;
std::vector<cudaEvent_t> g_event_pool;

cudaEvent_t pool_event() {
  if (!g_event_pool.empty()) {
    cudaEvent_t e = g_event_pool.back();
    g_event_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
  return e;
}

// Runs `launch` (which returns a cudaError_t), bracketed by events when timing is on.
template <class F>
int timed(const char* name, cudaStream_t s, F&& launch) {
  if (!g_prof_on) return launch_ok(launch());
  std::lock_guard<std::mutex> lk(g_prof_mu);
  cudaEvent_t a = pool_event(), b = pool_event();
  if (a) cudaEventRecord(a, s);
  const int rc = launch_ok(launch());
  if (a && b) {
    cudaEventRecord(b, s);
    g_prof.push_back({name, a, b});
  }
  return rc;
}

}  // namespace
}  // namespace mls

using namespace mls;

extern "C" size_t mls_workspace_size(const mls_problem* p) {
  if (validate(p) != MLS_OK) return 0;
  int head = 0, gemm = 0;
  current_pairs(head, gemm);
  return make_plan(p, head, gemm).total;
}

// How a problem's launches are cut, for tests that have to know which path a shape
// takes (not part of mls.h): out[0..5] = backward groups, partial-state slots of the
// forward and of the evaluation, extra pairs per token tile of both, bytes of the
// copies of split reductions; then per group of the backward the extra pairs, whether
// dH runs in wide units, and the units that share a long reduction.  Writes at most n
// values, returns how many there are or a negative MLS_ERR_* code.
extern "C" int mls_test_plan(const mls_problem* p, int64_t* out, int n) {
  const int rc = validate(p);
  if (rc) return rc;
  int head = 0, gemm = 0;
  current_pairs(head, gemm);
  const Plan pl = make_plan(p, head, gemm);
  std::vector<int64_t> v = {pl.ngroups,          pl.nparts, pl.eval_nparts, pl.split.extra,
                            pl.eval_split.extra, static_cast<int64_t>(pl.bwd_bytes - pl.off_split)};
  for (long long g = 0; g < pl.ngroups && static_cast<int>(v.size()) < n; ++g) {
    const GroupPlan gp = plan_group(p, pl, g, head, gemm);
    v.insert(v.end(), {gp.split.extra, gp.cut.wide ? 1 : 0, gp.cut.ksplit});
  }
  for (size_t i = 0; i < v.size() && static_cast<int>(i) < n; ++i) out[i] = v[i];
  return static_cast<int>(6 + 3 * pl.ngroups);
}

extern "C" int mls_head_loss_fwd(const mls_problem* p, const void* const* H, const void* const* W,
                                 const int32_t* targets, float* loss, float* tok_loss,
                                 float* tok_diag, int32_t* argmax, float* stats, void* ws,
                                 size_t ws_bytes, mls_stream_t stream) {
  int rc = validate(p);
  if (rc) return rc;
  if (!H || !W || !loss || (p->T > 0 && (!targets || !tok_loss || !stats))) return MLS_ERR_ARG;
  for (int m = 0; m < p->M; ++m) {
    if ((p->T > 0 && !H[m]) || !W[m]) return MLS_ERR_ARG;  // no rows to read when T = 0
    if (!aligned16(H[m]) || !aligned16(W[m])) return MLS_ERR_ALIGN;
  }
  DeviceState* dev = nullptr;
  if ((rc = device_state(&dev))) return rc;
  const Plan pl = make_plan(p, dev->head_pairs, dev->gemm_pairs);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (p->T == 0) return launch_ok(cudaMemsetAsync(loss, 0, sizeof(float), s));
  if ((rc = check_ws(pl, ws, ws_bytes, pl.total))) return rc;
  char* wsb = static_cast<char*>(ws);

  HeadParams hp;
  std::memset(&hp, 0, sizeof hp);
  fill_head_common(hp, p, pl, targets, dev->status);
  if ((rc = encode_head_maps(hp, p, pl, H, W))) return rc;
  hp.split = pl.split;
  hp.part = reinterpret_cast<float*>(wsb + pl.off_part);
  if ((rc = timed("head_fwd", s, [&] { return launch_head_fwd(hp, pl.elt == 4, p->tau == 1.0f, s); }))) return rc;

  MergeParams mp;
  std::memset(&mp, 0, sizeof mp);
  mp.part = hp.part;
  mp.nparts = pl.nparts;
  mp.M = p->M;
  mp.teacher = p->teacher;
  mp.T = p->T;
  mp.V = p->V;
  mp.L1 = hp.L1;
  mp.Ltau = hp.Ltau;
  mp.tau = p->tau;
  mp.alpha = p->alpha;
  for (int m = 0; m < p->M; ++m) mp.w[m] = p->w ? p->w[m] : 1.0f;
  mp.y = targets;
  mp.tok_loss = tok_loss;
  mp.tok_diag = tok_diag;
  mp.argmax = argmax;
  mp.stats = stats;
  mp.block_sum = reinterpret_cast<double*>(wsb + pl.off_bsum);
  mp.block_cnt = reinterpret_cast<long long*>(wsb + pl.off_bcnt);
  mp.status = dev->status;
  if ((rc = timed("merge", s, [&] { return launch_merge(mp, pl.merge_blocks, s); }))) return rc;
  return timed("final", s, [&] { return launch_final(mp.block_sum, mp.block_cnt, pl.merge_blocks, loss, s); });
}

extern "C" int mls_head_loss_bwd(const mls_problem* p, const void* const* H, const void* const* W,
                                 const int32_t* targets, const float* stats, float grad_scale,
                                 float* const* dH, float* const* dW, void* ws, size_t ws_bytes,
                                 mls_stream_t stream) {
  int rc = validate(p);
  if (rc) return rc;
  if (!H || !W || !dH || !dW || (p->T > 0 && (!targets || !stats))) return MLS_ERR_ARG;
  if (!std::isfinite(grad_scale)) return MLS_ERR_ARG;
  for (int m = 0; m < p->M; ++m) {
    if ((p->T > 0 && (!H[m] || !dH[m])) || !W[m] || !dW[m]) return MLS_ERR_ARG;
    if (!aligned16(H[m]) || !aligned16(W[m]) || !aligned16(dW[m]) || !aligned16(dH[m]))
      return MLS_ERR_ALIGN;
  }
  DeviceState* dev = nullptr;
  if ((rc = device_state(&dev))) return rc;
  const Plan pl = make_plan(p, dev->head_pairs, dev->gemm_pairs);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (p->T == 0) {
    for (int m = 0; m < p->M; ++m)
      if ((rc = launch_ok(cudaMemsetAsync(dW[m], 0, sizeof(float) * p->V * p->d[m], s)))) return rc;
    return MLS_OK;
  }
  if ((rc = check_ws(pl, ws, ws_bytes, pl.total))) return rc;
  char* wsb = static_cast<char*>(ws);
  const bool tf32 = pl.elt == 4;
  const int KE = 128 / pl.elt;
  float* inv_n = reinterpret_cast<float*>(wsb + pl.off_invn);
  void* G = wsb + pl.off_G;

  if ((rc = timed("count", s, [&] { return launch_count(targets, p->T, p->V, inv_n, dev->status, s); }))) return rc;

  HeadParams hp;
  std::memset(&hp, 0, sizeof hp);
  fill_head_common(hp, p, pl, targets, dev->status);
  if ((rc = encode_head_maps(hp, p, pl, H, W))) return rc;
  hp.stats = stats;
  hp.inv_n = inv_n;
  for (int m = 0; m < p->M; ++m) hp.coef[m] = grad_scale * (p->w ? p->w[m] : 1.0f);
  hp.one_minus_alpha = 1.0f - p->alpha;
  hp.alpha_over_tau = p->alpha / p->tau;

  // dW reads A = G viewed M-major and B = H viewed N-major, dH reads A = G
  // K-major and B = W viewed N-major, all in place.
  GemmParams gw, gh, gb;
  std::memset(&gw, 0, sizeof gw);
  std::memset(&gh, 0, sizeof gh);
  const CUtensorMapSwizzle mn_swizzle =
      tf32 ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B;
  for (int m = 0; m < p->M; ++m) {
    const void* Gm = static_cast<const char*>(G) + static_cast<size_t>(pl.elt) * p->T * pl.group * m;
    // the backward head kernel's TMA stores of dL/dz
    if (encode(&hp.mapG[m], Gm, pl.elt, pl.group, p->T, pl.group, KE / 2, 32, CU_TENSOR_MAP_SWIZZLE_64B))
      return MLS_ERR_CUDA;
    if (encode(&gh.mapA[m], Gm, pl.elt, pl.group, p->T, pl.group, KE, kGemmBM) ||
        encode(&gw.mapA[m], Gm, pl.elt, pl.group, p->T, pl.group, KE, KE, mn_swizzle) ||
        encode(&gw.mapB[m], H[m], pl.elt, p->d[m], p->T, p->d[m], KE, KE, mn_swizzle) ||
        encode(&gh.mapB[m], W[m], pl.elt, p->d[m], p->V, p->d[m], KE, KE, mn_swizzle))
      return MLS_ERR_CUDA;
  }

  for (long long g = 0; g < pl.ngroups; ++g) {
    const GroupPlan gp = plan_group(p, pl, g, dev->head_pairs, dev->gemm_pairs);
    const long long c0 = gp.c0, gc = gp.cols;
    hp.split = gp.split;
    hp.g_col0 = c0;
    if ((rc = timed("head_bwd", s, [&] { return launch_head_bwd(hp, tf32, p->tau == 1.0f, s); }))) return rc;
    // dW and dH of every sub-model in one persistent launch, the class with the
    // longer reduction (dH: the group's columns, dW: T) first.
    const int pairs = dev->gemm_pairs, M = p->M;
    const GemmCut& cut = gp.cut;
    float* split_ws = reinterpret_cast<float*>(wsb + pl.off_split);
    SplitSumParams sum;
    std::memset(&sum, 0, sizeof sum);
    std::memset(&gb, 0, sizeof gb);
    int units = 0, n_long = 0;
    long long split_off = 0;
    for (int i = 0; i < 2 * M; ++i) {
      const int m = i % M;
      const bool is_long = i < M, dh = is_long == cut.dh_long;
      gb.mapA[i] = dh ? gh.mapA[m] : gw.mapA[m];
      gb.mapB[i] = dh ? gh.mapB[m] : gw.mapB[m];
      GemmProblem& q = gb.prob[i];
      q.Mrows = static_cast<int>(dh ? p->T : gc);
      q.Ncols = p->d[m];
      q.K = static_cast<int>(dh ? gc : p->T);
      q.a_map = q.b_map = i;
      q.b_k0 = dh ? static_cast<int>(c0) : 0;
      float* out = dh ? dH[m] : dW[m] + c0 * p->d[m];
      q.accumulate = dh && g > 0 ? 1 : 0;
      q.a_mn = dh ? 0 : 1;
      q.tiles_m = static_cast<int>(ceil_div(q.Mrows, 2 * kGemmBM));
      q.tiles_n = static_cast<int>(ceil_div(p->d[m], kGemmBN));
      q.wide = cut.wide && dh ? 1 : 0;
      q.tile_begin = units;
      units += q.tiles_m * (q.wide ? (q.tiles_n + 1) / 2 : q.tiles_n) * (is_long ? cut.ksplit : 1);
      if (is_long && cut.ksplit > 1) {  // the units write their own sums, added up below
        q.ksplit = cut.ksplit;
        q.kb_split = cut.kb_split;
        sum.out[m] = out;
        sum.n4[m] = static_cast<long long>(q.Mrows) * p->d[m] / 4;
        sum.accumulate = q.accumulate;
        out = split_ws + split_off;
        q.accumulate = 0;
        sum.part[m] = out;
        split_off += static_cast<long long>(q.Mrows) * p->d[m];
      }
      if (encode_out(&gb.mapC[i], out, p->d[m], q.Mrows, q.ksplit > 1 ? q.ksplit : 1,
                     q.ksplit > 1 ? cut.part_floats / cut.ksplit : static_cast<long long>(q.Mrows) * p->d[m]))
        return MLS_ERR_CUDA;
      if (i == M - 1) n_long = units;
    }
    gb.nprob = 2 * M;
    gb.total_tiles = units;
    gb.status = dev->status;
    gb.chained = cut.chained ? 1 : 0;
    // persistent: one CTA pair per resident pair slot, never more pairs than units
    const int grid = 2 * (units < pairs ? units : pairs);
    schedule_two_class(gb, grid / 2, n_long, cut.cost_long, units - n_long, cut.cost_short);
    if ((rc = timed("gemm_bwd", s, [&] { return launch_gemm_mixed(gb, tf32, grid, s); }))) return rc;
    if (cut.ksplit > 1) {
      sum.nprob = M;
      sum.nsplit = cut.ksplit;
      sum.stride = cut.part_floats / cut.ksplit;
      if ((rc = timed("split_sum", s, [&] { return launch_split_sum(sum, s); }))) return rc;
    }
  }
  return MLS_OK;
}

extern "C" int mls_get_status(mls_stream_t stream) {
  DeviceState* dev = nullptr;
  const int rc = device_state(&dev);
  if (rc) return rc;
  if (cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess)
    return MLS_ERR_CUDA;
  int v = 0;
  if (cudaMemcpy(&v, dev->status, sizeof v, cudaMemcpyDeviceToHost) != cudaSuccess)
    return MLS_ERR_CUDA;
  const int zero = 0;
  if (cudaMemcpy(dev->status, &zero, sizeof zero, cudaMemcpyHostToDevice) != cudaSuccess)
    return MLS_ERR_CUDA;
  return v;
}

extern "C" const char* mls_strerror(int code) {
  switch (code) {
    case MLS_OK: return "success";
    case MLS_ERR_ARG: return "invalid argument";
    case MLS_ERR_ALIGN: return "device pointer not 16-byte aligned";
    case MLS_ERR_UNSUPPORTED: return "unsupported shape (row of H/W not a multiple of 16 bytes)";
    case MLS_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case MLS_ERR_CUDA: return "CUDA runtime or launch failure";
    case MLS_ERR_DEVICE: return "current device is not compute capability 10.3";
    case MLS_STATUS_BAD_TARGET: return "a target was >= V (token ignored)";
    case MLS_STATUS_TIMEOUT: return "a pipeline wait timed out; outputs are invalid";
    case MLS_STATUS_BAD_TARGET | MLS_STATUS_TIMEOUT: return "target >= V and a pipeline timeout";
    case MLS_STATUS_CHECK: return "an internal invariant failed (checked build)";
    case MLS_STATUS_DRAIN:
    case MLS_STATUS_TIMEOUT | MLS_STATUS_DRAIN:
      return "a pipeline timeout, and a shutdown wait ran out: the CUDA context is unreliable";
    default:
      return code > 0 && code < 16 ? "several status bits are set (MLS_STATUS_* in mls.h)" : "unknown code";
  }
}

extern "C" int mls_profile_enable(int on) {
  std::lock_guard<std::mutex> lk(g_prof_mu);
  g_prof_on = on != 0;
  for (auto& r : g_prof) {
    g_event_pool.push_back(r.a);
    g_event_pool.push_back(r.b);
  }
  g_prof.clear();
  return MLS_OK;
}

extern "C" int mls_profile_read(mls_kernel_time* out, int n) {
  std::lock_guard<std::mutex> lk(g_prof_mu);
  if (!g_prof.empty() && cudaEventSynchronize(g_prof.back().b) != cudaSuccess) return MLS_ERR_CUDA;
  int k = 0;
  const char* names[32];
  int launches[32];
  double ms[32];
  for (auto& r : g_prof) {
    float t = 0.f;
    cudaEventElapsedTime(&t, r.a, r.b);
    int i = 0;
    while (i < k && std::strcmp(names[i], r.name) != 0) ++i;
    if (i == k && k < 32) {
      names[k] = r.name;
      launches[k] = 0;
      ms[k] = 0.0;
      ++k;
    }
    if (i < 32) {
      launches[i] += 1;
      ms[i] += t;
    }
    g_event_pool.push_back(r.a);
    g_event_pool.push_back(r.b);
  }
  g_prof.clear();
  for (int i = 0; i < k && i < n; ++i) out[i] = {names[i], launches[i], ms[i]};
  return k;
}

// ------------------------------------------------------------------ forward without allocation
// Scratch for mls_head_loss_fwd_noalloc: a fixed device array that every GPU
// loading this library holds until the process exits.  Host code must not use
// the symbol's name as a device address; the address is looked up once per
// device with cudaGetSymbolAddress (that device current) and passed to the kernels.
static __device__ __align__(256) unsigned char g_noalloc_scratch[MLS_NOALLOC_SCRATCH_BYTES];

namespace mls {
namespace {
void* g_noalloc_ptr[kMaxDevices] = {};

int noalloc_scratch(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(MLS_ERR_CUDA, "cudaGetDevice", e);
  if (dev < 0 || dev >= kMaxDevices) return MLS_ERR_DEVICE;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_noalloc_ptr[dev]) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess || !ptr) return fail(MLS_ERR_CUDA, "cudaGetSymbolAddress(scratch)", e);
    g_noalloc_ptr[dev] = ptr;
  }
  *out = g_noalloc_ptr[dev];
  return MLS_OK;
}
}  // namespace
}  // namespace mls

extern "C" int mls_head_loss_fwd_noalloc(const mls_problem* p, const void* const* H,
                                         const void* const* W, const int32_t* targets, float* loss,
                                         float* tok_loss, float* tok_diag, int32_t* argmax,
                                         float* stats, mls_stream_t stream) {
  int rc = validate(p);
  if (rc) return rc;
  if (!H || !W || !loss || (p->T > 0 && (!targets || !tok_loss || !stats))) return MLS_ERR_ARG;
  for (int m = 0; m < p->M; ++m) {
    if ((p->T > 0 && !H[m]) || !W[m]) return MLS_ERR_ARG;  // no rows to read when T = 0
    if (!aligned16(H[m]) || !aligned16(W[m])) return MLS_ERR_ALIGN;
  }
  DeviceState* dev = nullptr;
  if ((rc = device_state(&dev))) return rc;
  const Plan pl = make_plan(p, dev->head_pairs, dev->gemm_pairs);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (p->T == 0) return launch_ok(cudaMemsetAsync(loss, 0, sizeof(float), s));
  if (pl.fwd_bytes > static_cast<size_t>(MLS_NOALLOC_SCRATCH_BYTES))
    return fail(MLS_ERR_WORKSPACE, "forward needs more scratch than MLS_NOALLOC_SCRATCH_BYTES");
  void* scratch = nullptr;
  if ((rc = noalloc_scratch(&scratch))) return rc;
  char* wsb = static_cast<char*>(scratch);
  // Every word of scratch that the kernels read is written earlier in the same
  // call (partials of valid rows, one sum per merge block), so nothing is cleared.

  HeadParams hp;
  std::memset(&hp, 0, sizeof hp);
  fill_head_common(hp, p, pl, targets, dev->status);
  if ((rc = encode_head_maps(hp, p, pl, H, W))) return rc;
  hp.split = pl.split;
  hp.part = reinterpret_cast<float*>(wsb + pl.off_part);
  if ((rc = timed("head_fwd", s, [&] { return launch_head_fwd(hp, pl.elt == 4, p->tau == 1.0f, s); })))
    return rc;

  MergeParams mp;
  std::memset(&mp, 0, sizeof mp);
  mp.part = hp.part;
  mp.nparts = pl.nparts;
  mp.M = p->M;
  mp.teacher = p->teacher;
  mp.T = p->T;
  mp.V = p->V;
  mp.L1 = hp.L1;
  mp.Ltau = hp.Ltau;
  mp.tau = p->tau;
  mp.alpha = p->alpha;
  for (int m = 0; m < p->M; ++m) mp.w[m] = p->w ? p->w[m] : 1.0f;
  mp.y = targets;
  mp.tok_loss = tok_loss;
  mp.tok_diag = tok_diag;
  mp.argmax = argmax;
  mp.stats = stats;
  mp.block_sum = reinterpret_cast<double*>(wsb + pl.off_bsum);
  mp.block_cnt = reinterpret_cast<long long*>(wsb + pl.off_bcnt);
  mp.status = dev->status;
  if ((rc = timed("merge", s, [&] { return launch_merge(mp, pl.merge_blocks, s); }))) return rc;
  return timed("final", s, [&] {
    return launch_final(mp.block_sum, mp.block_cnt, pl.merge_blocks, loss, s);
  });
}

extern "C" int mls_head_pairwise(const mls_problem* p, const void* const* H, const void* const* W,
                                 const int32_t* targets, float* tok_kl, int32_t* argmax,
                                 float* pair_stats, void* ws, size_t ws_bytes, mls_stream_t stream) {
  int rc = validate(p);
  if (rc) return rc;
  if (!H || !W || !pair_stats || (p->T > 0 && !tok_kl)) return MLS_ERR_ARG;
  for (int m = 0; m < p->M; ++m) {
    if ((p->T > 0 && !H[m]) || !W[m]) return MLS_ERR_ARG;  // no rows to read when T = 0
    if (!aligned16(H[m]) || !aligned16(W[m])) return MLS_ERR_ALIGN;
  }
  DeviceState* dev = nullptr;
  if ((rc = device_state(&dev))) return rc;
  const Plan pl = make_plan(p, dev->head_pairs, dev->gemm_pairs);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (p->T == 0)
    return launch_ok(cudaMemsetAsync(pair_stats, 0, sizeof(float) * 2 * p->M * p->M, s));
  if ((rc = check_ws(pl, ws, ws_bytes, pl.total))) return rc;
  char* wsb = static_cast<char*>(ws);

  EvalParams ep;
  std::memset(&ep, 0, sizeof ep);
  const int KE = 128 / pl.elt;
  for (int m = 0; m < p->M; ++m) {
    if (encode(&ep.mapH[m], H[m], pl.elt, p->d[m], p->T, p->d[m], KE, kHeadBM) ||
        encode(&ep.mapW[m], W[m], pl.elt, p->d[m], p->V, p->d[m], KE, eval_tile_cols(p->M) / 2))
      return MLS_ERR_CUDA;
    ep.nk[m] = static_cast<int>(ceil_div(p->d[m], KE));
  }
  ep.M = p->M;
  // units of a vocabulary tile, widest sub-model first (it overlaps the epilogue)
  for (int i = 0; i < p->M; ++i) ep.order[i] = i;
  for (int i = 0; i < p->M; ++i)
    for (int k = i + 1; k < p->M; ++k)
      if (p->d[ep.order[k]] > p->d[ep.order[i]]) {
        const int t = ep.order[i];
        ep.order[i] = ep.order[k];
        ep.order[k] = t;
      }
  // Slot schedule (M = 3): the narrower of the two TMEM-slot units goes first,
  // so the epilogue's first pass runs under the longer MMAs of the other.
  if (eval_slotted(p->M)) {
    const int t = ep.order[1];
    ep.order[1] = ep.order[2];
    ep.order[2] = t;
  }
  for (int i = 0; i < p->M; ++i) ep.pos[ep.order[i]] = i;
  ep.split = pl.eval_split;
  ep.T = p->T;
  ep.V = p->V;
  ep.L1 = 1.4426950408889634f;
  ep.status = dev->status;
  ep.part = reinterpret_cast<float*>(wsb + pl.off_epart);
  if ((rc = timed("pairwise", s, [&] { return launch_eval(ep, pl.elt == 4, s); }))) return rc;

  EvalMergeParams mp;
  std::memset(&mp, 0, sizeof mp);
  mp.part = ep.part;
  mp.nparts = pl.eval_nparts;
  mp.M = p->M;
  mp.T = p->T;
  mp.V = p->V;
  mp.y = targets;
  mp.tok_kl = tok_kl;
  mp.argmax = argmax;
  mp.block_acc = reinterpret_cast<double*>(wsb + pl.off_eacc);
  mp.block_cnt = reinterpret_cast<long long*>(wsb + pl.off_ecnt);
  mp.status = dev->status;
  if ((rc = timed("pairwise_merge", s, [&] { return launch_eval_merge(mp, pl.eval_merge_blocks, s); })))
    return rc;
  return timed("pairwise_final", s, [&] {
    return launch_eval_final(mp.block_acc, mp.block_cnt, pl.eval_merge_blocks, p->M, pair_stats, s);
  });
}

namespace {
int junction_check(long long T, int d_prev, int d_next, int dtype, const void* const* ptrs, int n) {
  if (T < 0 || T > INT_MAX || d_prev < 1 || d_next <= d_prev) return MLS_ERR_ARG;
  if (dtype != MLS_BF16 && dtype != MLS_FP32) return MLS_ERR_ARG;
  const int elt = dtype == MLS_BF16 ? 2 : 4;
  if ((static_cast<long long>(d_prev) * elt) % 16 || (static_cast<long long>(d_next) * elt) % 16)
    return MLS_ERR_UNSUPPORTED;
  for (int i = 0; i < n; ++i) {
    if (T > 0 && !ptrs[i]) return MLS_ERR_ARG;
    if (!aligned16(ptrs[i])) return MLS_ERR_ALIGN;
  }
  return MLS_OK;
}
}  // namespace

extern "C" int mls_junction_fwd(int64_t T, int32_t d_prev, int32_t d_next, int32_t in_dtype,
                                int32_t embed_first, const void* o, const void* e, void* x,
                                mls_stream_t stream) {
  const void* ptrs[3] = {o, e, x};
  int rc = junction_check(T, d_prev, d_next, in_dtype, ptrs, 3);
  if (rc) return rc;
  DeviceState* dev = nullptr;
  if ((rc = device_state(&dev))) return rc;
  JunctionParams jp{T, d_prev, d_next, embed_first ? 1 : 0, o, e, x, nullptr, nullptr, nullptr,
                    dev->status, dev->sms};
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  return timed("junction_fwd", s, [&] { return launch_junction_fwd(jp, in_dtype == MLS_FP32, s); });
}

extern "C" int mls_junction_bwd(int64_t T, int32_t d_prev, int32_t d_next, int32_t in_dtype,
                                int32_t embed_first, const void* o, const void* e, const void* g,
                                void* d_o, void* d_e, mls_stream_t stream) {
  const void* ptrs[5] = {o, e, g, d_o, d_e};
  int rc = junction_check(T, d_prev, d_next, in_dtype, ptrs, 5);
  if (rc) return rc;
  DeviceState* dev = nullptr;
  if ((rc = device_state(&dev))) return rc;
  JunctionParams jp{T, d_prev, d_next, embed_first ? 1 : 0, o, e, nullptr, g, d_o, d_e, dev->status,
                    dev->sms};
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  return timed("junction_bwd", s, [&] { return launch_junction_bwd(jp, in_dtype == MLS_FP32, s); });
}

// ------------------------------------------------------------------ speculative verify
namespace {
struct SpecPlan {
  long long Pd = 0, Pv = 0, ldz = 0, tiles = 0;
  bool few = false;     // few rows: logits by mls_logits.cu, tiles of kLogitsTile columns
  size_t off_ev = 0, off_ed = 0, off_sv = 0, off_sd = 0, off_fv = 0, off_fd = 0;
  size_t off_stv = 0, off_std = 0, total = 0;
};

int spec_validate(const mls_spec_problem* p) {
  if (!p || p->B < 0 || p->gamma < 0 || p->V < 1 || p->V > INT_MAX) return MLS_ERR_ARG;
  if (p->in_dtype != MLS_BF16 && p->in_dtype != MLS_FP32) return MLS_ERR_ARG;
  if (static_cast<long long>(p->B) * (p->gamma + 1) > INT_MAX) return MLS_ERR_ARG;
  const int elt = p->in_dtype == MLS_BF16 ? 2 : 4;
  if (p->d_verify < 1) return MLS_ERR_ARG;
  if ((static_cast<long long>(p->d_verify) * elt) % 16 != 0) return MLS_ERR_UNSUPPORTED;
  if (!p->greedy) {
    if (p->d_draft < 1) return MLS_ERR_ARG;
    if ((static_cast<long long>(p->d_draft) * elt) % 16 != 0) return MLS_ERR_UNSUPPORTED;
    if (!(p->temperature > 0.f) || !std::isfinite(p->temperature)) return MLS_ERR_ARG;
    if (!(p->top_p > 0.f && p->top_p <= 1.f)) return MLS_ERR_ARG;
    if (p->V > static_cast<long long>(kSpecMaxTiles) * kGemmBN || p->gamma > kSpecMaxGamma)
      return MLS_ERR_UNSUPPORTED;
  }
  return MLS_OK;
}

SpecPlan spec_plan(const mls_spec_problem* p) {
  SpecPlan pl;
  pl.Pv = static_cast<long long>(p->B) * (p->gamma + 1);
  pl.Pd = p->greedy ? 0 : static_cast<long long>(p->B) * p->gamma;
  pl.ldz = ceil_div(p->V, 4) * 4;
  // Few rows: bound by reading the heads (mls_logits.cu says more; at its
  // largest, 128 rows, the launch takes 83 us against the pair GEMM's 92).
  // Sampling keeps a row's tile table in shared memory, hence the bound on V.
  pl.few = pl.Pv <= kLogitsMaxRows && p->V <= static_cast<long long>(kSpecMaxTiles) * kLogitsTile;
  pl.tiles = ceil_div(p->V, pl.few ? kLogitsTile : kGemmBN);
  const size_t rows_e = p->greedy ? 0 : static_cast<size_t>(pl.Pv);  // e_t is only stored when sampling
  size_t o = 0;
  auto take = [&](size_t& off, size_t bytes) {
    off = o;
    o = align_up(o + bytes);
  };
  take(pl.off_ev, sizeof(float) * rows_e * pl.ldz);
  take(pl.off_ed, sizeof(float) * static_cast<size_t>(pl.Pd) * pl.ldz);
  take(pl.off_stv, sizeof(float) * 2 * static_cast<size_t>(pl.Pv) * pl.tiles);
  take(pl.off_std, sizeof(float) * 2 * static_cast<size_t>(pl.Pd) * pl.tiles);
  take(pl.off_fv, sizeof(float) * rows_e * pl.tiles);
  take(pl.off_fd, sizeof(float) * static_cast<size_t>(pl.Pd) * pl.tiles);
  take(pl.off_sv, sizeof(float) * kSpecStateWords * static_cast<size_t>(pl.Pv));
  take(pl.off_sd, sizeof(float) * kSpecStateWords * static_cast<size_t>(pl.Pd));
  pl.total = o;
  return pl;
}
}  // namespace

extern "C" size_t mls_spec_workspace_size(const mls_spec_problem* p) {
  if (spec_validate(p)) return 0;
  return spec_plan(p).total;
}

extern "C" int mls_spec_verify(const mls_spec_problem* p, const void* H_draft, const void* W_draft,
                               const void* H_verify, const void* W_verify,
                               const int32_t* draft_tokens, const float* uniforms,
                               int32_t* n_accepted, int32_t* next_token, void* ws, size_t ws_bytes,
                               mls_stream_t stream) {
  int rc = spec_validate(p);
  if (rc) return rc;
  if (p->B == 0) return MLS_OK;
  if (!H_verify || !W_verify || !n_accepted || !next_token || (p->gamma > 0 && !draft_tokens))
    return MLS_ERR_ARG;
  if (!p->greedy && (!uniforms || (p->gamma > 0 && (!H_draft || !W_draft)))) return MLS_ERR_ARG;
  if (!aligned16(H_verify) || !aligned16(W_verify) || !aligned16(H_draft) || !aligned16(W_draft))
    return MLS_ERR_ALIGN;
  const SpecPlan pl = spec_plan(p);
  if (!ws || (reinterpret_cast<uintptr_t>(ws) % kAlign) != 0 || ws_bytes < pl.total)
    return MLS_ERR_WORKSPACE;
  DeviceState* dev = nullptr;
  if ((rc = device_state(&dev))) return rc;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  char* wsb = static_cast<char*>(ws);
  const bool tf32 = p->in_dtype == MLS_FP32;
  const int elt = tf32 ? 4 : 2, KE = 128 / elt;
  auto at = [&](size_t off) { return reinterpret_cast<float*>(wsb + off); };

  SpecParams sp;
  std::memset(&sp, 0, sizeof sp);
  sp.V = p->V;
  sp.ldz = pl.ldz;
  sp.B = p->B;
  sp.gamma = p->gamma;
  sp.greedy = p->greedy ? 1 : 0;
  sp.tiles = static_cast<int>(pl.tiles);
  sp.tile_shift = pl.few ? 7 : 8;
  sp.scale = p->greedy ? 1.f : 1.4426950408889634f / p->temperature;
  sp.top_p = p->greedy ? 1.f : p->top_p;
  sp.ev = at(pl.off_ev);
  sp.ed = at(pl.off_ed);
  sp.stats_v = at(pl.off_stv);
  sp.stats_d = at(pl.off_std);
  sp.f_v = at(pl.off_fv);
  sp.f_d = at(pl.off_fd);
  sp.draft = draft_tokens;
  sp.u = uniforms;
  sp.state_v = at(pl.off_sv);
  sp.state_d = at(pl.off_sd);
  sp.n_accepted = n_accepted;
  sp.next_token = next_token;
  sp.status = dev->status;
  sp.sms = dev->sms;

  // Logits of the verify positions: one launch over the verifier's rows and
  // (sampling) the draft's, z = H W^T with both operands K-major; its epilogue
  // leaves per-tile softmax statistics (sampling) or the per-tile maximum and
  // argmax (greedy) instead of the logits.
  const void* Hs[2] = {H_verify, H_draft};
  const void* Ws[2] = {W_verify, W_draft};
  const int ds[2] = {p->d_verify, p->d_draft};
  const long long Ps[2] = {pl.Pv, pl.Pd};
  float* Cs[2] = {at(pl.off_ev), at(pl.off_ed)};
  float* Ss[2] = {at(pl.off_stv), at(pl.off_std)};
  if (pl.few) {
    LogitsParams lp;
    std::memset(&lp, 0, sizeof lp);
    const int first = Ps[1] > 0 && ds[1] > ds[0] ? 1 : 0;
    lp.n = static_cast<int>(ceil_div(pl.Pv, 16) * 16);
    for (int k = 0; k < 2; ++k) {
      const int m = k == 0 ? first : 1 - first;
      if (Ps[m] == 0) continue;
      const int i = lp.nprob++;
      if (encode(&lp.mapW[i], Ws[m], elt, ds[m], p->V, ds[m], KE, kLogitsTile) ||
          encode(&lp.mapH[i], Hs[m], elt, ds[m], Ps[m], ds[m], KE, lp.n))
        return MLS_ERR_CUDA;
      lp.prob[i] = {static_cast<int>(Ps[m]), static_cast<int>(ceil_div(ds[m], KE)),
                    static_cast<int>(pl.tiles), Cs[m], Ss[m]};
    }
    lp.greedy = sp.greedy;
    lp.scale = sp.scale;
    lp.V = p->V;
    lp.ldz = pl.ldz;
    lp.stats_ld = 2 * pl.tiles;
    lp.status = dev->status;
    const int units = static_cast<int>(pl.tiles) * lp.nprob;
    const int grid = units < dev->sms ? units : dev->sms;
    const int r = lp.prob[0].tiles % grid;
    if (lp.nprob > 1 && r > 0) {
      const long long fair = ceil_div(lp.prob[1].tiles, grid - r);
      const long long even = ceil_div(lp.prob[0].nk, lp.prob[1].nk);
      lp.catchup = static_cast<int>(fair < even ? fair : even);
    }
    if ((rc = timed("spec_logits", s, [&] { return launch_logits(lp, tf32, grid, s); }))) return rc;
    if (!p->greedy && (rc = timed("spec_rows", s, [&] { return launch_spec_rows(sp, s); }))) return rc;
    return timed("spec_sample", s, [&] { return launch_spec_sample(sp, s); });
  }
  GemmParams g;
  std::memset(&g, 0, sizeof g);
  int tiles = 0;
  for (int m = 0; m < 2; ++m) {
    if (Ps[m] == 0) continue;
    const int i = g.nprob++;
    if (encode(&g.mapA[i], Hs[m], elt, ds[m], Ps[m], ds[m], KE, kGemmBM) ||
        encode(&g.mapB[i], Ws[m], elt, ds[m], p->V, ds[m], KE, kGemmBHalf) ||
        (!p->greedy && encode(&g.mapC[i], Cs[m], 4, p->V, Ps[m], pl.ldz, 32, 32)))
      return MLS_ERR_CUDA;
    GemmProblem& pr = g.prob[i];
    pr.Mrows = static_cast<int>(Ps[m]);
    pr.Ncols = static_cast<int>(p->V);
    pr.K = ds[m];
    pr.a_map = pr.b_map = i;
    pr.tiles_n = static_cast<int>(pl.tiles);
    pr.tiles_m = static_cast<int>(ceil_div(Ps[m], 2 * kGemmBM));
    pr.m_fast = 1;
    pr.tile_begin = tiles;
    pr.epi = p->greedy ? kEpiArgmax : kEpiSoftmax;
    pr.epi_scale = sp.scale;
    pr.stats = Ss[m];
    pr.stats_ld = 2 * pl.tiles;
    tiles += pr.tiles_m * pr.tiles_n;
  }
  g.total_tiles = tiles;
  g.status = dev->status;
  const int grid = 2 * (tiles < dev->gemm_pairs ? tiles : dev->gemm_pairs);
  if ((rc = timed("spec_logits", s, [&] { return launch_gemm_stats(g, tf32, grid, s); }))) return rc;
  if (!p->greedy && (rc = timed("spec_rows", s, [&] { return launch_spec_rows(sp, s); })))
    return rc;
  return timed("spec_sample", s, [&] { return launch_spec_sample(sp, s); });
}
