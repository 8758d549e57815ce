// Logits of a few rows against a whole vocabulary, with the row statistics
// that the speculative verify step needs (the same outputs as the statistics
// epilogues of mls_gemm.cu).
//
// With up to kLogitsMaxRows rows the product is bound by reading the heads W
// from HBM, and a 256-row tile of the pair GEMM would spend its MMAs on padding
// (7 rows: as long as the reading itself).  So the operands change places: W's
// vocabulary rows are the M dimension and the hidden rows the N dimension of
// the MMA, whose time follows the rows there are.  One CTA per SM walks tiles
// of 128 vocabulary columns over both sub-models' heads, with 96 to 160 KB of W
// in flight per SM:
//   warp 8    TMA producer: 128 rows of W and the n rows of H per k-block
//   warp 9    MMA issuer
//   warps 0-7 epilogue: one vocabulary column per lane, one MMA column per row
//             (warps 0-3 take the even groups of 32 rows, warps 4-7 the odd ones);
//             a row's statistics combine over lanes, then over the warps
//             through shared memory, in a fixed order
// Tiles of 128 columns, not the pair GEMM's 256, so that 393 of them per head
// (V = 50304) spread evenly over 152 SMs: with 256 columns the greedy call
// below took 75 us.  Measured with V = 50304, widths 1024 / 3072, the whole
// verify call and this launch (events around it add about 5 us) against the
// pair GEMM: 7 rows 129 -> 91 us, 108 -> 70 us (412 MB at 6.3 TB/s); 48 rows
// 91 -> 74 us; 112 rows 91 -> 81 us; 112 rows greedily 68 -> 67 us.
#include "mls_device.cuh"
#include "mls_kernels.h"

namespace mls {
namespace {

constexpr int kTile = kLogitsTile;
constexpr int kEpi = 8;                           // epilogue warps
constexpr int kThreads = (kEpi + 2) * 32;
constexpr uint32_t kABytes = kTile * 128;         // W rows of a stage
constexpr uint32_t kStageBudget = 208 * 1024;
constexpr int kMaxStages = 10;
constexpr uint32_t kTmemCols = 256;               // 2 buffers x kLogitsMaxRows columns
constexpr uint64_t kDrainNs = 100000000ull;

// Shared-memory map past the operand stages.
struct Tail {
  uint64_t full[kMaxStages], empty[kMaxStages], accf[2], acce[2], drain;
  uint32_t tmem_slot;
  int abort;
  // per tile parity: a warp's maximum, its first column (greedy) or sum, per row
  float wmax[2][4][kLogitsMaxRows];
  float wsum[2][4][kLogitsMaxRows];
};

__host__ __device__ __forceinline__ uint32_t stage_bytes(int n) {
  return kABytes + ((static_cast<uint32_t>(n) * 128u + 1023u) & ~1023u);
}
__host__ __device__ __forceinline__ int stage_count(int n) {
  const int s = static_cast<int>(kStageBudget / stage_bytes(n));
  return s < kMaxStages ? s : kMaxStages;
}
constexpr uint32_t kLogitsSmem = 1024 + kStageBudget + sizeof(Tail);
static_assert(kLogitsSmem <= 227 * 1024, "logits kernel shared memory");
static_assert(kLogitsMaxRows * 2 <= static_cast<int>(kTmemCols), "accumulators fit in TMEM");

// The j-th unit of CTA c of G, or -1: the first problem's units round-robin,
// then the CTAs left one of them short take `catchup` of the second's each,
// and the rest go round-robin.
__device__ __forceinline__ int cta_unit(const LogitsParams& p, int c, int G, int j) {
  const int n0 = p.prob[0].tiles, n1 = p.nprob > 1 ? p.prob[1].tiles : 0;
  const int r = n0 % G, nl = n0 / G + (c < r ? 1 : 0);
  if (j < nl) return c + j * G;
  j -= nl;
  if (c >= r) {
    if (j < p.catchup) {
      const int s = c - r + j * (G - r);
      return s < n1 ? n0 + s : -1;
    }
    j -= p.catchup;
  }
  const int s = p.catchup * (G - r) + c + j * G;
  return s < n1 ? n0 + s : -1;
}

__device__ __forceinline__ float redux_max(float v) {
  float m;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
  return m;
}

// Lane l gets the sum over the warp's lanes of v[l] (a transpose by halves: 31
// shuffles for 32 sums).
__device__ __forceinline__ float transpose_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float keep = up ? v[i + o] : v[i], give = up ? v[i] : v[i + o];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return v[0];
}

template <bool kGreedy>
__device__ __forceinline__ void logits_epilogue(const LogitsParams& p, Tail* sh, uint32_t tmem,
                                                int warp, int lane) {
  const int quad = warp & 3, sub = warp >> 2;
  const int cols = (p.n + 31) & ~31;
  const uint32_t tl = tmem + (static_cast<uint32_t>(quad * 32) << 16);
  const int c = blockIdx.x, G = gridDim.x;
  int i = 0, u;
  for (int j = 0; (u = cta_unit(p, c, G, j)) >= 0; ++j, ++i) {
    const int pi = u >= p.prob[0].tiles ? 1 : 0;
    const LogitsProblem& pr = p.prob[pi];
    const int tile = u - (pi ? p.prob[0].tiles : 0);
    const uint32_t acc = static_cast<uint32_t>(i) & 1u;
    // All epilogue warps go on or leave together: the barriers below need all of them.
    const bool ok = mbar_wait(smem_u32(&sh->accf[acc]), static_cast<uint32_t>(i >> 1) & 1u, &sh->abort, p.status);
    if (!named_bar_and(1, kEpi * 32, ok)) break;
    tc_fence_after();
    const uint32_t ta = tl + acc * static_cast<uint32_t>(cols);
    const long long v0 = static_cast<long long>(tile) * kTile + quad * 32;
    const bool in = v0 + lane < p.V;
    float* wmax = sh->wmax[acc][quad];
    float* wsum = sh->wsum[acc][quad];
    float z[32];
#pragma unroll 1
    for (int r0 = sub * 32; r0 < pr.rows; r0 += 64) {
      tmem_ld32(ta + r0, z);
      float mine = -INFINITY, arg = 0.f;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const float zk = in ? z[k] : -INFINITY;
        const float m = fmaxf(redux_max(zk), -INFINITY);  // all NaN: -inf
        if (k == lane) mine = m;
        if (kGreedy) {
          const unsigned hit = __ballot_sync(0xffffffffu, zk == m);
          if (k == lane) arg = __int_as_float(static_cast<int>(v0) + (hit ? __ffs(hit) - 1 : 0));
        }
      }
      wmax[r0 + lane] = mine;
      if (kGreedy) wsum[r0 + lane] = arg;
    }
    if (kGreedy) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh->acce[acc]));
    }
    named_bar_sync(1, kEpi * 32);
    if constexpr (kGreedy) {
      const int row = threadIdx.x;
      if (row < pr.rows) {
        float m = -INFINITY;
        int a = tile * kTile;
        for (int w = 0; w < 4; ++w) {  // warps in vocabulary order: the first maximum wins
          const float mw = sh->wmax[acc][w][row];
          if (mw > m) {
            m = mw;
            a = __float_as_int(sh->wsum[acc][w][row]);
          }
        }
        float* s = pr.stats + row * p.stats_ld + 2 * tile;
        s[0] = m;
        s[1] = __int_as_float(a);
      }
    } else {
#pragma unroll 1
      for (int r0 = sub * 32; r0 < pr.rows; r0 += 64) {
        float m = -INFINITY;
#pragma unroll
        for (int w = 0; w < 4; ++w) m = fmaxf(m, sh->wmax[acc][w][r0 + lane]);
        tmem_ld32(ta + r0, z);
        float* out = pr.e + static_cast<long long>(r0) * p.ldz + v0 + lane;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          const float mk = __shfl_sync(0xffffffffu, m, k);
          z[k] = in ? fast_exp2((z[k] - mk) * p.scale) : 0.f;
          if (in && r0 + k < pr.rows) out[k * p.ldz] = z[k];
        }
        wsum[r0 + lane] = transpose_sum(z, lane);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh->acce[acc]));
      named_bar_sync(1, kEpi * 32);
      const int row = threadIdx.x;
      if (row < pr.rows) {
        float m = -INFINITY, s = 0.f;
        for (int w = 0; w < 4; ++w) {
          m = fmaxf(m, sh->wmax[acc][w][row]);
          s += sh->wsum[acc][w][row];
        }
        float* st = pr.stats + row * p.stats_ld + 2 * tile;
        st[0] = m;
        st[1] = s;
      }
    }
  }
}

template <bool kTF32, bool kGreedy>
__global__ void __launch_bounds__(kThreads, 1) logits_kernel(const __grid_constant__ LogitsParams p) {
  constexpr int KE = kTF32 ? 32 : 64;  // elements in 128 bytes of K
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
  Tail* sh = reinterpret_cast<Tail*>(smem_raw + (base - raw) + kStageBudget);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = stage_count(p.n);
  const uint32_t sbytes = stage_bytes(p.n);
  const int c = blockIdx.x, G = gridDim.x;

  if (threadIdx.x == 0) {
    sh->abort = 0;
    for (int s = 0; s < stages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&sh->accf[a]), 1);
      mbar_init(smem_u32(&sh->acce[a]), kEpi);
    }
    mbar_init(smem_u32(&sh->drain), 1);
    fence_barrier_init();
  }
  if (warp == kEpi + 1) {
    tmem_alloc(smem_u32(&sh->tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh->tmem_slot;

  if (warp == kEpi) {
    if (lane == 0) {
      int stage = 0, u;
      uint32_t phase = 0, filled = 0, lastpar = 0;
      bool ok = true;
      for (int j = 0; ok && (u = cta_unit(p, c, G, j)) >= 0; ++j) {
        const int pi = u >= p.prob[0].tiles ? 1 : 0;
        const int v0 = (u - (pi ? p.prob[0].tiles : 0)) * kTile;
        MLS_CHECK(p.status, v0 < p.V && p.prob[pi].rows <= p.n && p.n <= kLogitsMaxRows);
        for (int kb = 0; kb < p.prob[pi].nk; ++kb) {
          if (!mbar_wait(smem_u32(&sh->empty[stage]), phase ^ 1u, &sh->abort, p.status)) {
            ok = false;
            break;
          }
          const uint32_t bar = smem_u32(&sh->full[stage]), sa = base + static_cast<uint32_t>(stage) * sbytes;
          mbar_arrive_expect_tx(bar, kABytes + static_cast<uint32_t>(p.n) * 128u);
          tma_load_2d(sa, &p.mapW[pi], bar, kb * KE, v0);
          tma_load_2d(sa + kABytes, &p.mapH[pi], bar, kb * KE, 0);
          filled |= 1u << stage;
          lastpar = (lastpar & ~(1u << stage)) | (phase << stage);
          if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok)  // loads already issued must land before the shared memory goes away
        for (int s = 0; s < stages; ++s)
          if ((filled >> s) & 1u)
            mbar_wait_drain(smem_u32(&sh->full[s]), (lastpar >> s) & 1u, kDrainNs, p.status);
      chain_trigger();
    }
  } else if (warp == kEpi + 1) {
    if (lane == 0) {
      const uint32_t idesc = make_idesc(128, p.n, kTF32, false, false);
      const uint32_t cols = (static_cast<uint32_t>(p.n) + 31u) & ~31u;
      int stage = 0, i = 0, u;
      uint32_t phase = 0;
      bool ok = true;
      for (int j = 0; ok && (u = cta_unit(p, c, G, j)) >= 0; ++j, ++i) {
        const int nk = p.prob[u >= p.prob[0].tiles ? 1 : 0].nk;
        const uint32_t acc = static_cast<uint32_t>(i) & 1u;
        if (!mbar_wait(smem_u32(&sh->acce[acc]), (static_cast<uint32_t>(i >> 1) & 1u) ^ 1u, &sh->abort, p.status)) break;
        tc_fence_after();
        const uint32_t d = tmem + acc * cols;
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait(smem_u32(&sh->full[stage]), phase, &sh->abort, p.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = base + static_cast<uint32_t>(stage) * sbytes;
          const uint64_t a = make_sdesc(sa, 16), b = make_sdesc(sa + kABytes, 16);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)  // 4 x 32 bytes of K per stage
            mma_issue<kTF32>(d, a + 2u * kk, b + 2u * kk, idesc, (kb | kk) != 0);
          mma_commit(smem_u32(&sh->empty[stage]));
          if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok) mma_commit(smem_u32(&sh->accf[acc]));
      }
      // Every MMA this thread issued has finished before TMEM is released.
      mma_commit(smem_u32(&sh->drain));
      mbar_wait_drain(smem_u32(&sh->drain), 0, kDrainNs, p.status);
    }
    __syncwarp();
  } else {
    logits_epilogue<kGreedy>(p, sh, tmem, warp, lane);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kEpi + 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace

cudaError_t launch_logits(const LogitsParams& p, bool tf32, int grid, cudaStream_t s) {
  if (grid <= 0) return cudaSuccess;
  if (tf32) {
    if (p.greedy) logits_kernel<true, true><<<grid, kThreads, kLogitsSmem, s>>>(p);
    else logits_kernel<true, false><<<grid, kThreads, kLogitsSmem, s>>>(p);
  } else {
    if (p.greedy) logits_kernel<false, true><<<grid, kThreads, kLogitsSmem, s>>>(p);
    else logits_kernel<false, false><<<grid, kThreads, kLogitsSmem, s>>>(p);
  }
  return cudaGetLastError();
}

cudaError_t setup_logits_kernels() {
  cudaError_t e;
#define MLS_SET(TF, GR)                                                                             \
  e = cudaFuncSetAttribute(logits_kernel<TF, GR>, cudaFuncAttributeMaxDynamicSharedMemorySize,      \
                           kLogitsSmem);                                                            \
  if (e != cudaSuccess) return e;
  MLS_SET(true, true)
  MLS_SET(true, false)
  MLS_SET(false, true)
  MLS_SET(false, false)
#undef MLS_SET
  return cudaSuccess;
}

}  // namespace mls
