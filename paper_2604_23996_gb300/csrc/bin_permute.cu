// bin_permute.cu -- de-duplicated bin dispatch (Sec. 4.5, "DeDup").
//
// Every token is sent once to each bin that holds at least one of its top-k experts; the
// entry carries a bit mask of the chosen experts' slots inside the bin. Entries are grouped by
// bin (ascending) and ordered by token inside a bin. One cooperative launch, all integer work:
//   count    per-block pair counts per bin (warp ballots);
//   barrier  a bounded grid barrier (all blocks are resident: cooperative launch);
//   offsets  each block sums the count table: its prefix inside every bin and the bin bases;
//   scatter  stable positions from ballots, tokens and masks written, and the dispatch matrix
//            and per-modality expert counts added (integer atomics: order-independent).
#include <algorithm>
#include <mutex>

#include "device_common.cuh"
#include "ptx.cuh"
#include "smoes_internal.cuh"

namespace smoes {
namespace {

constexpr int kPermThreads = 256;                    // one token per thread and round
constexpr int kPermWarps = kPermThreads / 32;

// One token's selection: the set of its chosen experts at position bin * N_B + slot of a 128-bit
// set (plans hold at most 128 experts), so that a bin's mask is N_B consecutive bits, its experts in
// bytes (0xff: none) for the counts, and its modality (0 vision, 1 text). Bins, slots and masks per
// selected expert in registers of their own took 96 registers at k = 8: two blocks per SM, and two
// rounds for 131072 tokens.
constexpr int kSetWords = kMaxExpertsBf16 / 32;
template <int KM>
struct TokenSel {
  uint32_t set[kSetWords];
  uint32_t e4[(KM + 3) / 4];
  int m;
};

template <int KM>
__device__ __forceinline__ void empty_sel(TokenSel<KM>& s) {
#pragma unroll
  for (int w = 0; w < kSetWords; ++w) s.set[w] = 0u;
#pragma unroll
  for (int q = 0; q < (KM + 3) / 4; ++q) s.e4[q] = 0xffffffffu;
  s.m = 0;
}

// Token j's top-k and modality from memory, and the selection they make.
template <int KM>
__device__ __forceinline__ void load_topk(const PermParams& p, int j, int (&e)[KM], int& m) {
  m = 0;
#pragma unroll
  for (int i = 0; i < KM; ++i) e[i] = (j < p.T && i < p.k) ? __ldg(p.topk_idx + static_cast<size_t>(j) * p.k + i) : -1;
  if (j < p.T && p.is_vision) m = __ldg(p.is_vision + j) ? 0 : 1;
}
template <int KM>
__device__ __forceinline__ void make_sel(const PermParams& p, const uint8_t* s_pos, const int (&e)[KM], int m,
                                         TokenSel<KM>& s) {
  empty_sel<KM>(s);
  s.m = m;
#pragma unroll
  for (int i = 0; i < KM; ++i) {
    if (i < p.k) {
      if (e[i] >= 0 && e[i] < p.E) {
        const uint32_t pos = s_pos[e[i]];
        const uint32_t bit = 1u << (pos & 31u);
#pragma unroll
        for (int w = 0; w < kSetWords; ++w) s.set[w] |= (pos >> 5) == static_cast<uint32_t>(w) ? bit : 0u;
        s.e4[i >> 2] ^= (0xffu ^ static_cast<uint32_t>(e[i])) << (8 * (i & 3));
      } else {
        atomicOr(p.status, kStatusData);
      }
    }
  }
}

// The first bin's mask of a set; the set then moves on to the next bin.
__device__ __forceinline__ uint32_t next_mask(uint32_t (&set)[kSetWords], int NB, uint32_t nb_mask) {
  const uint32_t m = set[0] & nb_mask;
#pragma unroll
  for (int w = 0; w < kSetWords; ++w) set[w] = __funnelshift_rc(set[w], w + 1 < kSetWords ? set[w + 1] : 0u, NB);
  return m;
}

template <int KM>
__global__ void __launch_bounds__(kPermThreads) k_perm(const PermParams p) {
  __shared__ uint8_t s_pos[kMaxExperts];
  __shared__ int wcnt[kPermWarps][kMaxBins];
  __shared__ int base[kMaxBins];
  __shared__ int pre_s[kMaxBins], tot_s[kMaxBins];
  __shared__ int disp[kMaxBins * kMaxBins];
  __shared__ int ecnt[2 * kMaxExperts];
  __shared__ int ok_s;
  // a cooperative grid launched with programmatic serialization: the top-k of the kernel before
  // it are read only after that kernel has completed
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int K = p.K, NB = p.E / p.K;
  const uint32_t nb_mask = NB >= 32 ? 0xffffffffu : (1u << NB) - 1u;
  int e0[KM], m0;                                       // the first round's top-k, beside the tables
  load_topk<KM>(p, blockIdx.x * p.rounds * kPermThreads + threadIdx.x, e0, m0);
  for (int e = threadIdx.x; e < p.E; e += kPermThreads) s_pos[e] = static_cast<uint8_t>(p.expert_bin[e] * NB + p.expert_slot[e]);
  for (int i = threadIdx.x; i < K * K; i += kPermThreads) disp[i] = 0;
  for (int i = threadIdx.x; i < 2 * p.E; i += kPermThreads) ecnt[i] = 0;
  __syncthreads();

  // count: lane kb of each warp accumulates the warp's pairs in bin kb; the first round's
  // selections stay in registers for the scatter
  int cnt = 0;
  TokenSel<KM> s0;
  empty_sel<KM>(s0);
  for (int r = 0; r < p.rounds; ++r) {
    const int j = (blockIdx.x * p.rounds + r) * kPermThreads + threadIdx.x;
    TokenSel<KM> s;
    empty_sel<KM>(s);
    if (r > 0) load_topk<KM>(p, j, e0, m0);
    if (j < p.T) make_sel<KM>(p, s_pos, e0, m0, s);
    if (r == 0) s0 = s;
    for (int kb = 0; kb < K; ++kb) {
      const int c = __popc(__ballot_sync(0xffffffffu, next_mask(s.set, NB, nb_mask) != 0u));
      if (lane == kb) cnt += c;
    }
  }
  if (lane < kMaxBins) wcnt[warp][lane] = cnt;
  __syncthreads();
  if (threadIdx.x < K) {
    int t = 0;
    for (int w = 0; w < kPermWarps; ++w) t += wcnt[w][threadIdx.x];
    p.blk_counts[threadIdx.x * p.n_blocks + blockIdx.x] = t;     // bin-major
  }
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < K * K; i += kPermThreads) p.dispatch[i] = 0;
    if (p.expert_counts)
      for (int i = threadIdx.x; i < 2 * p.E; i += kPermThreads) p.expert_counts[i] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) ok_s = grid_barrier(p.sync, gridDim.x, p.limit_ns, p.status) ? 1 : 0;
  __syncthreads();
  if (!ok_s) return;

  // offsets: warp w sums bins w, w + 8, ... over all blocks (lanes stride the blocks, eight loads in
  // flight per lane)
  for (int kb = warp; kb < K; kb += kPermWarps) {
    int pre = 0, tot = 0;
    const int* row = p.blk_counts + kb * p.n_blocks;
    int b0 = lane;
    for (; b0 + 7 * 32 < p.n_blocks; b0 += 8 * 32) {
      int c[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) c[u] = __ldcg(row + b0 + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        tot += c[u];
        pre += b0 + 32 * u < static_cast<int>(blockIdx.x) ? c[u] : 0;
      }
    }
    for (; b0 < p.n_blocks; b0 += 32) {
      const int c = __ldcg(row + b0);
      tot += c;
      pre += b0 < static_cast<int>(blockIdx.x) ? c : 0;
    }
    pre = __reduce_add_sync(0xffffffffu, pre);
    tot = __reduce_add_sync(0xffffffffu, tot);
    if (lane == 0) {
      pre_s[kb] = pre;
      tot_s[kb] = tot;
    }
  }
  __syncthreads();
  if (warp == 0) {                                      // bin bases: exclusive scan over the bins
    const int t = lane < K ? tot_s[lane] : 0;
    int run = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, run, o);
      if (lane >= o) run += v;
    }
    if (lane < K) {
      base[lane] = run - t + pre_s[lane];
      if (blockIdx.x == 0) p.bin_offsets[lane] = run - t;
      if (blockIdx.x == 0 && lane == K - 1) p.bin_offsets[K] = run;
    }
  }
  __syncthreads();

  // scatter: per round, warp counts per bin -> exclusive scan over warps -> ballot ranks
  const unsigned lt_mask = (1u << lane) - 1u;
  for (int r = 0; r < p.rounds; ++r) {
    const int j = (blockIdx.x * p.rounds + r) * kPermThreads + threadIdx.x;
    const bool valid = j < p.T;
    int home = 0;
    if (valid) {
      home = p.home ? p.home[j] : static_cast<int>((static_cast<long long>(j) * K) / p.T);
      if (home < 0 || home >= K) {
        atomicOr(p.status, kStatusData);
        home = -1;
      }
    }
    TokenSel<KM> s;
    if (r == 0) {
      s = s0;
    } else {
      empty_sel<KM>(s);
      load_topk<KM>(p, j, e0, m0);
      if (valid) make_sel<KM>(p, s_pos, e0, m0, s);
    }
    if (p.rounds > 1) {                                 // (one round: wcnt still holds the warps' counts)
      uint32_t set[kSetWords];
#pragma unroll
      for (int w = 0; w < kSetWords; ++w) set[w] = s.set[w];
      for (int kb = 0; kb < K; ++kb) {
        const unsigned bal = __ballot_sync(0xffffffffu, next_mask(set, NB, nb_mask) != 0u);
        if (lane == 0) wcnt[warp][kb] = __popc(bal);
      }
      __syncthreads();
    }
    if (threadIdx.x < K) {                              // exclusive scan over warps, per bin
      int run = base[threadIdx.x];
      for (int w = 0; w < kPermWarps; ++w) {
        const int t = wcnt[w][threadIdx.x];
        wcnt[w][threadIdx.x] = run;
        run += t;
      }
      base[threadIdx.x] = run;                          // carried into the next round
    }
    __syncthreads();
    // lanes with the same dispatch home add their pairs with one atomic per (warp, bin, home)
    const unsigned same_home = __match_any_sync(0xffffffffu, home);
    for (int kb = 0; kb < K; ++kb) {
      const uint32_t mask = next_mask(s.set, NB, nb_mask);
      const unsigned bal = __ballot_sync(0xffffffffu, mask != 0u);
      if (mask) {
        const int pos = wcnt[warp][kb] + __popc(bal & lt_mask);
        p.perm_token[pos] = j;
        p.perm_mask[pos] = mask;
        const unsigned grp = bal & same_home;
        if (home >= 0 && lane == __ffs(grp) - 1) atomicAdd(&disp[home * K + kb], __popc(grp));
      }
    }
    if (valid && p.expert_counts) {
#pragma unroll
      for (int i = 0; i < KM; ++i) {
        const uint32_t e = (s.e4[i >> 2] >> (8 * (i & 3))) & 0xffu;
        if (e != 0xffu) atomicAdd(&ecnt[s.m * p.E + static_cast<int>(e)], 1);
      }
    }
    __syncthreads();                                    // wcnt reused by the next round
  }
  for (int i = threadIdx.x; i < K * K; i += kPermThreads)
    if (disp[i]) atomicAdd(p.dispatch + i, disp[i]);
  if (p.expert_counts)
    for (int i = threadIdx.x; i < 2 * p.E; i += kPermThreads)
      if (ecnt[i]) atomicAdd(p.expert_counts + i, ecnt[i]);
}
}  // namespace

// Scratch of the no-allocation permutation entry point (see smoes_bin_permute_noalloc): one copy
// per device that loads this library, alive until the process exits, shared by every call.
static __device__ __align__(256) unsigned char g_perm_static[sizeof(StaticPermScratch)];

// The host cannot use g_perm_static's name as a device address; it asks the runtime once per
// device, with that device current, and caches the answer.
cudaError_t static_perm_scratch(StaticPermScratch** out) {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static void* addr[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (addr[dev] == nullptr) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_perm_static);
    if (e != cudaSuccess) return e;
    addr[dev] = p;
  }
  *out = static_cast<StaticPermScratch*>(addr[dev]);
  return cudaSuccess;
}

// The plan's bin map and slots travel to the device as kernel parameters (2 KB, by value, so no
// host buffer is referenced once the launch returns); one block writes them into the fixed
// scratch and clears its status and grid-barrier words.
struct StaticPermMaps {
  int32_t expert_bin[kMaxExperts];
  int32_t expert_slot[kMaxExperts];
  int E;
};

__global__ void __launch_bounds__(kPermThreads) k_static_perm_prep(const StaticPermMaps m,
                                                                    StaticPermScratch* sp) {
  for (int e = threadIdx.x; e < m.E; e += kPermThreads) {
    sp->expert_bin[e] = m.expert_bin[e];
    sp->expert_slot[e] = m.expert_slot[e];
  }
  if (threadIdx.x < 4) {
    sp->status[threadIdx.x] = 0u;
    sp->sync[threadIdx.x] = 0u;
  }
}

cudaError_t launch_static_perm_prep(StaticPermScratch* sp, const int32_t* expert_bin,
                                    const int32_t* expert_slot, int E, cudaStream_t s) {
  if (E < 1 || E > kMaxExperts) return cudaErrorInvalidValue;
  StaticPermMaps m;
  for (int e = 0; e < kMaxExperts; ++e) {
    m.expert_bin[e] = e < E ? expert_bin[e] : 0;
    m.expert_slot[e] = e < E ? expert_slot[e] : 0;
  }
  m.E = E;
  k_static_perm_prep<<<1, kPermThreads, 0, s>>>(m, sp);
  return cudaGetLastError();
}

template <class F>
cudaError_t with_kernel(int k, F&& f) {
  if (k <= 2) return f(k_perm<2>);
  if (k <= 4) return f(k_perm<4>);
  if (k <= 6) return f(k_perm<6>);
  if (k <= 8) return f(k_perm<8>);
  return f(k_perm<16>);
}

// Blocks of the permutation: all must be resident at once (the grid barrier), and at most
// kStaticPermBlocks. Rounds of 256 tokens per block grow once the batch needs more blocks.
int perm_max_blocks(int k) {
  static std::mutex mu;
  static int cached[64][5] = {};
  const int v = k <= 2 ? 0 : k <= 4 ? 1 : k <= 6 ? 2 : k <= 8 ? 3 : 4;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  std::lock_guard<std::mutex> lock(mu);
  if (cached[dev][v] == 0) {
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
    const cudaError_t e = with_kernel(k, [&](auto kern) {
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPermThreads, 0);
    });
    if (e != cudaSuccess) return 1;
    cached[dev][v] = std::max(1, std::min(kStaticPermBlocks, sms * per_sm));
  }
  return cached[dev][v];
}
int perm_rounds(int T, int k) {
  const int units = (T + kPermThreads - 1) / kPermThreads;
  const int cap = perm_max_blocks(k);
  return units <= cap ? 1 : (units + cap - 1) / cap;
}
int perm_blocks(int T, int k) {
  const int per = kPermThreads * perm_rounds(T, k);
  return (T + per - 1) / per;
}

cudaError_t launch_bin_permute(const PermParams& p, cudaStream_t s) {
  if (p.n_blocks > perm_max_blocks(p.k)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.n_blocks);
  cfg.blockDim = dim3(kPermThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;    // every block resident: the barrier is safe
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return with_kernel(p.k, [&](auto kern) { return cudaLaunchKernelEx(&cfg, kern, p); });
}

}  // namespace smoes
