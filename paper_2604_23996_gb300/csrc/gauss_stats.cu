// gauss_stats.cu -- online statistics of the Gaussian modality score (Sec. 3.2, eqs. 5-7) and
// momentum-adaptive binning (Sec. 3.3, eqs. 10-11).
//
// Statistics update. The state (N_m, S_mu,m, S_var,m) of each modality m is kept in fp64 on the
// device. One pass over X forms, per feature and hard modality, the shifted sums
//   s1 = sum_{x in T_m} (x - c),   s2 = sum_{x in T_m} (x - c)^2,
// with the shift c = S_mu,m,t-1 / N_m,t-1 to fp32 precision (0 for an empty state): the previous
// mean is close to the batch mean, so the centred second moment
//   sum (x - mu_T)^2 = s2 - s1^2 / n,   mu_T = c + s1 / n,
// loses nothing to cancellation. k_stats_partial streams X once (bulk copies, 8 features per
// thread, fp32 sums over a contiguous run of rows per block) and writes one partial per block;
// k_stats_finalize sums the partials in block order (runs of 8 in fp32, then fp64) and applies
// eqs. (5)-(7) in fp64. Both are deterministic.
//
// Adaptive binning. k_adaptive_bins (one block, E <= 256 threads) updates the EMA expert loads
// of eq. (10) from this step's per-modality selection counts, forms the text bias f_spec of
// eq. (11), and ranks the experts by ascending f_spec (equal values in expert-index order); the
// rank cut into runs of N_B experts is the new expert -> bin map. All of it is fp64 with the
// rounding of separate multiplies, adds and a correctly rounded division, so the order, and
// with it the bin map, is reproducible bit for bit.
#include <cuda_bf16.h>

#include "device_common.cuh"
#include "ptx.cuh"
#include "smoes_internal.cuh"

namespace smoes {
namespace {

constexpr int kStatConsumers = 512;              // threads that sum rows
constexpr int kStatThreads = kStatConsumers + 32;   // and the warp whose lane 0 issues the copies
constexpr int kStatCols = 2048;                  // features per pass of a block (8 per thread)
constexpr int kStatStages = 4;
constexpr uint32_t kStatStageBytes = 32768;      // rows of one stage: as many as fit (at most 64)
constexpr uint32_t kStatMergeBytes = kStatConsumers * 8u * 4u * 4u;   // (s1, s2) x (v, t) per thread
constexpr int kStatMaxRows = 16384;              // rows per block (their labels stay in shared memory)

// x / n with the reciprocal formed once: GB300 has two fp64 FMAs per SM and clock, and an fp64 division
// takes many. The product is off by up to two ulp: enough for what is rounded to fp32 (one division per
// feature and thread for the shift cost 20 us of the pass over d = 2048). For what enters the fp64
// state its remainder, exact as an FMA, corrects it to the division's own rounding (Markstein's theorem
// on the correctly rounded reciprocal). Where the reciprocal leaves the normal range (n = 0 or
// subnormal) the division itself is taken; an infinite quotient has no remainder.
__device__ __forceinline__ bool has_inverse(double inv) {   // a normal number (its exponent bits: fp64 compares are slow too)
  return ((static_cast<uint32_t>(__double2hiint(inv)) >> 20 & 0x7ffu) - 1u) < 2046u;
}
__device__ __forceinline__ float div_f32(double x, double n, double inv) {
  return static_cast<float>(has_inverse(inv) ? x * inv : x / n);
}
__device__ __forceinline__ double div_f64(double x, double n, double inv) {
  if (!has_inverse(inv)) return x / n;
  const double q = x * inv, r = fma(-q, n, x);
  return isfinite(r) ? fma(r, inv, q) : q;
}
// Shift of a feature, the same in both kernels: the previous mean to fp32 precision, 0 for an empty state.
__device__ __forceinline__ float stat_shift(double n, double inv, double s_mu) {
  return n > 0.0 ? div_f32(s_mu, n, inv) : 0.f;
}

// Eight consecutive features of a staged row as four packed pairs.
template <bool kBf16>
__device__ __forceinline__ void staged8(const uint8_t* row, int f, uint64_t (&x)[4]) {
  if (kBf16) {
    const uint4 u = *reinterpret_cast<const uint4*>(row + 16 * f);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      x[q] = (static_cast<uint64_t>(w[q] & 0xffff0000u) << 32) | static_cast<uint32_t>(w[q] << 16);
  } else {
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(row + 32 * f);
    const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(row + 32 * f + 16);
    x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
  }
}

// Block b sums rows [b T / G, (b+1) T / G). part: [G][4][d] = (s1_v, s2_v, s1_t, s2_t);
// nvis: [G] vision rows of the block, -1 after a wait that ran out; block 0 also keeps a copy of N_{t-1}
// for the finalize kernel (which overwrites N).
//
// Bound by HBM. Rows are contiguous, so one thread streams them into a ring of four 32 KB stages
// with bulk copies (up to 128 KB in flight per SM, against the 64 KB of register loads of two
// 256-thread blocks that stopped while they summed), and 512 threads sum: w / 8 threads per row
// (rounded to warps), the rows of a stage dealt to 512 / that groups, whose sums are added in group
// order at the end. Packed fp32 pairs: three instructions per two features.
// 131072 x 2048 bf16, both kernels: 150.6 -> 92.6 us (5.8 TB/s of X).
template <bool kBf16>
__global__ void __launch_bounds__(kStatThreads, 1) k_stats_partial(const StatsParams p) {
  extern __shared__ __align__(128) uint8_t st_smem[];
  __shared__ __align__(8) uint64_t full[kStatStages], empty[kStatStages];
  __shared__ int abort_flag, nv_s[kStatThreads / 32];
  __shared__ double n_s[2], inv_s[2];
  constexpr int es = kBf16 ? 2 : 4;
  uint8_t* ring = st_smem;
  float* merge = reinterpret_cast<float*>(st_smem + kStatStages * kStatStageBytes);
  uint8_t* lab = st_smem + kStatStages * kStatStageBytes + kStatMergeBytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = gridDim.x, b = blockIdx.x;
  const int r0 = static_cast<int>(static_cast<long long>(b) * p.T / G);
  const int r1 = static_cast<int>(static_cast<long long>(b + 1) * p.T / G);
  WaitCtx wc{&abort_flag, p.status, p.limit_ns};
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int i = 0; i < kStatStages; ++i) {
      mbar_init(full + i, 1);
      mbar_init(empty + i, kStatConsumers / 32);
    }
    fence_mbar_init();
  }
  pdl_wait();                                      // X and the state may be written just before
  pdl_trigger();
  int nv = 0;
  for (int i = threadIdx.x; i < r1 - r0; i += kStatThreads) {
    const uint8_t v = __ldg(p.is_vision + r0 + i);
    lab[i] = v;
    nv += v != 0;
  }
  nv = __reduce_add_sync(0xffffffffu, nv);
  if (lane == 0) nv_s[warp] = nv;
  if (threadIdx.x < 2) {
    const double n = p.N[threadIdx.x];
    n_s[threadIdx.x] = n;
    inv_s[threadIdx.x] = 1.0 / n;
  }
  __syncthreads();
  const int w_max = min(p.d, kStatCols);
  const int R = max(1, min(64, static_cast<int>(kStatStageBytes) / (w_max * es)));   // rows per stage

  if (warp == kStatConsumers / 32) {
    // ------------------------------------------------------------------ bulk copies
    if (lane == 0) {
      int t = 0;
      for (int w = 0; w < kStatThreads / 32; ++w) t += nv_s[w];
      p.nvis[b] = t;
      if (b == 0) {
        p.N0[0] = n_s[0];
        p.N0[1] = n_s[1];
      }
      bool ok = true;
      int st = 0;
      uint32_t ph = 0;
      long issued = 0;
      for (int c0 = 0; c0 < p.d && ok; c0 += kStatCols) {
        const int w = min(kStatCols, p.d - c0);
        for (int j0 = r0; j0 < r1; j0 += R) {
          const int nr = min(R, r1 - j0);
          if (!mbar_wait(empty + st, ph ^ 1u, wc)) { ok = false; break; }
          uint8_t* dst = ring + st * kStatStageBytes;
          const uint8_t* src = static_cast<const uint8_t*>(p.X) + (static_cast<size_t>(j0) * p.d + c0) * es;
          mbar_arrive_expect_tx(full + st, static_cast<uint32_t>(nr * w * es));
          if (w == p.d) {
            bulk_load(dst, src, static_cast<uint32_t>(nr * w * es), full + st);
          } else {                                 // a column slice: row by row
            for (int r = 0; r < nr; ++r)
              bulk_load(dst + r * w * es, src + static_cast<size_t>(r) * p.d * es, static_cast<uint32_t>(w * es), full + st);
          }
          ++issued;
          if (++st == kStatStages) { st = 0; ph ^= 1u; }
        }
      }
      WaitCtx wd = wc;                             // every issued copy lands before the block exits
      int dummy = 0;
      wd.abort_flag = &dummy;
      if (wd.limit_ns < kWaitLimitNs) wd.limit_ns = kWaitLimitNs;   // (whatever the plan's own limit)
      for (long q = (issued > kStatStages ? issued - kStatStages : 0); q < issued; ++q)
        mbar_wait(full + (q % kStatStages), static_cast<uint32_t>((q / kStatStages) & 1), wd);
    }
  } else {
    // ------------------------------------------------------------------ sums
    bool ok = true;                                // (every pass meets its barriers, also after a timeout)
    int st = 0;
    uint32_t ph = 0;
    for (int c0 = 0; c0 < p.d; c0 += kStatCols) {
      const int w = min(kStatCols, p.d - c0);
      const int tpr = (w / 8 + 31) & ~31;          // threads per row
      const int ng = kStatConsumers / tpr;         // row groups (at least two)
      const int g = threadIdx.x / tpr, f = threadIdx.x % tpr;
      const bool act = g < ng && 8 * f < w;
      for (int i = threadIdx.x; i < 2 * w; i += kStatConsumers) {     // the negated shifts [2][w]
        const int m = i >= w ? 1 : 0;
        merge[i] = -stat_shift(n_s[m], inv_s[m], p.S_mu[static_cast<size_t>(m) * p.d + c0 + i - m * w]);
      }
      named_bar(1, kStatConsumers);
      uint64_t sh[2][4], s1[2][4], s2[2][4];       // packed pairs
#pragma unroll
      for (int m = 0; m < 2; ++m) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          s1[m][q] = s2[m][q] = 0ull;
          sh[m][q] = act ? *reinterpret_cast<const uint64_t*>(merge + m * w + 8 * f + 2 * q) : 0ull;
        }
      }
      named_bar(1, kStatConsumers);                // merge is rewritten by the sums below
      const uint32_t row_bytes = static_cast<uint32_t>(w * es);
      for (int j0 = r0; j0 < r1; j0 += R) {
        const int nr = min(R, r1 - j0);
        if (!ok || !warp_wait(full + st, ph, wc)) { ok = false; break; }
        if (act) {
          const uint8_t* rows = ring + st * kStatStageBytes;
          const uint8_t* lb = lab + (j0 - r0);
#pragma unroll 4
          for (int r = g; r < nr; r += ng) {
            uint64_t x[4];
            staged8<kBf16>(rows + r * row_bytes, f, x);
            if (lb[r]) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const uint64_t dv = fadd2(x[q], sh[0][q]);
                s1[0][q] = fadd2(s1[0][q], dv);
                s2[0][q] = ffma2(dv, dv, s2[0][q]);
              }
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const uint64_t dv = fadd2(x[q], sh[1][q]);
                s1[1][q] = fadd2(s1[1][q], dv);
                s2[1][q] = ffma2(dv, dv, s2[1][q]);
              }
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + st);
        if (++st == kStatStages) { st = 0; ph ^= 1u; }
      }
      // the groups' sums through shared memory, added in group order
      if (act) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          ulonglong2* o1 = reinterpret_cast<ulonglong2*>(merge + (g * 4 + 2 * m) * w + 8 * f);
          ulonglong2* o2 = reinterpret_cast<ulonglong2*>(merge + (g * 4 + 2 * m + 1) * w + 8 * f);
          o1[0] = make_ulonglong2(s1[m][0], s1[m][1]);
          o1[1] = make_ulonglong2(s1[m][2], s1[m][3]);
          o2[0] = make_ulonglong2(s2[m][0], s2[m][1]);
          o2[1] = make_ulonglong2(s2[m][2], s2[m][3]);
        }
      }
      named_bar(1, kStatConsumers);
      if (ok) {
        float* out = p.part + static_cast<size_t>(b) * 4 * p.d;
        for (int i = threadIdx.x; i < w; i += kStatConsumers) {      // float4 i of the 4 w sums
          const int v = 4 * i / w, c = 4 * i - v * w;                // (w is a multiple of 8)
          float4 t = *reinterpret_cast<const float4*>(merge + v * w + c);
          for (int q = 1; q < ng; ++q) {
            const float4 u = *reinterpret_cast<const float4*>(merge + (q * 4 + v) * w + c);
            t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
          }
          *reinterpret_cast<float4*>(out + static_cast<size_t>(v) * p.d + c0 + c) = t;
        }
      }
      named_bar(1, kStatConsumers);                // merge is rewritten by the next pass
    }
  }
  // a block whose wait ran out has no sums: its count says so, and the state stays as it was
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0 && *wc.abort_flag) p.nvis[b] = -1;
}

// One (modality, feature) column per (block column, 16 slices): slice t sums the partials of
// blocks [t G / 16, (t+1) G / 16) in order (runs of 8 in fp32, the runs in fp64), the slices are
// added in slice order in fp64; then eqs. (5)-(7) in fp64. The counts |T_m| are integer sums of
// nvis. The state and the reciprocals that do not depend on the sums are formed while the partials
// are in flight: every fp64 division on the way is about a microsecond here.
constexpr int kFinSlices = 16;
constexpr int kFinCols = 32;

__global__ void __launch_bounds__(kFinSlices * kFinCols) k_stats_finalize(const StatsParams p) {
  __shared__ double red[2][kFinSlices][kFinCols];
  __shared__ double inv_n_s[2];
  __shared__ long long cnt_s;
  pdl_wait();                                     // the partials of k_stats_partial
  pdl_trigger();
  const int col = threadIdx.x % kFinCols, sl = threadIdx.x / kFinCols;
  const int i2 = blockIdx.x * kFinCols + col;     // m * d + i
  const int m = i2 < 2 * p.d ? i2 / p.d : 0;
  const int i = i2 < 2 * p.d ? i2 % p.d : 0;
  const int G = p.G;
  const size_t at = static_cast<size_t>(m) * p.d + i;
  double N0 = 0.0, Smu0 = 0.0, Svar0 = 0.0, inv_N0 = 0.0, mean0 = 0.0;
  if (sl == 0) {
    N0 = p.N0[m];
    Smu0 = p.S_mu[at];
    Svar0 = p.S_var[at];
  }
  // runs of 8 block partials added in fp32 (their loads issued together), the runs in fp64: GB300's
  // fp64 rate is a small fraction of its fp32 rate, and one fp64 add per partial set this
  // kernel's time
  double a1 = 0.0, a2 = 0.0;
  if (i2 < 2 * p.d) {
    const int g0 = sl * G / kFinSlices, g1 = (sl + 1) * G / kFinSlices;
    for (int g = g0; g < g1; g += 8) {
      float v1[8], v2[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool in = g + u < g1;
        const float* base = p.part + static_cast<size_t>(in ? g + u : g0) * 4 * p.d;
        v1[u] = in ? __ldcg(base + static_cast<size_t>(2 * m) * p.d + i) : 0.f;
        v2[u] = in ? __ldcg(base + static_cast<size_t>(2 * m + 1) * p.d + i) : 0.f;
      }
      float r1 = 0.f, r2 = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        r1 += v1[u];
        r2 += v2[u];
      }
      a1 += static_cast<double>(r1);
      a2 += static_cast<double>(r2);
    }
  }
  if (sl == kFinSlices - 1) {                     // |T_v|: integer counts, lanes stride the blocks
    int nvis = 0;
    bool out = false;                             // a block has no sums
    for (int g = col; g < G; g += 32) {
      nvis += p.nvis[g];
      out = out || p.nvis[g] < 0;
    }
    nvis = __reduce_add_sync(0xffffffffu, nvis);
    out = __any_sync(0xffffffffu, out);
    const int cnt = col == 0 ? nvis : p.T - nvis;
    if (col < 2) inv_n_s[col] = cnt > 0 ? 1.0 / cnt : 0.0;
    if (col == 0) cnt_s = out ? -1 : nvis;
  }
  if (sl == 0) {                                  // (one warp of the block: fp64 is scarce)
    inv_N0 = 1.0 / N0;
    mean0 = div_f64(Smu0, N0, inv_N0);             // S_mu,t-1 / N_t-1 (used when N0 > 0)
  }
  red[0][sl][col] = a1;
  red[1][sl][col] = a2;
  __syncthreads();
  if (sl != 0 || i2 >= 2 * p.d || cnt_s < 0) return;
  double s1 = 0.0, s2 = 0.0;
#pragma unroll
  for (int t = 0; t < kFinSlices; ++t) {
    s1 += red[0][t][col];
    s2 += red[1][t][col];
  }
  const double n = m == 0 ? static_cast<double>(cnt_s) : static_cast<double>(p.T - cnt_s);
  const double inv_n = inv_n_s[m];
  const double beta = p.beta;
  const double N1 = beta * N0 + n;                                    // eq. (5)
  double Smu1 = beta * Smu0, Svar1 = beta * Svar0;
  const double inv_N1 = 1.0 / N1;
  if (n > 0.0) {
    const double c = static_cast<double>(stat_shift(N0, inv_N0, Smu0));
    const double db = div_f64(s1, n, inv_n);                          // batch mean - c
    const double m2 = fmax(s2 - s1 * db, 0.0);                        // sum (x - mu_b)^2
    Smu1 += n * (c + db);                                             // eq. (6)
    Svar1 += m2;                                                      // eq. (7)
    if (N0 > 0.0) {
      const double dm = (c - mean0) + db;                             // mu_b - S_mu,t-1 / N_t-1
      Svar1 += dm * dm * div_f64(beta * N0 * n, N1, inv_N1);
    }
  }
  p.S_mu[at] = Smu1;
  p.S_var[at] = Svar1;
  if (i == 0) p.N[m] = N1;
  if (p.mu_out) p.mu_out[at] = div_f32(Smu1, N1, inv_N1);
  if (p.var_out) p.var_out[at] = div_f32(Svar1, N1, inv_N1);
}

// Eqs. (10)-(11) and the stable ascending rank of f_spec; one thread per expert.
__global__ void __launch_bounds__(kMaxExperts) k_adaptive_bins(const BinsParams p) {
  __shared__ double f_s[kMaxExperts];
  pdl_wait();                                     // this step's counts
  pdl_trigger();
  const int e = threadIdx.x;
  double f = 0.5;
  if (e < p.E) {
    const double w_old = p.beta, w_new = 1.0 - p.beta;
    const double cv = __dadd_rn(__dmul_rn(w_old, p.C_bar[e]),
                                __dmul_rn(w_new, static_cast<double>(p.counts[e])));
    const double ct = __dadd_rn(__dmul_rn(w_old, p.C_bar[p.E + e]),
                                __dmul_rn(w_new, static_cast<double>(p.counts[p.E + e])));
    p.C_bar[e] = cv;                                                  // eq. (10)
    p.C_bar[p.E + e] = ct;
    const double tot = __dadd_rn(ct, cv);
    f = tot > 0.0 ? __ddiv_rn(ct, tot) : 0.5;                        // eq. (11); 0/0 -> neutral
    f_s[e] = f;
    if (p.f_spec) p.f_spec[e] = f;
  }
  __syncthreads();
  if (e < p.E) {
    int rank = 0;
    for (int o = 0; o < p.E; ++o) {
      const double g = f_s[o];
      rank += (g < f || (g == f && o < e)) ? 1 : 0;
    }
    p.expert_bin[e] = rank / p.N_B;
  }
}

}  // namespace

// Blocks of the statistics pass: one per SM, at least 32 rows each (and at most kStatMaxRows).
int stats_blocks(int T, int n_sms) {
  const int by_rows = (T + 31) / 32, by_labels = (T + kStatMaxRows - 1) / kStatMaxRows;
  const int g = by_rows < n_sms ? by_rows : n_sms;
  return g > by_labels ? (g > 1 ? g : 1) : (by_labels > 1 ? by_labels : 1);
}

cudaError_t launch_stats_update(const StatsParams& p, bool bf16, cudaStream_t s) {
  auto k = bf16 ? k_stats_partial<true> : k_stats_partial<false>;
  const int rows = (p.T + p.G - 1) / p.G;                // the labels of a block's rows
  const size_t smem = kStatStages * kStatStageBytes + kStatMergeBytes + static_cast<size_t>(round_up(rows, 16));
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(k, dim3(p.G), dim3(kStatThreads), smem, s, p);
  if (e != cudaSuccess) return e;
  const int blocks = (2 * p.d + kFinCols - 1) / kFinCols;
  return launch_pdl(k_stats_finalize, dim3(blocks), dim3(kFinSlices * kFinCols), 0, s, p);
}

cudaError_t launch_adaptive_bins(const BinsParams& p, cudaStream_t s) {
  if (p.E < 1 || p.E > kMaxExperts) return cudaErrorInvalidValue;
  return launch_pdl(k_adaptive_bins, dim3(1), dim3(kMaxExperts), 0, s, p);
}

}  // namespace smoes
