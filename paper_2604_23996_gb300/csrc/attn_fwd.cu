// attn_fwd.cu -- attention forward that also yields the attention-accumulated vision score (eqs.
// 2-4): O = softmax(s Q K^T + bias) V per head, and per query the head average of the weights'
// product with the carried score m, in one pass. Grouped-query attention: K and V have H_kv heads;
// query head h reads key/value head h / (H / H_kv).
//
// A work item is (sequence, head, pair of adjacent 128-query tiles); the tiles share one stream of
// 128-key blocks. Roles: a TMA producer, an MMA issuer, a warp that stages the keys' bias and carried
// score, and four softmax groups of four warps, one per tile and half of a block's keys, a query row
// per thread. For each block S = Q K^T goes to tensor memory; the row's two threads exchange their
// maxima, form the weights and keep the normaliser l = sum 2^(x - max) and the vision mass
// a = sum 2^(x - max) m (fp32, packed pairs). The weights return to tensor memory as bf16 over the
// scores they came from and are the A operand of O += P V. The maximum in use is raised only when a
// block's maximum exceeds it by more than 8 (a factor of 2^8; then l, a and O are rescaled).
//
// Bound by a tile's chain S -> softmax -> P V, which the other tile's hides in part. With the weights
// in tensor memory no P tile takes shared memory, and S, P and O of two tiles fill the 512 columns. One
// tile per CTA, its weights in shared memory, had every step of a block wait for the one before: 8 x 16 x
// 4096 causal with H_kv = 4 took 1270 us, now 560 (607 before the converged issue). Groups of a whole
// row (128 keys per thread, half the warps) took 735 us with the scores in registers and 643 us reading
// them twice. A vote in the softmax warps' waits, as the other roles have: 566 us, 1 x 16 x 512 16.1 -> 17.3.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <atomic>

#include "device_common.cuh"
#include "ptx.cuh"
#include "smoes_internal.cuh"

namespace smoes {
namespace {

constexpr int kAttnTile = 128;                // queries per tile, keys per block
constexpr int kAttnHd = 128;                  // head dimension handled here
constexpr uint32_t kAttnTileBytes = kAttnTile * kAttnHd * 2;   // a Q tile, K or V block (2 swizzle atoms)

// 2^x on the special-function unit (flushes results below 2^-126 to zero).
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Work items of a persistent kernel, dealt to the CTAs in rounds of gridDim.x that alternate in
// direction: in round r CTA c takes item r * G + c when r is even and r * G + (G - 1 - c) when it
// is odd. With the items ordered longest first, each CTA's total stays within about one item of
// the mean, where a plain stride gives the low-numbered CTAs the longest item of every round.
__device__ __forceinline__ int dealt_item(int round) {
  const int g = static_cast<int>(gridDim.x), c = static_cast<int>(blockIdx.x);
  return round * g + ((round & 1) ? g - 1 - c : c);
}

// Bounded wait with its slow path out of line: the softmax warps keep the wait context in
// memory instead of in registers, which they need for the scores.
__device__ __noinline__ bool wait_slow(uint64_t* bar, uint32_t parity, const WaitCtx& w) {
  return mbar_wait(bar, parity, w);
}
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, const WaitCtx& w) {
  return mbar_try_wait(bar, parity) || wait_slow(bar, parity, w);
}

// Bounded wait of a whole warp that runs ahead of the softmax warps: it sleeps between tries, which
// would otherwise take issue slots from them (a third of all instructions). Every lane returns the
// same answer: full-warp shuffles and votes follow, and a lane that had left at the limit alone would
// leave the others in them for good.
__device__ __forceinline__ bool wait_idle(uint64_t* bar, uint32_t parity, const WaitCtx& w) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const uint64_t t0 = global_ns();
  while (true) {
    __nanosleep(100);
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const bool over = global_ns() - t0 > w.limit_ns;
    if (over) raise_abort(w, 2u);
    if (__any_sync(0xffffffffu, over || *w.abort_flag)) return false;
  }
}

// Work item -> (sequence b, head h, query-tile pair pr). Pairs run longest (last) first; within
// a pair index the heads of all sequences follow each other, so concurrent items share L2 keys.
struct AttnItem {
  int b, h, qt0, nq;          // first query tile, tiles in the pair (1 or 2)
};

template <int kTiles>       // query tiles per item: 2, or 1 (see the launch)
__device__ __forceinline__ AttnItem decode_item(const AttnParams& p, int item) {
  const int n_pairs = (p.n_qtiles + kTiles - 1) / kTiles;
  const int BH = p.B * p.H;
  const int pr = n_pairs - 1 - item / BH;
  const int bh = item - (item / BH) * BH;
  AttnItem it;
  it.b = bh / p.H;
  it.h = bh - it.b * p.H;
  it.qt0 = kTiles * pr;
  it.nq = min(kTiles, p.n_qtiles - it.qt0);
  return it;
}

// Key blocks query tile qt attends to.
__device__ __forceinline__ int kblocks_of(const AttnParams& p, int qt) {
  const int nk = (p.S + kAttnTile - 1) / kAttnTile;
  return p.causal ? min(qt + 1, nk) : nk;
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Largest bias (log2 units) that a chunk may add to its maximum's term instead of to every score. The
// maximum is rounded at the bias's size, so the exponents f x + (g - max) can come out above 0 by half
// an ulp of it: at most 64 below 2^31, far from overflow. A larger bias swallows the scores, as it does
// in 64 bits from about 2^53: added to each, all of its keys weigh the same.
constexpr float kMaxChunkBias = 2147483648.f;

// What the keys of a 32-key chunk share. Labels and biases come in runs (an image, its text,
// padding), so most chunks hold one value of each: then neither is read per key and thread (a
// broadcast 16-byte load takes four cycles of the SM's shared-memory port; two per four keys
// were half of the score kernel's time), the bias joins the maximum's term in the exponent and the
// mass is the chunk's sum of weights times the score.
struct alignas(16) KeyChunk {
  float bias, m;
  uint32_t one_bias, one_m;   // all keys of the chunk have that value
};

__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// 32 lanes x 64 columns: both loads in flight, waited for inside the statement (tying the registers
// to a separate wait cost a move per register).
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t (&r)[64]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%64];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%65];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]),
        "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]),
        "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]),
        "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
        "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]),
        "=r"(r[63])
      : "r"(taddr), "r"(taddr + 32u)
      : "memory");
}
// 32 lanes x 16 columns from registers, not waited for.
__device__ __forceinline__ void tmem_st16_async(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]: A as 128 lanes (rows) of packed bf16 pairs along K.
__device__ __forceinline__ void umma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

constexpr float kRescale = 8.f;                // raise the maximum in use only past +2^8
constexpr int kHalf = kAttnTile / 2;           // keys of a block per softmax group

// Softmax groups: four of four warps, one per query tile and half of a block's keys, a query row
// per thread. Four warps per scheduler hide each other's tensor-memory loads and barrier waits: two
// groups with a row's 128 keys per thread ran at 0.42 instructions per cycle.
constexpr int kAttnThreads = 128 + 4 * 128;    // producer, MMA issuer, key terms, an idle warp, the groups
// The launch's 640 x 96 registers dealt anew: 56 for the first four warps, 104 for the softmax warps
// (128 x 56 + 512 x 104 = 60416 of 61440). setmaxnreg.inc waits without a limit for registers that the
// launch does not hold, so the launch is refused if the kernel was compiled to fewer.
constexpr int kFewerRegisters = 56, kMoreRegisters = 104;
constexpr int kDealtRegisters = 128 * kFewerRegisters + (kAttnThreads - 128) * kMoreRegisters;
__device__ __forceinline__ void attn_fewer_registers() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFewerRegisters)); }
__device__ __forceinline__ void attn_more_registers() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kMoreRegisters)); }

constexpr int kKtBlocks = 4;                   // key blocks per stage of key terms
constexpr int kKtStages = 2;
constexpr int kKtKeys = kKtBlocks * kAttnTile;
constexpr int kKtFloats = 2 * kKtKeys + kKtKeys / 32 * 4;   // bias * log2 e | carried score | chunks

// The warp that stages (bias * log2 e, carried score) of the keys, four blocks at a time, keys past
// S masked; loaded a stage ahead. kt: the stages, [kKtStages][kKtFloats]; full has count 32.
template <bool kFloatM, int kTiles>
__device__ __forceinline__ void stage_key_terms(const AttnParams& p, int n_items, float* kt, uint64_t* kt_full,
                                                uint64_t* kt_empty, const WaitCtx& wc) {
  constexpr int kN = kKtKeys / 32;
  const int lane = threadIdx.x & 31;
  bool ok = true;
  int st = 0;
  uint32_t ph = 0;
  for (int rd = 0; ok; ++rd) {
    const int item = dealt_item(rd);
    if (item >= n_items) break;
    const AttnItem w = decode_item<kTiles>(p, item);
    const int nkb = kblocks_of(p, w.qt0 + w.nq - 1);
    for (int kb = 0; kb < nkb; kb += kKtBlocks) {
      float b[kN], m[kN];
#pragma unroll
      for (int i = 0; i < kN; ++i) {
        const int key = kb * kAttnTile + 32 * i + lane;
        b[i] = -CUDART_INF_F;
        m[i] = 0.f;
        if (key < p.S) {
          const size_t tk = static_cast<size_t>(w.b) * p.S + key;
          b[i] = p.key_bias ? __ldg(p.key_bias + tk) * 1.4426950408889634f : 0.f;
          m[i] = kFloatM ? __ldg(p.m_prev + tk) : static_cast<float>(__ldg(p.is_vision + tk) != 0);
        }
      }
      if (!wait_idle(kt_empty + st, ph ^ 1u, wc)) { ok = false; break; }
      float* d = kt + st * kKtFloats;
      KeyChunk* ch = reinterpret_cast<KeyChunk*>(d + 2 * kKtKeys);
#pragma unroll
      for (int i = 0; i < kN; ++i) {
        d[32 * i + lane] = b[i];
        d[kKtKeys + 32 * i + lane] = m[i];
        KeyChunk c;
        c.bias = __shfl_sync(0xffffffffu, b[i], 0);
        c.m = __shfl_sync(0xffffffffu, m[i], 0);
        // (the maximum is then taken over the raw products: their factor has to be positive)
        const bool fits = fabsf(b[i]) < kMaxChunkBias || b[i] == -CUDART_INF_F;
        c.one_bias = __all_sync(0xffffffffu, fits && __float_as_uint(b[i]) == __float_as_uint(c.bias)) && p.scale_log2 > 0.f;
        c.one_m = __all_sync(0xffffffffu, __float_as_uint(m[i]) == __float_as_uint(c.m));
        if (lane == 0) ch[i] = c;
      }
      mbar_arrive(kt_full + st);
      if (++st == kKtStages) { st = 0; ph ^= 1u; }
    }
  }
}

// The half block's terms of a thread's 64 keys inside a stage of key terms (shared addresses).
struct HalfTerms {
  uint32_t bias, m, chunk;
};
__device__ __forceinline__ HalfTerms half_terms(const float* stage, int kb, int hf) {
  const uint32_t s = smem_u32(stage);
  const uint32_t k0 = static_cast<uint32_t>((kb % kKtBlocks) * kAttnTile + kHalf * hf);
  return HalfTerms{s + k0 * 4u, s + (kKtKeys + k0) * 4u, s + 2u * kKtKeys * 4u + k0 / 32u * 16u};
}
__device__ __forceinline__ KeyChunk key_chunk(const HalfTerms& h, int c) {
  const ulonglong2 v = lds_u64x2(h.chunk + 16u * c);
  KeyChunk k;
  k.bias = lo2(v.x);
  k.m = hi2(v.x);
  k.one_bias = static_cast<uint32_t>(v.y);
  k.one_m = static_cast<uint32_t>(v.y >> 32);
  return k;
}

// A row's 64 scores from tensor memory, as pairs x of f x + g per 32-key chunk (log2 units; f = 1 and
// g = 0 where biases are added key by key), keys above the diagonal masked (first_masked: the first
// one, 64 for none); returns their maximum. Factors are packed once: packed anew at every use they
// cost a move per score.
__device__ __forceinline__ float load_scores(uint32_t ts, const HalfTerms& h, float sc, int first_masked,
                                             uint64_t (&x)[kHalf / 2], uint64_t& f2, float (&g)[2]) {
  uint32_t r[64];
  __syncwarp();
  const KeyChunk ca = key_chunk(h, 0), cb = key_chunk(h, 1);
  tmem_ld64(ts, r);
#pragma unroll
  for (int i = 0; i < 32; ++i) x[i] = (static_cast<uint64_t>(r[2 * i + 1]) << 32) | r[2 * i];
  float f = sc;
  g[0] = ca.bias;
  g[1] = cb.bias;
  if (!(ca.one_bias && cb.one_bias)) {
    const uint64_t sc2 = pack2(sc, sc);
#pragma unroll
    for (int i4 = 0; i4 < kHalf / 4; ++i4) {
      const ulonglong2 bb = lds_u64x2(h.bias + 16u * i4);
      x[2 * i4] = ffma2(x[2 * i4], sc2, bb.x);
      x[2 * i4 + 1] = ffma2(x[2 * i4 + 1], sc2, bb.y);
    }
    f = 1.f;
    g[0] = g[1] = 0.f;
  }
  f2 = pack2(f, f);
  if (first_masked < kHalf) {
#pragma unroll
    for (int i = 0; i < kHalf / 2; ++i)
      x[i] = pack2(2 * i >= first_masked ? -CUDART_INF_F : lo2(x[i]), 2 * i + 1 >= first_masked ? -CUDART_INF_F : hi2(x[i]));
  }
  float mx[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const uint64_t* e = x + 16 * c;
    float c0 = fmaxf(lo2(e[0]), hi2(e[0])), c1 = fmaxf(lo2(e[1]), hi2(e[1]));
#pragma unroll
    for (int i = 2; i < 16; i += 2) {
      c0 = max3(c0, lo2(e[i]), hi2(e[i]));
      c1 = max3(c1, lo2(e[i + 1]), hi2(e[i + 1]));
    }
    mx[c] = fmaf(fmaxf(c0, c1), f, g[c]);
  }
  return fmaxf(mx[0], mx[1]);
}

// x becomes the weights 2^(f x + g - max in use) (nm: the negated maximum, 0 while every key is
// masked); their sum joins l, their product with the carried score a.
__device__ __forceinline__ void weigh(uint64_t (&x)[kHalf / 2], uint64_t f2, const float (&g)[2], float nm,
                                      const HalfTerms& h, float& l, float& a) {
  float sum[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const uint64_t gm2 = pack2(g[c] + nm, g[c] + nm);
    uint64_t s0 = 0ull, s1 = 0ull;
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      uint64_t* e = x + 16 * c + i;
      e[0] = ffma2(e[0], f2, gm2);
      e[1] = ffma2(e[1], f2, gm2);
      e[0] = pack2(ex2(lo2(e[0])), ex2(hi2(e[0])));
      e[1] = pack2(ex2(lo2(e[1])), ex2(hi2(e[1])));
      s0 = fadd2(s0, e[0]);
      s1 = fadd2(s1, e[1]);
    }
    s0 = fadd2(s0, s1);
    sum[c] = lo2(s0) + hi2(s0);
  }
  l += sum[0] + sum[1];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const KeyChunk kc = key_chunk(h, c);
    if (kc.one_m) {
      a = fmaf(kc.m, sum[c], a);
    } else {
      uint64_t a0 = 0ull, a1 = 0ull;
#pragma unroll
      for (int i4 = 0; i4 < 8; ++i4) {
        const ulonglong2 mm = lds_u64x2(h.m + 16u * (c * 8 + i4));
        a0 = ffma2(x[16 * c + 2 * i4], mm.x, a0);
        a1 = ffma2(x[16 * c + 2 * i4 + 1], mm.y, a1);
      }
      a0 = fadd2(a0, a1);
      a += lo2(a0) + hi2(a0);
    }
  }
}

constexpr int kKStages = 2, kVStages = 2;      // K and V blocks in flight

struct AttnLayout {
  uint32_t q, k, v, kt, mx, mrg, bars, total;
};
__host__ __device__ inline AttnLayout attn_layout() {
  AttnLayout L;
  uint32_t o = 0;
  L.q = o;    o += 2u * kAttnTileBytes;
  L.k = o;    o += kKStages * kAttnTileBytes;
  L.v = o;    o += kVStages * kAttnTileBytes;
  L.kt = o;   o += kKtStages * kKtFloats * 4u;             // the keys' terms
  L.mx = o;   o += 2u * 2u * 2u * kAttnTile * 4u;          // row maxima: tile x block parity x half
  L.mrg = o;  o += 2u * 2u * 2u * 2u * kAttnTile * 4u;     // (l, a) of a half: tile x item parity x half
  L.bars = o; o += 8u * 64u;
  L.total = o + 1024u;
  return L;
}

// M of a token from its heads' scores, in head order (eq. 3), optionally blended with the carried
// score (eq. 4).
__device__ __forceinline__ void average_heads(const AttnParams& p, int tok) {
  float sum = 0.f;
#pragma unroll 8
  for (int hh = 0; hh < p.H; ++hh) sum += __ldcg(p.part + static_cast<size_t>(hh) * p.T + tok);
  float mv = sum / static_cast<float>(p.H);
  if (p.xattn_norm) {
    const float an = __ldg(p.xattn_norm + tok), rn = __ldg(p.x_norm + tok);
    const float mprev = p.m_prev ? __ldg(p.m_prev + tok) : static_cast<float>(__ldg(p.is_vision + tok) != 0);
    mv = (an * mv + rn * mprev) / (an + rn);
  }
  reinterpret_cast<float2*>(p.M)[tok] = make_float2(mv, 1.f - mv);
}

template <bool kFloatM, int kTiles>
__global__ void __launch_bounds__(kAttnThreads, 1)
k_attn_fwd(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
           const __grid_constant__ CUtensorMap tmV, const AttnFwdParams fp) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const AttnParams& p = fp.a;
  const AttnLayout L = attn_layout();
  uint8_t* qs = base + L.q;
  uint8_t* ks = base + L.k;
  uint8_t* vs = base + L.v;
  float* kt = reinterpret_cast<float*>(base + L.kt);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + L.bars);
  uint64_t* q_full = bars;            // [2] per tile of the pair
  uint64_t* q_empty = bars + 2;       // [2] the item's last S has read Q
  uint64_t* k_full = bars + 4;        // [kKStages]
  uint64_t* k_empty = bars + 6;
  uint64_t* v_full = bars + 8;        // [kVStages]
  uint64_t* v_empty = bars + 10;
  uint64_t* kt_full = bars + 12;      // [kKtStages] count 32
  uint64_t* kt_empty = bars + 14;     // [kKtStages] count 16: a lane of every softmax warp
  uint64_t* s_full = bars + 16;       // [2] the tile's scores are in tensor memory
  uint64_t* mx_bar = bars + 18;       // [2] count 256: both halves' row maxima are written
  uint64_t* p_full = bars + 20;       // [tile][half] count 128: 64 keys' weights are in tensor memory; half 0's
                                      // also counts both halves' rescales of O (count 384)
  uint64_t* o_full = bars + 24;       // [2] the item's last P V has completed
  uint64_t* o_empty = bars + 26;      // [2] count 256: O has been read
  uint64_t* mrg_bar = bars + 28;      // [2] count 256: both halves' sums are written
  uint64_t* drain = bars + 30;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 31);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  int* last_head = abort_flag + 1;    // this CTA's head was its tile's last
  float* mxs = reinterpret_cast<float*>(base + L.mx);
  float* mrg = reinterpret_cast<float*>(base + L.mrg);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int n_items = ((p.n_qtiles + kTiles - 1) / kTiles) * p.B * p.H;
  WaitCtx wc{abort_flag, p.status, p.limit_ns};
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    for (int t = 0; t < 2; ++t) {
      mbar_init(q_full + t, 1);
      mbar_init(q_empty + t, 1);
      mbar_init(k_full + t, 1);
      mbar_init(k_empty + t, 1);
      mbar_init(v_full + t, 1);
      mbar_init(v_empty + t, 1);
      mbar_init(s_full + t, 1);
      mbar_init(p_full + 2 * t, 384);
      mbar_init(p_full + 2 * t + 1, 128);
      mbar_init(o_full + t, 1);
      mbar_init(o_empty + t, 256);
      mbar_init(mx_bar + t, 256);
      mbar_init(mrg_bar + t, 256);
    }
    for (int i = 0; i < kKtStages; ++i) {
      mbar_init(kt_full + i, 32);
      mbar_init(kt_empty + i, 16);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;    // S and P of the tiles at columns 0 and 128, O at 256 and 384
  pdl_wait();                          // inputs and outputs may be in use before this
  pdl_trigger();
  if (warp < 4) attn_fewer_registers();

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    {
      const int G = p.H / fp.Hkv;         // query heads per key/value head
      int st = 0, vst = 0;
      uint32_t ph = 0, vph = 0;
      int nqt[2] = {0, 0};              // items that used Q buffer t: its barrier phase
      long nk = 0, nv = 0;
      bool ok = true;
      for (int rd = 0; ok; ++rd) {
        const int item = dealt_item(rd);
        if (item >= n_items) break;
        const AttnItem w = decode_item<kTiles>(p, item);
        const int row0 = (w.b * p.H + w.h) * p.S, krow0 = (w.b * fp.Hkv + w.h / G) * p.S;
        for (int t = 0; t < w.nq && ok; ++t) {
          if (!warp_wait(q_empty + t, (static_cast<uint32_t>(nqt[t]) & 1u) ^ 1u, wc)) { ok = false; break; }
          ++nqt[t];
          if (elect_one()) {
            mbar_arrive_expect_tx(q_full + t, kAttnTileBytes);
            uint8_t* qd = qs + t * kAttnTileBytes;
            tma_load_2d(qd, &tmQ, q_full + t, 0, row0 + (w.qt0 + t) * kAttnTile);
            tma_load_2d(qd + kAttnTileBytes / 2, &tmQ, q_full + t, 64, row0 + (w.qt0 + t) * kAttnTile);
          }
          __syncwarp();
        }
        const int nkb = kblocks_of(p, w.qt0 + w.nq - 1);
        for (int kb = 0; kb < nkb && ok; ++kb) {
          if (!warp_wait(k_empty + st, ph ^ 1u, wc)) { ok = false; break; }
          if (elect_one()) {
            uint8_t* kd = ks + st * kAttnTileBytes;
            mbar_arrive_expect_tx(k_full + st, kAttnTileBytes);
            tma_load_2d(kd, &tmK, k_full + st, 0, krow0 + kb * kAttnTile);
            tma_load_2d(kd + kAttnTileBytes / 2, &tmK, k_full + st, 64, krow0 + kb * kAttnTile);
          }
          __syncwarp();
          ++nk;
          if (++st == kKStages) { st = 0; ph ^= 1u; }
          if (!warp_wait(v_empty + vst, vph ^ 1u, wc)) { ok = false; break; }
          if (elect_one()) {
            uint8_t* vd = vs + vst * kAttnTileBytes;
            mbar_arrive_expect_tx(v_full + vst, kAttnTileBytes);
            tma_load_2d(vd, &tmV, v_full + vst, 0, krow0 + kb * kAttnTile);
            tma_load_2d(vd + kAttnTileBytes / 2, &tmV, v_full + vst, 64, krow0 + kb * kAttnTile);
          }
          __syncwarp();
          ++nv;
          if (++vst == kVStages) { vst = 0; vph ^= 1u; }
        }
      }
      WaitCtx wd = wc;                  // every issued copy lands before the CTA may exit
      int dummy = 0;
      wd.abort_flag = &dummy;
      for (long q = (nk > kKStages ? nk - kKStages : 0); q < nk; ++q)
        mbar_wait(k_full + (q % kKStages), static_cast<uint32_t>((q / kKStages) & 1), wd);
      for (long q = (nv > kVStages ? nv - kVStages : 0); q < nv; ++q)
        mbar_wait(v_full + (q % kVStages), static_cast<uint32_t>((q / kVStages) & 1), wd);
      for (int t = 0; t < 2; ++t)
        if (nqt[t] > 0) mbar_wait(q_full + t, static_cast<uint32_t>(nqt[t] - 1) & 1u, wd);
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    {
      const uint32_t id_s = idesc_bf16(kAttnTile, kAttnTile, false, false);   // S = Q K^T (both K-major)
      const uint32_t id_o = idesc_bf16(kAttnTile, kAttnHd, false, true);      // O += P V (V MN-major)
      int st = 0, vst = 0;
      uint32_t ph = 0, vph = 0;
      int blk[2] = {0, 0};              // blocks of the tile so far: its score buffer and phases
      int nqt[2] = {0, 0};              // items of the tile so far
      bool ok = true;
      for (int rd = 0; ok; ++rd) {
        const int item = dealt_item(rd);
        if (item >= n_items) break;
        const AttnItem w = decode_item<kTiles>(p, item);
        int nb[2];
        nb[0] = kblocks_of(p, w.qt0);
        nb[1] = w.nq > 1 ? kblocks_of(p, w.qt0 + 1) : 0;
        const int nkb = nb[w.nq - 1];
        // slot j: for each tile O += P_{j-1} V_{j-1} (in two halves, as the weights arrive), then S_j
        // over the weights it has read (the MMAs of one thread run in order); the other tile's
        // softmax runs meanwhile
        for (int j = 0; j <= nkb && ok; ++j) {
          if (j < nkb && !warp_wait(k_full + st, ph, wc)) { ok = false; break; }
          if (j > 0 && !warp_wait(v_full + vst, vph, wc)) { ok = false; break; }
          for (int t = 0; t < w.nq && ok; ++t) {
            const uint32_t ts = tmem + static_cast<uint32_t>(t * kAttnTile);   // S, then P
            if (j > 0 && j <= nb[t]) {
              const uint32_t d = tmem + 256u + static_cast<uint32_t>(t * kAttnHd);
              const uint32_t vb = smem_u32(vs + vst * kAttnTileBytes);
              for (int hf = 0; hf < 2; ++hf) {
                if (!warp_wait(p_full + 2 * t + hf, static_cast<uint32_t>(blk[t] - 1) & 1u, wc)) { ok = false; break; }
                if (j == 1 && hf == 0 && !warp_wait(o_empty + t, (static_cast<uint32_t>(nqt[t] - 1) & 1u) ^ 1u, wc)) { ok = false; break; }
                tc_fence_after();
                if (elect_one()) {
#pragma unroll
                  for (int k4 = 0; k4 < 4; ++k4) {           // K = 16 keys per step
                    const int kk = 4 * hf + k4;
                    umma_bf16_ta(d, ts + 8u * kk, sdesc_sw128(vb + kk * 2048, kAttnTileBytes / 2, 1024), id_o,
                                 (j > 1 || kk > 0) ? 1u : 0u);
                  }
                  if (hf == 1 && j == nb[t]) umma_commit(o_full + t);
                }
                __syncwarp();
              }
              if (!ok) break;
            }
            if (j < nb[t]) {
              if (j == 0 && !warp_wait(q_full + t, static_cast<uint32_t>(nqt[t]++) & 1u, wc)) { ok = false; break; }
              tc_fence_after();
              const uint32_t qa = smem_u32(qs + t * kAttnTileBytes), kb = smem_u32(ks + st * kAttnTileBytes);
              if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < kAttnHd / 16; ++kk) {  // K = 16 of the head dimension per step
                  const uint32_t off = (kk >> 2) * (kAttnTileBytes / 2) + (kk & 3) * 32;
                  umma_bf16(ts, sdesc_sw128(qa + off, 16, 1024), sdesc_sw128(kb + off, 16, 1024), id_s, kk > 0 ? 1u : 0u);
                }
                umma_commit(s_full + t);
                if (j == nb[t] - 1) umma_commit(q_empty + t);  // Q may be replaced
              }
              __syncwarp();
              ++blk[t];
            }
          }
          if (!ok) break;
          if (j > 0) {
            if (elect_one()) umma_commit(v_empty + vst);
            __syncwarp();
            if (++vst == kVStages) { vst = 0; vph ^= 1u; }
          }
          if (j < nkb) {
            if (elect_one()) umma_commit(k_empty + st);
            __syncwarp();
            if (++st == kKStages) { st = 0; ph ^= 1u; }
          }
        }
      }
      if (elect_one()) umma_commit(drain);               // every issued MMA completes before TMEM is released
      WaitCtx wd = wc;
      int dummy = 0;
      wd.abort_flag = &dummy;
      mbar_wait(drain, 0, wd);
    }
  } else if (warp == 2) {
    stage_key_terms<kFloatM, kTiles>(p, n_items, kt, kt_full, kt_empty, wc);
  } else if (warp >= 4) {
    // ---------------------------------------------------------------- softmax groups (4 x 4 warps)
    attn_more_registers();
    const int grp = (warp - 4) >> 2;
    const int t = grp & 1;                     // query tile of the pair
    const int hf = grp >> 1;                   // half of each key block: keys [64 hf, 64 hf + 64)
    const int lg = warp & 3;                   // TMEM lane quarter of this warp
    const int row = lg * 32 + lane;            // query row of the tile == TMEM lane
    const uint32_t lane_off = static_cast<uint32_t>(lg * 32) << 16;
    const uint32_t ts = tmem + lane_off + static_cast<uint32_t>(t * kAttnTile);            // S, then P
    const uint32_t to = tmem + lane_off + 256u + static_cast<uint32_t>(t * kAttnHd + kHalf * hf);   // this half of O
    float* mxt = mxs + t * 4 * kAttnTile;      // [block parity][half][128]
    float* mrt = mrg + t * 8 * kAttnTile;      // [item parity][half][l | a][128]
    const float sc = p.scale_log2;
    int blk = 0, ng = 0, st = 0;
    uint32_t kph = 0;
    bool ok = true;
    for (int rd = 0; ok; ++rd) {
      const int item = dealt_item(rd);
      if (item >= n_items) break;
      const AttnItem w = decode_item<kTiles>(p, item);
      const int qt = w.qt0 + t;
      const int nkb = kblocks_of(p, w.qt0 + w.nq - 1);
      const int mine = t < w.nq ? kblocks_of(p, qt) : 0;
      float m_used = -CUDART_INF_F, l = 0.f, a = 0.f;
      for (int kb = 0; kb < nkb; ++kb) {
        if (kb % kKtBlocks == 0 && !wait_bar(kt_full + st, kph, wc)) { ok = false; break; }
        if (kb < mine) {
          const uint32_t bph = static_cast<uint32_t>(blk) & 1u;
          if (!wait_bar(s_full + t, bph, wc)) { ok = false; break; }
          ++blk;
          tc_fence_after();
          const HalfTerms h = half_terms(kt + st * kKtFloats, kb, hf);
          uint64_t x[kHalf / 2], f2;
          float g[2];
          const float mx = load_scores(ts + static_cast<uint32_t>(kHalf * hf), h, sc,
                                       p.causal && kb == qt ? row + 1 - kHalf * hf : kHalf, x, f2, g);
          // the row's maximum over both halves; past this exchange both have their scores in
          // registers, so the weights may overwrite them
          tc_fence_before();
          mxt[(bph * 2 + hf) * kAttnTile + row] = mx;
          mbar_arrive(mx_bar + t);
          if (!wait_bar(mx_bar + t, bph, wc)) { ok = false; break; }
          tc_fence_after();
          const float m_new = fmaxf(m_used, fmaxf(mx, mxt[(bph * 2 + (hf ^ 1)) * kAttnTile + row]));
          const bool raise = kb == 0 || m_new > m_used + kRescale;
          if (__any_sync(0xffffffffu, raise && kb > 0)) {    // rescale l, a and this half of O (rare)
            const float alpha = (raise && kb > 0) ? (m_used == -CUDART_INF_F ? 0.f : ex2(m_used - m_new)) : 1.f;
            l *= alpha;
            a *= alpha;
            // (S_j follows the tile's P V of block j - 1)
#pragma unroll 1
            for (int c = 0; c < kHalf / 16; ++c) {
              float v[16];
              tmem_ld16(to + 16u * c, v);
              uint32_t u[16];
#pragma unroll
              for (int q = 0; q < 16; ++q) u[q] = __float_as_uint(v[q] * alpha);
              tmem_st16_async(to + 16u * c, u);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          }
          // Each half rescales its own 64 columns of O, but the products of either half's weights add to
          // all 128. Half 0's are issued first, on p_full[2 t], so both halves arrive there with their
          // rescale done (or none needed): no product of block j reaches O before both rescales of
          // block j. The arrival comes a weigh() ahead of half 0's own, so the MMA warp waits no longer
          // for it. No thread can arrive for block j + 1 in the phase of block j: the scores of j + 1
          // are issued after these products. (Block 0 has no rescale and is counted alike.)
          tc_fence_before();
          mbar_arrive(p_full + 2 * t);
          if (raise) m_used = m_new;
          // weights, in bf16 to the half's 32 columns of P; a row whose keys are all masked so far
          // has weights 0
          weigh(x, f2, g, m_used == -CUDART_INF_F ? 0.f : -m_used, h, l, a);
          __syncwarp();
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) pk[i] = cvt_bf16x2(lo2(x[16 * c + i]), hi2(x[16 * c + i]));
            tmem_st16_async(ts + static_cast<uint32_t>(32 * hf + 16 * c), pk);
          }
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          tc_fence_before();
          mbar_arrive(p_full + 2 * t + hf);
        }
        if (kb % kKtBlocks == kKtBlocks - 1 || kb == nkb - 1) {
          __syncwarp();
          if (lane == 0) mbar_arrive(kt_empty + st);
          if (++st == kKtStages) { st = 0; kph ^= 1u; }
        }
      }
      if (!ok) break;
      if (mine == 0) continue;
      const uint32_t nt = static_cast<uint32_t>(ng++);     // this item's phase of the tile's barriers
      const int q = qt * kAttnTile + row;                  // query position in the sequence
      // both halves' sums (the maximum in use is the same)
      float* mb = mrt + (nt & 1u) * 4 * kAttnTile;
      mb[hf * 2 * kAttnTile + row] = l;
      mb[(hf * 2 + 1) * kAttnTile + row] = a;
      mbar_arrive(mrg_bar + t);
      if (!wait_bar(mrg_bar + t, nt & 1u, wc)) break;
      l = mb[row] + mb[2 * kAttnTile + row];               // in key order, the same in both halves
      const float il = 1.f / l;
      if (hf == 0)                                         // head result
        p.part[static_cast<size_t>(w.h) * p.T + static_cast<size_t>(w.b) * p.S + q] = (a + mb[3 * kAttnTile + row]) * il;
      // O / l: half a row per thread
      if (!wait_bar(o_full + t, nt & 1u, wc)) break;
      tc_fence_after();
      uint4* orow = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(fp.O) +
                                             ((static_cast<size_t>(w.b) * p.H + w.h) * p.S + q) * kAttnHd + kHalf * hf);
#pragma unroll 1
      for (int c = 0; c < kHalf / 32; ++c) {
        float v[32];
        tmem_ld32(to + 32u * c, v);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          orow[4 * c + u] = make_uint4(cvt_bf16x2(v[8 * u] * il, v[8 * u + 1] * il), cvt_bf16x2(v[8 * u + 2] * il, v[8 * u + 3] * il),
                                       cvt_bf16x2(v[8 * u + 4] * il, v[8 * u + 5] * il), cvt_bf16x2(v[8 * u + 6] * il, v[8 * u + 7] * il));
      }
      tc_fence_before();
      mbar_arrive(o_empty + t);
    }
    // One item per CTA: the tile's last head averages the heads here, in the warps that wrote this
    // head's scores. Reached on every path out of the loop, so the barriers complete and the ticket
    // is zero again for the next call also after a wait that ran out. With a second launch instead,
    // eager calls of 1 x 8 x 128 (3000 in a row), which the host bounds, take 12.0-13.8 us against
    // 9.9-11.1 (10.1-11.7 before this kernel had two tiles per item); in a graph the ticket costs 0.3 us
    // of 8.1 there and 0.1 of 15.6 at 1 x 16 x 512 (9.3 and 17.1 before).
    if (kTiles == 1 && grp == 0) {
      const AttnItem w = decode_item<kTiles>(p, dealt_item(0));
      __syncwarp();
      named_bar(1, 128);
      if (row == 0) {
        uint32_t* ticket = p.ticket + w.b * p.n_qtiles + w.qt0;
        __threadfence();                       // the four warps' scores, ordered before it by the barrier
        const bool last = atomicAdd(ticket, 1u) + 1u == static_cast<uint32_t>(p.H);
        if (last) *ticket = 0u;
        __threadfence();
        *last_head = last ? 1 : 0;
      }
      named_bar(1, 128);
      if (*last_head) average_heads(p, w.b * p.S + w.qt0 * kAttnTile + row);
    }
  }

  // the role branches leave single lanes running on their own: the warp reconverges before
  // the block barrier, so that no thread passes it while another of its warp is still working
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// The heads' average of a call with more tiles than SMs: a ticket per (sequence, query tile) taken at
// the end of every item instead, with its fences, stopped the CTA for microseconds between items:
// 639 -> 607 us on 8 x 16 x 4096, 71 -> 56 us on 16 x 32 x 256.
__global__ void __launch_bounds__(256) k_attn_average(const AttnParams p) {
  pdl_wait();                                  // the heads' scores of the kernel just before
  pdl_trigger();
  const int tok = blockIdx.x * 256 + threadIdx.x;
  if (tok < p.T) average_heads(p, tok);
}

}  // namespace

cudaError_t launch_attn_fwd(const AttnFwdParams& fp, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                            const CUtensorMap& tmV, int n_sms, cudaStream_t s) {
  const AttnParams& p = fp.a;
  if (p.hd != kAttnHd || p.S % kAttnTile != 0 || fp.Hkv < 1 || p.H % fp.Hkv != 0) return cudaErrorNotSupported;
  const uint32_t smem = attn_layout().total;
  // one tile per item while every tile has an SM to itself: a pair's blocks take longer than one
  // tile's (1 x 16 x 512: 20.1 against 16.6 us)
  const int tiles = p.n_qtiles * p.B * p.H;
  const bool single = tiles <= n_sms;
  const int n_items = single ? tiles : ((p.n_qtiles + 1) / 2) * p.B * p.H;
  const int grid = n_items < n_sms ? n_items : n_sms;
  auto launch = [&](auto k, std::atomic<int>& regs) -> cudaError_t {
    int held = regs.load(std::memory_order_relaxed);    // a constant of the build, asked for once
    if (held == 0) {
      cudaFuncAttributes fa;
      const cudaError_t e = cudaFuncGetAttributes(&fa, k);
      if (e != cudaSuccess) return e;
      regs.store(held = fa.numRegs, std::memory_order_relaxed);
    }
    if (held * kAttnThreads < kDealtRegisters) return cudaErrorInvalidConfiguration;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e != cudaSuccess ? e : launch_pdl(k, dim3(grid), dim3(kAttnThreads), smem, s, tmQ, tmK, tmV, fp);
  };
  static std::atomic<int> regs[4];
  const cudaError_t e = p.m_prev ? (single ? launch(k_attn_fwd<true, 1>, regs[0]) : launch(k_attn_fwd<true, 2>, regs[1]))
                                 : (single ? launch(k_attn_fwd<false, 1>, regs[2]) : launch(k_attn_fwd<false, 2>, regs[3]));
  if (e != cudaSuccess || single) return e;   // (one item per CTA: averaged by its last head)
  return launch_pdl(k_attn_average, dim3((p.T + 255) / 256), dim3(256), 0, s, p);
}

}  // namespace smoes
