// a5: decode attention straight from the NVFP4 KV cache (Sec. 2.1:
// z = softmax(Q K_hat^T / sqrt(d)) V_hat with quantized K and V).
//
// Split-KV ("flash-decoding").  The cached tokens of all sequences and KV heads
// are one list of 128-token stages, cut into equal runs, one per resident CTA
// (struct Walk).  Each CTA has a producer warp that streams its run's FP4 K/V
// codes and E4M3 scales into a 2-stage ring with 1-D bulk copies, and
// four consumer warps that each take two 16-token tiles of every stage (one
// barrier hand-off per two tiles; measured faster than 4 x 64-token stages).  A consumer
// dequantizes in registers (cvt e2m1x2 -> f16x2, times the E4M3 block scale:
// exact in f16) and runs mma.sync m16n8k16 with fp32 accumulation:
//   S^T[16 tok x 8 head] = K_hat[16 tok x 128] . Q^T[128 x 8]   (8 MMAs)
//   O^T[128 x 8 head]   += V_hat^T[128 x 16 tok] . P^T[16 x 8]  (8 MMAs)
// The up to 8 query heads that share a KV head (grouped-query attention) fill
// the MMA's N = 8.  Softmax is online, in fp32, in the log2 domain, with lazy
// rescaling (the running max moves only when a tile exceeds it by 2^8).  At
// the end of a (sequence, head) or of the run the four warps merge their
// partial (max, sum, O) and write one record; a combine kernel merges them.
//
// Lane roles (g = lane/4, t = lane%4), fixed by the m16n8k16 fragment layouts:
//   K: rows g and g+8 of the S tile, channels 32t..32t+31 (16 bytes, blocks 2t, 2t+1)
//   V: k-indices 2t, 2t+1, 2t+8, 2t+9, channels 16g..16g+15 (8 bytes, block g)
//   Q: head slot g, channels 32t..32t+31
// Row/k index m of a 16-token tile is token TOK(m) = (m&1)*4 + (m>>1&3) +
// (m&8): the V rows each lane reads are then t, t+4, t+8, t+12, so a V load
// instruction covers four consecutive token rows (measured faster on GB300
// than the orders that favour the K loads instead).  The channel order inside
// an MMA is permuted to match the lanes' contiguous bytes; neither
// permutation changes the dot products.
#include <cfloat>
#include <map>
#include <mutex>

#include "common.cuh"
#include "nvfp4_quant.cuh"

namespace nvfp4 {
namespace {

constexpr int kD = 128;
constexpr int kStageTok = 128;        // tokens per ring stage: the unit of work
constexpr int kChunk = 1024;          // the workspace holds at least one record per 1024 tokens and head
#ifndef NVFP4_ATTN_STAGES
#define NVFP4_ATTN_STAGES 2
#endif
#ifndef NVFP4_ATTN_MIN_CTAS
#define NVFP4_ATTN_MIN_CTAS 4
#endif
constexpr int kStages = NVFP4_ATTN_STAGES;  // 2 x 18 KiB ring + merge buffer: 4 CTAs per SM
constexpr int kConsumers = 4;         // consumer warps, 16 tokens of a stage each
constexpr int kThreads = 32 * (1 + kConsumers);
constexpr uint32_t kStageBytes = kStageTok * (64 + 8) * 2;  // K, V codes + scales: 18 KiB
static_assert(kStageTok % (16 * kConsumers) == 0, "stage tiling");
constexpr uint32_t kOffKc = 0, kOffVc = kStageTok * 64, kOffKs = 2 * kStageTok * 64, kOffVs = kOffKs + kStageTok * 8;
// Merge buffer: a head's channels with 2 floats of padding per 16, and heads
// 148 floats apart, so that a half-warp's 8-byte stores (4 channel groups, 4
// heads) meet 16 different bank pairs.
constexpr int kMergeHead = 148;
__device__ __forceinline__ int merge_channel(int c) { return c + 2 * (c >> 4); }
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRescaleLog2 = 8.0f;  // lazy rescale threshold (P stays <= 2^8 in f16)

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four packed e2m1x2 bytes -> four f16x2 (low nibble -> low half).
__device__ __forceinline__ void e2m1x8_to_f16x2(uint32_t w, uint32_t h[4]) {
  asm("{\n .reg .b8 b0, b1, b2, b3;\n mov.b32 {b0, b1, b2, b3}, %4;\n"
      " cvt.rn.f16x2.e2m1x2 %0, b0;\n cvt.rn.f16x2.e2m1x2 %1, b1;\n"
      " cvt.rn.f16x2.e2m1x2 %2, b2;\n cvt.rn.f16x2.e2m1x2 %3, b3;\n}"
      : "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3])
      : "r"(w));
}

// E1M2 nibbles (two's complement n, value n/2) decode to f16 n; the 1/2 goes
// into the block scale.  The nibble XOR 8 in the low mantissa bits of 1024.0
// (0x6400) reads as 1032 + n, and one f16x2 subtraction of 1032 leaves n.  A
// nibble in bits 4-7 of a half is decoded where it stands: 1024 + 16 (n + 8)
// minus 1152 leaves 16 n, and its block scale carries a further 1/16.  Both
// are exact, and the product with the scale is the same f16 either way
// (16 n times s / 16 is n times s, and s / 16 is exact in f16 for every E4M3
// scale), so the tensor-core operands are those of the shifted decode.
__device__ __forceinline__ uint32_t hsub2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
// K side: the eight nibbles n0..n7 of w (n0 lowest) -> h[i] = (n_i, n_{i+4}),
// with h[1] and h[3] holding 16 n (their scales carry the 1/16): one
// mask-and-xor and one subtraction per pair, one shift per word.  The channel
// order inside each group of eight differs from the E2M1 path; the queries
// are paired the same way, so every logit is the same sum.
__device__ __forceinline__ void e1m2x8_to_f16x2_paired(uint32_t w, uint32_t h[4]) {
  const uint32_t t = w >> 8;
  h[0] = hsub2((w & 0x000F000Fu) ^ 0x64086408u, 0x64086408u);
  h[1] = hsub2((w & 0x00F000F0u) ^ 0x64806480u, 0x64806480u);
  h[2] = hsub2((t & 0x000F000Fu) ^ 0x64086408u, 0x64086408u);
  h[3] = hsub2((t & 0x00F000F0u) ^ 0x64806480u, 0x64806480u);
}
// V side: byte k of two tokens' words a and b -> lo = (a, b) of the byte's
// low-nibble channel, hi = 16 (a, b) of its high-nibble channel (its scale
// carries the 1/16).
__device__ __forceinline__ void e1m2_token_pair(uint32_t wa, uint32_t wb, int k, uint32_t* lo, uint32_t* hi) {
  const uint32_t x = __byte_perm(wa, wb, 0x4400u + 0x1111u * k);  // bytes: a_k, a_k, b_k, b_k
  *lo = hsub2((x & 0x000F000Fu) ^ 0x64086408u, 0x64086408u);
  *hi = hsub2((x & 0x00F000F0u) ^ 0x64806480u, 0x64806480u);
}

template <bool kE1M2>
__device__ __forceinline__ void decode8(uint32_t w, uint32_t h[4]) {
  if (kE1M2) e1m2x8_to_f16x2_paired(w, h);
  else e2m1x8_to_f16x2(w, h);
}

// Two E4M3 bytes (low byte -> low half) -> f16x2, exact.
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t two_bytes) {
  uint32_t h;
  asm("{\n .reg .b16 s;\n cvt.u16.u32 s, %1;\n cvt.rn.f16x2.e4m3x2 %0, s;\n}" : "=r"(h) : "r"(two_bytes));
  return h;
}

__device__ __forceinline__ uint32_t hmul2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

__device__ __forceinline__ uint32_t f32x2_to_f16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t bcast_lo(uint32_t x) { return __byte_perm(x, x, 0x1010); }
__device__ __forceinline__ uint32_t bcast_hi(uint32_t x) { return __byte_perm(x, x, 0x3232); }

__device__ __forceinline__ void named_barrier_consumers() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kConsumers) : "memory");
}

// Token of row / k index m (0..15) of a 16-token tile.
__device__ __forceinline__ int tile_tok(int m) { return (m & 1) * 4 + ((m >> 1) & 3) + (m & 8); }

struct Params {
  const uint8_t* k_codes;
  const uint8_t* k_scales;
  const uint8_t* v_codes;
  const uint8_t* v_scales;
  const int32_t* seq_lens;
  const uint16_t* q;
  float* o_ws;
  float* ml_ws;
  int* status;
  int batch, hkv, capacity, hq, group, records, whole;
  float logit_mult;  // softmax_scale * g_K * log2(e)
  int fault_skip_stage;  // test-only: CTA 0's producer leaves its first stage unissued
};

// Which stages (128 cached tokens of one sequence and KV head) a CTA takes.
// The stages of all sequences and heads, sequence-major, are one list of T;
// CTA c takes units c R .. c R + R - 1, so every CTA has the same work
// whatever the lengths.  A (sequence, head)'s s stages then lie with at most
// (s - 2) / R + 2 CTAs in a row, each of which leaves one record of it; R is
// at least what keeps that within the workspace's `records` per head.  Where
// `whole` (room for one record only, or no head longer than three stages), a CTA
// takes whole (sequence, head)s instead and no lengths need be summed.
// A part of a head costs about as much as a stage beside its stages (merging
// four warps, writing a record), so where a CTA takes several stages each head
// counts one unit more, after its stages, and a run is R units: without it a
// run of one-stage heads took several times as long as the others (64 x 40
// heads of 1-3000 tokens 50 us).
struct Segment {  // a run of stages of one (sequence, KV head)
  int b, kvh, record, t_begin, t_end;
  bool last;  // of its (sequence, head)
};

__device__ __forceinline__ int cached_tokens(const Params& p, int b) {
  return max(0, min(__ldg(p.seq_lens + b), p.capacity));
}
__device__ __forceinline__ uint32_t stages_of(int tokens) {
  return static_cast<uint32_t>(tokens + kStageTok - 1) / kStageTok;
}

struct Walk {
  uint32_t R;        // units per CTA; 0: whole (sequence, head)s
  uint32_t at, end;  // next unit and end of this CTA's run; or (sequence, head)s
  uint32_t before;   // units before sequence b
  uint32_t extra;    // units of a head beside its stages
  int b;

  __device__ __forceinline__ uint32_t units_of(uint32_t stages) const { return stages ? stages + extra : 0u; }

  // By one converged warp.
  __device__ __forceinline__ void start(const Params& p) {
    if (p.whole) {
      R = 0;
      at = blockIdx.x;
      end = static_cast<uint32_t>(p.batch) * p.hkv;
      return;
    }
    const int lane = threadIdx.x & 31;
    const int per = (p.batch + 31) / 32, b0 = min(p.batch, lane * per), b1 = min(p.batch, b0 + per);
    uint32_t sum = 0, most = 0, filled = 0;
    for (int i = b0; i < b1; i += 4) {  // four lengths in flight per lane
      uint32_t s[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) s[j] = i + j < b1 ? stages_of(cached_tokens(p, i + j)) : 0u;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sum += s[j];
        most = max(most, s[j]);
        filled += s[j] != 0u;
      }
    }
    most = __reduce_max_sync(0xffffffffu, most);
    extra = __reduce_add_sync(0xffffffffu, sum) * p.hkv > gridDim.x ? 1u : 0u;
    sum += extra * filled;
    uint32_t incl = sum * p.hkv;  // units up to this lane's last sequence
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, sh);
      if (lane >= sh) incl += v;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    R = max(1u, (total + gridDim.x - 1) / gridDim.x);
    const uint32_t heads = static_cast<uint32_t>(p.batch) * p.hkv, whole = units_of(most);
    // Equal lengths, a little longer than a run, of enough heads: no run crosses a head.
    if (whole > R && whole <= R + 2 && whole * heads == total && 2 * heads >= gridDim.x) R = whole;
    if (most > 1) R = max(R, (most + p.records - 3) / (p.records - 1));
    at = min(blockIdx.x * R, total);
    end = min(at + R, total);
    // The lane whose sequences hold the first unit looks for its sequence.
    uint32_t first = incl - sum * p.hkv;
    int found = p.batch;
    if (at >= first && at < incl) {
      for (found = b0; found < b1; ++found) {
        const uint32_t n = units_of(stages_of(cached_tokens(p, found))) * p.hkv;
        if (at < first + n) break;
        first += n;
      }
    }
    const uint32_t owner = __ballot_sync(0xffffffffu, found < p.batch);
    const int src = owner ? __ffs(owner) - 1 : 0;
    b = __shfl_sync(0xffffffffu, found, src);
    before = __shfl_sync(0xffffffffu, first, src);
  }

  __device__ __forceinline__ bool next(const Params& p, Segment* s) {
    if (R == 0) {
      if (at >= end) return false;
      s->b = static_cast<int>(at) / p.hkv;
      s->kvh = static_cast<int>(at) - s->b * p.hkv;
      s->record = 0;
      s->last = true;
      s->t_begin = 0;
      s->t_end = cached_tokens(p, s->b);
      at += gridDim.x;
      return true;
    }
    while (at < end && b < p.batch) {
      const int len = cached_tokens(p, b);
      const uint32_t n = stages_of(len), units = units_of(n);
      if (at >= before + units * p.hkv) {
        before += units * p.hkv;
        ++b;
        continue;
      }
      s->b = b;
      s->kvh = static_cast<int>((at - before) / units);
      const uint32_t first = before + s->kvh * units;  // the head's first stage
      const uint32_t st = at - first, taken = min(units - st, end - at);
      at += taken;
      if (st >= n) continue;
      const uint32_t count = min(n - st, taken);
      s->record = static_cast<int>(blockIdx.x - first / R);
      s->last = st + count == n;
      s->t_begin = static_cast<int>(st) * kStageTok;
      s->t_end = min(s->t_begin + static_cast<int>(count) * kStageTok, len);
      return true;
    }
    return false;
  }
};

// kE1M2: the cache holds E1M2 elements (decoded to n, the scale carries 1/2).
template <bool kE1M2>
__global__ void __launch_bounds__(kThreads, NVFP4_ATTN_MIN_CTAS) attn_partial_kernel(const Params p) {
  extern __shared__ __align__(128) uint8_t smem[];
  uint8_t* ring = smem;
  float* sh_o = reinterpret_cast<float*>(smem + kStages * kStageBytes);  // [kConsumers][8][merge_channel(128)]
  float* sh_m = sh_o + kConsumers * 8 * kMergeHead;                      // [kConsumers][8]
  float* sh_l = sh_m + kConsumers * 8;
  uint64_t* full = reinterpret_cast<uint64_t*>(sh_l + kConsumers * 8);
  uint64_t* empty = full + kStages;
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kConsumers);
    }
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  griddep_wait_and_release();
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b < p.batch; b += kThreads)
      if (__ldg(p.seq_lens + b) > p.capacity) set_status(p.status, NVFP4_ERR_CAPACITY);

  Walk walk;
  walk.start(p);
  Segment it;
  if (warp == 0) {
    // ------------------------------------------------------------ producer ---
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued_parity[kStages];
      bool issued[kStages];
      for (int s = 0; s < kStages; ++s) issued[s] = false;
      bool skip_stage = p.fault_skip_stage && blockIdx.x == 0;
      while (!abort_flag && walk.next(p, &it)) {
        const size_t row0 = (static_cast<size_t>(it.b) * p.hkv + it.kvh) * p.capacity;
        for (int t0 = it.t_begin; t0 < it.t_end; t0 += kStageTok) {
          const int n = min(kStageTok, it.t_end - t0);
          const int n_even = (n + 1) & ~1;  // scale rows copied in 16-byte units (capacity is even)
          if (!mbar_wait_bounded(&empty[stage], phase ^ 1u, &abort_flag)) {
            set_status(p.status, NVFP4_ERR_TIMEOUT);
            abort_flag = 1;
            break;
          }
          if (skip_stage) {
            // Injected fault: the stage is neither armed nor loaded, so the
            // consumers' bounded wait on it runs out (NVFP4_ERR_TIMEOUT).
            skip_stage = false;
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
            continue;
          }
          uint8_t* st = ring + stage * kStageBytes;
          mbar_arrive_expect_tx(&full[stage], 2u * (n * 64 + n_even * 8));
          const size_t tok = row0 + t0;
          bulk_load(st + kOffKc, p.k_codes + tok * 64, n * 64, &full[stage]);
          bulk_load(st + kOffVc, p.v_codes + tok * 64, n * 64, &full[stage]);
          bulk_load(st + kOffKs, p.k_scales + tok * 8, n_even * 8, &full[stage]);
          bulk_load(st + kOffVs, p.v_scales + tok * 8, n_even * 8, &full[stage]);
          issued[stage] = true;
          issued_parity[stage] = phase;
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (abort_flag)
        for (int s = 0; s < kStages; ++s)
          if (issued[s]) mbar_wait_bounded(&full[s], issued_parity[s], nullptr);
    }
    return;
  }

  // -------------------------------------------------------------- consumers ---
  const int cw = warp - 1;  // consumer index: tiles cw, cw + 4, ... of each stage
  const int g = lane >> 2, t = lane & 3;
  const int rk0 = tile_tok(g), rk1 = tile_tok(g + 8);                    // K rows of this lane
  const int rv[4] = {tile_tok(2 * t), tile_tok(2 * t + 1), tile_tok(2 * t + 8), tile_tok(2 * t + 9)};  // V rows
  int stage = 0;
  uint32_t phase = 0;
  if (blockIdx.x == 0) {  // sequences without tokens have no segment
    for (int b = threadIdx.x - 32; b < p.batch; b += 32 * kConsumers) {
      if (__ldg(p.seq_lens + b) > 0) continue;
      float* ml = p.ml_ws + static_cast<size_t>(b) * p.hq * p.records * 2;
      for (int i = 0; i < p.hq * p.records; ++i) {
        ml[2 * i] = -INFINITY;
        ml[2 * i + 1] = 0.0f;
      }
    }
  }
  while (walk.next(p, &it)) {
    // Queries of head slot g: f16 after an exact power-of-two scaling that
    // keeps |q| < 1; the scaling is undone in the logit multiplier.
    const bool head_live = g < p.group;
    float qv[32];
    {
      const uint4* qp = reinterpret_cast<const uint4*>(
          p.q + (static_cast<size_t>(it.b) * p.hq + it.kvh * p.group + (head_live ? g : 0)) * kD + 32 * t);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 w = head_live ? __ldg(qp + i) : make_uint4(0, 0, 0, 0);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          qv[8 * i + 2 * k] = __uint_as_float(ws[k] << 16);
          qv[8 * i + 2 * k + 1] = __uint_as_float(ws[k] & 0xFFFF0000u);
        }
      }
    }
    float qmax = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; ++i) qmax = fmaxf(qmax, fabsf(qv[i]));
    qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, 1));
    qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, 2));
    const int qexp = qmax > 0.0f ? static_cast<int>((__float_as_uint(qmax) >> 23) & 0xFF) - 126 : 0;
    const float qscale = ldexpf(1.0f, -qexp);
    uint32_t qf[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      // k-step j = 2w + h.  E2M1 keys hold channel pairs (4j, 4j+1), (4j+2, 4j+3);
      // E1M2 keys (decoded in pairs i, i+4 of each word) hold (8w+2h, 8w+2h+4), (8w+2h+1, 8w+2h+5).
      const int c0 = kE1M2 ? 8 * (j >> 1) + 2 * (j & 1) : 4 * j;
      const int c1 = kE1M2 ? c0 + 4 : c0 + 1, c2 = kE1M2 ? c0 + 1 : c0 + 2, c3 = kE1M2 ? c0 + 5 : c0 + 3;
      qf[2 * j] = f32x2_to_f16x2(qv[c0] * qscale, qv[c1] * qscale);
      qf[2 * j + 1] = f32x2_to_f16x2(qv[c2] * qscale, qv[c3] * qscale);
    }
    const float mult_self = p.logit_mult / qscale;
    const float mult0 = __shfl_sync(0xffffffffu, mult_self, (2 * t) * 4);
    const float mult1 = __shfl_sync(0xffffffffu, mult_self, (2 * t + 1) * 4);

    float o[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.0f;
    float m_run[2] = {-INFINITY, -INFINITY};
    float l_run[2] = {0.0f, 0.0f};

    for (int t0 = it.t_begin; t0 < it.t_end; t0 += kStageTok) {
      int ok = 1;
      if (lane == 0) {
        ok = !abort_flag && mbar_wait_bounded(&full[stage], phase, &abort_flag);
        if (!ok && !abort_flag) {
          set_status(p.status, NVFP4_ERR_TIMEOUT);
          abort_flag = 1;
        }
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) return;
      const uint8_t* st = ring + stage * kStageBytes;
      // The warp's two tiles of the stage, unrolled: the second tile's loads,
      // decode and score MMAs interleave with the first tile's softmax and
      // value MMAs (same 96 registers, same 4 CTAs per SM): B=64, T=16384
      // 248.4 -> 241.3 us, bit-identical.
#pragma unroll
      for (int sub = 0; sub < kStageTok / (16 * kConsumers); ++sub) {
      const int r0 = 16 * (cw + kConsumers * sub);  // this warp's tile within the stage
      const int tile = t0 + r0;
      const int valid = it.t_end - tile;  // tokens of this warp's tile inside the segment (may be <= 0)
      if (valid > 0) {
        // ---- S^T = K_hat Q^T: 8 k-steps of 16 channels ---------------------
        const uint4 ka = *reinterpret_cast<const uint4*>(st + kOffKc + (r0 + rk0) * 64 + 16 * t);
        const uint4 kb = *reinterpret_cast<const uint4*>(st + kOffKc + (r0 + rk1) * 64 + 16 * t);
        uint32_t ksa = e4m3x2_to_f16x2(*reinterpret_cast<const uint16_t*>(st + kOffKs + (r0 + rk0) * 8 + 2 * t));
        uint32_t ksb = e4m3x2_to_f16x2(*reinterpret_cast<const uint16_t*>(st + kOffKs + (r0 + rk1) * 8 + 2 * t));
        if (kE1M2) { ksa = hmul2(ksa, 0x38003800u); ksb = hmul2(ksb, 0x38003800u); }  // times 1/2, exact
        const uint32_t sa_lo = bcast_lo(ksa), sa_hi = bcast_hi(ksa);
        const uint32_t sb_lo = bcast_lo(ksb), sb_hi = bcast_hi(ksb);
        float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        const uint32_t kaw[4] = {ka.x, ka.y, ka.z, ka.w};
        const uint32_t kbw[4] = {kb.x, kb.y, kb.z, kb.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          uint32_t ha[4], hb[4];
          decode8<kE1M2>(kaw[w], ha);
          decode8<kE1M2>(kbw[w], hb);
          const uint32_t sa = w < 2 ? sa_lo : sa_hi, sb = w < 2 ? sb_lo : sb_hi;
          // E1M2: the scales of the pairs decoded as 16 n (times 1/16, exact).
          const uint32_t sa1 = kE1M2 ? hmul2(sa, 0x2C002C00u) : sa, sb1 = kE1M2 ? hmul2(sb, 0x2C002C00u) : sb;
#pragma unroll
          for (int h = 0; h < 2; ++h) {  // k-step j = 2w + h uses bytes 2j and 2j+1
            const uint32_t a[4] = {hmul2(ha[2 * h], sa), hmul2(hb[2 * h], sb), hmul2(ha[2 * h + 1], sa1),
                                   hmul2(hb[2 * h + 1], sb1)};
            const int j = 2 * w + h;
            mma16816(s, a, qf[2 * j], qf[2 * j + 1]);
          }
        }
        // ---- online softmax over this tile (log2 domain) -------------------
        float x0 = s[0] * mult0, x1 = s[1] * mult1, x2 = s[2] * mult0, x3 = s[3] * mult1;
        uint32_t vs01_raw, vs89_raw;
        {
          const uint32_t s0 = st[kOffVs + (r0 + rv[0]) * 8 + g], s1 = st[kOffVs + (r0 + rv[1]) * 8 + g];
          const uint32_t s2 = st[kOffVs + (r0 + rv[2]) * 8 + g], s3 = st[kOffVs + (r0 + rv[3]) * 8 + g];
          vs01_raw = s0 | (s1 << 8);
          vs89_raw = s2 | (s3 << 8);
        }
        if (valid < 16) {  // ragged end of the segment: mask keys, zero the scales of absent values
          if (rk0 >= valid) x0 = x1 = -INFINITY;
          if (rk1 >= valid) x2 = x3 = -INFINITY;
          if (rv[0] >= valid) vs01_raw &= 0xFF00u;
          if (rv[1] >= valid) vs01_raw &= 0x00FFu;
          if (rv[2] >= valid) vs89_raw &= 0xFF00u;
          if (rv[3] >= valid) vs89_raw &= 0x00FFu;
        }
        float mx0 = fmaxf(x0, x2), mx1 = fmaxf(x1, x3);
        // The tile maximum is needed only when some logit exceeds the running
        // maximum by more than the lazy threshold: vote first, reduce then.
        if (__any_sync(0xffffffffu, mx0 > m_run[0] + kRescaleLog2 || mx1 > m_run[1] + kRescaleLog2)) {
#pragma unroll
          for (int sh = 4; sh < 32; sh <<= 1) {
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, sh));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, sh));
          }
          const bool up0 = mx0 > m_run[0] + kRescaleLog2, up1 = mx1 > m_run[1] + kRescaleLog2;
          const float al0 = up0 ? fast_exp2(m_run[0] - mx0) : 1.0f;
          const float al1 = up1 ? fast_exp2(m_run[1] - mx1) : 1.0f;
          if (up0) m_run[0] = mx0;
          if (up1) m_run[1] = mx1;
          l_run[0] *= al0;
          l_run[1] *= al1;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            o[i][0] *= al0; o[i][1] *= al1; o[i][2] *= al0; o[i][3] *= al1;
          }
        }
        const float p0 = fast_exp2(x0 - m_run[0]), p1 = fast_exp2(x1 - m_run[1]);
        const float p2 = fast_exp2(x2 - m_run[0]), p3 = fast_exp2(x3 - m_run[1]);
        l_run[0] += p0 + p2;
        l_run[1] += p1 + p3;
        // P^T fragments for the PV product: transpose the two 8x8 (token, head) blocks.
        const uint32_t pb0 = movmatrix_trans(f32x2_to_f16x2(p0, p1));
        const uint32_t pb1 = movmatrix_trans(f32x2_to_f16x2(p2, p3));

        // ---- O^T += V_hat^T P^T: 8 m-tiles, m-tile i = channels 16g+2i, 16g+2i+1
        uint32_t vs01 = e4m3x2_to_f16x2(vs01_raw), vs89 = e4m3x2_to_f16x2(vs89_raw);
        if (kE1M2) { vs01 = hmul2(vs01, 0x38003800u); vs89 = hmul2(vs89, 0x38003800u); }
        // E1M2: the high-nibble channels are decoded as 16 n; their scales carry 1/16 (exact).
        const uint32_t vs01_hi = kE1M2 ? hmul2(vs01, 0x2C002C00u) : vs01;
        const uint32_t vs89_hi = kE1M2 ? hmul2(vs89, 0x2C002C00u) : vs89;
        const uint2 va = *reinterpret_cast<const uint2*>(st + kOffVc + (r0 + rv[0]) * 64 + 8 * g);
        const uint2 vb = *reinterpret_cast<const uint2*>(st + kOffVc + (r0 + rv[1]) * 64 + 8 * g);
        const uint2 vc = *reinterpret_cast<const uint2*>(st + kOffVc + (r0 + rv[2]) * 64 + 8 * g);
        const uint2 vd = *reinterpret_cast<const uint2*>(st + kOffVc + (r0 + rv[3]) * 64 + 8 * g);
#pragma unroll
        for (int half = 0; half < 2; ++half) {  // bytes 0-3, then 4-7 of each token's 8-byte slice
          const uint32_t wa = half ? va.y : va.x, wb = half ? vb.y : vb.x;
          const uint32_t wc = half ? vc.y : vc.x, wd = half ? vd.y : vd.x;
          uint32_t f_lo_ab[4], f_hi_ab[4], f_lo_cd[4], f_hi_cd[4];
          if (kE1M2) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              e1m2_token_pair(wa, wb, k, &f_lo_ab[k], &f_hi_ab[k]);
              e1m2_token_pair(wc, wd, k, &f_lo_cd[k], &f_hi_cd[k]);
            }
          } else {
            // Pair the same channel of two tokens in one e2m1x2 byte (first token in the low nibble).
            const uint32_t lo_ab = (wa & 0x0F0F0F0Fu) | ((wb << 4) & 0xF0F0F0F0u);
            const uint32_t hi_ab = ((wa >> 4) & 0x0F0F0F0Fu) | (wb & 0xF0F0F0F0u);
            const uint32_t lo_cd = (wc & 0x0F0F0F0Fu) | ((wd << 4) & 0xF0F0F0F0u);
            const uint32_t hi_cd = ((wc >> 4) & 0x0F0F0F0Fu) | (wd & 0xF0F0F0F0u);
            e2m1x8_to_f16x2(lo_ab, f_lo_ab);
            e2m1x8_to_f16x2(hi_ab, f_hi_ab);
            e2m1x8_to_f16x2(lo_cd, f_lo_cd);
            e2m1x8_to_f16x2(hi_cd, f_hi_cd);
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t a[4] = {hmul2(f_lo_ab[k], vs01), hmul2(f_hi_ab[k], vs01_hi), hmul2(f_lo_cd[k], vs89),
                                   hmul2(f_hi_cd[k], vs89_hi)};
            mma16816(o[4 * half + k], a, pb0, pb1);
          }
        }
      }
      }  // tiles of the stage
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[stage]);
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }

    // ---- merge the consumer warps, write this segment's record ------------
    l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 4);
    l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 4);
    l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 8);
    l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 8);
    l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 16);
    l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 16);
    float* my_o = sh_o + cw * 8 * kMergeHead;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int c0 = merge_channel(16 * g + 2 * i);  // channels of accumulator rows g and g+8 of m-tile i
      *reinterpret_cast<float2*>(my_o + (2 * t) * kMergeHead + c0) = make_float2(o[i][0], o[i][2]);
      *reinterpret_cast<float2*>(my_o + (2 * t + 1) * kMergeHead + c0) = make_float2(o[i][1], o[i][3]);
    }
    if (g == 0) {
      sh_m[cw * 8 + 2 * t] = m_run[0]; sh_m[cw * 8 + 2 * t + 1] = m_run[1];
      sh_l[cw * 8 + 2 * t] = l_run[0]; sh_l[cw * 8 + 2 * t + 1] = l_run[1];
    }
    named_barrier_consumers();
    for (int idx = threadIdx.x - 32; idx < p.group * kD; idx += 32 * kConsumers) {
      const int h = idx / kD, c = idx % kD;
      float M = -INFINITY;
#pragma unroll
      for (int w = 0; w < kConsumers; ++w) M = fmaxf(M, sh_m[w * 8 + h]);
      float acc = 0.0f, L = 0.0f;
      if (M != -INFINITY) {
#pragma unroll
        for (int w = 0; w < kConsumers; ++w) {
          const float wt = fast_exp2(sh_m[w * 8 + h] - M);
          acc += wt * sh_o[(w * 8 + h) * kMergeHead + merge_channel(c)];
          L += wt * sh_l[w * 8 + h];
        }
      }
      const size_t rec = (static_cast<size_t>(it.b) * p.hq + it.kvh * p.group + h) * p.records + it.record;
      p.o_ws[rec * kD + c] = acc;
      if (c == 0) {
        p.ml_ws[rec * 2] = M;
        p.ml_ws[rec * 2 + 1] = L;
      }
    }
    if (it.last) {  // the records of this head that no segment leaves
      const int rest = p.records - it.record - 1;
      for (int i = threadIdx.x - 32; i < rest * p.group; i += 32 * kConsumers) {
        const int h = i / rest;
        const size_t rec = (static_cast<size_t>(it.b) * p.hq + it.kvh * p.group + h) * p.records + it.record + 1 + i - h * rest;
        p.ml_ws[rec * 2] = -INFINITY;
        p.ml_ws[rec * 2 + 1] = 0.0f;
      }
    }
    named_barrier_consumers();  // the merge buffer is rewritten by the next segment
  }
}

// out[b, h] = g_V * sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s
// Where the combine kernel puts o: bf16 [batch, heads, 128], or (kQuant) the
// NVFP4 A operand of the output projection: the bf16-rounded o of each query
// head's 128 channels quantized in 8 blocks of 16 with the static tensor scale
// g_out by the library's recipe, codes [batch, heads * 64] bytes and MMA-layout
// scales of the [batch, heads * 128] matrix (padding rows zero).
struct CombineOut {
  uint16_t* bf16;
  uint8_t* codes;
  uint8_t* scales;
  const float* g_out;
  int* status;
  int rows;
  uint32_t kgroups;
};

// One block per head, kD threads times kGroups.  A head's records come first
// in its slots; the others hold (-inf, 0) and an undefined O that is not used.
// The weights are formed one record per thread, then the records are added,
// one channel per thread; kGroups = 8 (few heads with many records) lets each
// group take every eighth one.  The first records' O is loaded beside the
// weights' inputs: usually that is all there is.
template <bool kQuant, int kGroups>
__global__ void __launch_bounds__(kD* kGroups) attn_combine_kernel(const float* __restrict__ o_ws,
                                                                   const float* __restrict__ ml_ws, int records,
                                                                   float gv, const CombineOut out) {
  constexpr int kT = kD * kGroups, kAhead = kGroups > 1 ? 8 : 4;
  __shared__ float sh_w[kT], sh_acc[kGroups][kD];
  __shared__ float2 sh_red[kT / 32];
  __shared__ int sh_used[kT / 32];
  griddep_wait_and_release();
  const size_t bh = static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = threadIdx.x % kD, group = threadIdx.x / kD;
  const float2* ml = reinterpret_cast<const float2*>(ml_ws) + bh * records;
  const float* o = o_ws + bh * records * kD + c;
  const float2 own = static_cast<int>(threadIdx.x) < records ? __ldg(ml + threadIdx.x) : make_float2(-INFINITY, 0.0f);
  float ahead[kAhead];
#pragma unroll
  for (int k = 0; k < kAhead; ++k) {
    const int i = group + k * kGroups;
    ahead[k] = i < records ? __ldg(o + static_cast<size_t>(i) * kD) : 0.0f;
  }
  float m = own.x;
  int used = own.x != -INFINITY ? static_cast<int>(threadIdx.x) + 1 : 0;  // the records in use come first
  for (int i = threadIdx.x + kT; i < records; i += kT) {
    const float x = __ldg(ml + i).x;
    m = fmaxf(m, x);
    if (x != -INFINITY) used = i + 1;
  }
  used = __reduce_max_sync(0xffffffffu, used);
#pragma unroll
  for (int sh = 16; sh; sh >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, sh));
  if (lane == 0) {
    sh_red[warp].x = m;
    sh_used[warp] = used;
  }
  __syncthreads();
  float M = sh_red[0].x;
  used = sh_used[0];
#pragma unroll
  for (int w = 1; w < kT / 32; ++w) {
    M = fmaxf(M, sh_red[w].x);
    used = max(used, sh_used[w]);
  }
  float acc = 0.0f, l = 0.0f;
  for (int i0 = 0; i0 < used; i0 += kT) {
    const int i = i0 + threadIdx.x;
    float w = 0.0f;
    if (i < used) {
      const float2 x = i0 == 0 ? own : __ldg(ml + i);
      w = fast_exp2(x.x - M);
      l += w * x.y;
    }
    sh_w[threadIdx.x] = w;
    __syncthreads();
    const int count = min(kT, used - i0);
    if (i0 == 0) {
#pragma unroll
      for (int k = 0; k < kAhead; ++k)
        if (group + k * kGroups < count) acc += sh_w[group + k * kGroups] * ahead[k];
    }
#pragma unroll 8
    for (int k = group + (i0 == 0 ? kAhead * kGroups : 0); k < count; k += kGroups)
      acc += sh_w[k] * __ldg(o + static_cast<size_t>(i0 + k) * kD);
    __syncthreads();
  }
#pragma unroll
  for (int sh = 16; sh; sh >>= 1) l += __shfl_xor_sync(0xffffffffu, l, sh);
  if (lane == 0) sh_red[warp].y = l;
  if (kGroups > 1) sh_acc[group][c] = acc;
  __syncthreads();
  if (group) return;
  float L = sh_red[0].y;
#pragma unroll
  for (int w = 1; w < kT / 32; ++w) L += sh_red[w].y;
#pragma unroll
  for (int k = 1; k < kGroups; ++k) acc += sh_acc[k][c];
  const float r = L > 0.0f ? __fdiv_rn(acc, L) * gv : 0.0f;
  uint16_t bits;
  asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(bits) : "f"(r));
  if (!kQuant) {
    out.bf16[bh * kD + c] = bits;
    return;
  }
  // Lanes 16j..16j+15 of a warp hold one 16-channel block of this head.
  const float g_in = __ldg(out.g_out);
  const bool g_ok = g_in > 0.0f && g_in <= FLT_MAX;
  if (!g_ok && bh == 0 && threadIdx.x == 0) set_status(out.status, NVFP4_ERR_INVALID_ARG);
  const float g = g_ok ? g_in : 1.0f;
  const float x = __uint_as_float(static_cast<uint32_t>(bits) << 16);
  float amax = fabsf(x);
#pragma unroll
  for (int sh = 1; sh < 16; sh <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, sh));
  const BlockScale bs = block_scale(amax, g, __fmul_rn(6.0f, g));
  // Lane pairs (2i, 2i+1) form one code byte, element 2i in the low nibble.
  const float mine = __fmul_rn(x, bs.mult);
  const float other = __shfl_xor_sync(0xffffffffu, mine, 1);
  uint32_t pair;  // the first source of the conversion goes to the high nibble
  asm("{\n .reg .b8 t;\n cvt.rn.satfinite.e2m1x2.f32 t, %1, %2;\n cvt.u32.u8 %0, t;\n}"
      : "=r"(pair)
      : "f"(other), "f"(mine));
  const uint32_t row = blockIdx.y, head = blockIdx.x;
  const uint32_t padded = (static_cast<uint32_t>(out.rows) + 127u) & ~127u;
  const uint64_t code_bytes = static_cast<uint64_t>(out.rows) * gridDim.x * (kD / 2);
  const uint64_t scale_bytes = static_cast<uint64_t>(padded) * out.kgroups * 4;
  const uint64_t code_off = static_cast<uint64_t>(row) * (gridDim.x * (kD / 2)) + head * (kD / 2) + c / 2;
  if ((c & 1) == 0 && in_bounds(out.status, code_off < code_bytes))
    out.codes[code_off] = g_ok ? static_cast<uint8_t>(pair & 0xFFu) : 0;
  const uint32_t kb = head * (kD / 16) + c / 16;
  const uint64_t sc_off = mma_scale_offset(row, kb, out.kgroups);
  if ((c & 15) == 0 && in_bounds(out.status, sc_off < scale_bytes))
    out.scales[sc_off] = g_ok ? static_cast<uint8_t>(bs.code) : 0;
  // Rows from batch up to the next multiple of 128 hold zero scales.
  if (row == 0 && c < kD / 16) {
    for (uint32_t pr = out.rows; pr < padded; ++pr) {
      const uint64_t off = mma_scale_offset(pr, head * (kD / 16) + c, out.kgroups);
      if (in_bounds(out.status, off < scale_bytes)) out.scales[off] = 0;
    }
  }
}

// Records per head that the workspace has to hold at least, and those that
// decode_attention_nvfp4_workspace_size asks for: with few sequences the CTAs
// (4 on each of 152 SMs) share a head, and lengths up to four times the mean
// are still spread evenly; S stages never leave more than S records.
// num_kv_heads is not known there: at least num_q_heads / 8.
int min_records(int capacity) { return (capacity + kChunk - 1) / kChunk; }
int64_t preferred_records(int64_t batch, int64_t num_q_heads, int64_t capacity) {
  const int64_t stages = (capacity + kStageTok - 1) / kStageTok, heads = batch * ((num_q_heads + 7) / 8);
  const int64_t spread = 4 * ((608 + heads - 1) / heads) + 1, least = min_records(static_cast<int>(capacity)) + 1;
  const int64_t want = spread > least ? spread : least;
  return want < stages ? want : stages;
}

constexpr size_t kRecordBytes = (kD + 2) * sizeof(float);  // O, max and sum of one head's segment
constexpr size_t kSmemBytes =
    kStages * kStageBytes + (kConsumers * 8 * kMergeHead + 2 * kConsumers * 8) * sizeof(float) + 2 * kStages * 8;

template <bool kE1M2>
int resident_ctas() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(d);
  if (it != cache.end()) return it->second;
  if (cudaFuncSetAttribute(attn_partial_kernel<kE1M2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(kSmemBytes)) != cudaSuccess)
    return 0;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, attn_partial_kernel<kE1M2>, kThreads, kSmemBytes) !=
          cudaSuccess ||
      per_sm <= 0)
    return 0;
  cache[d] = per_sm * sm_count();
  return cache[d];
}

// The partial kernel for the cache's element format, and its resident CTAs.
using PartialKernel = void (*)(const Params);
PartialKernel partial_kernel(const nvfp4_kv_cache* cache) {
  return cache->kv_format == NVFP4_KV_E1M2 ? attn_partial_kernel<true> : attn_partial_kernel<false>;
}
int resident_ctas(const nvfp4_kv_cache* cache) {
  return cache->kv_format == NVFP4_KV_E1M2 ? resident_ctas<true>() : resident_ctas<false>();
}
bool kv_format_ok(const nvfp4_kv_cache* cache) {
  return cache->kv_format == NVFP4_KV_E2M1 || cache->kv_format == NVFP4_KV_E1M2;
}

}  // namespace
}  // namespace nvfp4

using namespace nvfp4;

NVFP4_API size_t decode_attention_nvfp4_workspace_size(int32_t batch, int32_t num_q_heads, int32_t capacity) {
  if (batch <= 0 || num_q_heads <= 0 || capacity <= 0) return 0;
  return static_cast<size_t>(batch) * num_q_heads * preferred_records(batch, num_q_heads, capacity) * kRecordBytes;
}

namespace nvfp4 {
namespace {

// The smallest workspace that a call accepts; with less than
// decode_attention_nvfp4_workspace_size bytes fewer CTAs share a head.
size_t least_workspace(const nvfp4_kv_cache* cache, int32_t num_q_heads) {
  return static_cast<size_t>(cache->batch) * num_q_heads * min_records(cache->capacity) * kRecordBytes;
}

// Checks shared by the decode-attention entry points (all but the output
// buffers and the split-KV partials).
nvfp4_status attention_validate(const nvfp4_kv_cache* cache, const void* q_bf16, int32_t num_q_heads,
                                float softmax_scale) {
  if (!cache || !q_bf16 || !cache->seq_lens) return NVFP4_ERR_INVALID_ARG;
  if (!cache->k_codes || !cache->k_scales || !cache->v_codes || !cache->v_scales) return NVFP4_ERR_INVALID_ARG;
  if (!kv_format_ok(cache)) return NVFP4_ERR_INVALID_ARG;
  if (!(cache->k_gscale > 0.0f && cache->k_gscale <= FLT_MAX) || !(cache->v_gscale > 0.0f && cache->v_gscale <= FLT_MAX) ||
      !(softmax_scale > 0.0f && softmax_scale <= FLT_MAX))
    return NVFP4_ERR_INVALID_ARG;
  if (cache->head_dim != kD || cache->batch <= 0 || cache->num_kv_heads <= 0 || cache->capacity <= 0 ||
      cache->capacity % 2 || num_q_heads <= 0 || num_q_heads % cache->num_kv_heads ||
      num_q_heads / cache->num_kv_heads > 8)
    return NVFP4_ERR_SHAPE;
  if (static_cast<int64_t>(cache->batch) > 65535 || num_q_heads > 65535) return NVFP4_ERR_SHAPE;
  const int64_t n_items = static_cast<int64_t>(cache->batch) * cache->num_kv_heads * min_records(cache->capacity);
  if (n_items >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  return NVFP4_OK;
}

// Alignment of the query and cache arrays, then the partial kernel's
// parameters with its partials at `partials` and its grid size.
nvfp4_status attention_params(const nvfp4_kv_cache* cache, const void* q_bf16, int32_t num_q_heads,
                              float softmax_scale, float* partials, size_t partials_bytes, Params* prm,
                              int* grid) {
  if (!aligned(q_bf16, 16) || !aligned(cache->k_codes, 16) || !aligned(cache->v_codes, 16) ||
      !aligned(cache->k_scales, 16) || !aligned(cache->v_scales, 16))
    return NVFP4_ERR_ALIGN;
  const int ctas_max = resident_ctas(cache);
  if (ctas_max <= 0) return NVFP4_ERR_CUDA;
  const int64_t stages = (cache->capacity + kStageTok - 1) / kStageTok;
  const int64_t heads = static_cast<int64_t>(cache->batch) * cache->num_kv_heads;
  const int64_t fit = static_cast<int64_t>(partials_bytes / (kRecordBytes * cache->batch * num_q_heads));
  prm->k_codes = cache->k_codes;
  prm->k_scales = cache->k_scales;
  prm->v_codes = cache->v_codes;
  prm->v_scales = cache->v_scales;
  prm->seq_lens = cache->seq_lens;
  prm->q = static_cast<const uint16_t*>(q_bf16);
  prm->status = status_word_dev();
  prm->hkv = cache->num_kv_heads;
  prm->capacity = cache->capacity;
  prm->hq = num_q_heads;
  prm->group = num_q_heads / cache->num_kv_heads;
  prm->batch = cache->batch;
  // Never more than asked for, so that a larger workspace changes no result.
  const int64_t want = preferred_records(cache->batch, num_q_heads, cache->capacity);
  prm->records = static_cast<int>(fit < want ? fit : want);
  // Up to three stages a head's own work is shorter than what finding and
  // merging a run's parts costs (us, whole / runs: 1 x 40 heads, 154 tokens 5.9
  // / 7.0, 384 7.2 / 8.1, 512 8.1 / 6.2; 64 x 40: 10.2 / 11.3, 14.5 / 15.7).
  prm->whole = stages <= 3 || (stages <= 8 && 2 * heads >= ctas_max) || prm->records < 2;
  if (prm->whole) prm->records = 1;
  prm->logit_mult = softmax_scale * cache->k_gscale * kLog2e;
  prm->fault_skip_stage = take_fault(NVFP4_FAULT_ATTN_SKIP_STAGE) ? 1 : 0;
  // Every record the combine kernel reads is written by the partial kernel of
  // the same call, so nothing left from an earlier call needs clearing.
  prm->o_ws = partials;
  prm->ml_ws = prm->o_ws + static_cast<size_t>(cache->batch) * num_q_heads * prm->records * kD;
  const int64_t ctas = prm->whole ? heads : heads * stages;
  *grid = static_cast<int>(ctas < ctas_max ? ctas : ctas_max);
  return NVFP4_OK;
}

// The partial and the combine kernel.  With few heads of many records the
// combine's blocks take 8 x 128 threads (1 x 40 heads of 64 records: 4.3 ->
// 3.0 us); with more heads than SMs they would only crowd each other (both
// kernels, 8 x 32 heads of 8-9 records: 13.2 against 15.4 us).
template <bool kQuant>
nvfp4_status attention_launch(const nvfp4_kv_cache* cache, const Params& prm, int grid, const CombineOut& out,
                              cudaStream_t s) {
  const bool wide = prm.records > 8 && static_cast<int64_t>(prm.hq) * prm.batch <= sm_count();
  if (launch_pdl(partial_kernel(cache), dim3(grid), dim3(kThreads), kSmemBytes, s, prm) != cudaSuccess ||
      launch_pdl(wide ? attn_combine_kernel<kQuant, 8> : attn_combine_kernel<kQuant, 1>, dim3(prm.hq, prm.batch),
                 dim3(wide ? 8 * kD : kD), 0, s, static_cast<const float*>(prm.o_ws),
                 static_cast<const float*>(prm.ml_ws), prm.records, cache->v_gscale, out) != cudaSuccess)
    return NVFP4_ERR_CUDA;
  count_launches(2);
  return launch_status();
}

}  // namespace
}  // namespace nvfp4

NVFP4_API nvfp4_status decode_attention_nvfp4(const nvfp4_kv_cache* cache, const void* q_bf16, int32_t num_q_heads,
                                              float softmax_scale, void* out_bf16, void* workspace,
                                              size_t workspace_bytes, void* stream) {
  NVFP4_TRACE("decode_attention_nvfp4");
  if (!out_bf16 || !workspace) return NVFP4_ERR_INVALID_ARG;
  nvfp4_status st = attention_validate(cache, q_bf16, num_q_heads, softmax_scale);
  if (st != NVFP4_OK) return st;
  if (workspace_bytes < least_workspace(cache, num_q_heads)) return NVFP4_ERR_SHAPE;
  if (!aligned(out_bf16, 16) || !aligned(workspace, 16)) return NVFP4_ERR_ALIGN;
  Params prm;
  int grid = 0;
  st = attention_params(cache, q_bf16, num_q_heads, softmax_scale, static_cast<float*>(workspace), workspace_bytes, &prm,
                        &grid);
  if (st != NVFP4_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return attention_launch<false>(cache, prm, grid, CombineOut{static_cast<uint16_t*>(out_bf16)}, s);
}

NVFP4_API nvfp4_status decode_attention_nvfp4_quantize(const nvfp4_kv_cache* cache, const void* q_bf16,
                                                       int32_t num_q_heads, float softmax_scale, const float* g_out,
                                                       uint8_t* out_codes, uint8_t* out_scales, void* workspace,
                                                       size_t workspace_bytes, void* stream) {
  NVFP4_TRACE("decode_attention_nvfp4_quantize");
  if (!g_out || !out_codes || !out_scales || !workspace) return NVFP4_ERR_INVALID_ARG;
  nvfp4_status st = attention_validate(cache, q_bf16, num_q_heads, softmax_scale);
  if (st != NVFP4_OK) return st;
  if (workspace_bytes < least_workspace(cache, num_q_heads)) return NVFP4_ERR_SHAPE;
  if (!aligned(out_codes, 16) || !aligned(out_scales, 4) || !aligned(g_out, 4) || !aligned(workspace, 16))
    return NVFP4_ERR_ALIGN;
  Params prm;
  int grid = 0;
  st = attention_params(cache, q_bf16, num_q_heads, softmax_scale, static_cast<float*>(workspace), workspace_bytes, &prm,
                        &grid);
  if (st != NVFP4_OK) return st;
  CombineOut o{};
  o.codes = out_codes;
  o.scales = out_scales;
  o.g_out = g_out;
  o.status = status_word_dev();
  o.rows = cache->batch;
  o.kgroups = static_cast<uint32_t>(num_q_heads) * (kD / 64);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return attention_launch<true>(cache, prm, grid, o, s);
}

// ---------------------------------------------------------------------------
// Decode attention for callers that cannot allocate device memory.  The
// split-KV partials live in one file-scope device array instead of a caller
// workspace; every GPU that loads the library holds it until the process
// exits, and all calls share it.
namespace nvfp4 {
namespace {

static __device__ __align__(256) float g_attn_static_scratch[NVFP4_ATTN_STATIC_SCRATCH_BYTES / sizeof(float)];

// Device address of the static scratch for the current device, looked up once
// per device with that device current.  Host code must not hand the symbol
// itself to a kernel: on the host it is only a stand-in for the device array.
float* attn_static_scratch_dev() {
  static std::mutex mu;
  static std::map<int, float*> addr;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  auto it = addr.find(d);
  if (it != addr.end()) return it->second;
  float* p = nullptr;
  if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_attn_static_scratch) != cudaSuccess || !p) return nullptr;
  addr[d] = p;
  return p;
}

}  // namespace
}  // namespace nvfp4

NVFP4_API nvfp4_status decode_attention_nvfp4_static_scratch(const nvfp4_kv_cache* cache, const void* q_bf16,
                                                             int32_t num_q_heads, float softmax_scale,
                                                             void* out_bf16, void* stream) {
  NVFP4_TRACE("decode_attention_nvfp4_static_scratch");
  if (!out_bf16) return NVFP4_ERR_INVALID_ARG;
  nvfp4_status st = attention_validate(cache, q_bf16, num_q_heads, softmax_scale);
  if (st != NVFP4_OK) return st;
  // The partials must fit in the static scratch; larger problems are refused.
  if (least_workspace(cache, num_q_heads) > NVFP4_ATTN_STATIC_SCRATCH_BYTES) return NVFP4_ERR_SHAPE;
  if (!aligned(out_bf16, 16)) return NVFP4_ERR_ALIGN;
  float* scratch = attn_static_scratch_dev();
  if (!scratch) return NVFP4_ERR_CUDA;
  Params prm;
  int grid = 0;
  st = attention_params(cache, q_bf16, num_q_heads, softmax_scale, scratch, NVFP4_ATTN_STATIC_SCRATCH_BYTES, &prm, &grid);
  if (st != NVFP4_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return attention_launch<false>(cache, prm, grid, CombineOut{static_cast<uint16_t*>(out_bf16)}, s);
}
