// a4: quantize new K/V rows (optionally shifted by the Q-FIT post-RoPE vector
// m, Eq. 2) and write them into the NVFP4 KV cache; optionally rotate K by
// RoPE first (the fused RoPE -> shift -> quantize -> append step).
//
// A thread takes the same 16-element block of one, two or four heads of a token,
// of K or of V, so each block scale is computed once; eight lanes cover a row.
#include <cfloat>

#include "common.cuh"
#include "nvfp4_quant.cuh"

namespace nvfp4 {
namespace {

constexpr int kThreads = 256;

// kRope: K arrives before RoPE and is rotated here (rotate-half pairing,
// channel i with i + 64) with the (cos, sin) table row of its position, in
// fp32: y_i = x_i c_i - x_{i+64} s_i, y_{i+64} = x_i s_i + x_{i+64} c_i.
//
// A thread takes one 16-element block (of K or of V) of U consecutive heads of
// one token.  Eight lanes cover a row's blocks, a warp four head groups of K or
// of V (so that no lane idles while K is rotated); the RoPE partner block
// (channels 64 apart) is on lane l ^ 4.  The rotation depends on the token and
// the block only, so its (cos, sin) values, four times the bytes of a K block,
// are loaded once for U heads, and everything else that the thread reads is
// issued with them.
template <bool kRope, bool kE1M2, int U>
__global__ void __launch_bounds__(kThreads) kv_append_kernel(
    const uint16_t* __restrict__ k_in, const uint16_t* __restrict__ v_in, const int32_t* __restrict__ seq_idx,
    const int32_t* __restrict__ pos, const float* __restrict__ k_shift, const float* __restrict__ rope,
    uint32_t n_new, uint32_t hkv, FastDiv groups /* of U heads per token */, uint32_t batch, uint32_t capacity,
    uint8_t* __restrict__ kc, uint8_t* __restrict__ ks, uint8_t* __restrict__ vc, uint8_t* __restrict__ vs, float gk,
    float gv, int* status) {
  griddep_wait_and_release();
  const uint32_t n_groups = n_new * groups.d, total = (n_groups + 3u) / 4u * 64u;  // a K and a V warp per four
  const uint32_t lane = threadIdx.x & 31;
  const float qmax = kE1M2 ? 3.5f : 6.0f;  // largest element magnitude of the grid
  const float six_gk = __fmul_rn(qmax, gk), six_gv = __fmul_rn(qmax, gv);
  // 64 bits: a step may reach past 2^32 near the end.
  for (uint64_t c0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); c0 < total;
       c0 += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
    const uint32_t group = static_cast<uint32_t>(c0 >> 6) * 4u + (lane >> 3);
    const bool is_v = (c0 >> 5) & 1u;
    const bool live = group < n_groups;
    const uint32_t blk = lane & 7u;  // block within the 128-channel row
    const uint32_t tok = live ? groups.div(group) : 0;
    const uint32_t h0 = live ? (group - tok * groups.d) * U : 0;
    const uint64_t row0 = static_cast<uint64_t>(tok) * hkv + h0;
    const uint4* src = reinterpret_cast<const uint4*>((is_v ? v_in : k_in) + row0 * 128 + blk * 16);
    const int32_t b = __ldg(seq_idx + tok), p = __ldg(pos + tok);
    uint4 lo[U], hi[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      lo[u] = live ? __ldg(src + 16 * u) : make_uint4(0, 0, 0, 0);
      hi[u] = live ? __ldg(src + 16 * u + 1) : make_uint4(0, 0, 0, 0);
    }
    const bool bad = b < 0 || static_cast<uint32_t>(b) >= batch || p < 0 || static_cast<uint32_t>(p) >= capacity;
    float4 cs[kRope ? 8 : 1];
    if (kRope && !is_v) {
      // A position outside the cache is reported below; it rotates by row 0.
      const float4* row =
          reinterpret_cast<const float4*>(rope + (static_cast<uint64_t>(bad ? 0 : p) * 64 + (blk & 3u) * 16) * 2);
#pragma unroll
      for (int q = 0; q < 8; ++q) cs[q] = __ldg(row + q);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t h = h0 + u;
      float x[16];
      unpack_bf16x8(lo[u], x);
      unpack_bf16x8(hi[u], x + 8);
      if (kRope) {
        uint4 plo, phi;  // the partner block
        plo.x = __shfl_xor_sync(0xffffffffu, lo[u].x, 4);
        plo.y = __shfl_xor_sync(0xffffffffu, lo[u].y, 4);
        plo.z = __shfl_xor_sync(0xffffffffu, lo[u].z, 4);
        plo.w = __shfl_xor_sync(0xffffffffu, lo[u].w, 4);
        phi.x = __shfl_xor_sync(0xffffffffu, hi[u].x, 4);
        phi.y = __shfl_xor_sync(0xffffffffu, hi[u].y, 4);
        phi.z = __shfl_xor_sync(0xffffffffu, hi[u].z, 4);
        phi.w = __shfl_xor_sync(0xffffffffu, hi[u].w, 4);
        if (!is_v) {
          float xp[16];
          unpack_bf16x8(plo, xp);
          unpack_bf16x8(phi, xp + 8);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float cv0 = cs[q].x, sv0 = cs[q].y, cv1 = cs[q].z, sv1 = cs[q].w;
            const int e = 2 * q;
            x[e] = blk < 4 ? __fsub_rn(__fmul_rn(x[e], cv0), __fmul_rn(xp[e], sv0))
                           : __fadd_rn(__fmul_rn(xp[e], sv0), __fmul_rn(x[e], cv0));
            x[e + 1] = blk < 4 ? __fsub_rn(__fmul_rn(x[e + 1], cv1), __fmul_rn(xp[e + 1], sv1))
                               : __fadd_rn(__fmul_rn(xp[e + 1], sv1), __fmul_rn(x[e + 1], cv1));
          }
        }
      }
      if (!is_v && k_shift) {
        const float4* m4 = reinterpret_cast<const float4*>(k_shift + h * 128u + blk * 16u);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 m = __ldg(m4 + q);
          x[4 * q] = __fsub_rn(x[4 * q], m.x);
          x[4 * q + 1] = __fsub_rn(x[4 * q + 1], m.y);
          x[4 * q + 2] = __fsub_rn(x[4 * q + 2], m.z);
          x[4 * q + 3] = __fsub_rn(x[4 * q + 3], m.w);
        }
      }
      float amax = 0.0f;
#pragma unroll
      for (int i = 0; i < 16; ++i) amax = fmaxf(amax, fabsf(x[i]));
      const BlockScale bs = block_scale(amax, is_v ? gv : gk, is_v ? six_gv : six_gk);
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = __fmul_rn(x[i], bs.mult);
      const uint2 packed = kE1M2 ? make_uint2(e1m2x8(x), e1m2x8(x + 8)) : make_uint2(e2m1x8(x), e2m1x8(x + 8));
      if (!live) continue;
      if (bad) {
        if (blk == 0 && !is_v) set_status(status, NVFP4_ERR_CAPACITY);
        continue;
      }
      const uint64_t row = (static_cast<uint64_t>(b) * hkv + h) * capacity + static_cast<uint32_t>(p);
      if (!in_bounds(status, row < static_cast<uint64_t>(batch) * hkv * capacity && blk < 8u)) continue;
      reinterpret_cast<uint2*>((is_v ? vc : kc) + row * 64)[blk] = packed;
      (is_v ? vs : ks)[row * 8 + blk] = static_cast<uint8_t>(bs.code);
    }
  }
}

// The kernel for U heads per thread.
template <int U>
auto append_kernel(bool rope, bool e1m2) {
  return rope ? (e1m2 ? kv_append_kernel<true, true, U> : kv_append_kernel<true, false, U>)
              : (e1m2 ? kv_append_kernel<false, true, U> : kv_append_kernel<false, false, U>);
}

nvfp4_status append(const nvfp4_kv_cache* cache, const void* k_bf16, const void* v_bf16, const int32_t* seq_idx,
                    const int32_t* pos, int64_t n_new, const float* k_shift, const float* rope, void* stream) {
  if (!cache || !k_bf16 || !v_bf16 || !seq_idx || !pos) return NVFP4_ERR_INVALID_ARG;
  if (!cache->k_codes || !cache->k_scales || !cache->v_codes || !cache->v_scales) return NVFP4_ERR_INVALID_ARG;
  if (!(cache->k_gscale > 0.0f && cache->k_gscale <= FLT_MAX) || !(cache->v_gscale > 0.0f && cache->v_gscale <= FLT_MAX))
    return NVFP4_ERR_INVALID_ARG;
  if (cache->kv_format != NVFP4_KV_E2M1 && cache->kv_format != NVFP4_KV_E1M2) return NVFP4_ERR_INVALID_ARG;
  if (cache->head_dim != 128 || cache->batch <= 0 || cache->num_kv_heads <= 0 || cache->capacity <= 0 || n_new < 0)
    return NVFP4_ERR_SHAPE;
  if (n_new * cache->num_kv_heads * 32 >= (1ll << 32)) return NVFP4_ERR_SHAPE;
  if (!aligned(k_bf16, 16) || !aligned(v_bf16, 16) || !aligned(cache->k_codes, 16) || !aligned(cache->v_codes, 16) ||
      !aligned(cache->k_scales, 8) || !aligned(cache->v_scales, 8) || (k_shift && !aligned(k_shift, 16)) ||
      (rope && !aligned(rope, 16)))
    return NVFP4_ERR_ALIGN;
  if (n_new == 0) return NVFP4_OK;
  const bool e1m2 = cache->kv_format == NVFP4_KV_E1M2;
  const uint32_t heads = static_cast<uint32_t>(cache->num_kv_heads), tokens = static_cast<uint32_t>(n_new);
  // Heads per thread.  One while a thread per block does not fill the GPU
  // (latency); two beyond that; four with RoPE once even those are several
  // waves (the table's loads count, registers allow two CTAs per SM).  GB300,
  // U = 1 / 2 / 4, 8 heads with RoPE and shift: 64 tokens 2.2 / 2.8 / 4.0 us,
  // 1024 4.7 / 3.6 / 4.3, 4093 11.0 / 11.0 / 10.1, 65536 119 / 102 / 81;
  // without, 262144 tokens: 259 / 208 / 231.  (One block of K or V of one head
  // per thread with four such items in turn, before: 6.1, 6.4, 15.5, 167; 277.)
  const uint64_t items = static_cast<uint64_t>(tokens) * heads * 16, per_sm = items / sm_count();
  const uint32_t U = per_sm <= 512 || heads % 2 ? 1 : (rope && per_sm >= 2048 && heads % 4 == 0 ? 4 : 2);
  const auto kernel = U == 4   ? append_kernel<4>(rope, e1m2)
                      : U == 2 ? append_kernel<2>(rope, e1m2)
                               : append_kernel<1>(rope, e1m2);
  const uint64_t threads = (static_cast<uint64_t>(tokens) * (heads / U) + 3) / 4 * 64;
  uint64_t grid = (threads + kThreads - 1) / kThreads;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * 8;
  if (grid > cap) grid = cap;
  const cudaError_t e =
      launch_pdl(kernel, dim3(static_cast<int>(grid)), dim3(kThreads),
                 0, static_cast<cudaStream_t>(stream), static_cast<const uint16_t*>(k_bf16),
                 static_cast<const uint16_t*>(v_bf16), seq_idx, pos, k_shift, rope, tokens, heads,
                 FastDiv(heads / U), static_cast<uint32_t>(cache->batch),
                 static_cast<uint32_t>(cache->capacity), cache->k_codes, cache->k_scales, cache->v_codes,
                 cache->v_scales, cache->k_gscale, cache->v_gscale, status_word_dev());
  if (e != cudaSuccess) return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}

// table[p][i] = (cos, sin) of p * theta^(-2i/d): angle, sine and cosine in
// fp64, each of the two results rounded once to fp32.
__global__ void rope_table_kernel(float2* __restrict__ table, uint32_t n_pos, uint32_t half, double theta, double d) {
  griddep_wait_and_release();
  const uint64_t n = static_cast<uint64_t>(n_pos) * half;
  for (uint64_t k = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; k < n;
       k += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
    const uint32_t p = static_cast<uint32_t>(k / half), i = static_cast<uint32_t>(k % half);
    const double inv = pow(theta, -2.0 * static_cast<double>(i) / d);
    double sn, cs;
    sincos(static_cast<double>(p) * inv, &sn, &cs);
    table[k] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
  }
}

}  // namespace
}  // namespace nvfp4

using namespace nvfp4;

NVFP4_API nvfp4_status kv_append_nvfp4(const nvfp4_kv_cache* cache, const void* k_bf16, const void* v_bf16,
                                       const int32_t* seq_idx, const int32_t* pos, int64_t n_new,
                                       const float* k_shift, void* stream) {
  NVFP4_TRACE("kv_append_nvfp4");
  return append(cache, k_bf16, v_bf16, seq_idx, pos, n_new, k_shift, nullptr, stream);
}

NVFP4_API nvfp4_status kv_append_rope_nvfp4(const nvfp4_kv_cache* cache, const void* k_pre_bf16, const void* v_bf16,
                                            const int32_t* seq_idx, const int32_t* pos, int64_t n_new,
                                            const float* rope_table, int64_t rope_positions, const float* k_shift,
                                            void* stream) {
  NVFP4_TRACE("kv_append_rope_nvfp4");
  if (!cache || !rope_table) return NVFP4_ERR_INVALID_ARG;
  if (rope_positions < cache->capacity) return NVFP4_ERR_SHAPE;
  return append(cache, k_pre_bf16, v_bf16, seq_idx, pos, n_new, k_shift, rope_table, stream);
}

NVFP4_API nvfp4_status nvfp4_rope_table(float* table, int64_t n_pos, int32_t head_dim, float theta, void* stream) {
  NVFP4_TRACE("nvfp4_rope_table");
  if (n_pos < 0 || head_dim <= 0 || head_dim % 2 || n_pos * (head_dim / 2) >= (1ll << 40)) return NVFP4_ERR_SHAPE;
  if (!(theta > 1.0f && theta <= FLT_MAX)) return NVFP4_ERR_INVALID_ARG;
  if (n_pos == 0) return NVFP4_OK;
  if (!table) return NVFP4_ERR_INVALID_ARG;
  if (!aligned(table, 8)) return NVFP4_ERR_ALIGN;
  const uint64_t n = static_cast<uint64_t>(n_pos) * (head_dim / 2);
  uint64_t grid = (n + 255) / 256;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * 8;
  if (grid > cap) grid = cap;
  if (launch_pdl(rope_table_kernel, dim3(static_cast<int>(grid)), dim3(256), 0, static_cast<cudaStream_t>(stream),
                 reinterpret_cast<float2*>(table), static_cast<uint32_t>(n_pos), static_cast<uint32_t>(head_dim / 2),
                 static_cast<double>(theta), static_cast<double>(head_dim)) != cudaSuccess)
    return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}
