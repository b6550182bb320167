// a3: block-scaled NVFP4 x NVFP4 linear layer with bf16 output, on the
// 5th-generation tensor cores (tcgen05.mma kind::mxf4nvf4, 16-element blocks
// with UE4M3 scales, fp32 accumulation in tensor memory).
//
//   out[m, n] = bf16( g_a g_w sum_k a[m,k] w[n,k] )      (all linears, Appendix D.1)
//
// Persistent, warp-specialized CTAs (one per SM), tile 128 x BN x 256:
//   warp 0      TMA producer: the A and W tiles (codes via 2-D tensor maps
//               with the 128-byte swizzle) and their block scales (1-D bulk
//               copies).
//   warp 1      allocates 512 TMEM columns; one lane issues 4 MMAs of K = 64
//               per stage; its commit releases the stage.
//   warp 2      one lane copies each stage's block scales smem -> TMEM
//               (tcgen05.cp) as soon as the stage lands, so the copies run
//               ahead of, and in a different issue stream from, the MMAs.
//   warps 3..   epilogue: drain 128 accumulator columns into registers, hand
//               the accumulator back, scale by g_a g_w, round to bf16, stage in
//               swizzled shared memory and write with TMA stores.
// Every wait is bounded (NVFP4_ERR_TIMEOUT on expiry); the CTA then drains
// its copies and MMAs and frees TMEM before returning.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cfloat>
#include <map>
#include <mutex>

#include "common.cuh"
#include "nvfp4_quant.cuh"

namespace nvfp4 {
namespace {

#ifndef NVFP4_GEMM_PAIR_STAGES
#define NVFP4_GEMM_PAIR_STAGES 5
#endif

constexpr int BM = 128;
constexpr int BK = 256;  // elements per k-block = 128 bytes per row
constexpr uint32_t kTmemCols = 512;
constexpr int kEpiRows = 32, kEpiCols = 64;                 // one TMA store box (bf16)
constexpr uint32_t kEpiBufBytes = kEpiRows * kEpiCols * 2;  // 4 KiB per epilogue warp

// BN = 128: double-buffered TMEM accumulator, 4 epilogue warps.  BN = 256:
// one accumulator (TMEM also holds the scale slots) and 8 epilogue warps that
// drain it into registers and release it before storing.
template <int BN_, int STAGES_>
struct Cfg {
  static constexpr int BN = BN_;
  static constexpr int kStages = STAGES_;
  static constexpr int kAccBufs = BN == 128 ? 2 : 1;
  static constexpr int kEpiWarps = BN / 32;  // 128 accumulator columns each
  static constexpr int kThreads = 96 + 32 * kEpiWarps;  // producer, MMA, scale copier, epilogue
  static constexpr uint32_t kTileBytesA = BM * BK / 2;  // 16 KiB
  static constexpr uint32_t kTileBytesB = BN * BK / 2;
  static constexpr uint32_t kSfaBytes = 128 * (BK / 16);  // four 512-byte scale atoms
  static constexpr uint32_t kSfbBytes = kSfaBytes * (BN / 128);
  static constexpr uint32_t kStageBytes = kTileBytesA + kTileBytesB + kSfaBytes + kSfbBytes;
  static constexpr uint32_t kSfbColsPerMma = 4 * (BN / 128);
  static constexpr uint32_t kSfCols = 16 + 4 * kSfbColsPerMma;  // TMEM columns of one stage's scales
  static constexpr uint32_t kSfTmemCol = kAccBufs * BN;
  static constexpr size_t kSmemBytes =
      1024 /*align slack*/ + kStages * kStageBytes + kEpiWarps * kEpiBufBytes + 512 /*barriers*/;
  // Instruction descriptor, kind::mxf4nvf4: A and B packed E2M1 (format 1),
  // both K-major, UE4M3 scales (bit 23 = 0), N >> 3 at bit 17, M >> 4 at bit 24.
  static constexpr uint32_t kIdesc = (1u << 7) | (1u << 10) | (static_cast<uint32_t>(BN >> 3) << 17) |
                                     (static_cast<uint32_t>(BM >> 4) << 24);
  static_assert(kSfTmemCol + kStages * kSfCols <= kTmemCols, "TMEM budget");
  static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
};

// Shared-memory matrix descriptor of a K-major operand tile stored with the
// 128-byte swizzle: rows of 128 B, 8-row groups 1024 B apart (SBO).
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | (static_cast<uint64_t>(1024 >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}
// Descriptor of one 512-byte scale atom: 32 rows of 16 B, no swizzle, 8-row
// core matrices 128 B apart.
__device__ __forceinline__ uint64_t desc_sf(uint32_t saddr) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(128 >> 4) << 16) |
         (static_cast<uint64_t>(128 >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mma_fp4(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t sfa,
                                        uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%5], [%6], p;\n}" ::"r"(
          d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb)
      : "memory");
}

__device__ __forceinline__ void copy_sf_to_tmem(uint32_t taddr, uint64_t desc) {
  asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(desc) : "memory");
}

// 32 lanes x 32 consecutive fp32 columns; completion via tmem_ld_wait().
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr)
               : "memory");
  return v;
}

// Write one staged 32 x 64 bf16 box (rows of 128 B whose 16-byte chunks sit at
// chunk ^ (row % 8)) to out[y.., x..] with coalesced 16-byte stores: per
// instruction the warp writes 4 rows x 128 B; rows at or past M and chunks at or
// past N (N % 16 == 0, so a chunk is inside or outside) are skipped.  The
// CTA-pair epilogue's stores: against TMA stores of the same boxes they leave
// the TMA unit to the operand loads (32B prefill gate_up 731 -> 721 us, qkv 147.5
// -> 145.4, the other shapes unchanged).
__device__ __forceinline__ void store_box_lsu(uint32_t buf, uint16_t* out, int64_t ldo, int x, int y, int M, int N,
                                              int lane, int* status) {
  const int cc = lane & 7;
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int rr = 4 * it + (lane >> 3);
    const uint4 v = ld_shared_v4(buf + rr * 128 + ((cc ^ (rr & 7)) << 4));
    if (y + rr < M && x + cc * 8 < N && in_bounds(status, x + cc * 8 + 8 <= N))
      *reinterpret_cast<uint4*>(out + static_cast<int64_t>(y + rr) * ldo + x + cc * 8) = v;
  }
}

// Work-unit order: units walk the N tiles within groups of `group_m` row
// super-tiles, so the CTAs running at the same time share a few A and W
// tiles that stay in L2 instead of streaming all of A for every column.
__device__ __forceinline__ void unit_coords(int u, int msup, int tiles_n, int group_m, int* ms, int* nb) {
  const int per_group = group_m * tiles_n;
  const int group = u / per_group, r = u - group * per_group;
  const int rows = min(group_m, msup - group * group_m);
  *ms = group * group_m + r % rows;
  *nb = r / rows;
}

// Timeline build (-DNVFP4_TIMELINE): the 1-CTA kernel records, per CTA, the
// globaltimer at kernel entry (0), after its set-up (barriers, TMEM, the
// previous kernel's completion) (1), when the producer issued the first stage
// (2), when the first stage's data had landed for the MMA issuer (3), when the
// last MMA was issued (4), when the first epilogue warp saw the last tile's
// accumulator (5), when its stores had completed (6) and at exit (7).  The
// split-K kernel uses the same slots: 3 and 4 in the pair's leader only, 5
// when the first epilogue warp has drained the partial into shared memory,
// 6 when it has reduced and stored its box (CTAs that store one).
#ifdef NVFP4_TIMELINE
constexpr int kGemmTimelineCtas = 1024;
__device__ unsigned long long g_gemm_timeline[kGemmTimelineCtas][8];
__device__ __forceinline__ void gemm_stamp(int event) {
  if (blockIdx.x < kGemmTimelineCtas) g_gemm_timeline[blockIdx.x][event] = globaltimer_ns();
}
#else
__device__ __forceinline__ void gemm_stamp(int) {}
#endif

// Scale-format bit of the block-scaled MMA instruction descriptor (bit 23: UE8M0).
constexpr uint32_t kScaleE8M0 = 1u << 23;

struct GemmArgs {
  const uint8_t* sfa;
  const uint8_t* sfb;
  const float* ga;
  const float* gb;
  int M, N, K;
  int tiles_m, tiles_n;
  int* status;
  // OR-ed into the MMA instruction descriptor: 0 for UE4M3 block scales
  // (NVFP4), kScaleE8M0 for UE8M0 (MXFP4).  With ga == nullptr the epilogue
  // applies no global scale (MXFP4 has none).
  uint32_t idesc_fmt;
  // Fused SwiGLU + quantization epilogue (kSwiGLU): outputs.
  uint8_t* q_codes;   // [M, N/4] bytes: N/2 SwiGLU outputs per row
  uint8_t* q_scales;  // MMA layout for [M, N/2]
  const float* g_out;
  // Quantization of the fused output: 0 NVFP4 with the static scale g_out,
  // 1 MXFP4, 2 MXFP4 after the H_32 block rotation.
  uint32_t q_mode;
  // Test-only (nvfp4_debug_inject_fault): the first CTA, or both CTAs of the
  // first pair, leave their first stage neither armed nor loaded.
  int fault_skip_stage;
  // Row super-tiles per raster group (unit_coords).
  int group_m;
  // Pair kernel: units from this one on are 256 x 128 halves of a tile (the
  // last, partly filled wave); the number of tiles when no tile is split.
  int full_units;
  // Split-K kernel: CTA pairs per cluster, each taking one range of K; skinny
  // kernel: CTAs per cluster.
  int splits;
  // Skinny kernel: rows of the A box.
  int a_box_rows;
  // bf16 output [M, N] with row pitch ldo elements (the stores that do not
  // go through the output tensor map).
  uint16_t* out;
  int64_t ldo;
};

// Raster group for a GEMM with this K: with K <= 5120 the whole of A (M x K
// FP4) stays in L2 beside the W tiles in flight, so one group covers every
// row super-tile and W streams from DRAM once; longer K keeps groups of 8
// (measured on the 32B prefill shapes: gate_up 735 -> 715 us, qkv 147.5 ->
// 145.3 us with one group; down 362.5 us with 8 against 380.9 with one).
int raster_group(int64_t K, int64_t msup) {
  return static_cast<int>(K <= 5120 ? (msup < 1 ? 1 : msup) : 8);
}

template <class C>
__global__ void __launch_bounds__(C::kThreads, 1)
    nvfp4_gemm_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                      const __grid_constant__ CUtensorMap tmap_out, const GemmArgs args) {
  constexpr int BN = C::BN;
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + kStages * C::kTileBytesA;
  uint8_t* sEpi = sB + kStages * C::kTileBytesB;  // 1024-aligned: every tile above is a multiple of 1 KiB
  uint8_t* sSFA = sEpi + C::kEpiWarps * kEpiBufBytes;
  uint8_t* sSFB = sSFA + kStages * C::kSfaBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(sSFB + kStages * C::kSfbBytes);
  uint64_t* empty = full + kStages;
  uint64_t* sfready = empty + kStages;
  uint64_t* tfull = sfready + kStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint64_t* drain_cp = drain + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_cp + 1);
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kblocks = args.K / BK;
  const int kgroups = args.K / 64;
  // Work unit: one 128-row tile x one BN-column tile.
  const int msup = args.tiles_m;
  const int total_units = msup * args.tiles_n;
  const int cta_id = blockIdx.x, n_ctas = gridDim.x;
  if (threadIdx.x == 0) gemm_stamp(0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);  // the MMA commit that retires the stage
      mbar_init(&sfready[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], C::kEpiWarps);
    }
    mbar_init(drain, 1);
    mbar_init(drain_cp, 1);
    abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmap_a);
    prefetch_tmap(&tmap_b);
    prefetch_tmap(&tmap_out);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait_and_release();
  if (threadIdx.x == 0) gemm_stamp(1);
  const uint32_t tmem = *tmem_slot;

  auto fail = [&]() {
    set_status(args.status, NVFP4_ERR_TIMEOUT);
    abort_flag = 1;
  };

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------ TMA producer ---
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued_parity[kStages];
    bool issued[kStages];
    for (int s = 0; s < kStages; ++s) issued[s] = false;
    bool skip = args.fault_skip_stage && cta_id == 0;
#ifdef NVFP4_TIMELINE
    bool first_issue = true;
#endif
    for (int u = cta_id; u < total_units && !abort_flag; u += n_ctas) {
      int ms, nb;
      unit_coords(u, msup, args.tiles_n, args.group_m, &ms, &nb);
      const int mb = ms;
      const uint8_t* sfa_tile = args.sfa + (static_cast<size_t>(mb) * kgroups) * 512;
      const uint8_t* sfb_tiles = args.sfb + (static_cast<size_t>(nb) * (BN / 128) * kgroups) * 512;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!mbar_wait_bounded(&empty[stage], phase ^ 1u, &abort_flag)) { fail(); break; }
        if (skip) {
          skip = false;
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
          continue;
        }
        mbar_arrive_expect_tx(&full[stage], C::kStageBytes);
        tma_load_2d(sA + stage * C::kTileBytesA, &tmap_a, &full[stage], kb * (BK / 2), mb * BM);
        bulk_load(sSFA + stage * C::kSfaBytes, sfa_tile + static_cast<size_t>(kb) * C::kSfaBytes, C::kSfaBytes,
                  &full[stage]);
        // The stage's W scales: BN/128 row tiles of 2 KiB each.
#pragma unroll
        for (int j = 0; j < BN / 128; ++j)
          bulk_load(sSFB + stage * C::kSfbBytes + j * C::kSfaBytes,
                    sfb_tiles + (static_cast<size_t>(j) * kgroups) * 512 + static_cast<size_t>(kb) * C::kSfaBytes,
                    C::kSfaBytes, &full[stage]);
        tma_load_2d(sB + stage * C::kTileBytesB, &tmap_b, &full[stage], kb * (BK / 2), nb * BN);
#ifdef NVFP4_TIMELINE
        if (first_issue) gemm_stamp(2);
        first_issue = false;
#endif
        issued[stage] = true;
        issued_parity[stage] = phase;
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
    if (abort_flag) {
      // Let every copy destined for this CTA land before it exits.
      for (int s = 0; s < kStages; ++s)
        if (issued[s]) mbar_wait_bounded(&full[s], issued_parity[s], nullptr);
    }
  } else if (warp == 1 && lane == 0) {
    // ------------------------------------------------------- MMA issuer ---
    int stage = 0;
    uint32_t phase = 0;
    int local = 0;
    const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB), sSFA0 = smem_u32(sSFA), sSFB0 = smem_u32(sSFB);
    for (int u = cta_id; u < total_units && !abort_flag; u += n_ctas, ++local) {
      const int acc = local % C::kAccBufs;
      const uint32_t acc_phase = (local / C::kAccBufs) & 1;
      if (!mbar_wait_bounded(&tempty[acc], acc_phase ^ 1u, &abort_flag)) { fail(); break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem + acc * BN;
      bool ok = true;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!mbar_wait_bounded(&sfready[stage], phase, &abort_flag)) { fail(); ok = false; break; }
        if (local == 0 && kb == 0) gemm_stamp(3);
        tc_fence_after();
        const uint32_t sfa_col = tmem + C::kSfTmemCol + stage * C::kSfCols;
        const uint32_t sfb_col = sfa_col + 16;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          mma_fp4(d_tmem, desc_sw128(sA0 + stage * C::kTileBytesA + kk * 32),
                  desc_sw128(sB0 + stage * C::kTileBytesB + kk * 32), C::kIdesc | args.idesc_fmt, sfa_col + kk * 4,
                  sfb_col + kk * C::kSfbColsPerMma, (kb | kk) != 0);
        }
        tc_commit(&empty[stage]);
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      tc_commit(&tfull[acc]);
      gemm_stamp(4);
    }
    // Wait until every MMA issued above has retired before TMEM is freed.
    tc_commit(drain);
    mbar_wait_bounded(drain, 0, nullptr);
  } else if (warp == 2 && lane == 0) {
    // ---------------------------------------------- block scales -> TMEM ---
    // Slot `stage` is rewritten only after the stage's next `full` phase, which
    // the producer starts only after the MMAs that read the slot have retired.
    int stage = 0;
    uint32_t phase = 0;
    const uint32_t sSFA0 = smem_u32(sSFA), sSFB0 = smem_u32(sSFB);
    for (int u = cta_id; u < total_units && !abort_flag; u += n_ctas) {
      bool ok = true;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!mbar_wait_bounded(&full[stage], phase, &abort_flag)) { fail(); ok = false; break; }
        tc_fence_after();
        const uint32_t sfa_col = tmem + C::kSfTmemCol + stage * C::kSfCols;
        const uint32_t sfb_col = sfa_col + 16;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          copy_sf_to_tmem(sfa_col + kk * 4, desc_sf(sSFA0 + stage * C::kSfaBytes + kk * 512));
#pragma unroll
          for (int j = 0; j < BN / 128; ++j)
            copy_sf_to_tmem(sfb_col + kk * C::kSfbColsPerMma + j * 4,
                            desc_sf(sSFB0 + stage * C::kSfbBytes + j * C::kSfaBytes + kk * 512));
        }
        tc_commit(&sfready[stage]);
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
    }
    tc_commit(drain_cp);
    mbar_wait_bounded(drain_cp, 0, nullptr);
  } else if (warp >= 3) {
    // --------------------------------------------------------- epilogue ---
    const int quarter = warp & 3;                 // TMEM lanes this warp may access
    const int colbase = ((warp - 3) >> 2) * 128;  // accumulator columns this warp drains
    uint8_t* buf_ptr = sEpi + (warp - 3) * kEpiBufBytes;
    const uint32_t buf = smem_u32(buf_ptr);
    const float scale = args.ga ? __fmul_rn(__ldg(args.ga), __ldg(args.gb)) : 1.0f;
    int local = 0;
    for (int u = cta_id; u < total_units; u += n_ctas, ++local) {
      int ms, nb;
      unit_coords(u, msup, args.tiles_n, args.group_m, &ms, &nb);
      const int mb = ms;
      const int acc = local % C::kAccBufs;
      const uint32_t acc_phase = (local / C::kAccBufs) & 1;
      // Lane 0 waits and broadcasts, so the warp stays converged for the
      // .sync.aligned TMEM loads below even on the timeout path.
      int ok = 1;
      if (lane == 0) {
        ok = !abort_flag && mbar_wait_bounded(&tfull[acc], acc_phase, &abort_flag);
        if (!ok && !abort_flag) fail();
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      if (warp == 3 && lane == 0) gemm_stamp(5);
      tc_fence_after();
      // Drain 128 columns into registers, then hand the accumulator back.
      uint32_t r[128];
      const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BN + colbase;
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32(taddr + c * 32, r + 32 * c);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[acc]);

      // Two 32 x 64 bf16 boxes; row `lane` of a box is 8 chunks of 16 B stored
      // at chunk position (c ^ lane%8): the 128-byte swizzle the store expects.
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (lane == 0) bulk_wait_read_all();  // the previous box has left the buffer
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t* v = r + 64 * h + 8 * c;
          st_shared_v4(buf + lane * 128 + ((c ^ (lane & 7)) << 4),
                       pack_bf16x2(__uint_as_float(v[0]) * scale, __uint_as_float(v[1]) * scale),
                       pack_bf16x2(__uint_as_float(v[2]) * scale, __uint_as_float(v[3]) * scale),
                       pack_bf16x2(__uint_as_float(v[4]) * scale, __uint_as_float(v[5]) * scale),
                       pack_bf16x2(__uint_as_float(v[6]) * scale, __uint_as_float(v[7]) * scale));
        }
        fence_proxy_async_smem();
        __syncwarp();
        const int x = nb * BN + colbase + h * kEpiCols, y = mb * BM + quarter * 32;
        if (lane == 0 && x < args.N && y < args.M) {  // boxes reaching past M or N are clipped by the TMA unit
          tma_store_2d(&tmap_out, buf_ptr, x, y);
          bulk_commit_group();
        }
      }
    }
    if (lane == 0) bulk_wait_all();
    if (warp == 3 && lane == 0) gemm_stamp(6);
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (threadIdx.x == 0) gemm_stamp(7);
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// ------------------------------------------------------ CTA-pair kernel ---
// A pair of CTAs (a cluster of 2 on neighbouring SMs) computes a 256 x 256
// tile with tcgen05.mma.cta_group::2: each CTA holds its own 128 rows of A and
// its own 128-row half of the W tile in shared memory, and its 128 x 256 slice
// of the accumulator in its own TMEM.  Per SM this halves the W bytes loaded
// and the scale copies issued for the same FLOPs.  Each CTA loads the W scales
// of all 256 rows, so that each TMEM receives the full set.  The leader (rank 0)
// issues the copies and the MMAs; all loads are counted on its barriers.
//
// Per 256-deep k-block the MMAs take 512 cycles.  What kept it at 717 was no
// unit's rate but single threads' instruction streams: one producer issuing
// five loads and two expects (617 cycles per stage with MMAs and copies taken
// out), scale buffers held until the MMAs were done, and an MMA issuer that
// spent more than the last MMA's 128 cycles between two k-blocks.  So:
//   - each CTA loads its codes from warp 0 and its scales from another warp
//     (leader 3, peer 1); in the leader warp 1 issues the MMAs, warp 2 the copies;
//   - a CTA's W scales of a stage are two 128-row tiles of a 3-D map, one load.
//     (One multicast load for both CTAs was no faster, and no load goes to
//     several CTAs: replicas of this library run on several GPUs at once.)
//   - a stage's scale buffers are free for the next load once the copies have
//     read them (`full`), and TMEM slots once the MMAs have;
//   - codes and copies arrive on one barrier, so the MMA issuer waits once per
//     k-block, and it tests the next stage's barrier right after its commit;
//   - warps walk these loops converged and one elected lane issues, which
//     leaves descriptors in uniform registers (one copy warp then does what two
//     did).
// GB300, back to back: 8192 x 55296 x 5120 717 -> 641 us, 8192 x 5120 x 27648
// 361 -> 311, 8192 x 5120 x 8192 114 -> 97, 2048 x 17920 x 1536 29.1 -> 24.9
// (a form that kept W in shared memory for K <= 1536: 26.5).  The leader's warp 0
// with the scale loads beside the codes, and two copy warps: 661, 320, 99, 25.5.

__device__ __forceinline__ void mma_fp4_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t sfa, uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%5], [%6], p;\n}" ::"r"(
          d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb)
      : "memory");
}
__device__ __forceinline__ void copy_sf_to_tmem_pair(uint32_t taddr, uint64_t desc) {
  asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(desc) : "memory");
}
// Arrive on the barrier at this offset in every CTA of `mask` once all
// tcgen05 operations this thread issued for the pair have completed.
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                   smem_u32(bar)),
               "h"(mask)
               : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_slot)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// 2-D TMA load into this CTA's shared memory whose completion is counted on
// the barrier at offset `bar` in cluster CTA `lead` (the pair's even rank).
__device__ __forceinline__ void tma_load_2d_to(void* smem_dst, const void* tmap, uint64_t* bar, int x, int y,
                                               uint32_t lead) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(bar)), "r"(lead));
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(remote), "r"(x), "r"(y)
      : "memory");
}
// The same for a 3-D box at (0, y, z).
__device__ __forceinline__ void tma_load_3d_to(void* smem_dst, const void* tmap, uint64_t* bar, int y, int z,
                                               uint32_t lead) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(bar)), "r"(lead));
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(remote), "r"(0), "r"(y), "r"(z)
      : "memory");
}
// After a pipeline gave up: let the copies that this thread issued land before
// its CTA (or the CTA they go to) exits.  Copies whose barrier another CTA
// holds cannot be waited for here; a copy takes microseconds.
__device__ __forceinline__ void drain_delay() {
  const uint64_t t0 = globaltimer_ns();
  while (globaltimer_ns() - t0 < kDrainLimitNs) __nanosleep(100000);
}
// Arrive on the barrier at this shared-memory offset in CTA `rank` of the
// cluster, without release semantics.  Used only to hand the accumulator back:
// the arriving warp's TMEM loads have completed (tcgen05.wait::ld) and are
// ordered before the arrive by tcgen05.fence::before_thread_sync; no memory
// written by this thread is read by the waiter.  (A release.cluster arrive
// costs about a microsecond here, which stalled the MMAs at every tile.)
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint64_t* bar, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(bar)), "r"(rank));
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}

template <int STAGES_>
struct PairCfg {
  static constexpr int BN = 256;                 // MMA N (both halves of the pair)
  static constexpr int kStages = STAGES_;
  static constexpr int kEpiWarps = 8;            // 128 rows x 256 accumulator columns per CTA
  static constexpr int kScaleWarp = 3;           // the leader's scale producer; the peer's is warp 1
  static constexpr int kEpi0 = 4;                // first epilogue warp
  static constexpr int kThreads = 32 * (kEpi0 + kEpiWarps);
  static constexpr uint32_t kTileBytesA = BM * BK / 2;   // own 128 rows
  static constexpr uint32_t kTileBytesB = 128 * BK / 2;  // own half of the 256-row W tile
  static constexpr uint32_t kSfaBytes = 128 * (BK / 16);
  static constexpr uint32_t kSfbBytes = 2 * kSfaBytes;   // all 256 W rows
  static constexpr uint32_t kStageBytes = kTileBytesA + kTileBytesB + kSfaBytes + kSfbBytes;
  static constexpr uint32_t kSfCols = 16 + 32;
  static constexpr uint32_t kSfTmemCol = BN;
  static constexpr size_t kSmemBytes = 1024 + kStages * kStageBytes + kEpiWarps * kEpiBufBytes + 512 /*barriers*/;
  static constexpr uint32_t kIdesc = (1u << 7) | (1u << 10) | (static_cast<uint32_t>(BN >> 3) << 17) |
                                     (static_cast<uint32_t>(256 >> 4) << 24);
  static constexpr uint32_t kIdescHalf = (1u << 7) | (1u << 10) | (static_cast<uint32_t>(BN / 2 >> 3) << 17) |
                                         (static_cast<uint32_t>(256 >> 4) << 24);
  static_assert(kSfTmemCol + kStages * kSfCols <= kTmemCols, "TMEM budget");
  static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
};

template <class C, bool kSwiGLU>
__global__ void __launch_bounds__(C::kThreads, 1)
    nvfp4_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                           const __grid_constant__ CUtensorMap tmap_b_half,
                           const __grid_constant__ CUtensorMap tmap_sfa, const __grid_constant__ CUtensorMap tmap_sfb,
                           const GemmArgs args) {
  constexpr int BN = C::BN;
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + kStages * C::kTileBytesA;
  uint8_t* sEpi = sB + kStages * C::kTileBytesB;
  uint8_t* sSFA = sEpi + C::kEpiWarps * kEpiBufBytes;
  uint8_t* sSFB = sSFA + kStages * C::kSfaBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(sSFB + kStages * C::kSfbBytes);  // codes landed, scales in TMEM
  uint64_t* empty = full + kStages;
  uint64_t* sffull = empty + kStages;  // block scales landed (loaded first, so copies overlap the codes)
  uint64_t* tfull = sffull + kStages;
  uint64_t* tempty = tfull + 1;
  uint64_t* drain = tempty + 1;
  uint64_t* drain_cp = drain + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_cp + 1);
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kblocks = args.K / BK;
  const int kgroups = args.K / 64;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int msup = (args.tiles_m + 1) / 2;
  const int tiles = msup * args.tiles_n;
  // The tiles of a partly filled last wave are split into two 256 x 128 units
  // each when all of those fit in it.
  const int total_units = 2 * tiles - args.full_units;
  const int pair_id = blockIdx.x / 2, n_pairs = gridDim.x / 2;
  // Tile (ms, nb) of unit u and its columns: half -1 all 256, else 128 from 128 * half.
  auto coords = [&](int u, int* ms, int* nb, int* half) {
    *half = -1;
    const int s = u - args.full_units;
    if (s >= 0) {
      *half = s & 1;
      u = args.full_units + (s >> 1);
    }
    unit_coords(u, msup, args.tiles_n, args.group_m, ms, nb);
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      // The commit of the copies that put the stage's scales into TMEM, in the
      // leader also an expect_tx that covers both CTAs' code bytes.  It frees
      // the stage's scale buffers for the next load.
      mbar_init(&full[s], leader ? 2 : 1);
      mbar_init(&empty[s], 1);
      mbar_init(&sffull[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, 2 * C::kEpiWarps);
    mbar_init(drain, 1);
    mbar_init(drain_cp, 1);
    abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmap_a);
    prefetch_tmap(&tmap_b);
    prefetch_tmap(&tmap_b_half);
    prefetch_tmap(&tmap_sfa);
    prefetch_tmap(&tmap_sfb);
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  griddep_wait_and_release();
  const uint32_t tmem = *tmem_slot;

  auto fail = [&]() {
    set_status(args.status, NVFP4_ERR_TIMEOUT);
    abort_flag = 1;
  };

  // A producer warp walks this pair's units and k-blocks; prep(ms, nb, half)
  // gives a unit's start rows, and load(stage, kb, rows, wide), in one
  // lane, fills a stage once `free` says that it may be rewritten.
  auto produce = [&](uint64_t* free, auto&& prep, auto&& load) {
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    // Test-only injected fault: both CTAs of pair 0 leave their first stage
    // neither armed nor loaded, so no copy is ever in flight for it and the
    // consumers' bounded waits on it run out.
    bool skip = args.fault_skip_stage && pair_id == 0;
    for (int u = pair_id; u < total_units && !abort_flag; u += n_pairs) {
      int ms, nb, half;
      coords(u, &ms, &nb, &half);
      const bool wide = half < 0;
      const int2 rows = prep(ms, nb, half);
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!mbar_wait_bounded(&free[stage], phase ^ 1u, &abort_flag)) { fail(); break; }
        if (issuer && !skip) load(stage, kb, rows, wide);
        skip = false;
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
    if (abort_flag) drain_delay();
  };

  // A CTA's own A scales and both tiles of the W scales (a half unit needs only
  // the first); 8 rows of 256 bytes are the four 512-byte atoms of one (128-row
  // tile, k-block).
  auto load_scales = [&](int stage, int kb, int a_tile, int w_tile) {
    if (leader) mbar_arrive_expect_tx(&sffull[stage], 2 * (C::kSfaBytes + C::kSfbBytes));
    tma_load_2d_to(sSFA + stage * C::kSfaBytes, &tmap_sfa, &sffull[stage], 0, a_tile * kgroups * 2 + kb * 8, 0);
    tma_load_3d_to(sSFB + stage * C::kSfbBytes, &tmap_sfb, &sffull[stage], kb * 8, w_tile, 0);
  };
  if (warp == 0) {
    // ------------------------------------------------------ producer: codes ---
    produce(empty,
            [&](int ms, int nb, int half) {
              return make_int2(min(ms * 2 + static_cast<int>(rank), args.tiles_m - 1) * BM,  // a spare CTA redoes the last tile
                               nb * BN + (half < 0 ? static_cast<int>(rank) * 128
                                                   : half * 128 + static_cast<int>(rank) * 64));
            },
            [&](int stage, int kb, int2 rows, bool wide) {
              uint8_t* a_dst = sA + stage * C::kTileBytesA;
              uint8_t* b_dst = sB + stage * C::kTileBytesB;
              const CUtensorMap* map_b = wide ? &tmap_b : &tmap_b_half;
              const int kx = kb * (BK / 2);
              if (leader)  // both CTAs' codes are counted on the leader's barrier
                mbar_arrive_expect_tx(&full[stage],
                                      2 * (C::kTileBytesA + (wide ? C::kTileBytesB : C::kTileBytesB / 2)));
              tma_load_2d_to(a_dst, &tmap_a, &full[stage], kx, rows.x, 0);
              tma_load_2d_to(b_dst, map_b, &full[stage], kx, rows.y, 0);
            });
  } else if (leader ? warp == C::kScaleWarp : warp == 1) {
    // ----------------------------------------------------- producer: scales ---
    // A stage's scale buffers are free once the copies have read them: the
    // peer's `full` barrier says so, the leader's a little later (codes landed).
    produce(full,
            [&](int ms, int nb, int half) {
              return make_int2(min(ms * 2 + static_cast<int>(rank), args.tiles_m - 1), nb * 2 + max(half, 0));
            },
            [&](int stage, int kb, int2 tiles, bool) { load_scales(stage, kb, tiles.x, tiles.y); });
  } else if (warp == 1 && leader) {
    // ------------------------------------------------ MMA issuer (leader) ---
    // The whole warp walks the loop and one elected lane issues, so that the
    // descriptors stay in uniform registers: between two k-blocks the issuer
    // has only the last MMA's ~128 cycles for its barrier and its commit.
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    int local = 0;
    const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
    const uint64_t a_desc0 = desc_sw128(smem_u32(sA)), b_desc0 = desc_sw128(smem_u32(sB));
    bool ready = false;  // the next stage was seen full
    // Lanes decide together: a wait that runs out in one of them ends all.
    const auto wait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, &abort_flag)) != 0;
    };
    for (int u = pair_id; u < total_units; u += n_pairs, ++local) {
      if (!wait(tempty, (local & 1) ^ 1u)) { fail(); break; }
      tc_fence_after();
      const uint32_t idesc =
          (u < args.full_units ? C::kIdesc : C::kIdescHalf) | args.idesc_fmt;
      bool ok = true;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!ready && !wait(&full[stage], phase)) { fail(); ok = false; break; }
        tc_fence_after();
        const uint32_t sfa_col = utmem + C::kSfTmemCol + stage * C::kSfCols, sfb_col = sfa_col + 16;
        const uint64_t a_desc = a_desc0 + static_cast<uint32_t>(stage) * (C::kTileBytesA >> 4);
        const uint64_t b_desc = b_desc0 + static_cast<uint32_t>(stage) * (C::kTileBytesB >> 4);
        const int next = stage + 1 == kStages ? 0 : stage + 1;
        const uint32_t next_phase = next ? phase : phase ^ 1u;
        if (issuer) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_fp4_pair(utmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, sfa_col + kk * 4, sfb_col + kk * 8,
                         (kb | kk) != 0);
          tc_commit_pair(&empty[stage], 0x3);
        }
        ready = __all_sync(0xffffffffu, mbar_test_wait(&full[next], next_phase)) != 0;
        stage = next;
        phase = next_phase;
      }
      if (!ok) break;
      if (issuer) tc_commit_pair(tfull, 0x3);
    }
    if (issuer) tc_commit_pair(drain, 0x1);
    mbar_wait_bounded(drain, 0, nullptr);
  } else if (warp == 2 && leader) {
    // ------------------------------------- leader: block scales -> TMEM ---
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
    const uint64_t sfa_desc0 = desc_sf(smem_u32(sSFA)), sfb_desc0 = desc_sf(smem_u32(sSFB));
    for (int u = pair_id; u < total_units && !abort_flag; u += n_pairs) {
      bool ok = true;
      int ms, nb, half;
      coords(u, &ms, &nb, &half);
      const bool wide = half < 0;
      for (int kb = 0; kb < kblocks; ++kb) {
        // The scales have landed, and the MMAs that read this TMEM slot are done.
        if (!mbar_wait_bounded(&sffull[stage], phase, &abort_flag) ||
            !mbar_wait_bounded(&empty[stage], phase ^ 1u, &abort_flag)) { fail(); ok = false; break; }
        tc_fence_after();
        const uint32_t sfa_col = utmem + C::kSfTmemCol + stage * C::kSfCols, sfb_col = sfa_col + 16;
        const uint64_t sfa_desc = sfa_desc0 + static_cast<uint32_t>(stage) * (C::kSfaBytes >> 4);
        const uint64_t sfb_desc = sfb_desc0 + static_cast<uint32_t>(stage) * (C::kSfbBytes >> 4);
        if (issuer) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            copy_sf_to_tmem_pair(sfa_col + kk * 4, sfa_desc + kk * (512 >> 4));
            copy_sf_to_tmem_pair(sfb_col + kk * 8, sfb_desc + kk * (512 >> 4));
            if (wide) copy_sf_to_tmem_pair(sfb_col + kk * 8 + 4, sfb_desc + (C::kSfaBytes + kk * 512) / 16);
          }
          tc_commit_pair(&full[stage], 0x3);
        }
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
    }
    if (issuer) tc_commit_pair(drain_cp, 0x1);
    mbar_wait_bounded(drain_cp, 0, nullptr);
  } else if (kSwiGLU && warp >= C::kEpi0) {
    // ------------------------------------- epilogue: SwiGLU + NVFP4 output ---
    // W rows are interleaved in blocks of 16 (gate, then the matching up), so
    // each 32-column TMEM load gives a thread 16 gate and 16 up values of its
    // row: one 16-element block of h = SiLU(gate) * up, quantized here with
    // the static scale g_out by the library's recipe.  A warp's 128 columns
    // are 64 outputs = 4 blocks = 32 code bytes and one 32-bit scale word.
    constexpr int kEpi0 = C::kEpi0;
    const int quarter = warp & 3;
    const int colbase = ((warp - kEpi0) >> 2) * 128;
    const float scale = args.ga ? __fmul_rn(__ldg(args.ga), __ldg(args.gb)) : 1.0f;
    const float g_in = args.q_mode == 0 ? __ldg(args.g_out) : 1.0f;
    const bool g_ok = g_in > 0.0f && g_in <= FLT_MAX;
    if (!g_ok && blockIdx.x == 0 && threadIdx.x == 32 * kEpi0) set_status(args.status, NVFP4_ERR_INVALID_ARG);
    const float g = g_ok ? g_in : 1.0f, six_g = __fmul_rn(6.0f, g);
    const uint32_t q_cols = static_cast<uint32_t>(args.N) >> 1;  // SwiGLU outputs per row
    const uint32_t q_kgroups = q_cols >> 6;
    int local = 0;
    for (int u = pair_id; u < total_units; u += n_pairs, ++local) {
      int ms, nb, half;
      coords(u, &ms, &nb, &half);
      const int mb = ms * 2 + static_cast<int>(rank);  // mb >= tiles_m: nothing is stored
      int ok = 1;
      if (lane == 0) {
        ok = !abort_flag && mbar_wait_bounded(tfull, local & 1, &abort_flag);
        if (!ok && !abort_flag) fail();
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      tc_fence_after();
      uint32_t r[128];
      const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + colbase;
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32(taddr + c * 32, r + 32 * c);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_relaxed(tempty, 0);
      if (half >= 0 && colbase) continue;  // a half tile: columns 0..127 of the accumulator
      // The MMAs of the next tile run while this warp computes and stores.
      const uint32_t row = static_cast<uint32_t>(mb * BM + quarter * 32 + lane);
      const uint32_t oc0 =
          static_cast<uint32_t>(nb) * (BN / 2) + static_cast<uint32_t>((colbase + 128 * max(half, 0)) / 2);
      uint32_t codes[8], sc = 0;
      if (args.q_mode == 0) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float h[16];
          float amax = 0.0f;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            // SiLU(x) = x sigmoid(x) = x/2 (1 + tanh(x/2)): one MUFU operation.
            const float half_g = __uint_as_float(r[32 * c + i]) * (0.5f * scale);
            const float up = __uint_as_float(r[32 * c + 16 + i]) * scale;
            h[i] = fmaf(half_g, tanh_approx(half_g), half_g) * up;
            amax = fmaxf(amax, fabsf(h[i]));
          }
          const BlockScale bs = block_scale(amax, g, six_g);
#pragma unroll
          for (int i = 0; i < 16; ++i) h[i] = __fmul_rn(h[i], bs.mult);
          codes[2 * c] = g_ok ? e2m1x8(h) : 0u;
          codes[2 * c + 1] = g_ok ? e2m1x8(h + 8) : 0u;
          sc |= (g_ok ? bs.code : 0u) << (8 * c);
        }
      } else {
        // MXFP4: two TMEM loads give 32 consecutive outputs, one 32-element
        // block (optionally rotated by H_32 / sqrt(32)) with one E8M0 scale,
        // stored for both 16-element halves in the MMA scale word.
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          float h[32];
#pragma unroll
          for (int cc = 0; cc < 2; ++cc) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float half_g = __uint_as_float(r[32 * (2 * j + cc) + i]) * (0.5f * scale);
              const float up = __uint_as_float(r[32 * (2 * j + cc) + 16 + i]) * scale;
              h[16 * cc + i] = fmaf(half_g, tanh_approx(half_g), half_g) * up;
            }
          }
          if (args.q_mode == 2) hadamard32(h);
          float amax = 0.0f;
#pragma unroll
          for (int i = 0; i < 32; ++i) amax = fmaxf(amax, fabsf(h[i]));
          const uint32_t code = mx_scale_code(amax);
          const float inv = mx_inv_scale(code);
#pragma unroll
          for (int i = 0; i < 32; ++i) h[i] = __fmul_rn(h[i], inv);
          codes[4 * j] = e2m1x8(h);
          codes[4 * j + 1] = e2m1x8(h + 8);
          codes[4 * j + 2] = e2m1x8(h + 16);
          codes[4 * j + 3] = e2m1x8(h + 24);
          sc |= (code | (code << 8)) << (16 * j);
        }
      }
      if (mb < args.tiles_m) {
        // Scales for every row of the 128-row tile (rows past M hold zeros: A's
        // missing rows load as zeros), codes for rows < M.
        const uint64_t sc_off = mma_scale_offset(row, oc0 / 16, q_kgroups);
        const uint64_t sc_bytes = static_cast<uint64_t>((args.M + 127) & ~127) * (q_cols / 16);
        if (in_bounds(args.status, sc_off % 4 == 0 && sc_off + 4 <= sc_bytes))
          *reinterpret_cast<uint32_t*>(args.q_scales + sc_off) = sc;
        const uint64_t code_off = static_cast<uint64_t>(row) * (q_cols / 2) + oc0 / 2;
        if (row < static_cast<uint32_t>(args.M) &&
            in_bounds(args.status, code_off + 32 <= static_cast<uint64_t>(args.M) * (q_cols / 2))) {
          uint4* dst = reinterpret_cast<uint4*>(args.q_codes + code_off);
          dst[0] = make_uint4(codes[0], codes[1], codes[2], codes[3]);
          dst[1] = make_uint4(codes[4], codes[5], codes[6], codes[7]);
        }
      }
    }
  } else if (warp >= C::kEpi0) {
    // --------------------------------------------------------- epilogue ---
    constexpr int kEpi0 = C::kEpi0;
    const int quarter = warp & 3;
    const int colbase = ((warp - kEpi0) >> 2) * 128;
    const uint32_t buf = smem_u32(sEpi + (warp - kEpi0) * kEpiBufBytes);
    const float scale = args.ga ? __fmul_rn(__ldg(args.ga), __ldg(args.gb)) : 1.0f;
    int local = 0;
    for (int u = pair_id; u < total_units; u += n_pairs, ++local) {
      int ms, nb, half;
      coords(u, &ms, &nb, &half);
      const int mb = ms * 2 + static_cast<int>(rank);  // mb >= tiles_m: nothing is stored
      int ok = 1;
      if (lane == 0) {
        ok = !abort_flag && mbar_wait_bounded(tfull, local & 1, &abort_flag);
        if (!ok && !abort_flag) fail();
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      tc_fence_after();
      uint32_t r[128];
      const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + colbase;
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_ld32(taddr + c * 32, r + 32 * c);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_relaxed(tempty, 0);
      if (half >= 0 && colbase) continue;  // a half tile: columns 0..127 of the accumulator
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t* v = r + 64 * h + 8 * c;
          st_shared_v4(buf + lane * 128 + ((c ^ (lane & 7)) << 4),
                       pack_bf16x2(__uint_as_float(v[0]) * scale, __uint_as_float(v[1]) * scale),
                       pack_bf16x2(__uint_as_float(v[2]) * scale, __uint_as_float(v[3]) * scale),
                       pack_bf16x2(__uint_as_float(v[4]) * scale, __uint_as_float(v[5]) * scale),
                       pack_bf16x2(__uint_as_float(v[6]) * scale, __uint_as_float(v[7]) * scale));
        }
        const int x = nb * BN + 128 * max(half, 0) + colbase + h * kEpiCols, y = mb * BM + quarter * 32;
        __syncwarp();
        if (x < args.N && y < args.M) store_box_lsu(buf, args.out, args.ldo, x, y, args.M, args.N, lane, args.status);
        __syncwarp();  // the next box overwrites the staging buffer
      }
    }
  }

  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, kTmemCols);
}

// ------------------------------------------------- split-K cluster kernel ---
// For decode-sized M the 256 x 256 pair tiles are too few to occupy the GPU,
// and 128 x 128 tiles on single CTAs make every SM receive all of A and a W
// tile for the whole K (the k-loop is bound by the bytes each SM must take
// in).  Here a cluster of 2S CTAs computes one 256 x 256 tile: its S CTA
// pairs (ranks 2s and 2s + 1) each run the pair kernel's pipeline over one
// contiguous range of the k-blocks, so each W byte is still read once and
// each SM takes in 1/S of the tile's operands.  The S fp32 partial
// accumulators are then summed across the cluster in distributed shared
// memory: every CTA drains its 128 x 256 partial from TMEM into its own
// (now idle) operand ring, and after a cluster barrier the S CTAs holding the
// same 128 rows each reduce a share of the 32 x 64 output boxes, reading the
// other partials remotely and adding them in split order (so the result does
// not depend on which CTA reduces), scale by g_a g_w, round to bf16 and store
// with TMA.  One tile per cluster; no persistent loop.

// 16-byte chunk j of partial-buffer row `row` (1 KiB rows of 256 fp32): the
// chunk index is XOR-ed with row % 8 so that both the row-per-lane drain and
// the row-contiguous reduction touch every bank once per 8 lanes.
__device__ __forceinline__ uint32_t part_offset(uint32_t row, uint32_t j) {
  return row * 1024u + ((j ^ (row & 7u)) << 4);
}

// Load from a shared::cluster address (a CTA's shared memory mapped with mapa).
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t cluster_addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(cluster_addr)
               : "memory");
  return v;
}
__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
// One 32 x 64 output box of the split-K reduction: rows 32q .. 32q + 31 of
// the CTA's slice, 16-byte column chunk j (lane & 15 picks the chunk, lane >> 4
// the row of a pair).  The S partials (cluster ranks 2t + half) are read in
// batches of B row pairs with all S x B loads of a batch in flight, added in
// split order (the result does not depend on which CTA reduces), scaled,
// rounded to bf16 and written to the 128-byte-swizzled staging box.
template <int S, int B>
__device__ __forceinline__ void reduce_box(uint32_t part0, uint32_t half, int q, uint32_t j, int lane, float scale,
                                           uint32_t buf) {
  uint32_t base[S];
#pragma unroll
  for (int t = 0; t < S; ++t)
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(base[t]) : "r"(part0), "r"(2u * t + half));
  const uint32_t cchunk = static_cast<uint32_t>((lane & 15) >> 1);
#pragma unroll 1
  for (int b = 0; b < 16 / B; ++b) {
    float4 v[S][B];
#pragma unroll
    for (int t = 0; t < S; ++t)
#pragma unroll
      for (int i = 0; i < B; ++i) {
        const uint32_t rr = static_cast<uint32_t>(2 * (b * B + i) + (lane >> 4));
        v[t][i] = ld_cluster_f4(base[t] + part_offset(static_cast<uint32_t>(q * 32) + rr, j));
      }
#pragma unroll
    for (int i = 0; i < B; ++i) {
      float4 acc = v[0][i];
#pragma unroll
      for (int t = 1; t < S; ++t) {
        acc.x += v[t][i].x;
        acc.y += v[t][i].y;
        acc.z += v[t][i].z;
        acc.w += v[t][i].w;
      }
      const uint32_t rr = static_cast<uint32_t>(2 * (b * B + i) + (lane >> 4));
      st_shared_v2(buf + rr * 128 + ((cchunk ^ (rr & 7u)) << 4) + (lane & 1) * 8,
                   pack_bf16x2(acc.x * scale, acc.y * scale), pack_bf16x2(acc.z * scale, acc.w * scale));
    }
  }
}

template <class C>
__global__ void __launch_bounds__(C::kThreads, 1)
    nvfp4_gemm_splitk_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                             const __grid_constant__ CUtensorMap tmap_sfa,
                             const __grid_constant__ CUtensorMap tmap_sfb,
                             const __grid_constant__ CUtensorMap tmap_out, const GemmArgs args) {
  constexpr int BN = C::BN;
  constexpr int kStages = C::kStages;
  constexpr int kEpi0 = C::kEpi0;
  static_assert(C::kEpiWarps == 8, "eight reduction warps");
  static_assert(128u * 1024u <= kStages * (C::kTileBytesA + C::kTileBytesB), "the partial fits in the ring");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + kStages * C::kTileBytesA;
  uint8_t* sEpi = sB + kStages * C::kTileBytesB;
  uint8_t* sSFA = sEpi + C::kEpiWarps * kEpiBufBytes;
  uint8_t* sSFB = sSFA + kStages * C::kSfaBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(sSFB + kStages * C::kSfbBytes);
  uint64_t* empty = full + kStages;
  uint64_t* sffull = empty + kStages;
  uint64_t* tfull = sffull + kStages;
  uint64_t* drain = tfull + 1;
  uint64_t* drain_cp = drain + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_cp + 1);
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = args.splits;
  const int kblocks = args.K / BK;
  const int kgroups = args.K / 64;
  const uint32_t rank = cluster_ctarank();
  const uint32_t half = rank & 1u, split = rank >> 1, lead = rank & ~1u;
  const bool leader = half == 0;
  const int tile = blockIdx.x / (2 * S);
  const int msup = (args.tiles_m + 1) / 2;
  int ms, nb;
  unit_coords(tile, msup, args.tiles_n, args.group_m, &ms, &nb);
  const int k0 = static_cast<int>(split) * kblocks / S, k1 = (static_cast<int>(split) + 1) * kblocks / S;
  const int mb = ms * 2 + static_cast<int>(half);  // mb >= tiles_m: a spare CTA, nothing is stored
  if (threadIdx.x == 0) gemm_stamp(0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], leader ? 2 : 1);  // as in the pair kernel
      mbar_init(&empty[s], 1);
      mbar_init(&sffull[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(drain, 1);
    mbar_init(drain_cp, 1);
    abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmap_a);
    prefetch_tmap(&tmap_b);
    prefetch_tmap(&tmap_sfa);
    prefetch_tmap(&tmap_sfb);
    prefetch_tmap(&tmap_out);
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  griddep_wait_and_release();
  if (threadIdx.x == 0) gemm_stamp(1);
  const uint32_t tmem = *tmem_slot;

  auto fail = [&]() {
    set_status(args.status, NVFP4_ERR_TIMEOUT);
    abort_flag = 1;
  };

  bool have_partial = false;  // epilogue warps: this CTA's partial is in shared memory
  // The pair kernel's roles over one range of k-blocks.
  auto produce = [&](uint64_t* free, auto&& load) {
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    // Test-only injected fault, as in the pair kernel: the first stage of the
    // first pair is neither armed nor loaded.
    bool skip = args.fault_skip_stage && tile == 0 && split == 0;
    for (int kb = k0; kb < k1; ++kb) {
      if (!mbar_wait_bounded(&free[stage], phase ^ 1u, &abort_flag)) { fail(); break; }
      if (issuer && !skip) load(stage, kb);
      skip = false;
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
    if (abort_flag) drain_delay();
  };
  const int a_tile = min(mb, args.tiles_m - 1);  // a spare CTA reloads the last tile
  auto load_scales = [&](int stage, int kb) {
    if (leader) mbar_arrive_expect_tx(&sffull[stage], 2 * (C::kSfaBytes + C::kSfbBytes));
    tma_load_2d_to(sSFA + stage * C::kSfaBytes, &tmap_sfa, &sffull[stage], 0, a_tile * kgroups * 2 + kb * 8, lead);
    tma_load_3d_to(sSFB + stage * C::kSfbBytes, &tmap_sfb, &sffull[stage], kb * 8, nb * 2, lead);
  };
  if (warp == 0) {
    // ------------------------------------------------------ producer: codes ---
    const int b_row = nb * BN + static_cast<int>(half) * 128;
    produce(empty, [&](int stage, int kb) {
      if (leader) mbar_arrive_expect_tx(&full[stage], 2 * (C::kTileBytesA + C::kTileBytesB));
      tma_load_2d_to(sA + stage * C::kTileBytesA, &tmap_a, &full[stage], kb * (BK / 2), a_tile * BM, lead);
      tma_load_2d_to(sB + stage * C::kTileBytesB, &tmap_b, &full[stage], kb * (BK / 2), b_row, lead);
      if (kb == k0) gemm_stamp(2);
    });
  } else if (leader ? warp == C::kScaleWarp : warp == 1) {
    // ----------------------------------------------------- producer: scales ---
    produce(full, load_scales);
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer (leader) ---
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
    const uint64_t a_desc0 = desc_sw128(smem_u32(sA)), b_desc0 = desc_sw128(smem_u32(sB));
    bool ok = true;
    for (int kb = k0; kb < k1; ++kb) {
      if (!mbar_wait_bounded(&full[stage], phase, &abort_flag)) { fail(); ok = false; break; }
      if (kb == k0) gemm_stamp(3);
      tc_fence_after();
      const uint32_t sfa_col = utmem + C::kSfTmemCol + stage * C::kSfCols, sfb_col = sfa_col + 16;
      const uint64_t a_desc = a_desc0 + static_cast<uint32_t>(stage) * (C::kTileBytesA >> 4);
      const uint64_t b_desc = b_desc0 + static_cast<uint32_t>(stage) * (C::kTileBytesB >> 4);
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_fp4_pair(utmem, a_desc + 2 * kk, b_desc + 2 * kk, C::kIdesc | args.idesc_fmt, sfa_col + kk * 4,
                       sfb_col + kk * 8, (kb != k0) | (kk != 0));
        tc_commit_pair(&empty[stage], static_cast<uint16_t>(3u << lead));
      }
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
    if (issuer) {
      if (ok) tc_commit_pair(tfull, static_cast<uint16_t>(3u << lead));
      gemm_stamp(4);
      tc_commit_pair(drain, static_cast<uint16_t>(1u << lead));
    }
    mbar_wait_bounded(drain, 0, nullptr);
  } else if (warp == 2 && leader) {
    // ------------------------------------- leader: block scales -> TMEM ---
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
    const uint64_t sfa_desc0 = desc_sf(smem_u32(sSFA)), sfb_desc0 = desc_sf(smem_u32(sSFB));
    for (int kb = k0; kb < k1; ++kb) {
      if (!mbar_wait_bounded(&sffull[stage], phase, &abort_flag) ||
          !mbar_wait_bounded(&empty[stage], phase ^ 1u, &abort_flag)) { fail(); break; }
      tc_fence_after();
      const uint32_t sfa_col = utmem + C::kSfTmemCol + stage * C::kSfCols, sfb_col = sfa_col + 16;
      const uint64_t sfa_desc = sfa_desc0 + static_cast<uint32_t>(stage) * (C::kSfaBytes >> 4);
      const uint64_t sfb_desc = sfb_desc0 + static_cast<uint32_t>(stage) * (C::kSfbBytes >> 4);
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          copy_sf_to_tmem_pair(sfa_col + kk * 4, sfa_desc + kk * (512 >> 4));
          copy_sf_to_tmem_pair(sfb_col + kk * 8, sfb_desc + kk * (512 >> 4));
          copy_sf_to_tmem_pair(sfb_col + kk * 8 + 4, sfb_desc + (C::kSfaBytes + kk * 512) / 16);
        }
        tc_commit_pair(&full[stage], static_cast<uint16_t>(3u << lead));
      }
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
    if (issuer) tc_commit_pair(drain_cp, static_cast<uint16_t>(1u << lead));
    mbar_wait_bounded(drain_cp, 0, nullptr);
  } else if (warp >= kEpi0) {
    // ------------------------------- drain the partial into shared memory ---
    // The last MMA has completed (tfull), so every operand copy has landed
    // and been read: the ring is free for the partial.
    const int quarter = warp & 3;
    const int colbase = ((warp - kEpi0) >> 2) * 128;
    int ok = 1;
    if (lane == 0) {
      ok = !abort_flag && mbar_wait_bounded(tfull, 0, &abort_flag);
      if (!ok && !abort_flag) fail();
    }
    if (__shfl_sync(0xffffffffu, ok, 0)) {
      tc_fence_after();
      const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + colbase;
      const uint32_t row = static_cast<uint32_t>(quarter * 32 + lane);
      const uint32_t part0 = smem_u32(smem);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t r[64];
        tmem_ld32(taddr + 64 * h, r);
        tmem_ld32(taddr + 64 * h + 32, r + 32);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 16; ++c)
          st_shared_v4(part0 + part_offset(row, static_cast<uint32_t>(colbase / 4 + 16 * h + c)), r[4 * c],
                       r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
      }
      have_partial = true;
      if (warp == kEpi0 && lane == 0) gemm_stamp(5);
    }
  }

  // Every CTA's partial is written (or its CTA gave up) before any is read.
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();

  if (warp >= kEpi0 && !abort_flag) {
    // ------------------------------------------ reduce and store (one box) ---
    // Box p (0..15) covers rows 32 (p % 4) .. +31 and columns 64 (p / 4) .. +63
    // of this CTA's 128 x 256 slice; split s reduces boxes s, s + S, ...
    const int p = static_cast<int>(split) + (warp - kEpi0) * S;
    const bool all_ok = __all_sync(0xffffffffu, have_partial ? 1 : 0);
    if (p < 16 && mb < args.tiles_m && all_ok) {
      const int q = p & 3, pc = p >> 2;
      const float scale = args.ga ? __fmul_rn(__ldg(args.ga), __ldg(args.gb)) : 1.0f;
      uint8_t* buf_ptr = sEpi + (warp - kEpi0) * kEpiBufBytes;
      const uint32_t buf = smem_u32(buf_ptr), part0 = smem_u32(smem);
      const uint32_t j = static_cast<uint32_t>(pc * 16 + (lane & 15));
      if (S == 2) reduce_box<2, 8>(part0, half, q, j, lane, scale, buf);
      else if (S == 3) reduce_box<3, 4>(part0, half, q, j, lane, scale, buf);
      else reduce_box<4, 4>(part0, half, q, j, lane, scale, buf);
      fence_proxy_async_smem();
      __syncwarp();
      const int x = nb * BN + pc * 64, y = mb * BM + q * 32;
      if (lane == 0 && x < args.N && y < args.M) {
        tma_store_2d(&tmap_out, buf_ptr, x, y);
        bulk_commit_group();
        bulk_wait_all();
        if (warp == kEpi0) gemm_stamp(6);
      }
    }
  }

  // No CTA leaves while another may still read its partial.
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  if (threadIdx.x == 0) gemm_stamp(7);
  if (warp == 1) tmem_dealloc_pair(tmem, kTmemCols);
}

// ------------------------------------------------ skinny (M <= 128) kernel ---
// One row tile of activations: the call streams W once and the time is W's
// bytes.  A tile is 128 W rows; a cluster of S CTAs splits its K, so that
// every SM holds W loads in flight whatever N is, and two CTAs share an SM
// (one's set-up, drain and reduction under the other's stream).  The A box
// carries only the M rows rounded up to 8; the MMA's 128 A rows read on into
// whatever follows in shared memory, which only reaches accumulator rows that
// are never stored.
// The S fp32 partials ([rows, 128], 512-byte rows with swizzled 16-byte
// chunks, in the idle ring) are added across the cluster in split order, each
// CTA taking a share of the columns: deterministic for a given shape.
//   warp 0  TMA producer of the codes; before it waits for the previous kernel
//           it prefetches its first W k-blocks into L2, while the activation
//           is still being quantized (a prefetch of something that kernel
//           writes would be harmless: L2 is the point of coherence)
//   warp 1  TMEM allocation, MMAs
//   warp 2  scale copies into TMEM, ahead of the MMAs
//   warp 3  producer of the block scales
//   warps 4-7  drain, reduction, stores
// Each role is a converged warp that issues through one elected lane, as in
// the pair kernel.
// Measured with the activation's quantization before it (graph replay, W from
// DRAM), against the kernels that served these shapes before, 1 row: 5120 x
// 5120 13.6 -> 8.3 us, 7168 x 5120 14.5 -> 8.9, 27648 x 5120 31.1 -> 17.3 (W's
// bytes at the copy rate: 11.7), 5120 x 13824 23.1 -> 12.8; 32 rows: 14.6 ->
// 11.3, 15.1 -> 12.0, 29.4 -> 19.7, 19.5 -> 14.8.
template <int ROWS_>
struct SkinnyCfg {
  static constexpr int kRows = ROWS_;                      // A rows held per k-block: 32, 64 or 128
  static constexpr int kStages = ROWS_ == 32 ? 4 : 3;
  static constexpr int kEpiWarps = 4;
  static constexpr int kThreads = 128 + 32 * kEpiWarps;
  static constexpr uint32_t kTileBytesA = kRows * BK / 2;
  static constexpr uint32_t kTileBytesB = 128 * BK / 2;
  static constexpr uint32_t kSfBytes = 128 * (BK / 16);    // of A and of W: four 512-byte atoms
  static constexpr uint32_t kTmemCols = 256;               // two CTAs per SM
  static constexpr uint32_t kSfTmemCol = 128;              // 32 columns per stage after the accumulator
  static constexpr size_t kSmemBytes = 1024 + kStages * (kTileBytesA + kTileBytesB + 2 * kSfBytes) + 256 /*barriers*/;
  static constexpr uint32_t kIdesc = (1u << 7) | (1u << 10) | (static_cast<uint32_t>(128 >> 3) << 17) |
                                     (static_cast<uint32_t>(BM >> 4) << 24);
  static_assert(kSfTmemCol + kStages * 32 <= kTmemCols, "TMEM budget");
  static_assert(2 * (kSmemBytes + 1024) <= 228 * 1024, "two CTAs per SM");
  static_assert(kRows * 512u <= kStages * (kTileBytesA + kTileBytesB), "the partial fits in the ring");
};

constexpr int kSkinnyPrefetch = 4;  // W k-blocks per CTA: what arrives while a small activation is quantized

// Prefetch one 2-D box into L2.
__device__ __forceinline__ void tma_prefetch_2d(const void* tmap, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                   reinterpret_cast<uint64_t>(tmap)),
               "r"(x), "r"(y)
               : "memory");
}

// 16-byte chunk j (0..31) of row `row` of the skinny partial (512-byte rows).
__device__ __forceinline__ uint32_t skinny_part_offset(uint32_t row, uint32_t j) {
  return row * 512u + ((j ^ (row & 7u)) << 4);
}

// Add the cluster's S partials over this CTA's share of the 32 column chunks in
// split order, scale, round to bf16 and store; 128 threads, one chunk of one row each per step.
template <int S>
__device__ __forceinline__ void skinny_reduce(uint32_t part0, uint32_t rank, uint32_t tid, int n0, float scale,
                                              const GemmArgs& args) {
  uint32_t base[S];
#pragma unroll
  for (int t = 0; t < S; ++t)
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(base[t]) : "r"(part0), "r"(t));
  const uint32_t j0 = 32 * rank / S, chunks = 32 * (rank + 1) / S - j0, items = args.M * chunks;
  constexpr int kBatch = S > 4 ? 1 : 2;  // loads of kBatch x S partial chunks in flight per thread
  for (uint32_t i0 = tid; i0 < items; i0 += 128 * kBatch) {
    float4 v[kBatch][S];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const uint32_t i = i0 + 128 * b, row = i / chunks, j = j0 + i - row * chunks;
      if (i < items) {
#pragma unroll
        for (int t = 0; t < S; ++t) v[b][t] = ld_cluster_f4(base[t] + skinny_part_offset(row, j));
      }
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const uint32_t i = i0 + 128 * b, row = i / chunks, j = j0 + i - row * chunks;
      const int n = n0 + static_cast<int>(4 * j);
      if (i >= items || n >= args.N) continue;  // N % 16 == 0: a chunk is inside or outside
      float4 acc = v[b][0];
#pragma unroll
      for (int t = 1; t < S; ++t) {
        acc.x += v[b][t].x;
        acc.y += v[b][t].y;
        acc.z += v[b][t].z;
        acc.w += v[b][t].w;
      }
      if (in_bounds(args.status, row < static_cast<uint32_t>(args.M) && n + 4 <= args.N))
        *reinterpret_cast<uint2*>(args.out + static_cast<int64_t>(row) * args.ldo + n) =
            make_uint2(pack_bf16x2(acc.x * scale, acc.y * scale), pack_bf16x2(acc.z * scale, acc.w * scale));
    }
  }
}

// SwiGLU and quantization of the fp32 tile in this CTA's own ring (one CTA per
// tile).  W rows are interleaved in blocks of 16 (gate, then the matching up),
// so a thread takes 32 columns of a row: one 16-element block c of the output.
// A warp takes 8 rows and step, lanes 8c..8c+7 those of block c (whose chunks
// the swizzle spreads over all banks); the two halves of a 32-element block are
// lanes l and l ^ 8.  The arithmetic is the CTA-pair kernel's, element by
// element.
__device__ __forceinline__ void skinny_swiglu(const uint8_t* part, uint32_t warp, uint32_t lane, int nb, float scale,
                                              const GemmArgs& args) {
  const float g_in = args.q_mode == 0 ? __ldg(args.g_out) : 1.0f;
  const bool g_ok = g_in > 0.0f && g_in <= FLT_MAX;
  if (!g_ok && blockIdx.x == 0 && warp == 0 && lane == 0) set_status(args.status, NVFP4_ERR_INVALID_ARG);
  const float g = g_ok ? g_in : 1.0f, six_g = __fmul_rn(6.0f, g);
  const uint32_t q_cols = static_cast<uint32_t>(args.N) >> 1, oc0 = static_cast<uint32_t>(nb) * 64;
  const uint32_t M = static_cast<uint32_t>(args.M), c = lane >> 3;
  const uint64_t sc_bytes = 128ull * (q_cols / 16), code_bytes = static_cast<uint64_t>(M) * (q_cols / 2);
  auto store_scales = [&](uint32_t row, uint32_t sc) {
    const uint64_t off = mma_scale_offset(row, oc0 / 16, q_cols >> 6);
    if (in_bounds(args.status, off % 4 == 0 && off + 4 <= sc_bytes)) *reinterpret_cast<uint32_t*>(args.q_scales + off) = sc;
  };
  for (uint32_t r0 = 8 * warp; r0 < M; r0 += 32) {
    const uint32_t row = r0 + (lane & 7);
    float v[32], h[16];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 x = row < M ? *reinterpret_cast<const float4*>(part + skinny_part_offset(row, 8 * c + q))
                               : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      v[4 * q] = x.x;
      v[4 * q + 1] = x.y;
      v[4 * q + 2] = x.z;
      v[4 * q + 3] = x.w;
    }
    float amax = 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float half_g = v[i] * (0.5f * scale), up = v[16 + i] * scale;
      h[i] = fmaf(half_g, tanh_approx(half_g), half_g) * up;
    }
    if (args.q_mode == 2) {  // hadamard32, its last stage across the lanes
#pragma unroll
      for (int s = 1; s < 16; s <<= 1)
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if ((i & s) == 0) {
            const float a = h[i], b = h[i + s];
            h[i] = __fadd_rn(a, b);
            h[i + s] = __fsub_rn(a, b);
          }
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float other = __shfl_xor_sync(0xffffffffu, h[i], 8);
        h[i] = __fmul_rn(c & 1 ? __fsub_rn(other, h[i]) : __fadd_rn(h[i], other), __uint_as_float(kInvSqrt32Bits));
      }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) amax = fmaxf(amax, fabsf(h[i]));
    uint32_t code;
    float mult;
    if (args.q_mode == 0) {
      const BlockScale bs = block_scale(amax, g, six_g);
      code = g_ok ? bs.code : 0u;
      mult = bs.mult;
    } else {
      code = mx_scale_code(fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 8)));
      mult = mx_inv_scale(code);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) h[i] = __fmul_rn(h[i], mult);
    uint32_t sc = code << (8 * c);
    sc |= __shfl_xor_sync(0xffffffffu, sc, 8);
    sc |= __shfl_xor_sync(0xffffffffu, sc, 16);
    const uint64_t off = static_cast<uint64_t>(row) * (q_cols / 2) + oc0 / 2 + 8 * c;
    if (row < M && in_bounds(args.status, off + 8 <= code_bytes))
      *reinterpret_cast<uint2*>(args.q_codes + off) = make_uint2(g_ok ? e2m1x8(h) : 0u, g_ok ? e2m1x8(h + 8) : 0u);
    if (c == 0) store_scales(row, sc);
  }
  // Scales of the 128-row tile's further rows: those of zeros.
  const uint32_t zero = args.q_mode == 0 ? (g_ok ? block_scale(0.0f, g, six_g).code : 0u) : mx_scale_code(0.0f);
  for (uint32_t row = ((M + 7) & ~7u) + 32 * warp + lane; row < 128; row += 128) store_scales(row, zero * 0x01010101u);
}

// kSwiGLU: one CTA per tile (args.splits == 1).
template <class C, bool kSwiGLU = false>
__global__ void __launch_bounds__(C::kThreads, 2)
    nvfp4_gemm_skinny_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                             const GemmArgs args) {
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;  // the MMA's reads past a short A slot end inside sB
  uint8_t* sB = sA + kStages * C::kTileBytesA;
  uint8_t* sSFA = sB + kStages * C::kTileBytesB;
  uint8_t* sSFB = sSFA + kStages * C::kSfBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(sSFB + kStages * C::kSfBytes);
  uint64_t* empty = full + kStages;
  uint64_t* sffull = empty + kStages;
  uint64_t* tfull = sffull + kStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull + 1);
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = args.splits;
  const int kblocks = args.K / BK;
  const int split = static_cast<int>(cluster_ctarank());
  const int nb = blockIdx.x / S;
  const int k0 = split * kblocks / S, k1 = (split + 1) * kblocks / S;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 2);  // the codes' expect_tx, and the commit of the scale copies
      mbar_init(&empty[s], 1);
      mbar_init(&sffull[s], 1);
    }
    mbar_init(tfull, 1);
    abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmap_a);
    prefetch_tmap(&tmap_b);
    for (int kb = k0; kb < min(k1, k0 + kSkinnyPrefetch); ++kb) tma_prefetch_2d(&tmap_b, kb * (BK / 2), nb * 128);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, C::kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait_and_release();
  const uint32_t tmem = *tmem_slot;

  auto fail = [&]() {
    set_status(args.status, NVFP4_ERR_TIMEOUT);
    abort_flag = 1;
  };

  bool have_partial = false;
  // Walks this CTA's k-blocks: load(stage, kb) in one lane once `free` allows.
  auto produce = [&](uint64_t* free, auto&& load) {
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    bool skip = args.fault_skip_stage && blockIdx.x == 0;
    for (int kb = k0; kb < k1; ++kb) {
      if (!mbar_wait_bounded(&free[stage], phase ^ 1u, &abort_flag)) { fail(); break; }
      if (issuer && !skip) load(stage, kb);
      skip = false;
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
    if (abort_flag) drain_delay();
  };
  if (warp == 0) {
    // ------------------------------------------------------ producer: codes ---
    const uint32_t bytes = static_cast<uint32_t>(args.a_box_rows) * (BK / 2) + C::kTileBytesB;
    produce(empty, [&](int stage, int kb) {
      mbar_arrive_expect_tx(&full[stage], bytes);
      tma_load_2d(sB + stage * C::kTileBytesB, &tmap_b, &full[stage], kb * (BK / 2), nb * 128);
      tma_load_2d(sA + stage * C::kTileBytesA, &tmap_a, &full[stage], kb * (BK / 2), 0);
    });
  } else if (warp == 3) {
    // ----------------------------------------------------- producer: scales ---
    // A stage's scale buffers are free once the previous copies have read
    // them, which its `full` phase includes.
    const uint8_t* sfb_tile = args.sfb + static_cast<size_t>(nb) * kblocks * C::kSfBytes;
    produce(full, [&](int stage, int kb) {
      const size_t off = static_cast<size_t>(kb) * C::kSfBytes;
      mbar_arrive_expect_tx(&sffull[stage], 2 * C::kSfBytes);
      bulk_load(sSFB + stage * C::kSfBytes, sfb_tile + off, C::kSfBytes, &sffull[stage]);
      bulk_load(sSFA + stage * C::kSfBytes, args.sfa + off, C::kSfBytes, &sffull[stage]);
    });
  } else if (warp == 1) {
    // ------------------------------------------------------- MMA issuer ---
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
    const uint64_t a_desc0 = desc_sw128(smem_u32(sA)), b_desc0 = desc_sw128(smem_u32(sB));
    for (int kb = k0; kb < k1; ++kb) {
      if (!mbar_wait_bounded(&full[stage], phase, &abort_flag)) { fail(); break; }
      tc_fence_after();
      const uint32_t sfa_col = utmem + C::kSfTmemCol + stage * 32, sfb_col = sfa_col + 16;
      const uint64_t a_desc = a_desc0 + static_cast<uint32_t>(stage) * (C::kTileBytesA >> 4);
      const uint64_t b_desc = b_desc0 + static_cast<uint32_t>(stage) * (C::kTileBytesB >> 4);
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_fp4(utmem, a_desc + 2 * kk, b_desc + 2 * kk, C::kIdesc | args.idesc_fmt, sfa_col + kk * 4,
                  sfb_col + kk * 4, (kb != k0) | (kk != 0));
        tc_commit(&empty[stage]);
      }
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
    // Also on the timeout path: every MMA issued has retired before TMEM is freed.
    if (issuer) tc_commit(tfull);
    mbar_wait_bounded(tfull, 0, nullptr);
  } else if (warp == 2) {
    // ---------------------------------------------- block scales -> TMEM ---
    const bool issuer = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
    const uint64_t sfa_desc0 = desc_sf(smem_u32(sSFA)), sfb_desc0 = desc_sf(smem_u32(sSFB));
    for (int kb = k0; kb < k1; ++kb) {
      // The scales have landed, and the MMAs that read this TMEM slot are done.
      if (!mbar_wait_bounded(&sffull[stage], phase, &abort_flag) ||
          !mbar_wait_bounded(&empty[stage], phase ^ 1u, &abort_flag)) { fail(); break; }
      tc_fence_after();
      const uint32_t sfa_col = utmem + C::kSfTmemCol + stage * 32, sfb_col = sfa_col + 16;
      const uint64_t off = static_cast<uint32_t>(stage) * (C::kSfBytes >> 4);
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          copy_sf_to_tmem(sfa_col + kk * 4, sfa_desc0 + off + kk * (512 >> 4));
          copy_sf_to_tmem(sfb_col + kk * 4, sfb_desc0 + off + kk * (512 >> 4));
        }
        tc_commit(&full[stage]);
      }
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
    // The MMAs that read the last copies are waited for above; on the timeout
    // path copies may be in flight still.
    if (abort_flag) drain_delay();
  } else if (warp >= 4) {
    // ------------------------------- drain the partial into shared memory ---
    const int quarter = warp & 3;  // TMEM lanes this warp may access = accumulator rows
    int ok = 1;
    if (lane == 0) {
      ok = mbar_wait_bounded(tfull, 0, &abort_flag) && !abort_flag;
      if (!ok && !abort_flag) fail();
    }
    if (__shfl_sync(0xffffffffu, ok, 0)) {
      tc_fence_after();
      if (quarter * 32 < C::kRows) {
        const uint32_t row = static_cast<uint32_t>(quarter * 32 + lane), part0 = smem_u32(smem);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t r[32];
          tmem_ld32(tmem + (static_cast<uint32_t>(quarter * 32) << 16) + c * 32, r);
          tmem_ld_wait();
#pragma unroll
          for (int q = 0; q < 8; ++q)
            st_shared_v4(part0 + skinny_part_offset(row, static_cast<uint32_t>(8 * c + q)), r[4 * q], r[4 * q + 1],
                         r[4 * q + 2], r[4 * q + 3]);
        }
      }
      have_partial = true;
    }
  }

  // Every CTA's partial is written (or its CTA gave up) before any is read.
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();

  if (warp >= 4 && !abort_flag && __all_sync(0xffffffffu, have_partial ? 1 : 0)) {
    const float scale = args.ga ? __fmul_rn(__ldg(args.ga), __ldg(args.gb)) : 1.0f;
    const uint32_t part0 = smem_u32(smem);
    const uint32_t tid = threadIdx.x - 128;
    const int n0 = nb * 128;
    if constexpr (kSwiGLU) {
      skinny_swiglu(smem, tid >> 5, tid & 31, nb, scale, args);
    } else switch (S) {
      case 1: skinny_reduce<1>(part0, split, tid, n0, scale, args); break;
      case 2: skinny_reduce<2>(part0, split, tid, n0, scale, args); break;
      case 3: skinny_reduce<3>(part0, split, tid, n0, scale, args); break;
      case 4: skinny_reduce<4>(part0, split, tid, n0, scale, args); break;
      case 5: skinny_reduce<5>(part0, split, tid, n0, scale, args); break;
      case 6: skinny_reduce<6>(part0, split, tid, n0, scale, args); break;
      case 7: skinny_reduce<7>(part0, split, tid, n0, scale, args); break;
      default: skinny_reduce<8>(part0, split, tid, n0, scale, args); break;
    }
  }

  // No CTA leaves while another may still read its partial.
  cluster_sync_all();
  if (warp == 1) tmem_dealloc(tmem, C::kTmemCols);
}

// ------------------------------------- quantize-in-prologue linear kernel ---
// a1 + a2 + a3 in one launch for an activation of at most 32 rows and K of
// at most 1536: every CTA reads the whole bf16 activation x (at most 96 KB,
// an L2 hit after the first CTA), reduces its amax, forms the tensor scale g_a
// and quantizes x into its own shared memory in the MMA layout (codes in the
// 128-byte-swizzled K-major tiles the tensor core reads, block scales in
// 512-byte atoms), exactly as nvfp4_quantize_dynamic would; no grid barrier
// is needed because each CTA does the reduction itself.  A and its scales then
// stay resident (A scales in TMEM for the whole K) while the producer streams
// only W through a 5-stage ring, from the kernel's first instruction on.
//   warp 0      TMA producer for W codes and scales (skips the prologue)
//   warps 1-11  prologue (amax, then quantization), then:
//   warp 1      TMEM allocation; MMAs
//   warp 2      scale copies: each stage's W scales, for the CTA's first tile
//               with that k-block's A scales
//   warps 4, 8  epilogue, 64 of 128 columns each (the two warps that reach
//               TMEM lanes 0-31, where the at most 32 rows are)
// Latency-bound (12 CTAs at N = 1536, 0.02 of HBM): what counts is the chain
// x -> amax -> block scales -> scale copies -> MMAs -> stores.  A's rows and
// scales past M are whatever shared memory holds; they only reach accumulator
// rows that are never stored.  16 x 1536 x 1536 back to back 9.1 -> 6.5 us, 32
// rows 10.3 -> 7.9, 16 x 17920 x 1536 9.6 -> 7.0 (before: padding zeroed, one
// thread combining the warps' maxima, all A scales copied before the first
// MMA, TMA stores).
struct DynCfg {
  static constexpr int BN = 128;
  static constexpr int kStages = 5;
  static constexpr int kMaxKb = 6;                          // K <= 1536
  static constexpr int kMaxRows = 32;                       // M <= 32
  static constexpr int kEpiWarps = 2;
  // The others only help with the prologue, whose per-block arithmetic
  // (E4M3 scale, reciprocal, 16 conversions) is latency-bound with few warps.
  static constexpr int kThreads = 384;
  static constexpr int kProThreads = kThreads - 32;          // warps 1-11
  static constexpr uint32_t kTileBytesA = BM * BK / 2;       // 16 KiB per k-block
  static constexpr uint32_t kTileBytesB = BN * BK / 2;       // 16 KiB per stage
  static constexpr uint32_t kSfaBytes = 128 * (BK / 16);     // 2 KiB per k-block: four 512-byte atoms
  static constexpr uint32_t kSfbBytes = kSfaBytes;
  static constexpr uint32_t kSfaResCol = 2 * BN;             // A scales: 16 columns per k-block
  static constexpr uint32_t kSfbCol = kSfaResCol + 16 * kMaxKb;  // W scales: 16 columns per stage
  static constexpr size_t kSmemBytes = 1024 + kMaxKb * (kTileBytesA + kSfaBytes) +
                                       kStages * (kTileBytesB + kSfbBytes) + kEpiWarps * kEpiBufBytes + 512;
  static constexpr uint32_t kIdesc = (1u << 7) | (1u << 10) | (static_cast<uint32_t>(BN >> 3) << 17) |
                                     (static_cast<uint32_t>(BM >> 4) << 24);
  static_assert(kSfbCol + kStages * 16 <= kTmemCols, "TMEM budget");
  static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
};

struct DynArgs {
  const uint16_t* x;  // bf16 [M, K], row pitch ldx elements
  int64_t ldx;
  const uint8_t* sfb;
  const float* gb;
  float* g_out;  // optional: g_a
  uint16_t* out;
  int64_t ldo;
  FastDiv kb16;  // 16-element blocks per row
  int M, N, K;
  int tiles_n;
  int* status;
  int fault_skip_stage;  // as in GemmArgs
};

__device__ __forceinline__ void named_barrier(uint32_t id, uint32_t threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void st_shared_v2_u32(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void st_shared_u8(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <class C>
__global__ void __launch_bounds__(C::kThreads, 1)
    nvfp4_linear_dyn_kernel(const __grid_constant__ CUtensorMap tmap_b, const DynArgs args) {
  constexpr int BN = C::BN;
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;                                        // resident A, one 16 KiB tile per k-block
  uint8_t* sB = sA + C::kMaxKb * C::kTileBytesA;
  uint8_t* sEpi = sB + kStages * C::kTileBytesB;
  uint8_t* sSFA = sEpi + C::kEpiWarps * kEpiBufBytes;        // resident A scale atoms
  uint8_t* sSFB = sSFA + C::kMaxKb * C::kSfaBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(sSFB + kStages * C::kSfbBytes);
  uint64_t* empty = full + kStages;
  uint64_t* sfready = empty + kStages;
  uint64_t* tfull = sfready + kStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint64_t* drain_cp = drain + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_cp + 1);
  __shared__ volatile int abort_flag;
  __shared__ uint32_t warp_max[C::kThreads / 32];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kblocks = args.K / BK;
  const int kgroups = args.K / 64;
  const int total_units = args.tiles_n;
  const int cta_id = blockIdx.x, n_ctas = gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&sfready[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], C::kEpiWarps);
    }
    mbar_init(drain, 1);
    mbar_init(drain_cp, 1);
    abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmap_b);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait_and_release();
  const uint32_t tmem = *tmem_slot;

  auto fail = [&]() {
    set_status(args.status, NVFP4_ERR_TIMEOUT);
    abort_flag = 1;
  };

  if (warp == 0) {
    // ------------------------------------------------------ TMA producer ---
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued = 0, issued_parity = 0;  // one bit per stage
      bool skip = args.fault_skip_stage && cta_id == 0;
      for (int u = cta_id; u < total_units && !abort_flag; u += n_ctas) {
        const uint8_t* sfb_tile = args.sfb + (static_cast<size_t>(u) * kgroups) * 512;
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait_bounded(&empty[stage], phase ^ 1u, &abort_flag)) { fail(); break; }
          if (skip) {
            skip = false;
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
            continue;
          }
          mbar_arrive_expect_tx(&full[stage], C::kTileBytesB + C::kSfbBytes);
          bulk_load(sSFB + stage * C::kSfbBytes, sfb_tile + static_cast<size_t>(kb) * C::kSfbBytes, C::kSfbBytes,
                    &full[stage]);
          tma_load_2d(sB + stage * C::kTileBytesB, &tmap_b, &full[stage], kb * (BK / 2), u * BN);
          issued |= 1u << stage;
          issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (abort_flag)
        for (int s = 0; s < kStages; ++s)
          if (issued >> s & 1u) mbar_wait_bounded(&full[s], issued_parity >> s & 1u, nullptr, kDrainLimitNs);
    }
  } else {
    // ------------------------------- prologue: g_a and A into shared memory ---
    // Thread pt owns the 16-element blocks pt, pt + 352, ... of x in row-major
    // block order; they stay in registers from the amax pass to the
    // quantization pass, so x is read once.
    constexpr int kKeep = 10;
    static_assert(kKeep * C::kProThreads >= C::kMaxRows * C::kMaxKb * (BK / 16), "x fits in registers");
    const uint32_t pt = threadIdx.x - 32;
    const uint32_t live = static_cast<uint32_t>(args.M) * args.kb16.d;
    auto block_src = [&](uint32_t b) {
      const uint32_t r = args.kb16.div(b), j = b - r * args.kb16.d;
      return reinterpret_cast<const uint4*>(args.x + static_cast<int64_t>(r) * args.ldx + j * 16);
    };
    uint4 lo[kKeep], hi[kKeep];
#pragma unroll
    for (int i = 0; i < kKeep; ++i) {
      const uint32_t b = pt + i * C::kProThreads;
      lo[i] = hi[i] = make_uint4(0, 0, 0, 0);
      if (b < live) {
        const uint4* src = block_src(b);
        lo[i] = __ldg(src);
        hi[i] = __ldg(src + 1);
      }
    }
    const uint32_t sA0 = smem_u32(sA), sSFA0 = smem_u32(sSFA);
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < kKeep; ++i) m = max(m, max(amax_bits_bf16x8(lo[i]), amax_bits_bf16x8(hi[i])));
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) warp_max[warp] = m;
    named_barrier(1, C::kProThreads);
    // g_a = amax / (6 * 448), or 1 for an all-zero tensor: the dynamic
    // quantizer's tensor scale, bit for bit, in every thread.
    const float amax_x = __uint_as_float(
        __reduce_max_sync(0xffffffffu, lane >= 1 && lane < C::kThreads / 32 ? warp_max[lane] : 0u) << 16);
    const float g = amax_x > 0.0f ? __fdiv_rn(amax_x, 2688.0f) : 1.0f, six_g = __fmul_rn(6.0f, g);
    if (blockIdx.x == 0 && pt == 0 && args.g_out) *args.g_out = g;
    // One 16-element block: E4M3 scale and 16 E2M1 codes, stored where the
    // TMA load of the two-call path would have put them (row r at r * 128 in
    // its k-block tile, 16-byte chunk c at (c ^ r % 8) * 16) and the scale
    // byte at its place in the 512-byte atom of its 64-element group.
    auto quantize_block = [&](uint32_t b, const uint4 v0, const uint4 v1) {
      const uint32_t r = args.kb16.div(b), j = b - r * args.kb16.d;
      float xf[16];
      unpack_bf16x8(v0, xf);
      unpack_bf16x8(v1, xf + 8);
      const float amax = __uint_as_float(max(amax_bits_bf16x8(v0), amax_bits_bf16x8(v1)) << 16);
      const BlockScale bs = block_scale(amax, g, six_g);
      float q[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) q[i] = __fmul_rn(xf[i], bs.mult);
      const uint32_t kb = j >> 4, e = j & 15u;
      st_shared_v2_u32(sA0 + kb * C::kTileBytesA + r * 128u + (((e >> 1) ^ (r & 7u)) << 4) + (e & 1u) * 8u,
                       e2m1x8(q), e2m1x8(q + 8));
      st_shared_u8(sSFA0 + (j >> 2) * 512u + (r & 31u) * 16u + ((r >> 5) & 3u) * 4u + (j & 3u), bs.code);
    };
#pragma unroll
    for (int i = 0; i < kKeep; ++i) {
      const uint32_t b = pt + i * C::kProThreads;
      if (b < live) quantize_block(b, lo[i], hi[i]);
    }
    fence_proxy_async_smem();  // the tensor core reads A and its scales through the async proxy
    named_barrier(1, C::kProThreads);

    if (warp == 1) {
      // ------------------------------------------------------- MMA issuer ---
      const bool issuer = elect_one();
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
      const uint64_t a_desc0 = desc_sw128(sA0), b_desc0 = desc_sw128(smem_u32(sB));
      bool ok = true;
      for (int u = cta_id; ok && u < total_units && !abort_flag; u += n_ctas, ++local) {
        const int acc = local & 1;
        const uint32_t acc_phase = (local >> 1) & 1;
        if (!mbar_wait_bounded(&tempty[acc], acc_phase ^ 1u, &abort_flag)) { fail(); break; }
        tc_fence_after();
        const uint32_t d_tmem = utmem + acc * BN;
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait_bounded(&sfready[stage], phase, &abort_flag)) { fail(); ok = false; break; }
          tc_fence_after();
          const uint32_t sfa_col = utmem + C::kSfaResCol + kb * 16, sfb_col = utmem + C::kSfbCol + stage * 16;
          const uint64_t a_desc = a_desc0 + static_cast<uint32_t>(kb) * (C::kTileBytesA >> 4);
          const uint64_t b_desc = b_desc0 + static_cast<uint32_t>(stage) * (C::kTileBytesB >> 4);
          if (issuer) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_fp4(d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, C::kIdesc, sfa_col + kk * 4, sfb_col + kk * 4,
                      (kb | kk) != 0);
            tc_commit(&empty[stage]);
          }
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (ok && issuer) tc_commit(&tfull[acc]);
      }
      if (issuer) tc_commit(drain);
      mbar_wait_bounded(drain, 0, nullptr);
    } else if (warp == 2) {
      // ------------------------------------------- block scales -> TMEM ---
      const bool issuer = elect_one();
      int stage = 0;
      uint32_t phase = 0;
      const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
      const uint64_t sfa_desc0 = desc_sf(sSFA0), sfb_desc0 = desc_sf(smem_u32(sSFB));
      bool ok = true;
      for (int u = cta_id; ok && u < total_units && !abort_flag; u += n_ctas) {
        const bool with_a = u == cta_id;
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait_bounded(&full[stage], phase, &abort_flag)) { fail(); ok = false; break; }
          tc_fence_after();
          const uint32_t sfa_col = utmem + C::kSfaResCol + kb * 16, sfb_col = utmem + C::kSfbCol + stage * 16;
          const uint64_t sfa_desc = sfa_desc0 + static_cast<uint32_t>(kb) * (C::kSfaBytes >> 4);
          const uint64_t sfb_desc = sfb_desc0 + static_cast<uint32_t>(stage) * (C::kSfbBytes >> 4);
          if (issuer) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              if (with_a) copy_sf_to_tmem(sfa_col + kk * 4, sfa_desc + kk * (512 >> 4));
              copy_sf_to_tmem(sfb_col + kk * 4, sfb_desc + kk * (512 >> 4));
            }
            tc_commit(&sfready[stage]);
          }
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (issuer) tc_commit(drain_cp);
      mbar_wait_bounded(drain_cp, 0, nullptr);
    } else if (warp == 4 || warp == 8) {
      // --------------------------------------------------------- epilogue ---
      // 32 rows x 64 columns; row `lane` of the staged box is 8 chunks of 16 B
      // at chunk position (c ^ lane % 8).
      const int colbase = warp == 8 ? kEpiCols : 0;
      const uint32_t buf = smem_u32(sEpi + (warp == 8 ? kEpiBufBytes : 0));
      const float scale = __fmul_rn(g, __ldg(args.gb));
      int local = 0;
      for (int u = cta_id; u < total_units; u += n_ctas, ++local) {
        const int acc = local & 1;
        const uint32_t acc_phase = (local >> 1) & 1;
        int ok = 1;
        if (lane == 0) {
          ok = !abort_flag && mbar_wait_bounded(&tfull[acc], acc_phase, &abort_flag);
          if (!ok && !abort_flag) fail();
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) break;
        tc_fence_after();
        uint32_t r[64];
        const uint32_t taddr = tmem + acc * BN + colbase;
        tmem_ld32(taddr, r);
        tmem_ld32(taddr + 32, r + 32);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[acc]);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint32_t* v = r + 8 * c;
          st_shared_v4(buf + lane * 128 + ((c ^ (lane & 7)) << 4),
                       pack_bf16x2(__uint_as_float(v[0]) * scale, __uint_as_float(v[1]) * scale),
                       pack_bf16x2(__uint_as_float(v[2]) * scale, __uint_as_float(v[3]) * scale),
                       pack_bf16x2(__uint_as_float(v[4]) * scale, __uint_as_float(v[5]) * scale),
                       pack_bf16x2(__uint_as_float(v[6]) * scale, __uint_as_float(v[7]) * scale));
        }
        __syncwarp();
        const int cc = lane & 7, x = u * BN + colbase + cc * 8;
        if (x < args.N) {  // N % 16 == 0: a chunk is inside or outside
#pragma unroll
          for (int it = 0; it < 8; ++it) {
            const int rr = 4 * it + (lane >> 3);
            if (rr < args.M && in_bounds(args.status, x + 8 <= args.N))
              *reinterpret_cast<uint4*>(args.out + static_cast<int64_t>(rr) * args.ldo + x) =
                  ld_shared_v4(buf + rr * 128 + ((cc ^ (rr & 7)) << 4));
          }
        }
        __syncwarp();  // the next tile overwrites the box
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// ------------------------------------------------------------------- host ---

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// Row-major [rows, K/2] byte matrix, box of 128 bytes x box_rows rows, 128-B swizzle.
bool make_code_map(CUtensorMap* map, const uint8_t* base, int64_t rows, int64_t K, uint32_t box_rows) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(K / 2), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(K / 2)};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(BK / 2), box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// MMA-layout block scales of a [rows, K] operand viewed as [bytes / 256, 256]
// bytes; a box of 8 rows is one (128-row tile, k-block) group of four atoms.
// pair: [row tiles, K / 32, 256] bytes and boxes of two row tiles.
bool make_scale_map(CUtensorMap* map, const uint8_t* base, int64_t rows, int64_t K, bool pair) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  const cuuint64_t tile_rows = static_cast<cuuint64_t>(K / 32), tiles = static_cast<cuuint64_t>((rows + 127) / 128);
  cuuint64_t dims[3] = {256, pair ? tile_rows : tile_rows * tiles, tiles};
  cuuint64_t strides[2] = {256, 256 * tile_rows};
  cuuint32_t box[3] = {256, 8, 2};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, pair ? 3 : 2, const_cast<uint8_t*>(base), dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// bf16 [M, N] output with row pitch ldo, stored in 32 x 64 boxes, 128-B swizzle.
bool make_out_map(CUtensorMap* map, void* base, int64_t M, int64_t N, int64_t ldo) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(M)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(ldo * 2)};
  cuuint32_t box[2] = {kEpiCols, kEpiRows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Per-device, per-configuration launch set-up: the shared-memory opt-in and
// the number of clusters resident on the GPU at once (persistent grid).
template <class C>
int resident_ctas() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(d);
  if (it != cache.end()) return it->second;
  if (cudaFuncSetAttribute(nvfp4_gemm_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(C::kSmemBytes)) != cudaSuccess)
    return 0;
  const int n = sm_count();  // one CTA per SM (launch bounds and shared memory allow no more)
  cache[d] = n;
  return n;
}

template <class C>
nvfp4_status launch(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a, const uint8_t* w_codes,
                    const uint8_t* w_scales, const float* g_w, int64_t M, int64_t N, int64_t K, void* out_bf16,
                    int64_t ldo, cudaStream_t stream, uint32_t idesc_fmt) {
  const int64_t tiles_m = (M + BM - 1) / BM, tiles_n = (N + C::BN - 1) / C::BN;
  const int64_t units = tiles_m * tiles_n;
  if (units >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  CUtensorMap ma, mb, mo;
  if (!make_code_map(&ma, a_codes, M, K, BM) || !make_code_map(&mb, w_codes, N, K, C::BN) ||
      !make_out_map(&mo, out_bf16, M, N, ldo))
    return NVFP4_ERR_CUDA;
  const int ctas_max = resident_ctas<C>();
  if (ctas_max <= 0) return NVFP4_ERR_CUDA;
  GemmArgs args = {};
  args.idesc_fmt = idesc_fmt;
  args.sfa = a_scales;
  args.sfb = w_scales;
  args.ga = g_a;
  args.gb = g_w;
  args.M = static_cast<int>(M);
  args.N = static_cast<int>(N);
  args.K = static_cast<int>(K);
  args.tiles_m = static_cast<int>(tiles_m);
  args.tiles_n = static_cast<int>(tiles_n);
  args.group_m = raster_group(K, units / tiles_n);
  args.status = status_word_dev();
  args.fault_skip_stage = take_fault(NVFP4_FAULT_GEMM_SKIP_STAGE) ? 1 : 0;
  const int ctas = static_cast<int>(units < ctas_max ? units : ctas_max);
  if (launch_pdl(nvfp4_gemm_kernel<C>, dim3(ctas), dim3(C::kThreads), C::kSmemBytes, stream, ma, mb, mo, args) !=
      cudaSuccess)
    return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}

template <class C, bool kSwiGLU>
int resident_pairs() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(d);
  if (it != cache.end()) return it->second;
  if (cudaFuncSetAttribute(nvfp4_gemm_pair_kernel<C, kSwiGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(C::kSmemBytes)) != cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2 * (sm_count() / 2), 1, 1);
  cfg.blockDim = dim3(C::kThreads, 1, 1);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, nvfp4_gemm_pair_kernel<C, kSwiGLU>, &cfg) != cudaSuccess ||
      clusters <= 0) {
    cudaGetLastError();
    return 0;
  }
  cache[d] = clusters;
  return clusters;
}

// kSwiGLU: out_bf16 is unused; the fused outputs go through
// args.q_codes / q_scales / g_out, which the caller fills in `extra`.
template <class C, bool kSwiGLU = false>
nvfp4_status launch_pair(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a, const uint8_t* w_codes,
                         const uint8_t* w_scales, const float* g_w, int64_t M, int64_t N, int64_t K, void* out_bf16,
                         int64_t ldo, cudaStream_t stream, const GemmArgs* extra = nullptr,
                         uint32_t idesc_fmt = 0) {
  const int64_t tiles_m = (M + BM - 1) / BM, tiles_n = (N + C::BN - 1) / C::BN;  // a column tail reads zeros
  const int64_t units = ((tiles_m + 1) / 2) * tiles_n;
  if (units >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  CUtensorMap ma, mb, mb_half, msa, msb;
  if (!make_code_map(&ma, a_codes, M, K, BM) || !make_code_map(&mb, w_codes, N, K, 128) ||
      !make_code_map(&mb_half, w_codes, N, K, 64) ||
      !make_scale_map(&msa, a_scales, M, K, false) || !make_scale_map(&msb, w_scales, N, K, true))
    return NVFP4_ERR_CUDA;
  const int pairs_max = resident_pairs<C, kSwiGLU>();
  if (pairs_max <= 0) return NVFP4_ERR_CUDA;
  GemmArgs args = {};
  if (extra) args = *extra;
  args.idesc_fmt = idesc_fmt;
  args.sfa = a_scales;
  args.sfb = w_scales;
  args.ga = g_a;
  args.gb = g_w;
  args.M = static_cast<int>(M);
  args.N = static_cast<int>(N);
  args.K = static_cast<int>(K);
  args.tiles_m = static_cast<int>(tiles_m);
  args.tiles_n = static_cast<int>(tiles_n);
  args.group_m = raster_group(K, units / tiles_n);
  args.status = status_word_dev();
  args.fault_skip_stage = take_fault(NVFP4_FAULT_GEMM_SKIP_STAGE) ? 1 : 0;
  args.out = static_cast<uint16_t*>(out_bf16);
  args.ldo = ldo;
  // Tiles of a last wave that fills at most half of the pairs are split in
  // two: a half takes about two thirds of a tile's time (GB300, 76 pairs: 1000
  // x 5120 x 13824, 80 tiles, 38.5 -> 34.0 us; 256 x 27648 x 5120, 108 tiles,
  // 22.9 -> 21.3; 8192 x 5120 x 27648, 640 tiles, 316.9 -> 312.1).
  const int64_t last = units % pairs_max;
  const bool split = last > 0 && 2 * last <= pairs_max;
  args.full_units = static_cast<int>(split ? units - last : units);
  const int64_t total = 2 * units - args.full_units;
  const int pairs = static_cast<int>(total < pairs_max ? total : pairs_max);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2 * pairs, 1, 1);
  cfg.blockDim = dim3(C::kThreads, 1, 1);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, nvfp4_gemm_pair_kernel<C, kSwiGLU>, ma, mb, mb_half, msa, msb, args) != cudaSuccess)
    return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}

using SplitCfg = PairCfg<NVFP4_GEMM_PAIR_STAGES>;

// Clusters of `size` CTAs of the split-K kernel that are resident on the GPU
// at once (0 if that cluster shape cannot be launched).
int resident_split_clusters(int size) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, int> cache;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find({d, size});
  if (it != cache.end()) return it->second;
  int clusters = 0;
  if (cudaFuncSetAttribute(nvfp4_gemm_splitk_kernel<SplitCfg>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(SplitCfg::kSmemBytes)) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(size * (sm_count() / size), 1, 1);
    cfg.blockDim = dim3(SplitCfg::kThreads, 1, 1);
    cfg.dynamicSmemBytes = SplitCfg::kSmemBytes;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&clusters, nvfp4_gemm_splitk_kernel<SplitCfg>, &cfg) != cudaSuccess)
      clusters = 0;
  }
  cudaGetLastError();
  cache[{d, size}] = clusters;
  return clusters;
}

// Pairs per tile for the split-K kernel: among S = 2..4 with every tile's
// cluster of 2S CTAs resident at once, the one with the fewest k-blocks per
// pair (ties: the smaller S, less to reduce); 0 if none.  On GB300 clusters
// of 4, 6 and 8 CTAs of this kernel fit about 36, 24 and 16 at a time, so the
// 14B decode qkv (28 tiles) takes S = 2 and the o and down GEMMs (20 tiles)
// S = 3.  The cross-CTA reduction costs ~3-4 us, which only pays with a long
// K: measured back to back on GB300, 256 x 7168 x 5120 11.9 -> 11.1 us,
// 256 x 5120 x 5120 11.8 -> 10.7 us, 256 x 5120 x 13824 24.8 -> 15.2 us, but
// 16 x 1536 x 1536 (6 k-blocks) 5.7 -> 7.2 us; so K needs 16 k-blocks.
constexpr int64_t kSplitMinKblocks = 16;
int choose_splits(int64_t tiles, int64_t kblocks) {
  if (kblocks < kSplitMinKblocks) return 0;
  int best = 0;
  int64_t best_kb = kblocks;
  for (int S = 2; S <= 4; ++S) {
    if (kblocks < S || tiles > resident_split_clusters(2 * S)) continue;
    const int64_t kb = (kblocks + S - 1) / S;
    if (kb < best_kb) { best = S; best_kb = kb; }
  }
  return best;
}

nvfp4_status launch_splitk(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a, const uint8_t* w_codes,
                           const uint8_t* w_scales, const float* g_w, int64_t M, int64_t N, int64_t K, void* out_bf16,
                           int64_t ldo, cudaStream_t stream, uint32_t idesc_fmt, int splits) {
  using C = SplitCfg;
  const int64_t tiles_m = (M + BM - 1) / BM, tiles_n = N / C::BN;
  const int64_t tiles = ((tiles_m + 1) / 2) * tiles_n;
  if (tiles * 2 * splits >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  CUtensorMap ma, mb, msa, msb, mo;
  if (!make_code_map(&ma, a_codes, M, K, BM) || !make_code_map(&mb, w_codes, N, K, 128) ||
      !make_scale_map(&msa, a_scales, M, K, false) || !make_scale_map(&msb, w_scales, N, K, true) ||
      !make_out_map(&mo, out_bf16, M, N, ldo))
    return NVFP4_ERR_CUDA;
  GemmArgs args = {};
  args.idesc_fmt = idesc_fmt;
  args.sfa = a_scales;
  args.sfb = w_scales;
  args.ga = g_a;
  args.gb = g_w;
  args.M = static_cast<int>(M);
  args.N = static_cast<int>(N);
  args.K = static_cast<int>(K);
  args.tiles_m = static_cast<int>(tiles_m);
  args.tiles_n = static_cast<int>(tiles_n);
  args.group_m = raster_group(K, tiles / tiles_n);
  args.splits = splits;
  args.status = status_word_dev();
  args.fault_skip_stage = take_fault(NVFP4_FAULT_GEMM_SKIP_STAGE) ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2 * splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(tiles * 2 * splits), 1, 1);
  cfg.blockDim = dim3(C::kThreads, 1, 1);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, nvfp4_gemm_splitk_kernel<C>, ma, mb, msa, msb, mo, args) != cudaSuccess)
    return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}

// Clusters of `size` CTAs of the skinny kernel resident on the GPU at once
// (0 if that cluster shape cannot be launched).  The occupancy query counts
// one CTA of a kernel that allocates TMEM per SM; two of these share one (256
// of 512 columns each, and their shared memory fits).  Timing agrees: the
// step from one wave to two lies at twice the query's figures (92 clusters of
// 3, 72 of 4, 56 of 5, 46 of 6).
template <class C, bool kSwiGLU = false>
int resident_skinny_clusters(int size) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, int> cache;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find({d, size});
  if (it != cache.end()) return it->second;
  int clusters = 0;
  if (cudaFuncSetAttribute(nvfp4_gemm_skinny_kernel<C, kSwiGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(C::kSmemBytes)) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(size * (2 * sm_count() / size), 1, 1);
    cfg.blockDim = dim3(C::kThreads, 1, 1);
    cfg.dynamicSmemBytes = C::kSmemBytes;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, nvfp4_gemm_skinny_kernel<C, kSwiGLU>, &cfg) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, nvfp4_gemm_skinny_kernel<C, kSwiGLU>, C::kThreads,
                                                      C::kSmemBytes) != cudaSuccess)
      clusters = 0;
    else if (per_sm == 1)
      clusters *= 2;
  }
  cudaGetLastError();
  cache[{d, size}] = clusters;
  return clusters;
}

// CTAs per tile of the skinny kernel, or 0 where another kernel is faster.
// The largest S <= 8 whose clusters are all resident at once: a second wave
// costs more than a longer k-loop, and within one wave more CTAs stream
// faster (1 row, 5120 x 13824, S = 1, 2, 4, 6, 7: 28.3, 18.5, 14.8, 13.4, 19.1
// us with the activation's quantization; 27648 x 5120, S = 1, 2, 4: 18.5,
// 22.7, 25.8, before the scales had a producer of their own).  More rows make the reduction dearer: above 32 rows S stays
// at 4 unless each CTA keeps 4-5 k-blocks (128 rows, 1536 x 5120, S = 4, 8:
// 12.2, 14.0; 1536 x 13824: 17.2, 14.9).
// K <= 1536 is never split: nvfp4_linear_dynamic's sums are in one order.
// Against the kernels for other shapes: unsplit with a short K and at most one
// 128 x 128 tile per SM the single-CTA kernel is as fast (1536 x 2048: 8.3
// against 8.2 us); with 65-128 rows A is half of what an SM takes in, and the
// skinny kernel is ahead only when it splits by three or more (7168 x 5120:
// 14.8 against 15.8 us; 14336 x 5120 by two: 17.9 against 17.0) or when the
// last wave of single CTAs would be mostly empty (27648 x 5120, 216 tiles on
// 152 SMs: 24.6 against 26.7; 55296 x 5120, 432 tiles: 45.8 against 38.3).
template <class C>
int choose_skinny_splits(int64_t tiles, int64_t kblocks) {
  const int64_t sms = sm_count();
  if (sms <= 0 || (C::kRows == 128 && kblocks <= 8)) return 0;
  int best = 1;
  if (kblocks > DynCfg::kMaxKb) {
    const int64_t cap = C::kRows == 32 ? 8 : (C::kRows == 64 ? kblocks / 4 : kblocks / 5);
    for (int s = 2; s <= 8 && s <= kblocks && s <= (cap < 4 ? 4 : cap); ++s)
      if (tiles <= resident_skinny_clusters<C>(s)) best = s;
  } else if (tiles <= sms) {
    return 0;
  }
  if (C::kRows == 128 && (best == 2 || (best == 1 && 4 * ((tiles + sms - 1) / sms) * sms <= 5 * tiles))) return 0;
  return best;
}

// kSwiGLU: out_bf16 is unused; the fused outputs go through *extra.
template <class C, bool kSwiGLU = false>
nvfp4_status launch_skinny(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a, const uint8_t* w_codes,
                           const uint8_t* w_scales, const float* g_w, int64_t M, int64_t N, int64_t K, void* out_bf16,
                           int64_t ldo, cudaStream_t stream, uint32_t idesc_fmt, int splits,
                           const GemmArgs* extra = nullptr) {
  const int64_t tiles_n = (N + 127) / 128;
  if (resident_skinny_clusters<C, kSwiGLU>(splits) <= 0) return NVFP4_ERR_CUDA;  // also the shared-memory opt-in
  if (tiles_n * splits >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  GemmArgs args = kSwiGLU ? *extra : GemmArgs{};
  args.a_box_rows = static_cast<int>((M + 7) & ~7ll);
  CUtensorMap ma, mb;
  if (!make_code_map(&ma, a_codes, M, K, args.a_box_rows) || !make_code_map(&mb, w_codes, N, K, 128))
    return NVFP4_ERR_CUDA;
  args.idesc_fmt = idesc_fmt;
  args.sfa = a_scales;
  args.sfb = w_scales;
  args.ga = g_a;
  args.gb = g_w;
  args.M = static_cast<int>(M);
  args.N = static_cast<int>(N);
  args.K = static_cast<int>(K);
  args.splits = splits;
  args.status = status_word_dev();
  args.fault_skip_stage = take_fault(NVFP4_FAULT_GEMM_SKIP_STAGE) ? 1 : 0;
  args.out = static_cast<uint16_t*>(out_bf16);
  args.ldo = ldo;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(tiles_n * splits), 1, 1);
  cfg.blockDim = dim3(C::kThreads, 1, 1);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, nvfp4_gemm_skinny_kernel<C, kSwiGLU>, ma, mb, args) != cudaSuccess) return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}

// nvfp4_linear_dynamic: one persistent CTA per 128-column tile of W, at most
// one per SM.
nvfp4_status launch_dynamic(const uint16_t* x, int64_t M, int64_t K, int64_t ldx, const uint8_t* w_codes,
                            const uint8_t* w_scales, const float* g_w, int64_t N, void* out_bf16, int64_t ldo,
                            float* g_out, cudaStream_t stream) {
  using C = DynCfg;
  static std::mutex mu;
  static std::map<int, bool> ready;
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return NVFP4_ERR_CUDA;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!ready[d]) {
      if (cudaFuncSetAttribute(nvfp4_linear_dyn_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(C::kSmemBytes)) != cudaSuccess)
        return NVFP4_ERR_CUDA;
      ready[d] = true;
    }
  }
  const int64_t tiles_n = (N + C::BN - 1) / C::BN;
  CUtensorMap mb;
  if (!make_code_map(&mb, w_codes, N, K, C::BN)) return NVFP4_ERR_CUDA;
  DynArgs args = {};
  args.x = x;
  args.ldx = ldx;
  args.sfb = w_scales;
  args.gb = g_w;
  args.g_out = g_out;
  args.out = static_cast<uint16_t*>(out_bf16);
  args.ldo = ldo;
  args.kb16 = FastDiv(static_cast<uint32_t>(K / 16));
  args.M = static_cast<int>(M);
  args.N = static_cast<int>(N);
  args.K = static_cast<int>(K);
  args.tiles_n = static_cast<int>(tiles_n);
  args.status = status_word_dev();
  args.fault_skip_stage = take_fault(NVFP4_FAULT_GEMM_SKIP_STAGE) ? 1 : 0;
  const int sms = sm_count();
  if (sms <= 0) return NVFP4_ERR_CUDA;
  const int ctas = static_cast<int>(tiles_n < sms ? tiles_n : sms);
  if (launch_pdl(nvfp4_linear_dyn_kernel<C>, dim3(ctas), dim3(C::kThreads), C::kSmemBytes, stream, mb, args) !=
      cudaSuccess)
    return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}

#ifndef NVFP4_GEMM_BN
#define NVFP4_GEMM_BN 0  // 0: choose per shape
#endif
#ifndef NVFP4_GEMM_SPLITK
#define NVFP4_GEMM_SPLITK 1  // 0: never use the split-K kernel
#endif
#ifndef NVFP4_GEMM_PAIR
#define NVFP4_GEMM_PAIR 1  // 0: never use the CTA-pair kernel
#endif
}  // namespace
}  // namespace nvfp4

using namespace nvfp4;

namespace nvfp4 {
namespace {
// Kernel choice for one block-scaled linear (arguments already validated).
nvfp4_status linear_dispatch(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a,
                             const uint8_t* w_codes, const uint8_t* w_scales, const float* g_w, int64_t M, int64_t N,
                             int64_t K, void* out_bf16, int64_t ldo, cudaStream_t s, uint32_t idesc_fmt) {
  const int64_t tiles_m = (M + BM - 1) / BM;
  if (tiles_m == 1) {
    const int64_t tiles = (N + 127) / 128, kblocks = K / BK;
    const int splits = M <= 32   ? choose_skinny_splits<SkinnyCfg<32>>(tiles, kblocks)
                       : M <= 64 ? choose_skinny_splits<SkinnyCfg<64>>(tiles, kblocks)
                                 : choose_skinny_splits<SkinnyCfg<128>>(tiles, kblocks);
    const auto kernel = M <= 32   ? launch_skinny<SkinnyCfg<32>>
                        : M <= 64 ? launch_skinny<SkinnyCfg<64>>
                                  : launch_skinny<SkinnyCfg<128>>;
    if (splits)
      return kernel(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K, out_bf16, ldo, s, idesc_fmt, splits,
                    nullptr);
  }
  // The CTA pair, unless its 256 x 256 tiles would leave most pairs idle
  // (decode-sized M): then, with a long K, the split-K clusters, else 128 x
  // 128 tiles on single CTAs, which spread the W stream over more SMs than
  // the pairs would (measured faster at M = 256 with N = 5120 or 7168, slower
  // with N = 27648).
  using Pair = PairCfg<NVFP4_GEMM_PAIR_STAGES>;
  // A column tail (N % 256 != 0) costs the pairs at most one tile column of
  // zeros, and single CTAs still take twice as long: 8192 x 7296 x 5120 191 ->
  // 92 us, 256 x 27520 x 5120 28.7 -> 21.3, 2048 x 2176 x 8192 28.8 -> 15.6.
  // Only with a short K and at most one 128 x 128 tile per SM are single CTAs
  // as fast or faster (K = 1536: 2048 x 1152 6.3 against 7.2 us, 1024 x 2304
  // 6.2 / 6.3; K = 2048: 256 x 9728 7.7 / 7.3).
  const bool single = K / BK <= 6 && tiles_m * ((N + 127) / 128) <= sm_count();
  if (NVFP4_GEMM_PAIR && tiles_m >= 2 && !single) {
    const int64_t pair_units = ((tiles_m + 1) / 2) * ((N + 255) / 256);
    if (2 * pair_units >= resident_pairs<Pair, false>())
      return launch_pair<Pair>(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K, out_bf16, ldo, s, nullptr,
                               idesc_fmt);
  }
  // Too few pair tiles for the GPU: split K across clusters of CTA pairs.
  if (NVFP4_GEMM_SPLITK && N % 256 == 0) {
    const int splits = choose_splits(((tiles_m + 1) / 2) * (N / 256), K / BK);
    if (splits)
      return launch_splitk(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K, out_bf16, ldo, s, idesc_fmt,
                           splits);
  }
  // Single CTAs: BN = 128 (measured faster than 256 at M <= 256 on GB300).
  const int bn = NVFP4_GEMM_BN ? NVFP4_GEMM_BN : 128;
  if (bn == 256)
    return launch<Cfg<256, 3>>(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K, out_bf16, ldo, s, idesc_fmt);
  return launch<Cfg<128, 5>>(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K, out_bf16, ldo, s, idesc_fmt);
}

// Whether the fused gate_up + SwiGLU runs in the skinny kernel, one CTA per 128
// W rows: two CTAs share an SM and only the A rows that exist are copied.  K is
// not split: the sums, and with them every output byte, are those of the
// pairs.  us, pairs -> skinny:
//   up to 32 rows: 1 row, 27648 x 5120 27.5 -> 17.2, 17920 x 1536 9.8 -> 7.5,
//     12288 x 8192 23.6 -> 15.4, 4096 x 2048 7.2 -> 6.3; 32 rows: 22.4 -> 17.2,
//     9.0 -> 7.3, 16.6 -> 15.4, 6.6 -> 6.2.  A few tiles with a long K leave
//     each SM one CTA, whose ring streams slower than the pairs' (2048 x 8192
//     12.3 against 11.8, 4096 x 13824, 32 rows, 18.8 against 17.1; 2048 x 4096
//     7.7 against 7.9): those stay with the pairs;
//   more rows, whose larger A slots leave three ring stages: ahead when all
//     tiles are resident at once and some SMs hold two (48 rows: 27648 x 5120
//     26.2 -> 18.2, 38912 x 1536 12.8 -> 9.9, 22528 x 8192 28.4 -> 23.6; 96 rows
//     20.6 -> 19.3, 11.7 -> 10.7, 28.4 -> 24.3), and up to 64 rows with fewer
//     tiles unless K is long (12288 x 5120 14.9 -> 12.7, 16384 x 1536 9.0 -> 7.9;
//     12288 x 8192 17.0 -> 17.1, 8192 x 4096, 64 rows, 9.6 -> 10.5); not with a
//     second wave (40960 x 5120, 64 rows, 28.8 -> 32.5).
bool swiglu_in_skinny(int64_t M, int64_t tiles, int64_t kblocks) {
  const int64_t sms = sm_count();
  if (M <= 32) return kblocks <= 16 || tiles > 32;
  if (M > 128 || tiles > 2 * sms) return false;
  return tiles > sms || (M <= 64 && kblocks <= 20 && 8 * tiles >= 5 * sms);
}

// Kernel choice for the fused gate_up + SwiGLU (arguments already validated).
nvfp4_status swiglu_dispatch(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a,
                             const uint8_t* w_codes, const uint8_t* w_scales, const float* g_w, int64_t M, int64_t N,
                             int64_t K, cudaStream_t s, const GemmArgs& extra, uint32_t idesc_fmt) {
  if (swiglu_in_skinny(M, N / 128, K / BK)) {
    const auto kernel = M <= 32   ? launch_skinny<SkinnyCfg<32>, true>
                        : M <= 64 ? launch_skinny<SkinnyCfg<64>, true>
                                  : launch_skinny<SkinnyCfg<128>, true>;
    return kernel(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K, nullptr, 0, s, idesc_fmt, 1, &extra);
  }
  return launch_pair<PairCfg<NVFP4_GEMM_PAIR_STAGES>, true>(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K,
                                                           nullptr, 0, s, &extra, idesc_fmt);
}

}  // namespace
}  // namespace nvfp4

NVFP4_API nvfp4_status nvfp4_linear(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a,
                                    const uint8_t* w_codes, const uint8_t* w_scales, const float* g_w, int64_t M,
                                    int64_t N, int64_t K, void* out_bf16, int64_t ldo, void* stream) {
  NVFP4_TRACE("nvfp4_linear");
  if (!a_codes || !a_scales || !g_a || !w_codes || !w_scales || !g_w || !out_bf16) return NVFP4_ERR_INVALID_ARG;
  if (M <= 0 || N <= 0 || K <= 0 || K % BK || N % 16 || ldo < N || ldo % 8) return NVFP4_ERR_SHAPE;
  if (M >= (1ll << 31) || N >= (1ll << 31) || K >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  if (!aligned(a_codes, 16) || !aligned(w_codes, 16) || !aligned(a_scales, 16) || !aligned(w_scales, 16) ||
      !aligned(out_bf16, 16) || !aligned(g_a, 4) || !aligned(g_w, 4))
    return NVFP4_ERR_ALIGN;
  return linear_dispatch(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, N, K, out_bf16, ldo,
                         static_cast<cudaStream_t>(stream), 0);
}

NVFP4_API nvfp4_status nvfp4_linear_dynamic(const void* x_bf16, int64_t M, int64_t K, int64_t ld_x,
                                            const uint8_t* w_codes, const uint8_t* w_scales, const float* g_w,
                                            int64_t N, void* out_bf16, int64_t ldo, float* g_a_out, void* stream) {
  NVFP4_TRACE("nvfp4_linear_dynamic");
  if (!x_bf16 || !w_codes || !w_scales || !g_w || !out_bf16) return NVFP4_ERR_INVALID_ARG;
  if (M <= 0 || N <= 0 || K <= 0 || K % BK || N % 16 || ldo < N || ldo % 8 || ld_x < K) return NVFP4_ERR_SHAPE;
  if (M > DynCfg::kMaxRows || K > static_cast<int64_t>(DynCfg::kMaxKb) * BK) return NVFP4_ERR_UNSUPPORTED;
  if (N >= (1ll << 31) || ld_x >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  if (!aligned(x_bf16, 16) || ld_x % 8 || !aligned(w_codes, 16) || !aligned(w_scales, 16) || !aligned(out_bf16, 16) ||
      !aligned(g_w, 4) || !aligned(g_a_out, 4))
    return NVFP4_ERR_ALIGN;
  return launch_dynamic(static_cast<const uint16_t*>(x_bf16), M, K, ld_x, w_codes, w_scales, g_w, N, out_bf16, ldo,
                        g_a_out, static_cast<cudaStream_t>(stream));
}

NVFP4_API nvfp4_status mxfp4_linear(const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* w_codes,
                                    const uint8_t* w_scales, int64_t M, int64_t N, int64_t K, void* out_bf16,
                                    int64_t ldo, void* stream) {
  NVFP4_TRACE("mxfp4_linear");
  if (!a_codes || !a_scales || !w_codes || !w_scales || !out_bf16) return NVFP4_ERR_INVALID_ARG;
  if (M <= 0 || N <= 0 || K <= 0 || K % BK || N % 16 || ldo < N || ldo % 8) return NVFP4_ERR_SHAPE;
  if (M >= (1ll << 31) || N >= (1ll << 31) || K >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  if (!aligned(a_codes, 16) || !aligned(w_codes, 16) || !aligned(a_scales, 16) || !aligned(w_scales, 16) ||
      !aligned(out_bf16, 16))
    return NVFP4_ERR_ALIGN;
  return linear_dispatch(a_codes, a_scales, nullptr, w_codes, w_scales, nullptr, M, N, K, out_bf16, ldo,
                         static_cast<cudaStream_t>(stream), kScaleE8M0);
}

NVFP4_API nvfp4_status nvfp4_linear_swiglu_quantize(const uint8_t* a_codes, const uint8_t* a_scales, const float* g_a,
                                                    const uint8_t* w_codes, const uint8_t* w_scales, const float* g_w,
                                                    int64_t M, int64_t I, int64_t K, const float* g_out,
                                                    uint8_t* out_codes, uint8_t* out_scales, void* stream) {
  NVFP4_TRACE("nvfp4_linear_swiglu_quantize");
  if (!a_codes || !a_scales || !g_a || !w_codes || !w_scales || !g_w || !g_out || !out_codes || !out_scales)
    return NVFP4_ERR_INVALID_ARG;
  if (M <= 0 || I <= 0 || K <= 0 || K % BK || I % 128) return NVFP4_ERR_SHAPE;
  if (M >= (1ll << 31) || 2 * I >= (1ll << 31) || K >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  if (!aligned(a_codes, 16) || !aligned(w_codes, 16) || !aligned(a_scales, 16) || !aligned(w_scales, 16) ||
      !aligned(out_codes, 16) || !aligned(out_scales, 4) || !aligned(g_a, 4) || !aligned(g_w, 4) || !aligned(g_out, 4))
    return NVFP4_ERR_ALIGN;
  GemmArgs extra = {};
  extra.q_codes = out_codes;
  extra.q_scales = out_scales;
  extra.g_out = g_out;
  return swiglu_dispatch(a_codes, a_scales, g_a, w_codes, w_scales, g_w, M, 2 * I, K,
                         static_cast<cudaStream_t>(stream), extra, 0);
}

NVFP4_API nvfp4_status mxfp4_linear_swiglu_quantize(const uint8_t* a_codes, const uint8_t* a_scales,
                                                    const uint8_t* w_codes, const uint8_t* w_scales, int64_t M,
                                                    int64_t I, int64_t K, int rotate, uint8_t* out_codes,
                                                    uint8_t* out_scales, void* stream) {
  NVFP4_TRACE("mxfp4_linear_swiglu_quantize");
  if (!a_codes || !a_scales || !w_codes || !w_scales || !out_codes || !out_scales) return NVFP4_ERR_INVALID_ARG;
  if (rotate != 0 && rotate != 1) return NVFP4_ERR_INVALID_ARG;
  if (M <= 0 || I <= 0 || K <= 0 || K % BK || I % 128) return NVFP4_ERR_SHAPE;
  if (M >= (1ll << 31) || 2 * I >= (1ll << 31) || K >= (1ll << 31)) return NVFP4_ERR_SHAPE;
  if (!aligned(a_codes, 16) || !aligned(w_codes, 16) || !aligned(a_scales, 16) || !aligned(w_scales, 16) ||
      !aligned(out_codes, 16) || !aligned(out_scales, 4))
    return NVFP4_ERR_ALIGN;
  GemmArgs extra = {};
  extra.q_codes = out_codes;
  extra.q_scales = out_scales;
  extra.q_mode = rotate ? 2u : 1u;
  return swiglu_dispatch(a_codes, a_scales, nullptr, w_codes, w_scales, nullptr, M, 2 * I, K,
                         static_cast<cudaStream_t>(stream), extra, kScaleE8M0);
}

namespace nvfp4 {
namespace {
// out row 32j + t = gate row 16j + t, out row 32j + 16 + t = up row 16j + t
// (t < 16); one thread moves 16 bytes.
__global__ void interleave_gate_up_kernel(const uint4* __restrict__ gate, const uint4* __restrict__ up,
                                          uint4* __restrict__ out, uint64_t row_chunks, uint64_t n) {
  griddep_wait_and_release();
  for (uint64_t k = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; k < n;
       k += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
    const uint64_t orow = k / row_chunks, c = k - orow * row_chunks;
    const uint64_t j = orow >> 5, t = orow & 31u;
    const uint64_t irow = 16 * j + (t & 15u);
    out[k] = __ldg((t < 16 ? gate : up) + irow * row_chunks + c);
  }
}
}  // namespace
}  // namespace nvfp4

NVFP4_API nvfp4_status nvfp4_interleave_gate_up(const void* w_gate, const void* w_up, int64_t I, int64_t row_bytes,
                                                void* w_out, void* stream) {
  NVFP4_TRACE("nvfp4_interleave_gate_up");
  if (!w_gate || !w_up || !w_out) return NVFP4_ERR_INVALID_ARG;
  if (I <= 0 || I % 16 || row_bytes <= 0 || row_bytes % 16) return NVFP4_ERR_SHAPE;
  if (!aligned(w_gate, 16) || !aligned(w_up, 16) || !aligned(w_out, 16)) return NVFP4_ERR_ALIGN;
  const uint64_t row_chunks = static_cast<uint64_t>(row_bytes) / 16, n = 2 * static_cast<uint64_t>(I) * row_chunks;
  uint64_t grid = (n + 255) / 256;
  const uint64_t cap = static_cast<uint64_t>(sm_count()) * 8;
  if (grid > cap) grid = cap;
  if (launch_pdl(interleave_gate_up_kernel, dim3(static_cast<int>(grid)), dim3(256), 0,
                 static_cast<cudaStream_t>(stream), static_cast<const uint4*>(w_gate), static_cast<const uint4*>(w_up),
                 static_cast<uint4*>(w_out), row_chunks, n) != cudaSuccess)
    return NVFP4_ERR_CUDA;
  count_launches(1);
  return launch_status();
}

#ifdef NVFP4_TIMELINE
// Timeline build only (not part of the C ABI of include/nvfp4.h): copy the
// per-CTA stamps of the last 1-CTA GEMM launch ([1024][8] uint64, ns, zero
// where a CTA or event did not occur) to host memory, then clear them.
// Synchronizes the device.
extern "C" __attribute__((visibility("default"))) int nvfp4_timeline_gemm(unsigned long long* host) {
  if (cudaDeviceSynchronize() != cudaSuccess) return 1;
  if (cudaMemcpyFromSymbol(host, nvfp4::g_gemm_timeline, sizeof(nvfp4::g_gemm_timeline)) != cudaSuccess) return 1;
  static unsigned long long zero[nvfp4::kGemmTimelineCtas * 8];
  return cudaMemcpyToSymbol(nvfp4::g_gemm_timeline, zero, sizeof(zero)) == cudaSuccess ? 0 : 1;
}
#endif
