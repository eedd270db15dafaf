// Prefill projections on the 5th-generation tensor cores: a persistent,
// warp-specialised tcgen05 GEMM, out[m][n] = A[m] . W[n] (A = bf16
// activations [M][K], W = bf16 weights [N][K], fp32 accumulation in TMEM),
// followed by the fused epilogues of epilogue.cuh.
//
//   warp 0      : TMA producer -- one lane streams 128x64 A and up to 256x64 W
//                 tiles (128-byte swizzle) into a shared-memory ring,
//                 completion tracked by mbarrier transaction bytes;
//   warp 1      : MMA issuer -- allocates 512 TMEM columns (two 128x256 fp32
//                 accumulators), one lane issues tcgen05.mma kind::f16
//                 (M=128, N=256, K=16) and frees ring slots / publishes
//                 finished accumulators with tcgen05.commit;
//   warps 2..9  : epilogue -- two warps per 32 TMEM lanes (rows), half the
//                 columns each, 32 at a time with tcgen05.ld, and the fused
//                 epilogue, overlapping the next tile's main loop
//                 (double-buffered accumulators).
// Tiles are visited in groups of 8 M-blocks per N sweep so the A and W
// working sets of the concurrently running CTAs stay L2-resident.
// Eight epilogue warps: where a launch has one or two tiles per CTA the epilogue
// is exposed, and four warps kept too few reads in flight (8B width, 1024 rows,
// per CTA: O 19 -> 13 us, QKV 10 -> 3; 0.5B width, 512 rows: QKV 6.5-11 -> 2-4.5,
// gate/up 9.5 -> 4.6). Measured and not kept: launching the next kernel and
// requesting its first weights under the last epilogue (small widths 1-3% faster,
// 8B width 2-6% slower).
// Every mbarrier wait is bounded (DEVERR_TIMEOUT instead of a hang).
#include "kernels.h"

#include <cudaTypedefs.h>

namespace {

constexpr int BM = 128, BK = 64, GROUP_M = 8;
constexpr int A_BYTES = BM * BK * 2;  // 16 KB
constexpr int EPI_WARPS = 8;
constexpr int NUM_THREADS = 64 + 32 * EPI_WARPS;

// BN_: columns of the output tile that the ring holds (256: 256, 224 or 192 at
// run time; or 128; gemm_tile_n chooses). SPLIT: the A operand is the sum of two
// 16-bit terms (hi + lo) and every k-step issues two MMAs into the same
// accumulator. The ring takes as many stages as fit in 200 KB, at most 6
// (BN 256: 4, split 3; BN 128: 6, split 4).
//
// AROWS < 128 (gate/up and logits of at most AROWS activation rows, 16 or 64, whose
// weights are too wide for the few-token kernel): each stage
// holds [A (AROWS rows) | A_lo (AROWS rows, SPLIT) | B]; the MMA still reads
// 128 A rows from the tile, rows AROWS..127 falling in the same stage's
// following bytes (landed, so stable; their accumulator rows are never
// stored). Without the padding rows a stage is smaller, so more of them --
// more weight bytes in flight per SM -- fit (up to 12).
//
// RING: the ring's byte budget (the residual kind's epilogue staging takes 32 KB).
template <bool SPLIT, int BN_, int AROWS = 128, int RING = 200 * 1024>
struct GCfg {
  static constexpr int BN = BN_;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr uint32_t TMEM_COLS = 2 * BN;
  static constexpr int A_TERMS = SPLIT ? 2 : 1;
  static constexpr bool SMALL = AROWS < BM;
  static constexpr int A_TILE = AROWS * BK * 2;  // bytes of one A term in a stage
  static constexpr int STAGE_BYTES = A_TERMS * A_TILE + B_BYTES;
  static constexpr int MAX_STAGES = SMALL ? 12 : 6;
  static constexpr int STAGES = RING / STAGE_BYTES > MAX_STAGES ? MAX_STAGES : RING / STAGE_BYTES;
  static_assert(!SMALL || STAGE_BYTES - (A_TERMS - 1) * A_TILE >= A_BYTES, "the MMA's 128-row read stays in its stage");
  static constexpr int BAR_BYTES = 8 * (2 * STAGES + 4) + 16;
  static constexpr int SMEM = STAGES * STAGE_BYTES + BAR_BYTES + 1024;
};

template <int KIND, bool SPLIT, int BN, int AROWS>
using GCfgK = GCfg<SPLIT, BN, AROWS, (KIND == EPI_RESID ? 192 : 200) * 1024>;

// Residual epilogue staging: each epilogue warp's 32 rows x 32 accumulator
// columns; 16-byte chunk j of row r lies at chunk j ^ (r & 7), so that both the
// row-wise stores and the 4-row loads hit distinct banks.
template <int KIND>
constexpr int epi_smem() { return KIND == EPI_RESID ? EPI_WARPS * 32 * 32 * 4 : 0; }

AXON_DEV void tile_coords(int t, int num_m, int num_n, int& mb, int& nb) {
  const int per_group = GROUP_M * num_n;
  const int g = t / per_group;
  const int first_m = g * GROUP_M;
  const int gm = min(GROUP_M, num_m - first_m);
  const int local = t - g * per_group;
  nb = local / gm;
  mb = first_m + (local - nb * gm);
}

template <int KIND, typename T16, bool SPLIT, int BN_, int AROWS>
__global__ void __launch_bounds__(NUM_THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmAlo, int M, int N, int K, int width, EpiArgs ep, GemmGroup grp) {
  using C = GCfgK<KIND, SPLIT, BN_, AROWS>;
  constexpr bool SMALL = C::SMALL;
  constexpr int BN = C::BN;
  constexpr int B_BYTES = C::B_BYTES;
  constexpr bool ANY_WIDTH = BN == 256 && !SMALL;
  const int bn = ANY_WIDTH ? width : BN;  // columns of this launch's tiles
  constexpr uint32_t TMEM_COLS = C::TMEM_COLS;
  constexpr int STAGES = C::STAGES;
  constexpr int STAGE_BYTES = C::STAGE_BYTES;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  // ring: [STAGES] A tiles, [STAGES] A_lo tiles (SPLIT), [STAGES] B tiles;
  // AROWS < 128: per stage [A | A_lo | B]
  const uint32_t sA = base, sAlo = base + STAGES * A_BYTES, sB = base + STAGES * A_BYTES * C::A_TERMS;
  auto a_at = [&](int s) { return SMALL ? base + s * STAGE_BYTES : sA + s * A_BYTES; };
  auto alo_at = [&](int s) { return SMALL ? base + s * STAGE_BYTES + C::A_TILE : sAlo + s * A_BYTES; };
  auto b_at = [&](int s) { return SMALL ? base + s * STAGE_BYTES + C::A_TERMS * C::A_TILE : sB + s * B_BYTES; };
  const uint32_t bars = base + STAGES * STAGE_BYTES;
  const uint32_t tmem_slot = bars + 8 * (2 * STAGES + 4);
  float* const epi_tile = reinterpret_cast<float*>(smem_raw + (bars + C::BAR_BYTES - raw));  // epi_smem<KIND>()
  const uint32_t* tmem_slot_ptr =
      reinterpret_cast<const uint32_t*>(smem_raw + (tmem_slot - raw));
  auto full_bar = [&](int s) { return bars + 8 * s; };
  auto empty_bar = [&](int s) { return bars + 8 * (STAGES + s); };
  auto accf_bar = [&](int i) { return bars + 8 * (2 * STAGES + i); };
  auto acce_bar = [&](int i) { return bars + 8 * (2 * STAGES + 2 + i); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(accf_bar(i), 1);
      mbar_init(acce_bar(i), 32 * EPI_WARPS);
    }
    fence_mbar_init();
    fence_proxy_async();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    if (SPLIT) tma_prefetch_desc(&tmAlo);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;

  grid_dep_wait();
  // grouped: the m-blocks the routing plan laid out (read after the wait,
  // when the plan kernel's writes are visible)
  const bool grouped = grp.mb_expert != nullptr;
  const int num_m = grouped ? __ldcg(grp.n_mblocks) : (M + BM - 1) / BM, num_n = (N + bn - 1) / bn;
  const int tiles = num_m * num_n, KB = K / BK;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        int mb, nb;
        tile_coords(t, num_m, num_n, mb, nb);
        if (grouped) {
          mb = t / num_n;
          nb = t - mb * num_n;
        }
        const int wrow = grouped ? __ldcg(grp.mb_expert + mb) * N + nb * bn : nb * bn;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1;
          if (!mbar_wait(empty_bar(s), ph ^ 1, ep.err)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(full_bar(s), STAGE_BYTES - (BN - bn) * (BK * 2));
          tma_load_2d(a_at(s), &tmA, full_bar(s), kb * BK, mb * BM);
          if (SPLIT) tma_load_2d(alo_at(s), &tmAlo, full_bar(s), kb * BK, mb * BM);
          tma_load_2d(b_at(s), &tmB, full_bar(s), kb * BK, wrow);
        }
      }
      // every copy lands before the CTA's shared memory goes away (all were consumed
      // unless a wait ran out)
      for (int j = it > STAGES ? it - STAGES : 0; j < it; ++j) mbar_wait(full_bar(j % STAGES), (j / STAGES) & 1, ep.err);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_f32acc(BM, bn, MmaFmt<T16>::v);
      int it = 0, lt = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++lt) {
        const int buf = lt & 1;
        const uint32_t aph = (lt >> 1) & 1;
        if (!mbar_wait(acce_bar(buf), aph ^ 1, ep.err)) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * BN;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1;
          if (!mbar_wait(full_bar(s), ph, ep.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = smem_desc_sw128(a_at(s));
          const uint64_t bd = smem_desc_sw128(b_at(s));
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)  // +32 bytes along K inside the swizzle atom
            tc_mma_f16(d, ad + 2 * k, bd + 2 * k, idesc, (kb != 0 || k != 0) ? 1u : 0u);
          if (SPLIT) {
            const uint64_t ald = smem_desc_sw128(alo_at(s));
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) tc_mma_f16(d, ald + 2 * k, bd + 2 * k, idesc, 1u);
          }
          tc_commit(empty_bar(s));
        }
        if (ok) tc_commit(accf_bar(buf));
      }
    }
    __syncwarp();
  } else {
    // two warps per TMEM lane quarter (the one that a warp may read), half the
    // tile's columns each
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    // whole groups of 32 columns: the first half takes the odd one
    const int mid = (bn / 32 + 1) / 2 * 32;
    const int cb = half ? mid : 0, ce = half ? bn : mid;
    const int row = q4 * 32 + lane;
    int lt = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++lt) {
      int mb, nb;
      tile_coords(t, num_m, num_n, mb, nb);
      if (grouped) {
        mb = t / num_n;
        nb = t - mb * num_n;
      }
      const int buf = lt & 1;
      const uint32_t aph = (lt >> 1) & 1;
      const int m = mb * BM + row;
      const bool mval = m < M && (!grp.row_valid || grp.row_valid[m] >= 0);
      float rinv = 1.f;  // read while the tile's products run
      if (KIND != EPI_RESID && KIND != EPI_ROWSCALE && mval) rinv = row_rinv(ep, m);
      int seq = 0, pos = 0;
      if (KIND == EPI_QKV && mval) pos = row_seq_pos(ep, m, seq);
      const bool got = __all_sync(0xffffffffu, mbar_wait(accf_bar(buf), aph, ep.err));
      if (!got) break;
      tc_fence_after();
      unsigned long long best = 0ull;
      const uint32_t taddr = tmem + (static_cast<uint32_t>(q4 * 32) << 16) + buf * BN;
      if (KIND == EPI_RESID) {
        // Through shared memory, 32 columns at a time: the warp stages its 32
        // rows x 32 accumulator columns, then every global access (residual
        // read, x, a and a_lo writes) covers 4 rows x 128 bytes per
        // instruction, lane (r, c) taking row 4i + r, columns 4c .. 4c+3.
        float* tw = epi_tile + (warp - 2) * 32 * 32;
        const int lr = lane >> 3, lc = (lane & 7) * 4;
        const int mrow = mb * BM + q4 * 32 + lr;  // + 4i: the lane's rows
        bool rv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int mm = mrow + 4 * i;
          rv[i] = mm < M && (!grp.row_valid || grp.row_valid[mm] >= 0);
        }
        // residual slices of group c0 (8 rows x 4 columns per lane), loaded
        // one group ahead so that their round trip overlaps the previous
        // group's stores
        auto load_x = [&](int c0, float4 (&xr)[8]) {
          const int n = nb * bn + c0 + lc;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            xr[i] = (rv[i] && n < N) ? __ldcg(reinterpret_cast<const float4*>(
                                           ep.x + static_cast<long long>(mrow + 4 * i) * ep.N + n))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float rs[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) rs[i] = 0.f;
        float4 xcur[8], xnext[8];
        load_x(cb, xcur);
#pragma unroll 1
        for (int c0 = cb; c0 < ce; c0 += 32) {
          if (c0 + 32 < ce) load_x(c0 + 32, xnext);
          uint32_t v[2][16];
          tmem_ld16(taddr + c0, v[0]);
          tmem_ld16(taddr + c0 + 16, v[1]);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j)
            *reinterpret_cast<float4*>(tw + lane * 32 + 4 * (j ^ (lane & 7))) =
                make_float4(__uint_as_float(v[j >> 2][(j & 3) * 4]), __uint_as_float(v[j >> 2][(j & 3) * 4 + 1]),
                            __uint_as_float(v[j >> 2][(j & 3) * 4 + 2]), __uint_as_float(v[j >> 2][(j & 3) * 4 + 3]));
          __syncwarp();
          const int n = nb * bn + c0 + lc;
          const float4 g4 = n < N ? *reinterpret_cast<const float4*>(ep.gain + n) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int rl = 4 * i + lr;
            float part = 0.f;
            if (rv[i] && n < N) {
              const float4 acc = *reinterpret_cast<const float4*>(tw + rl * 32 + (lc ^ (4 * (rl & 7))));
              const float4 xo = xcur[i];
              const float xn[4] = {xo.x + acc.x, xo.y + acc.y, xo.z + acc.z, xo.w + acc.w};
              const long long off = static_cast<long long>(mrow + 4 * i) * ep.N + n;
              *reinterpret_cast<float4*>(ep.x + off) = make_float4(xn[0], xn[1], xn[2], xn[3]);
              const float ag[4] = {xn[0] * g4.x, xn[1] * g4.y, xn[2] * g4.z, xn[3] * g4.w};
              *reinterpret_cast<uint2*>(static_cast<T16*>(ep.a_out) + off) =
                  make_uint2(pack2<T16>(ag[0], ag[1]), pack2<T16>(ag[2], ag[3]));
              if (ep.a_lo_out) {
                float lo[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) lo[k] = ag[k] - to_f(from_f<T16>(ag[k]));
                *reinterpret_cast<uint2*>(static_cast<T16*>(ep.a_lo_out) + off) =
                    make_uint2(pack2<T16>(lo[0], lo[1]), pack2<T16>(lo[2], lo[3]));
              }
              part = ((xn[0] * xn[0] + xn[1] * xn[1]) + xn[2] * xn[2]) + xn[3] * xn[3];
            }
            rs[i] += part;
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i) xcur[i] = xnext[i];
        }
        // a row's half tile: the 8 lanes of the row, fixed tree order
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          rs[i] += __shfl_xor_sync(0xffffffffu, rs[i], 1);
          rs[i] += __shfl_xor_sync(0xffffffffu, rs[i], 2);
          rs[i] += __shfl_xor_sync(0xffffffffu, rs[i], 4);
        }
        if ((lane & 7) == 0) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (rv[i]) ep.ss_out[static_cast<long long>(mrow + 4 * i) * ep.ss_out_stride + 2 * nb + half] = rs[i];
        }
      }
#pragma unroll 1
      for (int c2 = cb; c2 < ce && KIND != EPI_RESID; c2 += 32) {
        uint32_t v2[2][16];
        tmem_ld16(taddr + c2, v2[0]);
        tmem_ld16(taddr + c2 + 16, v2[1]);
        const int n2 = nb * bn + c2;
        // both chunks' rotation pairs and biases are requested together
        QkvIn in[KIND == EPI_QKV ? 2 : 1];
        if (KIND == EPI_QKV && mval) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (n2 + 16 * h < N) load_qkv16p(ep, pos, n2 + 16 * h, in[KIND == EPI_QKV ? h : 0]);
        }
        tmem_wait_ld();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int n0 = n2 + 16 * h;
          if (!mval || n0 >= N) continue;
          float f[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(v2[h][i]);
          if (KIND == EPI_QKV) {
            epi_qkv16p<T16>(ep, m, seq, pos, n0, f, rinv, in[KIND == EPI_QKV ? h : 0]);
          } else if (KIND == EPI_SWIGLU) {
            epi_swiglu16<T16>(ep, m, n0, f, rinv);
          } else if (KIND == EPI_ROWSCALE) {
            epi_rowscale16(ep, m, n0, f);
          } else {
            const unsigned long long k = epi_logits16(ep, m, n0, f, rinv);
            best = k > best ? k : best;
          }
        }
      }
      tc_fence_before();
      mbar_arrive(acce_bar(buf));

      if (KIND == EPI_LOGITS && mval) argmax_commit(ep.keys + m, best);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

template <int KIND, typename T16, bool SPLIT, int BN, int AROWS>
cudaError_t launch_kind(const LaunchCtx& lc, const GemmMaps& maps, int M, int N, int K, const EpiArgs& ep,
                        const GemmGroup& grp, int width) {
  const int tiles = ((M + BM - 1) / BM) * ((N + width - 1) / width);
  // grouped: the tile count is known only on the device; one CTA per SM
  const int grid = grp.mb_expert ? lc.num_sms : (tiles < lc.num_sms ? tiles : lc.num_sms);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = GCfgK<KIND, SPLIT, BN, AROWS>::SMEM + epi_smem<KIND>();
  cfg.stream = lc.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = lc.pdl ? 1 : 0;
  const GemmMaps& g = BN == 256 ? maps : *maps.n128;
  const CUtensorMap& ta = AROWS == 16 ? g.a16 : (AROWS == 64 ? g.a64 : g.a);
  const CUtensorMap& w = width == 224 ? g.w224 : (width == 192 ? g.w192 : g.w);
  const CUtensorMap& tlo = SPLIT ? (AROWS == 16 ? g.a_lo16 : (AROWS == 64 ? g.a_lo64 : g.a_lo)) : ta;
  return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<KIND, T16, SPLIT, BN, AROWS>, ta, w, tlo, M, N, K, width, ep, grp);
}

}  // namespace

bool make_tma_2d_16(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, bool f16) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(base) & 15) || ((cols * 2) & 15)) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(BK), box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_tma_3d_16(CUtensorMap* map, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint32_t box1,
                    uint32_t box2, bool f16) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(base) & 15) || ((d0 * 2) & 15)) return false;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {d0 * 2, d0 * d1 * 2};
  cuuint32_t box[3] = {static_cast<cuuint32_t>(BK), box1, box2};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base),
            dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_tma_2d_plain(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_cols,
                       uint32_t box_rows, bool f16) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(base) & 15) || ((cols * 2) & 15) || ((box_cols * 2) & 15)) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base),
            dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {
template <int KIND, typename T16, bool SPLIT, int BN, int AROWS>
cudaError_t set_smem1() {
  return cudaFuncSetAttribute(gemm_tc_kernel<KIND, T16, SPLIT, BN, AROWS>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              GCfgK<KIND, SPLIT, BN, AROWS>::SMEM + epi_smem<KIND>());
}
template <int KIND, typename T16, bool SPLIT>
cudaError_t set_smem() {
  cudaError_t e = set_smem1<KIND, T16, SPLIT, 256, 128>();
  if (e == cudaSuccess) e = set_smem1<KIND, T16, SPLIT, 128, 128>();
  return e;
}
// The small-M layouts.
template <int KIND, typename T16, bool SPLIT>
cudaError_t set_smem_few() {
  cudaError_t e = set_smem1<KIND, T16, SPLIT, 256, 16>();
  if (e == cudaSuccess) e = set_smem1<KIND, T16, SPLIT, 128, 16>();
  if (e == cudaSuccess) e = set_smem1<KIND, T16, SPLIT, 256, 64>();
  if (e == cudaSuccess) e = set_smem1<KIND, T16, SPLIT, 128, 64>();
  return e;
}
template <typename T16>
cudaError_t prepare_gemm_t() {
  cudaError_t e = set_smem<EPI_QKV, T16, false>();
  if (e == cudaSuccess) e = set_smem<EPI_QKV, T16, true>();
  if (e == cudaSuccess) e = set_smem<EPI_RESID, T16, false>();
  if (e == cudaSuccess) e = set_smem<EPI_SWIGLU, T16, false>();
  if (e == cudaSuccess) e = set_smem<EPI_LOGITS, T16, false>();
  if (e == cudaSuccess) e = set_smem<EPI_ROWSCALE, T16, false>();
  if (e == cudaSuccess) e = set_smem_few<EPI_SWIGLU, T16, false>();
  if (e == cudaSuccess) e = set_smem_few<EPI_LOGITS, T16, false>();
  return e;
}
template <typename T16, int BN>
cudaError_t launch_t(const LaunchCtx& lc, int kind, const GemmMaps& maps, int M, int N, int K, const EpiArgs& ep,
                     const GemmGroup& grp, int width) {
  switch (kind) {
    case EPI_QKV:
      return maps.split ? launch_kind<EPI_QKV, T16, true, BN, 128>(lc, maps, M, N, K, ep, grp, width)
                        : launch_kind<EPI_QKV, T16, false, BN, 128>(lc, maps, M, N, K, ep, grp, width);
    case EPI_RESID: return launch_kind<EPI_RESID, T16, false, BN, 128>(lc, maps, M, N, K, ep, grp, width);
    case EPI_SWIGLU: return launch_kind<EPI_SWIGLU, T16, false, BN, 128>(lc, maps, M, N, K, ep, grp, width);
    case EPI_ROWSCALE: return launch_kind<EPI_ROWSCALE, T16, false, BN, 128>(lc, maps, M, N, K, ep, grp, width);
    default: return launch_kind<EPI_LOGITS, T16, false, BN, 128>(lc, maps, M, N, K, ep, grp, width);
  }
}
// The small-M layouts (gate/up and logits); LO: a two-term operand.
template <typename T16, bool LO, int BN, int AROWS>
cudaError_t launch_few(const LaunchCtx& lc, int kind, const GemmMaps& maps, int M, int N, int K, const EpiArgs& ep) {
  return kind == EPI_SWIGLU ? launch_kind<EPI_SWIGLU, T16, LO, BN, AROWS>(lc, maps, M, N, K, ep, GemmGroup{}, BN)
                            : launch_kind<EPI_LOGITS, T16, LO, BN, AROWS>(lc, maps, M, N, K, ep, GemmGroup{}, BN);
}
template <int BN, int AROWS>
cudaError_t launch_few_t(const LaunchCtx& lc, int kind, const GemmMaps& maps, int M, int N, int K, const EpiArgs& ep,
                         bool lo) {
  if (!lc.f16) return launch_few<bf16, false, BN, AROWS>(lc, kind, maps, M, N, K, ep);
  return lo ? launch_few<f16, true, BN, AROWS>(lc, kind, maps, M, N, K, ep)
            : launch_few<f16, false, BN, AROWS>(lc, kind, maps, M, N, K, ep);
}
template <int BN>
cudaError_t launch_bn(const LaunchCtx& lc, int kind, const GemmMaps& maps, int M, int N, int K, const EpiArgs& ep,
                      const GemmGroup& grp, int arows, int width, bool lo) {
  if (arows == 16) return launch_few_t<BN, 16>(lc, kind, maps, M, N, K, ep, lo);
  if (arows == 64) return launch_few_t<BN, 64>(lc, kind, maps, M, N, K, ep, lo);
  return lc.f16 ? launch_t<f16, BN>(lc, kind, maps, M, N, K, ep, grp, width)
                : launch_t<bf16, BN>(lc, kind, maps, M, N, K, ep, grp, width);
}
}  // namespace

// Output-tile width for an M x N product: the cheapest count of waves, each
// priced by its width. A wave costs less than its columns: at 128 the
// reads of A weigh more and the tensor cores idle (down projection of 8B width,
// a wave of 128 / 192 / 224 / 256 columns 63 / 83.5 / 89 / 92 us: the weights
// below). 192 and 224 fill waves that the others leave half empty (8B width, 1024
// rows: QKV 128 62.7 us, 192 54.4, 256 59.0; down 256 92.0, 224 89.4; 1300 rows: O 128
// 63.5, 192 54.7, 256 60.1; down 186 / 157 / 167; 32B width, 512 rows: O 256 46.9, 192
// 40.8; 1024 rows: down 128 348, 192 283, 256 303). At most 64 rows (the small-M
// stages) and the grouped products know 128 and 256 only: 128 where 256-wide tiles
// leave the last wave mostly idle.
int gemm_tile_n(const LaunchCtx& lc, const GemmMaps& maps, int M, int N) {
  if (!maps.n128) return 256;
  const long long mt = (M + BM - 1) / BM;
  auto waves = [&](int bn) { return (mt * ((N + bn - 1) / bn) + lc.num_sms - 1) / lc.num_sms; };
  if (!maps.mid || M <= 64) return waves(128) * (128 + 16) * 100 < waves(256) * (256 + 16) * 85 ? 128 : 256;
  constexpr int WIDTH[4] = {256, 224, 192, 128}, COST[4] = {146, 139, 132, 100};
  int best = 0;
  for (int i = 1; i < 4; ++i)
    if (waves(WIDTH[i]) * COST[i] < waves(WIDTH[best]) * COST[best]) best = i;
  return WIDTH[best];
}

cudaError_t prepare_gemm_kernels() {
  cudaError_t e = prepare_gemm_t<bf16>();
  if (e == cudaSuccess) e = prepare_gemm_t<f16>();
  if (e == cudaSuccess) e = set_smem_few<EPI_SWIGLU, f16, true>();
  if (e == cudaSuccess) e = set_smem_few<EPI_LOGITS, f16, true>();
  return e;
}

cudaError_t launch_gemm_tc(const LaunchCtx& lc, int kind, const GemmMaps& maps, int M, int N, int K,
                           const EpiArgs& ep, int tile_n, const GemmGroup* group, bool lo) {
  if (M < 1 || N < 1 || K < BK || (K % BK)) return cudaErrorInvalidValue;
  const GemmGroup grp = group ? *group : GemmGroup{};
  if (grp.mb_expert && (!grp.n_mblocks || (M % BM))) return cudaErrorInvalidValue;
  if (kind == EPI_ROWSCALE && !grp.mb_expert) return cudaErrorInvalidValue;
  // at most 16 (64) rows -- one M block -- and activation boxes of 16 (64)
  // rows: the small-M stage layouts
  const bool few = maps.few && !grp.mb_expert && (kind == EPI_SWIGLU || kind == EPI_LOGITS);
  const int arows = !few || M > 64 ? 128 : (M <= 16 ? 16 : 64);
  if (lo && !(lc.f16 && maps.has_lo && arows < BM)) return cudaErrorInvalidValue;
  const bool mid = maps.mid && arows == 128 && !grp.mb_expert;
  if (tile_n != 256 && tile_n != 128 && !(mid && (tile_n == 192 || tile_n == 224))) return cudaErrorInvalidValue;
  if (tile_n == 128) {
    if (!maps.n128) return cudaErrorInvalidValue;
    return launch_bn<128>(lc, kind, maps, M, N, K, ep, grp, arows, 128, lo);
  }
  return launch_bn<256>(lc, kind, maps, M, N, K, ep, grp, arows, tile_n, lo);
}
