// Projections of few tokens (decode batches, short prompts) on tcgen05:
// out[m][n] = act[m] . W[n] for M <= 128 tokens (more in tiles of 128, where a
// product has few of them), fused epilogues as in epilogue.cuh.
//
// The product is bound by streaming W once. Here the weights are the 128-row
// operand of the MMA and the tokens its N dimension (16, 32, 64 or 128), so that a
// stage of 64 columns moves 16 KB of weights and only the token rows that exist,
// and K is split over the CTAs of a cluster: a projection of few 128-row tiles
// still has weight requests in flight on every SM. Each CTA leaves its fp32
// partial tile in its own shared memory; after one cluster barrier CTA r sums,
// in rank order, the partials of tokens r, r + ks, ... over distributed shared
// memory and runs their epilogues. No partials or tickets go through L2 (the
// 64-row fp32 partials of a split through L2 cost more than the idle SMs).
//
// Measured against the kernels that it replaced (the GEMV up to 32 tokens, split-K
// GEMM through L2, unsplit GEMM): 8B width, 64 tokens in fp16, one layer over a paged
// cache 308 -> 229 us of which the attention takes 99 (QKV 36.9 -> 20.3 us, O 29 ->
// 15.2, gate/up 50 -> 43.4 (235 MB), down 53 -> 28.4 (117 MB)); 32B width, 16 tokens,
// one layer 253 -> 222 us. About 5 us of each launch are fixed: launch, first
// weights, cluster barrier, epilogue.
//
//   warp 0 : TMA producer; requests the first stages' weights before the
//            preceding kernel has finished (they depend on nothing);
//   warp 1 : MMA issuer;
//   warps 2..7 : the tokens' norm scales, meanwhile;
//   all eight: accumulators to shared memory, sums and epilogues.
#include "kernels.h"

namespace {

constexpr int SK_THREADS = 256;
constexpr int SK_BN = 128;                // weight rows per tile
constexpr int SK_W_BYTES = SK_BN * 64 * 2;  // weights of a stage
constexpr int SK_PITCH = SK_BN + 4;       // floats per token row of the partial tile
constexpr int SK_MAX_STAGES = 12;
constexpr int SK_MAX_KS = 5;
constexpr int SK_MISC = 8 * (2 * SK_MAX_STAGES + 1) + 8 + 128 * 4;  // barriers, TMEM slot, norm scales

AXON_DEV uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
AXON_DEV void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
AXON_DEV float4 ld_cluster4(uint32_t addr, uint32_t rank) {
  float4 v;
  asm volatile(
      "{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %4, %5;\n ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [ra];\n}"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "r"(addr), "r"(rank)
      : "memory");
  return v;
}

// nt: token columns of the MMA (16, 32, 64, 128); lo: the activations are two
// 16-bit terms (a second MMA set on the second one); stages of the ring.
template <int KIND, typename T16>
__global__ void __launch_bounds__(SK_THREADS, 2)
    skinny_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA,
                  const __grid_constant__ CUtensorMap tmAlo, int M_all, int N, int K, EpiArgs ep, int ks, int nt, int lo,
                  int stages, int row0, int tiles_m) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const int act_bytes = nt * 128;
  const int stage_bytes = SK_W_BYTES + act_bytes * (1 + lo);
  const uint32_t misc = base + stages * stage_bytes;
  auto full_bar = [&](int s) { return misc + 8 * s; };
  auto empty_bar = [&](int s) { return misc + 8 * (SK_MAX_STAGES + s); };
  const uint32_t acc_bar = misc + 8 * (2 * SK_MAX_STAGES);
  const uint32_t tmem_slot = acc_bar + 8;
  float* const rinv_s = reinterpret_cast<float*>(smem_raw + (tmem_slot + 8 - raw));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t cols = nt < 32 ? 32u : static_cast<uint32_t>(nt);

  grid_dep_launch();
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(acc_bar, 1);
    fence_mbar_init();
    fence_proxy_async();
    tma_prefetch_desc(&tmW);
    tma_prefetch_desc(&tmA);
    if (lo) tma_prefetch_desc(&tmAlo);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<const uint32_t*>(smem_raw + (tmem_slot - raw));

  const int rank = ks > 1 ? static_cast<int>(cluster_rank()) : 0;
  // tile: 128 weight rows x nt tokens; the token tiles of one weight tile are
  // neighbours, so that its weights are read from memory once
  const int tile = blockIdx.x / ks / tiles_m, n_tile = tile * SK_BN;
  const int m_tile = (blockIdx.x / ks - tile * tiles_m) * nt;
  const int M = min(M_all - m_tile, nt);  // tokens of this tile
  const int KB = K / 64, kb0 = rank * KB / ks, nkb = (rank + 1) * KB / ks - kb0;

  if (warp == 0) {
    if (lane == 0) {
      // weights are read once: they should not push the cache and activations out of L2
      const uint64_t policy = createpolicy_evict_first();
      auto load_w = [&](int i) {
        const int s = i % stages;
        mbar_arrive_expect_tx(full_bar(s), stage_bytes);
        tma_load_2d_hint(base + s * stage_bytes, &tmW, full_bar(s), (kb0 + i) * 64, n_tile, policy);
      };
      auto load_a = [&](int i) {
        const int s = i % stages;
        const uint32_t dst = base + s * stage_bytes + SK_W_BYTES;
        tma_load_2d(dst, &tmA, full_bar(s), (kb0 + i) * 64, row0 + m_tile);
        if (lo) tma_load_2d(dst + act_bytes, &tmAlo, full_bar(s), (kb0 + i) * 64, row0 + m_tile);
      };
      const int ahead = nkb < stages ? nkb : stages;
      for (int i = 0; i < ahead; ++i) load_w(i);
      grid_dep_wait();
      for (int i = 0; i < ahead; ++i) load_a(i);
      for (int i = ahead; i < nkb; ++i) {
        if (!mbar_wait(empty_bar(i % stages), ((i / stages) & 1) ^ 1, ep.err)) {
          // copies in flight land before the shared memory is reused
          for (int j = i - stages; j < i; ++j) mbar_wait(full_bar(j % stages), (j / stages) & 1, ep.err);
          break;
        }
        load_w(i);
        load_a(i);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_f32acc(SK_BN, nt, MmaFmt<T16>::v);
      bool ok = true;
      for (int i = 0; i < nkb; ++i) {
        const int s = i % stages;
        ok = mbar_wait(full_bar(s), (i / stages) & 1, ep.err);
        if (!ok) break;
        tc_fence_after();
        const uint64_t wd = smem_desc_sw128(base + s * stage_bytes);
        const uint64_t ad = smem_desc_sw128(base + s * stage_bytes + SK_W_BYTES);
#pragma unroll
        for (int k = 0; k < 4; ++k) tc_mma_f16(tmem, wd + 2 * k, ad + 2 * k, idesc, (i != 0 || k != 0) ? 1u : 0u);
        if (lo) {
          const uint64_t ld = smem_desc_sw128(base + s * stage_bytes + SK_W_BYTES + act_bytes);
#pragma unroll
          for (int k = 0; k < 4; ++k) tc_mma_f16(tmem, wd + 2 * k, ld + 2 * k, idesc, 1u);
        }
        tc_commit(empty_bar(s));
      }
      tc_commit(acc_bar);
    }
    __syncwarp();
  }
  grid_dep_wait();
  // the tokens' norm scales, eight tokens' reads in flight per warp
  if (KIND != EPI_RESID && warp >= 2) {
    if (ep.rinv) {
      for (int m = threadIdx.x - 64; m < M; m += SK_THREADS - 64)
        rinv_s[m] = ep.rinv[static_cast<long long>(m_tile + m) * ep.rinv_stride];
    } else {
      constexpr int U = 8;
      for (int m0 = (warp - 2) * U; m0 < M; m0 += 6 * U) {
        float s[U];
#pragma unroll
        for (int u = 0; u < U; ++u) s[u] = 0.f;
        for (int i = lane; i < ep.ss_parts; i += 32) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (m0 + u < M) s[u] += ep.ss[static_cast<long long>(m_tile + m0 + u) * ep.ss_stride + i];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          s[u] = warp_sum(s[u]);
          if (lane == 0 && m0 + u < M) rinv_s[m0 + u] = 1.0f / sqrtf(s[u] * ep.inv_D + ep.eps);
        }
      }
    }
  }

  // tasks (token, 16 rows): eight neighbouring lanes hold one token's tile.
  // The first task's global inputs are requested while the product runs.
  const int mine = (M - rank + ks - 1) / ks;  // tokens rank, rank + ks, ...
  float4 xin[4];
  QkvIn qin;
  auto load_in = [&](int t) {
    const int m = rank + (t >> 3) * ks, n0 = n_tile + (t & 7) * 16;
    if (t >= mine * 8 || n0 >= N) return;
    if (KIND == EPI_RESID) load_resid16(ep, m_tile + m, n0, xin);
    if (KIND == EPI_QKV) load_qkv16(ep, m_tile + m, n0, qin);
  };
  load_in(threadIdx.x);

  // accumulators -> [token][weight row] in the ring's memory (every stage was
  // consumed); a warp reads its lane quarter, the two halves of the CTA take
  // alternate groups of 16 tokens
  mbar_wait(acc_bar, 0, ep.err);
  __syncthreads();  // also: the norm scales
  tc_fence_after();
  float* const part = reinterpret_cast<float*>(smem_raw + (base - raw));
  {
    const uint32_t taddr = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const int row = (warp & 3) * 32 + lane;
    for (int c = (warp >> 2) * 16; c < nt && c < M; c += 32) {
      uint32_t v[16];
      tmem_ld16(taddr + c, v);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; ++i) part[(c + i) * SK_PITCH + row] = __uint_as_float(v[i]);
    }
  }
  tc_fence_before();
  if (ks > 1)
    cluster_sync();
  else
    __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, cols);
  }

  // ks > 1: the sums over the cluster, a token row (512 contiguous bytes of every
  // peer) per warp and step, into this CTA's own rows behind the partials. (Read
  // by the tasks themselves, 64 bytes per lane, the sums of 64 tokens took 7 us.)
  const float* src = part;
  if (ks > 1) {
    float* const sums = part + nt * SK_PITCH;
    src = sums;
    for (int t = warp; t < mine; t += SK_THREADS / 32) {
      const uint32_t at = base + ((rank + t * ks) * SK_PITCH + lane * 4) * 4;
      float4 v[SK_MAX_KS];
#pragma unroll
      for (int r = 0; r < SK_MAX_KS; ++r)
        if (r < ks) v[r] = ld_cluster4(at, r);
      float4 s = v[0];
#pragma unroll
      for (int r = 1; r < SK_MAX_KS; ++r) {
        if (r >= ks) break;
        s.x += v[r].x;
        s.y += v[r].y;
        s.z += v[r].z;
        s.w += v[r].w;
      }
      *reinterpret_cast<float4*>(sums + t * SK_PITCH + lane * 4) = s;
    }
    __syncthreads();
  }
  for (int t0 = 0; t0 < mine * 8; t0 += SK_THREADS) {
    const int t = t0 + threadIdx.x;
    const int c = t & 7, m = rank + (t >> 3) * ks, n0 = n_tile + c * 16;
    const bool on = t < mine * 8 && n0 < N;
    float ssum = 0.f;
    unsigned long long best = 0ull;
    if (t0 > 0) load_in(t);
    if (on) {
      float f[16];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(src + (t >> 3) * SK_PITCH + c * 16 + 4 * i);
        f[4 * i] = v.x;
        f[4 * i + 1] = v.y;
        f[4 * i + 2] = v.z;
        f[4 * i + 3] = v.w;
      }
      if (KIND == EPI_QKV) {
        epi_qkv16x<T16>(ep, m_tile + m, n0, f, rinv_s[m], qin);
      } else if (KIND == EPI_RESID) {
        ssum = epi_resid16x<T16>(ep, m_tile + m, n0, f, xin);
      } else if (KIND == EPI_SWIGLU) {
        epi_swiglu16<T16>(ep, m_tile + m, n0, f, rinv_s[m]);
      } else {
        best = epi_logits16(ep, m_tile + m, n0, f, rinv_s[m]);
      }
    }
    if (KIND == EPI_RESID) {
      // the row's norm partial of this tile, in a fixed order
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) ssum += __shfl_xor_sync(0xffffffffu, ssum, o);
      if (on && c == 0) ep.ss_out[static_cast<long long>(m_tile + m) * ep.ss_out_stride + tile] = ssum;
    } else if (KIND == EPI_LOGITS) {
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const unsigned long long k = __shfl_xor_sync(0xffffffffu, best, o);
        best = k > best ? k : best;
      }
      if (on && c == 0) argmax_commit(ep.keys + m_tile + m, best);
    }
  }
  __syncwarp();
  if (ks > 1) cluster_sync();  // peers may still read this CTA's partials
}

template <int KIND, typename T16>
cudaError_t launch_kind(const LaunchCtx& lc, const CUtensorMap& w, const CUtensorMap& a, const CUtensorMap& alo, int M,
                        int N, int K, const EpiArgs& ep, const SkinnyPlan& pl, int row0) {
  cudaLaunchConfig_t cfg = {};
  const int tiles_m = (M + pl.nt - 1) / pl.nt;
  cfg.gridDim = dim3((N + SK_BN - 1) / SK_BN * tiles_m * pl.ks);
  cfg.blockDim = dim3(SK_THREADS);
  const int lo = pl.lo ? 1 : 0;
  cfg.dynamicSmemBytes = 1024 + pl.stages * (SK_W_BYTES + pl.nt * 128 * (1 + lo)) + SK_MISC;
  cfg.stream = lc.stream;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (pl.ks > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = pl.ks;
    attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (lc.pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, skinny_kernel<KIND, T16>, w, a, alo, M, N, K, ep, pl.ks, pl.nt, lo, pl.stages, row0,
                            tiles_m);
}

template <typename T16>
cudaError_t launch_t(const LaunchCtx& lc, int kind, const CUtensorMap& w, const CUtensorMap& a, const CUtensorMap& alo,
                     int M, int N, int K, const EpiArgs& ep, const SkinnyPlan& pl, int row0) {
  switch (kind) {
    case EPI_QKV: return launch_kind<EPI_QKV, T16>(lc, w, a, alo, M, N, K, ep, pl, row0);
    case EPI_RESID: return launch_kind<EPI_RESID, T16>(lc, w, a, alo, M, N, K, ep, pl, row0);
    case EPI_SWIGLU: return launch_kind<EPI_SWIGLU, T16>(lc, w, a, alo, M, N, K, ep, pl, row0);
    case EPI_LOGITS: return launch_kind<EPI_LOGITS, T16>(lc, w, a, alo, M, N, K, ep, pl, row0);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T16>
cudaError_t prepare_t() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto* k) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SKINNY_MAX_SMEM);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  };
  set(skinny_kernel<EPI_QKV, T16>);
  set(skinny_kernel<EPI_RESID, T16>);
  set(skinny_kernel<EPI_SWIGLU, T16>);
  set(skinny_kernel<EPI_LOGITS, T16>);
  return e;
}

}  // namespace

// Clusters of ks CTAs that fit the device at one CTA per SM (index ks).
static int g_clusters[SK_MAX_KS + 1] = {};

cudaError_t prepare_skinny_kernels() {
  cudaError_t e = prepare_t<bf16>();
  if (e == cudaSuccess) e = prepare_t<f16>();
  for (int ks = 1; ks <= SK_MAX_KS && e == cudaSuccess; ++ks) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ks);
    cfg.blockDim = dim3(SK_THREADS);
    cfg.dynamicSmemBytes = SKINNY_MAX_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&g_clusters[ks], skinny_kernel<EPI_QKV, bf16>, &cfg);
  }
  return e;
}

bool make_act_maps(ActMaps* maps, const void* act, const void* act_lo, long long rows, long long lo_rows, long long K,
                   bool f16) {
  const uint32_t box[4] = {16, 32, 64, 128};
  maps->lo = act_lo != nullptr;
  for (int i = 0; i < 4; ++i) {
    if (!make_tma_2d_16(&maps->t[i], act, rows, K, box[i], f16)) return false;
    if (act_lo && !make_tma_2d_16(&maps->l[i], act_lo, lo_rows, K, box[i], f16)) return false;
  }
  return true;
}

SkinnyPlan skinny_plan(const LaunchCtx& lc, int M, int N, int K, bool lo) {
  SkinnyPlan pl;
  if (M < 1 || (K & 63)) return pl;
  pl.nt = M <= 16 ? 16 : (M <= 32 ? 32 : (M <= 64 ? 64 : 128));
  pl.lo = lo;
  const int tiles_m = (M + pl.nt - 1) / pl.nt, tiles = (N + SK_BN - 1) / SK_BN * tiles_m, KB = K / 64;
  const int stage = SK_W_BYTES + pl.nt * 128 * (lo ? 2 : 1);
  // More than 128 tokens: only where the tiles leave at least half the SMs without
  // work and K is long enough to share.
  if (tiles_m > 1 && (2 * tiles > lc.num_sms || K < 2048)) return pl;
  const int per_sm = pl.nt == 128 ? 1 : 2;
  if (tiles > per_sm * g_clusters[1]) return pl;
  const int budget = (per_sm == 1 ? SKINNY_MAX_SMEM : SKINNY_MAX_SMEM / 2) - 1024 - SK_MISC - 1024;
  pl.stages = budget / stage;
  if (pl.stages > SK_MAX_STAGES) pl.stages = SK_MAX_STAGES;
  // As many CTAs per tile as the clusters resident at a time allow, with at
  // least 4 K blocks each. Beyond 5 (4 with the wider token tiles, whose
  // activation rows every CTA of a tile reads again) a launch got no shorter,
  // and a second wave of clusters doubles it (8B width, 8 tokens, QKV, 3 / 4 / 5 /
  // 6 CTAs: 16.9 / 15.9 / 15.5 / 24.4 us; 64 tokens: 24.9 / 23.4 / 25.4 / 34.7).
  int ks = pl.nt <= 32 ? SK_MAX_KS : 4;
  while (ks > 1 && (KB / ks < 4 || tiles > per_sm * g_clusters[ks])) --ks;
  pl.ks = ks;
  return pl;
}

cudaError_t launch_skinny(const LaunchCtx& lc, int kind, const CUtensorMap& w, const ActMaps& act, int M, int N, int K,
                          const EpiArgs& ep, const SkinnyPlan& pl, int row0) {
  if (pl.ks < 1 || pl.ks > SK_MAX_KS || M < 1 || N < 1 || (K & 63) || K / 64 < pl.ks || pl.stages < 2 ||
      (pl.lo && !act.lo))
    return cudaErrorInvalidValue;
  const int i = pl.nt == 16 ? 0 : (pl.nt == 32 ? 1 : (pl.nt == 64 ? 2 : 3));
  const CUtensorMap& lo = pl.lo ? act.l[i] : act.t[i];
  return lc.f16 ? launch_t<f16>(lc, kind, w, act.t[i], lo, M, N, K, ep, pl, row0)
                : launch_t<bf16>(lc, kind, w, act.t[i], lo, M, N, K, ep, pl, row0);
}
