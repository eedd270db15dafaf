// Prefill attention on the 5th-generation tensor cores: causal grouped-query
// flash attention over the block-structured KV cache (layout in k_attn.cu),
// 16-bit modes.
//
// A tile is 128 rows = PW consecutive positions x the H/G query heads of one
// kv head (PW = 128 / (H/G), so up to H/G - 1 rows are padding); a CTA owns
// two such tiles (consecutive positions) and streams the keys they see
// through one ring, 128 keys at a time:
//   warps 0..3, 4..7 : softmax of tile 0, tile 1 -- one thread per row, so
//                      that the row maximum and sum need no shuffles;
//   warp 8           : TMA producer -- Q once (a 3-D box of 64 dims x H/G
//                      heads x PW positions per chunk), then K and V as eight
//                      16-token cache blocks per stage, lane i fetching the
//                      table entry of block i and issuing its boxes;
//   warp 9           : MMA issuer -- S = Q K^T into TMEM, O += P V with P
//                      read back from TMEM and O accumulating in TMEM.
// The 512 TMEM columns hold S0, S1 (128 each) and O0, O1 (HD each); a tile's
// probabilities (16-bit, 64 columns) and their second terms (8 columns) overwrite
// its scores. The issuer alternates the tiles, so one tile's softmax runs under the
// other's MMAs.
//
// Rounding of the probabilities, which must cost no more than in the mma.sync
// kernel: O is rescaled in TMEM whenever a row's maximum has grown, so that the
// largest probability is 1 and enters P V exactly; the row sum takes the rounded
// values; and since a maximum over 128 keys leaves fewer of a row's running
// maxima exact than one over 32, the first KT2 keys of a tile have a second 16-bit
// term (one more MMA of 16 keys). rms error of one layer in fp16, this / mma.sync, at
// scores of standard deviation 1.0, 1.64 (8B width) and 2.5: 0.982, 0.992, 0.994; without
// the second terms 1.010, 1.012, 1.005; rescaled only on a growth of 2^8 and with an
// unrounded sum 1.059, 1.103, 1.147; with second terms of all keys 0.789, 0.857, 0.913 at
// 22 % more time. Whole prefills against 64 bits, 8B width, fp16, 512 tokens: mma.sync 8.53e-4,
// this 8.50e-4 (rescaled on 2^8: 8.65e-4).
//
// Bound: at head_dim 128 a 128 x 128 tile takes 544 tensor cycles and nearly as many
// exponential-unit cycles, and the softmax's issue slots come to about the
// same. Measured by events against the mma.sync kernel (4 warps x 16 rows, scores in
// registers, k_attn.cu; still taken for short prompts) and this one with the lagging
// maximum: 8B width, 8191 positions under a 4096-key window 1681 / 387 / 432 us,
// 32B width, 4 x 2048 positions 916 / 243 / 269 us, 8B width, 1024 positions
// 62 / 28.8 / 30.9 us.
#include <math.h>

#include "kernels.h"

namespace {

constexpr int TC_THREADS = 320;
constexpr int KT = 128;  // keys per tile
constexpr int KT2 = 16;  // the first keys of a tile: their probabilities have two 16-bit terms

template <int HD>
struct ACfg {
  static constexpr int CH = HD / 64;                   // 64-dim chunks (128-byte swizzled rows)
  static constexpr int CHUNK = 128 * 128;              // bytes of one 128-row chunk
  static constexpr int TILE = CH * CHUNK;              // Q, K or V tile
  static constexpr int STAGES = HD == 128 ? 5 : 8;     // K and V tiles in flight
  static constexpr int BARS = 2 * STAGES + 1 + 2 + 2 + 2;
  static constexpr int SMEM = 2 * TILE + STAGES * TILE + 8 * BARS + 16 + 1024;
};

AXON_DEV void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem desc] (A: 128 lanes, two 16-bit values per column).
AXON_DEV void tc_mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(
          d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

AXON_DEV void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,"
      "%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
AXON_DEV void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,"
      "%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
AXON_DEV void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
AXON_DEV void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

AXON_DEV float ex2(float v) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
// Two fp32 values in one 64-bit register: the packed FMA and add take one
// issue slot for both.
AXON_DEV uint64_t pk2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
AXON_DEV void upk2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
AXON_DEV uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
AXON_DEV uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// Probabilities lie in [0, 1]: no saturation needed.
template <typename T> AXON_DEV uint32_t pack_p(float lo, float hi);
template <> AXON_DEV uint32_t pack_p<bf16>(float lo, float hi) { return pack_bf2(lo, hi); }
template <> AXON_DEV uint32_t pack_p<f16>(float lo, float hi) {
  __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
// What the two 16-bit roundings in p lost of a and e.
template <typename T> AXON_DEV uint32_t pack_rest(float a, float e, uint32_t p);
template <> AXON_DEV uint32_t pack_rest<bf16>(float a, float e, uint32_t p) {
  return pack_bf2(a - bf_lo(p), e - bf_hi(p));
}
template <> AXON_DEV uint32_t pack_rest<f16>(float a, float e, uint32_t p) {
  const float2 r = __half22float2(*reinterpret_cast<__half2*>(&p));
  return pack_p<f16>(a - r.x, e - r.y);
}
// lo += the low, hi += the high 16-bit value of p.
template <typename T> AXON_DEV void add_p(float& lo, float& hi, uint32_t p);
template <> AXON_DEV void add_p<bf16>(float& lo, float& hi, uint32_t p) {
  asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n add.f32.bf16 %0, l, %0;\n add.f32.bf16 %1, h, %1;\n}"
      : "+f"(lo), "+f"(hi)
      : "r"(p));
}
template <> AXON_DEV void add_p<f16>(float& lo, float& hi, uint32_t p) {
  asm("{\n .reg .f16 l, h;\n mov.b32 {l, h}, %2;\n add.f32.f16 %0, l, %0;\n add.f32.f16 %1, h, %1;\n}"
      : "+f"(lo), "+f"(hi)
      : "r"(p));
}

// The V tile as the B operand of P V: N = dims (contiguous in memory), K =
// tokens at 128-byte pitch; 8-token groups 1024 bytes apart, the second 64
// dims one chunk further.
template <int HD>
AXON_DEV uint64_t v_desc(uint32_t addr) {
  uint64_t d = smem_desc_sw128(addr);
  d &= ~(static_cast<uint64_t>(0x3FFFu) << 16);
  d |= static_cast<uint64_t>(ACfg<HD>::CHUNK >> 4) << 16;
  return d;
}

// The work item of a CTA: sequence b and tile pair `pb` (positions pb * 2 * PW
// onward of its chunk). Prompts of one length: pairs counted down from the
// end, all sequences and kv heads of a pair together, so that the launch ends
// with the short items. Variable-length: a linear index over the sequences'
// pairs (at most rows / (2 PW) + B of them), found by scanning the offsets
// 32 sequences at a time. Returns false when the CTA has no item.
AXON_DEV bool find_item(const AttnArgs& p, const AttnVarlen& vl, int B, int PC, int item, int& b, int& pb, int& row0,
                        int& S, int& past) {
  if (!vl.cu) {
    const int n = (p.S + PC - 1) / PC;
    b = item % B;
    pb = n - 1 - item / B;
    row0 = b * p.S;
    S = p.S;
    past = 0;
    return pb >= 0;
  }
  const int lane = threadIdx.x & 31;
  int before = 0;
  for (int b0 = 0; b0 < B; b0 += 32) {
    int r0 = 0, len = 0, ps = 0;
    if (b0 + lane < B) {
      r0 = vl.cu[b0 + lane];
      const int r1 = vl.cu[b0 + lane + 1];
      ps = vl.past[b0 + lane];
      len = r1 - r0;
      // inconsistent offsets (reported by the row-map kernel): no work
      if (r0 < 0 || r1 > vl.rows || len < 0 || len > p.S || ps < 0 || ps + len > p.blocks_per_seq * 16) len = 0;
    }
    const int mine = (len + PC - 1) / PC;
    int end = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += t;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, item < before + end);
    if (hit) {
      const int src = __ffs(hit) - 1;
      b = b0 + src;
      row0 = __shfl_sync(0xffffffffu, r0, src);
      S = __shfl_sync(0xffffffffu, len, src);
      past = __shfl_sync(0xffffffffu, ps, src);
      pb = before + __shfl_sync(0xffffffffu, end, src) - 1 - item;  // counted down
      return true;
    }
    before += __shfl_sync(0xffffffffu, end, 31);
  }
  return false;
}

template <int HD, typename T16>
__global__ void __launch_bounds__(TC_THREADS, 1)
    attn_prefill_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                           const __grid_constant__ CUtensorMap tmV, AttnArgs p, int B, int PW, int pool_row0,
                           int pool_rows, AttnVarlen vl) {
  using C = ACfg<HD>;
  constexpr int NS = C::STAGES;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t sQ = base, sKV = base + 2 * C::TILE, bars = sKV + NS * C::TILE;
  auto kv_full = [&](int s) { return bars + 8 * s; };
  auto kv_empty = [&](int s) { return bars + 8 * (NS + s); };
  const uint32_t q_full = bars + 8 * (2 * NS);
  auto s_full = [&](int w) { return bars + 8 * (2 * NS + 1 + w); };
  auto p_full = [&](int w) { return bars + 8 * (2 * NS + 3 + w); };
  auto o_full = [&](int w) { return bars + 8 * (2 * NS + 5 + w); };
  const uint32_t tmem_slot = bars + 8 * C::BARS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int HPG = p.H / p.G;

  grid_dep_launch();
  // the set-up runs under the previous kernel's tail
  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(kv_full(s), 1);
      mbar_init(kv_empty(s), 1);
    }
    mbar_init(q_full, 1);
    for (int w = 0; w < 2; ++w) {
      mbar_init(s_full(w), 1);
      mbar_init(p_full(w), 128);
      mbar_init(o_full(w), 1);
    }
    fence_mbar_init();
    fence_proxy_async();
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  if (warp == 9) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<const uint32_t*>(smem_raw + (tmem_slot - raw));
  grid_dep_wait();

  const int g = blockIdx.x % p.G;
  int b = 0, pb = 0, row0 = 0, S = 0, past = 0;
  const bool item = find_item(p, vl, B, 2 * PW, blockIdx.x / p.G, b, pb, row0, S, past);
  const int p0 = pb * 2 * PW;  // first position of the chunk in tile 0
  const int nw = !item ? 0 : (p0 + PW < S ? 2 : 1);  // tiles with rows
  // Keys klo .. pend-1 are visible to some row (klo > 0 only under a sliding
  // window), from block jlo on.
  const int W = p.window;
  const int pend = past + min(p0 + nw * PW, S);
  const int klo = (W > 0 && past + p0 >= W) ? past + p0 - W + 1 : 0;
  const int jlo = klo >> 4, jend = (pend + 15) >> 4;
  const int nt = (jend - jlo + 7) >> 3;
  const int tail = (jend - jlo) * 16 - (nt - 1) * KT;  // keys of the last tile, a multiple of 16

  if (!item) {
    // a spare CTA of a variable-length batch: only TMEM to give back
  } else if (warp == 8) {
    // -------------------------------------------------------------- producer
    if (lane == 0) {
      mbar_arrive_expect_tx(q_full, nw * HPG * PW * HD * 2);
      for (int w = 0; w < nw; ++w)
        for (int c = 0; c < C::CH; ++c)
          tma_load_3d(sQ + w * C::TILE + c * C::CHUNK, &tmQ, q_full, c * 64, g * HPG, row0 + p0 + w * PW);
    }
    // pool row of this lane's block of key tile t; past the last block and for
    // table entries out of range (reported) the row lies outside the pool,
    // where a box reads zeros
    auto pool_row = [&](int t) {
      const int j = jlo + t * 8 + lane;
      if (lane >= 8 || t >= nt || j >= jend) return pool_rows;
      const int blk =
          p.block_table ? p.block_table[static_cast<long long>(b) * p.bt_stride + j] : b * p.blocks_per_seq + j;
      if (blk < 0 || blk >= p.num_blocks) {
        set_err(p.err, DEVERR_BLOCK);
        return pool_rows;
      }
      return pool_row0 + (blk * p.G + g) * 16;
    };
    int next = pool_row(0), it = 0;
    bool ok = true;
    for (int t = 0; t < nt && ok; ++t) {
      const int y = next;
      next = pool_row(t + 1);
      for (int kv = 0; kv < 2; ++kv, ++it) {
        const int s = it % NS;
        ok = __all_sync(0xffffffffu, mbar_wait(kv_empty(s), ((it / NS) & 1) ^ 1, p.err));
        if (!ok) break;
        if (lane == 0) mbar_arrive_expect_tx(kv_full(s), C::TILE);
        __syncwarp();
        if (lane < 8)
          for (int c = 0; c < C::CH; ++c)
            tma_load_2d(sKV + s * C::TILE + c * C::CHUNK + lane * 2048, kv ? &tmV : &tmK, kv_full(s), c * 64, y);
      }
    }
    // every copy lands before the CTA's shared memory goes away (all were consumed
    // unless a wait ran out)
    mbar_wait(q_full, 0, p.err);
    for (int i = it > NS ? it - NS : 0; i < it; ++i) mbar_wait(kv_full(i % NS), (i / NS) & 1, p.err);
  } else if (warp == 9) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t id_s = idesc_f32acc(128, KT, MmaFmt<T16>::v);
      constexpr uint32_t id_o = idesc_f32acc(128, HD, MmaFmt<T16>::v) | (1u << 16);  // B stored N-contiguous
      auto issue_s = [&](int w, int slot) {
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint32_t off = (k >> 2) * C::CHUNK + (k & 3) * 32;
          tc_mma_f16(tmem + w * KT, smem_desc_sw128(sQ + w * C::TILE + off),
                     smem_desc_sw128(sKV + slot * C::TILE + off), id_s, k != 0);
        }
        tc_commit(s_full(w));
      };
      bool ok = mbar_wait(q_full, 0, p.err) && mbar_wait(kv_full(0), 0, p.err);
      if (ok) {
        tc_fence_after();
        for (int w = 0; w < nw; ++w) issue_s(w, 0);
        tc_commit(kv_empty(0));
      }
      for (int t = 0; t < nt && ok; ++t) {
        const int iv = 2 * t + 1, ik = 2 * t + 2;
        const int sv = iv % NS, sk = ik % NS;
        const bool more = t + 1 < nt;
        ok = mbar_wait(kv_full(sv), (iv / NS) & 1, p.err) && (!more || mbar_wait(kv_full(sk), (ik / NS) & 1, p.err));
        for (int w = 0; w < nw && ok; ++w) {
          ok = mbar_wait(p_full(w), t & 1, p.err);
          if (!ok) break;
          tc_fence_after();
          const int ks = more ? KT / 16 : tail / 16;
          for (int k = 0; k < ks; ++k) {
            const uint64_t vd = v_desc<HD>(sKV + sv * C::TILE + k * 2048);
            tc_mma_f16_ts(tmem + 2 * KT + w * HD, tmem + w * KT + k * 8, vd, id_o, (t != 0 || k != 0) ? 1u : 0u);
            if (k < KT2 / 16) tc_mma_f16_ts(tmem + 2 * KT + w * HD, tmem + w * KT + KT / 2 + k * 8, vd, id_o, 1u);
          }
          // MMAs run in issue order: the next scores may overwrite the
          // probabilities just issued, and s_full implies that O is up to date
          if (more)
            issue_s(w, sk);
          else
            tc_commit(o_full(w));
        }
        if (ok) {
          tc_commit(kv_empty(sv));
          if (more) tc_commit(kv_empty(sk));
        }
      }
    }
    __syncwarp();
  } else {
    // --------------------------------------------------------------- softmax
    const int w = warp >> 2;
    if (w < nw) {
      const int i = threadIdx.x & 127;  // row of the tile
      const int pl = i / HPG, h = i - pl * HPG;
      const int ip = p0 + w * PW + pl;
      const bool valid = i < HPG * PW && ip < S;
      const int pos = valid ? past + ip : -1;
      const int lo = (W > 0 && pos >= W) ? pos - W + 1 : 0;
      const uint32_t lanes = static_cast<uint32_t>((warp & 3) * 32) << 16;
      const uint32_t tS = tmem + lanes + w * KT, tO = tmem + lanes + 2 * KT + w * HD;
      const float sl2 = p.scale_log2;
      float m = -INFINITY, l = 0.f;
      bool ok = true;
      for (int t = 0; t < nt; ++t) {
        ok = __all_sync(0xffffffffu, mbar_wait(s_full(w), t & 1, p.err));
        if (!ok) break;
        tc_fence_after();
        // short prompts and single tokens end in a short tile: its columns past
        // the last key (in steps of 64) are neither exponentiated nor multiplied
        const bool half = t == nt - 1 && tail <= 64;
        float s[KT];
        tmem_ld32(tS, reinterpret_cast<uint32_t*>(s));
        tmem_ld32(tS + 32, reinterpret_cast<uint32_t*>(s) + 32);
        if (!half) {
          tmem_ld32(tS + 64, reinterpret_cast<uint32_t*>(s) + 64);
          tmem_ld32(tS + 96, reinterpret_cast<uint32_t*>(s) + 96);
        }
        tmem_wait_ld();
        if (half) {
#pragma unroll
          for (int c = 64; c < KT; ++c) s[c] = -INFINITY;
        }
        const int tok0 = (jlo + t * 8) * 16;
        // padding rows reach no output: they alone never ask for the mask
        if (!__all_sync(0xffffffffu, !valid || (tok0 + KT - 1 <= pos && tok0 >= lo))) {
#pragma unroll
          for (int c = 0; c < KT; ++c) s[c] = (tok0 + c <= pos && tok0 + c >= lo) ? s[c] : -INFINITY;
        }
        float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
        for (int c = 4; c < KT; c += 8) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            mx[u] = c + 4 + u < KT ? fmaxf(mx[u], fmaxf(s[c + u], s[c + 4 + u])) : fmaxf(mx[u], s[c + u]);
        }
        const float mt = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sl2;
        if (__any_sync(0xffffffffu, mt > m)) {
          const float nm = fmaxf(m, mt);
          const float f = m == -INFINITY ? 0.f : ex2(m - nm);
          l *= f;
          m = nm;
          if (t > 0) {
            const uint64_t f2 = pk2(f, f);
#pragma unroll 1
            for (int c = 0; c < HD; c += 32) {
              float o[32];
              tmem_ld32(tO + c, reinterpret_cast<uint32_t*>(o));
              tmem_wait_ld();
#pragma unroll
              for (int u = 0; u < 32; u += 2) upk2(mul2(pk2(o[u], o[u + 1]), f2), o[u], o[u + 1]);
              tmem_st32(tO + c, reinterpret_cast<uint32_t*>(o));
            }
          }
        }
        const float nb = m == -INFINITY ? 0.f : -m;
        const uint64_t sl2p = pk2(sl2, sl2), nbp = pk2(nb, nb);
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c0 = 0; c0 < KT; c0 += 64) {
          if (c0 == 64 && half) break;
          uint32_t pr[32], rest[8];
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            float a, e;
            upk2(fma2(pk2(s[c0 + 2 * c], s[c0 + 2 * c + 1]), sl2p, nbp), a, e);
            a = ex2(a);
            e = ex2(e);
            pr[c] = pack_p<T16>(a, e);
            if (c0 == 0 && c < KT2 / 2) {
              rest[c & 7] = pack_rest<T16>(a, e, pr[c]);
              sum[(c & 1) * 2] += a;
              sum[(c & 1) * 2 + 1] += e;
              if ((c & 7) == 7) tmem_st8(tS + KT / 2 + (c & ~7), rest);
            } else {
              add_p<T16>(sum[(c & 1) * 2], sum[(c & 1) * 2 + 1], pr[c]);
            }
          }
          tmem_st32(tS + c0 / 2, pr);
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(p_full(w));
        l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
      }
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(o_full(w), 0, p.err));
      if (ok) {
        tc_fence_after();
        const float inv = l > 0.f ? 1.f / l : 0.f;
        uint4* dst = reinterpret_cast<uint4*>(static_cast<T16*>(p.o) +
                                              (static_cast<long long>(row0) + ip) * p.H * HD + (g * HPG + h) * HD);
#pragma unroll 1
        for (int c = 0; c < HD; c += 32) {
          uint32_t o[32];
          tmem_ld32(tO + c, o);
          tmem_wait_ld();
          if (valid) {
#pragma unroll
            for (int u = 0; u < 32; u += 8) {
              float v[8];
#pragma unroll
              for (int k = 0; k < 8; ++k) v[k] = __uint_as_float(o[u + k]) * inv;
              dst[(c + u) >> 3] = make_uint4(pack2<T16>(v[0], v[1]), pack2<T16>(v[2], v[3]), pack2<T16>(v[4], v[5]),
                                             pack2<T16>(v[6], v[7]));
            }
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int HD, typename T16>
cudaError_t launch_hd(const LaunchCtx& lc, const AttnArgs& a, const AttnMaps& maps, int layer, int B,
                      const AttnVarlen& vl) {
  const int PW = attn_tile_positions(a.H, a.G), PC = 2 * PW;
  const long long pairs = vl.cu ? vl.rows / PC + B : static_cast<long long>((a.S + PC - 1) / PC) * B;
  const int layer_rows = a.num_blocks * a.G * 16;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(pairs * a.G));
  cfg.blockDim = dim3(TC_THREADS);
  cfg.dynamicSmemBytes = ACfg<HD>::SMEM;
  cfg.stream = lc.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = lc.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, attn_prefill_tc_kernel<HD, T16>, maps.q, maps.k, maps.v, a, B, PW,
                            layer * layer_rows, maps.pool_rows, vl);
}

template <int HD, typename T16>
cudaError_t prepare_hd() {
  return cudaFuncSetAttribute(attn_prefill_tc_kernel<HD, T16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              ACfg<HD>::SMEM);
}

}  // namespace

cudaError_t prepare_attn_tc_kernels() {
  cudaError_t e = prepare_hd<64, bf16>();
  if (e == cudaSuccess) e = prepare_hd<64, f16>();
  if (e == cudaSuccess) e = prepare_hd<128, bf16>();
  if (e == cudaSuccess) e = prepare_hd<128, f16>();
  return e;
}

bool make_attn_maps(AttnMaps* maps, const void* q, long long rows, const void* kpool, const void* vpool,
                    long long pool_rows, int H, int G, int d, bool f16) {
  if (pool_rows > 0x7fffff00ll) return false;  // box rows are 32-bit coordinates
  maps->pool_rows = static_cast<int>(pool_rows);
  return make_tma_3d_16(&maps->q, q, d, H, rows, H / G, attn_tile_positions(H, G), f16) &&
         make_tma_2d_16(&maps->k, kpool, pool_rows, d, 16, f16) && make_tma_2d_16(&maps->v, vpool, pool_rows, d, 16, f16);
}

cudaError_t launch_attn_prefill_tc(const LaunchCtx& lc, const AttnArgs& a, const AttnMaps& maps, int layer, int B,
                                   const AttnVarlen* vl) {
  const AttnVarlen v = vl ? *vl : AttnVarlen{};
  if (a.H / a.G > 16 || B < 1 || a.S < 1) return cudaErrorInvalidValue;
  if (a.d == 64)
    return lc.f16 ? launch_hd<64, f16>(lc, a, maps, layer, B, v) : launch_hd<64, bf16>(lc, a, maps, layer, B, v);
  if (a.d == 128)
    return lc.f16 ? launch_hd<128, f16>(lc, a, maps, layer, B, v) : launch_hd<128, bf16>(lc, a, maps, layer, B, v);
  return cudaErrorInvalidValue;
}
