// Persistent decode step: one cooperative launch runs a whole decode step
// (embedding, L x [QKV, attention, O, gate/up, down], LM head, greedy token)
// for B <= 8 sequences, with one CTA per SM.
//
// Why: at decode, every projection of a small model moves a few MB, which the
// GPU streams in a microsecond or two, while a chain of ~5L+3 dependent
// kernel launches pays the kernel boundary (grid drain, launch, first loads)
// at every link. The weights do not depend on the activations and never wait: in
// every CTA a producer warp streams that CTA's share of every weight matrix of
// the step, in consumption order, through a shared-memory ring (2D TMA tensor
// copies completing on mbarriers), running ahead across layer and phase
// boundaries as far as the ring allows. The eight consumer warps take weight
// tiles from the ring and run the same mma.sync products, reductions and fused
// epilogues as the decode GEMV kernels.
//
// Exchange between CTAs: flagged words. Every value that one phase hands to the
// next (operands, q, the newest k and v, attention outputs, residual, norm
// partials) is stored as an 8-byte word {32 bits of data, flag}, the flag naming
// the launch and layer, and a reader polls the words that it needs until they
// carry the flag. A word is written and read whole, so no fence, barrier or
// counter stands between a producer's store and its consumers: one trip through
// L2 instead of the five of a grid barrier (release of the data, arrival, poll,
// data load, staging). Measured per step, grid barriers / flagged words: 135M
// width, 30 layers, 1 sequence 605 / 370 us; 0.5B width, 4 layers, 577 cached tokens
// 134 / 101 us; 8B width, 2 layers, fp16, 1151 cached tokens 222 / 190 us.
//   Data words: one-term mode, two neighbouring 16-bit values; two-term modes, the
// two terms of one value; fp32 for the residual and the norm partials.
//   Reuse: each buffer has one writing phase per layer, and a phase cannot begin
// writing layer l + 1 before every reader of layer l is done: its inputs depend,
// through the phases between, on the outputs of all of that buffer's readers (the
// newest k and v are awaited even where their position lies outside the cache).
//   Flags: epoch + layer + 1, the epoch advanced by L + 1 with every launch, so that
// what an earlier layer or launch left never matches. Before the 32-bit flags would
// wrap (after some 10^8 steps) the last CTA of a launch clears the buffers and starts the
// epoch anew; 0 is never a flag.
// The first layer's operand is the embedding, which every CTA computes itself.
//
// Work split: a projection phase is cut into items of 16 weight rows x all
// of K; item i of a phase goes to CTA (i + rot) mod grid, rot advancing by
// the phase's item count so that consecutive phases continue the round
// robin and every CTA streams about the same number of bytes per step. The
// producer and the consumers of a CTA walk the same item sequence. Attention
// items are the (split, kv head, sequence) triples of the split-KV decode
// attention, run by the consumer warps with the shared decode-attention code
// (last-arriver merge across splits); their cache blocks are requested before q
// has arrived.
//
// Waits (persist_wait.cuh): every wait has a limit of looks. A poll of words that runs
// out sets DEVERR_TIMEOUT and a grid-wide abort flag; after that no poll blocks, the
// weights stream to the end of the step as ever, the kernel runs to its end on garbage
// and the host sees the error bit. (Ring waits that gave up on the abort would release
// slots whose copies are in flight, and the producer would re-arm their barriers. To
// look at the full barrier as well before each copy costs 2 to 3 % at 8B and 32B width.) A
// ring wait of its own runs out only when a copy has not landed for a second or more;
// it is reported alike, and no wait of the CTA blocks after it. Before it exits, the
// producer waits (bounded) for its copies in flight.
#include <type_traits>

#include "attn_tile.cuh"
#include "persist_wait.cuh"

namespace {

constexpr int PCW = 8;                     // consumer warps (= DEC_WARPS)
constexpr int PTHREADS = (PCW + 1) * 32;   // + 1 producer warp
constexpr int KC = 512;                    // weight columns per ring stage (one 64-column chunk per warp)
constexpr int BOXC = PERSIST_BOX_COLS;     // columns per TMA box: a stage is 2 boxes of 16 rows x 256
constexpr int BOX_BYTES = 16 * BOXC * 2;   // 8 KB, rows dense (512 bytes)
constexpr int STAGE_BYTES = 2 * BOX_BYTES;
constexpr int RED_FLOATS = PCW * 16 * 9;   // cross-warp partials of one item: [warp][row][token + pad]
constexpr uint64_t PWAIT_NS = 2000000000ull;
// Operand vectors in flight per thread (staging).
constexpr int BATCH = 4;
constexpr int SMEM_LIMIT = 232448;         // 227 KB opt-in per CTA

static_assert(PCW == DEC_WARPS, "attention items run on the consumer warps");

// How the 16-bit operand terms of the projections enter the MMAs (proj_phase).
constexpr int TERMS_ONE = 0, TERMS_PAIRED = 1, TERMS_TWO = 2;

// Shared-memory layout. SM ("small", head_dim 128): the attention items stage
// one key block per warp (decode_smem1), so the weight ring gets the space a
// second stage would take: 9 ring stages instead of 5.
template <int HD, bool SM>
struct PLayout {
  static constexpr int ATTN = SM ? static_cast<int>(decode_smem1<HD>()) : static_cast<int>(decode_smem<HD>());
  static constexpr int RED = 2 * RED_FLOATS * 4;
  static constexpr int MISC = 256;  // rinv[8], abort flag
  static constexpr int STATIC_EST = 1024;  // static shared (the merge flag), with margin
  static constexpr int NS = (SMEM_LIMIT - ATTN - RED - MISC - STATIC_EST - 1024) / (STAGE_BYTES + 16);
  static constexpr int BARS = 2 * NS * 8;
  static constexpr int RING_OFF = 0;
  static constexpr int ATTN_OFF = RING_OFF + NS * STAGE_BYTES;
  static constexpr int RED_OFF = ATTN_OFF + ATTN;
  static constexpr int BAR_OFF = RED_OFF + RED;
  static constexpr int MISC_OFF = BAR_OFF + BARS;
  static constexpr int BYTES = MISC_OFF + MISC + 1024;  // + alignment slack
  static_assert(NS >= 3, "ring too small");
};

AXON_DEV void consumer_sync() { asm volatile("bar.sync 1, %0;" ::"n"(PCW * 32) : "memory"); }

AXON_DEV uint4 lds16(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}

AXON_DEV int first_item(int rot) {
  const int i = static_cast<int>(blockIdx.x) - rot;  // rot < gridDim.x
  return i < 0 ? i + static_cast<int>(gridDim.x) : i;
}

AXON_DEV int next_rot(int rot, const PersistPhase& ph) {
  rot += ph.rot_step;  // items mod grid
  return rot >= static_cast<int>(gridDim.x) ? rot - static_cast<int>(gridDim.x) : rot;
}

template <int HD, bool SM>
struct Ring {
  uint32_t base;  // shared address of stage 0
  uint32_t bars;  // full[NS] then empty[NS]
  AXON_DEV uint32_t full(int s) const { return bars + 8 * s; }
  AXON_DEV uint32_t empty(int s) const { return bars + 8 * (PLayout<HD, SM>::NS + s); }
};

// Word `i` of an exchange buffer.
AXON_DEV uint2* ll_word(uint4* base, int i) { return reinterpret_cast<uint2*>(base) + i; }
// Layout of a projection operand: the 2^SH vectors of one producing item at the
// start of STRIDE vectors (128-byte lines) of its own -- items of several CTAs
// in one line made every store fight the other writers and all the pollers for
// that line (36 norm partials in 3 lines, polled by 152 CTAs, took 2 us longer to
// arrive than the operand stored beside them). The residual producers (items of
// 16 values) put the item's norm partial behind its values.
template <bool LO> struct OpD {  // after O and down
  static constexpr int SH = LO ? 3 : 2, STRIDE = LO ? 16 : 8;
};

AXON_DEV uint32_t lo_halves(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x5410); }
AXON_DEV uint32_t hi_halves(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x7632); }
// The two 16-bit terms of a value in one word: its rounding (low half) and what
// the rounding lost.
template <typename T16>
AXON_DEV uint32_t two_terms(float v) { return pack2<T16>(v, v - to_f(from_f<T16>(v))); }

// Exchange of an attention item (attn_decode_item).
template <bool LO>
struct LLAttn {
  static constexpr bool on = true;
  const uint4* q;  // [B][H][d], both terms per word
  const uint4* k;  // [B][G][d], two values per word
  const uint4* v;
  uint4* o;  // [B][H][d], as the projections' operands
  uint32_t flag;
  PersistGrid* g;
  volatile int* s_abort;
  int* err;

  // A fragments of rows r (first terms) and r + 8 (second terms); off: element
  // offset of the row.
  template <int HD>
  AXON_DEV void load_q(uint32_t (&qa)[HD / 16][4], long long off, bool row, int qd) const {
    if (!row) {
#pragma unroll
      for (int kk = 0; kk < HD / 16; ++kk) qa[kk][0] = qa[kk][1] = qa[kk][2] = qa[kk][3] = 0u;
      return;
    }
    const int src = static_cast<int>(off >> 1) + qd;  // elements 2 qd, 2 qd + 1
#pragma unroll
    for (int k0 = 0; k0 < HD / 16; k0 += 4) {
      uint4 w[8];
      poll_vecs<8>(w, [&](int i) { return q + src + (k0 * 2 + i) * 4; }, flag, g, s_abort, err);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        qa[k0 + (i >> 1)][(i & 1) * 2] = lo_halves(w[i].x, w[i].z);
        qa[k0 + (i >> 1)][(i & 1) * 2 + 1] = hi_halves(w[i].x, w[i].z);
      }
    }
  }
  // The newest token's key and value, into row `tok` of a staged block [K | V] if
  // that is their place.
  template <int HD>
  AXON_DEV void patch(uint32_t stage, long long off, int tok, int lane, bool store) const {
    constexpr int VECS = HD / 4;  // four values per vector
    constexpr int N = 2 * VECS / 32;
    uint4 w[N];
    auto src = [&](int u) {
      const int t = lane + u * 32, kv = t / VECS;
      return (kv ? v : k) + static_cast<int>(off >> 2) + (t - kv * VECS);
    };
    poll_vecs<N>(w, src, flag, g, s_abort, err);
    if (!store) return;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int t = lane + u * 32, kv = t / VECS, i = t - kv * VECS;
      const uint32_t dst = swz<HD>(stage + kv * 16 * HD * 2, tok, i >> 1) + (i & 1) * 8;
      asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(dst), "r"(w[u].x), "r"(w[u].z) : "memory");
    }
  }
  // Output element `idx`; neighbouring lanes hold neighbouring elements.
  template <typename T16>
  AXON_DEV void store_o(long long idx, float val) const {
    if (LO) {
      st_word(ll_word(o, static_cast<int>(idx)), two_terms<T16>(val), flag);
    } else {
      const float other = __shfl_xor_sync(0xffffffffu, val, 1);
      if ((idx & 1) == 0) st_word(ll_word(o, static_cast<int>(idx >> 1)), pack2<T16>(val, other), flag);
    }
  }
};

// ----------------------------------------------------------------- producer
// Streams this CTA's items of one matrix (in the item order the consumers
// walk): per ring stage one or two TMA boxes of 16 rows x 256 columns, one
// instruction each; rows >= N and columns >= K arrive as zeros.
template <int HD, bool SM>
AXON_DEV void stream_matrix(const Ring<HD, SM>& R, const CUtensorMap* map, const PersistPhase& ph, int& rot, uint32_t& stage,
                            bool& stop, PersistGrid* g, volatile int* s_abort, int* err, int lane) {
  constexpr int NS = PLayout<HD, SM>::NS;
  const int n = ph.items, K = ph.K;
  const int i0 = first_item(rot);
  rot = next_rot(rot, ph);
  // Weights are read once per step: they should not evict the key/value
  // cache or the activations from L2.
  const uint64_t policy = createpolicy_evict_first();
#pragma unroll 1
  for (int i = i0; i < n && !stop; i += gridDim.x) {
#pragma unroll 1
    for (int k0 = 0; k0 < K && !stop; k0 += KC) {
      const int slot = static_cast<int>(stage % NS);
      int ok = 1;
      if (lane == 0) {
        if (stage >= static_cast<uint32_t>(NS))  // the consumers released this slot's previous use?
          ok = ring_wait(R.empty(slot), ((stage / NS) - 1) & 1u, g, s_abort, err) ? 1 : 0;
        if (ok) {
          const bool two = k0 + BOXC < K;
          mbar_arrive_expect_tx(R.full(slot), two ? STAGE_BYTES : BOX_BYTES);
          const uint32_t dst = R.base + slot * STAGE_BYTES;
          tma_load_2d_hint(dst, map, R.full(slot), k0, i * 16, policy);
          if (two) tma_load_2d_hint(dst + BOX_BYTES, map, R.full(slot), k0 + BOXC, i * 16, policy);
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) {
        stop = true;
        break;
      }
      ++stage;
    }
  }
}

// ----------------------------------------------------------------- consumers
struct CState {
  int rot = 0;
  uint32_t stage = 0;
  int buf = 0;
};

// One ring stage's fragments of a warp: its 64-column chunk of 16 weight rows
// (rows r, r + 8 x 16 columns), the token-r operand (x) and, with a second MMA
// set, its second term (y).
struct Frag {
  uint4 w0, w1, w2, w3, x0, x1, y0, y1;
};

// Wait for the ring slot of the next stage (columns k0 .. of K, operand columns
// from ka on in shared memory), copy the fragments to registers, release the slot.
template <int HD, bool SM, bool WANT_Y>
AXON_DEV bool load_stage(const Ring<HD, SM>& R, CState& cs, PersistGrid* g, volatile int* s_abort, int* err, int k_left,
                         int ka, int warp, int lane, int r, int q, bool tok_ok, uint32_t xrow, uint32_t yrow, Frag& f) {
  constexpr int NS = PLayout<HD, SM>::NS;
  const int sl = static_cast<int>(cs.stage % NS);
  ring_wait(R.full(sl), (cs.stage / NS) & 1u, g, s_abort, err);
  const bool on = warp * 64 < k_left;
  f.x0 = f.x1 = make_uint4(0, 0, 0, 0);
  if (WANT_Y) f.y0 = f.y1 = make_uint4(0, 0, 0, 0);
  if (on) {
    // chunk `warp` = box warp/4, columns (warp%4)*64 of its dense 512-byte rows
    const uint32_t rs = R.base + sl * STAGE_BYTES + (warp >> 2) * BOX_BYTES + (warp & 3) * 128 + q * 32;
    f.w0 = lds16(rs + r * (BOXC * 2));
    f.w1 = lds16(rs + r * (BOXC * 2) + 16);
    f.w2 = lds16(rs + (r + 8) * (BOXC * 2));
    f.w3 = lds16(rs + (r + 8) * (BOXC * 2) + 16);
    if (tok_ok) {
      const uint32_t off = (ka + warp * 64 + 16 * q) * 2;
      f.x0 = lds16(xrow + off);
      f.x1 = lds16(xrow + off + 16);
      if (WANT_Y) {
        f.y0 = lds16(yrow + off);
        f.y1 = lds16(yrow + off + 16);
      }
    }
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(R.empty(sl));  // fragments are in registers: slot free
  ++cs.stage;
  return on;
}

// Every lane issues every MMA (mma.sync is warp-collective); token slots >= B
// feed zeros. Two accumulators halve the dependent chain.
template <typename T16, bool WANT_Y>
AXON_DEV void mma_stage(float (&acc)[2][4], const Frag& f) {
  const uint32_t A0[8] = {f.w0.x, f.w0.y, f.w0.z, f.w0.w, f.w1.x, f.w1.y, f.w1.z, f.w1.w};
  const uint32_t A1[8] = {f.w2.x, f.w2.y, f.w2.z, f.w2.w, f.w3.x, f.w3.y, f.w3.z, f.w3.w};
  const uint32_t Bv[8] = {f.x0.x, f.x0.y, f.x0.z, f.x0.w, f.x1.x, f.x1.y, f.x1.z, f.x1.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t a[4] = {A0[2 * j], A1[2 * j], A0[2 * j + 1], A1[2 * j + 1]};
    const uint32_t bb[2] = {Bv[2 * j], Bv[2 * j + 1]};
    mma16816<T16>(acc[j & 1], a, bb);
  }
  if (WANT_Y) {
    const uint32_t Bl[8] = {f.y0.x, f.y0.y, f.y0.z, f.y0.w, f.y1.x, f.y1.y, f.y1.z, f.y1.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t a[4] = {A0[2 * j], A1[2 * j], A0[2 * j + 1], A1[2 * j + 1]};
      const uint32_t bb[2] = {Bl[2 * j], Bl[2 * j + 1]};
      mma16816<T16>(acc[j & 1], a, bb);
    }
  }
}

// What a projection phase reads and writes beside its weights.
struct PhaseIO {
  const uint4* act;  // operand words [B][K]; null: the embedding times gain_in
  int sh, stride;    // their layout (OpD; 30 / 0: dense)
  uint32_t f_in;     // their flag
  const float* gain_in;
  // residual kind: x in (null: the embedding) and out, the next operand and its partials
  const uint4* x_in;
  uint32_t f_x;
  uint4* x_out;
  uint4* a_out;
  const float* gain;
  // QKV
  const float* bias;
  uint4* q_out;
  uint4* k_out;
  uint4* v_out;
  void* k_cache;
  void* v_cache;
  // gate/up
  uint4* u_out;
  uint32_t f_out;
};

// One projection phase: items of 16 rows x K, products on mma.sync with the
// weight tile from the ring and the B <= 8 token rows of the operand; epilogue
// `kind`. All phases run this one body: a phase is a few hundred instructions
// executed once, and with a specialised copy per phase (111 KB of code) every
// phase missed the instruction cache (3900 line fetches per SM and step at 135M
// width; 530 us per step against 370 with this body, 66 KB).
//
// MODE (compile time, so that each kernel carries only its own inner loop):
//   TERMS_ONE    one 16-bit term per token (bf16 mode);
//   TERMS_PAIRED two terms, B <= 4: token slot 2b of the MMA's N dimension
//                holds token b's first term and slot 2b+1 its second, and
//                the reduction adds the two accumulator columns (no extra
//                MMA, no extra load);
//   TERMS_TWO    two terms, B = 5..8: a second MMA set takes the second
//                terms.
//
// Per item the consumer warps only run the products and the cross-warp sum;
// the item's 16 x B sums go to a shared buffer and the epilogues run in
// batches of up to 32 / B items, eight lanes per (item, token), so that their
// global reads overlap instead of stalling the weight stream item after item;
// the first batch's reads are requested before the products. The LM head, with no
// such reads, takes batches of up to 64 items, a thread per (item, token) (0.5B width, 3
// layers, 62 items per CTA, bf16, 8 sequences in batches of 4 / of 62: 166 / 153 us); its
// argmax keeps a per-CTA best key per token in shared memory and commits it
// once per phase.
template <int HD, bool SM, typename T16, int MODE>
AXON_DEV void proj_phase(const Ring<HD, SM>& R, CState& cs, const PersistArgs& A, int kind, const PersistPhase& ph, const PhaseIO& io,
                         float* red_base, float* rinv_s, unsigned long long* best_s, uint8_t* act_sm, PersistGrid* g,
                         volatile int* s_abort, int tid) {
  constexpr bool LO = MODE != TERMS_ONE;
  constexpr bool paired = MODE == TERMS_PAIRED;
  const bool NORM = kind != EPI_RESID;  // the accumulator takes the operand's norm scale
  const int warp = tid >> 5, lane = tid & 31, r = lane >> 2, q = lane & 3;
  const int B = A.B, G0 = static_cast<int>(gridDim.x);
  const int n = ph.items, K = ph.K;
  const int i_first = first_item(cs.rot);
  cs.rot = next_rot(cs.rot, ph);
  if (i_first >= n) return;
  // The phase's B x K operand goes to shared memory (both terms), rows padded by
  // 16 bytes so that the 8 token rows of a fragment load hit distinct banks, with
  // the norm partials behind it (the attention staging region is free during a
  // projection phase): once, for all items, where it fits beside the epilogue
  // buffer; else in pieces of KP columns for each item. KP < K only for wide MLPs
  // at head_dim 64, whose down projection has no more items than CTAs.
  const int parts = A.D >> 4, KP = ph.KP, pitch = KP * 2 + 16;
  float* ss_s = reinterpret_cast<float*>(act_sm + ph.ss_off);
  float* vbuf = reinterpret_cast<float*>(act_sm + ph.vb_off);

  // Epilogue task of this thread in a batch of items from i0 on (ph.cap of them at
  // most, so that every task has a thread): eight lanes per (item, token).
  const int i8 = tid & 7, t_slot = ((tid >> 3) * ph.inv_B) >> 16, t_b = (tid >> 3) - t_slot * B;
  struct Pre {
    uint4 x;
    float2 gn, cs;
    float b0, b1;
  } pre;
  // the task's global inputs
  auto load_in = [&](int n0) {
    const int b = t_b;
    if (kind == EPI_RESID) {
      if (io.x_in) {
        pre.x = ld_words(io.x_in + ((b * A.D + n0) >> 1) + i8);
      } else {
        int id = A.tokens[b];
        id = id < 0 || id >= A.V ? 0 : id;  // reported where the operand is formed
        const uint32_t e =
            *reinterpret_cast<const uint32_t*>(static_cast<const T16*>(A.embed) + static_cast<long long>(id) * A.D + n0 + 2 * i8);
        const T16* eh = reinterpret_cast<const T16*>(&e);
        pre.x = make_uint4(__float_as_uint(to_f(eh[0])), io.f_x, __float_as_uint(to_f(eh[1])), io.f_x);
      }
      pre.gn = *reinterpret_cast<const float2*>(io.gain + n0 + 2 * i8);
    }
    if (kind == EPI_QKV) {
      pre.b0 = io.bias ? io.bias[n0 + i8] : 0.f;
      pre.b1 = io.bias ? io.bias[n0 + 8 + i8] : 0.f;
      const int c = n0 & (HD - 1);  // within a head: every region is a multiple of d
      const int pos = min(max(A.ctx[b], 0), A.max_pos - 1);
      pre.cs = A.rope[static_cast<long long>(pos) * (HD / 2) + (c >> 4) * 8 + i8];
    }
  };
  if (kind == EPI_LOGITS && tid < B) best_s[tid] = 0ull;
  // Operand columns kp .. kp + kn (and, the first time, the norm partials) to
  // shared memory.
  auto stage = [&](int kp, int kn, bool first) {
    if (!io.act) {
      // embedding: operand E[token] * gain (both terms), sum of squares per 16 columns
#pragma unroll 1
      for (int it = tid; it < B * parts; it += PCW * 32) {
        const int b = it / parts, c = it - b * parts;
        int id = A.tokens[b];
        if (id < 0 || id >= A.V) {
          set_err(A.err, DEVERR_TOKEN);
          id = 0;
        }
        const T16* e = static_cast<const T16*>(A.embed) + static_cast<long long>(id) * A.D + c * 16;
        float s = 0.f;
#pragma unroll 1
        for (int k = 0; k < 16; k += 2) {
          const float v0 = to_f(e[k]), v1 = to_f(e[k + 1]);
          const float a0 = v0 * io.gain_in[c * 16 + k], a1 = v1 * io.gain_in[c * 16 + k + 1];
          s += v0 * v0;
          s += v1 * v1;
          *reinterpret_cast<uint32_t*>(act_sm + b * pitch + (c * 16 + k) * 2) = pack2<T16>(a0, a1);
          if (LO)
            *reinterpret_cast<uint32_t*>(act_sm + (B + b) * pitch + (c * 16 + k) * 2) =
                pack2<T16>(a0 - to_f(from_f<T16>(a0)), a1 - to_f(from_f<T16>(a1)));
        }
        ss_s[it] = s;
      }
      return;
    }
    // operand words, then norm partials: two words per vector
    constexpr int VE = LO ? 2 : 4;  // values per vector
    const int per_row = kn / VE, row_stride = K / VE;
    const int act0 = kp / VE;
    const int n_act = B * per_row, n_ss = NORM && first ? B * parts : 0;
    const uint32_t inv_row = kn == KP ? ph.inv_row : ph.inv_row_last;
    auto row_of = [&](int c) { return B == 1 ? 0 : static_cast<int>(__umulhi(static_cast<uint32_t>(c), inv_row)); };  // c / per_row
    const int total = n_act + n_ss;
    auto batch = [&](auto count, int c0) {
      constexpr int U = decltype(count)::value;
      uint4 w[U];
      poll_vecs<U>(
          w,
          [&](int u) -> const uint4* {
            const int c = c0 + u * PCW * 32;
            if (c < n_act) {
              const int row = row_of(c), v = act0 + row * row_stride + (c - row * per_row);
              return io.act + (v >> io.sh) * io.stride + (v & ((1 << io.sh) - 1));
            }
            return c < total ? io.act + (c - n_act) * OpD<LO>::STRIDE + (1 << OpD<LO>::SH) : nullptr;
          },
          io.f_in, g, s_abort, A.err);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int c = c0 + u * PCW * 32, row = row_of(c), piece = c - row * per_row;
        if (c < n_act) {
          if (LO) {
            *reinterpret_cast<uint32_t*>(act_sm + row * pitch + piece * 4) = lo_halves(w[u].x, w[u].z);
            *reinterpret_cast<uint32_t*>(act_sm + (B + row) * pitch + piece * 4) = hi_halves(w[u].x, w[u].z);
          } else {
            *reinterpret_cast<uint2*>(act_sm + row * pitch + piece * 8) = make_uint2(w[u].x, w[u].z);
          }
        } else if (c < total) {
          ss_s[c - n_act] = __uint_as_float(w[u].x);
        }
      }
    };
    // Vectors in flight per thread: as many as there are, up to BATCH (8 and 12 grew
    // the body past the instruction cache: 135M width 7.2 -> 7.6 and 9.1 ms for 16
    // steps and a prompt).
    int c0 = tid;
#pragma unroll 1
    for (; c0 - tid + 2 * PCW * 32 < total; c0 += BATCH * PCW * 32) batch(std::integral_constant<int, BATCH>{}, c0);
    if (c0 - tid + PCW * 32 < total)
      batch(std::integral_constant<int, 2>{}, c0);
    else if (c0 - tid < total)
      batch(std::integral_constant<int, 1>{}, c0);
  };
  // Token slot r of the MMA's N dimension holds token r, or (paired) the
  // first or second term of token r / 2.
  const int tb = paired ? (r >> 1) : r;
  const bool term_lo = paired && (r & 1);
  const bool tok_ok = tb < B;
  const int tsafe = tok_ok ? tb : 0;
  const uint32_t xrow = smem_u32(act_sm) + (term_lo ? B + tsafe : tsafe) * pitch;
  const uint32_t yrow = smem_u32(act_sm) + (B + tsafe) * pitch;
  constexpr bool want_y = LO && !paired;

  // Epilogues of the buffered items slot 0 .. nslots-1 (items i0 + slot * grid).
  auto flush = [&](int i0, int nslots) {
    consumer_sync();  // sums of the last item and the norm scales visible
    if (kind == EPI_LOGITS) {
      EpiArgs ep;
      memset(&ep, 0, sizeof(ep));
      ep.N = A.V;
      ep.logits = A.logits;
      ep.logits_stride = A.V;
#pragma unroll 1
      for (int t = tid; t < nslots * B; t += PCW * 32) {
        const int slot = t / B, b = t - slot * B;
        float v[16];
#pragma unroll
        for (int rr = 0; rr < 16; ++rr) v[rr] = vbuf[(slot * B + b) * 16 + rr];
        atomicMax(best_s + b, epi_logits16(ep, b, (i0 + slot * G0) * 16, v, rinv_s[b]));
      }
    } else {
      const bool ok = t_slot < nslots;
      const int b = t_b, n0 = (i0 + (ok ? t_slot * G0 : 0)) * 16;
      {
        const float* v = vbuf + (ok ? t_slot * B + b : 0) * 16;
        if (kind == EPI_RESID) {
          // elements n0 + 2 i8, + 1: x += v, next operand x * gain, x^2
          float x0 = 0.f, x1 = 0.f;
          const int e0 = b * A.D + n0 + 2 * i8;
          if (ok) {
            uint4 xw[1] = {pre.x};
            if (xw[0].y != io.f_x || xw[0].w != io.f_x)
              poll_vecs<1>(xw, [&](int) { return io.x_in + (e0 >> 1); }, io.f_x, g, s_abort, A.err);
            x0 = __uint_as_float(xw[0].x) + v[2 * i8];
            x1 = __uint_as_float(xw[0].z) + v[2 * i8 + 1];
            const float a0 = x0 * pre.gn.x, a1 = x1 * pre.gn.y;
            uint4* dst = io.a_out + (e0 >> 4) * OpD<LO>::STRIDE;
            if (LO)
              st_words(dst + i8, two_terms<T16>(a0), two_terms<T16>(a1), io.f_out);
            else
              st_word(ll_word(dst, i8), pack2<T16>(a0, a1), io.f_out);
          }
          float sq = x0 * x0 + x1 * x1;
          sq += __shfl_xor_sync(0xffffffffu, sq, 1);
          sq += __shfl_xor_sync(0xffffffffu, sq, 2);
          sq += __shfl_xor_sync(0xffffffffu, sq, 4);
          if (ok) {
            if (i8 == 0)
              st_words(io.a_out + (e0 >> 4) * OpD<LO>::STRIDE + (1 << OpD<LO>::SH), __float_as_uint(sq), 0u, io.f_out);
            st_words(io.x_out + (e0 >> 1), __float_as_uint(x0), __float_as_uint(x1), io.f_out);
          }
        } else if (kind == EPI_SWIGLU) {
          const float rs = rinv_s[b];
          const float u = gate_act(v[i8] * rs, A.act == ACT_GELU_TANH) * (v[8 + i8] * rs);
          const int e = b * A.F + (n0 >> 1) + i8;
          if (LO) {
            if (ok) st_word(ll_word(io.u_out, e), two_terms<T16>(u), io.f_out);
          } else {
            const float other = __shfl_xor_sync(0xffffffffu, u, 1);
            if (ok && (i8 & 1) == 0) st_word(ll_word(io.u_out, e >> 1), pack2<T16>(u, other), io.f_out);
          }
        } else {
          // QKV: dims j and j + d/2 of one head (rotation partners)
          const int Hd = A.H * HD, Gd = A.G * HD;
          constexpr int half = HD / 2;
          const int region = n0 < Hd ? 0 : (n0 < Hd + Gd ? 1 : 2);
          const int base = region == 0 ? 0 : (region == 1 ? Hd : Hd + Gd);
          const int head = (n0 - base) / HD, j = (((n0 - base) & (HD - 1)) >> 4) * 8 + i8;
          const float rs = rinv_s[b];
          float lo = v[i8] * rs + pre.b0, hi = v[8 + i8] * rs + pre.b1;
          if (region < 2) {
            const float t1 = lo, t2 = hi;
            lo = t1 * pre.cs.x - t2 * pre.cs.y;
            hi = t2 * pre.cs.x + t1 * pre.cs.y;
          }
          // neighbouring dims share the words and cache stores of k and v: the even
          // lane takes the pair of the lower half, the odd lane that of the upper
          const bool odd = i8 & 1;
          const float got = __shfl_xor_sync(0xffffffffu, odd ? lo : hi, 1);
          if (ok && region == 0) {
            const int dst = (b * A.H + head) * HD + j;
            st_word(ll_word(io.q_out, dst), two_terms<T16>(lo), io.f_out);
            st_word(ll_word(io.q_out, dst + half), two_terms<T16>(hi), io.f_out);
          } else if (ok) {
            const uint32_t two = odd ? pack2<T16>(got, hi) : pack2<T16>(lo, got);
            const int dim = odd ? half + j - 1 : j;
            st_word(ll_word(region == 1 ? io.k_out : io.v_out, ((b * A.G + head) * HD + dim) >> 1), two, io.f_out);
            EpiArgs ke;
            ke.max_pos = A.max_pos;
            ke.block_table = A.block_table;
            ke.bt_stride = ke.blocks_per_seq = A.blocks_per_seq;
            ke.num_blocks = A.num_blocks;
            ke.G = A.G;
            ke.d = HD;
            ke.err = A.err;
            const long long off = kv_offset(ke, b, A.ctx[b], head);
            if (off >= 0)
              *reinterpret_cast<uint32_t*>(static_cast<T16*>(region == 1 ? io.k_cache : io.v_cache) + off + dim) = two;
          }
        }
      }
    }
  };

  int slot = 0, i0 = i_first;
#pragma unroll 1
  for (int i = i_first; i < n; i += G0) {
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    // a batch's first item: its tasks' inputs, requested ahead of the products
    if (slot == 0 && t_slot < ph.cap && i0 + t_slot * G0 < n) load_in((i0 + t_slot * G0) * 16);
#pragma unroll 1
    for (int kp = 0; kp < K; kp += KP) {
      const int kn = min(KP, K - kp);
      if (i == i_first || KP < K) {
        consumer_sync();  // the region's previous use is over
        stage(kp, kn, i == i_first && kp == 0);
        consumer_sync();
      }
      // two stages at a time: their loads overlap
#pragma unroll 1
      for (int k = 0; k < kn; k += 2 * KC) {
        Frag f0, f1;
        const bool on0 = load_stage<HD, SM, want_y>(R, cs, g, s_abort, A.err, kn - k, k, warp, lane, r, q, tok_ok, xrow,
                                                    yrow, f0);
        bool on1 = false;
        if (k + KC < kn)
          on1 = load_stage<HD, SM, want_y>(R, cs, g, s_abort, A.err, kn - k - KC, k + KC, warp, lane, r, q, tok_ok, xrow,
                                           yrow, f1);
        if (on0) mma_stage<T16, want_y>(acc, f0);
        if (on1) mma_stage<T16, want_y>(acc, f1);
      }
    }
    if (NORM && i == i_first && PCW - 1 - warp < B) {
      // norm scale of token b, by the warps that hold the fewest K chunks
      const int b = PCW - 1 - warp;
      float rp = 0.f;
#pragma unroll 1
      for (int j = lane; j < parts; j += 32) rp += ss_s[b * parts + j];
      rp = warp_sum(rp);
      if (lane == 0) rinv_s[b] = 1.0f / sqrtf(rp * A.inv_D + A.eps);
    }
    // Accumulator of lane (r, q): rows r, r+8 x token slots 2q, 2q+1.
    float* red = red_base + cs.buf * RED_FLOATS;
    if (paired) {  // slots 2q, 2q+1 = the two terms of token q
      red[(warp * 16 + r) * 9 + q] = (acc[0][0] + acc[1][0]) + (acc[0][1] + acc[1][1]);
      red[(warp * 16 + r + 8) * 9 + q] = (acc[0][2] + acc[1][2]) + (acc[0][3] + acc[1][3]);
    } else {
      red[(warp * 16 + r) * 9 + 2 * q] = acc[0][0] + acc[1][0];
      red[(warp * 16 + r) * 9 + 2 * q + 1] = acc[0][1] + acc[1][1];
      red[(warp * 16 + r + 8) * 9 + 2 * q] = acc[0][2] + acc[1][2];
      red[(warp * 16 + r + 8) * 9 + 2 * q + 1] = acc[0][3] + acc[1][3];
    }
    consumer_sync();
    if (tid < B * 16) {
      const int b = tid >> 4, rr = tid & 15;
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < PCW; ++w) sum += red[(w * 16 + rr) * 9 + b];
      vbuf[(slot * B + b) * 16 + rr] = sum;
    }
    cs.buf ^= 1;
    if (++slot == ph.cap || i + G0 >= n) {
      flush(i0, slot);
      if (i + G0 < n) consumer_sync();  // buffer free again
      i0 = i + G0;
      slot = 0;
    }
  }
  if (kind == EPI_LOGITS) consumer_sync();
  if (kind == EPI_LOGITS && tid < B) argmax_commit(A.keys + tid, best_s[tid]);
}

template <int HD, bool SM, typename T16, int MODE>
__global__ void __launch_bounds__(PTHREADS, 1) persist_decode_kernel(PersistArgs A) {
  constexpr bool LO = MODE != TERMS_ONE;  // fp16 mode carries the split operand
  constexpr int NS = PLayout<HD, SM>::NS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Ring<HD, SM> R;
  R.base = smem_u32(sm + PLayout<HD, SM>::RING_OFF);
  R.bars = smem_u32(sm + PLayout<HD, SM>::BAR_OFF);
  uint8_t* attn_sm = sm + PLayout<HD, SM>::ATTN_OFF;
  float* red_base = reinterpret_cast<float*>(sm + PLayout<HD, SM>::RED_OFF);
  float* rinv_s = reinterpret_cast<float*>(sm + PLayout<HD, SM>::MISC_OFF);
  volatile int* s_abort = reinterpret_cast<volatile int*>(sm + PLayout<HD, SM>::MISC_OFF + 64);
  unsigned long long* best_s = reinterpret_cast<unsigned long long*>(sm + PLayout<HD, SM>::MISC_OFF + 128);
  PersistGrid* g = A.grid;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(R.full(s), 1);
      mbar_init(R.empty(s), PCW);
    }
    *s_abort = 0;
    fence_mbar_init();
  }
  __syncthreads();

  if (warp == PCW) {
    // ------------------------------------------------------------ producer
    int rot = 0;
    uint32_t stage = 0;
    bool stop = false;
#pragma unroll 1
    for (int i = 0; i <= 4 * A.L && !stop; ++i) {
      stream_matrix<HD, SM>(R, A.wmaps + i, A.ph[i == 4 * A.L ? 4 : i & 3], rot, stage, stop, g, s_abort, A.err, lane);
    }
    // Copies still in flight must land before the CTA's shared memory goes
    // away: wait for the last use of every slot.
    if (lane == 0) {
      for (uint32_t j = stage > static_cast<uint32_t>(NS) ? stage - NS : 0u; j < stage; ++j) {
        if (!mbar_try_wait(R.full(static_cast<int>(j % NS)), (j / NS) & 1u)) {
          const uint64_t t0 = global_ns();
          while (!mbar_try_wait(R.full(static_cast<int>(j % NS)), (j / NS) & 1u))
            if (global_ns() - t0 > PWAIT_NS) {
              set_err(A.err, DEVERR_TIMEOUT);
              break;
            }
        }
      }
    }
    return;
  }

  // -------------------------------------------------------------- consumers
  const int tid = threadIdx.x;
  CState cs;
  const int B = A.B;
  const uint32_t epoch = ld_volatile(&g->epoch);

  PhaseIO io;
  memset(&io, 0, sizeof(io));
  io.q_out = A.ll_q;
  io.k_out = A.ll_k;
  io.v_out = A.ll_v;
  io.u_out = A.ll_u;
#pragma unroll 1
  for (int step = 0; step <= 4 * A.L; ++step) {
    const int l = step >> 2;
    const bool head = step == 4 * A.L;
    const uint32_t flag = epoch + 1u + static_cast<uint32_t>(l);
    const PersistLayer* w = A.layers + l;  // (the head reads none)
    int kind;
    io.f_out = io.f_in = flag;
    if (head || (step & 3) == 0) {
      // QKV + bias + RoPE + KV store, or final norm + LM head + argmax
      kind = head ? EPI_LOGITS : EPI_QKV;
      io.act = l ? A.ll_ad : nullptr;
      io.gain_in = head ? A.gf : w->g1;
      io.sh = OpD<LO>::SH;
      io.stride = OpD<LO>::STRIDE;
      io.f_in = flag - 1u;
      if (!head) {
        io.bias = w->bqkv;
        io.k_cache = w->kc;
        io.v_cache = w->vc;
      }
    } else if ((step & 3) == 2) {
      // gate/up + SwiGLU
      kind = EPI_SWIGLU;
      io.act = A.ll_ao;
      io.sh = OpD<LO>::SH;
      io.stride = OpD<LO>::STRIDE;
    } else {
      kind = EPI_RESID;
      if ((step & 3) == 1) {
        // split-KV attention, then the O projection + residual; next operand x * g2
        AttnArgs p;
        memset(&p, 0, sizeof(p));
        p.k = w->kc;
        p.v = w->vc;
        p.ctx = A.ctx;
        p.block_table = A.block_table;
        p.bt_stride = A.blocks_per_seq;
        p.blocks_per_seq = A.blocks_per_seq;
        p.num_blocks = A.num_blocks;
        p.H = A.H;
        p.G = A.G;
        p.d = A.d;
        p.S = 1;
        p.splits = A.splits;
        p.window = A.window;
        p.scale_log2 = A.scale_log2;
        p.part = A.attn_part;
        p.counter = A.attn_cnt;
        p.err = A.err;
        const LLAttn<LO> ll{A.ll_q, A.ll_k, A.ll_v, A.ll_o, flag, g, s_abort, A.err};
        const int items = A.splits * A.G * B;
#pragma unroll 1
        for (int it = blockIdx.x; it < items; it += gridDim.x) {
          consumer_sync();  // the staging memory is free
          const int s = it % A.splits, gg = (it / A.splits) % A.G, b = it / (A.splits * A.G);
          attn_decode_item<HD, T16, true, 1, SM ? 1 : 2>(p, s, gg, b, attn_sm, tid, ll);
        }
        io.act = A.ll_o;
        io.sh = 30;
        io.stride = 0;
        io.x_in = l ? A.ll_xd : nullptr;
        io.f_x = flag - 1u;
        io.x_out = A.ll_xo;
        io.a_out = A.ll_ao;
        io.gain = w->g2;
      } else {
        // down projection + residual; next operand x * (next norm's gain)
        io.act = A.ll_u;
        io.sh = 30;
        io.stride = 0;
        io.x_in = A.ll_xo;
        io.f_x = flag;
        io.x_out = A.ll_xd;
        io.a_out = A.ll_ad;
        io.gain = w->gnext;
      }
    }
    proj_phase<HD, SM, T16, MODE>(R, cs, A, kind, A.ph[head ? 4 : step & 3], io, red_base, rinv_s, best_s, attn_sm, g, s_abort, tid);
  }
  // Last CTA out: greedy token, context advance, keys cleared for the next step,
  // epoch of the next launch.
  consumer_sync();
  if (tid == 0 && atom_add_acq_rel_gpu(reinterpret_cast<int*>(&g->exit), 1) == static_cast<int>(gridDim.x) - 1) {
#pragma unroll 1
    for (int b = 0; b < B; ++b) {
      const unsigned long long k = atomicExch(A.keys + b, 0ull);
      if (A.next) A.next[b] = static_cast<int>(0xffffffffu - static_cast<uint32_t>(k & 0xffffffffull));
      A.ctx[b] += 1;
    }
    uint32_t next = epoch + static_cast<uint32_t>(A.L) + 1u;
    if (next > 0xfffffffeu - static_cast<uint32_t>(A.L)) {  // its last flag would be next + L + 1
#pragma unroll 1
      for (unsigned i = 0; i < A.ll_vecs; ++i) A.ll_ao[i] = make_uint4(0u, 0u, 0u, 0u);
      next = 0u;
    }
    g->abort = 0u;
    g->exit = 0u;
    g->epoch = next;
  }
}

// The phases' constants for this launch.
template <int HD, bool SM, int MODE>
bool plan_phases(PersistArgs& a, int nctas) {
  constexpr bool LO = MODE != TERMS_ONE;
  constexpr int ATTN = PLayout<HD, SM>::ATTN, VE = LO ? 2 : 4;
  const int N[5] = {a.Nqkv, a.D, 2 * a.F, a.D, a.V}, K[5] = {a.D, a.H * a.d, a.D, a.F, a.D};
  const int rows = LO ? 2 * a.B : a.B;
  for (int i = 0; i < 5; ++i) {
    PersistPhase& p = a.ph[i];
    p.K = K[i];
    p.items = (N[i] + 15) / 16;
    p.rot_step = p.items % nctas;
    const int ss_bytes = i == 1 || i == 3 ? 0 : a.B * (a.D / 16) * 4;  // norm partials (a multiple of 16 bytes)
    const int room = ATTN - 8 * a.B * 64 - ss_bytes;
    p.KP = rows * (K[i] * 2 + 16) <= room ? K[i] : (room / rows - 16) / (4 * KC) * (2 * KC);
    if (p.KP < 2 * KC && p.KP < K[i]) return false;
    p.ss_off = rows * (p.KP * 2 + 16);
    p.vb_off = p.ss_off + ss_bytes;
    p.cap = (ATTN - p.vb_off) / (a.B * 64);
    const int most = i == 4 ? 64 : PCW * 4 / a.B;
    if (p.cap > most) p.cap = most;
    p.inv_row = 0xffffffffu / static_cast<uint32_t>(p.KP / VE) + 1u;
    const int last = K[i] % p.KP ? K[i] % p.KP : p.KP;
    p.inv_row_last = 0xffffffffu / static_cast<uint32_t>(last / VE) + 1u;
    p.inv_B = 65536u / static_cast<uint32_t>(a.B) + 1u;
    if (p.cap < 1) return false;
  }
  return true;
}

template <int HD, bool SM, typename T16, int MODE>
cudaError_t launch_t(const PersistArgs& args, int nctas, cudaStream_t st) {
  PersistArgs a = args;
  if (!plan_phases<HD, SM, MODE>(a, nctas)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nctas);
  cfg.blockDim = dim3(PTHREADS);
  cfg.dynamicSmemBytes = PLayout<HD, SM>::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, persist_decode_kernel<HD, SM, T16, MODE>, a);
}

template <int HD, bool SM, typename T16, int MODE>
cudaError_t prepare_one(int* per_sm) {
  cudaError_t e = cudaFuncSetAttribute(persist_decode_kernel<HD, SM, T16, MODE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, PLayout<HD, SM>::BYTES);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, persist_decode_kernel<HD, SM, T16, MODE>, PTHREADS,
                                                       PLayout<HD, SM>::BYTES);
}

// The kernels a (head_dim, type) launches: bf16 one term; fp16 paired
// (B <= 4) and two sets (B > 4). Head_dim 64 takes the layout whose
// attention region stages two key blocks per warp, head_dim 128 the small
// one (measured at head_dim 128: the two-stage layout's 5-stage ring lost to
// the launch chain at 8B width, B = 8, bf16, 4.19 against 3.59 ms per step,
// and tied it at 32B width, B = 1, fp16). Resident CTAs per SM = the smaller
// count.
template <int HD, typename T16>
cudaError_t prepare_t(int* per_sm) {
  constexpr bool SMALL = HD == 128;
  if constexpr (!std::is_same<T16, f16>::value) {
    return prepare_one<HD, SMALL, T16, TERMS_ONE>(per_sm);
  } else {
    int a = 0, b = 0;
    cudaError_t e = prepare_one<HD, SMALL, T16, TERMS_PAIRED>(&a);
    if (e == cudaSuccess) e = prepare_one<HD, SMALL, T16, TERMS_TWO>(&b);
    *per_sm = a < b ? a : b;
    return e;
  }
}

template <int HD, typename T16>
cudaError_t launch_mode(const PersistArgs& a, int nctas, cudaStream_t st) {
  constexpr bool SMALL = HD == 128;
  if constexpr (!std::is_same<T16, f16>::value)
    return launch_t<HD, SMALL, T16, TERMS_ONE>(a, nctas, st);
  else
    return a.B <= 4 ? launch_t<HD, SMALL, T16, TERMS_PAIRED>(a, nctas, st)
                    : launch_t<HD, SMALL, T16, TERMS_TWO>(a, nctas, st);
}

// Whether B activation rows (two terms each in fp16 mode) of K columns stage
// in an attention region of `attn` bytes next to the epilogue buffer.
bool stages_in(int attn, bool use_f16, int B, int K) {
  const int rows = use_f16 ? 2 * B : B;
  return static_cast<long long>(rows) * (K * 2 + 16) <= attn - 8 * B * 16 * 4;
}

}  // namespace

int persist_ctas_per_sm(int head_dim, bool use_f16) {
  int n = 0;
  cudaError_t e;
  if (head_dim == 64)
    e = use_f16 ? prepare_t<64, f16>(&n) : prepare_t<64, bf16>(&n);
  else if (head_dim == 128)
    e = use_f16 ? prepare_t<128, f16>(&n) : prepare_t<128, bf16>(&n);
  else
    return 0;
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

bool persist_fits(int head_dim, bool use_f16, int B, int D, int kmax) {
  if (B < 1 || B > PERSIST_MAX_B) return false;
  // The normed operand of QKV, gate/up and the LM head (K = D) must stage in
  // shared memory next to the epilogue buffer; at head_dim 128 (small layout)
  // every projection's operand (K up to kmax) must.
  // The norm partials (D / 16 floats per token) lie behind a K = D operand.
  const int attn = head_dim == 64 ? PLayout<64, false>::ATTN : PLayout<128, true>::ATTN;
  if (!stages_in(attn - B * (D >> 4) * 4, use_f16, B, D)) return false;
  // Head_dim 64 stages a wider operand (the down projection's) in pieces, up to
  // twice the room (0.5B width, 4 layers, fp16, persistent / launch chain: 5
  // sequences 163 / 175 us, 8 sequences 200 / 180).
  if (head_dim == 64) return stages_in(2 * attn, use_f16, B, kmax);
  if (head_dim == 128) return stages_in(PLayout<128, true>::ATTN, use_f16, B, kmax);
  return false;
}

cudaError_t launch_persist_decode(const PersistArgs& a, int head_dim, bool use_f16, int nctas, cudaStream_t st) {
  if (a.B < 1 || a.B > PERSIST_MAX_B || (a.D & 63) || (a.F & 63) || ((a.H * a.d) & 63)) return cudaErrorInvalidValue;
  if (head_dim == 64) return use_f16 ? launch_mode<64, f16>(a, nctas, st) : launch_mode<64, bf16>(a, nctas, st);
  if (head_dim == 128) return use_f16 ? launch_mode<128, f16>(a, nctas, st) : launch_mode<128, bf16>(a, nctas, st);
  return cudaErrorInvalidValue;
}
