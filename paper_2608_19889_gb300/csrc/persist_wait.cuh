// Bounded waits of the persistent decode step (k_persist.cu): ring mbarriers and
// polls of flagged words.
#pragma once

#include "kernels.h"

namespace {

// Looks until a wait gives up: a poll is a round trip to L2 (4M of them take
// seconds), a look at an mbarrier some tens of cycles or more.
constexpr uint32_t POLL_LOOKS = 1u << 22, RING_LOOKS = 1u << 26;

AXON_DEV unsigned ld_volatile(const unsigned* p) { return *reinterpret_cast<const volatile unsigned*>(p); }

// Every wait of the step is bounded by its looks: the one that runs out sets the
// error bit and the grid-wide abort flag, which the others see every few
// thousand looks. (Counting looks instead of reading the clock keeps the waits
// short: the code of a layer should fit the instruction cache.) s_abort, the CTA's
// own flag: ABORT_POLLS ends its polls of words; its ring goes on as ever, since
// copies land whatever the words hold, and no slot is released or armed out of
// turn. ABORT_RING: a ring wait of the CTA itself ran out, and none blocks any more.
constexpr int ABORT_POLLS = 1, ABORT_RING = 2;

AXON_DEV void wait_tick(uint32_t looks, uint32_t limit, int bits, PersistGrid* g, volatile int* s_abort, int* err) {
  if ((looks & 4095u) == 0) {
    if (looks >= limit) {
      set_err(err, DEVERR_TIMEOUT);
      atomicExch(&g->abort, 1u);
      *s_abort = bits;
    }
    if (!*s_abort && ld_volatile(&g->abort)) *s_abort = ABORT_POLLS;
  }
}

// Wait for phase `parity` of a ring mbarrier.
AXON_DEV bool ring_wait(uint32_t bar, uint32_t parity, PersistGrid* g, volatile int* s_abort, int* err) {
#pragma unroll 1
  for (uint32_t looks = 0; !mbar_try_wait(bar, parity);) {
    if (*s_abort & ABORT_RING) return false;
    wait_tick(++looks, RING_LOOKS, ABORT_POLLS | ABORT_RING, g, s_abort, err);
  }
  return true;
}

AXON_DEV uint4 ld_words(const uint4* p) {
  uint4 v;
  asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p)
               : "memory");
  return v;
}
AXON_DEV void st_words(uint4* p, uint32_t d0, uint32_t d1, uint32_t flag) {
  asm volatile("st.volatile.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(d0), "r"(flag), "r"(d1), "r"(flag)
               : "memory");
}
AXON_DEV void st_word(uint2* p, uint32_t d, uint32_t flag) {
  asm volatile("st.volatile.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(d), "r"(flag) : "memory");
}

// N vectors of two words each, looked at together until all carry `flag`.
template <int N, typename F>
AXON_DEV void poll_vecs(uint4 (&w)[N], F src, uint32_t flag, PersistGrid* g, volatile int* s_abort, int* err,
                        uint32_t limit = POLL_LOOKS) {
  uint32_t looks = 0;
#pragma unroll 1
  for (;;) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const uint4* p = src(i);
      w[i] = p ? ld_words(p) : make_uint4(0u, flag, 0u, flag);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) ok = ok && w[i].y == flag && w[i].w == flag;
    if (ok || *s_abort) return;
    wait_tick(++looks, limit, ABORT_POLLS, g, s_abort, err);
  }
}

}  // namespace
