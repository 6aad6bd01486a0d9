// Barriers of the flow decoder's cluster step whose phases more than one warp or CTA has to agree on: the K/V ring and the hand-over of a stage's rows.
// Plain C++, so that the host can walk them as well.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define DC_HD __host__ __device__ __forceinline__
#else
#define DC_HD inline
#endif

namespace dc {

constexpr uint32_t CLU_KVS = 4;   // slots

// Items of one attention job of n key blocks, in the order in which the products consume them: K0 K1 K2 V0 K3 V1 ... V(n-1).
DC_HD int clu_item_k(int b) { return b < 2 ? b : 2 * b - 2; }
DC_HD int clu_item_v(int b, int n) { return b + 2 < n ? 2 * b + 3 : 2 * n - (n - b); }
DC_HD void clu_item(int i, int n, bool* is_v, int* b) {
  if (i == 2 * n - 1) { *is_v = true; *b = n - 1; }
  else if (n >= 2 && i == 2 * n - 2) { *is_v = true; *b = n - 2; }
  else if (i < 2) { *is_v = false; *b = i; }
  else if (i & 1) { *is_v = true; *b = (i - 3) >> 1; }
  else { *is_v = false; *b = (i >> 1) + 1; }
}

// A wait for a phase of a barrier, told by its parity, passes at once while the phase BEFORE it is still open.  So the rule for every ring: who waits for a
// phase has waited for the one before, or stands behind a barrier that implies it.  A slot of this ring holds K and V blocks in turn, the scores' warp waits
// for the K blocks only and the output's warp for the V blocks only, and neither knows what the other has waited for: from four key blocks on V(n-2) follows
// K(n-2) into its slot.  Hence two "full" barriers per slot, one of each kind: every phase of one is waited for by one and the same warp.
DC_HD uint32_t clu_kv_full(bool is_v, uint32_t slot) { return (is_v ? CLU_KVS : 0u) + slot; }
struct CluKvPhases {              // a waiting warp's count of its barriers' phases, one bit each
  uint32_t bits = 0;
  DC_HD uint32_t next(uint32_t slot) {
    const uint32_t parity = (bits >> slot) & 1u;
    bits ^= 1u << slot;
    return parity;
  }
};

// The barrier on which the CTAs of a cluster signal that their rows of the n-th stage handed over in bulk are there, and its phase.  Two in turn: a CTA may
// signal stage n + 1 while another still waits for a signal of stage n, but none stage n + 2, because every CTA has passed a cluster barrier behind its wait.
DC_HD uint32_t clu_hand(uint32_t n) { return n & 1u; }
DC_HD uint32_t clu_hand_parity(uint32_t n) { return (n >> 1) & 1u; }

}  // namespace dc
