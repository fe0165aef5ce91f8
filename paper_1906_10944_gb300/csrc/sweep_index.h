// Index arithmetic of the band sweeps (sweep.cu) that decides which shared
// memory they read: plain integers, so that a host program can enumerate it.
#pragma once

#ifdef __CUDACC__
#define GENEO_HD __host__ __device__ __forceinline__
#else
#define GENEO_HD inline
#endif

namespace geneo {

// Bytes between the start of the dynamic shared memory and the row slots: mbarriers
// and padding.  The tensor-core sweep loads before it masks, also blocks left of a
// row's band (below), so the entries before the first slot that it loads lie here.
// (Skipping those blocks cost the loop 1.5 %: 2.97 for 2.92 ms at 512 bands of order
// 6000, half width 360, 8 columns.)
constexpr int kSlotLead = 512;
GENEO_HD constexpr int slot_lead(int C) { return C > 1 ? 1792 : kSlotLead; }

// row blocks before a block that its owner reads: those the band reaches, and
// all that the other blocks of the cluster solve between two of its own (so
// that every value sent is waited for)
GENEO_HD int reach_blocks(int w, int B, int C) {
  const int r = (w + B - 1) / B;
  return r > C - 1 ? r : C - 1;
}
// blocks of B rows in the ring of solved rows (and of partial sums): the
// reach, and the slots of block k itself and of the C - 1 blocks that may
// arrive before the owner of k reads on (rounded up to 32 rows, the columns
// the multiply-add sweep takes at a time)
GENEO_HD int ring_blocks(int w, int B, int C) {
  const int r = reach_blocks(w, B, C) + C, m = B < 32 ? 32 / B : 1;
  return m > 1 ? (r + 2 * m - 1) / m * m : r;
}
// The forward sweep's first block for block kk of a matrix of half width w: the
// first in band, and no later than the first that arrived since the owner's last
// block.  A class is launched with the C of its widest matrix, so for the others
// that may lie left of the band: up to (C - 1) B - w columns, whose products are
// with zeros.
GENEO_HD int forward_first(int kk, int w, int B, int C) {
  const int j = kk * B > w ? (kk * B - w) / B : 0, a = kk - C + 1;
  const int m = j < a ? j : a;
  return m > 0 ? m : 0;
}
// element offset, from the start of the row slot, of entry (row r of block kk,
// column c) whose row is row r mod SR of the slot
GENEO_HD int slot_offset(int kk, int r, int c, int w, int ld, int B, int SR) {
  return (r % SR) * ld + w - kk * B - r + c;
}

}  // namespace geneo
