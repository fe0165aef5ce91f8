// Index arithmetic of the band sweeps (sweep.cu) that decides which shared
// memory they read: plain integers, so that a host program can enumerate it.
#pragma once

#ifdef __CUDACC__
#define GENEO_HD __host__ __device__ __forceinline__
#else
#define GENEO_HD inline
#endif

namespace geneo {

// Bytes between the start of the dynamic shared memory and the row slots
// (mbarriers and padding).  The tensor-core sweep loads before it masks: the
// entries left of a row's band that it loads from the first slot end here.
constexpr int kSlotLead = 512;

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
// The forward sweep's first block for block kk (rows kb = kk B ..) of a matrix
// of half width w: the first in band, and no later than the first that arrived
// since the owner's last block.  A class is launched with the C of its widest
// matrix, so for the others that may lie left of the band: such a block is
// waited for and not read.
GENEO_HD int forward_first(int kk, int w, int B, int C) {
  const int j = (kk * B - w + B) / B - 1, a = kk - C + 1;
  const int m = j < a ? j : a;
  return m > 0 ? m : 0;
}
// whether a column of block j lies in the band of a row of block kk > j
GENEO_HD bool block_in_band(int kk, int j, int w, int B) { return j * B + B > kk * B - w; }
// element offset, from the start of the row slot, of entry (row r of block kk,
// column c) whose row is row r mod SR of the slot
GENEO_HD int slot_offset(int kk, int r, int c, int w, int ld, int B, int SR) {
  return (r % SR) * ld + w - kk * B - r + c;
}

}  // namespace geneo
