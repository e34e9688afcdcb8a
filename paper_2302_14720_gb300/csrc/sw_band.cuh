// sw_band.cuh -- the masks of a Hoshen-Kopelman scan down a 32-column band,
// shared by the tiled and the one-CTA path.
#pragma once
#include <stdint.h>

namespace sw {

// ------------------------------------------------- row masks of the band scan
//
// Phase 1 of the tiled path, and the one-CTA path, label sites by a
// Hoshen-Kopelman scan down each 32-column band: the rows are visited top to
// bottom, every run (a maximal stretch of east bonds inside one row word)
// takes the label of the run above it that it is bonded to, or a new label
// (its first site) when it has no bond upwards, and a run bonded to several
// runs above that carry different labels makes those labels equivalent (a
// union). What each run of a row needs -- which of its columns passes the
// label down, which columns join a further run above -- follows from four bit
// masks of the row, computed for all runs of a word at once.

// Bits j of D whose interval (previous bit of D below j, j] holds a bit of X
// (for the lowest bit of D the interval starts at bit 0). One addition scans
// all intervals: a bit of X outside D starts a carry that runs up through the
// bits outside D and stops on the next bit of D.
__device__ __forceinline__ uint32_t carry_hit(uint32_t X, uint32_t D) {
  const uint32_t nd = ~D;
  return ((nd + (X & nd)) & D) | (X & D);
}

// Masks of row word B given the row word A above it in the same band. eB, eA:
// east bonds inside the tile (bit 31 = bond into the next word, not part of a
// run here); vB, vA: valid columns; D: south bonds from A into B.
//   R: run starts of B;
//   F: the first column of each run of B with a bond upwards -- the run takes
//      the label of the site above that column;
//   S: F, plus the start of every run with no bond upwards (a new label);
//   M: the other bonds upwards that reach a run of A different from the one
//      reached by the previous bond of the same run of B -- each asks for a
//      union of that run's label with the label of the run of B.
struct RowMasks {
  uint32_t R, S, F, M;
};
__device__ __forceinline__ RowMasks row_masks(uint32_t eB, uint32_t vB, uint32_t eA, uint32_t vA, uint32_t D) {
  const uint32_t RB = ~(eB << 1) & vB;
  const uint32_t RA = ~(eA << 1) & vA;
  const uint32_t F = carry_hit(RB, D);
  const uint32_t M = carry_hit(RA, D) & ~F;
  // runs of B that hold a bit of D: the same scan on the reversed word, where
  // a run's start is the top of its interval
  const uint32_t withD = __brev(carry_hit(__brev(D), __brev(RB)));
  RowMasks m;
  m.R = RB;
  m.F = F;
  m.M = M;
  m.S = F | (RB & ~withD);
  return m;
}

// Sum of v over the lanes below this one.
__device__ __forceinline__ int warp_exclusive_sum(int v, int lane) {
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  return incl - v;
}

}  // namespace sw
