// Gather tables of the shared-memory row kernels: for each of 32 consecutive states the row
// entries it sums, in an order that spreads a warp's reads over the shared-memory banks.
//
// A thread that sums d random entries of a staged row reads one per slot.  Random addresses
// cost a warp 3.5 shared-memory wavefronts per 4-byte slot (of 1) and 6.3 per 16-byte slot (of
// 4), and the order of a thread's own terms is free, so the table picks it: slot by slot,
// each lane takes the entry whose bank is still unused in this slot and most in demand later.
// Measured on the tables of the 18-site Hubbard cluster (4-byte entries): 28.8 wavefronts per
// state instead of 64.1; 16 sites, 16-byte entries: 23.0 per eight lanes instead of 40.3.
//
// Terms carry a phase (a sign, or a coefficient class).  Slots run phase by phase, each phase
// as many slots as the longest of the 32 lists, so the phase of a slot is the same in all
// lanes; lanes without a term left read one of the zero entries that follow the staged row, in
// a bank nobody else uses.
//
// Layout: records of four slots, rec[group * stride + state], so a warp reads 256 consecutive
// bytes per group; hdr[warp] holds the slot ends of phases 0 .. 7, cumulative, 16 bits each.
#pragma once

#include "common.cuh"

namespace hphi {

constexpr int kGatherPhases = 8;
// lanes that share one pass over the banks for entries of the given width, which is also the
// number of zero entries after a staged row
__host__ __device__ constexpr int gather_lanes(int entry_bytes) {
  return entry_bytes <= 4 ? 32 : (entry_bytes <= 8 ? 16 : 8);
}

// records are read in chunks of this many groups; a table has whole chunks allocated
constexpr int kGatherChunk = 4;

// end of phase f from a warp's header
__device__ __forceinline__ int gather_end(const uint4& h, int f) {
  const uint32_t w = f < 2 ? h.x : f < 4 ? h.y : f < 6 ? h.z : h.w;
  return (int)((f & 1) ? (w >> 16) : (w & 0xffffu));
}

}  // namespace hphi
