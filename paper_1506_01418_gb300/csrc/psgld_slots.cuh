// psgld_slots.cuh -- where the units of a part keep the sums of a row that
// spans several of them (psgld_units.cu): per unit a head slot, for the row
// that goes on from the unit before, and a tail slot, for the row that goes
// on in the next, ldk floats each.
//
// In 64 bits: one part may hold every entry (block-diagonal data), and
// 3.4e7 entries at K = 512 (8 a unit) already need 2^32 floats.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define PSGLD_HD __host__ __device__ __forceinline__
#else
#define PSGLD_HD inline
#endif

namespace psgld {

PSGLD_HD int64_t head_slot(int64_t unit, int32_t ldk) { return 2 * unit * ldk; }
PSGLD_HD int64_t tail_slot(int64_t unit, int32_t ldk) { return (2 * unit + 1) * ldk; }

// Floats for the slots of a part of n entries in units of `unit`.
PSGLD_HD int64_t slot_floats(int64_t n, int32_t unit, int32_t ldk) { return 2 * (n / unit + 1) * ldk; }

}  // namespace psgld
