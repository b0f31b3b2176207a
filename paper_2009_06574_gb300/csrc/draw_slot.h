// Places of a drawing block's records: a ring slot holds one chunk's triangles
// behind a blank record, so that a lane's next triangle is the place of the
// lowest set bit of its mask, counted from 1, and a lane without a triangle (mask
// 0) has a place too, which nothing writes while the ring is in use. Compiles for
// the device and, for tests, for the host.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define HEXFC_SLOT __device__ __forceinline__
#define HEXFC_SLOT_CONST __host__ __device__ constexpr
#else
#define HEXFC_SLOT inline
#define HEXFC_SLOT_CONST constexpr
inline int __ffs(int v) { return __builtin_ffs(v); }
#endif

namespace hexfc {

constexpr int kSlotBlank = 0;
HEXFC_SLOT_CONST int slot_records(int chunk) { return chunk + 1; }
// The place of triangle j of the chunk.
HEXFC_SLOT_CONST int slot_place(int j) { return j + 1; }
// The place of the next triangle of the mask m (kSlotBlank: none).
HEXFC_SLOT int next_place(uint32_t m) { return __ffs((int)m); }

}  // namespace hexfc
