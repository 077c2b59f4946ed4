// span.cuh -- positions in a particle array, in 32 bits over the whole range of a species
// (at most 2^31 - 1 particles).  Plain C++: the arithmetic is tested on the host.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define PIC_HD __host__ __device__ __forceinline__
#else
#define PIC_HD inline
#endif

namespace pic {

// A position that a loop forms, past its share's end too.  Unsigned: shares end below 2^31
// and a round steps past the end by a few thousand, so it does not wrap, where a signed
// one wrapped to a negative value that passes the test for the end.
typedef uint32_t Slot;
PIC_HD Slot slot_at(Slot base, unsigned offset) { return base + offset; }
PIC_HD bool slot_before(Slot p, int end) { return p < (Slot)end; }

// Rows of 32 that hold n particles; none for a negative n (the difference of two offsets
// of which a sort that timed out has written one).
PIC_HD int slot_rows(int n) { return n > 0 ? (int)(((uint32_t)n + 31u) >> 5) : 0; }

}  // namespace pic
