// Words of a match stream, two 16-bit entries each (see gate_multi.cu).  Plain C++ as well, so that the bit tricks can be
// checked on the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SR_BITS __host__ __device__ __forceinline__
#else
#define SR_BITS static inline
#endif

namespace sr {

constexpr uint32_t kLocNone = 0x7FFFu;    // bit 15 clear, far above any row: shifts to 0
constexpr uint32_t kLocRow = 0x8000u;     // | index of the symbol's mask row

// Top bit of each half of x that is not zero.
SR_BITS uint32_t set_halves(uint32_t x) { return (((x & 0x7FFF7FFFu) + 0x7FFF7FFFu) | x) & 0x80008000u; }

// Top bit of each half of stream word v with matches beside the main diagonal, whose places are in `at`: a mask row (or
// a chain), or a single position from `strip` on.  A symbol of the removed common prefix that occurs again in the text is
// no match of what is left of the pair.
SR_BITS uint32_t matches_beside(uint32_t v, uint32_t at, int strip) {
    // strip is below 2^15, so that no half borrows from the other
    const uint32_t left = ((v & 0x7FFF7FFFu) | 0x80008000u) - (uint32_t)strip * 0x10001u;
    return set_halves(v ^ at) & set_halves(v ^ (kLocNone * 0x10001u)) & (left | v);
}

}  // namespace sr
