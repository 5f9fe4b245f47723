// The rotating accumulators of the residue product with four real products
// (residue.cu), apart from the kernel so that a host program can check them.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ROT_FN __host__ __device__ __forceinline__
#else
#define ROT_FN inline
#endif

// The accumulator drained after chunk c of a unit of nc, other than at the unit's
// end: Re (0), Im (1) or none (-1).
ROT_FN int drained_after(int c, int nc) { return (c & 3) == 3 && c + 1 < nc ? (c & 4 ? 0 : 1) : -1; }

// Which of three buffers holds which accumulator: one that ends moves to the free
// buffer, and its old one is free once it is drained.  Every role follows the same
// sequence of ends: those of drained_after, and Re and Im at the end of a unit.
//
// A buffer is used again, by either accumulator, when the end of its last use is drained.  The
// drains signal that end by its number, on a ring of kEnds barriers.  (By the buffer, on
// one barrier each, the parity of a phase says too little: the accumulators belong to
// different warps, one of which may be six chunks ahead of the other, and would take
// the drain before the one it needs for it where a unit's length leaves short uses, such
// as 12 or 44 chunks.  On the ring that would take ends kEnds apart.)
struct AccState {
    static constexpr uint32_t kEnds = 8;
    uint32_t b[2] = {0, 1}, free = 2, drains = 0;  // drains: parity of each buffer's
    uint32_t ends = 0, last = 0x0F0F0F;            // ends so far; a byte a buffer: its last one, modulo 2 kEnds
    ROT_FN void end(int t) {
        const uint32_t old = t == 0 ? b[0] : b[1];
        if (t == 0) b[0] = free;
        else b[1] = free;
        free = old;
        drains ^= 1u << old;
        last = (last & ~(0xFFu << (8 * old))) | (ends & (2 * kEnds - 1)) << (8 * old);
        ends++;
    }
    // The barrier that the next end is signalled on
    ROT_FN uint32_t signal() const { return ends & (kEnds - 1); }
    // The barrier and the phase's parity to wait for before `buf` is used again (an unused
    // buffer: the phase before a fresh barrier's first, which has passed)
    ROT_FN uint32_t wait_on(uint32_t buf) const { return last >> (8 * buf) & (kEnds - 1); }
    ROT_FN uint32_t wait_parity(uint32_t buf) const { return last >> (8 * buf + 3) & 1; }
};
static_assert(AccState::kEnds == 8, "bits of last");
