// Per-thread tallies of a walk, reduced when a CTA finishes a medium.
#ifndef MCMIE_TALLY_H
#define MCMIE_TALLY_H

#include <stdint.h>

#ifdef __CUDACC__
#define MCX_HD __host__ __device__ __forceinline__
#else
#define MCX_HD inline
#endif

namespace mcx {

// A thread counts its flights in 32 bits, although one warp may carry a whole
// medium of 2^31 photons (launch shape, sharing of a batch). So the count is
// handed on to the medium's total (Tally::due) whenever the warp takes new
// photons, MAX_ITEM at a time at most, and on every flight of a photon from its
// LOOK_FLIGHTS-th on: between two looks a thread ends at most MAX_ITEM + 1
// photons of at most LOOK_FLIGHTS flights each. (No slower at tau 5, 0.5 % on
// the plume's walk. A 64-bit count, one more instruction a flight, takes 1 % on
// an H-G walk and 1.5 % on the plume's; a sum at each photon's end 1.5 to 2.7 %
// on 64 media.)
constexpr uint32_t MAX_ITEM = 1u << 15, LOOK_FLIGHTS = 1u << 16, HOLD_FLIGHTS = 1u << 30;
static_assert(HOLD_FLIGHTS + (MAX_ITEM + 1ull) * LOOK_FLIGHTS < (1ull << 32), "a count that stays must not wrap");

struct Tally {
    uint32_t steps = 0;         // flights since the last that were handed on
    uint32_t n_refl = 0, n_far = 0, n_side = 0, n_ball = 0;   // photons of weight one, at most 2^31
    long long refl = 0, far = 0, side = 0, ball = 0, abs = 0; // 2^-32 weight units

    MCX_HD uint32_t due()       // flights to hand on now (0: none yet)
    {
        if (steps < HOLD_FLIGHTS) return 0;
        const uint32_t n = steps;
        steps = 0;
        return n;
    }
};

}  // namespace mcx

#endif
