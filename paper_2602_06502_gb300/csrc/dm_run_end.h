// dm_run_end.h -- where a prompt's run of resident blocks ends, by three
// probes a round.  No CUDA types: the host tests compile it too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DM_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define DM_HOST_DEVICE inline
#endif

namespace dm {

// The blocks 0 .. nblk - 1 of a prompt whose block 0 is resident (nblk >= 1).
// A round probes blocks b[0 .. 2] (below nblk, in any order) and leaves a
// quarter of the range; the first round starts at `guess`, a block thought to
// be the first missing one (0: no idea).
//
// The resident blocks are a leading run, unless a lookup gave up (it counts as
// missing, and its call ends with its status) or two keys collide.  A higher
// block may then be resident above a missing one: the range is closed at once
// and the run ends at the lowest block found missing, so no later round
// computes blocks from an empty range.
struct RunEnd {
    uint32_t lo, hi;   // block lo is resident; hi is not, or is the prompt's end
    uint32_t b[3];

    DM_HOST_DEVICE RunEnd(uint32_t nblk, uint32_t guess) : lo(0), hi(nblk) {
        b[0] = guess ? guess - 1 : nblk / 4;
        if (b[0] >= nblk) b[0] = nblk - 1;
        b[1] = guess < nblk ? guess : nblk - 1;
        b[2] = nblk / 2 < b[0] ? b[0] : nblk / 2;
    }
    DM_HOST_DEVICE bool open() const { return hi > lo + 1; }
    DM_HOST_DEVICE void narrow(const bool (&in)[3]) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int q = 0; q < 3; ++q) {
            if (in[q]) lo = b[q] > lo ? b[q] : lo;
            else hi = b[q] < hi ? b[q] : hi;
        }
        const uint32_t step = (hi - lo) / 4, rest = (hi - lo) & 3u;
        const uint32_t x = lo + step + (rest > 2), y = lo + 2 * step + (rest > 1), z = lo + 3 * step + rest;
        b[0] = x > lo ? x : lo + 1;
        b[1] = y > b[0] ? y : b[0];
        b[2] = z < hi ? z : hi - 1;
        b[2] = b[2] > b[1] ? b[2] : b[1];
    }
};

}  // namespace dm
