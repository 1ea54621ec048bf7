// Control flow of bounded waits, apart from the instructions it runs on, so
// that the host can run it as well (threads and counters in the place of
// warps and barriers; no GPU).
#pragma once
#include <cuda_runtime.h>

namespace fe {

// One round of a fill warp of k_phase1_ts over its NST stages; whether to go
// on, which is the same in every fill warp. All of them call it in every
// round: vote(ok) is a barrier of the fill warps that returns whether all were
// ok, so a warp that left without it would leave the others waiting there.
//   moved    the round realigns (the same in every warp)
//   copy()   the warp's own bulk copies; false if one of its waits gave up
//   free(k)  whether stage k may be written (one thread waits for it)
//   realign(k)  the warps' common copy of stage k
template <int NST, class Copy, class Free, class Realign, class Vote>
__host__ __device__ __forceinline__ bool ts_fill_round(bool moved, Copy &&copy, Free &&free, Realign &&realign,
                                                       Vote &&vote) {
    // (the vote follows the copies: a warp that gave up alone takes the others with it before the next round)
    if (!moved) return vote(copy());
#pragma unroll 1
    for (int k = 0; k < NST; k++) {
        if (!vote(free(k))) return false;
        realign(k);
    }
    return true;
}

// A warp's copies into its one buffer, one on its way at a time, and the waits
// for them. After a wait that gave up (over() ended it) the warp takes no more
// copies and waits no more: its barrier's phase is not over, so another copy
// asked for on it would be counted wrongly, and a wait per item left would
// each run to its limit.
struct CopyWait {
    unsigned parity = 0;
    bool pending = false, dead = false;
    template <class Start>
    __host__ __device__ __forceinline__ void ask(Start &&start) {
        if (dead) return;
        start();
        pending = true;
    }
    // here(parity): whether the copy has arrived; over(): whether to give up. False: the buffer holds nothing.
    template <class Here, class Over>
    __host__ __device__ __forceinline__ bool arrived(Here &&here, Over &&over) {
        if (dead) return false;
        while (!here(parity))
            if (over()) {
                dead = true;
                return false;
            }
        parity ^= 1u;
        pending = false;
        return true;
    }
    // before the warp leaves: a copy still on its way (there is none unless a wait gave up) is given one more limit
    template <class Here, class Over>
    __host__ __device__ __forceinline__ void leave(Here &&here, Over &&over) {
        if (pending)
            while (!here(parity))
                if (over()) return;
    }
};

}  // namespace fe
