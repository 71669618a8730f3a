// Handing out the units of a persistent attention kernel.  The grid has one block per unit; as many as fit run, and a running CTA takes
// the next unit that no block has started (cluster launch control) when its producer has all but issued the loads of the current
// one.  The list is sorted by decreasing cost, so this is greedy longest-first scheduling by the real times: a fixed round-robin
// left the chip 16 to 20 % idle on lists of a few units per SM, and 1 to 2 % on long ones.  The producer puts every unit it takes into
// a ring from which the other roles read it; an entry without keys ends the list.
#pragma once
#include "common.h"
#include "sm100_ptx.cuh"

namespace mpipe {

constexpr int kUnitRing = 4;
struct UnitRing {
    uint4 answer;                          // of the last request (16-byte aligned by its type)
    mpipe_work_item_t item[kUnitRing];     // `seg` holds the head
    uint64_t answered, full[kUnitRing], empty[kUnitRing];
};
__device__ __forceinline__ void unit_ring_init(UnitRing* r, int readers) {
    mbar_init(&r->answered, 1);
    for (int i = 0; i < kUnitRing; ++i) {
        mbar_init(&r->full[i], 1);
        mbar_init(&r->empty[i], readers);
    }
}

// Producer side (one thread).
struct UnitSource {
    UnitRing* ring;
    volatile int* abort_flag;
    uint32_t taken = 0, asked = 0;
    bool outstanding = false;              // a request whose answer has not been seen
    bool ended = false;                    // an answer without a block has come: no more may be asked for
    __device__ __forceinline__ void ask() {
        mbar_expect_tx(&ring->answered, 16);
        clc_try_cancel(&ring->answer, &ring->answered);
        ++asked;
        outstanding = true;
    }
    // The unit of the outstanding request, -1 at the end of the list (or after a time-out, *ok = false).
    __device__ __forceinline__ int take(bool* ok) {
        *ok = mbar_wait(&ring->answered, (asked - 1) & 1, abort_flag);
        if (!*ok) return -1;
        outstanding = false;
        const int u = clc_block_of(&ring->answer);
        ended = u < 0;
        fence_async_smem();                // the answer has been read before the next one is asked for
        return u;
    }
    __device__ __forceinline__ bool put(const mpipe_work_item_t& it) {
        const uint32_t slot = taken % kUnitRing;
        if (!mbar_wait(&ring->empty[slot], ((taken / kUnitRing) & 1) ^ 1, abort_flag)) return false;
        ring->item[slot] = it;
        mbar_arrive(&ring->full[slot]);    // (release: the entry is visible to whoever sees the phase complete)
        ++taken;
        return true;
    }
    // After a time-out: nothing of this grid shall start any more, or every further block would run into its own time-out.  An answer
    // still on its way is waited for first: the barrier counts one at a time.
    __device__ __forceinline__ void cancel_rest() {
        int dummy = 0;
        while (!ended) {
            if (!outstanding) ask();
            if (!mbar_wait_budget(&ring->answered, (asked - 1) & 1, &dummy, 10000000ll)) return;
            outstanding = false;
            ended = clc_block_of(&ring->answer) < 0;
            fence_async_smem();
        }
    }
};
// Reader side (a whole warp): the i-th unit of this CTA; false at the end of the list or after a time-out.
__device__ __forceinline__ bool next_unit(UnitRing* r, uint32_t i, mpipe_work_item_t* it, int lane, volatile int* abort_flag) {
    const uint32_t slot = i % kUnitRing;
    if (!mbar_wait(&r->full[slot], (i / kUnitRing) & 1, abort_flag)) return false;
    *it = r->item[slot];
    __syncwarp();
    if (lane == 0) mbar_arrive(&r->empty[slot]);
    return it->kv_len > 0;
}

}  // namespace mpipe
