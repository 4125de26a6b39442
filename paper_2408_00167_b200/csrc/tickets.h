// How the ranges of a scoring unit learn that all of them have published their row statistics: two counters per unit in
// global memory, zero before and after every call.  Every range publishes once and leaves once, in this order and
// however it ends -- also after a wait that ran out, when it has nothing to publish and has waited for nobody -- so that the
// last one to leave can set both back to zero and a call finds nothing of the one before it.  (A range that gives up lets its
// neighbours read statistics that were never written; the status word says so of the whole call.)
#pragma once

#ifdef __CUDACC__
#define FINCH_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define FINCH_HOST_DEVICE inline
#endif

namespace finch {

struct Tickets {
    int *published, *left;  // ranges of a unit that have published / that need the counters no more
    int ranges;             // of a unit

    FINCH_HOST_DEVICE static int add(int *counter) {
#ifdef __CUDA_ARCH__
        return atomicAdd(counter, 1);
#else
        return __atomic_fetch_add(counter, 1, __ATOMIC_ACQ_REL);
#endif
    }
    FINCH_HOST_DEVICE void publish(int unit) const { add(published + unit); }
    FINCH_HOST_DEVICE void leave(int unit) const {
        if (add(left + unit) == ranges - 1) {
            published[unit] = 0;
            left[unit] = 0;
        }
    }
    // A range from its own statistics to those of all ranges: own() waits until the former are written, all(counter, ranges)
    // until the counter has come to `ranges`; either is false when it gives up.  good: nothing has failed before.
    template <typename Own, typename All>
    FINCH_HOST_DEVICE bool pass(int unit, bool good, const Own &own, const All &all) const {
        good = good && own();
        publish(unit);
        good = good && all(published + unit, ranges);
        leave(unit);
        return good;
    }
};

}  // namespace finch
