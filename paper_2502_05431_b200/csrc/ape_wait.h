// How long a wait may last, and the wait for what the other blocks of a cluster send.  No PTX in here: the rule can be run on the host.
#pragma once

#ifdef __CUDACC__
#define APE_DEVICE __device__ __forceinline__
#else
#define APE_DEVICE inline
#endif

namespace ape {

// Every wait in the library is bounded: after about a second (2^31 SM cycles) the waiter raises the CTA's
// abort flag and the device status word, and every role of the CTA leaves its loop.
constexpr long long kWaitCycles = 1ll << 31;
// The wait for what other blocks send does not end for the abort flag, and not before theirs have: a block whose own wait has run out sends its
// rows all the same, after it has let its copies and products drain (2^24 cycles for each role), and a block that left before that
// would leave copies behind that land in the shared memory of whichever block comes next.
constexpr long long kReceiveCycles = 4 * kWaitCycles;

// arrived(): all that is sent to this block is here; now(): cycles.  Returns false, after give_up(), when even kReceiveCycles were not enough.
template <typename Arrived, typename Now, typename GiveUp>
APE_DEVICE bool wait_received(Arrived arrived, Now now, GiveUp give_up) {
    if (arrived()) return true;
    const long long t0 = now();
    while (!arrived()) {
        if (now() - t0 > kReceiveCycles) { give_up(); return false; }
    }
    return true;
}

}  // namespace ape
