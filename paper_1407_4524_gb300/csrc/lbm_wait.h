// lbm_wait.h -- the clock of the bounded device waits (plain C++, so that the
// rule runs on the host too).
#pragma once

#ifdef __CUDACC__
#define LBM_WAIT_FN __host__ __device__ __forceinline__
#else
#define LBM_WAIT_FN inline
#endif

namespace lbm {

constexpr unsigned long long STAGE_WAIT_NS = 1000000000ull; // a wait gives up after one second of polling
// A gap between two looks at the clock counts for at most this much.  Polls are
// microseconds apart; a longer gap means that the context was switched out, and
// the copy waited for lands after it is back: one gap, however long, must not
// end the wait.
constexpr unsigned long long STAGE_GAP_NS = STAGE_WAIT_NS / 8;

struct WaitClock {
    unsigned long long last, spent;
};

// now: the clock, at or after c.last; true when the wait has to give up
LBM_WAIT_FN bool wait_over(WaitClock &c, unsigned long long now) {
    const unsigned long long gap = now - c.last;
    c.last = now;
    c.spent += gap < STAGE_GAP_NS ? gap : STAGE_GAP_NS;
    return c.spent > STAGE_WAIT_NS;
}

} // namespace lbm
