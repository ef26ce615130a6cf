// bounded_wait.cuh -- a wait with a time limit that all threads of a block end
// alike, shared by the inner solver's kernel and a host-side check (plain C++,
// no CUDA needed).
//
// Every thread of a block polls the same condition, which once true stays true
// until the block's next barrier.  A thread whose limit runs out adds itself to
// a count in shared memory and polls on.  The wait has failed when the count is
// the whole block, and from then on it stays that: a thread that sees the
// condition come true takes itself off the count again, by compare-and-swap, but
// never off a full one.  So either all threads return false, or all true: one
// that has returned true is not in the count, which then cannot fill up, and the
// others, however late, see the condition as well.  Without this a condition
// that comes true around the limit sends the threads of a block different ways,
// and they meet different barriers.
//
// The loops end: a thread polls at most `limit`, then until the others have run
// out too or the condition has come true for it as for them.
#pragma once

#ifndef __CUDACC__
#ifndef __host__
#define __host__
#endif
#ifndef __device__
#define __device__
#endif
#ifndef __forceinline__
#define __forceinline__ inline
#endif
#endif

// poll(): the condition; now(): nanoseconds; count: load(), add() and
// cas(expected, value) on the block's counter, 0 before the first wait and after
// every one that has succeeded.
template <typename Poll, typename Now, typename Count>
__host__ __device__ __forceinline__ bool bounded_wait(Poll poll, Now now, Count count, int nthreads,
                                                      unsigned long long limit) {
    unsigned long long t0 = 0;
    for (int i = 0;; ++i) {
        if (poll()) return true;
        if ((i & 15) == 15) {  // (a poll may itself wait a while)
            const unsigned long long t = now();
            if (!t0) t0 = t;
            else if (t - t0 > limit) break;
        }
    }
    count.add();
    for (;;) {
        if (count.load() >= nthreads) return false;
        if (!poll()) continue;
        for (;;) {
            const int c = count.load();
            if (c >= nthreads) return false;
            if (count.cas(c, c - 1)) return true;
        }
    }
}
