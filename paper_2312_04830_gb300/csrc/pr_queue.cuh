// A block's queue of cells to be finished together: its threads push entries
// in rounds of at most one a thread (atomicAdd on the count), and whenever a
// block's worth has gathered, every thread finishes one.
#pragma once

#ifdef __CUDACC__
#define PRQ_FN __device__ __forceinline__
#define PRQ_BARRIER() __syncthreads()
#else
#define PRQ_FN static inline   // host build: the test supplies PRQ_BARRIER
#endif

namespace prk {

// After a round's pushes (queue room: two blocks' worth; at most one less than
// a block's worth is left over, so a round never adds up to two): with a
// block's worth, every thread finishes one of the newest entries.
// `finish(e)` takes entry e.  The count is read once, by every thread, between
// two barriers: a thread that read it in a loop of its own could see the next
// round's pushes and enter the body without the others.  The last barrier
// keeps the next round's pushes off entries that are still being read.
template <class Finish>
PRQ_FN void queue_round(int *q_n, int tid, int threads, Finish finish)
{
    PRQ_BARRIER();   // the round's entries are written
    const int n = *q_n;
    PRQ_BARRIER();   // every thread has the count
    if (n >= threads) {
        if (tid == 0) *q_n = n - threads;
        finish(n - threads + tid);
        PRQ_BARRIER();
    }
}

// After the last round: fewer entries than threads.
template <class Finish>
PRQ_FN void queue_rest(const int *q_n, int tid, Finish finish)
{
    if (tid < *q_n) finish(tid);
}

}  // namespace prk
