// The work queue of the batched solve: two lists of systems that persistent CTAs
// take from. Plain C++ but for the atomic addition, which the caller passes, so
// that it also runs on the host.
#pragma once
#ifdef __CUDACC__
#define HPL_QUEUE __device__ __forceinline__
#else
#define HPL_QUEUE inline
#endif

namespace hplgb {
namespace bt {

// Cleared by every run.
struct Queue {
    unsigned int counter[2];    // next index in list 0 / list 1
    unsigned int gave_up;       // CTAs that left with the queue not empty
};

// Table index of the next system (list l: sz[l] of them from lo[l] on), from the
// preferred list if it has any; -1 when both are empty.
template <class Add>
HPL_QUEUE int queue_next(Queue* q, const int (&lo)[2], const int (&sz)[2], int pref, Add add) {
    for (int i = 0; i < 2; i++) {
        const int l = pref ^ i;
        if (sz[l] > 0 && (int)*(volatile unsigned int*)&q->counter[l] < sz[l]) {
            const int t = (int)add(&q->counter[l], 1u);
            if (t < sz[l]) return lo[l] + t;
        }
    }
    return -1;
}

// A CTA that takes no further systems (a wait of its own gave up) leaves them to
// the others. The last of all ctas to leave so marks what is still queued: a
// system that nobody takes must not keep the record of an earlier run.
template <class Add, class Mark>
HPL_QUEUE void queue_give_up(Queue* q, const int (&lo)[2], const int (&sz)[2], unsigned ctas, Add add, Mark mark) {
    if (add(&q->gave_up, 1u) != ctas - 1) return;
    for (int i = queue_next(q, lo, sz, 0, add); i >= 0; i = queue_next(q, lo, sz, 0, add)) mark(i);
}

}  // namespace bt
}  // namespace hplgb
