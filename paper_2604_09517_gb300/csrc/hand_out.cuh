// Hands a value from one thread of a CTA to all of them, one barrier deep.
// Plain C++, so that the protocol also runs on the host.
#pragma once
#ifdef __CUDACC__
#define HPL_HAND_OUT __device__ __forceinline__
#else
#define HPL_HAND_OUT inline
#endif

namespace hplgb {

// The leader's value, in every thread; words: two words that all threads share;
// pass: each thread's own count of calls, 0 at the first. The words alternate,
// because nothing keeps the leader from writing its next value while a thread
// has yet to read this one: the calls may follow each other with no barrier
// between them. The word is written again two calls later, after the next
// call's barrier, which every thread reaches with this call's read behind it.
template <class Sync>
HPL_HAND_OUT int hand_out(int* words, int& pass, bool leader, int value, Sync sync) {
    int* w = words + (pass & 1);
    pass ^= 1;
    if (leader) *w = value;
    sync();
    return *w;
}

}  // namespace hplgb
