// Barrier of the blocks of one problem in the one-kernel operator-splitting
// solve, with a bounded wait.  Word is the barrier's word in memory (device: global
// memory; the test runs the same code on host threads).
#pragma once

namespace rt3d {

// The barrier's word (zero before) counts the arrivals in its low half and those
// that have more to do in the half above; its top bit says that a wait gave
// up.  One atomic and one polled load carry all of it.
constexpr unsigned long long kBarGone = 1ull << 63;

// Arrive and wait for all nblk arrivals: how many of them had more to do, or a
// negative number where a wait gave up, this one after at most `polls` polls.
template <class Word>
__host__ __device__ inline int bar_wait(Word word, int nblk, bool more, int polls)
{
    word.arrive(more ? (1ull << 32) + 1 : 1ull);
    unsigned long long v;
    int n = 0;
    do v = word.load();
    while ((int)v < nblk && ++n < polls);
    return (int)v < nblk ? -1 : (int)(v >> 32);
}

// After a wait at the last barrier that returned a negative number: the same
// answer for all that arrive there.  The top bit is set while the arrivals are
// incomplete, and then every later reader sees it; where they are complete
// without it (some have passed) nothing is set and the wait has succeeded after
// all.  At an earlier barrier no agreement is needed: who gives up does not
// arrive at the next one, which nobody passes then.  (Apart from bar_wait, whose
// loop is in every sweep: with this in it the 17^3 solve took 1.2% longer.)
template <class Word>
__host__ __device__ inline int bar_settle(Word word, int nblk)
{
    unsigned long long v = word.load();
    while ((int)v < nblk && !(v & kBarGone)) {
        const unsigned long long seen = v;
        v = word.cas(seen, seen | kBarGone);      // what was there
        if (v == seen) return -1;
    }
    return (int)(v >> 32);
}

}  // namespace rt3d
