// How the CTAs of the persistent serving kernel agree to leave, free of CUDA: one word holds the number
// of CTAs that hold or are taking a unit and a closed bit. A CTA enters before it claims a unit and
// leaves when the unit is done; the kernel closes only from 0, in one atomic step, so that either the
// closing CTA finds an entered one and does not close, or the entering CTA finds the word closed and
// claims nothing: no CTA is left to walk a unit alone while the others have gone. (Two words, one read
// and then the other set, let a CTA enter in between.) serve.cu runs it on device atomics, a CPU test on
// words of its own.
#pragma once

#ifdef __CUDACC__
#define RS_CLOSE_FN __host__ __device__ __forceinline__
#else
#define RS_CLOSE_FN inline
#endif

namespace rs {
namespace life {

constexpr int CLOSED = 1 << 30;

// Word: int add(int) (returns the old value), int cas(int expected, int desired) (returns the old
// value), int load().

// Enter before claiming a unit; false: closed.
template <class Word>
RS_CLOSE_FN bool enter(Word &w)
{
    if (!(w.add(1) & CLOSED)) return true;
    w.add(-1);
    return false;
}

template <class Word>
RS_CLOSE_FN void leave(Word &w)
{
    w.add(-1);
}

// Close if no CTA has entered; true: closed by this call.
template <class Word>
RS_CLOSE_FN bool close(Word &w)
{
    return w.cas(0, CLOSED) == 0;
}

template <class Word>
RS_CLOSE_FN bool closed(Word &w)
{
    return (w.load() & CLOSED) != 0;
}

}  // namespace life
}  // namespace rs
