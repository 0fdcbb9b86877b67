// gcp_noalloc_hot.h -- how the replicas of hot rows lie in the scratch of the
// allocation-free gradient (gcp_noalloc.cu), and which of what is found there
// a kernel may use.
//
// The scratch is shared by every call on a device, and only the caller orders
// the calls.  Where two overlap all the same, their results are undefined, but
// a kernel must not leave the arrays that it was given: each takes the word
// and the rows that it finds through hot_word_for and row_in_mode, which
// hold whatever is there to the shape of the kernel's own call.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define NA_HD __host__ __device__
#else
#define NA_HD
#endif

namespace gcpna {

constexpr int kHot = 32;               // hot rows of a mode at most
constexpr int kRepFloats = 23 * 1024;  // replica rows, shared out evenly over the modes

// Floats of a replica row, and of one mode's share of the replicas.
NA_HD constexpr int row_floats(int R) { return (R + 3) & ~3; }
NA_HD constexpr int mode_floats(int d) { return (kRepFloats / d) & ~3; }

// Replicas of each of n hot rows: 4, 8, 16 or 32, as many as fit the mode's
// share, or 0 where n is 0 or too large for four of each.
NA_HD inline int replicas(int n, int R, int d) {
    const int row = n * row_floats(R), share = mode_floats(d);
    if (n < 1 || n > kHot || 4 * row > share) return 0;
    int r = 4;
    while (r < 32 && 2 * r * row <= share) r *= 2;
    return r;
}

// n and their replicas in one word, which is read once by whoever uses it, so
// that the two always belong together.
NA_HD inline int hot_word(int n, int R, int d) {
    const int r = replicas(n, R, d);
    return r ? n | r << 8 : 0;
}

// The word as it may be used by a call of this rank and order: as it is if it
// was written for such a call, else 0 (no hot rows).
NA_HD inline int hot_word_for(int word, int R, int d) { return word == hot_word(word & 255, R, d) ? word : 0; }
NA_HD inline int hot_count(int word) { return word & 255; }
NA_HD inline int hot_replicas(int word) { return word >> 8; }

NA_HD inline bool row_in_mode(int row, int64_t dim) { return row >= 0 && row < dim; }

}  // namespace gcpna
