// The word of a post of merges (gwcp_wide.cu): how many merges the post holds and how many
// have been handed out, in one word. Plain integer functions, so that a host program can walk
// through every interleaving of walkers with them.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define GWCP_POST_FN __host__ __device__ __forceinline__
#else
#define GWCP_POST_FN inline
#endif

namespace gwcp {

// A walker draws a merge by adding 1 to the word: the value before the add holds both the merge
// drawn and the number of merges of the very post it was drawn from. (With the number in a
// word of its own, read after the draw, a walker that drew past the end of one post could
// hold its draw against the next, larger post in the same place: a merge done twice, `done`
// one too high, and the poster leaving with a merge still in flight.)
constexpr uint32_t kPostClosed = 0;  // no merges: nothing can be drawn
GWCP_POST_FN uint32_t post_open(uint32_t merges) { return merges << 16; }
GWCP_POST_FN uint32_t post_merge(uint32_t word) { return word & 0xFFFFu; }   // the merge drawn with this value
GWCP_POST_FN uint32_t post_merges(uint32_t word) { return word >> 16; }      // of so many
// Whether the value holds a merge. Walkers add only after they have seen a value that does, so
// a post is overdrawn by at most one draw per walker and the low half never carries.
GWCP_POST_FN bool post_left(uint32_t word) { return post_merge(word) < post_merges(word); }

}  // namespace gwcp
