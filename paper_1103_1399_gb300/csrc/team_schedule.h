// Which buffer of a team's exchange each step uses (team.cu), in one place so that a
// host program can check the order of every pair of accesses.
#pragma once

#ifdef __CUDACC__
#define QAA_HD __host__ __device__
#else
#define QAA_HD
#endif

namespace qaa {

// Cluster form, shared memory of one CTA: two buffers for its own transposes, then two
// that its partners fill, in turn by step.  The transposes stay out of what the partners
// fill: a partner that has its words of step j may send step j + 1 while other threads
// of this CTA still read their last transpose of step j (each partner's words come
// from some of the threads only).
constexpr int kClusterBuffers = 4;
QAA_HD constexpr int cluster_transpose(int j, int k) { return (void)j, k; }  // k: 0, 1
QAA_HD constexpr int cluster_receive(int j) { return 2 + (j & 1); }

// Word form, global memory: buffers in turn by step.  A receiver empties a slot in step
// j, after it has taken the word; its sender stores the next word there in step j +
// kWordBuffers.  Behind the takes and emptyings of step j a warp of each CTA runs a
// fence, and the CTA's stores of step j + kWordFenceLag wait for it.  The emptying is
// before the next store if a fence of the receiver, words sent behind it and a fence of
// the sender behind those words' arrival lie in between: twice the lag.  (Two CTAs on an
// SM have no room for a fence warp: thread 0 runs the fence between the transposes of step
// j + 1, whose barriers put it before that step's stores: a lag of one.)
constexpr int kWordBuffers = 4;
constexpr int kWordFenceLag = 2;
QAA_HD constexpr int word_buffer(int j) { return j % kWordBuffers; }
static_assert(kWordBuffers >= 2 * kWordFenceLag, "a fence on both sides between the emptying of a slot and its next use");

}  // namespace qaa
