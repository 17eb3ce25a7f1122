// Rule of the hand-overs from several writing warps to the one that issues MMAs, through barriers of the SM (bar.arrive, bar.sync),
// which have no limit of their own.  Hand-overs are numbered 0, 1, 2, ...; every warp takes part in every one of them, also after
// one of its waits has run out:
//   - a writing warp in order arrives and goes on; it reaches hand-over p + 1 only after an answer (an mbarrier with a limit) to p,
//     so p is complete by then;
//   - a writing warp that has failed has no answer to pace it: it waits at every later hand-over until it is complete;
//   - the MMA warp waits at every hand-over, failed or not;
//   - even and odd hand-overs go through barriers of their own.
// So no warp arrives at a barrier whose last-but-one hand-over (the one before on that barrier) is still open: in order at p it has
// seen p - 1 complete, and its first hand-over after a failure at p - 1 is p, on the other barrier, with p - 2 complete.  No
// arrival can be counted for a hand-over that it does not belong to, and as every wait between two hand-overs has a limit, all
// warps reach the last one.  (On one barrier, or with failed warps that do not wait, eight warps can complete hand-overs without
// the MMA warp, which then waits for arrivals that have been used up.)
#pragma once

#if defined(__CUDACC__)
#define UOE_HAND_OVER_FN __host__ __device__ constexpr
#else
#define UOE_HAND_OVER_FN constexpr
#endif

namespace uoe {
UOE_HAND_OVER_FN int hand_over_barrier(int p) { return p & 1; }              // which of the two barriers
UOE_HAND_OVER_FN bool hand_over_waits(bool failed) { return failed; }        // whether a writing warp waits there

#if defined(__CUDACC__)
// A writing warp's part in a hand-over of THREADS threads on barrier `id`; `failed` is the same in the whole warp.  (The branch marked as
// the rare one: image block forward 179.5 us and 180.6 as predicated instructions; unmarked it spills registers.)
template <int THREADS>
__device__ __forceinline__ void hand_over_write(int id, bool failed) {
    if (__builtin_expect(hand_over_waits(failed), 0)) asm volatile("bar.sync %0, %1;" :: "r"(id), "n"(THREADS) : "memory");
    else asm volatile("bar.arrive %0, %1;" :: "r"(id), "n"(THREADS) : "memory");
}
// The MMA warp's part
template <int THREADS>
__device__ __forceinline__ void hand_over_take(int id) { asm volatile("bar.sync %0, %1;" :: "r"(id), "n"(THREADS) : "memory"); }
#endif
}  // namespace uoe
