// Hand-over of positions from the warp on the chain to the warps that absorb them beside it (rt_leaf_small.cu, rt_backward_loop.cu): a ring
// of kSlots entries, each with a barrier that says "entry ready" and one that says "entry read by every absorbing warp".
//
// A waiter sees only the parity of a barrier's phase, so it must never be more than one phase behind.  The chain depends on the warp that
// owns the next position, not on the others: one of those can be kSlots hand-overs behind.  With one ready barrier for all entries it would
// then wait for a parity that has come and gone twice, the chain for an entry that nobody frees any more, until the time limit ends both.  With a
// ready barrier per entry the read barrier of the same entry keeps the two at most one phase apart.
#pragma once

#ifdef __CUDACC__
#define RT_HANDOVER_FN __host__ __device__ constexpr
#else
#define RT_HANDOVER_FN constexpr
#endif

namespace rt {

struct Handover {
  static constexpr int kSlots = 4;
  static constexpr int kReadyBars = kSlots;                                                  // barriers "entry ready"
  static RT_HANDOVER_FN int slot(int j) { return j % kSlots; }                               // entry of hand-over j, and its read barrier
  static RT_HANDOVER_FN int ready_bar(int j) { return j % kReadyBars; }
  static RT_HANDOVER_FN unsigned ready_parity(int j) { return (unsigned)(j / kReadyBars) & 1u; }
  static RT_HANDOVER_FN unsigned read_parity(int j) { return (unsigned)(j / kSlots) & 1u; }  // of hand-over j's entry having been read
};

}  // namespace rt
