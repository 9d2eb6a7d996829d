// Hand-back of the streamed forward's two stage buffers (tc_wide.cuh): the
// commit of stage t's MMAs completes barrier slot(t), and a producer warp with
// a task of stage t waits there for stage t - 2, which used the same buffer.
//
// A wait by parity tells completion j of a barrier from completion j - 1 only
// if the waiter knows that j - 1 has happened, and from j + 1 only if that
// cannot have happened.  A warp's tasks skip stages (by at most one), so it
// does not see every completion itself.  With one barrier per buffer, what it
// has to know is that stage t - 4 is done, and after a task of stage t - 1 it
// has only seen stage t - 3: right as long as commits arrive in order, which
// is not promised.  With four barriers it has to know of stage t - 6.  Its
// last task, of stage t - 2 or t - 1, saw stage t - 4 or t - 3 complete; the
// MMAs of t - 4 were issued after every task of t - 4 was written, and those
// tasks' warps had seen t - 6.  Stage t + 2, the next completion of the same
// barrier, needs stage t, hence this warp.
#pragma once
#ifdef __CUDACC__
#define IMG_RING_FN __host__ __device__ constexpr
#else
#define IMG_RING_FN constexpr
#endif

namespace img {
namespace fwd_ring {

constexpr int kProducers = 15;          // producer warps
constexpr int kSlots = 4;               // barriers
constexpr int kBuffers = 2;             // stage buffers
IMG_RING_FN int slot(int t) { return t % kSlots; }
// Parity of stage t's completion of its barrier.
IMG_RING_FN unsigned parity(int t) { return (unsigned)(t / kSlots) & 1u; }
// Warps that take tasks of stages of ntask tasks each (task id goes to warp id
// % warps): at most two stages' tasks in flight, so that a warp's next task is
// at most two stages on.  Small arrays have as few as 4 tasks per stage.
IMG_RING_FN int warps(int ntask) { return kProducers < kBuffers * ntask ? kProducers : kBuffers * ntask; }

}  // namespace fwd_ring
}  // namespace img
