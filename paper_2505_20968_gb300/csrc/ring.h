// Hand-over of the stages of a shared-memory ring from a producer (bulk copies) to a consumer
// that gives them back, with waits that may give up.  The rules a role follows are here, its
// barriers and work are passed in, so that the rules can be run on the host against a model of
// the barriers (no CUDA).
//
// A stage's two barriers complete one phase per use: "full" (armed by the producer with the bytes
// of its copies, arrival count 1) and "empty" (the consumer's).  What the rules keep, also when a
// wait gives up at any point:
//   - "full" is armed and a stage filled only after the consumer has given the stage back, so no
//     phase is armed twice and no copy lands in a stage that another copy is filling;
//   - a stage is given back only after its copies have landed and been used;
//   - at the end every copy has landed: once no role touches the ring any more, the producer
//     waits for those of the stages it filled last.
#pragma once

#if defined(__CUDACC__)
#define PRD_RING_FN __host__ __device__ __forceinline__
#else
#define PRD_RING_FN inline
#endif

namespace prd {

// stage and phase parity of the it-th use of a ring of n stages
struct RingPos {
  int s = 0;
  unsigned ph = 0;
  PRD_RING_FN void next(int n) {
    if (++s == n) {
      s = 0;
      ph ^= 1;
    }
  }
};

// Producer: fills up to `iters` stages in turn and returns how many it filled.
// wait_empty(s, parity): bounded wait, false when it gives up; fill(s): arms "full" and copies.
template <class W, class F>
PRD_RING_FN int ring_produce(int iters, int n, W&& wait_empty, F&& fill) {
  RingPos p;
  int it = 0;
  for (; it < iters; ++it, p.next(n)) {
    if (it >= n && !wait_empty(p.s, p.ph ^ 1)) break;
    fill(p.s);
  }
  return it;
}

// Producer, before the ring's memory is laid out anew: waits until the consumer has given back
// every stage of the `iters` filled; false when a wait gives up.
template <class W>
PRD_RING_FN bool ring_close(int iters, int n, W&& wait_empty) {
  for (int k = iters > n ? iters - n : 0; k < iters; ++k)
    if (!wait_empty(k % n, (unsigned)(k / n) & 1u)) return false;
  return true;
}

// Consumer: takes the next stage.  wait_full(s, parity, limit): bounded wait of at most `limit`
// polls, false when it gives up; use(s, landed): works on the stage and gives it back if it has
// landed, does neither otherwise.  After a wait that gave up nothing is waited for or taken.
template <class W, class U>
PRD_RING_FN void ring_take(RingPos& p, int n, int& limit, W&& wait_full, U&& use) {
  if (!wait_full(p.s, p.ph, limit)) limit = 0;
  use(p.s, limit > 0);
  p.next(n);
}

// Once no role touches the ring any more: the copies of the stages filled last.
// landed(s, parity) waits for a stage's copies.
template <class L>
PRD_RING_FN void ring_drain(int filled, int n, L&& landed) {
  for (int k = filled > n ? filled - n : 0; k < filled; ++k) landed(k % n, (unsigned)(k / n) & 1u);
}

}  // namespace prd
