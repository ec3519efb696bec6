// The refill of a ring's stage, apart from the instructions that do it, so that
// the host can check its order.
#pragma once

#ifdef __CUDACC__
#define MAPE_REFILL_FN __device__ __forceinline__
#else
#define MAPE_REFILL_FN inline
#endif

namespace mape_detail {

// By every lane of the warp that feeds a ring, after it has used the chunk in
// the stage.  ok: no wait of the lane has run out so far; emptied(): waits until
// every reader has handed the stage back, false when its time ran out;
// all(b): the warp's vote; refill(): arms the stage's barrier and starts the copy.
// After a wait that ran out the stage is left alone: its barrier may still be
// within a phase, and arming it again would be one arrival too many.
template <typename Emptied, typename All, typename Refill>
MAPE_REFILL_FN bool refill_stage(bool ok, Emptied emptied, All all, Refill refill) {
  if (!emptied()) ok = false;
  if (all(ok)) refill();
  return ok;
}

}  // namespace mape_detail
