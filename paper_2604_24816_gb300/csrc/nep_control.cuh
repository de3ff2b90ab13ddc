// nep_control.cuh -- the rebuild decision (device side), taken by one thread after the positions have changed and
// before the rebuild chain.
#pragma once

#include "nep_common.cuh"

namespace nep {

// What decides: an earlier kernel already did; an MD step (displacement past skin/2, or every
// rebuild_every steps); a check after an upload that kept the list (displacement only, the step counters are
// not touched); or a rebuild in any case.
enum : int { DECIDE_DONE = 0, DECIDE_STEP = 1, DECIDE_CHECK = 2, DECIDE_FORCE = 3 };

// Sets do_rebuild and, for the row walks of the coming evaluation, skip_far: the far bands can be left out while no
// atom moved far enough since the build to bring a far-band pair inside rc_R.  Returns do_rebuild.
__device__ __forceinline__ int decide_rebuild(Control *ctrl, int decide) {
  if (decide == DECIDE_DONE) return ctrl->do_rebuild;
  int rb = ctrl->moved;
  if (decide == DECIDE_STEP) {
    ctrl->steps += 1;
    ctrl->steps_since += 1;
    if (ctrl->rebuild_every > 0 && ctrl->steps_since >= ctrl->rebuild_every) rb = 1;
    ctrl->fb_count = 0; // of the evaluation to come
    ctrl->pending = 1;  // this step's closing half kick: done by the next step's opening kick or the final one
  }
  if (decide == DECIDE_FORCE) rb = 1;
  ctrl->do_rebuild = rb;
  if (rb) {
    ctrl->moved = 0;
    ctrl->steps_since = 0;
    ctrl->rebuilds += 1;
    ctrl->dmax2 = 0.f;
  }
  ctrl->skip_far = (rb ? 0.f : ctrl->dmax2) < ctrl->far_dmax2 ? 1 : 0;
  return rb;
}

}  // namespace nep
