// Host interface of the fused split step (fk_split.cu).
#pragma once

#include "fk_internal.cuh"

namespace fk {

// What a fused split step needs beside StepArgs (whose geom and part are the
// split plan's): the partial sums of the state after the velocity step and
// that state on the two boundary planes (rows with v1 < 0: x = 0, rows with
// v1 > 0: x = h_max).
struct SplitArgs {
  StepArgs a;
  double *pe_mid, *see_mid, *vac_mid;  // [n_tiles]
  void* h_wall;                        // [nv1][pitch]
};

// Tiles and chunks of a fused split step for these sizes; false if a plan
// does not fit (rows too wide for a tile of two of them) or the passes are
// faster.  half: the grid's streaming units are half units.
bool plan_split(int precision, bool strang, int nx, int nv1, int pitch, int i_neg, bool half,
                int sms, Geom* gm);
// One Lie (strang = false) or Strang step of f_in into f_out, without its
// finalize; the second also adds the mid-step fluxes' share to a.st.
cudaError_t launch_split_step(const SplitArgs& sa, int precision, bool strang, bool bgk,
                              cudaStream_t s);

}  // namespace fk
