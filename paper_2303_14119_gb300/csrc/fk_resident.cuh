// Host interface of the resident step kernel (fk_resident.cu).
#pragma once

#include "fk_internal.cuh"

namespace fk {

// Several steps in one launch: between its steps a unit tells the launch's
// finalize CTAs that its planes are done and waits for the coefficients of
// the new state.  Both counters start at kCountZero.
struct Resident {
  unsigned* arrive;  // one count per unit and step; kGoStop: no further step
  unsigned* go;      // n_fin counts per step; kGoStop: no further step
  unsigned n_units;
  unsigned n_fin;    // finalize CTAs
  int n_steps;
  double* lv_odd;    // the velocity-edge partials of odd steps
};
constexpr unsigned kCountZero = 0xFFFFFFFFu;  // so that one memset prepares a launch
constexpr unsigned kGoStop = 1u << 24;        // above any count of a launch
constexpr int kResidentSteps = 128;           // most steps of a launch

struct ResidentArgs {
  StepArgs a;   // step 0's; odd steps swap f_in and f_out
  FinOut o;
  Resident rs;
  unsigned long long* xch;  // [rows][kFinMaxBlocks] exchange of block sums, all bits set
};

// Words of the block that holds a launch's counters and exchange slots; every
// bit of it is set before a launch.
int resident_scratch_words();
// Shared memory of a CTA and how many fit on an SM (0: the kernel cannot run).
size_t resident_smem_bytes(int precision, const Geom& gm, int pitch);
int resident_ctas_per_sm(int precision, const Geom& gm, int pitch, bool padded);
// n_steps <= kResidentSteps steps; scratch: resident_scratch_words() 32-bit words.
cudaError_t launch_resident(const StepArgs& a, const FinOut& o, int precision, bool bgk,
                            int n_steps, double* lv_odd, unsigned* scratch, cudaStream_t s);

}  // namespace fk
