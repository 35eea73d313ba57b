// The sweep kernels that few programs run: of launches limited to one CTA an SM,
// and of teams with many sections.  A module of their own, loaded when the first
// of them is set up: a module is loaded as a whole, and with them in
// hiccl_sweep.cu's (which nvcc then compresses) the first hiccl_init of a process
// took 10.6 ms instead of 3.0.

#include "hiccl_sweep_kernels.cuh"

namespace hiccl {

SweepKernel sweep_rare_kernel(uint32_t kernel) {
  switch (kernel) {
    case SWEEP_COPY: return sweep_copy_kernel<true>;
    case SWEEP_FOLD: return sweep_fold_kernel<true>;
    case SWEEP_FP8: return sweep_fp8_kernel<true>;
    case SWEEP_NARROW: return sweep_narrow_kernel<true>;
    case SWEEP_SHIFT: return sweep_shift_kernel<true>;
    case SWEEP_TEAM: return sweep_team_kernel<true>;
    default: return sweep_fp8_team_kernel<true>;
  }
}

}  // namespace hiccl
