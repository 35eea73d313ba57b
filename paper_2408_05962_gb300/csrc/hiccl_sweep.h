// Launch interface of the sweep kernels (hiccl_sweep.cu).
#pragma once

#include <cuda_runtime.h>

#include "hiccl_internal.h"

namespace hiccl {

struct SweepArgs {
  const SweepClass *classes;            // of this launch
  const uint32_t *toks;
  const unsigned long long *ptrs;
  const uint32_t *hints;                // of this launch
  uint32_t nclass;
  uint32_t units;
  uint32_t groups = 0;                  // of a fold's ring
  uint32_t sections = 0;                // whose values a team's CTA holds
  unsigned long long minus0 = 0x8000000080000000ull;   // two binary32 -0 (see mul2)
  uint32_t unit0[SWEEP_PREFIX];         // first units, for searching without a memory access
  SweepClass first[SWEEP_INLINE];       // the classes themselves, where there are few
};

typedef void (*SweepKernel)(const SweepArgs);
// the form of a kernel for one CTA an SM, or of a team's for many sections (hiccl_sweep_rare.cu)
SweepKernel sweep_rare_kernel(uint32_t kernel);

// Set the kernel of a launch up (`one`: for one CTA an SM), once per device, with
// it current; the index tells kernels apart.  (Loading a kernel takes up to a
// millisecond, so a kernel is set up for the first program that runs it.)
cudaError_t sweep_prepare(const SweepLaunch &L, bool one);
constexpr uint32_t SWEEP_KERNEL_FORMS = 2 * SWEEP_KERNELS;
uint32_t sweep_kernel_index(const SweepLaunch &L, bool one);
// one_per_sm: at most one CTA on an SM (CTAS_PER_SM = 1) of so many; 0: no limit
cudaError_t sweep_launch(const SweepLaunch &L, const SweepArgs &A, unsigned one_per_sm, cudaStream_t s);

}  // namespace hiccl
