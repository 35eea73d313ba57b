// Launches of the sweep kernels (hiccl_sweep_kernels.cuh), and those that most
// programs run.

#include <algorithm>

#include "hiccl_sweep_kernels.cuh"

namespace hiccl {

// dynamic shared memory: at most SWEEP_MAX_DEPTH saved values of 16 words for
// each of 256 threads beside the rings of eight warps, and the values of many
// sections; more than half an SM's keeps a second CTA off it
constexpr size_t SWEEP_MAX_SMEM = SWEEP_MAX_DEPTH * 16 * 4 * 256 + 8 * FP8_SLOTS * FP8_STEP, SWEEP_HALF_SM = 120 * 1024,
                 SWEEP_MANY_SMEM = SWEEP_MAX_SMEM + SWEEP_TEAM_MAX * FP8_STEP;
static_assert(SWEEP_MANY_SMEM <= 227 * 1024, "a CTA's shared memory");

namespace {

bool many_sections(const SweepLaunch &L) { return L.sections > SWEEP_TEAM_STATIC; }
bool is_team(const SweepLaunch &L) { return L.kernel == SWEEP_TEAM || L.kernel == SWEEP_FP8_TEAM; }

// the kernel of a launch (one: for one CTA an SM, which teams are limited to as they are)
SweepKernel kernel_of(const SweepLaunch &L, bool one) {
  if (is_team(L) ? many_sections(L) : one) return sweep_rare_kernel(L.kernel);
  switch (L.kernel) {
    case SWEEP_COPY: return sweep_copy_kernel<false>;
    case SWEEP_FOLD: return sweep_fold_kernel<false>;
    case SWEEP_FP8: return sweep_fp8_kernel<false>;
    case SWEEP_NARROW: return sweep_narrow_kernel<false>;
    case SWEEP_SHIFT: return sweep_shift_kernel<false>;
    case SWEEP_TEAM: return sweep_team_kernel<false>;
    default: return sweep_fp8_team_kernel<false>;
  }
}

}  // namespace

cudaError_t sweep_prepare(const SweepLaunch &L, bool one) {
  return cudaFuncSetAttribute(kernel_of(L, one), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              many_sections(L) ? SWEEP_MANY_SMEM : SWEEP_MAX_SMEM);
}
uint32_t sweep_kernel_index(const SweepLaunch &L, bool one) {
  return 2 * L.kernel + (is_team(L) ? many_sections(L) : one);
}

cudaError_t sweep_launch(const SweepLaunch &L, const SweepArgs &A, unsigned one_per_sm, cudaStream_t s) {
  const bool team = is_team(L), fp8 = L.kernel == SWEEP_FP8 || L.kernel == SWEEP_FP8_TEAM;
  // One CTA an SM: CTAs of up to 16 warps (the usual ones, one at a time: All-to-all
  // of 64 ranks x 4 MiB 314 us, Reduce-scatter 254 us, 110 and 73 us step by step),
  // copies and FP8 folds walking over their units in a single wave (91 us), the
  // other folds in waves, as their registers do not suffice for the walk (53 us)
  const bool one = one_per_sm && !team;
  SweepArgs B = A;
  B.sections = L.sections;
  if (L.kernel == SWEEP_FOLD) B.groups = !one && L.units < SHORT_UNITS ? FOLD_GROUPS_SHORT : FOLD_GROUPS;
  size_t per_warp = (size_t)L.stack_words * 4 * 32;
  if (L.kernel == SWEEP_FOLD) per_warp += B.groups * RING_GROUP * 512;
  if (fp8) per_warp += FP8_SLOTS * FP8_STEP;
  unsigned warps = L.threads / 32;
  if (one) {
    warps = std::min(SWEEP_ONE_THREADS / 32, std::max(1u, (L.units + one_per_sm - 1) / one_per_sm));
    while (warps > 1 && warps * per_warp > SWEEP_MAX_SMEM) --warps;
  }
  unsigned grid = team ? L.units : (L.units + warps - 1) / warps;
  if (one && L.kernel != SWEEP_FOLD && L.kernel != SWEEP_NARROW) grid = std::min(grid, one_per_sm);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(warps * 32);
  cfg.dynamicSmemBytes = warps * per_warp;
  if (many_sections(L)) cfg.dynamicSmemBytes += L.sections * (fp8 ? FP8_STEP : 512);
  if (one_per_sm && cfg.dynamicSmemBytes < SWEEP_HALF_SM) cfg.dynamicSmemBytes = SWEEP_HALF_SM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel_of(L, one), B);
}

}  // namespace hiccl
