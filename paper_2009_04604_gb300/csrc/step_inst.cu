// step_inst.cu -- explicit instantiation of one part of the fused step for one
// lattice and storage type. The build compiles this file once per part and pair,
// with -DLBM_STEP_PART=<0|1|2>, -DLBM_STEP_LATTICE=<D2Q9|D3Q19|D3Q27> and
// -DLBM_STEP_STORE=<double|float|__half|__nv_bfloat16>; without them it defines nothing.
#include "step.cuh"

#if defined(LBM_STEP_LATTICE) && defined(LBM_STEP_STORE) && defined(LBM_STEP_PART)
namespace lbm {
#if LBM_STEP_PART == 0
LBM_STEP_PART0(, LBM_STEP_LATTICE, LBM_STEP_STORE)
#elif LBM_STEP_PART == 1
LBM_STEP_PART1(, LBM_STEP_LATTICE, LBM_STEP_STORE)
#else
LBM_STEP_PART2(, LBM_STEP_LATTICE, LBM_STEP_STORE)
#endif
}  // namespace lbm
#endif
