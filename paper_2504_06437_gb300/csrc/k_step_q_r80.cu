// One-controller step kernels of the planar quadrotor model, 80-register form
// (see DBM_STEP_MAXNREG_R80), without and with far-field cells.
#include "kernels.cuh"

namespace dbm {

__global__ void __maxnreg__(DBM_STEP_MAXNREG_R80) step_q8_r80(const __grid_constant__ CtrlDesc D,
                                                         const double* __restrict__ x0,
                                                         const double* __restrict__ xref) {
  step_body<1, 8>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG_R80) step_q14_r80(const __grid_constant__ CtrlDesc D,
                                                          const double* __restrict__ x0,
                                                          const double* __restrict__ xref) {
  step_body<1, 14>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG_R80) step_q8_r80_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<1, 8, false, false, true>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG_R80) step_q14_r80_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<1, 14, false, false, true>(D, x0, xref);
}

}  // namespace dbm
