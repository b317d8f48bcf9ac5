// One-controller step kernels of the 5-state planar quadrotor with far-field cells:
// plain, with smoothing, with the grid map.
#include "kernels.cuh"

namespace dbm {

__global__ void __maxnreg__(DBM_STEP_MAXNREG) step_p8_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<3, 8, false, false, true>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG) step_p14_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<3, 14, false, false, true>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG) step_p8_sgf_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<3, 8, true, false, true>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG) step_p14_sgf_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<3, 14, true, false, true>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG) step_p8_grid_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<3, 8, true, true, true>(D, x0, xref);
}

__global__ void __maxnreg__(DBM_STEP_MAXNREG) step_p14_grid_far(
    const __grid_constant__ CtrlDesc D, const double* __restrict__ x0,
    const double* __restrict__ xref) {
  step_body<3, 14, true, true, true>(D, x0, xref);
}

}  // namespace dbm
