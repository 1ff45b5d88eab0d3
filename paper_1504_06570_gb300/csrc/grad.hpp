// Parameters of the adjoint kernels (grad.cu), filled by phosim_grad.
#pragma once

#include "phosim_device.cuh"

namespace phosim {

constexpr int kMaxGradParams = 128;
// Gradient sums of one source and surface, in the order the adjoint kernel reduces them: 32 for the monomials of
// the Zernike figure (kZPoly of them), then 32 for the misalignments (the force on the surface, k = 0..2, and the torque,
// k = 3..5, in its frame, in the words 32 + k + 8 g, g = 0..3)
constexpr int kGradWords = 64;

// a Zernike figure's second derivatives in x and y by the monomials u^a v^b, a + b <= 4, row by row in b
struct ZernikeHessian {
    double xx[15], xy[15], yy[15];
};

struct GradParams {
    int n_params;
    int first_surface;                                   // the first surface with a parameter: the sweep ends there
    uint8_t shift[PHOSIM_MAX_SURFACES];                  // 1: a decenter of this surface is a parameter
    uint8_t tilt[PHOSIM_MAX_SURFACES];                   // 1: a tilt is
    uint8_t figure[PHOSIM_MAX_SURFACES];                 // 1: a Zernike coefficient is
    int32_t param_surface[kMaxGradParams], param_field[kMaxGradParams];
    double axis[PHOSIM_MAX_SURFACES][6][3];              // of each field: the direction of its shift, the axis of its rotation
    ZernikeHessian hessian[PHOSIM_MAX_SURFACES];         // of the surfaces with a figure
    const double* zmono;                                 // PHOSIM_MAX_ZERNIKE x kZPoly monomials of Z_j
    const double* seeds;                                 // per source: Ax, Ay, Bxx, Bxy, Byy, mean x, mean y, 0
    double* sums;                                        // n_src x n_surf x kGradWords, added to
    double* grad;                                        // n_src x n_params, written by launch_grad_finish
};

cudaError_t launch_grad(const TraceParams& P, const GradParams& G, const BatchList& L, int blocks, cudaStream_t st);
cudaError_t launch_grad_finish(const TraceParams& P, const GradParams& G, cudaStream_t st);
cudaError_t grad_occupancy(int* blocks_per_sm);

}  // namespace phosim
