// Shared by the refinement residual's kernels: the monomial coefficients of
// eqs. A2D / A3D (helm_resid.cu) and the fixed-point kernels (helm_resid_fx.cu).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace helm {

struct ResidQArgs {
  int64_t n[3];
  // 3D: c0[4 cx + 2 cy + cz][2 b + c], c1[2 cy + cz][2 b + c]; 2D: c0[2 cx + cy][b], c1[cy][b]
  double2 c0[8][4];
  double2 c1[4][4];
  // 3D corrections of the end classes against the same class inside y and z:
  // dc0[cls][bc] = c0[cls][bc] - c0[cls & 4][bc], dc1[cyz][bc] = c1[cyz][bc] - c1[0][bc]
  double2 dc0[8][4];
  double2 dc1[4][4];
};

// Tensor map of a [nx][ny][nz] complex128 array viewed as [nx][ny][2 nz]
// FP64, with a box of bz complex values x by rows along y; false if it cannot
// be made.
bool residual_map(CUtensorMap* m, const double2* v, const int64_t* n, int bz, int by);

// r = f - A u in 64-bit fixed point (helm_resid_fx.cu): complex64 r and the
// block sums of |r|^2, |f|^2 (*nblocks pairs, at most residual_fx_blocks).
// cudaErrorNotSupported: 3D without tensor maps (nothing launched).
cudaError_t launch_residual_fx(int dim, const ResidQArgs& q, const double2* f, const double2* u, float2* r,
                               double* sums, int64_t* nblocks, const int* skip, int* err, cudaStream_t st);
int64_t residual_fx_blocks(int dim, const int64_t* n);

}  // namespace helm
