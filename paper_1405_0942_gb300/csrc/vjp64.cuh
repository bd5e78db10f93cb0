// Arguments of the FP64 stage VJP passes (kern_f64_vjp.cu).
#pragma once

#include "glemur_dev.cuh"

namespace glemur {

struct VjpArgs {
  int nx, ny, nz;
  double h2[3];            // 2 h_a
  double s[3];             // B0s_a = s_a B0_a
  const double* y;         // the stage's input (displacement, 3N)
  const double* B0s;       // 3N
  const double* Bb;        // the stage's B, 3N
  const double* rec;       // its node records (G and 1/det G)
  const double* lam_next;  // lam', 3N
  const double* ly[6];     // stage-input adjoints of the later stages, 3N each
  double cb, ca[6];        // dt b_s; dt a_js (j > s)
  double *lamP, *lamg;     // adjoints of P_a and g_a, 9N each (P's zero on the boundary)
  double *lamr, *lamB;     // of 1/det G (N) and of B (3N), from the current
  double* ly_out;          // this stage's input adjoint, 3N (s > 0)
  double* lam;             // result (s = 0), 3N
  double* mu_B0;           // accumulated, 3N
  int grid, threads;
  WarpShare inner, faces, bound;  // interior, inner face and all boundary nodes
  FastDiv dx, dy, dz;
};

cudaError_t prepare_f64_vjp();
cudaError_t launch_f64_vjp(const VjpArgs& a, int stage, cudaStream_t s);

}  // namespace glemur
