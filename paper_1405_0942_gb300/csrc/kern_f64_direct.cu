// FP64 (GLEMUR_FP64) stages with the direct-derivative current.
//
// The classic current at a node needs first and second differences of x,
// first differences of B0s and nothing another thread has formed, so a stage
// is one dense pass over the interior nodes (split64.cuh), every value loaded
// from the node's neighbours through L1 (19 points of the stage input, 7 of
// B0s).  It is bound by the FP64 pipe, which the equal shares of node warps
// keep evenly busy: 65^3, an attempt 1.51 ms on shared-memory tiles (32 x 8
// columns, one CTA of 8 warps per SM at 180-226 registers: 135 CTAs for 152
// SMs, a stage 244 us where the pipe's time for its instructions was 106),
// 0.755 ms on two CTAs of 8 warps per SM, 0.697 ms on one of 16 (128
// registers).
#include "split64.cuh"

namespace glemur {

namespace {

// Direct current at interior node n (section "Diagnostics", the classic
// method): dB/dX of B = V / det G, V = sum_a g_a b_a, by the product rule,
//   det D_c B = D_c V - V (D_c det) / det,
//   D_c V = sum_a S_ac b_a + g_a D_c b_a,  D_c det = sum_a (g_a+1 x g_a+2) . S_ac,
// with the second differences S_ac of x; the antisymmetric part of
// dB/dx = dB/dX (dx/dX)^-1 in covariant form is
//   J = (c_0 g_0 + c_1 g_1 + c_2 g_2) / det,  c_a = D_{a+1} B . g_{a+2} - D_{a+2} B . g_{a+1}
// (six inner products instead of the product with the inverse).  The scale 4
// of the pure second differences S_aa (index space: g_a is twice a first
// difference) rides on b_a and on one FMA.  Returns V, det^2 J and 1/det.
__device__ __forceinline__ void direct_current(const SplitArgs& a, const double* __restrict__ y,
                                               int N, int n, double V[3], double Jd2[3],
                                               double& r, double& det) {
  const int st[3] = {1, a.nx, a.nx * a.ny};
  double g[3][3], s[3][3], x[3][3];  // x[0] = S_12, x[1] = S_02, x[2] = S_01; 4 s[a] = S_aa
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double* v = y + c * N + n;
    const double yc = __ldg(v);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const double p = __ldg(v + st[e]), m = __ldg(v - st[e]);
      g[e][c] = p - m;
      s[e][c] = fma(-2.0, yc, p + m);
      const int p1 = st[(e + 1) % 3], p2 = st[(e + 2) % 3];
      x[e][c] = (__ldg(v + p1 + p2) - __ldg(v + p1 - p2)) -
                (__ldg(v - p1 + p2) - __ldg(v - p1 - p2));
    }
  }
#pragma unroll
  for (int e = 0; e < 3; ++e) g[e][e] += a.h2[e];
  double cof[3][3];
#pragma unroll
  for (int e = 0; e < 3; ++e) cross64(g[(e + 1) % 3], g[(e + 2) % 3], cof[e]);
  det = dot3(g[0], cof[0]);
  r = recip(det);
  double b[3], b4[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    b[e] = __ldg(&a.B0s[e * N + n]);
    b4[e] = 4.0 * b[e];
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) V[c] = g[0][c] * b[0] + g[1][c] * b[1] + g[2][c] * b[2];
  double DB[3][3];  // det D_c B
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;  // S_{c1 c} = x[c2], S_{c2 c} = x[c1]
    double Dd = 4.0 * dot3(cof[c], s[c]);
#pragma unroll
    for (int i = 0; i < 3; ++i) Dd = fma(cof[c1][i], x[c2][i], fma(cof[c2][i], x[c1][i], Dd));
    Dd *= r;
    double Db[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const double* q = a.B0s + e * N + n;
      Db[e] = __ldg(q + st[c]) - __ldg(q - st[c]);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double t = s[c][i] * b4[c];
      t = fma(x[c2][i], b[c1], t);
      t = fma(x[c1][i], b[c2], t);
#pragma unroll
      for (int e = 0; e < 3; ++e) t = fma(g[e][i], Db[e], t);
      DB[c][i] = fma(-V[i], Dd, t);
    }
  }
  double cc[3];
#pragma unroll
  for (int e = 0; e < 3; ++e)
    cc[e] = dot3_sub(DB[(e + 1) % 3], g[(e + 2) % 3], DB[(e + 2) % 3], g[(e + 1) % 3]);
#pragma unroll
  for (int c = 0; c < 3; ++c) Jd2[c] = cc[0] * g[0][c] + cc[1] * g[1][c] + cc[2] * g[2][c];
}

template <int S>
__global__ void __launch_bounds__(DENSE_T2, 1) k_direct64(const SplitArgs a) {
  int cur;
  if (!dense_start<S == 0>(a, cur)) return;
  __shared__ double red[32];
  const DevState* st = a.st;
  const int N = a.nx * a.ny * a.nz;
  const double* d = a.d[cur];
  double* dout = const_cast<double*>(a.d[cur ^ 1]);
  const double* y = S == 0 ? d : a.ys[S & 1];
  double* ynext = a.ys[(S + 1) & 1];
  double an[5];
#pragma unroll
  for (int j = 0; j < 5; ++j) an[j] = S < 5 && j <= S ? st->dta[S < 5 ? S + 1 : 0][j] : 0.0;
  Acc<double> acc;
  int tb, te;
  cta_range(a.inner_c, tb, te);
  for (int t = tb + threadIdx.x; t < te; t += blockDim.x) {
    int i, j, k;
    const int n = interior_node(a, t, i, j, k);
    double V[3], J[3], u[3], r, det;
    direct_current(a, y, N, n, V, J, r, det);
    if (le_zero(det))  // NaN: reported by the error norm
      atomicOr(&a.st->flags, S == 0 ? FLAG_COLLAPSED : FLAG_FOLDED_TRIAL);
    const double r2 = r * r;
    // u = J x B with J = Jd2 r^2, B = V r
    cross64(J, V, u);
    const double r3 = r2 * r;
#pragma unroll
    for (int c = 0; c < 3; ++c) u[c] *= r3;
    if (S == 0 && a.diag) acc.max_xi(dot3(u, u), dot3(V, V) * r2, dot3(J, J) * (r2 * r2));
    split_emit<S, LdRO>(a, d, dout, ynext, an, N, n, k, u, acc);
  }
  pdl_trigger();
  if (S == 5) {
    const double v = block_reduce<true>(acc.lam, red);
    if (threadIdx.x == 0) put_partial(a, PART_LAMBDA, v);
  }
  if (S == 0 && a.diag) {
    double v = block_reduce<true>(acc.xi2(), red);
    if (threadIdx.x == 0) put_partial(a, PART_XI2, v);
    v = block_reduce<true>(acc.xis2(), red);
    if (threadIdx.x == 0) {
      put_partial(a, PART_XIS2, v);
      put_partial(a, PART_E, 0.0);  // interior nodes only: no energy
    }
  }
}

}  // namespace

// Let the stages ask for DENSE_SMEM.
cudaError_t prepare_f64_direct() {
  void (*k[6])(const SplitArgs) = {k_direct64<0>, k_direct64<1>, k_direct64<2>,
                                   k_direct64<3>, k_direct64<4>, k_direct64<5>};
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 6 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(k[i], cudaFuncAttributeMaxDynamicSharedMemorySize, DENSE_SMEM);
  return e;
}

// Launch stage `stage`.
cudaError_t launch_f64_direct(const SplitArgs& a, int stage, cudaStream_t s) {
  const dim3 g(a.grid_c), nt(a.threads_c);
  switch (stage) {
    case 0: return launch_pdl(k_direct64<0>, g, nt, DENSE_SMEM, s, a);
    case 1: return launch_pdl(k_direct64<1>, g, nt, DENSE_SMEM, s, a);
    case 2: return launch_pdl(k_direct64<2>, g, nt, DENSE_SMEM, s, a);
    case 3: return launch_pdl(k_direct64<3>, g, nt, DENSE_SMEM, s, a);
    case 4: return launch_pdl(k_direct64<4>, g, nt, DENSE_SMEM, s, a);
    case 5: return launch_pdl(k_direct64<5>, g, nt, DENSE_SMEM, s, a);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace glemur
