// FP64 stage VJP of the reverse step, from the data the forward recompute
// keeps (dense passes, see split64.cuh).
//
// With the stage-input adjoints ly_j of the later stages (zero for the last)
// the adjoint of k_s is dt (b_s lam' + sum_{j>s} a_js ly_j); the stage's VJP
// (adjoint.cu states the steps) then gives ly_s and its share of mu, and after
// the first stage lam = lam' + sum_s ly_s.  So no stage reads or writes the
// adjoint of any other k.  Three passes per stage, all bound by the FP64
// pipe:
//   current    interior nodes: reverse of u = J x B and of the current, from
//              the node's record (G and 1/det G) and B around it;
//   pull-back  interior nodes and the inner parts of the faces: gather of the
//              adjoint of B, reverse of B = G B0s / det G.  With B itself at
//              hand the adjoint of det G is -r (lam_B . B + r lam_r), r = 1 /
//              det G, without forming G B0s again.  Edges and corners have no
//              interior neighbour: nothing reaches them;
//   positions  interior nodes: gather of the adjoints of g_a over the
//              difference stencils that contain the node.  Along an axis of n
//              nodes those of node p are the central ones at p -+ 1, weight
//              +-1, or on a face the one-sided one, weight +-4, and the
//              one-sided one two nodes away, weight -+1.
// 242 FP64-pipe instructions per interior node and stage (120 + 82 + 39),
// without forming G again in the first two passes, B0s's product in the
// second and every k's adjoint in the third; pull-back 64 -> 43 us at 64^3;
// the gradient over four steps there 8.27 -> 7.34 ms.
#include "split64.cuh"
#include "vjp64.cuh"

namespace glemur {

namespace {

// The node's record of pass B (kern_f64_split.cu, node_record).
__device__ __forceinline__ void load_record(const VjpArgs& a, int t, double g[3][3], double& r) {
  const double2* q = reinterpret_cast<const double2*>(a.rec) + ((size_t)(t >> 5) * 160 + (t & 31));
  const double2 q0 = __ldg(q), q1 = __ldg(q + 32), q2 = __ldg(q + 64), q3 = __ldg(q + 96),
                q4 = __ldg(q + 128);
  g[0][0] = q0.x; g[0][1] = q0.y; g[0][2] = q1.x;
  g[1][0] = q1.y; g[1][1] = q2.x; g[1][2] = q2.y;
  g[2][0] = q3.x; g[2][1] = q3.y; g[2][2] = q4.x;
  r = q4.y;
}

template <int S>
__global__ void __launch_bounds__(DENSE_T2, 1) k_vjp_current(const VjpArgs a) {
  pdl_wait();
  const int N = a.nx * a.ny * a.nz;
  const int st[3] = {1, a.nx, a.nx * a.ny};
  int tb, te;
  cta_range(a.inner, tb, te);
  for (int t = tb + threadIdx.x; t < te; t += blockDim.x) {
    int i, j, k;
    const int n = interior_node(a, t, i, j, k);
    double G[3][3], P[3][3], r;
    load_record(a, t, G, r);
    double B[3], lu[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double* b = a.Bb + c * N + n;
#pragma unroll
      for (int e = 0; e < 3; ++e) P[e][c] = __ldg(b + st[e]) - __ldg(b - st[e]);
      B[c] = __ldg(b);
      // adjoint of k_S (b_2 = b_5 = 0)
      double v = 0.0;
      if (S != 1 && S != 4) v = a.cb * __ldg(&a.lam_next[c * N + n]);
#pragma unroll
      for (int q = S + 1; q < 6; ++q) {
        const double l = __ldg(&a.ly[q][c * N + n]);
        v = (S == 4 || S == 1) && q == S + 1 ? a.ca[q] * l : fma(a.ca[q], l, v);
      }
      lu[c] = v;
    }
    double cc[3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
      cc[e] = dot3_sub(P[(e + 1) % 3], G[(e + 2) % 3], P[(e + 2) % 3], G[(e + 1) % 3]);
    double V[3], J[3], lJ[3], lB[3], lV[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      V[c] = cc[0] * G[0][c] + cc[1] * G[1][c] + cc[2] * G[2][c];
      J[c] = V[c] * r;
    }
    cross64(B, lu, lJ);  // u = J x B: lam_J = B x lam_u, lam_B = lam_u x J
    cross64(lu, J, lB);
#pragma unroll
    for (int c = 0; c < 3; ++c) lV[c] = lJ[c] * r;
    double lc[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) lc[e] = dot3(lV, G[e]);
    // c_a = P_{a+1} . g_{a+2} - P_{a+2} . g_{a+1}, V = sum_a c_a g_a
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const int e1 = (e + 1) % 3, e2 = (e + 2) % 3;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        a.lamP[(e * 3 + c) * N + n] = lc[e2] * G[e1][c] - lc[e1] * G[e2][c];
        a.lamg[(e * 3 + c) * N + n] =
            fma(lc[e1], P[e2][c], fma(-lc[e2], P[e1][c], cc[e] * lV[c]));
      }
    }
    a.lamr[n] = dot3(lJ, V);
#pragma unroll
    for (int c = 0; c < 3; ++c) a.lamB[c * N + n] = lB[c];
  }
  pdl_trigger();
}

// Reverse of B = G B0s / det G at a node from the adjoint lB of B: mu_B0, and
// the adjoints of the columns g_a on top of lg.
__device__ __forceinline__ void pullback_node64(const VjpArgs& a, int N, int n,
                                                const double G[3][3], double r,
                                                const double lB[3], double lr, double lg[3][3]) {
  double B[3], b[3], lW[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    B[c] = __ldg(&a.Bb[c * N + n]);
    b[c] = __ldg(&a.B0s[c * N + n]);
    lW[c] = lB[c] * r;
  }
  // B = W r, W = sum_a g_a b_a: lam_r = lam_B . W + lr = lam_B . B / r + lr
  const double ldet = -r * fma(r, lr, dot3(lB, B));
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    double cr[3];
    cross64(G[(e + 1) % 3], G[(e + 2) % 3], cr);
    const int q = e * N + n;
    a.mu_B0[q] = fma(a.s[e], dot3(lW, G[e]), a.mu_B0[q]);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      a.lamg[(e * 3 + c) * N + n] = fma(b[e], lW[c], fma(ldet, cr[c], lg[e][c]));
  }
}

// A face's inner node (axis A, s = +1 the low face, -1 the high one): only
// its interior neighbour's difference P_A contains B there.
template <int A>
__device__ __forceinline__ void pullback_face(const VjpArgs& a, int N, int n, int s) {
  const int st[3] = {1, a.nx, a.nx * a.ny};
  double G[3][3];
  gcol<A == 0, LdRO>(a.y, N, n, 1, s, G[0]);
  gcol<A == 1, LdRO>(a.y, N, n, a.nx, s, G[1]);
  gcol<A == 2, LdRO>(a.y, N, n, a.nx * a.ny, s, G[2]);
#pragma unroll
  for (int e = 0; e < 3; ++e) G[e][e] += a.h2[e];
  double lB[3], lg[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double l = __ldg(&a.lamP[(A * 3 + c) * N + n + s * st[A]]);
    lB[c] = s > 0 ? -l : l;
  }
  pullback_node64(a, N, n, G, recip(det3(G[0], G[1], G[2])), lB, 0.0, lg);
}

__global__ void __launch_bounds__(DENSE_T2, 1) k_vjp_pullback(const VjpArgs a) {
  pdl_wait();
  const int N = a.nx * a.ny * a.nz;
  const int st[3] = {1, a.nx, a.nx * a.ny};
  int tb, te;
  cta_range(a.inner, tb, te);
  for (int t = tb + threadIdx.x; t < te; t += blockDim.x) {
    int i, j, k;
    const int n = interior_node(a, t, i, j, k);
    double G[3][3], r, lg[3][3], lB[3];
    load_record(a, t, G, r);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      // P_a(m) = B(m + e_a) - B(m - e_a); P's adjoint is zero on the boundary
      lB[c] = __ldg(&a.lamB[c * N + n]);
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const double* l = a.lamP + (e * 3 + c) * N + n;
        lB[c] += __ldg(l - st[e]) - __ldg(l + st[e]);
        lg[e][c] = a.lamg[(e * 3 + c) * N + n];
      }
    }
    pullback_node64(a, N, n, G, r, lB, __ldg(&a.lamr[n]), lg);
  }
  // the faces take up where the interior left off
  const int nw = blockDim.x >> 5;
  int wb = (threadIdx.x >> 5) - ((te - tb + 31) >> 5);
  while (wb < 0) wb += nw;
  cta_range(a.faces, tb, te, gridDim.x - 1 - blockIdx.x);
  for (int b = tb + 32 * wb + (threadIdx.x & 31); b < te; b += blockDim.x) {
    int i, j, k;
    const int n = boundary_node(a, b, i, j, k);
    if (n < 0) continue;
    if (k == 0 || k == a.nz - 1)
      pullback_face<2>(a, N, n, k == 0 ? 1 : -1);
    else if (j == 0 || j == a.ny - 1)
      pullback_face<1>(a, N, n, j == 0 ? 1 : -1);
    else
      pullback_face<0>(a, N, n, i == 0 ? 1 : -1);
  }
  pdl_trigger();
}

// FIRST: the step's first stage, whose stage-input adjoint completes lam.
template <bool FIRST>
__global__ void __launch_bounds__(DENSE_T2, 1) k_vjp_positions(const VjpArgs a) {
  pdl_wait();
  const int N = a.nx * a.ny * a.nz;
  const int st[3] = {1, a.nx, a.nx * a.ny};
  const int ext[3] = {a.nx, a.ny, a.nz};
  int tb, te;
  cta_range(a.inner, tb, te);
  for (int t = tb + threadIdx.x; t < te; t += blockDim.x) {
    int id[3];
    const int n = interior_node(a, t, id[0], id[1], id[2]);
    double ly[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const int p = id[e];
      const double wm = p == 1 ? 4.0 : 1.0, wp = p == ext[e] - 2 ? -4.0 : -1.0;
      const double* l = a.lamg + e * 3 * N + n;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        ly[c] = fma(wm, __ldg(l + c * N - st[e]), ly[c]);
        ly[c] = fma(wp, __ldg(l + c * N + st[e]), ly[c]);
      }
      if (p == 2) {
#pragma unroll
        for (int c = 0; c < 3; ++c) ly[c] -= __ldg(l + c * N - 2 * st[e]);
      }
      if (p == ext[e] - 3) {
#pragma unroll
        for (int c = 0; c < 3; ++c) ly[c] += __ldg(l + c * N + 2 * st[e]);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int q = c * N + n;
      if (!FIRST) {
        a.ly_out[q] = ly[c];
      } else {
        double v = __ldg(&a.lam_next[q]) + ly[c];
#pragma unroll
        for (int m = 1; m < 6; ++m) v += __ldg(&a.ly[m][q]);
        a.lam[q] = v;
      }
    }
  }
  if (FIRST) {  // line-tied: no position adjoint is added on the boundary
    const int nw = blockDim.x >> 5;
    int wb = (threadIdx.x >> 5) - ((te - tb + 31) >> 5);
    while (wb < 0) wb += nw;
    cta_range(a.bound, tb, te, gridDim.x - 1 - blockIdx.x);
    for (int b = tb + 32 * wb + (threadIdx.x & 31); b < te; b += blockDim.x) {
      int i, j, k;
      const int n = boundary_node(a, b, i, j, k);
      if (n < 0) continue;
      for (int c = 0; c < 3; ++c) a.lam[c * N + n] = __ldg(&a.lam_next[c * N + n]);
    }
  }
  pdl_trigger();
}

template <int S>
cudaError_t launch_stage(const VjpArgs& a, cudaStream_t s) {
  const dim3 g(a.grid), t(a.threads);
  cudaError_t e = launch_pdl(k_vjp_current<S>, g, t, DENSE_SMEM, s, a);
  if (e == cudaSuccess) e = launch_pdl(k_vjp_pullback, g, t, DENSE_SMEM, s, a);
  if (e == cudaSuccess) e = launch_pdl(k_vjp_positions<S == 0>, g, t, DENSE_SMEM, s, a);
  return e;
}

}  // namespace

cudaError_t prepare_f64_vjp() {
  void (*k[9])(const VjpArgs) = {k_vjp_current<0>, k_vjp_current<1>,     k_vjp_current<2>,
                                 k_vjp_current<3>, k_vjp_current<4>,     k_vjp_current<5>,
                                 k_vjp_pullback,   k_vjp_positions<true>, k_vjp_positions<false>};
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 9 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(k[i], cudaFuncAttributeMaxDynamicSharedMemorySize, DENSE_SMEM);
  return e;
}

// The VJP of stage s: ly_s into a.ly_out (s > 0) or lam (s = 0), mu_B0 +=.
cudaError_t launch_f64_vjp(const VjpArgs& a, int stage, cudaStream_t s) {
  switch (stage) {
    case 0: return launch_stage<0>(a, s);
    case 1: return launch_stage<1>(a, s);
    case 2: return launch_stage<2>(a, s);
    case 3: return launch_stage<3>(a, s);
    case 4: return launch_stage<4>(a, s);
    case 5: return launch_stage<5>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace glemur
