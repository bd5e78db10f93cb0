// FP64 stage evaluation in two passes, without halo recomputation.
//
// On GB300 the FP64 pipe (2 lanes per SM per cycle, 1/64 of FP32) bounds
// the FP64 step, not HBM.  The fused stage kernel recomputes B on the tile
// halo (about 1.7 B evaluations per node) and the stage input on the
// halo-2 tile (about 2.5 combines per node); for FP64 those FP64
// instructions cost more than the extra HBM traffic of writing B once.  So
// the FP64 path evaluates each stage as
//   pass B:  B = G B0s / det G and 1/det G at every node, from the stage
//            input y_s (index-space differences: central inside,
//            second-order one-sided on boundary faces; eq. "B
//            transformation"); at interior nodes also the differences g_a
//            themselves (the current needs them again);
//   pass C:  the mimetic current J = (c_0 g_0 + c_1 g_1 + c_2 g_2)/det G
//            and u = J x B at interior nodes (eqs. "current discrete" to
//            "current matrix equation", eq. "magneto friction"), writing
//            k_s and, pointwise, the next stage input
//            y_{s+1} = d + sum_{j<=s} dt a_{s+1,j} k_j; the last stage
//            writes the fifth-order update and the embedded error instead.
// Pass C reads g_a (and 1/det G) as pass B stored them, side by side for a
// warp's nodes, rather than forming g_a again from the stage input's
// neighbours: 12 fewer FP64 additions per interior node and stage for 80
// bytes written and read (five 16-byte accesses each way), which HBM (used at
// well under a fifth of its bandwidth by these passes) absorbs.
// Each pass is one CTA per SM over equal shares of the node warps (see
// split64.cuh), launched as a programmatic dependent of the one before it.
// The per-CTA partials (Lambda, E_M, xi) keep the fused kernel's layout.
#include "split64.cuh"
#include "tma.cuh"

namespace glemur {

// Where interior node t's record for pass C starts: the records of a warp's
// 32 nodes lie side by side, value by value, so each of a record's five
// 16-byte accesses is one contiguous 512 bytes for the warp.  FP64 and memory
// instructions share an issue queue here, and a warp's accesses hold it for
// every 128-byte line they touch: with the records one after another (80
// bytes apart) those five touched 100 lines, of 200 in all, in a pass whose
// FP64 instructions take 864 cycles a node warp (129 x 97 x 75: 1029 -> 1019
// us an attempt).
__device__ __forceinline__ double2* node_record(const SplitArgs& a, int t) {
  return reinterpret_cast<double2*>(a.Gb) + ((size_t)(t >> 5) * 160 + (t & 31));
}

// det G, 1/det G and B = G B0s / det G at node n from its columns (eq. "B
// transformation"); B stored at node nw (n itself, or a periodic ghost node
// that carries n's B); with G the node's record for pass C (interior nodes).
// Returns the node's energy term zeta |B|^2 det G if `energy`.
template <bool WITH_G>
__device__ __forceinline__ double split_B_finish(const SplitArgs& a, int N, int n, int t, int i,
                                                 int j, int k, bool state, bool energy, int nw,
                                                 double g0[3], double g1[3], double g2[3]) {
  g0[0] += a.h2[0];
  g1[1] += a.h2[1];
  g2[2] += a.h2[2];
  const double det = det3(g0, g1, g2);
  if (le_zero(det))  // NaN: reported by the error norm
    atomicOr(&a.st->flags, state ? FLAG_COLLAPSED : FLAG_FOLDED_TRIAL);
  const double r = recip(det);
  if (WITH_G) {
    // the node's differences and 1/det G for pass C
    double2* q = node_record(a, t);
    q[0] = make_double2(g0[0], g0[1]);
    q[32] = make_double2(g0[2], g1[0]);
    q[64] = make_double2(g1[1], g1[2]);
    q[96] = make_double2(g2[0], g2[1]);
    q[128] = make_double2(g2[2], r);
  }
  const double b0 = __ldg(&a.B0s[n]), b1 = __ldg(&a.B0s[N + n]), b2 = __ldg(&a.B0s[2 * N + n]);
  double B[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    B[c] = (g0[c] * b0 + g1[c] * b1 + g2[c] * b2) * r;
    a.Bb[c * N + nw] = B[c];
  }
  if (!energy) return 0.0;
  // eq. "magnetic energy": zeta halves per boundary index coordinate
  const int nb = (i == 0 || i == a.nx - 1) + (j == 0 || j == a.ny - 1) + (k == 0 || k == a.nz - 1);
  const double zeta = nb == 0 ? 1.0 : nb == 1 ? 0.5 : nb == 2 ? 0.25 : 0.125;
  return zeta * dot3(B, B) * det;
}

// B at an interior node (central differences), storing G for pass C.
template <class LD>
__device__ __forceinline__ double split_B_interior(const SplitArgs& a,
                                                   const double* __restrict__ y, int N, int n,
                                                   int t, int i, int j, int k, bool state,
                                                   bool energy) {
  double g0[3], g1[3], g2[3];
  gcol<false, LD>(y, N, n, 1, 1, g0);
  gcol<false, LD>(y, N, n, a.nx, 1, g1);
  gcol<false, LD>(y, N, n, a.nx * a.ny, 1, g2);
  return split_B_finish<true>(a, N, n, t, i, j, k, state, energy, n, g0, g1, g2);
}

// B at a boundary node (or, with periodic z, at the partner of a ghost
// node): one-sided along the axes with sx, sy, sz != 0 (+1 low face, -1
// high face), central along the others; the variant is a template
// argument, so each runs its own FP64 instructions only.
template <bool OX, bool OY, bool OZ, class LD>
__device__ __forceinline__ double split_B_bvar(const SplitArgs& a, const double* __restrict__ y,
                                               int N, int n, int i, int j, int k, int sx,
                                               int sy, int sz, bool state, bool energy,
                                               int nw) {
  double g0[3], g1[3], g2[3];
  gcol<OX, LD>(y, N, n, 1, sx, g0);
  gcol<OY, LD>(y, N, n, a.nx, sy, g1);
  gcol<OZ, LD>(y, N, n, a.nx * a.ny, sz, g2);
  return split_B_finish<false>(a, N, n, 0, i, j, k, state, energy, nw, g0, g1, g2);
}

template <class LD>
__device__ __forceinline__ double split_B_boundary(const SplitArgs& a,
                                                   const double* __restrict__ y, int N, int n,
                                                   int i, int j, int k, int sx, int sy, int sz,
                                                   bool state, bool energy, int nw) {
#define GLEMUR_BVAR(X, Y, Z) \
  return split_B_bvar<X, Y, Z, LD>(a, y, N, n, i, j, k, sx, sy, sz, state, energy, nw)
  switch ((sx != 0) * 4 + (sy != 0) * 2 + (sz != 0)) {
    case 0: GLEMUR_BVAR(false, false, false);
    case 1: GLEMUR_BVAR(false, false, true);
    case 2: GLEMUR_BVAR(false, true, false);
    case 3: GLEMUR_BVAR(false, true, true);
    case 4: GLEMUR_BVAR(true, false, false);
    case 5: GLEMUR_BVAR(true, false, true);
    case 6: GLEMUR_BVAR(true, true, false);
    default: GLEMUR_BVAR(true, true, true);
  }
#undef GLEMUR_BVAR
}

// Pass B (stage s): B and 1/det G at every node, interior nodes (central
// differences) and boundary nodes (one-sided on their faces) in separate
// dense loops -- in one loop the compiler evaluates the one-sided variants
// under predicates for every node, and predicated-off FP64 instructions
// still take FP64-pipe slots; in the diagnostic launch also the energy
// partials (eq. "magnetic energy").
template <int S, class LD>
__device__ __forceinline__ void pass_B(const SplitArgs& a, int cur, double* red) {
  const int N = a.nx * a.ny * a.nz;
  const double* y = S == 0 ? a.d[cur] : a.ys[S & 1];
  const bool energy = S == 0 && a.diag;
  double eacc = 0.0;
  int tb, te;
  cta_range(a.inner_b, tb, te);
#pragma unroll 2  // two nodes' loads in flight (48 -> 64 registers, +1 % at 64^3)
  for (int t = tb + threadIdx.x; t < te; t += blockDim.x) {
    int i, j, k;
    const int n = interior_node(a, t, i, j, k);
    eacc += split_B_interior<LD>(a, y, N, n, t, i, j, k, S == 0, energy);
  }
  // the boundary nodes take up where the interior ones left off
  const int nw = blockDim.x >> 5;
  int wb = (threadIdx.x >> 5) - ((te - tb + 31) >> 5);
  while (wb < 0) wb += nw;
  cta_range(a.bound_b, tb, te, gridDim.x - 1 - blockIdx.x);
  for (int b = tb + 32 * wb + (threadIdx.x & 31); b < te; b += blockDim.x) {
    int i, j, k;
    const int n = boundary_node(a, b, i, j, k);
    if (n < 0) continue;
    const int sx = i == 0 ? 1 : (i == a.nx - 1 ? -1 : 0);
    const int sy = j == 0 ? 1 : (j == a.ny - 1 ? -1 : 0);
    const int sz = k == 0 ? 1 : (k == a.nz - 1 ? -1 : 0);
    if (a.periodic && sz != 0) {
      // a ghost plane carries its partner's B (section "Boundary
      // Conditions"); it is not part of the period's energy
      const int kk = sz > 0 ? a.nz - 2 : 1;
      const int np = (kk * a.ny + j) * a.nx + i;
      split_B_boundary<LD>(a, y, N, np, i, j, kk, sx, sy, 0, S == 0, false, n);
    } else {
      eacc += split_B_boundary<LD>(a, y, N, n, i, j, k, sx, sy, sz, S == 0, energy, n);
    }
  }
  pdl_trigger();
  if (energy) {
    const double v = block_reduce<false>(eacc, red);
    if (threadIdx.x == 0) put_partial(a, PART_E, v);
  }
}

template <int S>
__global__ void __launch_bounds__(DENSE_T, 1) k_split_B(const SplitArgs a) {
  int cur;
  if (!dense_start<S == 0>(a, cur)) return;
  __shared__ double red[32];
  pass_B<S, LdRO>(a, cur, red);
}

// One octilateral loop of the next-nearest-neighbour current (section
// "Next Nearest Neighbor Mimetic Approach") in the index surface spanned by
// P and Q: the eight in-plane neighbours V_1..V_8 at (along P, along Q) =
// (1,-1), (1,0), (1,1), (0,1), (-1,1), (-1,0), (-1,-1), (0,-1) with
// positions r_m.  Returns twice the circulation and twice the vector area
// (the common factor 1/2 cancels in M J = c):
//   circulation with edge-mean B (eq. "current discrete", eight edges):
//     sum_m (B_m + B_m+1)/2 . (r_m+1 - r_m) = sum_m B_m . e_m / 2 with
//     e_m = r_m+1 - r_m-1;
//   vector area (eq. "sum of eight triangles": four corner triangles plus
//   the inner quadrilateral): a surface spanning the loop, so its vector area
//   is the loop's, which the three quadrilaterals V_1 V_2 V_3 V_4, V_1 V_4
//   V_5 V_8 and V_5 V_6 V_7 V_8 give as half the cross products of their
//   diagonals: e_2 x e_3 + (r_5 - r_1) x (r_8 - r_4) + e_6 x e_7.
// The pass is bound by the FP64 pipe, so everything is in the e_m: e_2..e_7
// are differences of the displacement plus label offsets, r_5 - r_1 = e_2 +
// e_4, r_8 - r_4 = e_5 + e_7, and the loop closes: e_8 = -(e_2 + e_4 + e_6),
// e_1 = -(e_3 + e_5 + e_7).  81 FP64 instructions a loop, where positions
// relative to the node and eight cross products took 128, and one reciprocal
// for the solve's three divisions: 64^3, pass C of stage 3 217 -> 137 us; a
// 65^3 attempt 1.55 -> 1.05 ms.
template <int P, int Q, class LD>
__device__ __forceinline__ void nnn_loop(const SplitArgs& a, const double* __restrict__ y,
                                         int N, int n, double& circ2, double area2[3]) {
  const int sp = P == 0 ? 1 : (P == 1 ? a.nx : a.nx * a.ny);
  const int sq = Q == 0 ? 1 : (Q == 1 ? a.nx : a.nx * a.ny);
  const double hp = 0.5 * a.h2[P], hq = 0.5 * a.h2[Q];
  const int v[8] = {n + sp - sq, n + sp, n + sp + sq, n + sq,
                    n - sp + sq, n - sp, n - sp - sq, n - sq};
  double e2[3], e3[3], e4[3], e5[3], e6[3], e7[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double r[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) r[m] = LD::ld(&y[c * N + v[m]]);
    e2[c] = r[2] - r[0];
    e3[c] = r[3] - r[1];
    e4[c] = r[4] - r[2];
    e5[c] = r[5] - r[3];
    e6[c] = r[6] - r[4];
    e7[c] = r[7] - r[5];
  }
  e2[Q] += a.h2[Q];
  e3[P] -= hp;
  e3[Q] += hq;
  e4[P] -= a.h2[P];
  e5[P] -= hp;
  e5[Q] -= hq;
  e6[Q] -= a.h2[Q];
  e7[P] += hp;
  e7[Q] -= hq;
  double f[3], g[3];  // r_5 - r_1, r_8 - r_4
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    f[c] = e2[c] + e4[c];
    g[c] = e5[c] + e7[c];
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double* b = a.Bb + c * N;
    const double m1 = g[c] + e3[c], m8 = f[c] + e6[c];  // -e_1, -e_8
    circ2 = c == 0 ? LD::ld(&b[v[1]]) * e2[c] : fma(LD::ld(&b[v[1]]), e2[c], circ2);
    circ2 = fma(LD::ld(&b[v[2]]), e3[c], circ2);
    circ2 = fma(LD::ld(&b[v[3]]), e4[c], circ2);
    circ2 = fma(LD::ld(&b[v[4]]), e5[c], circ2);
    circ2 = fma(LD::ld(&b[v[5]]), e6[c], circ2);
    circ2 = fma(LD::ld(&b[v[6]]), e7[c], circ2);
    circ2 = fma(-LD::ld(&b[v[0]]), m1, circ2);
    circ2 = fma(-LD::ld(&b[v[7]]), m8, circ2);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
    double t = e2[c1] * e3[c2];
    t = fma(-e2[c2], e3[c1], t);
    t = fma(e6[c1], e7[c2], t);
    t = fma(-e6[c2], e7[c1], t);
    t = fma(f[c1], g[c2], t);
    area2[c] = fma(-f[c2], g[c1], t);
  }
}

// The next-nearest-neighbour current at interior node n and B there: the
// three loops (surfaces r = 0, 1, 2 spanned by p = r+1, q = r+2 mod 3,
// counter-clockwise about +r) give the rows of M and the entries of c in
// eq. "current matrix equation", solved by the adjugate,
// J = (c_0 a_1 x a_2 + c_1 a_2 x a_0 + c_2 a_0 x a_1) / det M.
template <class LD>
__device__ __forceinline__ void nnn_current(const SplitArgs& a, const double* __restrict__ y,
                                            int N, int n, double J[3], double B[3]) {
  double M[3][3], cr[3];
  nnn_loop<1, 2, LD>(a, y, N, n, cr[0], M[0]);
  nnn_loop<2, 0, LD>(a, y, N, n, cr[1], M[1]);
  nnn_loop<0, 1, LD>(a, y, N, n, cr[2], M[2]);
  double adj[3][3];  // adj[r] = a_{r+1} x a_{r+2}
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const double* u = M[(r + 1) % 3];
    const double* v = M[(r + 2) % 3];
    adj[r][0] = u[1] * v[2] - u[2] * v[1];
    adj[r][1] = u[2] * v[0] - u[0] * v[2];
    adj[r][2] = u[0] * v[1] - u[1] * v[0];
  }
  const double rM = recip(dot3(M[0], adj[0]));
#pragma unroll
  for (int c = 0; c < 3; ++c)
    J[c] = (cr[0] * adj[0][c] + cr[1] * adj[1][c] + cr[2] * adj[2][c]) * rM;
#pragma unroll
  for (int c = 0; c < 3; ++c) B[c] = LD::ld(&a.Bb[c * N + n]);
}

// Pass C (stage s): current and velocity at interior nodes; k_s and the
// next stage input, or (s = 5) the update, the error and k6.  CURL 0: the
// nearest-neighbour current; CURL 2: the next-nearest-neighbour current (a
// comparison option).
template <int S, int CURL, class LD>
__device__ __forceinline__ void pass_C(const SplitArgs& a, int cur, double* red) {
  constexpr bool FINAL = S == 5;
  const DevState* st = a.st;
  const int N = a.nx * a.ny * a.nz;
  const double* d = a.d[cur];
  double* dout = const_cast<double*>(a.d[cur ^ 1]);
  double* ynext = a.ys[(S + 1) & 1];
  double an[5];  // dt a_{S+1, j}: next stage input (non-final stages)
#pragma unroll
  for (int j = 0; j < 5; ++j) an[j] = (!FINAL && j <= S) ? LD::ld(&st->dta[S + 1][j]) : 0.0;
  Acc<double> acc;
  const int sy = a.nx, sz = a.nx * a.ny;
  int tb, te;
  cta_range(a.inner_c, tb, te);
  for (int t = tb + threadIdx.x; t < te; t += blockDim.x) {
    int i, j, k;
    const int n = interior_node(a, t, i, j, k);
    double J[3], B[3], u[3];
    if constexpr (CURL == 2) {
      nnn_current<LD>(a, S == 0 ? d : a.ys[S & 1], N, n, J, B);
    } else {
      double g0[3], g1[3], g2[3], P0[3], P1[3], P2[3];
      const double2* q = node_record(a, t);
      const double2 q0 = LD::ld2(q), q1 = LD::ld2(q + 32), q2 = LD::ld2(q + 64),
                    q3 = LD::ld2(q + 96), q4 = LD::ld2(q + 128);
      g0[0] = q0.x; g0[1] = q0.y; g0[2] = q1.x;
      g1[0] = q1.y; g1[1] = q2.x; g1[2] = q2.y;
      g2[0] = q3.x; g2[1] = q3.y; g2[2] = q4.x;
      const double r = q4.y;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double* b = a.Bb + c * N;
        P0[c] = LD::ld(&b[n + 1]) - LD::ld(&b[n - 1]);
        P1[c] = LD::ld(&b[n + sy]) - LD::ld(&b[n - sy]);
        P2[c] = LD::ld(&b[n + sz]) - LD::ld(&b[n - sz]);
        B[c] = LD::ld(&b[n]);
      }
      const double c0 = dot3_sub(P1, g2, P2, g1);
      const double c1 = dot3_sub(P2, g0, P0, g2);
      const double c2 = dot3_sub(P0, g1, P1, g0);
#pragma unroll
      for (int c = 0; c < 3; ++c) J[c] = (c0 * g0[c] + c1 * g1[c] + c2 * g2[c]) * r;
    }
    u[0] = J[1] * B[2] - J[2] * B[1];
    u[1] = J[2] * B[0] - J[0] * B[2];
    u[2] = J[0] * B[1] - J[1] * B[0];
    if (S == 0 && a.diag) acc.max_xi(dot3(u, u), dot3(B, B), dot3(J, J));
    split_emit<S, LD>(a, d, dout, ynext, an, N, n, k, u, acc);
  }
  pdl_trigger();
  if (FINAL) {
    const double v = block_reduce<true>(acc.lam, red);
    if (threadIdx.x == 0) put_partial(a, PART_LAMBDA, v);
  }
  if (S == 0 && a.diag) {
    double v = block_reduce<true>(acc.xi2(), red);
    if (threadIdx.x == 0) put_partial(a, PART_XI2, v);
    v = block_reduce<true>(acc.xis2(), red);
    if (threadIdx.x == 0) put_partial(a, PART_XIS2, v);
  }
}

template <int S, int CURL>
__global__ void __launch_bounds__(CURL == 2 ? DENSE_T2 : DENSE_T, 1) k_split_C(const SplitArgs a) {
  int cur;
  if (!dense_start<false>(a, cur)) return;
  __shared__ double red[32];
  pass_C<S, CURL, LdRO>(a, cur, red);
}

// ---- persistent attempts ------------------------------------------------
//
// One cooperative launch runs whole attempts: the twelve passes and the
// step control, with no kernel boundary between them.  Each CTA keeps the
// node ranges it has in the per-pass kernels (one CTA per SM, all resident),
// and instead of a grid-wide boundary after each pass it waits only for the
// node planes its next pass reads:
//   pass B of stage s at plane p reads the stage input at planes p-2..p+2,
//     written by pass C of stage s-1 (the one-sided boundary stencil reaches
//     two planes; the same wait orders pass C's earlier reads of the B, G
//     and stage-input buffers that pass B now overwrites);
//   pass C of stage s at plane p reads B at planes p-1..p+1 from pass B.
// A CTA publishes a finished pass by adding one to the completion counter
// of every plane its work touched (after a fence that makes its writes
// visible at device scope); a wait reads the counters through L2 until they
// reach (CTAs touching the plane) x (passes done).  The last CTA to finish
// an attempt runs the step control and releases the others; the next
// attempt's first pass reads the state the control selected.  All data
// another CTA may have written is loaded through L2 (LdL2).  Every wait is
// bounded: after 2 s it raises FLAG_TIMEOUT and status TIMEOUT and the CTA
// leaves; the others see the flag in their own waits and leave too.
// Results are bit-identical to the per-pass kernels: each node's
// arithmetic is the same.  Measured on GB300 it is slower than the per-pass
// kernels chained by programmatic dependent launch (16^3: 76 against 56 us an
// attempt, 64^3: 344 against 302), so it runs only on request
// (GLEMUR_PERSIST=1).

constexpr unsigned long long PERSIST_WAIT_NS = 2000000000ull;

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Spin until *p >= want (bounded); false on timeout or abort.
__device__ __forceinline__ bool persist_wait(const int* p, int want, DevState* st,
                                             unsigned long long t0) {
  for (;;) {
    if (ld_acquire(p) >= want) return true;
    if (ld_acquire(&st->flags) & FLAG_TIMEOUT) return false;
    if (globaltimer_ns() - t0 > PERSIST_WAIT_NS) return false;
  }
}

// The t-th plane of the intervals [lo - r, hi + r] (clipped to [kmin,
// kmax]) taken in turn, or -1 past their end.
__device__ __forceinline__ int persist_plane_at(const int* iv, int nint, int r, int kmin,
                                                int kmax, int t) {
  for (int q = 0; q < nint; ++q) {
    const int lo = iv[2 * q], hi = iv[2 * q + 1];
    if (lo > hi) continue;
    const int a = max(lo - r, kmin), b = min(hi + r, kmax);
    if (a > b) continue;
    if (t <= b - a) return a + t;
    t -= b - a + 1;
  }
  return -1;
}

__device__ __forceinline__ void persist_abort(DevState* st) {
  atomicOr(&st->flags, FLAG_TIMEOUT);
  atomicExch(&st->status, ST_TIMEOUT);
}

// The whole CTA: wait for the counters of planes [lo - r, hi + r] (clipped
// to [kmin, kmax]) of every interval to reach touch x phases, one thread
// per plane (a second round of planes per thread where there are more
// planes than threads); true for every thread when all are reached.
__device__ __forceinline__ bool persist_wait_planes(const int* iv, int nint, int r, int kmin,
                                                    int kmax, const int* cnt, const int* touch,
                                                    int phases, DevState* st) {
  const unsigned long long t0 = globaltimer_ns();
  bool ok = true;
  for (int t = threadIdx.x;; t += blockDim.x) {
    const int p = persist_plane_at(iv, nint, r, kmin, kmax, t);
    if (p < 0) break;
    ok = ok && persist_wait(&cnt[p], touch[p] * phases, st, t0);
  }
  return __syncthreads_and(ok);
}

// The whole CTA, after its pass: one completion for every plane of every
// interval, one thread per plane, each after a device-scope fence (the
// barrier before it makes the CTA's writes part of what the fence orders).
__device__ __forceinline__ void persist_publish(const int* iv, int nint, int* cnt) {
  __syncthreads();
  for (int t = threadIdx.x;; t += blockDim.x) {
    const int p = persist_plane_at(iv, nint, 0, 0, 1 << 30, t);
    if (p < 0) break;
    __threadfence();
    atomicAdd(&cnt[p], 1);
  }
}

template <int CURL>
__global__ void __launch_bounds__(CURL == 2 ? DENSE_T2 : DENSE_T, 1)
    k_attempts_persist(const SplitArgs a, const PersistArgs pa) {
  __shared__ double red[32];
  __shared__ double sh[96];
  __shared__ int ok, last;
  DevState* st = a.st;
  const int G = gridDim.x;
  const int* ivB = pa.ivB + blockIdx.x * 2 * PERSIST_BI;
  const int* ivC = pa.ivC + blockIdx.x * 2;
  for (int att = 0; att < pa.n_attempts; ++att) {
    if (LdL2::ldi(&st->status) != ST_OK ||
        __ldcg(&st->n_accept) >= __ldcg(&st->target))
      return;
    const int cur = LdL2::ldi(&st->cur);
#define GLEMUR_PERSIST_STAGE(SS)                                                          \
    if (SS > 0 && !persist_wait_planes(ivB, PERSIST_BI, 2, 1, a.nz - 2, pa.cntC,          \
                                       pa.touchC, att * 6 + SS, st)) {                    \
      if (threadIdx.x == 0) persist_abort(st);                                            \
      return;                                                                             \
    }                                                                                     \
    pass_B<SS, LdL2>(a, cur, red);                                                        \
    if (!(SS == 2 && (int)blockIdx.x == pa.test_withhold))                                \
      persist_publish(ivB, PERSIST_BI, pa.cntB);                                          \
    if (!persist_wait_planes(ivC, 1, 1, 0, a.nz - 1, pa.cntB, pa.touchB,                  \
                             att * 6 + SS + 1, st)) {                                     \
      if (threadIdx.x == 0) persist_abort(st);                                            \
      return;                                                                             \
    }                                                                                     \
    pass_C<SS, CURL, LdL2>(a, cur, red);                                                  \
    persist_publish(ivC, 1, pa.cntC);
    GLEMUR_PERSIST_STAGE(0)
    GLEMUR_PERSIST_STAGE(1)
    GLEMUR_PERSIST_STAGE(2)
    GLEMUR_PERSIST_STAGE(3)
    GLEMUR_PERSIST_STAGE(4)
    GLEMUR_PERSIST_STAGE(5)
#undef GLEMUR_PERSIST_STAGE
    // end of the attempt: the last CTA to arrive runs the step control
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned old = atomicAdd(&pa.bar[0], 1u);
      last = old == (unsigned)(G * (att + 1) - 1);
    }
    __syncthreads();
    if (last) {
      __threadfence();
      control_block<LdCoherent>(st, a.part, a.nblocks, a.diag, pa.dtlog, sh, [] {});
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        atomicExch(&pa.bar[1], (unsigned)(att + 1));
      }
    } else {
      if (threadIdx.x == 0) {
        const unsigned long long t0 = globaltimer_ns();
        ok = 1;
        while (ld_acquire(&pa.bar[1]) < (unsigned)(att + 1)) {
          if ((ld_acquire(&st->flags) & FLAG_TIMEOUT) ||
              globaltimer_ns() - t0 > PERSIST_WAIT_NS) {
            ok = 0;
            break;
          }
        }
        __threadfence();
      }
      __syncthreads();
      if (!ok) {
        if (threadIdx.x == 0) persist_abort(st);
        return;
      }
    }
    __syncthreads();
  }
}

// The persistent kernel's launch (cooperative: every CTA resident, or the
// launch fails).
cudaError_t launch_f64_persist(const SplitArgs& a, const PersistArgs& pa, int grid, int curl,
                               cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(a.threads_b);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (curl == 2) return cudaLaunchKernelEx(&cfg, k_attempts_persist<2>, a, pa);
  return cudaLaunchKernelEx(&cfg, k_attempts_persist<0>, a, pa);
}

// Let the passes ask for DENSE_SMEM.
cudaError_t prepare_f64_split() {
  void (*k[18])(const SplitArgs) = {
      k_split_B<0>,    k_split_B<1>,    k_split_B<2>,    k_split_B<3>,    k_split_B<4>,
      k_split_B<5>,    k_split_C<0, 0>, k_split_C<1, 0>, k_split_C<2, 0>, k_split_C<3, 0>,
      k_split_C<4, 0>, k_split_C<5, 0>, k_split_C<0, 2>, k_split_C<1, 2>, k_split_C<2, 2>,
      k_split_C<3, 2>, k_split_C<4, 2>, k_split_C<5, 2>};
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 18 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(k[i], cudaFuncAttributeMaxDynamicSharedMemorySize, DENSE_SMEM);
  return e;
}

// Launch the passes of stage s with the current `curl` (0 nearest, 2
// next-nearest neighbours); pass B alone without pass_c.
cudaError_t launch_f64_split(const SplitArgs& a, int stage, cudaStream_t s, int curl,
                             bool pass_c) {
  if (stage < 0 || stage > 5 || (curl != 0 && curl != 2)) return cudaErrorInvalidValue;
  const dim3 gb(a.grid_b), gc(a.grid_c), tb(a.threads_b), tc(a.threads_c);
  cudaError_t e = cudaSuccess;
#define GLEMUR_SPLIT_CASE(SS)                                                          \
  case SS:                                                                             \
    e = launch_pdl(k_split_B<SS>, gb, tb, DENSE_SMEM, s, a);                           \
    if (e == cudaSuccess && pass_c)                                                    \
      e = curl == 2 ? launch_pdl(k_split_C<SS, 2>, gc, tc, DENSE_SMEM, s, a)           \
                    : launch_pdl(k_split_C<SS, 0>, gc, tc, DENSE_SMEM, s, a);          \
    break;
  switch (stage) {
    GLEMUR_SPLIT_CASE(0)
    GLEMUR_SPLIT_CASE(1)
    GLEMUR_SPLIT_CASE(2)
    GLEMUR_SPLIT_CASE(3)
    GLEMUR_SPLIT_CASE(4)
    GLEMUR_SPLIT_CASE(5)
    default:
      return cudaErrorInvalidValue;
  }
#undef GLEMUR_SPLIT_CASE
  return e;
}

}  // namespace glemur
