// What the dense FP64 kernels share (the two-pass stages and the direct
// stage): node ranges of a one-wave grid, the loads, the per-CTA partials and
// the output of a stage at a node.
#pragma once

#include "control.cuh"
#include "stage_kernels.cuh"

namespace glemur {

// How the passes load data that another CTA of the same launch may have
// written: the per-pass kernels use the read-only path (__ldg) -- each pass
// only reads what earlier launches wrote -- while the persistent attempt
// kernel, whose CTAs read each other's results within one launch, uses
// ordinary (weak) global loads: the read-only path may keep lines from an
// earlier pass, whereas weak loads that follow, in causality order, an
// acquire that observed the writer's release must return the released
// values (the PTX memory model; the waits below are exactly that pattern).
// The loads are volatile asm so that the compiler neither merges loads of
// one address from different passes nor moves them across the waits.
struct LdRO {
  __device__ static __forceinline__ double ld(const double* p) { return __ldg(p); }
  __device__ static __forceinline__ double2 ld2(const double2* p) { return __ldg(p); }
  __device__ static __forceinline__ int ldi(const int* p) { return *p; }
};
struct LdL2 {
  __device__ static __forceinline__ double ld(const double* p) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
  }
  __device__ static __forceinline__ double2 ld2(const double2* p) {
    double2 v;
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
  }
  __device__ static __forceinline__ int ldi(const int* p) {
    int v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
  }
};

// How the dense passes are spread.  The FP64 pipe belongs to an SM's
// quarter: it takes a warp instruction every 64 cycles, and a single warp
// keeps it 97 % busy (a dependent DFMA takes 67).  So what counts is that
// every quarter gets the same number of node warps.  A pass runs one CTA per
// SM, each over an equal range of whole warps of nodes, and the CTA's warps
// (a multiple of four, warp w on quarter w mod 4) take the range's node warps
// in turn, so the quarters of an SM differ by one at most.  (Four CTAs of
// eight warps per SM, each with twelve node warps, gave the first quarter 16
// where the mean is 12.25: 64^3.)  Small grids get no more warps per CTA than
// an SM's share, four at least, so that one node warp has a quarter to
// itself.  Together with the variant groups of boundary_node, index division
// by multiplication and no 64-bit division, an attempt went from 95 to 56 us
// at 16^3, 106 to 74 at 33^3, 211 to 155 at 48^3 and 349 to 302 at 64^3.
//
// CTA b's range [begin, end) of the nodes w shares out.  (Pass B takes the
// boundary's in reverse, so that one CTA does not get both extra warps.)
__device__ __forceinline__ void cta_range(const WarpShare& w, int& begin, int& end,
                                          int b = blockIdx.x) {
  begin = 32 * (b * w.each + min(b, w.extra));
  end = min(begin + 32 * (w.each + (b < w.extra)), w.n);
}

// Interior nodes enumerated densely: t in [0, (nx-2)(ny-2)(nz-2)) -> node.
// A warp then holds 32 interior nodes, so the interior code (central
// differences only) runs with no boundary lanes in it.
template <class Args>
__device__ __forceinline__ int interior_node(const Args& a, int t, int& i, int& j, int& k) {
  const int r = a.dx.div(t), q = a.dy.div(r);
  i = 1 + t - r * a.dx.d;
  j = 1 + r - q * a.dy.d;
  k = 1 + q;
  return (k * a.ny + j) * a.nx + i;
}

// Boundary nodes enumerated in groups of one stencil variant each (which
// axes are one-sided): the inner parts of the two z faces, the two y faces
// and the two x faces (one boundary index coordinate), the edges along x, y
// and z (two), then the eight corners.  Every group starts a new warp, so no
// warp runs more than one variant: a warp with n of them takes its quarter of
// the SM n times as long, and with the groups packed one warp at their end
// had four -- 14000 cycles of a 33000-cycle pass B at 64^3, most of it at
// 16^3.  b in [0, boundary_items); -1 for the idle lanes of a group's last
// warp.  The host's persistent-kernel plan mirrors this order.
template <class Args>
__device__ __forceinline__ int boundary_node(const Args& a, int b, int& i, int& j, int& k) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int xi = nx - 2, yi = ny - 2, zi = nz - 2;
  const int fz = xi * yi, fy = xi * zi, fx = yi * zi;
  bool idle;
  if (b < pad32(2 * fz)) {
    idle = b >= 2 * fz;
    k = b < fz ? 0 : nz - 1;
    const int r = b < fz ? b : b - fz, q = a.dx.div(r);
    i = 1 + r - q * xi;
    j = 1 + q;
  } else if ((b -= pad32(2 * fz)) < pad32(2 * fy)) {
    idle = b >= 2 * fy;
    j = b < fy ? 0 : ny - 1;
    const int r = b < fy ? b : b - fy, q = a.dx.div(r);
    i = 1 + r - q * xi;
    k = 1 + q;
  } else if ((b -= pad32(2 * fy)) < pad32(2 * fx)) {
    idle = b >= 2 * fx;
    i = b < fx ? 0 : nx - 1;
    const int r = b < fx ? b : b - fx, q = a.dy.div(r);
    j = 1 + r - q * yi;
    k = 1 + q;
  } else if ((b -= pad32(2 * fx)) < pad32(4 * xi)) {
    idle = b >= 4 * xi;
    const int e = a.dx.div(b);
    i = 1 + b - e * xi;
    j = (e & 1) ? ny - 1 : 0;
    k = (e & 2) ? nz - 1 : 0;
  } else if ((b -= pad32(4 * xi)) < pad32(4 * yi)) {
    idle = b >= 4 * yi;
    const int e = a.dy.div(b);
    j = 1 + b - e * yi;
    i = (e & 1) ? nx - 1 : 0;
    k = (e & 2) ? nz - 1 : 0;
  } else if ((b -= pad32(4 * yi)) < pad32(4 * zi)) {
    idle = b >= 4 * zi;
    const int e = a.dz.div(b);
    k = 1 + b - e * zi;
    i = (e & 1) ? nx - 1 : 0;
    j = (e & 2) ? ny - 1 : 0;
  } else {
    b -= pad32(4 * zi);
    idle = b >= 8;
    i = (b & 1) ? nx - 1 : 0;
    j = (b & 2) ? ny - 1 : 0;
    k = (b & 4) ? nz - 1 : 0;
  }
  return idle ? -1 : (k * ny + j) * nx + i;
}

// One column of G from the stage input y along an axis of node stride
// `stride`, without the 2 h_a e_a term.  ONE = false: the central
// difference v(n+s) - v(n-s).  ONE = true: the second-order one-sided
// difference into the domain, (4 v(n+s) - 3 v(n)) - v(n+2s) at the low face
// (sg = +1) and (3 v(n) - 4 v(n-s)) + v(n-2s) at the high face (sg = -1),
// both as sg times the first form with s -> sg s: the signs ride on
// constants chosen by a select (multiplying by -1 is exact), so both faces
// run the same three FP64 instructions per component.
template <bool ONE, class LD>
__device__ __forceinline__ void gcol(const double* __restrict__ y, int N, int n, int stride,
                                     int sg, double out[3]) {
  const int s = sg * stride;
  const double c4 = sg > 0 ? 4.0 : -4.0, m3 = sg > 0 ? -3.0 : 3.0, m1 = sg > 0 ? -1.0 : 1.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double* v = y + c * N;
    if (!ONE)
      out[c] = LD::ld(&v[n + stride]) - LD::ld(&v[n - stride]);
    else
      out[c] = fma(m1, LD::ld(&v[n + 2 * s]), fma(c4, LD::ld(&v[n + s]), m3 * LD::ld(&v[n])));
  }
}

// The start of a dense pass: false if stepping has stopped.  FIRST: the
// first kernel of an attempt, which waits before it reads anything; the
// others read the control state ahead of the wait (see launch_pdl).
template <bool FIRST>
__device__ __forceinline__ bool dense_start(const SplitArgs& a, int& cur) {
  if (FIRST) pdl_wait();
  const DevState* st = a.st;
  const bool stop = !a.force && (st->status != ST_OK || st->n_accept >= st->target);
  cur = st->cur;
  if (!FIRST) pdl_wait();
  return !stop;
}

// This CTA's partial of kind `kind`; the slots of the partial stride beyond
// this launch's grid are zeroed (neutral for the sums and for the maxima of
// non-negative values), so a pass with fewer CTAs than the stride leaves no
// stale slot behind.
__device__ __forceinline__ void put_partial(const SplitArgs& a, int kind, double v) {
  double* p = a.part + kind * a.nblocks;
  p[blockIdx.x] = v;
  for (int b = gridDim.x + blockIdx.x; b < a.nblocks; b += gridDim.x) p[b] = 0.0;
}

__device__ __forceinline__ void cross64(const double a[3], const double b[3], double o[3]) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

// a.b - c.d as one multiply and five FMAs (one FP64 instruction fewer than
// two dot products and a subtraction)
__device__ __forceinline__ double dot3_sub(const double a[3], const double b[3],
                                           const double c[3], const double d[3]) {
  double t = a[0] * b[0];
  t = fma(a[1], b[1], t);
  t = fma(a[2], b[2], t);
  t = fma(-c[0], d[0], t);
  t = fma(-c[1], d[1], t);
  return fma(-c[2], d[2], t);
}

// Stage S's output at interior node n of plane k from its velocity u: k_S and
// the next stage input y_{S+1} = d + sum_{j<=S} dt a_{S+1,j} k_j, or (S = 5)
// the fifth-order update, the embedded error and k6.
template <int S, class LD>
__device__ __forceinline__ void split_emit(const SplitArgs& a, const double* d, double* dout,
                                           double* ynext, const double an[5], int N, int n,
                                           int k, const double u[3], Acc<double>& acc) {
  constexpr bool FINAL = S == 5;
  const DevState* st = a.st;
  const int sz = a.nx * a.ny;
  if (!FINAL) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a.k[S][c * N + n] = u[c];
      // next stage input y_{S+1} = d + sum_{j<=S} dt a_{S+1,j} k_j
      double v = LD::ld(&d[c * N + n]);
#pragma unroll
      for (int jj = 0; jj < S; ++jj) v = fma(an[jj], LD::ld(&a.k[jj][c * N + n]), v);
      v = fma(an[S], u[c], v);
      ynext[c * N + n] = v;
      // periodic in z: the ghost of an end plane holds the same
      // displacement (its position differs by the period)
      if (a.periodic && (k == 1 || k == a.nz - 2))
        ynext[c * N + n + (k == 1 ? 1 : -1) * (a.nz - 2) * sz] = v;
    }
  } else {
    const double b0 = LD::ld(&st->dtb[0]), b2 = LD::ld(&st->dtb[2]),
                 b3 = LD::ld(&st->dtb[3]), b5 = LD::ld(&st->dtb[5]);
    const double e0 = LD::ld(&st->dte[0]), e2 = LD::ld(&st->dte[2]),
                 e3 = LD::ld(&st->dte[3]), e4 = LD::ld(&st->dte[4]),
                 e5 = LD::ld(&st->dte[5]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double k1 = LD::ld(&a.k[0][c * N + n]), k3 = LD::ld(&a.k[2][c * N + n]),
                   k4 = LD::ld(&a.k[3][c * N + n]), k5 = LD::ld(&a.k[4][c * N + n]);
      double up = b0 * k1;
      up = fma(b2, k3, up);
      up = fma(b3, k4, up);
      up = fma(b5, u[c], up);
      double er = e0 * k1;
      er = fma(e2, k3, er);
      er = fma(e3, k4, er);
      er = fma(e4, k5, er);
      er = fma(e5, u[c], er);
      const double dn = LD::ld(&d[c * N + n]) + up;
      dout[c * N + n] = dn;
      if (a.periodic && (k == 1 || k == a.nz - 2))
        dout[c * N + n + (k == 1 ? 1 : -1) * (a.nz - 2) * sz] = dn;
      acc.max_lam(fabs(er));
      if (a.k[5]) a.k[5][c * N + n] = u[c];
    }
  }
}

}  // namespace glemur
