// Mixed-precision mimetic stage kernel: a CTA owns a MX x WARPS column tile
// (two x-neighbouring output columns per thread) and marches along z, one B
// plane per iteration, with what the current needs along z carried in
// registers.
//
// Iteration q of a CTA forms B = G B0s / det G (eq. "B transformation") at
// plane q of the tile + halo 1 and the current and velocity (section
// "Mimetic Operators", eq. "magneto friction") at plane q - 1 of the tile's
// own nodes.  A thread forms B at its own nodes of every plane, so it already
// holds what the current of plane q - 1 needs there: the columns of G and
// 1/det G from iteration q - 1, and B of planes q - 2, q - 1, q.  Shared
// memory is read for the in-plane neighbours only, and a plane of B lives for
// one iteration (two slots).  The halo points of B (a row below and above the
// tile, a pair of columns left and right) are the second pairs of three
// warps, another three in every CTA so that the SM's schedulers share them.
//
// What bounds it: at 384^3 HBM (84 B per node-stage are read and written, 85 %
// of the measured copy bandwidth), at 128^3 and below, where the fields fit
// in L2, instruction issue and the latency of an iteration.  So a thread's
// two nodes go through the arithmetic as one packed FP32 pair
// (fma.rn.f32x2 and kin: one issue slot for both), through 8-byte shared and
// global accesses, and share every index, branch and barrier: 344 issue
// slots per node in stage 4 where one node per thread on 32-wide tiles took
// 542 with the same carried registers, and 564 re-reading G and B from
// shared memory.  An attempt: 384^3 7.16 -> 4.87 ms, 128^3 351 -> 243 us,
// 48^3 70 -> 59 us, 101 x 90 x 75 (plain copies) 197 -> 159 us (the last 12
// and 15 us by choose_kz_march's planes per CTA).  Measured and
// left: one column per thread (384^3 6.2 ms at 24 warps per SM, 6.5 ms at
// 16), 16 or 4 warps per CTA (5.7, 5.6 ms).  128 registers, 2 CTAs per SM.
//
// The stage input y_s (halo 2) and B0s (halo 1) arrive in rings of planes,
// two iterations ahead of their use.  Two loaders fill the same layout
// (component-major planes MP floats wide whose column 4 is the tile's first):
//   TMA = true   cp.async.bulk.tensor boxes of all three components, which
//                must start on a 16-byte boundary (hence 4 columns left of
//                the tile) and need rows of a multiple of 16 bytes, so nx a
//                multiple of 4;
//   TMA = false  4-byte cp.async copies of the needed points, any grid
//                (and 4-byte global accesses: rows may start anywhere).
// The centre values (d, k_j) of a thread's nodes are loaded one plane ahead.
#pragma once

#include "stage_kernels.cuh"

namespace glemur {

constexpr int MX = 64;      // tile width (nodes)
constexpr int MP = MX + 8;  // row pitch of the planes in shared memory (floats)

template <int WARPS>
struct MarchGeo {
  static constexpr int NTH = 32 * WARPS;             // threads per CTA
  static constexpr int TH = WARPS;                   // tile height (nodes)
  static constexpr int YHt = TH + 4;                 // stage-input box height (halo 2)
  static constexpr int YCSt = MP * YHt, YPLt = 3 * YCSt;
  static constexpr int YSTRt = (YPLt * 4 + 127) / 128 * 32;  // ring slot stride (floats)
  static constexpr int ZHt = TH + 2;                 // B0 box height (halo 1), B plane
  static constexpr int ZCSt = MP * ZHt, ZPLt = 3 * ZCSt;
  static constexpr int ZSTRt = (ZPLt * 4 + 127) / 128 * 32;  // slot stride (floats)
  static constexpr unsigned YBYTESt = YPLt * 4, ZBYTESt = ZPLt * 4;
  // planes q - 1, q, q + 1 in use, q + 2 and q + 3 in flight (the slot of
  // q - 2 is the one q + 3 goes to; at the last plane nothing is in flight
  // and q - 2 is still there for the one-sided difference)
  static constexpr int YRING = 5, ZRING = 3;
  // points a thread copies per plane without TMA (halo 2, halo 1)
  static constexpr int LWY = MX + 4, LPY = (LWY * YHt + NTH - 1) / NTH;
  static constexpr int LWZ = MX + 2, LPZ = (LWZ * ZHt + NTH - 1) / NTH;
  static constexpr size_t smem_bytes() {
    return 128 + (size_t)(YRING * YSTRt + (ZRING + 2) * ZSTRt) * 4;
  }
};

// ---- packed FP32 pairs

typedef unsigned long long f2;
__device__ __forceinline__ f2 f2pack(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2split(f2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 f2dup(float a) { return f2pack(a, a); }
__device__ __forceinline__ f2 f2add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 f2neg(f2 a) { return f2mul(a, 0xbf800000bf800000ull); }  // (-1, -1)
__device__ __forceinline__ f2 f2dot(const f2 a[3], const f2 b[3]) {
  return f2fma(a[2], b[2], f2fma(a[1], b[1], f2mul(a[0], b[0])));
}
__device__ __forceinline__ f2 f2lds(const float* p) { return *reinterpret_cast<const f2*>(p); }
__device__ __forceinline__ void f2sts(float* p, f2 v) { *reinterpret_cast<f2*>(p) = v; }
// a + b = s + e exactly
__device__ __forceinline__ void f2two_diff(f2 a, f2 b, f2& s, f2& e) {  // of a - b
  s = f2sub(a, b);
  const f2 bb = f2sub(s, a);
  e = f2sub(f2sub(a, f2sub(s, bb)), f2add(b, bb));
}
__device__ __forceinline__ void f2two_sum(f2 a, f2 b, f2& s, f2& e) {
  s = f2add(a, b);
  const f2 bb = f2sub(s, a);
  e = f2add(f2sub(a, f2sub(s, bb)), f2sub(b, bb));
}

// det3 of stage_kernels.cuh (float-float, rounded once), operation for
// operation, on a pair.  The error of a product a b rounded to p comes as
// its negative, fma(-a, b, p).
__device__ __forceinline__ f2 f2det3(const f2 g0[3], const f2 g1[3], const f2 g2[3]) {
  f2 th[3], ntl[3];
  constexpr int ia[3] = {1, 2, 0}, ib[3] = {2, 0, 1};
  f2 n1[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) n1[r] = f2neg(g1[r]);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const f2 p = f2mul(g1[ia[r]], g2[ib[r]]), npe = f2fma(n1[ia[r]], g2[ib[r]], p);
    const f2 q = f2mul(g1[ib[r]], g2[ia[r]]), nqe = f2fma(n1[ib[r]], g2[ia[r]], q);
    f2 s, se;
    f2two_diff(p, q, s, se);
    const f2 lo = f2add(se, f2sub(nqe, npe));
    const f2 n0 = f2neg(g0[r]);
    th[r] = f2mul(g0[r], s);
    ntl[r] = f2fma(n0, lo, f2fma(n0, s, th[r]));
  }
  f2 s01, e01, s, e2;
  f2two_sum(th[0], th[1], s01, e01);
  f2two_sum(s01, th[2], s, e2);
  const f2 lo = f2sub(f2add(e01, e2), f2add(f2add(ntl[0], ntl[1]), ntl[2]));
  return f2add(s, lo);
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int LEFT>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// ---- points and planes

// A pair of B points (x, x + 1): its index in the B0 and B planes (component
// 0) -- one row more in the stage-input planes -- and what does not change
// from plane to plane.  code: which of the two are needed and lie in the grid
// (bits 0, 1), which lies on an x face (2, 3; at most one, with the step
// xs = +-1 into the domain), the row on the lower or upper y face (4, 5).
struct MarchPair {
  int z0, code, xs;
  template <class Gm>
  __device__ __forceinline__ void init(int col, int row, int i0, int j0, int nx, int ny) {
    const int gi = i0 + col, gj = j0 - 1 + row;  // col: -2, 0, 2, .. MX; row: 0 .. TH + 1
    z0 = row * MP + col + 4;
    code = xs = 0;
    if (gj < 0 || gj >= ny) return;
    // left of the tile only the second point is needed, right of it the first
    code = (col >= 0 && gi < nx) | (col < MX && gi + 1 >= 0 && gi + 1 < nx) << 1;
    if (code == 0) return;
    xs = gi == 0 ? 1 : -1;
    code |= (gi == 0 || gi == nx - 1) << 2 | (gi + 1 == nx - 1) << 3 | (gj == 0) << 4 |
            (gj == ny - 1) << 5;
  }
  __device__ __forceinline__ bool any() const { return (code & 3) != 0; }
  __device__ __forceinline__ bool xface() const { return (code & 12) != 0; }
};

// Stage-input planes around plane q in shared memory.
struct MarchRing {
  const float* ym2;
  const float* ym;
  const float* yq;
  const float* yp;
  const float* yp2;
};

// The one-sided second-order difference sgn (4 p1 - 3 p0 - p2).
__device__ __forceinline__ float march_side(float p0, float p1, float p2, float sgn) {
  return sgn * ((4.0f * p1 - 3.0f * p0) - p2);
}

// Columns of G (index-space differences of x, central inside, one-sided on
// the faces), det G, 1/det G and B at a pair of points of plane q (sz: z
// stencil, 0 central, 1 lower face, 2 upper face); yc: the stage input there
// one plane below (at a thread's own nodes the centre of its next output).
template <class Gm>
__device__ __forceinline__ void march_B(const StageArgs<float>& a, const MarchPair& pt, int sz,
                                        const MarchRing& R, const float* __restrict__ zq,
                                        f2 g[3][3], f2& det, f2& r, f2 B[3], f2 yc[3]) {
  constexpr int CS = Gm::YCSt, ZC = Gm::ZCSt;
  const int x0 = pt.z0 + MP;
  const float* yq = R.yq + x0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float c0, c1;
    f2split(f2lds(yq + c * CS), c0, c1);
    g[0][c] = f2pack(c1 - yq[c * CS - 1], yq[c * CS + 2] - c0);
    g[1][c] = f2sub(f2lds(yq + c * CS + MP), f2lds(yq + c * CS - MP));
    yc[c] = f2lds(R.ym + x0 + c * CS);
    g[2][c] = f2sub(f2lds(R.yp + x0 + c * CS), yc[c]);
  }
  // One-sided along the axis of a face.  x faces are lanes of one warp in each
  // row of the first and last tile; y faces are whole rows, z faces planes.
  if (pt.xface()) {
    const float* v = yq + (pt.code >> 3 & 1);
    const float sg = (float)pt.xs;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float o = march_side(v[c * CS], v[c * CS + pt.xs], v[c * CS + 2 * pt.xs], sg);
      float e0, e1;
      f2split(g[0][c], e0, e1);
      g[0][c] = f2pack(pt.code & 4 ? o : e0, pt.code & 8 ? o : e1);
    }
  }
  if (pt.code >> 4) {
    const int st = pt.code & 16 ? MP : -MP;
    const float sg = pt.code & 16 ? 1.0f : -1.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float* v = yq + c * CS;
      g[1][c] = f2pack(march_side(v[0], v[st], v[2 * st], sg),
                       march_side(v[1], v[st + 1], v[2 * st + 1], sg));
    }
  }
  if (sz) {
    const float* q1 = (sz == 1 ? R.yp : R.ym) + x0;
    const float* q2 = (sz == 1 ? R.yp2 : R.ym2) + x0;
    const float sg = sz == 1 ? 1.0f : -1.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float* v = yq + c * CS;
      g[2][c] = f2pack(march_side(v[0], q1[c * CS], q2[c * CS], sg),
                       march_side(v[1], q1[c * CS + 1], q2[c * CS + 1], sg));
    }
  }
#pragma unroll
  for (int e = 0; e < 3; ++e) g[e][e] = f2add(g[e][e], f2dup(a.h2f[e]));
  det = f2det3(g[0], g[1], g[2]);
  float d0, d1;
  f2split(det, d0, d1);
  r = f2pack(recip(d0), recip(d1));
  const float* z = zq + pt.z0;
  const f2 b0 = f2lds(z), b1 = f2lds(z + ZC), b2 = f2lds(z + 2 * ZC);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    B[c] = f2mul(f2fma(g[2][c], b2, f2fma(g[1][c], b1, f2mul(g[0][c], b0))), r);
}

// det <= 0 at a node of the grid (NaN: reported by the error norm).
__device__ __forceinline__ int march_bad(const MarchPair& pt, f2 det) {
  float d0, d1;
  f2split(det, d0, d1);
  return ((pt.code & 1) && d0 <= 0.0f) || ((pt.code & 2) && d1 <= 0.0f);
}

// eq. "magnetic energy" of a pair: zeta halves per boundary index coordinate.
__device__ __forceinline__ void march_energy(const MarchPair& pt, int sz, const f2 B[3], f2 det,
                                             Acc<float>& acc) {
  float w0, w1;
  f2split(f2mul(f2dot(B, B), det), w0, w1);
  const float zyz = ((pt.code >> 4) ? 0.5f : 1.0f) * (sz ? 0.5f : 1.0f);
  if (pt.code & 1) acc.add_e(((pt.code & 4) ? 0.5f : 1.0f) * zyz * w0);
  if (pt.code & 2) acc.add_e(((pt.code & 8) ? 0.5f : 1.0f) * zyz * w1);
}

// A node pair of a field in global memory, at element i; VEC: 8-byte
// aligned rows.
template <bool VEC>
__device__ __forceinline__ f2 march_ld(const float* base, unsigned i, bool second) {
  if constexpr (VEC) return __ldg(reinterpret_cast<const f2*>(base + i));
  return f2pack(__ldg(base + i), second ? __ldg(base + i + 1) : 0.0f);
}
template <bool VEC>
__device__ __forceinline__ void march_st(float* base, unsigned i, bool second, f2 v) {
  if constexpr (VEC) {
    *reinterpret_cast<f2*>(base + i) = v;
  } else {
    float a, b;
    f2split(v, a, b);
    base[i] = a;
    if (second) base[i + 1] = b;
  }
}

// Centre values of a thread's pair: d (not in the first stage, whose input
// is the state) and the k_j of the next stage input (S < 5: k_0 .. k_{S-1})
// or of the update and error (S = 5: k1, k3, k4, k5).
template <int S>
struct MarchCentre {
  static constexpr int NK = S == 5 ? 4 : S;
  f2 d[3];
  f2 k[NK > 0 ? NK : 1][3];
  // OLD: what stages before the previous one wrote; LAST: the previous
  // stage's k (k_{S-1}, the last of the list)
  template <bool VEC, bool OLD, bool LAST>
  __device__ __forceinline__ void issue(const StageArgs<float>& a, const float* d_, int N,
                                        unsigned i, bool second) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (OLD && S > 0) d[c] = march_ld<VEC>(d_, i + c * N, second);
#pragma unroll
      for (int j = 0; j < NK; ++j)
        if (j < NK - 1 ? OLD : LAST)
          k[j][c] = march_ld<VEC>(a.k[S == 5 ? (j == 0 ? 0 : j + 1) : j], i + c * N, second);
    }
  }
};

// Current, velocity and the stage's outputs at the thread's pair of plane m:
// the B plane bm there, P2 the z difference of B, G and 1/det G of plane m,
// yc its stage input, i the pair's first element.  A pair's node on an
// x face is written too, with velocity 0: k is 0 there, so its stage input is
// the fixed boundary position again, and its update that position's bits (d +
// 0 would turn a negative zero).
template <class Gm, int S, bool VEC>
__device__ __forceinline__ void march_out(const StageArgs<float>& a, const MarchPair& own,
                                          bool second, const float* __restrict__ bm,
                                          const f2 P2[3], const f2 g[3][3], f2 r,
                                          const f2 yc[3], const MarchCentre<S>& ce,
                                          const f2* __restrict__ co, float* dout, int N,
                                          unsigned i, bool diag, Acc<float>& acc) {
  f2 P0[3], P1[3], B[3], J[3], u[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float* b = bm + own.z0 + c * Gm::ZCSt;
    B[c] = f2lds(b);
    float b0, b1;
    f2split(B[c], b0, b1);
    P0[c] = f2pack(b1 - b[-1], b[2] - b0);
    P1[c] = f2sub(f2lds(b + MP), f2lds(b - MP));
  }
  const f2 c0 = f2sub(f2dot(P1, g[2]), f2dot(P2, g[1]));
  const f2 c1 = f2sub(f2dot(P2, g[0]), f2dot(P0, g[2]));
  const f2 c2 = f2sub(f2dot(P0, g[1]), f2dot(P1, g[0]));
#pragma unroll
  for (int c = 0; c < 3; ++c)
    J[c] = f2mul(f2fma(c2, g[2][c], f2fma(c1, g[1][c], f2mul(c0, g[0][c]))), r);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int e = (c + 1) % 3, f = (c + 2) % 3;
    u[c] = f2fma(J[e], B[f], f2neg(f2mul(J[f], B[e])));
  }
  if (own.xface()) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float u0, u1;
      f2split(u[c], u0, u1);
      u[c] = f2pack((own.code & 4) ? 0.0f : u0, (own.code & 8) ? 0.0f : u1);
    }
  }
  if (diag) {
    float u0, u1, b0, b1, j0, j1;
    f2split(f2dot(u, u), u0, u1);
    f2split(f2dot(B, B), b0, b1);
    f2split(f2dot(J, J), j0, j1);
    if (!(own.code & 4)) acc.max_xi(u0, b0, j0);
    if (second && !(own.code & 8)) acc.max_xi(u1, b1, j1);
  }
  if constexpr (S < 5) {
    float* ynext = a.ys[(S + 1) & 1];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      f2 v = S == 0 ? yc[c] : ce.d[c];
#pragma unroll
      for (int j = 0; j < S; ++j) v = f2fma(co[j], ce.k[j][c], v);
      v = f2fma(co[S], u[c], v);
      march_st<VEC>(a.k[S], i + c * N, second, u[c]);
      march_st<VEC>(ynext, i + c * N, second, v);
    }
  } else {
    // fifth-order update (b_2 = b_5 = 0) and embedded error (b_2 - b*_2 = 0)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const f2 k1 = ce.k[0][c], k3 = ce.k[1][c], k4 = ce.k[2][c], k5 = ce.k[3][c];
      const f2 up = f2fma(co[3], u[c], f2fma(co[2], k4, f2fma(co[1], k3, f2mul(co[0], k1))));
      const f2 er = f2fma(
          co[8], u[c], f2fma(co[7], k5, f2fma(co[6], k4, f2fma(co[5], k3, f2mul(co[4], k1)))));
      f2 dn = f2add(ce.d[c], up);
      if (own.xface()) {
        float d0, d1, n0, n1;
        f2split(ce.d[c], d0, d1);
        f2split(dn, n0, n1);
        dn = f2pack((own.code & 4) ? d0 : n0, (own.code & 8) ? d1 : n1);
      }
      march_st<VEC>(dout, i + c * N, second, dn);
      float e0, e1;
      f2split(er, e0, e1);
      acc.max_lam(fabsf(e0));
      if (second) acc.max_lam(fabsf(e1));
      if (a.k6) march_st<VEC>(a.k6, i + c * N, second, u[c]);
    }
  }
}

// Wait for a barrier's phase (bounded, as mbar_wait_bounded); false at once
// when another thread of the CTA has given up.
__device__ __forceinline__ bool march_wait(uint64_t* bar, unsigned parity,
                                           volatile int* gave_up) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*gave_up) return false;
    if (globaltimer_ns() - t0 > TMA_WAIT_NS) {
      *gave_up = 1;
      return false;
    }
  }
}

// Stage S (0..5).  Iteration `it` (plane q = qa + it) waits for the planes
// issued two iterations before and issues y plane q + 3 and B0 plane q + 2;
// the prologue's planes (y qa - 1 .. qa + 2, B0 qa, qa + 1) come first.
//
// With TMA an iteration's own B needs no other thread's work, so the barrier
// between iterations is split: warps arrive at the end of iteration q and
// wait for one another only after their own B of plane q + 1, before they
// store it (into the slot whose last readers were in iteration q), refill the
// ring and read their neighbours' B.  (Three warps have a halo pair more than
// the others; with one __syncthreads per iteration 384^3 takes 5.04 ms.)
//
// These waits are bounded.  A thread whose wait gives up tells the others
// (`gave_up`), which then stop waiting; all run out their iterations on void
// data, FLAG_TIMEOUT voids the attempt, thread 0 waits (bounded again) for
// every box still in flight and the CTA returns.  The test hook (a.tma_test)
// adds a barrier that no copy completes to the prologue's wait (1) or to the
// loop's first wait (2); the real copies do complete.
template <int WARPS, int S, bool TMA>
__device__ __forceinline__ void march_body(const StageArgs<float>& a, const TmaMaps* maps) {
  using Gm = MarchGeo<WARPS>;
  constexpr bool FINAL = S == 5;
  constexpr int YR = Gm::YRING, ZR = Gm::ZRING;
  const DevState* st = a.st;
  // Before pdl_wait() only what the previous stage of the attempt does not
  // write: it triggers this launch after its own pdl_wait(), so every kernel
  // before it has completed.  (The first stage follows the step control or
  // anything else, so it waits first.)
  if (S == 0) pdl_wait();
  if (!a.force && (st->status != ST_OK || st->n_accept >= st->target)) {
    if (S > 0) pdl_wait();
    return;
  }
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ double red[32];
  // three for the loop (a barrier is armed again an iteration after every
  // thread has seen it complete), the prologue's, the test hook's, the warps'
  __shared__ uint64_t bars[6];
  __shared__ int gave_up;
  unsigned char* base =
      smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);  // 128-byte aligned
  float* yr = reinterpret_cast<float*>(base);  // [YR][YSTRt]
  float* zr = yr + YR * Gm::YSTRt;             // [ZR][ZSTRt]
  float* bs = zr + ZR * Gm::ZSTRt;             // [2][ZSTRt]
  const int i0 = blockIdx.x * MX, j0 = blockIdx.y * Gm::TH;
  const int k0 = blockIdx.z * a.kz, k1 = min(a.nz, k0 + a.kz);
  const int N = a.nx * a.ny * a.nz, nxy = a.nx * a.ny;
  const int cur = st->cur;
  const float* d = a.d[cur];
  float* dout = const_cast<float*>(a.d[cur ^ 1]);
  const float* y = S == 0 ? d : a.ys[S & 1];
  const CUtensorMap* ymap = TMA ? (S == 0 ? &maps->d[cur] : &maps->ys[S & 1]) : nullptr;
  // B planes qa .. qb; y planes up to yl
  const int qa = max(k0 - 1, 0), qb = min(k1, a.nz - 1), yl = min(qb + 1, a.nz - 1);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;

  // copies without TMA: this thread's points
  int yoff[Gm::LPY], zoff[Gm::LPZ];
  if constexpr (!TMA) {
#pragma unroll
    for (int t = 0; t < Gm::LPY; ++t) {
      const int p = threadIdx.x + t * Gm::NTH;
      const int gi = i0 - 2 + p % Gm::LWY, gj = j0 - 2 + p / Gm::LWY;
      yoff[t] = p < Gm::LWY * Gm::YHt && gi >= 0 && gi < a.nx && gj >= 0 && gj < a.ny
                    ? gj * a.nx + gi : -1;
    }
#pragma unroll
    for (int t = 0; t < Gm::LPZ; ++t) {
      const int p = threadIdx.x + t * Gm::NTH;
      const int gi = i0 - 1 + p % Gm::LWZ, gj = j0 - 1 + p / Gm::LWZ;
      zoff[t] = p < Gm::LWZ * Gm::ZHt && gi >= 0 && gi < a.nx && gj >= 0 && gj < a.ny
                    ? gj * a.nx + gi : -1;
    }
  }
  auto copy_y = [&](float* dst, int q) {
#pragma unroll
    for (int t = 0; t < Gm::LPY; ++t) {
      if (yoff[t] < 0) continue;
      const int p = threadIdx.x + t * Gm::NTH;
      float* o = dst + (p / Gm::LWY) * MP + p % Gm::LWY + 2;
      const float* s = y + (q * nxy + yoff[t]);
#pragma unroll
      for (int c = 0; c < 3; ++c) cp_async4(o + c * Gm::YCSt, s + c * N);
    }
  };
  auto copy_z = [&](float* dst, int q) {
#pragma unroll
    for (int t = 0; t < Gm::LPZ; ++t) {
      if (zoff[t] < 0) continue;
      const int p = threadIdx.x + t * Gm::NTH;
      float* o = dst + (p / Gm::LWZ) * MP + p % Gm::LWZ + 3;
      const float* s = a.B0s + (q * nxy + zoff[t]);
#pragma unroll
      for (int c = 0; c < 3; ++c) cp_async4(o + c * Gm::ZCSt, s + c * N);
    }
  };

  // dt-scaled coefficients as pairs: a_{S+1, j} of the next stage input, or
  // b and b - b* of the update and error
  __shared__ f2 co[9];
  if (S < 5 && threadIdx.x <= S) co[threadIdx.x] = f2dup(st->dtaf[S < 5 ? S + 1 : 0][threadIdx.x]);
  if (S == 5 && threadIdx.x < 9) {
    const int t = threadIdx.x, jb = t == 0 ? 0 : (t == 3 ? 5 : t + 1), je = t == 4 ? 0 : t - 3;
    co[t] = f2dup(t < 4 ? st->dtbf[jb] : st->dtef[je]);
  }
  const bool diag = S == 0 && a.diag != 0;
  Acc<float> acc;
  // the thread's own pair and, for three warps, a halo pair: the rows below
  // and above the tile, then the columns left and right of it
  MarchPair own, halo;
  own.init<Gm>(2 * lane, w + 1, i0, j0, a.nx, a.ny);
  halo.z0 = halo.code = halo.xs = 0;
  const int wr = (w + blockIdx.x + blockIdx.y + blockIdx.z) % WARPS;
  if (wr == 0) halo.init<Gm>(2 * lane, 0, i0, j0, a.nx, a.ny);
  if (wr == 1) halo.init<Gm>(2 * lane, Gm::TH + 1, i0, j0, a.nx, a.ny);
  if (wr == 2 && lane < 2 * Gm::TH)
    halo.init<Gm>(lane < Gm::TH ? -2 : MX, 1 + lane % Gm::TH, i0, j0, a.nx, a.ny);
  // outputs: pairs in the grid, off the y faces
  const bool out_xy = own.any() && !(own.code >> 4);
  const bool second = (own.code & 2) != 0;
  unsigned n = (unsigned)(k0 * nxy + (j0 + w) * a.nx + i0 + 2 * lane);
  MarchCentre<S> ce;
  const bool first_out = out_xy && k0 >= 1 && k0 <= a.nz - 2;
  if (first_out) ce.template issue<TMA, true, false>(a, d, N, n, second);
  // prologue: B0 planes, then (after the wait) stage-input planes
  if constexpr (TMA) {
    if (threadIdx.x == 0) {
      for (int i = 0; i < 5; ++i) mbar_init(&bars[i], 1);
      mbar_init(&bars[5], WARPS);
      gave_up = 0;
      fence_barrier_init();
      if (a.tma_test) mbar_arrive_expect_tx(&bars[4], 16u);
      unsigned bytes = 0;
      for (int q = qa - 1; q <= qa + 2; ++q)
        if (q >= 0 && q <= yl) bytes += Gm::YBYTESt;
      for (int q = qa; q <= qa + 1; ++q)
        if (q <= qb) bytes += Gm::ZBYTESt;
      mbar_arrive_expect_tx(&bars[3], bytes);
      for (int q = qa; q <= qa + 1; ++q)
        if (q <= qb)
          tma_load_4d(zr + (q - qa) * Gm::ZSTRt, &maps->b0, i0 - 4, j0 - 1, q, 0, &bars[3]);
    }
  } else {
    for (int q = qa; q <= qa + 1; ++q)
      if (q <= qb) copy_z(zr + (q - qa) * Gm::ZSTRt, q);
  }
  if (S > 0) pdl_wait();
  // a grid that leaves room for the next stage's beside it lets that one in
  // now; a larger one only when its own CTAs are done
  if (a.early) pdl_trigger();
  if constexpr (TMA) {
    if (threadIdx.x == 0)
      for (int q = qa - 1; q <= qa + 2; ++q)
        if (q >= 0 && q <= yl)
          tma_load_4d(yr + (q - qa + 1) * Gm::YSTRt, ymap, i0 - 4, j0 - 2, q, 0, &bars[3]);
  } else {
    for (int q = qa - 1; q <= qa + 2; ++q)
      if (q >= 0 && q <= yl) copy_y(yr + (q - qa + 1) * Gm::YSTRt, q);
    cp_async_commit();
  }
  if (first_out) ce.template issue<TMA, false, true>(a, d, N, n, second);

  // ring offsets: y planes q - 1 .. q + 3, B0 planes q .. q + 2
  int yo[YR], zo[ZR];
#pragma unroll
  for (int t = 0; t < YR; ++t) yo[t] = t * Gm::YSTRt;
#pragma unroll
  for (int t = 0; t < ZR; ++t) zo[t] = t * Gm::ZSTRt;

  bool ok = true;
  if constexpr (TMA) {
    // an earlier stage of this attempt gave up: so does this one
    const bool skip = threadIdx.x == 0 && (st->flags & FLAG_TIMEOUT);
    if (__syncthreads_or(skip)) {
      if (threadIdx.x == 0) mbar_wait_bounded(&bars[3], 0);
      return;
    }
    ok = mbar_wait_bounded(&bars[3], 0);
    if (a.tma_test == 1) ok = ok && mbar_wait_bounded(&bars[4], 0);
    if (__syncthreads_or(!ok)) {
      if (threadIdx.x == 0) {
        atomicOr(&a.st->flags, FLAG_TIMEOUT);
        mbar_wait_bounded(&bars[3], 0);  // the prologue's boxes still in flight
      }
      return;
    }
  } else {
    cp_async_wait<0>();
    __syncthreads();
  }

  // carried along z: G and 1/det G of plane q - 1 (its B, and B of plane
  // q - 2, are the thread's own entries of the two B slots)
  f2 gc[3][3], rc = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) gc[0][c] = gc[1][c] = gc[2][c] = 0;
  int bo = 0;       // this iteration's B slot
  int ba = 0;       // the barrier this iteration arms
  unsigned pw = 0;  // parity of the barrier it waits for
  int issued = -1;  // the last iteration that issued boxes (thread 0)
#pragma unroll 1  // twice the code no longer stays in the instruction cache (48^3: 59 -> 71 us)
  for (int q = qa; q <= qb; ++q) {
    const int it = q - qa;
    if constexpr (TMA) {
      if (it >= 2) {
        const int bw = ba == 2 ? 0 : ba + 1;  // the barrier of iteration it - 2
        ok = march_wait(&bars[bw], pw, &gave_up) && ok;
        if (a.tma_test == 2 && it == 2) ok = march_wait(&bars[4], 0, &gave_up) && ok;
        pw ^= bw == 2;
      }
    } else {
      if (q + 3 <= yl) copy_y(yr + yo[4], q + 3);
      if (q + 2 <= qb) copy_z(zr + zo[2], q + 2);
      cp_async_commit();
    }
    const int sz = q == 0 ? 1 : (q == a.nz - 1 ? 2 : 0);
    // q - 2 sits where q + 3 would go, q + 2 one before
    const MarchRing R{yr + yo[4], yr + yo[0], yr + yo[1], yr + yo[2], yr + yo[3]};
    const float* zq = zr + zo[0];
    float* bq = bs + bo;
    const float* bm = bs + (Gm::ZSTRt - bo);  // plane q - 1
    f2 gn[3][3], rn = 0, det = 0, Bn[3] = {0, 0, 0}, yc[3] = {0, 0, 0};
#pragma unroll
    for (int c = 0; c < 3; ++c) gn[0][c] = gn[1][c] = gn[2][c] = 0;
    if (own.any()) march_B<Gm>(a, own, sz, R, zq, gn, det, rn, Bn, yc);
    if constexpr (TMA) {
      if (it >= 1) ok = march_wait(&bars[5], (it - 1) & 1, &gave_up) && ok;
      if (threadIdx.x == 0 && ok) {
        const bool ly = q + 3 <= yl, lz = q + 2 <= qb;
        uint64_t* bar = &bars[ba];
        mbar_arrive_expect_tx(bar, (ly ? Gm::YBYTESt : 0u) + (lz ? Gm::ZBYTESt : 0u));
        if (ly) tma_load_4d(yr + yo[4], ymap, i0 - 4, j0 - 2, q + 3, 0, bar);
        if (lz) tma_load_4d(zr + zo[2], &maps->b0, i0 - 4, j0 - 1, q + 2, 0, bar);
        issued = it;
      }
      ba = ba == 2 ? 0 : ba + 1;
    }
    if (own.any()) {
      f2 P2[3];
      acc.bad |= march_bad(own, det);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float* b = bq + own.z0 + c * Gm::ZCSt;
        P2[c] = f2sub(Bn[c], f2lds(b));  // B of plane q - 2 was there
        f2sts(b, Bn[c]);
      }
      if (diag && q >= k0 && q < k1) march_energy(own, sz, Bn, det, acc);
      const int m = q - 1;  // the plane of this iteration's outputs
      if (out_xy && m >= k0 && m >= 1)
        march_out<Gm, S, TMA>(a, own, second, bm, P2, gc, rc, yc, ce, co, dout, N, n - nxy,
                              diag, acc);
    }
    if (halo.any()) {
      f2 gh[3][3], dh, rh, Bh[3], yh[3];
      march_B<Gm>(a, halo, sz, R, zq, gh, dh, rh, Bh, yh);
      acc.bad |= march_bad(halo, dh);
#pragma unroll
      for (int c = 0; c < 3; ++c) f2sts(bq + halo.z0 + c * Gm::ZCSt, Bh[c]);
    }
    if (q >= k0) {
      if (out_xy && q >= 1 && q > k0 && q < k1 && q <= a.nz - 2)
        ce.template issue<TMA, true, true>(a, d, N, n, second);
      n += nxy;  // in plane q + 1
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int e = 0; e < 3; ++e) gc[e][c] = gn[e][c];
    rc = rn;
    bo = Gm::ZSTRt - bo;
    const int y_first = yo[0], z_first = zo[0];
#pragma unroll
    for (int t = 0; t < YR - 1; ++t) yo[t] = yo[t + 1];
    yo[YR - 1] = y_first;
#pragma unroll
    for (int t = 0; t < ZR - 1; ++t) zo[t] = zo[t + 1];
    zo[ZR - 1] = z_first;
    if constexpr (TMA) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars[5]);
    } else {
      cp_async_wait<1>();  // what the next iteration reads has landed
      __syncthreads();
    }
  }
  if constexpr (TMA) {
    if (__syncthreads_or(!ok)) {
      if (threadIdx.x == 0) {
        atomicOr(&a.st->flags, FLAG_TIMEOUT);
        for (int j = max(issued - 2, 0); j <= issued; ++j)  // boxes still in flight
          mbar_wait_bounded(&bars[j % 3], (j / 3) & 1);
      }
      return;
    }
  }
  if (!a.early) pdl_trigger();
  if (__syncthreads_or(acc.bad) && threadIdx.x == 0)
    atomicOr(&a.st->flags, S == 0 ? FLAG_COLLAPSED : FLAG_FOLDED_TRIAL);
  write_partials<float, float>(a, FINAL, diag, acc, red);
}

template <int WARPS, int S, int MINB>
__global__ void __launch_bounds__(32 * WARPS, MINB)
    k_stage_march_tma(const StageArgs<float> a, const __grid_constant__ TmaMaps maps) {
  march_body<WARPS, S, true>(a, &maps);
}
template <int WARPS, int S, int MINB>
__global__ void __launch_bounds__(32 * WARPS, MINB) k_stage_march(const StageArgs<float> a) {
  march_body<WARPS, S, false>(a, nullptr);
}

// Launch stage `stage` (0..5) on `grid`: with tensor maps the TMA loader,
// without (null) the plain copies.
template <int WARPS, int MINB>
cudaError_t launch_stage_march_t(const StageArgs<float>& a, const TmaMaps* maps, int stage,
                                 dim3 grid, cudaStream_t s) {
  const size_t smem = MarchGeo<WARPS>::smem_bytes();
  const dim3 nt(32 * WARPS);
#define GLEMUR_MARCH_CASE(SS)                                                                \
  case SS:                                                                                   \
    return maps ? launch_pdl(k_stage_march_tma<WARPS, SS, MINB>, grid, nt, smem, s, a, *maps) \
                : launch_pdl(k_stage_march<WARPS, SS, MINB>, grid, nt, smem, s, a);
  switch (stage) {
    GLEMUR_MARCH_CASE(0)
    GLEMUR_MARCH_CASE(1)
    GLEMUR_MARCH_CASE(2)
    GLEMUR_MARCH_CASE(3)
    GLEMUR_MARCH_CASE(4)
    GLEMUR_MARCH_CASE(5)
    default:
      return cudaErrorInvalidValue;
  }
#undef GLEMUR_MARCH_CASE
}

template <int WARPS, int MINB>
cudaError_t prepare_stage_march_t() {
  const int sm = (int)MarchGeo<WARPS>::smem_bytes();
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaSuccess;
#define GLEMUR_MARCH_PREP(SS)                                                                  \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stage_march_tma<WARPS, SS, MINB>, at, sm);  \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stage_march<WARPS, SS, MINB>, at, sm);
  GLEMUR_MARCH_PREP(0)
  GLEMUR_MARCH_PREP(1)
  GLEMUR_MARCH_PREP(2)
  GLEMUR_MARCH_PREP(3)
  GLEMUR_MARCH_PREP(4)
  GLEMUR_MARCH_PREP(5)
#undef GLEMUR_MARCH_PREP
  return e;
}

template <int WARPS, int MINB>
int stage_march_ctas_per_sm_t(bool tma) {
  int n = 0;
  const size_t sm = MarchGeo<WARPS>::smem_bytes();
  if (tma)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_stage_march_tma<WARPS, 3, MINB>,
                                                  32 * WARPS, sm);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_stage_march<WARPS, 3, MINB>, 32 * WARPS,
                                                  sm);
  return n;
}

}  // namespace glemur
