// Device-side definitions shared by the GB300 kernels of the relaxation step.
//
// Storage.  The library keeps the displacement d = x - X (X the label grid)
// rather than x: every stencil only needs differences of x, and
// x(m + e_a) - x(m - e_a) = d(m + e_a) - d(m - e_a) + 2 h_a e_a, so X never
// has to be formed and FP32 storage (mixed mode) keeps its precision in the
// part that moves.  B0 is stored pre-scaled, B0s_a = B0_a * 4 h_{a+1} h_{a+2},
// so that with the index-space differences g_a = 2 h_a dx/dX_a the pull-back
// of eq. "B transformation" is B = (g_0 B0s_0 + g_1 B0s_1 + g_2 B0s_2)/det G
// (the h factors cancel), and E_M = sum zeta |B|^2 det G / 16.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace glemur {

// CTA tile: TX x TY output columns, marching in z.
constexpr int TX = 32;
constexpr int TY = 8;
constexpr int NT = TX * TY;
// Displacement tile with a halo of 2 (the mimetic current needs B at the
// six neighbours, and B at a node needs x at its own neighbours).
constexpr int XW = TX + 4, XH = TY + 4, XP = XW * XH;
// B tile with a halo of 1.
constexpr int BW = TX + 2, BH = TY + 2, BP = BW * BH;
// Displacement tile with a halo of 1 (direct current).
constexpr int DW = TX + 2, DH = TY + 2, DP = DW * DH;
// Error flags raised by the stage kernels: det G <= 0 in the accepted state
// (stage 1 input: fatal) or in a trial stage input (the attempt is
// rejected with the largest shrink).
constexpr unsigned FLAG_COLLAPSED = 1u;
constexpr unsigned FLAG_FOLDED_TRIAL = 2u;
// A bounded wait for a tile load gave up (the attempt's results are void).
constexpr unsigned FLAG_TIMEOUT = 4u;

// Device status codes (same values as glemur_status).
constexpr int ST_OK = 0;
constexpr int ST_COLLAPSED = -3;
constexpr int ST_NONFINITE = -4;
constexpr int ST_DT_UNDERFLOW = -5;
constexpr int ST_TIMEOUT = -8;

// Control state of the time integration, resident in the workspace.  The
// step-control kernel updates it after every attempt, so the host never has
// to synchronise between attempts.
struct DevState {
  double dt;          // step size of the next attempt
  double dt_last;     // step size of the last accepted attempt
  double t;           // time of the accepted state
  double lambda;      // error estimate of the last attempt
  double lambda0, dt_min, grow_max, shrink_min, safety;
  long long n_accept, n_reject;
  long long target;   // attempts stop (no-op) once n_accept reaches this
  int consec;         // consecutive rejections
  int cur;            // which displacement buffer holds the accepted state
  int status;         // ST_OK or an error status
  unsigned flags;     // FLAG_* raised by stage kernels in this attempt
  int max_rejects;
  int replay;         // 1: accept the next attempt whatever its error
  // dt-scaled Cash-Karp coefficients of the pending attempt
  double dta[6][6];
  double dtb[6];
  double dte[6];
  float dtaf[6][6];
  float dtbf[6];
  float dtef[6];
  // diagnostics reduced from the state the last diagnostic launch saw
  double E, xi, xi_sin;
};

// Partial-result slots per CTA (see StageArgs::part).
enum { PART_LAMBDA = 0, PART_E = 1, PART_XI2 = 2, PART_XIS2 = 3, NPART = 4 };

template <typename T>
struct StageArgs {
  int nx, ny, nz;
  int kz;              // planes per CTA along z
  double h2[3];        // 2 h_a
  float h2f[3];        // 2 h_a rounded to float (mixed precision)
  const T* d[2];       // ping-pong displacement buffers (3N each)
  const T* B0s;        // pre-scaled B0 (3N)
  T* k[5];             // stage derivatives k1..k5 (3N each)
  T* k6;               // if set, the last stage also stores k6 here
  T* ys[2];            // stage inputs: y_s in ys[s & 1] (s >= 1), 3N each;
                       // boundary entries hold the fixed boundary positions
  int stage;           // 0..5 (stage s+1 of Cash-Karp)
  int diag;            // reduce E_M / xi partials in this launch
  int force;           // run even if the step target is reached
  int early;           // trigger the next launch at the start (see launch_pdl)
  DevState* st;
  double* part;        // [NPART][nblocks] per-CTA partials
  int nblocks;
  // test hook of the bounded tile waits: 0 (off); 1 or 2 make the TMA
  // stage kernels also wait, at the prologue (1) or at the first wait
  // inside the plane loop (2), on a barrier that no copy completes, so that
  // wait gives up and the attempt fails without any fault
  int tma_test;
};

// Programmatic dependent launch.  The kernels of an attempt are launched
// with launch_pdl: the next kernel of the stream may then be scheduled onto
// SMs that the current one has left while its last CTAs still run.  Each
// such kernel calls pdl_trigger() (its own successor may be scheduled once
// all of its CTAs have started and called it) and pdl_wait():
// griddepcontrol.wait returns once the preceding grids have completed and
// their memory operations are visible.  Every path through such a kernel
// passes pdl_wait(), so completion stays transitive along the stream.  Before
// it, a kernel reads and writes nothing an earlier kernel of the stream
// touches, with one exception, which rests on this rule: every stage (both
// its passes) triggers after its own pdl_wait().  So when what follows a stage
// starts, everything before that stage is complete, and a stage after an
// attempt's first, a pass after an attempt's first and the step control may
// read ahead of their wait what the stage or pass before them does not write
// (the control state but its flags, and the partials of the first stage's
// diagnostics).  The step control triggers before its wait, so an attempt's
// first stage or pass, like anything else that may follow it, waits first.
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Host side: launch `k` on stream s, programmatic serialisation allowed
// unless the environment sets GLEMUR_PDL=0 (then an ordinary launch).  A
// grid launched this way is placed on SMs as slots free up, not spread
// evenly at launch: the one-wave FP64 passes therefore size their grid to
// exactly the CTAs per SM that each of them can hold.
bool pdl_enabled();
template <typename... Exp, typename... Act>
cudaError_t launch_pdl(void (*k)(Exp...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       Act&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<Act&&>(args)...);
}

// Division of 0 <= n < 2^31 by a divisor fixed on the host, as a multiply and
// a shift (Granlund & Montgomery, PLDI 1994): an integer division by a
// variable takes some 25 instructions and 200 cycles of latency.
struct FastDiv {
  unsigned m;
  int s, d;
  __device__ __forceinline__ int div(int n) const {
    return (int)((__umulhi((unsigned)n, m) + (unsigned)n) >> s);
  }
};
inline FastDiv fast_div(int d) {
  FastDiv f;
  f.d = d;
  f.s = 0;
  while ((1ll << f.s) < d) ++f.s;
  f.m = (unsigned)(((1ull << 32) * ((1ull << f.s) - (unsigned)d)) / (unsigned)d + 1);
  return f;
}

// n items in whole warps over the CTAs of a grid: `each` warps a CTA, one
// more for the first `extra` (host-side division, no 64-bit one per thread).
struct WarpShare {
  int n, each, extra;
};
inline WarpShare warp_share(long long n, int grid) {
  const long long w = (n + 31) / 32;
  return WarpShare{(int)n, (int)(w / grid), (int)(w % grid)};
}

// Arguments of the FP64 two-pass stages (pass B: B and 1/det G at every
// node; pass C: current, k_s and the next stage input).
struct SplitArgs {
  int nx, ny, nz;
  double h2[3];        // 2 h_a
  const double* d[2];  // ping-pong displacements
  const double* B0s;   // pre-scaled B0 (3N)
  double* k[6];        // k1..k5 (k[5] = optional k6)
  double* ys[2];       // stage inputs: y_s in ys[s & 1] (s >= 1), 3N each;
                       // boundary entries hold the fixed boundary positions
  double* Bb;          // B, 3N
  double* Gb;          // per interior node 10 doubles: g_0, g_1, g_2
                       // (index-space differences, 3 components each) and
                       // 1/det G -- written by pass B, read by pass C
                       // (node_record)
  int diag, force;
  int periodic;        // periodic in z: planes 0, nz-1 are ghosts of nz-2, 1
  DevState* st;
  double* part;        // [NPART][nblocks] per-CTA partials
  int nblocks;         // partial stride: the largest of the grids
  int grid_b, threads_b;  // CTAs of pass B, threads of each
  int grid_c, threads_c;  // of pass C (or the direct stage)
  WarpShare inner_b, bound_b, inner_c;  // interior and boundary nodes of each
  FastDiv dx, dy, dz;     // by nx - 2, ny - 2, nz - 2
};
// Most threads of a dense pass's CTA (one CTA per SM): 32 warps at 64
// registers a thread, since the warps of a quarter come to the end of a node
// together and wait for the next one's loads together, so fewer, fuller
// rounds win (64^3, 12.25 node warps a quarter: 16, 24, 32 warps per SM take
// 322, 320, 302 us an attempt; 129 x 97 x 75: 1034, 1019, 1020).  16 warps at
// 128 for the next-nearest-neighbour pass C and the direct stage.
constexpr int DENSE_T = 1024, DENSE_T2 = 512;
// Dynamic shared memory none of them uses: more than half of an SM's, so
// that two CTAs never share one (a programmatic launch fills an SM that fell
// free with two where it can, and leaves another without: 33^3 99 against 90
// us an attempt, 64^3 at 16 warps 486 against 338).
constexpr int DENSE_SMEM = 118784;

// The persistent FP64 attempt kernel's plan and synchronisation state
// (workspace memory): per node plane, completion counters of pass B and
// pass C and how many CTAs contribute to each; per CTA, the plane
// intervals its pass-B work touches (at most 6: interior planes and the
// boundary face blocks) and its pass-C interval (interior planes); an
// arrival counter and a release generation for the end of each attempt.
constexpr int PERSIST_BI = 6;  // pass-B intervals per CTA
struct PersistArgs {
  int* cntB;            // [nz]
  int* cntC;            // [nz]
  const int* touchB;    // [nz] contributions per plane and pass-B phase
  const int* touchC;    // [nz]
  const int* ivB;       // [G][PERSIST_BI][2] (lo, hi) inclusive, lo > hi: empty
  const int* ivC;       // [G][2]
  unsigned* bar;        // [2] arrivals, released generation
  double* dtlog;        // accepted step-size ring
  int n_attempts;       // attempts this launch
  int test_withhold;    // test hook: this CTA never publishes pass B of
                        // stage 3, so waits on it give up (-1: off)
};

// Boundary nodes as pass B enumerates them (boundary_node): seven groups of
// one stencil variant each, padded to whole warps.
__host__ __device__ constexpr int pad32(int n) { return (n + 31) & ~31; }
__host__ __device__ constexpr int boundary_items(int nx, int ny, int nz) {
  return pad32(2 * (nx - 2) * (ny - 2)) + pad32(2 * (nx - 2) * (nz - 2)) +
         pad32(2 * (ny - 2) * (nz - 2)) + pad32(4 * (nx - 2)) + pad32(4 * (ny - 2)) +
         pad32(4 * (nz - 2)) + 32;
}

// What the on-demand diagnostics (diagnostics.cu) need of a context.
struct DiagCtx {
  int nx, ny, nz;
  double lo[3], h[3];
  int precision, curl, periodic;
  const void* const* dbuf_dev;  // device copy of the two displacement buffers
  const void* B0s;              // pre-scaled B0 in storage precision
  const DevState* st;           // .cur selects the accepted displacement
  double* part;                 // NPART * max_blocks doubles of scratch
  int max_blocks;
  double* stage;                // 3N doubles of scratch
  cudaStream_t s;
};

// 1/v, FP64: Newton-Raphson refinement of the hardware approximation
// rcp.approx.ftz.f64, y <- y + y (1 - v y): each step squares the relative
// error (the classical iteration for reciprocals, e.g. Muller et al.,
// Handbook of Floating-Point Arithmetic, ch. on Newton-Raphson division),
// so two steps take the approximation to within an ulp or two of the
// correctly rounded 1/v in 4 FMAs, where the IEEE division costs about 12
// FP64-pipe instructions -- a quarter of the FP64 work of forming B.  For
// |v| in [2^-1022, 2^1022]: 0, subnormal v, inf and NaN give NaN, larger
// finite v 0.  Its callers pass det G (a value <= 0 is flagged), det M of the
// next-nearest-neighbour current (NaN where the loops are degenerate: the
// error norm reports it) and y^4 of fifth_root (within [1e-24, 1e24]).
__device__ __forceinline__ double recip(double v) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
  double e = fma(-v, y, 1.0);
  y = fma(y, e, y);
  e = fma(-v, y, 1.0);
  return fma(y, e, y);
}

// max of two non-negative doubles that propagates NaN (of either sign),
// on the integer pipes: the bit patterns of non-negative doubles order like
// unsigned integers and every NaN pattern lies above +inf.  (All maxima of
// the step -- error norms, xi^2 -- are of non-negative values; -0 must not
// occur.)  GB300's FP64 pipe is 1/64 of its FP32 rate, so FP64 compares in
// reductions and per-node maxima are worth avoiding.
__device__ __forceinline__ double nanmax(double a, double b) {
  const unsigned long long ua = (unsigned long long)__double_as_longlong(a);
  const unsigned long long ub = (unsigned long long)__double_as_longlong(b);
  return __longlong_as_double((long long)(ua > ub ? ua : ub));
}

// a > b for non-negative doubles (a NaN a counts as larger), on the integer
// pipes (see nanmax); the float overload is the plain compare.
__device__ __forceinline__ bool gt_nonneg(double a, double b) {
  return (unsigned long long)__double_as_longlong(a) > (unsigned long long)__double_as_longlong(b);
}
__device__ __forceinline__ bool gt_nonneg(float a, float b) { return a > b || a != a; }
// not a NaN (integer test for doubles)
__device__ __forceinline__ bool not_nan(double a) {
  return ((unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull) <=
         0x7ff0000000000000ull;
}
__device__ __forceinline__ bool not_nan(float a) { return a == a; }
// a <= 0 (false for NaN), integer test for doubles
__device__ __forceinline__ bool le_zero(double a) {
  return __double_as_longlong(a) <= 0 && not_nan(a);  // sign bit set, or +0
}
__device__ __forceinline__ bool le_zero(float a) { return a <= 0.0f; }

}  // namespace glemur
