// crkfr_volume_lanes.cuh -- the lane-form kernels of the cRKFR step (sm_103a):
// the persistent volume kernel (single solve and batched), the face/update
// kernel (single solve and batched) and their shared-memory layouts.
//
// Volume: element-local cRK stages with the flux-differencing residual, the
// b-weighted volume residual and the face traces of the time averages (eqs.
// crkfr.inner, entropy.cons.flux.dev, entropy.cons.noncons.dev,
// disc.avg.flux), mapped for throughput:
//
//  * a CTA holds 32 elements (16 or 8 where the layout would not fit,
//    LaneLayout::EPB); warp w handles line index w of every element and lane l
//    handles element l, so every shared-memory access of a warp touches 32
//    different elements at the same offset: with an odd element stride there
//    are no bank conflicts;
//  * each thread owns one x-line (N+1 nodes): u^n, the stage combination, the
//    pair data and the whole x-direction flux differencing stay in
//    registers; only the y (and z) lines go through shared memory;
//  * residuals of earlier stages that later stages still need (dense
//    tableaux, N >= 4) stay with the owner thread;
//  * 2D Euler in FP32 (N <= 4): the thread's x-line and y-line are
//    flux-differenced together, one in each half of packed FP32x2
//    instructions (crkfr_f2.cuh), which halves the instructions of the pair
//    fluxes;
//  * the next tile's u^n arrives by TMA bulk copy while the current tile
//    computes (persistent CTAs, one mbarrier, bounded waits);
//  * the register budget (resident CTAs per SM) is set per variant from
//    measurements; the batched form compiles a second shape and lets its
//    autotuner choose.
#pragma once
#include <type_traits>

#include "crkfr_f2.cuh"
#include "crkfr_kernels.cuh"
#include "crkfr_limiter.cuh"

namespace crk {

// stage j's residual is needed by a stage later than j+1
__host__ __device__ constexpr bool rk_saved(int N, int j) {
  bool need = false;
  for (int i = j + 2; i < rk_stages(N); ++i) need = need || (rk_a(N, i, j) != 0.0);
  return need;
}
__host__ __device__ constexpr int rk_slot(int N, int j) {
  int s = 0;
  for (int k = 0; k < j; ++k) s += rk_saved(N, k) ? 1 : 0;
  return s;
}
__host__ __device__ constexpr int rk_nsaved(int N) { return rk_slot(N, rk_stages(N)); }

// The x-line and the y-line of one thread in the two halves of packed FP32
// pairs (2D Euler, FP32 form).  Both lines are flux-differenced in a frame
// rotated to the line: the y half holds (rho, v_y, v_x, p, aux), so the
// normal direction is the first velocity component in both halves, and the
// momentum results of the y half come out in (normal, tangential) order.
template <class EQ>
struct PackXY {
  static constexpr bool value = EQ::DIM == 2 && !EQ::NC;
  // pair-data / residual component of the x line -> of the y half
  __host__ __device__ static constexpr int rot(int c) { return c == 1 ? 2 : (c == 2 ? 1 : c); }
};

// Component of the pair data or residual of a line in direction y, seen in a
// frame reflected across the diagonal so that y becomes the first direction:
// swap of the x and y vector components (velocity / momentum, and the
// magnetic field for GLM-MHD).  The systems and their two-point fluxes are
// invariant under this relabelling, and it is its own inverse.
template <class EQ>
__host__ __device__ constexpr int swap_xy(int c) {
  return c == 1 ? 2 : c == 2 ? 1 : (EQ::NC && c == 5) ? 6 : (EQ::NC && c == 6) ? 5 : c;
}

// PRE: the coefficients carry 1/dx of each line, else the residual is scaled
// at the end
template <class EQ, int N, bool PRE>
__device__ __forceinline__ void line_residual_xy(const f2 (&q)[N + 1][EQ::P], f2 (&acc)[N + 1][EQ::M],
                                                 f2 (&fend)[2][EQ::M], const PhysParams<f2>& pp,
                                                 const RefTab<float>& tb, f2 inv_dx) {
  constexpr int n = N + 1, M = EQ::M;
  const float2 (&A)[6][6] = tb.A2[PRE ? 0 : 1];
  const float2 (&B)[6][6] = tb.B2[PRE ? 0 : 1];
#pragma unroll
  for (int k = 0; k < n; ++k)
#pragma unroll
    for (int v = 0; v < M; ++v) acc[k][v] = f2(0.0f);
  if constexpr (EQ::VOL == VOL_CENTRAL) {
    // sum_q D_pq f(q_q) (line_differences), D_bb = 0 at the inner nodes
#pragma unroll
    for (int b = 1; b < N; ++b) {
      f2 f[M];
      EQ::flux(0, q[b], f, pp);
#pragma unroll
      for (int a = 0; a < n; ++a)
        if (a != b)
#pragma unroll
          for (int v = 0; v < M; ++v) acc[a][v] += f2(B[a][b]) * f[v];
    }
    EQ::flux(0, q[0], fend[0], pp);
    EQ::flux(0, q[N], fend[1], pp);
#pragma unroll
    for (int a = 0; a < n; ++a)
#pragma unroll
      for (int v = 0; v < M; ++v) {
        acc[a][v] += f2(B[a][0]) * fend[0][v];
        acc[a][v] += f2(B[a][N]) * fend[1][v];
      }
  } else {
#pragma unroll
    for (int a = 0; a < n; ++a)
#pragma unroll
      for (int b = a + 1; b < n; ++b) {
        f2 f[M];
        EQ::two_point(0, q[a], q[b], f, pp);
#pragma unroll
        for (int v = 0; v < M; ++v) {
          acc[a][v] += f2(EQ::half(v) ? B[a][b] : A[a][b]) * f[v];
          acc[b][v] += f2(EQ::half(v) ? B[b][a] : A[b][a]) * f[v];
        }
      }
    // end points last: the fluxes there stay live only until the face sums
    EQ::flux(0, q[0], fend[0], pp);
    EQ::flux(0, q[N], fend[1], pp);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      acc[0][v] += f2(A[0][0]) * fend[0][v];
      acc[N][v] += f2(A[N][N]) * fend[1][v];
    }
  }
  if constexpr (!PRE) {
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
      for (int v = 0; v < M; ++v) acc[k][v] *= inv_dx;
  }
}

// Time averages at the two end points of one line in direction D (the face
// nodes of the two faces normal to D): U = sum_i b_i u^(i), F^D = sum_i b_i
// f^D(u^(i)) (eq. disc.avg.flux), lambda_D(u^n).  One record per end.  (The
// average of the non-conservative product, F^nc,D = sum_i b_i B^D g^D of Sec.
// 2.3, enters only its own element's update: nonconservative_ends.)
template <class EQ, typename R>
struct FaceAcc {
  static constexpr int M = EQ::M;
  R U[2][M], F[2][M], lam[2];
};

// The own non-conservative face term at one node of direction D's face (c = 0 or
// N): in the update it appears as the jump's -F^nc_own times the correction
// factor, against + B(u^n) g^avg(U).  Both carry B(u^n) g(u^n), which is large where they
// nearly cancel, so each is taken without it: the jump as B(u^n) (g^avg(U) -
// g(u^n)), and F^nc - B(u^n) g(u^n) as a part of R-bar, + (1/(w_0 dx)) of it at xi = 0
// and - (1/(w_N dx)) at xi = 1.  Added stage by stage with b_i, minus one at
// the first: neither accumulators over the stages nor a component of the
// face record (GLM-MHD 128^2, N = 4, FP32: 28 record components instead of 37, 36
// accumulators less).  A single stage (RKFR) has nothing to add, and the stage-wise
// flux takes B(u^(j)) (g^avg - g)(u^(j)) in the jump.  Against F^nc
// whole in R-bar, rms error of FP32 over 40 (RKFR 20) seeded runs of all degrees: EC 0.98,
// central 0.97, stage-wise 0.96, RKFR EC 0.98, central 0.94.
template <class EQ, int N, typename R>
__device__ __forceinline__ void nonconservative_ends(int d, int c, const R* q, R bi, const MeshArgs& ma,
                                                     const RefTab<R>& tb, R (&rb)[EQ::M]) {
  if (c != 0 && c != N) return;
  R g[2], nc[EQ::M];
#pragma unroll
  for (int v = 0; v < EQ::M; ++v) nc[v] = R(0);
  EQ::ncg(d, q, g);
  EQ::nc_apply(d, q, g, nc);
  const R s = bi * inv_dx_of<R>(ma, d) * (c == 0 ? tb.iw0 : -tb.iwN);
#pragma unroll
  for (int v = 1; v < EQ::M; ++v) rb[v] += s * nc[v];   // no mass
}

// Register budget of the 2D Euler lane kernels of degree 4 and 5 (resident
// CTAs per SM) and the highest degree that takes the packed x/y form by
// default.  FP32, us per volume launch: degree 4 (128^2) packed at 2 CTAs 49.0,
// at 3 CTAs 60, at 1 CTA 59.7, scalar at 3 CTAs 57.9, at 4 CTAs 68.7; degree 5
// (97x61) scalar at 2 CTAs 47.6, at 3 CTAs 76, packed at 2 CTAs 49.0, at 1 CTA
// 53.8 (the packed one won on the larger solves of a batch, so it is the batched
// form's second shape).
constexpr int kMinB4 = 3, kMinB4Pack = 2, kMinB5 = 2, kPackMaxN = 4;
// degree 2, FP32: 4 CTAs per SM (256^2: 26.7 us per volume launch, 27.4 at 5, 30.5 at
// 6, 39.4 at 8); degree 3: 3 CTAs (256^2: 47.5, 50.6 at 2, 49.7 at 4)
constexpr int kMinB2 = 4, kMinB3 = 3;
// GLM-MHD (9 variables, 13 pair data): 2 CTAs per SM where the layout allows
// it, which needs the shared memory of the next tile's staging buffer
// (128^2, N = 4, FP32: 174 against 206 us per volume launch with one): no such
// buffer there (PersistLayout::STAGE)
constexpr int kMinBNc = 2;

// Kernel shapes: SH = 0 is the measured default of each variant; SH = 1 is the
// alternative the batched form's autotuner also times: the scalar form (no
// x/y packing) at one resident CTA per SM more than the packed default, for the
// scalar default of degree 5 (FP32) the packed form, else one CTA fewer (fewer
// spills, fewer warps).
template <class EQ, int N, typename R, int SH = 0>
struct LaneLayout;

template <class EQ, int N, typename R>
struct LaneLayout<EQ, N, R, 0> {
  static constexpr int DIM = EQ::DIM, M = EQ::M, P = EQ::P, n = N + 1;
  static constexpr int NP = ipow(n, DIM), NF = NP / n, S = rk_stages(N);
  static constexpr int O_Q = 0;                                // [P][NP] pair data (also staging)
  static constexpr int O_RY = O_Q + P * NP;                    // [M][NP] y (+z) residual
  static constexpr int O_U0 = O_RY + (DIM > 1 ? M * NP : 0);   // [M][NP] u^n
  static constexpr int SZ0 = O_U0 + M * NP;
  static constexpr int SZ = SZ0 | 1;                           // odd element stride: no bank conflicts
  // Elements per CTA: 32 (a warp = one line of 32 elements) where the layout
  // fits in shared memory, else 16 or 8 (a warp = 2 or 4 lines): FP64 in 3D and
  // GLM-MHD N = 5, FP32 3D N >= 4.  Lines of different offsets in a warp can meet in a
  // bank; in FP64 an access is served per half-warp, so 16 elements have none.
  // us per volume launch against one thread per line with the stages in shared
  // memory (4 to 8 warps per SM), which this replaced: 3D FP64 N = 3 22x20x19
  // 1498 -> 1193, N = 4 14^3 3942 -> 1714, N = 5 10^3 4755 -> 1238, FP32 N = 4 32^3 3432 -> 862 (8
  // elements; 937 with 16), N = 5 24^3 3993 -> 931 (16; 959 with 8), GLM-MHD FP64
  // N = 5 64^2 7191 -> 1826.  3D FP32 N = 3: 1588 with 32, 1605 with 16, 1706 with 8 (64^3).
  static constexpr size_t kSmemCta = 227 * 1024 - 16;   // the mbarrier after the layout
  static constexpr bool fits_with(int e) { return sizeof(R) * (size_t)SZ * e <= kSmemCta && e * NF <= 1024; }
  static constexpr int EPB = fits_with(32) ? 32 : fits_with(16) && !(DIM == 3 && N == 4) ? 16 : 8;
  static constexpr int THREADS = EPB * NF;
  // resident CTAs of a layout with fewer than 32 elements: what shared memory
  // holds (with the staging buffer), up to 512 threads
  static constexpr int small_minb() {
    const size_t stage = sizeof(double) * (size_t)M * EPB * NP, b = bytes() + stage <= kSmemCta ? bytes() + stage : bytes();
    const int by_smem = (int)(228 * 1024 / (b + 1040)), by_threads = 512 / THREADS;
    const int m = by_smem < by_threads ? by_smem : by_threads;
    return m > 1 ? m : 1;
  }
  static constexpr size_t bytes() { return sizeof(R) * (size_t)SZ * EPB; }
  // packed x/y form (2D Euler, FP32 pair fluxes)
  static constexpr bool PACK = PackXY<EQ>::value && sizeof(R) == 4 && N <= kPackMaxN;
  // CTAs per SM the register allocation aims at (the packed form holds both
  // lines' pair data at once)
  static constexpr int MINB = EQ::NC ? (2 * (bytes() + 1024) <= 228 * 1024 ? kMinBNc : 1)
                            : EPB < 32 ? small_minb()
                            : (THREADS <= 128) ? ((N == 2 && sizeof(R) == 4) ? kMinB2 : PACK ? kMinB3 : 4)
                            : (DIM == 2) ? (N == 4 ? (PACK ? kMinB4Pack : kMinB4) : N == 5 ? kMinB5 : 1) : 1;
  static constexpr bool fits() { return fits_with(EPB); }
};

template <class EQ, int N, typename R>
struct LaneLayout<EQ, N, R, 1> : LaneLayout<EQ, N, R, 0> {
  using B = LaneLayout<EQ, N, R, 0>;
  static constexpr bool PACK = N == 5 && PackXY<EQ>::value && sizeof(R) == 4;
  static constexpr int MINB = PACK ? B::MINB : B::PACK ? B::MINB + 1 : (B::MINB > 1 ? B::MINB - 1 : 1);
};

// SH = 2: the same form in tiles of 8 or 16 elements (whole warps where NF allows),
// which spread a mesh more evenly over the SMs (FP64, Variant::volume).
template <class EQ, int N, typename R>
struct LaneLayout<EQ, N, R, 2> : LaneLayout<EQ, N, R, 0> {
  using B = LaneLayout<EQ, N, R, 0>;
  static constexpr int EPB = B::DIM == 3 || B::NF % 4 == 0 ? 8 : 16;
  static constexpr int THREADS = EPB * B::NF;
  // eight warps per SM keep the FP64 pipe as busy as the default's 12 to 16, with
  // 255 registers: 97x61 N = 5 856 -> 833 us per step, N = 4 551 -> 529, others within 1%
  static constexpr int W = (THREADS + 31) / 32, MINB = W < 8 ? 8 / W : 1;
  static constexpr size_t bytes() { return sizeof(R) * (size_t)B::SZ * EPB; }
};

// face_accumulate for both lines of the packed form at once (x-line ends in
// the low halves, y-line ends in the high halves, the latter in the frame of
// the y-line); the wave speeds are taken separately
template <class EQ, int N>
__device__ __forceinline__ void face_accumulate_xy(FaceAcc<EQ, f2>& fa, const f2 (&q)[N + 1][EQ::P],
                                                   const f2 (&fend)[2][EQ::M], f2 b, bool first,
                                                   const PhysParams<f2>& pp) {
  constexpr int M = EQ::M;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    f2 uu[M];
    EQ::cons_from_pair(q[side ? N : 0], uu, pp);
    if (first) {
#pragma unroll
      for (int v = 0; v < M; ++v) {
        fa.U[side][v] = f2(0.0f);
        fa.F[side][v] = f2(0.0f);
      }
    }
#pragma unroll
    for (int v = 0; v < M; ++v) {
      fa.U[side][v] += b * uu[v];
      fa.F[side][v] += b * fend[side][v];
    }
  }
}

template <class EQ, int N, typename R, int D>
__device__ __forceinline__ void face_accumulate(FaceAcc<EQ, R>& fa, const R (&q)[N + 1][EQ::P],
                                                const R (&fend)[2][EQ::M], R b, bool first,
                                                const PhysParams<R>& pp) {
  constexpr int M = EQ::M;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const R* qs = q[side ? N : 0];
    R uu[M];
    EQ::cons_from_pair(qs, uu, pp);
    if (first) {
      fa.lam[side] = EQ::wave_speed(D, qs, pp);
#pragma unroll
      for (int v = 0; v < M; ++v) {
        fa.U[side][v] = R(0);
        fa.F[side][v] = R(0);
      }
    }
#pragma unroll
    for (int v = 0; v < M; ++v) {
      fa.U[side][v] += b * uu[v];
      fa.F[side][v] += b * fend[side][v];
    }
  }
}

// Record of one face node: U, F, lambda [, u^n] (C components, each
// store coalesced over the warp's elements).  u^n of the two end nodes
// (non-conservative system) is read from shared memory: un0 / unN point at
// variable 0 of the end nodes, variables NP apart.
template <class EQ, typename R, int NF>
__device__ __forceinline__ void write_records(R* __restrict__ trace, const FaceAcc<EQ, R>& fa, int d, long long E,
                                              long long e, int f, const R* un0, const R* unN, int NPv) {
  constexpr int M = EQ::M;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    R* dst = trace + trace_index<EQ, NF>(d, side, f, 0, E, e);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      dst[(size_t)v * E] = fa.U[side][v];
      dst[(size_t)(M + v) * E] = fa.F[side][v];
    }
    dst[(size_t)(2 * M) * E] = fa.lam[side];
    if constexpr (EQ::NC) {
#pragma unroll
      for (int v = 0; v < M; ++v) dst[(size_t)(2 * M + 1 + v) * E] = (side ? unN : un0)[v * NPv];
    }
  }
}

// Prefetch of the next tile's u^n into the staging buffer (TMA bulk copies,
// one per variable), issued by thread 0 once the current tile's staging data
// has been consumed.  src == nullptr: nothing to prefetch.
struct Prefetch {
  const double* src;        // u^n of variable 0 of the next tile
  long long var_stride;     // doubles between variables (E * NP of the next tile's solve)
  unsigned bytes;           // bytes per variable (32 * NP * 8)
  double* staging;
  unsigned long long* bar;
};

template <int M>
__device__ __forceinline__ void issue_prefetch(const Prefetch& pf) {
  fence_proxy_async_smem();
  mbar_arrive_expect_tx(pf.bar, M * pf.bytes);
#pragma unroll
  for (int v = 0; v < M; ++v)
    bulk_copy_g2s(pf.staging + (size_t)v * (pf.bytes / 8), pf.src + (size_t)v * pf.var_stride, pf.bytes, pf.bar);
}

// One tile of 32 elements starting at e0 (the CTA's whole shared memory sm).
// staged != nullptr: u^n of the tile already sits in shared memory as FP64,
// [var][32][NP] (the tile's slice of the global layout).  S1 = 1: a single
// stage with b = 1 (R-bar = R(u), face records of u), the volume part of one
// stage of the multi-stage RKFR step.
// PRE: a single solve's reference table (the flux-differencing coefficients
// carry 1/dx); false for the batched kernels
template <class EQ, int N, typename R, int SH = 0, int S1 = 0, bool PRE = false>
__device__ __forceinline__ void volume_lanes_tile(const double* __restrict__ u, R* __restrict__ rbar,
                                                  R* __restrict__ trace, const DevState* __restrict__ st,
                                                  const MeshArgs& ma, const PhysParams<R>& pp, const RefTab<R>& tb,
                                                  long long e0, R dtR, R* sm, const double* staged = nullptr,
                                                  Prefetch pf = Prefetch{nullptr, 0, 0, nullptr, nullptr}) {
  using L = LaneLayout<EQ, N, R, SH>;
  constexpr int DIM = L::DIM, M = L::M, P = L::P, n = L::n, NP = L::NP, NF = L::NF, S = S1 ? S1 : L::S;
  // 2D, FP64, degree 5 and GLM-MHD: the x-line and the y-line go through one copy
  // of the pair loop (a rolled loop over the two directions, the y-line in the
  // frame of swap_xy), with the pair data read back from shared memory: half the
  // code of two inlined copies, and no pair data held across the barrier.
  // Measured per launch: degree 5 (97x61) 1269 against 1294 us, the GLM-MHD
  // vortex at degree 4 (128^2) 3.27 against 3.58 ms, at degree 3 (61x45) 306
  // against 319 us; in FP32 two copies are the faster form (degree 5, 97x61,
  // 47.6 against 51 us; GLM-MHD degree 4, 128^2, 174 against 193 us, and 255 us
  // with the pair loop rolled over shared memory).
  constexpr bool ROLL = !L::PACK && DIM == 2 && sizeof(R) == 8 && (N >= 5 || EQ::NC);
  // 2D Euler, FP32, degree 5: the plain coefficients and a scaling per line for
  // single solves too, so that a solve and the same solve in a batch round alike
  // (the scaling is 48 of about 1500 instructions a stage)
  constexpr bool TPRE = PRE && !(DIM == 2 && !EQ::NC && sizeof(R) == 4 && N == 5);
  constexpr int NS = rk_nsaved(N) > 0 ? rk_nsaved(N) : 1;

  const int tid = threadIdx.x;
  const int l = tid / L::EPB;          // line index (warp-uniform with 32 elements)
  const int el = tid % L::EPB;         // element within the CTA
  const long long E = ma.E;
  const int nel = (int)min((long long)L::EPB, E - e0);
  const bool active = el < nel;
  R* my = sm + (size_t)el * L::SZ;
  constexpr bool PACK = L::PACK;
  const PhysParams<f2> pp2{f2(float(pp.gamma)), f2(float(pp.inv_gm1)), f2(float(pp.c_h)), f2(float(pp.inv4)), f2(float(pp.ch2))};

  // ---- u^n: coalesced into shared memory (staging in the Q region), then own x-line to registers
  // (index arithmetic with compile-time divisors only).  FP32 form: the hardware conversion, one
  // issue slot on the FP64 pipe, which this kernel leaves otherwise idle (the integer d2f_int is
  // about twenty ALU instructions; measured 59.5 -> 56.6 us per launch, 2D Euler 256^2, N = 3)
  // each variable's 32 NP values are n rounds of the CTA's 32 NF threads:
  // the node offsets of the rounds are computed once, the variable loop only
  // adds its stride
  static_assert(L::EPB * NP == n * L::THREADS, "a tile's values per variable are n rounds of the CTA");
  int tofs[n];
  bool tok[n];
#pragma unroll
  for (int j = 0; j < n; ++j) {
    const int r = tid + j * L::THREADS, ee = r / NP;
    tofs[j] = ee * L::SZ + L::O_U0 + r % NP;
    tok[j] = ee < nel;
  }
  {
    const double* src = staged ? staged + tid : u + (size_t)e0 * NP + tid;
    const size_t vstride = staged ? (size_t)L::EPB * NP : (size_t)E * NP;
#pragma unroll 1
    for (int v = 0; v < M; ++v, src += vstride) {
#pragma unroll
      for (int j = 0; j < n; ++j)
        if (tok[j]) {
          const double x = src[j * L::THREADS];
          if constexpr (sizeof(R) == 4) sm[tofs[j] + v * NP] = __double2float_rn(x);
          else sm[tofs[j] + v * NP] = x;
        }
    }
  }
  __syncthreads();
  // the staging buffer is free: start the next tile's copy, overlapped with this tile's work
  if (pf.src && tid == 0) issue_prefetch<M>(pf);

  R rb[n][M], ax[n][M], rs[NS][n][M];
#pragma unroll
  for (int k = 0; k < n; ++k)
#pragma unroll
    for (int v = 0; v < M; ++v) { rb[k][v] = R(0); ax[k][v] = R(0); }
  // face sums of the ends of this thread's x-line (faces normal to x), y-line and z-line
  FaceAcc<EQ, R> fx, fy, fz;
  FaceAcc<EQ, f2> fxy;   // packed form: both lines' face sums

  // the stage loop stays rolled: one stage's code is large, and S copies of it
  // would overflow the instruction cache; the tableau comes from the parameters
#pragma unroll 1
  for (int i = 0; i < S; ++i) {
    const R bi = S1 ? R(1) : tb.b[i];
    // ---------------- node phase (own x-line): stage state and pair data
    R q[ROLL ? 1 : n][P];
    if (active) {
      // w = dt sum_j a_ij R_j: the last stage's residual (x part from registers,
      // y/z part from shared memory), then the saved ones stage by stage, so that
      // the slot, its address and the coefficient are taken once per stage, not
      // once per value (volume launch, FP32: 2D Euler 128^2 N = 4 97 -> 50 us,
      // 97x61 N = 5 98 -> 51 us, GLM-MHD 128^2 N = 4 491 -> 255 us)
      R w[n][M];
      if (i > 0) {
        const R ap = dtR * tb.a[i][i - 1], bp = tb.b[i - 1];
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int v = 0; v < M; ++v) {
            const R r = ax[k][v] + (DIM > 1 ? my[L::O_RY + v * NP + l * n + k] : R(0));
            rb[k][v] += bp * r;
            w[k][v] = DIM == 1 ? mulr(ap, r) : ap * r;   // 1D: rounded as in k_volume_pairs
            if constexpr (rk_nsaved(N) > 0) ax[k][v] = r;
          }
        if constexpr (rk_nsaved(N) > 0) {
          const int sp = tb.slot[i - 1];
          if (sp >= 0) {
#pragma unroll
            for (int k = 0; k < n; ++k)
#pragma unroll
              for (int v = 0; v < M; ++v) rs[sp][k][v] = ax[k][v];
          }
#pragma unroll 1
          for (int j = 0; j < i - 1; ++j) {
            const R c = dtR * tb.a[i][j];
            const int sj = tb.slot[j];
            if (sj >= 0 && c != R(0)) {
#pragma unroll
              for (int k = 0; k < n; ++k)
#pragma unroll
                for (int v = 0; v < M; ++v) w[k][v] += c * rs[sj][k][v];
            }
          }
        }
      } else {
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int v = 0; v < M; ++v) w[k][v] = R(0);
      }
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const int p = l * n + k;
        R uu[M];
#pragma unroll
        for (int v = 0; v < M; ++v) uu[v] = my[L::O_U0 + v * NP + p] - w[k][v];
        R* qk = q[ROLL ? 0 : k];
        EQ::pair_data(uu, qk, pp);
        if constexpr (EQ::NC && !EQ::NCS && !S1) {
          static_assert(DIM == 2, "the y coordinate of x-line l is l");
          const R bd = i == 0 ? bi - R(1) : bi;
          nonconservative_ends<EQ, N, R>(0, k, qk, bd, ma, tb, rb[k]);
          nonconservative_ends<EQ, N, R>(1, l, qk, bd, ma, tb, rb[k]);
        }
        if (DIM > 1) {
#pragma unroll
          for (int c = 0; c < P; ++c) my[L::O_Q + c * NP + p] = qk[c];
        }
        if constexpr (ROLL && EQ::NCS) {
          // face traces of this stage: the ends of the x-line, and the whole
          // x-line where it lies on a face normal to y
          if (k == 0) write_stage_prims<EQ, N, R>(trace, 0, 0, l, i, E, e0 + el, qk);
          if (k == N) write_stage_prims<EQ, N, R>(trace, 0, 1, l, i, E, e0 + el, qk);
          if (l == 0) write_stage_prims<EQ, N, R>(trace, 1, 0, k, i, E, e0 + el, qk);
          if (l == N) write_stage_prims<EQ, N, R>(trace, 1, 1, k, i, E, e0 + el, qk);
        }
      }
      if constexpr (EQ::NCS && !ROLL) {
        // face traces of this stage at the ends of the x-line (stage-wise
        // non-conservative flux)
        write_stage_prims<EQ, N, R>(trace, 0, 0, l, i, E, e0 + el, q[0]);
        write_stage_prims<EQ, N, R>(trace, 0, 1, l, i, E, e0 + el, q[N]);
      }
      // ---------------- x-direction flux differencing, all in registers
      // (packed form: together with the y-line below)
      if constexpr (!PACK && !ROLL) {
        R fend[2][M];
        line_differences<EQ, N, R, TPRE>(0, q, ax, fend, pp, tb, 0, inv_dx_of<R>(ma, 0));
        face_accumulate<EQ, N, R, 0>(fx, q, fend, bi, i == 0, pp);
      }
    }
    if constexpr (PACK) {
      __syncthreads();   // Q of this stage visible; RY of the last stage consumed
      if (active) {
        // y-line l: nodes (i = l, j = 0..N); x-line in the low halves, y-line in the high halves
        R qy[n][P];
        f2 q2[n][P], acc2[n][M], fe2[2][M];
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int c = 0; c < P; ++c) qy[k][c] = my[L::O_Q + c * NP + l + k * n];
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int c = 0; c < P; ++c) q2[k][c] = f2(q[k][c], qy[k][PackXY<EQ>::rot(c)]);
        line_residual_xy<EQ, N, TPRE>(q2, acc2, fe2, pp2, tb, f2(inv_dx_of<float>(ma, 0), inv_dx_of<float>(ma, 1)));
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int v = 0; v < M; ++v) {
            ax[k][v] = acc2[k][v].v.x;
            my[L::O_RY + v * NP + l + k * n] = acc2[k][PackXY<EQ>::rot(v)].v.y;
          }
        if (i == 0) {
#pragma unroll
          for (int sd = 0; sd < 2; ++sd) {
            fx.lam[sd] = EQ::wave_speed(0, q[sd ? N : 0], pp);
            fy.lam[sd] = EQ::wave_speed(1, qy[sd ? N : 0], pp);
          }
        }
        face_accumulate_xy<EQ, N>(fxy, q2, fe2, f2(bi), i == 0, pp2);
      }
      __syncthreads();   // RY complete
    } else if constexpr (ROLL) {
      __syncthreads();   // Q of this stage visible; RY of the last stage consumed
      if (active) {
#pragma unroll 1
        for (int dir = 0; dir < 2; ++dir) {
          // x-line l: nodes l n + k; y-line l: nodes l + k n (2D)
          const int base = dir ? l : l * n, stride = dir ? n : 1;
          R qd[n][P], ad[n][M], fe[2][M];
#pragma unroll
          for (int k = 0; k < n; ++k)
#pragma unroll
            for (int c = 0; c < P; ++c) qd[k][c] = my[L::O_Q + (dir ? swap_xy<EQ>(c) : c) * NP + base + k * stride];
          line_differences<EQ, N, R, TPRE>(0, qd, ad, fe, pp, tb, dir, dir ? inv_dx_of<R>(ma, 1) : inv_dx_of<R>(ma, 0));
          if (dir == 0) {
#pragma unroll
            for (int k = 0; k < n; ++k)
#pragma unroll
              for (int v = 0; v < M; ++v) ax[k][v] = ad[k][v];
            face_accumulate<EQ, N, R, 0>(fx, qd, fe, bi, i == 0, pp);
          } else {
#pragma unroll
            for (int k = 0; k < n; ++k)
#pragma unroll
              for (int v = 0; v < M; ++v) my[L::O_RY + swap_xy<EQ>(v) * NP + base + k * n] = ad[k][v];
            // accumulated in the swapped frame; swapped back when written
            face_accumulate<EQ, N, R, 0>(fy, qd, fe, bi, i == 0, pp);
          }
        }
      }
      __syncthreads();   // RY complete
    } else if (DIM > 1) {
      __syncthreads();   // Q of this stage visible; RY of the last stage consumed
      if (active) {
        // y-line l: nodes (i = l % n, j = 0..N, k = l / n)
        const int base = (l % n) + (l / n) * n * n;
        R qy[n][P], ay[n][M], fend[2][M];
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int c = 0; c < P; ++c) qy[k][c] = my[L::O_Q + c * NP + base + k * n];
        if constexpr (EQ::NCS) {
          static_assert(DIM == 2, "stage-wise non-conservative flux: 2D only");
          write_stage_prims<EQ, N, R>(trace, 1, 0, l, i, E, e0 + el, qy[0]);
          write_stage_prims<EQ, N, R>(trace, 1, 1, l, i, E, e0 + el, qy[N]);
        }
        line_differences<EQ, N, R, TPRE>(DIM > 1 ? 1 : 0, qy, ay, fend, pp, tb, 1, inv_dx_of<R>(ma, 1));
        face_accumulate<EQ, N, R, (DIM > 1 ? 1 : 0)>(fy, qy, fend, bi, i == 0, pp);
#pragma unroll
        for (int k = 0; k < n; ++k)
#pragma unroll
          for (int v = 0; v < M; ++v) my[L::O_RY + v * NP + base + k * n] = ay[k][v];
      }
      if (DIM == 3) {
        __syncthreads();
        if (active) {
          // z-line l: nodes (i, j) = (l % n, l / n), k = 0..N
          const int base = l;
          R qz[n][P], az[n][M], fend[2][M];
#pragma unroll
          for (int k = 0; k < n; ++k)
#pragma unroll
            for (int c = 0; c < P; ++c) qz[k][c] = my[L::O_Q + c * NP + base + k * n * n];
          line_differences<EQ, N, R, TPRE>(DIM - 1, qz, az, fend, pp, tb, 2, inv_dx_of<R>(ma, DIM - 1));
          face_accumulate<EQ, N, R, DIM - 1>(fz, qz, fend, bi, i == 0, pp);
#pragma unroll
          for (int k = 0; k < n; ++k)
#pragma unroll
            for (int v = 0; v < M; ++v) my[L::O_RY + v * NP + base + k * n * n] += az[k][v];
        }
      }
      __syncthreads();   // RY complete
    }
  }

  // ---- last stage's residual, Rbar to shared (Q region) then coalesced store
  if (active) {
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const int p = l * n + k;
#pragma unroll
      for (int v = 0; v < M; ++v) {
        R r = ax[k][v] + (DIM > 1 ? my[L::O_RY + v * NP + p] : R(0));
        my[L::O_Q + v * NP + p] = rb[k][v] + (S1 ? R(1) : tb.b[S - 1]) * r;
      }
    }
  }
  __syncthreads();
  {
    int qofs[n];
    bool qok[n];
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const int r = tid + j * L::THREADS, ee = r / NP;
      qofs[j] = ee * L::SZ + L::O_Q + r % NP;
      qok[j] = ee < nel;
    }
    R* dst = rbar + (size_t)e0 * NP + tid;
#pragma unroll 1
    for (int v = 0; v < M; ++v, dst += (size_t)E * NP) {
#pragma unroll
      for (int j = 0; j < n; ++j)
        if (qok[j]) dst[j * L::THREADS] = sm[qofs[j] + v * NP];
    }
  }
  // ---- face records [DIM][2][NF][C][E]: this thread owns the two ends of its
  // x-, y- and z-line, i.e. face node f = l of every face; consecutive lanes
  // write consecutive records
  if (active) {
    const R* u0 = my + L::O_U0;
    // end nodes: x-line l (l n, l n + N), y-line l (by, by + N n), z-line l (l, l + N n^2)
    const int by = (l % n) + (l / n) * n * n;
    if constexpr (PACK) {
#pragma unroll
      for (int sd = 0; sd < 2; ++sd)
#pragma unroll
        for (int v = 0; v < M; ++v) {
          fx.U[sd][v] = fxy.U[sd][v].v.x;
          fx.F[sd][v] = fxy.F[sd][v].v.x;
          fy.U[sd][v] = fxy.U[sd][PackXY<EQ>::rot(v)].v.y;
          fy.F[sd][v] = fxy.F[sd][PackXY<EQ>::rot(v)].v.y;
        }
    }
    write_records<EQ, R, NF>(trace, fx, 0, E, e0 + el, l, u0 + l * n, u0 + l * n + N, NP);
    if constexpr (ROLL) {
      FaceAcc<EQ, R> fyo;
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        fyo.lam[sd] = fy.lam[sd];
#pragma unroll
        for (int v = 0; v < M; ++v) {
          fyo.U[sd][swap_xy<EQ>(v)] = fy.U[sd][v];
          fyo.F[sd][swap_xy<EQ>(v)] = fy.F[sd][v];
        }
      }
      write_records<EQ, R, NF>(trace, fyo, 1, E, e0 + el, l, u0 + by, u0 + by + N * n, NP);
    } else if (DIM > 1) {
      write_records<EQ, R, NF>(trace, fy, 1, E, e0 + el, l, u0 + by, u0 + by + N * n, NP);
    }
    if (DIM > 2) write_records<EQ, R, NF>(trace, fz, 2, E, e0 + el, l, u0 + l, u0 + l + N * n * n, NP);
  }
}

// shared memory of the persistent lane kernels: lane layout, then the FP64
// staging buffer of one tile, then the mbarrier
template <class EQ, int N, typename R, int SH = 0>
struct PersistLayout {
  using L = LaneLayout<EQ, N, R, SH>;
  static constexpr size_t O_STAGE = (L::bytes() + 15) & ~(size_t)15;
  static constexpr size_t WANT = sizeof(double) * (size_t)EQ::M * L::EPB * L::NP;
  static constexpr bool STAGE = !EQ::NC && O_STAGE + WANT + 16 <= 227 * 1024;
  static constexpr size_t STAGE_BYTES = STAGE ? WANT : 0;
  static constexpr size_t O_BAR = O_STAGE + STAGE_BYTES;
  static constexpr size_t bytes() { return O_BAR + 16; }
  static constexpr bool fits() { return L::fits() && bytes() <= 227 * 1024; }
};

// Persistent volume kernel for one solve: CTA b handles tiles b, b + grid, ...;
// u^n of whole tiles arrives by TMA bulk copy one tile ahead.  first = false
// (later stages of a multi-stage RKFR step) takes the dt the step's first
// launch recorded.
struct NoTileWork {
  __device__ void operator()(long long, const float*) const {}
};

// after_tile(e0, sm): more work on a finished tile whose u^n is still in the
// lane layout's u^n region of sm (the rest of the layout is free)
template <class EQ, int N, typename R, int S1, class After = NoTileWork, int SH = 0>
__device__ __forceinline__ void volume_lanes_persistent(const double* __restrict__ u, R* __restrict__ rbar,
                                                        R* __restrict__ trace, DevState* __restrict__ st,
                                                        const MeshArgs& ma, const PhysParams<R>& pp,
                                                        const RefTab<R>& tb, int slot, bool first,
                                                        After after_tile = After{}) {
  using PL = PersistLayout<EQ, N, R, SH>;
  constexpr int M = EQ::M, NP = PL::L::NP, EPB = PL::L::EPB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* sm = reinterpret_cast<R*>(smem_raw);
  double* staging = reinterpret_cast<double*>(smem_raw + PL::O_STAGE);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + PL::O_BAR);
  const long long E = ma.E;
  const unsigned ntiles = (unsigned)((E + EPB - 1) / EPB);
  auto whole = [&](unsigned t) { return PL::STAGE && ma.tma_ok && (long long)(t + 1) * EPB <= E; };
  auto pf_of = [&](unsigned t) {
    return Prefetch{u + (size_t)t * EPB * NP, E * NP, (unsigned)(EPB * NP * sizeof(double)), staging, bar};
  };
  __shared__ double s_dt;
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    s_dt = first ? step_begin(st, slot, ma.cfl, ma.dt_fixed, blockIdx.x == 0) : st->dt;
  }
  __syncthreads();
  const R dtR = dt_as<R>(s_dt);
  unsigned phase = 0;
  unsigned t = blockIdx.x;
  if (t < ntiles && whole(t) && threadIdx.x == 0) issue_prefetch<M>(pf_of(t));
  for (; t < ntiles; t += gridDim.x) {
    const bool staged = whole(t);
    if (staged) {
      const bool ok = mbar_wait_bounded(bar, phase);
      if (__syncthreads_or(!ok)) {
        // the copy may still be in flight: thread 0 waits for it once more
        // (bounded) before the CTA's shared memory is released
        if (threadIdx.x == 0) {
          atomicOr(&st->status, ST_TIMEOUT);
          mbar_wait_bounded(bar, phase);
        }
        return;
      }
      phase ^= 1u;
    }
    const unsigned tn = t + gridDim.x;
    const Prefetch pf = (tn < ntiles && whole(tn)) ? pf_of(tn) : Prefetch{nullptr, 0, 0, nullptr, nullptr};
    volume_lanes_tile<EQ, N, R, SH, S1, true>(u, rbar, trace, st, ma, pp, tb, (long long)t * EPB, dtR, sm,
                                       staged ? staging : nullptr, pf);
    __syncthreads();   // shared memory is reused by the next tile
    if constexpr (!std::is_same<After, NoTileWork>::value) {
      after_tile((long long)t * EPB, reinterpret_cast<const float*>(sm));
      __syncthreads();
    }
  }
}

template <class EQ, int N, typename R, int SH = 0>
__global__ void __launch_bounds__(LaneLayout<EQ, N, R, SH>::THREADS, LaneLayout<EQ, N, R, SH>::MINB)
k_volume_lanes(const double* __restrict__ u, R* __restrict__ rbar, R* __restrict__ trace,
               DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb,
               int slot) {
  volume_lanes_persistent<EQ, N, R, 0, NoTileWork, SH>(u, rbar, trace, st, ma, pp, tb, slot, true);
}

// The volume kernel of the limited FP32 step, which also evaluates the
// limiter's raw coefficients of every tile it has finished: rho p at the nodes
// from the tile's FP32 u^n (the same values k_alpha_raw converts), staged in
// the pair-data region, then one lane per element takes the energy fraction
// and the coefficient; near a clip threshold it leaves -1 for k_alpha_fix's
// FP64 evaluation (measured: the FP64 evaluation here stalled the tile on
// fronts, 110.2 against 108.5 us per step).  It also empties the touched list
// for k_alpha_smooth.
template <class EQ, int N, typename R>
__global__ void __launch_bounds__(LaneLayout<EQ, N, R>::THREADS, LaneLayout<EQ, N, R>::MINB)
k_volume_lanes_ind(const double* __restrict__ u, R* __restrict__ rbar, R* __restrict__ trace,
                   DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb,
                   int slot, double* __restrict__ araw, unsigned* __restrict__ tcount, const LimTab lt) {
  static_assert(sizeof(R) == 4 && !EQ::NC, "the FP32 Euler form");
  using L = LaneLayout<EQ, N, R>;
  constexpr int DIM = EQ::DIM, n = N + 1, NP = L::NP;
  if (blockIdx.x == 0 && threadIdx.x == 0) *tcount = 0u;
  auto indicator = [&](long long e0, const float* sm) {
    float* smw = const_cast<float*>(sm);
    const int tid = threadIdx.x, l = tid / L::EPB, el = tid % L::EPB;
    const int nel = (int)min((long long)L::EPB, ma.E - e0);
    float* my = smw + (size_t)el * L::SZ;
    if (el < nel) {
      const float gm1 = ma.gamma_f - 1.0f;
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const int p = l * n + k;
        const float rho = my[L::O_U0 + p], Et = my[L::O_U0 + (DIM + 1) * NP + p];
        float mm = 0.0f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
          const float mk = my[L::O_U0 + (1 + d) * NP + p];
          mm += mk * mk;
        }
        my[L::O_Q + p] = gm1 * (rho * Et - 0.5f * mm);
      }
    }
    __syncthreads();
    if (tid < L::EPB && el < nel) {
      const float En = indicator_of_values<EQ, N, float>([&](int p) { return my[L::O_Q + p]; }, lt);
      const float a = alpha_of_energy_f32(En, lt);
      araw[e0 + el] = a >= 0.0f ? f2d_int(a) : -1.0;   // k_alpha_fix takes it in FP64
    }
  };
  volume_lanes_persistent<EQ, N, R, 0>(u, rbar, trace, st, ma, pp, tb, slot, true, indicator);
}

// volume part of one RKFR stage (input: the stage state)
template <class EQ, int N, typename R>
__global__ void __launch_bounds__(LaneLayout<EQ, N, R>::THREADS, LaneLayout<EQ, N, R>::MINB)
k_volume_lanes_stage(const double* __restrict__ u, R* __restrict__ rbar, R* __restrict__ trace,
                     DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb,
                     int slot, int first) {
  volume_lanes_persistent<EQ, N, R, 1>(u, rbar, trace, st, ma, pp, tb, slot, first != 0);
}

}  // namespace crk

namespace crk {

// ---------------------------------------------------------------------------
// Face + update kernel, lane form: 32 elements per CTA.  The jumps are computed
// with warp = face node, lane = element (every record a warp loads, own and
// neighbour, is a run of 32 consecutive elements of the [DIM][2][NF][C][E] trace
// array), the update with a thread per node in memory order.
// ---------------------------------------------------------------------------
template <class EQ, int N, typename R>
struct FaceLaneLayout {
  static constexpr int DIM = EQ::DIM, M = EQ::M, n = N + 1;
  static constexpr int NP = ipow(n, DIM), NF = NP / n;
  static constexpr int EPB = 32 * NF <= 1024 ? 32 : 16;   // elements per CTA (16: 3D, N = 5)
  static constexpr int THREADS = EPB * NF;
  // scaled jumps of every face: [DIM][side][M][face node][EPB elements], rows of
  // LD values (phase A writes a row per warp; in phase B the lanes of a warp
  // read several face nodes of few elements: 2 f + e falls into distinct banks)
  static constexpr int LD = EPB + 2;
  __host__ __device__ static constexpr int jump(int d, int side, int v) { return ((d * 2 + side) * M + v) * NF * LD; }
  static constexpr size_t bytes() { return sizeof(R) * (size_t)jump(DIM, 0, 0); }
  static constexpr bool fits() { return THREADS <= 1024 && bytes() <= 227 * 1024; }
  // Register budget of the face kernels, in resident threads per SM: the update
  // waits for memory, and registers spent on loads ahead of phase A (96 of
  // them) cost more warps than they hid.  us per launch, FP32, budget none /
  // 1024 / 1280 / 1536: 2D Euler 256^2 N = 3 29.8 / 23.0 / 21.0 / 22.7, TGV
  // 64^3 N = 3 797 / 559 / 556 / 513; GLM-MHD 128^2 N = 4 none / 768 / 1024 /
  // 1536 57.6 / 29.0 / 29.9 / 52 (spills); 64 batched solves 267 / 234 (1024) /
  // 221 (1152) / 228 (1280); RKFR 256^2 176 / 126 / 126 / 129.  3D N = 1, whose jumps
  // are most of its work, spills at 1536: 1024 (22x20x19 14.3 -> 10.5, 48^3 69.8 -> 53.5;
  // 768 56.4, 1280 54.6; the limited step's 15.7 -> 14.9, RKFR 32^3 31.0 -> 30.6).
  static constexpr int minb(int t) { return t / THREADS > 1 ? t / THREADS : 1; }
  // 1D: 512, for the values loaded ahead; none for the form with a thread per line.
  static constexpr bool WIDE = sizeof(R) == 8 || DIM == 1;
  static constexpr int MINB = minb(WIDE ? 512 : EQ::NC ? 768 : DIM == 3 ? (N == 1 ? 1024 : 1536) : 1280),
                       MINB1 = DIM == 1 ? 1 : minb(WIDE ? 512 : EQ::NC ? 768 : DIM == 3 && N == 1 ? 1024 : 1152),
                       MINB_OUT = DIM == 1 ? 1 : MINB;
};

// One tile of EPB elements starting at e0 (sj: the CTA's shared memory; slot:
// step parity of the CFL reduction).
//
// Phase A (warp = line index l, lane = element): every warp computes the Rusanov
// jumps of face node f = l of all 2 DIM faces of its elements, scaled by
// their correction factor, into shared memory: every record load is a run of 32
// elements, the same loads for every warp.
// Phase B (thread = node, in memory order): the tile's values of a variable are
// n contiguous runs of the CTA's threads; each node's increment (eq.
// crkfr.non.cons.final) is -dt R-bar plus the jumps of the faces it lies on,
// then the update, the CFL reduction and the store.  u^n, R-bar and u^{n+1} move
// in whole lines; with a thread per x-line (lane = element) each access of a
// warp touched 32 different lines, 20 x 32 of them per warp against 72 of the
// records (2D Euler, N = 3).  us per launch against that form, FP32: 2D Euler
// 256^2 N = 3 28.4 -> 21.0 (launches back to back; 22.4 us after an L2 flush,
// 5.4 TB/s of the algorithmic 116 B per node), 128^2 N = 4
// 18.9 -> 12.8, TGV 64^3 649 -> 513, GLM-MHD 128^2 N = 4 57.4 -> 29.0, RKFR 256^2
// 151 -> 124, 64 batched solves 329 -> 221; FP64 within 4% either way (its
// FP64 pipe is the bound).
// RK = true: stage mode of the multi-stage RKFR step (RkStage): the increment
// is the stage's K_j, combined with the earlier stages' into the next stage
// state (eq. rkfr1) or, at the last stage, into u^{n+1} (eq. rkfr2).
// FUSED: a tile of the fused single-launch step (crkfr_fused.cuh): dt comes
// from the caller (dt_fused), slot is the CFL reduction's write slot itself,
// and R-bar and the face records, written by other CTAs in the same launch,
// are read through L2.
// touched != nullptr (subcell blending limiter): the elements the limiter
// touches (blending coefficient of the element or of a face neighbour above
// zero, flagged by k_alpha_smooth) are left out -- k_face_update_limited takes
// them -- and u^{n+1} of the others goes to uout (the limited step keeps u^n
// intact).
template <class EQ, int N, typename R, bool RK = false, bool FUSED = false>
__device__ __forceinline__ void face_lanes_tile(double* __restrict__ u, const R* __restrict__ rbar,
                                                const R* __restrict__ trace, DevState* __restrict__ st,
                                                const MeshArgs& ma, const PhysParams<R>& pp, const RefTab<R>& tb,
                                                unsigned e0, int slot, R* __restrict__ sj,
                                                const RkStage<R>& rk = RkStage<R>{nullptr, nullptr, 0, 1},
                                                R dt_fused = R(0), const unsigned char* __restrict__ touched = nullptr,
                                                double* __restrict__ uout = nullptr) {
  using L = FaceLaneLayout<EQ, N, R>;
  constexpr int DIM = L::DIM, M = L::M, n = L::n, NP = L::NP, NF = L::NF, T = L::THREADS, LD = L::LD;
  constexpr bool F32 = sizeof(R) == 4;
  const int tid = threadIdx.x;
  const long long E = ma.E;
  // a volume CTA that timed out left its records unwritten: leave u^n as it is
  // (another output buffer gets it)
  if constexpr (!FUSED) {
    if (st->status & ST_TIMEOUT) {
      if (uout && !touched) {
        const size_t vt = (size_t)E * NP;
        for (int j = 0; j < n; ++j) {
          const int r = tid + j * T;
          if (r / NP < (int)min((long long)L::EPB, E - (long long)e0))
            for (int v = 0; v < M; ++v) uout[v * vt + (size_t)e0 * NP + r] = u[v * vt + (size_t)e0 * NP + r];
        }
      }
      return;
    }
  }
  const R dtR = FUSED ? dt_fused : step_dt<R>(st);
  const int nel = (int)min((long long)L::EPB, E - (long long)e0);
  const size_t vs = (size_t)E * NP;   // values per variable
  const size_t g0 = (size_t)e0 * NP + tid;

  // 1D: u^n and R-bar of all rounds ahead of phase A.  A round is M values a
  // thread there, and a mesh of a few thousand elements has less than one warp
  // per scheduler: each round's loads would be waited for in turn (us per step, FP32, before and
  // after: 2046 elements N = 1 10.4 -> 9.5, N = 5 14.6 -> 12.5, 30000 elements N = 3 14.3 -> 13.3, N = 5 23.8 ->
  // 22.8; 65536 N = 5 39.2 -> 37.4; FP64 within 1%, N = 1 20.1 -> 18.7).
  constexpr int AHEAD = DIM == 1 ? n : 1;
  double ua[AHEAD][M];
  R ra[AHEAD][M];
  if constexpr (DIM == 1) {
#pragma unroll
    for (int j = 0; j < n; ++j)
      if ((tid + j * T) / NP < nel)
#pragma unroll
        for (int v = 0; v < M; ++v) {
          ua[j][v] = u[g0 + j * T + v * vs];
          ra[j][v] = ldx<FUSED>(rbar + g0 + j * T + v * vs);
        }
  }

  // ---- phase A: scaled jumps, -dt J^- g_R'(1)/dx at the xi = 1 faces and
  // +dt J^+ (-g_L'(0))/dx at the xi = 0 faces
  {
    const int l = tid / L::EPB, el = tid % L::EPB;
    const unsigned e = e0 + el;
    if (el < nel && !(touched && touched[e])) {
      unsigned ec[3] = {0, 0, 0};
      elem_coords<DIM>(e, ma, ec);
#pragma unroll
      for (int d = 0; d < DIM; ++d)
#pragma unroll
        for (int side = 1; side >= 0; --side) {
          R J[M];
          face_jump<EQ, N, R, FUSED>(trace, E, d, side, e, neighbour_of(e, ec, d, side ? +1 : -1, ma), l, J, pp, tb);
          const R sc = side ? -(dtR * tb.iwN * inv_dx_of<R>(ma, d)) : dtR * tb.iw0 * inv_dx_of<R>(ma, d);
#pragma unroll
          for (int v = 0; v < M; ++v) sj[L::jump(d, side, v) + l * LD + el] = mulr(sc, J[v]);
        }
    }
  }
  __syncthreads();

  // ---- phase B
  R lam = R(0);
  bool bad = false;
  double* dst = uout ? uout : u;
  const bool last = !RK || rk.j == rk.s - 1;   // uniform over the grid
  if (RK && !last) dst = rk.uout;
  // FP64: a lower bound of the new state's maximum wave speed, from the warps
  // that have reduced theirs so far
  float thr = 0.0f;
  if constexpr (!F32) {
    if (last) thr = lambda_seen(st, FUSED ? slot : slot ^ 1);
  }
#pragma unroll AHEAD
  for (int j = 0; j < n; ++j) {
    const int r = tid + j * T, ee = r / NP, p = r % NP;
    const bool on = ee < nel && !(touched && touched[e0 + ee]);
    const size_t g = g0 + j * T;
    double un[M];
    if (on) {
      R du[M];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        if constexpr (DIM == 1) {
          un[v] = ua[j][v];
          du[v] = ra[j][v];
        } else {
          un[v] = u[g + v * vs];
          du[v] = ldx<FUSED>(rbar + g + v * vs);
        }
      }
      // the jumps of the faces the node lies on (one at most per direction: one
      // addition, whichever side), then -dt R-bar
      R t[M];
      int rem = p;
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        const int c = rem % n, stride = ipow(n, d);
        rem /= n;
        const int f = (p % stride) + (p / (stride * n)) * stride;
        R td[M];
#pragma unroll
        for (int v = 0; v < M; ++v) td[v] = R(0);
        if (c == 0 || c == N) {
          const R* src = sj + (c == N ? L::jump(0, 1, 0) : 0) + f * LD + ee;
#pragma unroll
          for (int v = 0; v < M; ++v) td[v] = src[L::jump(d, 0, v)];
        }
#pragma unroll
        for (int v = 0; v < M; ++v) t[v] = d == 0 ? td[v] : t[v] + td[v];
      }
#pragma unroll
      for (int v = 0; v < M; ++v) du[v] = mad(-dtR, du[v], t[v]);
      if constexpr (RK) {
        // du is this stage's K_j: keep it for the later stages and combine it
        // with the earlier ones (a_{j+1,q}, or b_q at the last stage)
        const R cj = last ? tb.b[rk.j] : tb.a[rk.j + 1][rk.j];
        R acc[M];
#pragma unroll
        for (int v = 0; v < M; ++v) {
          if (!last) rk.k[(size_t)rk.j * M * vs + v * vs + g] = du[v];
          acc[v] = mulr(cj, du[v]);
        }
#pragma unroll 1
        for (int q = 0; q < rk.j; ++q) {
          const R c = last ? tb.b[q] : tb.a[rk.j + 1][q];
          if (c != R(0)) {
#pragma unroll
            for (int v = 0; v < M; ++v) acc[v] = mad(c, rk.k[(size_t)q * M * vs + v * vs + g], acc[v]);
          }
        }
#pragma unroll
        for (int v = 0; v < M; ++v) du[v] = acc[v];
      }
      // u^{n+1} = u^n + du in FP64
#pragma unroll
      for (int v = 0; v < M; ++v) {
        if constexpr (F32) un[v] += f2d_int(du[v]);
        else un[v] += du[v];
        dst[g + v * vs] = un[v];
      }
    }
    if constexpr (F32) {
      if (last && on) {
        R lk;
        bad = bad || !physical_state<EQ, R>(un, ma, lk);
        lam = fmax(lam, lk);
      }
    } else {
      if (last) wave_speeds_fp64<EQ>(on, un, ma, thr, lam, bad);
    }
  }
  // the CFL reduction of the new state (RKFR: after the last stage only)
  if (last) reduce_lambda<R>(lam, bad, st, FUSED ? slot : slot ^ 1);
}

// n contiguous values of one line, in 16-byte accesses where VEC says that lines start
// on such a boundary (an array that does and an even n, or four floats, give it)
template <int n, bool VEC, typename T>
__device__ __forceinline__ void load_line(const T* __restrict__ src, T (&out)[n]) {
  constexpr int W = 16 / (int)sizeof(T);
  if constexpr (VEC && n % W == 0) {
#pragma unroll
    for (int k = 0; k < n / W; ++k) {
      const uint4 x = reinterpret_cast<const uint4*>(src)[k];
      memcpy(&out[k * W], &x, 16);
    }
  } else {
#pragma unroll
    for (int k = 0; k < n; ++k) out[k] = src[k];
  }
}
template <int n, bool VEC, typename T>
__device__ __forceinline__ void store_line(T* __restrict__ dst, const T (&in)[n]) {
  constexpr int W = 16 / (int)sizeof(T);
  if constexpr (VEC && n % W == 0) {
#pragma unroll
    for (int k = 0; k < n / W; ++k) {
      uint4 x;
      memcpy(&x, &in[k * W], 16);
      reinterpret_cast<uint4*>(dst)[k] = x;
    }
  } else {
#pragma unroll
    for (int k = 0; k < n; ++k) dst[k] = in[k];
  }
}

// 1D: a thread per element (its line of n nodes), the jumps of its two faces in
// registers, no exchange and no barrier.  The face part of a small mesh is one
// round trip to memory, which the two phases of face_lanes_tile make two, and an
// RKFR stage is a chain of them: the earlier increments K_q come in one load of
// all of a line's values per q here, not one per round and q.  Arithmetic and
// order are face_lanes_tile's: the same bits.  us per step, EC flux, two phases ->
// here: RKFR FP32 N = 3 64 elements 27.9 -> 20.6, 262144 130 -> 100, N = 5 64 77.5 -> 48.5, 9000
// 83.7 -> 60.0, 262144 545 -> 357, FP64 N = 5 2046 247 -> 224; limited FP32 N = 3 64 14.0 -> 11.3;
// the single-stage update's figures are at Variant::face_by_line.
// VEC: u and the output start on 16-byte boundaries (this library's own arrays do).
template <class EQ, int N, typename R, bool RK = false, bool VEC = true>
__device__ __forceinline__ void face_line(double* __restrict__ u, const R* __restrict__ rbar,
                                          const R* __restrict__ trace, DevState* __restrict__ st, const MeshArgs& ma,
                                          const PhysParams<R>& pp, const RefTab<R>& tb, int slot,
                                          const RkStage<R>& rk = RkStage<R>{nullptr, nullptr, 0, 1},
                                          const unsigned char* __restrict__ touched = nullptr,
                                          double* __restrict__ uout = nullptr) {
  static_assert(EQ::DIM == 1, "one line per element");
  constexpr int M = EQ::M, n = N + 1;
  constexpr bool F32 = sizeof(R) == 4;
  const long long E = ma.E;
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t vs = (size_t)E * n, g = (size_t)e * n;
  bool on = (long long)e < E;
  // as face_lanes_tile: u^n stays, another output buffer gets it
  if (st->status & ST_TIMEOUT) {
    if (uout && !touched && on)
      for (int v = 0; v < M; ++v)
        for (int k = 0; k < n; ++k) uout[v * vs + g + k] = u[v * vs + g + k];
    return;
  }
  on = on && !(touched && touched[e]);
  const bool last = !RK || rk.j == rk.s - 1;   // uniform over the grid
  double* dst = uout ? uout : u;
  if (RK && !last) dst = rk.uout;
  const R dtR = step_dt<R>(st);
  double un[M][n];
  if (on) {
    R du[M][n];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      load_line<n, true>(rbar + v * vs + g, du[v]);
      load_line<n, VEC>(u + v * vs + g, un[v]);
    }
    const unsigned ec[3] = {e, 0, 0};
    R J[2][M];
#pragma unroll
    for (int side = 1; side >= 0; --side) {
      face_jump<EQ, N, R>(trace, E, 0, side, e, neighbour_of(e, ec, 0, side ? +1 : -1, ma), 0, J[side], pp, tb);
      const R sc = side ? -(dtR * tb.iwN * inv_dx_of<R>(ma, 0)) : dtR * tb.iw0 * inv_dx_of<R>(ma, 0);
#pragma unroll
      for (int v = 0; v < M; ++v) J[side][v] = mulr(sc, J[side][v]);
    }
#pragma unroll
    for (int v = 0; v < M; ++v)
#pragma unroll
      for (int k = 0; k < n; ++k) du[v][k] = mad(-dtR, du[v][k], k == 0 ? J[0][v] : k == N ? J[1][v] : R(0));
    if constexpr (RK) {
      const R cj = last ? tb.b[rk.j] : tb.a[rk.j + 1][rk.j];
      R acc[M][n];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        if (!last) store_line<n, true>(rk.k + (size_t)rk.j * M * vs + v * vs + g, du[v]);
#pragma unroll
        for (int k = 0; k < n; ++k) acc[v][k] = mulr(cj, du[v][k]);
      }
#pragma unroll 1
      for (int q = 0; q < rk.j; ++q) {
        const R c = last ? tb.b[q] : tb.a[rk.j + 1][q];
        if (c != R(0)) {
#pragma unroll
          for (int v = 0; v < M; ++v) {
            R kq[n];
            load_line<n, true>(rk.k + (size_t)q * M * vs + v * vs + g, kq);
#pragma unroll
            for (int k = 0; k < n; ++k) acc[v][k] = mad(c, kq[k], acc[v][k]);
          }
        }
      }
#pragma unroll
      for (int v = 0; v < M; ++v)
#pragma unroll
        for (int k = 0; k < n; ++k) du[v][k] = acc[v][k];
    }
#pragma unroll
    for (int v = 0; v < M; ++v) {
#pragma unroll
      for (int k = 0; k < n; ++k) {
        if constexpr (F32) un[v][k] += f2d_int(du[v][k]);
        else un[v][k] += du[v][k];
      }
    }
  }
  // the reduction's atomics are under way when the stores begin
  if (last) {
    R lam = R(0);
    bool bad = false;
    float thr = 0.0f;
    if constexpr (!F32) thr = lambda_seen(st, slot ^ 1);
#pragma unroll
    for (int k = 0; k < n; ++k) {
      double uu[M];
#pragma unroll
      for (int v = 0; v < M; ++v) uu[v] = un[v][k];
      if constexpr (F32) {
        if (on) {
          R lk;
          bad = bad || !physical_state<EQ, R>(uu, ma, lk);
          lam = fmax(lam, lk);
        }
      } else {
        wave_speeds_fp64<EQ>(on, uu, ma, thr, lam, bad);
      }
    }
    reduce_lambda<R>(lam, bad, st, slot ^ 1);
  }
  if (on) {
#pragma unroll
    for (int v = 0; v < M; ++v) store_line<n, VEC>(dst + v * vs + g, un[v]);
  }
}

template <class EQ, int N, typename R>
__global__ void __launch_bounds__(32)
k_face_update_line(double* __restrict__ u, const R* __restrict__ rbar, const R* __restrict__ trace,
                   DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb, int slot) {
  face_line<EQ, N, R>(u, rbar, trace, st, ma, pp, tb, slot);
}

template <class EQ, int N, typename R>
__global__ void __launch_bounds__(FaceLaneLayout<EQ, N, R>::THREADS, FaceLaneLayout<EQ, N, R>::MINB)
k_face_update_lanes(double* __restrict__ u, const R* __restrict__ rbar, const R* __restrict__ trace,
                    DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb,
                    int slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  face_lanes_tile<EQ, N, R>(u, rbar, trace, st, ma, pp, tb, blockIdx.x * (unsigned)FaceLaneLayout<EQ, N, R>::EPB, slot,
                            reinterpret_cast<R*>(smem_raw));
}

// the same with the outputs of a step that keeps no record of its own
// (cr_step_noalloc); a kernel apart, since the pointers cost the plain one 1.5%
template <class EQ, int N, typename R>
__global__ void __launch_bounds__(FaceLaneLayout<EQ, N, R>::THREADS, FaceLaneLayout<EQ, N, R>::MINB_OUT)
k_face_update_lanes_out(double* __restrict__ u, const R* __restrict__ rbar, const R* __restrict__ trace,
                        DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb,
                        int slot, const FaceOut fo) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (blockIdx.x == 0) {
    if (fo.dt && threadIdx.x == 0) *fo.dt = st->dt;
    if (fo.reset && threadIdx.x < kLamSpread) st->lam_bits[slot][threadIdx.x] = 0ull;
  }
  if constexpr (EQ::DIM == 1) {
    // the caller's arrays: any 8-byte boundary
    const RkStage<R> none{nullptr, nullptr, 0, 1};
    if (((reinterpret_cast<size_t>(u) | reinterpret_cast<size_t>(fo.u)) & 15) == 0)
      face_line<EQ, N, R>(u, rbar, trace, st, ma, pp, tb, slot, none, nullptr, fo.u);
    else
      face_line<EQ, N, R, false, false>(u, rbar, trace, st, ma, pp, tb, slot, none, nullptr, fo.u);
  } else {
    face_lanes_tile<EQ, N, R>(u, rbar, trace, st, ma, pp, tb, blockIdx.x * (unsigned)FaceLaneLayout<EQ, N, R>::EPB,
                              slot, reinterpret_cast<R*>(smem_raw), RkStage<R>{nullptr, nullptr, 0, 1}, R(0), nullptr,
                              fo.u);
  }
}

// the limited step's elements that the limiter does not touch: the plain
// update from u^n (uin) into uout (touched: the flags of k_alpha_smooth)
template <class EQ, int N, typename R>
__global__ void __launch_bounds__(FaceLaneLayout<EQ, N, R>::THREADS, FaceLaneLayout<EQ, N, R>::MINB1)
k_face_update_lanes_clean(double* __restrict__ uin, double* __restrict__ uout, const R* __restrict__ rbar,
                          const R* __restrict__ trace, const unsigned char* __restrict__ touched,
                          DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb,
                          int slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if constexpr (EQ::DIM == 1)
    face_line<EQ, N, R>(uin, rbar, trace, st, ma, pp, tb, slot, RkStage<R>{nullptr, nullptr, 0, 1}, touched, uout);
  else
    face_lanes_tile<EQ, N, R>(uin, rbar, trace, st, ma, pp, tb, blockIdx.x * (unsigned)FaceLaneLayout<EQ, N, R>::EPB,
                              slot, reinterpret_cast<R*>(smem_raw), RkStage<R>{nullptr, nullptr, 0, 1}, R(0), touched,
                              uout);
}

// face / update part of stage rk.j of the multi-stage RKFR step
template <class EQ, int N, typename R>
__global__ void __launch_bounds__(FaceLaneLayout<EQ, N, R>::THREADS, FaceLaneLayout<EQ, N, R>::MINB1)
k_face_stage_lanes(double* __restrict__ u, const R* __restrict__ rbar, const R* __restrict__ trace,
                   DevState* __restrict__ st, const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb,
                   int slot, const RkStage<R> rk) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if constexpr (EQ::DIM == 1)
    face_line<EQ, N, R, true>(u, rbar, trace, st, ma, pp, tb, slot, rk);
  else
    face_lanes_tile<EQ, N, R, true>(u, rbar, trace, st, ma, pp, tb,
                                    blockIdx.x * (unsigned)FaceLaneLayout<EQ, N, R>::EPB, slot,
                                    reinterpret_cast<R*>(smem_raw), rk);
}

// ---------------------------------------------------------------------------
// Batched persistent form: many independent solves of one degree.  Each
// persistent CTA walks a work list of 32-element tiles spanning all solves
// (grid-stride); the solve's mesh, buffers and step record come from a
// device table.
// ---------------------------------------------------------------------------
struct BatchSolve {
  MeshArgs ma;
  double* u;
  void* rbar;
  void* trace;
  DevState* st;
  unsigned ntiles;     // tiles of this solve
  unsigned pad;
};
struct BatchTile {
  unsigned solve;
  unsigned e0;
};

template <class EQ, int N, typename R, int SH = 0>
__global__ void __launch_bounds__(LaneLayout<EQ, N, R, SH>::THREADS, LaneLayout<EQ, N, R, SH>::MINB)
k_volume_batched(const BatchSolve* __restrict__ solves, const BatchTile* __restrict__ tiles, unsigned ntiles,
                 const PhysParams<R> pp, const RefTab<R> tb, int slot) {
  using PL = PersistLayout<EQ, N, R>;
  constexpr int M = EQ::M, NP = LaneLayout<EQ, N, R>::NP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* sm = reinterpret_cast<R*>(smem_raw);
  double* staging = reinterpret_cast<double*>(smem_raw + PL::O_STAGE);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + PL::O_BAR);
  auto whole = [&](const BatchTile& t) {
    const BatchSolve& bs = solves[t.solve];
    return bs.ma.tma_ok && (long long)t.e0 + 32 <= bs.ma.E;
  };
  auto pf_of = [&](const BatchTile& t) {
    const BatchSolve& bs = solves[t.solve];
    return Prefetch{bs.u + (size_t)t.e0 * NP, bs.ma.E * NP, (unsigned)(32 * NP * sizeof(double)), staging, bar};
  };
  if (threadIdx.x == 0) mbar_init(bar, 1);
  __syncthreads();
  unsigned phase = 0;
  unsigned it = blockIdx.x;
  if (it < ntiles && threadIdx.x == 0) {
    const BatchTile t0 = tiles[it];
    if (whole(t0)) issue_prefetch<M>(pf_of(t0));
  }
  for (; it < ntiles; it += gridDim.x) {
    const BatchTile t = tiles[it];
    const BatchSolve& bs = solves[t.solve];
    const bool staged = whole(t);
    if (staged) {
      const bool ok = mbar_wait_bounded(bar, phase);
      if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {
          atomicOr(&bs.st->status, ST_TIMEOUT);
          mbar_wait_bounded(bar, phase);
        }
        return;
      }
      phase ^= 1u;
    }
    Prefetch pf{nullptr, 0, 0, nullptr, nullptr};
    if (it + gridDim.x < ntiles) {
      const BatchTile tn = tiles[it + gridDim.x];
      if (whole(tn)) pf = pf_of(tn);
    }
    const MeshArgs ma = bs.ma;
    // dt of this solve's step; its first tile records the step
    __shared__ double s_dt;
    if (threadIdx.x == 0) s_dt = step_begin(bs.st, slot, ma.cfl, ma.dt_fixed, t.e0 == 0);
    __syncthreads();
    volume_lanes_tile<EQ, N, R, SH>(bs.u, (R*)bs.rbar, (R*)bs.trace, bs.st, ma, pp, tb, (long long)t.e0,
                                dt_as<R>(s_dt), sm, staged ? staging : nullptr, pf);
    __syncthreads();   // shared memory is reused by the next tile
  }
}

template <class EQ, int N, typename R>
__global__ void __launch_bounds__(FaceLaneLayout<EQ, N, R>::THREADS, FaceLaneLayout<EQ, N, R>::MINB1)
k_face_batched(const BatchSolve* __restrict__ solves, const BatchTile* __restrict__ tiles, unsigned ntiles,
               const PhysParams<R> pp, const RefTab<R> tb, int slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  for (unsigned it = blockIdx.x; it < ntiles; it += gridDim.x) {
    const BatchTile t = tiles[it];
    const MeshArgs ma = solves[t.solve].ma;
    face_lanes_tile<EQ, N, R>(solves[t.solve].u, (const R*)solves[t.solve].rbar, (const R*)solves[t.solve].trace,
                              solves[t.solve].st, ma, pp, tb, t.e0, slot, reinterpret_cast<R*>(smem_raw));
    __syncthreads();   // the jump buffer is reused by the next tile
  }
}

}  // namespace crk
