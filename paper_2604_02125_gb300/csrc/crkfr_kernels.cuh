// crkfr_kernels.cuh -- shared pieces of the cRKFR step kernels on sm_103a (the
// step's kernels are in crkfr_volume_lanes.cuh):
//
//  line_differences  flux differencing along one line (Sec. 3, eqs.
//                 entropy.cons.flux.dev, entropy.cons.noncons.dev)
//  face_jump      the jump of one face node: one time-averaged Rusanov flux
//                 (eq. numflux.cons) and the reduced-communication
//                 non-conservative flux B(u^{n,+-}) g^avg(U) (Sec. 2.3)
//  k_lambda       CFL reduction of a state (first step after set_state).
//  k_totals       FP64 quadrature-weighted totals (diagnostics).
// and the mesh and reference-element parameters, the step record and its
// fence-free CFL protocol (reduce_lambda / step_begin), element coordinates
// and periodic neighbours, the face-record layout.
//
// Layouts in HBM:
//   u     [M][E][NP] FP64        state, updated in place by the face / update kernel
//   rbar  [M][E][NP] R           sum_i b_i R(u^(i))
//   trace [DIM][2][NF][C][E] R   face data; side 0 = xi_d = 0 face, side 1 = xi_d = 1;
//         per face node C components, each contiguous over the elements
//         (a warp's 32 consecutive elements load one 128-byte line):
//         U (M), F^d (M), lambda_d(u^n) (1) [+ GLM-MHD: u^n (M)]
#pragma once
#include "crkfr_async.cuh"
#include "crkfr_physics.cuh"

namespace crk {

// Division of n < 2^31 by an invariant d >= 1 with one wide multiply:
// q = (n * m) >> (32 + l), l = ceil(log2 d), m = ceil(2^(32+l) / d) < 2^33.
// With m = 2^(32+l)/d + eps, 0 <= eps < 1, the quotient is n/d + n eps / 2^(32+l)
// and n eps / 2^(32+l) < 2^31 / 2^(32+l) <= 1/(2d), too small to change floor(n/d).
struct FastDiv {
  unsigned long long m;
  unsigned shift;   // 32 + l
  unsigned d;
};
__host__ __device__ inline FastDiv make_fastdiv(unsigned d) {
  unsigned l = 0;
  while ((1ull << l) < d) ++l;
  FastDiv f;
  f.d = d;
  f.shift = 32 + l;
  f.m = (((1ull << (32 + l)) + d - 1) / d);
  return f;
}
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv& f) {
  return (unsigned)(((unsigned long long)n * f.m) >> f.shift);
}

struct MeshArgs {
  long long E;          // elements; E * (N+1)^dim < 2^31 nodes per solve
  int cells[3];
  FastDiv cdiv[3];      // division by cells[k]
  double inv_dx[3];
  double cfl, dt_fixed;
  double gamma, c_h;
  float inv_dx_f[3], gamma_f, gm1_f, c_h_f;   // FP32 copies (no conversions on the FP64 pipe); gm1 = gamma - 1
  int tma_ok;           // state base 16-byte aligned and E * NP even: whole tiles can be bulk-copied
};
template <typename R> __device__ __forceinline__ R inv_dx_of(const MeshArgs& ma, int d);
template <> __device__ __forceinline__ double inv_dx_of<double>(const MeshArgs& ma, int d) { return ma.inv_dx[d]; }
template <> __device__ __forceinline__ float inv_dx_of<float>(const MeshArgs& ma, int d) { return ma.inv_dx_f[d]; }

// Coefficients of the flux differencing, D_pq = l_q'(xi_p) on [0,1].  A[d] and
// B[d] carry 1/dx_d of a single solve (d < 3), so its residuals need no scaling
// at the end of a line; A[3] and B[3] are without it (the batched kernels, which
// share one table among solves of different sizes, scale).
//   A: the pair coefficient of an unscaled row of the two-point flux, 2 D_pq
//      (Euler) or D_pq / 2 (GLM-MHD, whose two-point flux comes out times 4)
//   B: D_pq (rows scaled by two, the central flux, the non-conservative term)
// FP32: A2, B2 as ready register pairs (x, y) of the packed FP32x2 pair loop,
// [0] with 1/dx and 1/dy, [1] without (measured 53.8 -> 52.5 us per volume
// launch, 2D Euler 256^2, N = 3, against forming the pairs in the loop, and
// 52.7 -> 51.4 us for the folded 1/dx).
constexpr int kTabPlain = 3;
template <typename R>
struct RefTabPairs {};
template <>
struct RefTabPairs<float> {
  float2 A2[2][6][6], B2[2][6][6];
};
template <typename R>
struct RefTab : RefTabPairs<R> {
  R A[4][6][6], B[4][6][6];
  R iw0, iwN;      // 1/w_0, 1/w_N
  double w[6];     // quadrature weights (FP64, diagnostics)
  R a[7][7], b[7]; // Butcher tableau of the degree (same values as rk_a / rk_b)
  signed char slot[7];   // register slot of a stage residual needed beyond the next stage, else -1
};

// Step record of one solve.  The CFL reduction needs no fence and no
// ticket: the wave-speed maximum of a state is accumulated by fire-and-forget
// atomics into lam_bits[slot], where slot alternates with the step parity
// (the host passes it to every kernel); the volume kernel of the step that
// starts from that state reads it (kernel boundaries order the two), derives
// dt, records the step and clears the other slot for the new state.
// The fused single-launch step (crkfr_fused.cuh) reduces into a third slot: it
// rotates read / write / clear slots modulo 3, because its clear and its
// reductions happen within one launch.  epoch[] carries its per-step tile
// readiness value the same way.
// Each slot is spread over kLamSpread words: warp w of CTA b reduces into word
// (b NW + w) mod kLamSpread, and the step start takes the maximum of the
// words -- thousands of warps' atomics on a single word would serialise.
constexpr int kLamSpread = 32;
struct DevState {
  unsigned long long lam_bits[3][kLamSpread];   // max over nodes of sum_d lambda_d / dx_d (bits of a non-negative double)
  unsigned epoch[3];   // fused step: readiness value of the step that starts from a slot
  unsigned pad0;
  double dt;           // dt of the last step (set when the step starts)
  double t;            // time after the last step
  double lam_max;      // wave-speed maximum the last step's dt came from
  long long steps;
  unsigned status;     // bit 0: non-physical state, bit 1: barrier timeout
  unsigned pad;
};

constexpr unsigned ST_NONPHYS = 1u, ST_TIMEOUT = 2u;

// One stage of the multi-stage RKFR step (eq. rkfr.non.cons), for the face /
// update kernels in stage mode.  Stage j (0-based) of s forms the increment
// K_j = -dt R_FR(u^(j)) at every node and combines it with the earlier ones:
// u^(j+1) = u^n + sum_{q<=j} a_{j+1,q} K_q into uout, or, at the last stage,
// u^{n+1} = u^n + sum_q b_q K_q into the state (followed by the CFL
// reduction).  k holds K_0..K_{s-2}, [stage][var][elem][node].
template <typename R>
struct RkStage {
  R* k;
  double* uout;
  int j, s;
};

// What one face / update launch writes besides the state in place: u^{n+1} into
// another buffer (nullptr: in place), the step's dt, and (reset) zeros into the
// CFL slot the step has read, so that a record used for one step at a time
// starts the next one clean.
struct FaceOut {
  double* u;
  double* dt;
  int reset;
};

// ---------------------------------------------------------------------------
// CFL reduction: every warp takes its maximum with shuffles and folds it into
// its word of lam_bits[slot] with one 64-bit atomicMax (non-negative doubles order like
// their bit patterns; the result is not waited for).  Must be reached by every
// lane of the warp.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void reduce_lambda(T lam, bool bad, DevState* st, int slot) {
  for (int o = 16; o > 0; o >>= 1) lam = fmax(lam, __shfl_xor_sync(0xffffffffu, lam, o));
  const unsigned anybad = __ballot_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    if (anybad) atomicOr(&st->status, ST_NONPHYS);
    // a warp whose lanes did no work (maximum 0) leaves the slot alone: the
    // atomics of thousands of idle warps on one word would serialise
    if (lam > T(0)) {
      const unsigned word = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) % kLamSpread;
      atomicMax(&st->lam_bits[slot][word], (unsigned long long)__double_as_longlong((double)lam));
    }
  }
}

// dt of the step that starts now, from the wave-speed maximum of its initial
// state: cfl / max_nodes sum_d lambda_d/dx_d, or the fixed dt.  Every caller
// computes the same value; the one with lead set (one per solve and launch)
// records the step and clears the other slot for the new state's reduction.
__device__ __forceinline__ double step_begin_slots(DevState* st, int slot, int clear_slot, double cfl, double dt_fixed,
                                                   bool lead) {
  // all words loaded at once (one round trip), then reduced
  unsigned long long w[kLamSpread];
#pragma unroll
  for (int k = 0; k < kLamSpread; ++k) w[k] = st->lam_bits[slot][k];
  unsigned long long bits = 0ull;
#pragma unroll
  for (int k = 0; k < kLamSpread; ++k) bits = max(bits, w[k]);
  const double lam = __longlong_as_double((long long)bits);
  const double dt = dt_fixed > 0.0 ? dt_fixed : cfl / lam;
  if (lead) {
#pragma unroll 8
    for (int k = 0; k < kLamSpread; ++k) st->lam_bits[clear_slot][k] = 0ull;
    st->dt = dt;
    st->t += dt;
    st->steps += 1;
    st->lam_max = lam;
    if (!(lam > 0.0) || !isfinite(lam)) atomicOr(&st->status, ST_NONPHYS);
  }
  return dt;
}
__device__ __forceinline__ double step_begin(DevState* st, int slot, double cfl, double dt_fixed, bool lead) {
  return step_begin_slots(st, slot, slot ^ 1, cfl, dt_fixed, lead);
}


// Loads of data another CTA wrote earlier in the same launch (fused step):
// through L2 (ld.global.cg), never the non-coherent path or a stale L1 line.
template <bool COH, typename T>
__device__ __forceinline__ T ldx(const T* p) {
  if constexpr (COH) return __ldcg(p);
  else return *p;
}

// the current step's dt in the path's arithmetic (face kernels, after the
// volume kernel of the same step has recorded it)
template <typename R>
__device__ __forceinline__ R dt_as(double dt) {
  if constexpr (sizeof(R) == 4) return d2f_int(dt);
  else return dt;
}
template <typename R>
__device__ __forceinline__ R step_dt(const DevState* st) {
  return dt_as<R>(st->dt);
}


template <class EQ>
__host__ __device__ constexpr int trace_comps() { return EQ::NC ? 3 * EQ::M + 1 : 2 * EQ::M + 1; }
// component c of the record of face node f of face (d, side) of element e
template <class EQ, int NF>
__host__ __device__ __forceinline__ size_t trace_index(int d, int side, int f, int c, long long E, long long e) {
  return ((((size_t)(d * 2 + side) * NF + f) * trace_comps<EQ>() + c) * (size_t)E) + (size_t)e;
}
// Stage-wise non-conservative flux (EQ::NCS): after the records, the seven
// primitives of every stage's face trace, [DIM][2][NF][stage][7][E].
template <class EQ, int N>
__host__ __device__ constexpr size_t ncs_values_per_elem() {
  return (size_t)EQ::DIM * 2 * (ipow(N + 1, EQ::DIM) / (N + 1)) * rk_stages(N) * 7;
}
template <class EQ, int N>
__host__ __device__ __forceinline__ size_t ncs_index(int d, int side, int f, int j, int c, long long E, long long e) {
  constexpr int NF = ipow(N + 1, EQ::DIM) / (N + 1), S = rk_stages(N);
  const size_t base = (size_t)EQ::DIM * 2 * NF * trace_comps<EQ>() * (size_t)E;
  return base + (((((size_t)(d * 2 + side) * NF + f) * S + j) * 7 + c) * (size_t)E) + (size_t)e;
}
// the primitives of stage j at face node f of face (d, side) of element e
template <class EQ, int N, typename R>
__device__ __forceinline__ void write_stage_prims(R* __restrict__ trace, int d, int side, int f, int j, long long E,
                                                  long long e, const R* q) {
  if constexpr (EQ::NCS) {
    R w[7];
    EQ::stage_prims(q, w);
#pragma unroll
    for (int c = 0; c < 7; ++c) trace[ncs_index<EQ, N>(d, side, f, j, c, E, e)] = w[c];
  }
}

// node index of the first node of line l in direction d, and its stride
template <int n>
__device__ __forceinline__ int line_base(int l, int stride) { return (l % stride) + (l / stride) * stride * n; }

// element coordinates (x fastest) of element e
template <int DIM>
__device__ __forceinline__ void elem_coords(unsigned e, const MeshArgs& ma, unsigned (&c)[3]) {
  unsigned r = e;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    const unsigned q = (k == DIM - 1) ? 0u : fdiv(r, ma.cdiv[k]);
    c[k] = (k == DIM - 1) ? r : r - q * (unsigned)ma.cells[k];
    r = q;
  }
}
// periodic neighbour of element e (coordinates c) in direction d, offset +-1
__device__ __forceinline__ unsigned neighbour_of(unsigned e, const unsigned (&c)[3], int d, int off,
                                                 const MeshArgs& ma) {
  unsigned stride = 1;
  for (int k = 0; k < d; ++k) stride *= (unsigned)ma.cells[k];
  const unsigned nd = (unsigned)ma.cells[d];
  if (off > 0) return c[d] + 1 == nd ? e - (nd - 1) * stride : e + stride;
  return c[d] == 0 ? e + (nd - 1) * stride : e - stride;
}

// Flux differencing along one line of n = N+1 nodes in direction d from the
// pair data q: acc_p = (1/dx) (sum_q 2 D_pq f_S(q_p, q_q) [+ B(q_p) sum_q D_pq g(q_q)]).
// Every pair is evaluated once (f_S is symmetric); D_pp f(q_p) only at the two
// end points of a GLL line, where D_pp is non-zero.  The central flux,
// (f(q_p) + f(q_q))/2, is differenced as sum_q D_pq f(q_q), the same sum since
// the rows of D add up to zero.  fend: the physical fluxes at the two ends.
// PRE: coefficients with 1/dx of direction td; else the plain ones, and the
// result is scaled by inv_dx.
template <class EQ, int N, typename R, bool PRE>
__device__ __forceinline__ void line_differences(int d, const R (&q)[N + 1][EQ::P], R (&acc)[N + 1][EQ::M],
                                                 R (&fend)[2][EQ::M], const PhysParams<R>& pp, const RefTab<R>& tb,
                                                 int td, R inv_dx) {
  constexpr int n = N + 1, M = EQ::M;
  const R (&A)[6][6] = tb.A[PRE ? td : kTabPlain];
  const R (&B)[6][6] = tb.B[PRE ? td : kTabPlain];
  EQ::flux(d, q[0], fend[0], pp);
  EQ::flux(d, q[N], fend[1], pp);
  if constexpr (EQ::VOL == VOL_CENTRAL) {
#pragma unroll
    for (int a = 0; a < n; ++a)
#pragma unroll
      for (int v = 0; v < M; ++v) acc[a][v] = B[a][0] * fend[0][v] + B[a][N] * fend[1][v];
#pragma unroll
    for (int b = 1; b < N; ++b) {
      R f[M];
      EQ::flux(d, q[b], f, pp);
#pragma unroll
      for (int a = 0; a < n; ++a)
        if (a != b)   // D_bb = 0 at the inner nodes
#pragma unroll
          for (int v = 0; v < M; ++v) acc[a][v] += B[a][b] * f[v];
    }
  } else {
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
      for (int v = 0; v < M; ++v) acc[k][v] = R(0);
    const R c0 = R(2) * B[0][0], cN = R(2) * B[N][N];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      // 1D: rounded by itself, as in the form with a lane per pair (the sum of two
      // products below would leave the fused one to the compiler)
      acc[0][v] = EQ::DIM == 1 ? mulr(c0, fend[0][v]) : c0 * fend[0][v];
      acc[N][v] = EQ::DIM == 1 ? mulr(cN, fend[1][v]) : cN * fend[1][v];
    }
#pragma unroll
    for (int a = 0; a < n; ++a)
#pragma unroll
      for (int b = a + 1; b < n; ++b) {
        R f[M];
        EQ::two_point(d, q[a], q[b], f, pp);
#pragma unroll
        for (int v = 0; v < M; ++v) {
          acc[a][v] += (EQ::half(v) ? B[a][b] : A[a][b]) * f[v];
          acc[b][v] += (EQ::half(v) ? B[b][a] : A[b][a]) * f[v];
        }
      }
  }
  if constexpr (EQ::NC) {
    // sum_q D_pq B(u_p) g(u_q) = B(u_p) (D g)_p (no factor 2)
#pragma unroll
    for (int a = 0; a < n; ++a) {
      R dg[2] = {R(0), R(0)};
#pragma unroll
      for (int b = 0; b < n; ++b) {
        R g[2];
        EQ::ncg(d, q[b], g);
        dg[0] += B[a][b] * g[0];
        dg[1] += B[a][b] * g[1];
      }
      EQ::nc_apply(d, q[a], dg, acc[a]);
    }
  }
  if constexpr (!PRE) {
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
      for (int v = 0; v < M; ++v) acc[k][v] *= inv_dx;
  }
}

// physicality and sum_d lambda_d/dx_d of an updated state; the FP32 form
// evaluates the wave speeds in FP32 (the dt reduction is a max)
template <class EQ, typename R>
__device__ __forceinline__ bool physical_state(const double* uu, const MeshArgs& ma, R& lam) {
  if constexpr (sizeof(R) == 8) {
    if constexpr (EQ::NC) return EQ::physical(uu, ma.gamma, ma.c_h, lam, ma.inv_dx);
    else return EQ::physical(uu, ma.gamma, lam, ma.inv_dx);
  } else {
    float uf[EQ::M];
#pragma unroll
    for (int v = 0; v < EQ::M; ++v) uf[v] = d2f_rz(uu[v]);
    if constexpr (EQ::NC) return EQ::physical(uf, ma.gamma_f, ma.c_h_f, lam, ma.inv_dx_f);
    else return EQ::physical(uf, ma.gamma_f, lam, ma.inv_dx_f);
  }
}

// A lower bound (FP32, rounded toward zero) of the maximum that the CFL slot
// will hold: what the warps sharing this warp's word have reduced so far.
__device__ __forceinline__ float lambda_seen(const DevState* st, int slot) {
  const unsigned word = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) % kLamSpread;
  const unsigned long long b = *reinterpret_cast<const volatile unsigned long long*>(&st->lam_bits[slot][word]);
  return d2f_rz(__longlong_as_double((long long)b));
}

// Physicality and wave speeds of the warp's nodes (on: the lane has one) in the
// FP64 form.  Only a node that could raise the maximum is evaluated in FP64:
// one whose FP32 upper bound is below thr, a lower bound of the maximum, and
// which is certainly physical cannot change the result, which stays exactly the
// FP64 maximum over all nodes.  The evaluation (a division, square roots, about
// thirty instructions on the FP64 pipe) was half of this kernel's FP64 work.
// Called by whole warps; thr is raised to the warp's maximum.
template <class EQ>
__device__ __forceinline__ void wave_speeds_fp64(bool on, const double* uu, const MeshArgs& ma, float& thr, double& lam,
                                                 bool& bad) {
  bool need = false;
  if (on) {
    float uf[EQ::M], up;
#pragma unroll
    for (int v = 0; v < EQ::M; ++v) uf[v] = d2f_rz(uu[v]);
    const bool sure = EQ::speed_bound(uf, MeshSpeeds{ma.gamma_f, ma.gm1_f, ma.c_h_f, ma.inv_dx_f}, up);
    need = !sure || !(up < thr);
  }
  if (__any_sync(0xffffffffu, need)) {
    if (need) {
      double lk;
      bad = !physical_state<EQ, double>(uu, ma, lk) || bad;
      lam = fmax(lam, lk);
    }
    // non-negative floats order like their bits; fmaxf drops the NaN of a value
    // beyond the FP32 range, and thr stays the bound it was
    thr = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(thr, d2f_rz(lam)))));
  }
}

// the C components of the record of face node f of face (d, side) of element e
template <class EQ, int N, typename R, bool COH = false>
__device__ __forceinline__ void load_face_record(const R* __restrict__ trace, long long E, int d, int side, int f,
                                                 long long e, R (&rec)[trace_comps<EQ>()]) {
  constexpr int NF = ipow(N + 1, EQ::DIM) / (N + 1), C = trace_comps<EQ>();
  const R* p = trace + trace_index<EQ, NF>(d, side, f, 0, E, e);
#pragma unroll
  for (int c = 0; c < C; ++c) rec[c] = ldx<COH>(p + (size_t)c * E);
}

// Jump J = F^num - F_own [+ B(u^n_own) g^avg(U)] at one face node
// from the own record o and the other side's record x (eq. numflux.cons and
// the reduced-communication non-conservative flux of Sec. 2.3).
template <class EQ, typename R>
__device__ __forceinline__ void jump_of(const R* o, const R* x, int d, int side_own, R* J, const PhysParams<R>& pp) {
  constexpr int M = EQ::M;
  const R lam = fmax(o[2 * M], x[2 * M]);
  // own is the '-' state when it is the xi = 1 side: U+ - U- = sgn (Ux - Uo)
  const R sgn = side_own == 1 ? R(1) : R(-1);
#pragma unroll
  for (int v = 0; v < M; ++v)
    J[v] = mad(R(0.5), o[M + v] + x[M + v], mulr(R(-0.5) * lam * sgn, x[v] - o[v])) - o[M + v];
  if constexpr (EQ::NC) {
    // + B(u^n_own) (g^avg(U) - g(u^n_own)) (the stage-wise flux adds its own sum in
    // face_jump instead); the rest of - F^nc_own is part of R-bar
    // (nonconservative_ends)
    if constexpr (!EQ::NCS) {
      R un[M], q[EQ::P];
#pragma unroll
      for (int v = 0; v < M; ++v) un[v] = o[2 * M + 1 + v];
      EQ::pair_data(un, q, pp);
      R g[2];
      g[0] = R(0.5) * ((o[5 + d] - un[5 + d]) + (x[5 + d] - un[5 + d]));
      g[1] = R(0.5) * ((o[8] - un[8]) + (x[8] - un[8]));
      EQ::nc_apply(d, q, g, J);
    }
  }
}

template <class EQ, int N, typename R, bool COH = false>
__device__ __forceinline__ void face_jump(const R* __restrict__ trace, long long E, int d, int side_own, long long e_own,
                                          long long e_oth, int f, R* J, const PhysParams<R>& pp, const RefTab<R>& tb) {
  constexpr int C = trace_comps<EQ>();
  R o[C], x[C];
  load_face_record<EQ, N, R, COH>(trace, E, d, side_own, f, e_own, o);
  load_face_record<EQ, N, R, COH>(trace, E, d, 1 - side_own, f, e_oth, x);
  jump_of<EQ, R>(o, x, d, side_own, J, pp);
  if constexpr (EQ::NCS) {
    // + sum_j b_j B(u^(j)_own) (g^avg - g)(u^(j)), F^nc_own of eq.
    // bad.numflux.non.cons included
#pragma unroll 1
    for (int j = 0; j < rk_stages(N); ++j) {
      R wo[7], wx[7];
#pragma unroll
      for (int c = 0; c < 7; ++c) {
        wo[c] = trace[ncs_index<EQ, N>(d, side_own, f, j, c, E, e_own)];
        wx[c] = trace[ncs_index<EQ, N>(d, 1 - side_own, f, j, c, E, e_oth)];
      }
      R go[2], gx[2], g[2], nc[EQ::M];
      EQ::ncg_prims(d, wo, go);
      EQ::ncg_prims(d, wx, gx);
      g[0] = R(0.5) * (gx[0] - go[0]);
      g[1] = R(0.5) * (gx[1] - go[1]);
#pragma unroll
      for (int v = 0; v < EQ::M; ++v) nc[v] = R(0);
      EQ::nc_apply_prims(d, wo, g, nc);
#pragma unroll
      for (int v = 0; v < EQ::M; ++v) J[v] += tb.b[j] * nc[v];
    }
  }
}

// CFL reduction of the current state (used after set_state); wave speeds in
// the path's arithmetic R, like the reduction of the face / update kernel
template <class EQ, int N, typename R>
__global__ void __launch_bounds__(256)
k_lambda(const double* __restrict__ u, DevState* __restrict__ st, const MeshArgs ma, int slot, int fresh) {
  constexpr int M = EQ::M, NP = ipow(N + 1, EQ::DIM);
  const long long E = ma.E;
  const unsigned gid = blockIdx.x * blockDim.x + threadIdx.x;
  // fresh: drop the timeout an earlier step left in a reused record.  Only that bit,
  // which nothing in this launch sets: a store of 0 could fall on either side of
  // the other warps' atomicOr of ST_NONPHYS.
  if (fresh && gid == 0) atomicAnd(&st->status, ~ST_TIMEOUT);
  R lam = R(0);
  bool bad = false;
  if (gid < (unsigned)(E * NP)) {
    const unsigned e = gid / NP;
    const int p = (int)(gid % NP);
    double uu[M];
#pragma unroll
    for (int v = 0; v < M; ++v) uu[v] = u[((size_t)v * E + e) * NP + p];
    bad = !physical_state<EQ, R>(uu, ma, lam);
  }
  reduce_lambda<R>(lam, bad, st, slot);
}

// FP64 quadrature-weighted totals: per block partial sums, fixed order
template <class EQ, int N>
__global__ void __launch_bounds__(256)
k_totals(const double* __restrict__ u, double* __restrict__ part, const MeshArgs ma, const RefTab<double> tb) {
  constexpr int DIM = EQ::DIM, M = EQ::M, n = N + 1, NP = ipow(n, DIM), K = M + 2;
  const long long E = ma.E;
  const unsigned gid = blockIdx.x * blockDim.x + threadIdx.x;
  double acc[K];
#pragma unroll
  for (int k = 0; k < K; ++k) acc[k] = 0.0;
  if (gid < (unsigned)(E * NP)) {
    const unsigned e = gid / NP;
    const int p = (int)(gid % NP);
    double wq = 1.0;
    int rem = p;
#pragma unroll
    for (int d = 0; d < DIM; ++d) { wq *= tb.w[rem % n] / ma.inv_dx[d]; rem /= n; }
    double uu[M];
#pragma unroll
    for (int v = 0; v < M; ++v) { uu[v] = u[((size_t)v * E + e) * NP + p]; acc[v] = wq * uu[v]; }
    double rho = uu[0], ke = 0.0, p_;
    if constexpr (EQ::NC) {
      double vv = (uu[1] * uu[1] + uu[2] * uu[2] + uu[3] * uu[3]) / rho;
      ke = 0.5 * vv;
      p_ = (ma.gamma - 1.0) * (uu[4] - ke - 0.5 * (uu[5] * uu[5] + uu[6] * uu[6] + uu[7] * uu[7]) - 0.5 * uu[8] * uu[8]);
    } else {
      double mm = 0.0;
#pragma unroll
      for (int k = 0; k < DIM; ++k) mm += uu[1 + k] * uu[1 + k];
      ke = 0.5 * mm / rho;
      p_ = (ma.gamma - 1.0) * (uu[DIM + 1] - ke);
    }
    acc[M] = wq * ke;
    acc[M + 1] = wq * (-rho * (log(p_) - ma.gamma * log(rho)) / (ma.gamma - 1.0));
  }
  __shared__ double s[K][256];
#pragma unroll
  for (int k = 0; k < K; ++k) s[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h)
#pragma unroll
      for (int k = 0; k < K; ++k) s[k][threadIdx.x] += s[k][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) part[(size_t)blockIdx.x * K + k] = s[k][0];
}

}  // namespace crk
