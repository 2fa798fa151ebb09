// crkfr_volume_pairs.cuh -- the 1D volume kernel with a lane per pair of nodes,
// for meshes too small to fill the chip with a thread per element.
#pragma once
#include "crkfr_volume_lanes.cuh"

namespace crk {

// G lanes per element: lane g < n(n-1)/2 evaluates one pair flux of a stage, lane
// k <= N owns node k (stage state, pair data, residual); the lanes beyond repeat the
// last pair and node.  32 / G elements per CTA of one warp.
template <class EQ, int N>
struct PairLanes {
  static constexpr int n = N + 1, PAIRS = n * (n - 1) / 2;
  static constexpr int G = N == 2 ? 4 : N == 3 ? 8 : 16;
  static constexpr int EPB = 32 / G;
  static_assert(PAIRS <= G && n <= G, "a lane per pair and per node");
};

// The cRK stages of a few elements per warp (1D).  The lane form keeps the
// n(n-1)/2 pair fluxes of a line in one thread, one after the other; below a
// few thousand elements that chain is the launch's time, on a chip with one
// warp per SM or none.  Here a stage is one node evaluation, one exchange of the
// pair data, one pair flux and n - 1 exchanges of fluxes, on n(n-1)/2 times the
// lanes.  Each node adds its pair fluxes in the order of line_differences,
// and every product that meets a sum is rounded by itself (mulr, Euler::value): both
// forms give the same bits.  us per step (volume and face kernel, EC flux)
// with a thread per element -> here: 64 elements FP64 N = 3 54 -> 23.5, N = 5 167 -> 39,
// FP32 N = 3 10.5 -> 8.5, N = 5 18.5 -> 12.2; 2048 elements FP64 N = 3 54 -> 25, N = 5
// 167 -> 55, FP32 N = 5 19.3 -> 12.8.  In FP64 a warp instruction occupies the SM's
// FP64 pipe for 18 cycles whatever its lanes hold, so the lanes spent on
// repeats set the crossover (Variant::kPairElems).
template <class EQ, int N, typename R>
__global__ void __launch_bounds__(32)
k_volume_pairs(const double* __restrict__ u, R* __restrict__ rbar, R* __restrict__ trace, DevState* __restrict__ st,
               const MeshArgs ma, const PhysParams<R> pp, const RefTab<R> tb, int slot) {
  static_assert(EQ::DIM == 1 && !EQ::NC && EQ::VOL != VOL_CENTRAL, "1D Euler with a two-point flux");
  using PG = PairLanes<EQ, N>;
  constexpr int n = N + 1, M = EQ::M, P = EQ::P, G = PG::G, S = rk_stages(N);
  constexpr int NS = rk_nsaved(N) > 0 ? rk_nsaved(N) : 1;
  const int lane = threadIdx.x, g = lane % G, base = lane - g;
  const long long E = ma.E, e0 = (long long)blockIdx.x * PG::EPB + lane / G;
  const bool active = e0 < E;
  const long long e = active ? e0 : E - 1;
  const int k = g < N ? g : N;

  // the pair of this lane (pairs in lexicographic order), and for this node the
  // other node's pair lane and coefficients, in the order of that node
  int pa = N - 1, pb = N;
  {
    int idx = 0;
#pragma unroll
    for (int a = 0; a < n; ++a)
#pragma unroll
      for (int b = a + 1; b < n; ++b, ++idx)
        if (g == idx) { pa = a; pb = b; }
  }
  int src[N];
  R cA[N], cB[N];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int q = j < k ? j : j + 1;
    const int lo = min(k, q), hi = max(k, q);
    src[j] = base + lo * (2 * n - lo - 1) / 2 + hi - lo - 1;
    cA[j] = tb.A[0][k][q];
    cB[j] = tb.B[0][k][q];
  }
  const R diag = k == 0 ? R(2) * tb.B[0][0][0] : k == N ? R(2) * tb.B[0][N][N] : R(0);

  double dt = 0.0;
  if (lane == 0) dt = step_begin(st, slot, ma.cfl, ma.dt_fixed, blockIdx.x == 0);
  const R dtR = dt_as<R>(__shfl_sync(0xffffffffu, dt, 0));

  R u0[M], rb[M], r[M], rs[NS][M], U[M], F[M], lam = R(0);
#pragma unroll
  for (int v = 0; v < M; ++v) {
    const double x = u[((size_t)v * E + e) * n + k];
    if constexpr (sizeof(R) == 4) u0[v] = __double2float_rn(x);
    else u0[v] = x;
    rb[v] = r[v] = U[v] = F[v] = R(0);
  }
#pragma unroll 1
  for (int i = 0; i < S; ++i) {
    R w[M];
#pragma unroll
    for (int v = 0; v < M; ++v) w[v] = R(0);
    if (i > 0) {
      const R ap = dtR * tb.a[i][i - 1], bp = tb.b[i - 1];
#pragma unroll
      for (int v = 0; v < M; ++v) {
        rb[v] += bp * r[v];
        w[v] = mulr(ap, r[v]);
      }
      if constexpr (rk_nsaved(N) > 0) {
        const int sp = tb.slot[i - 1];
        if (sp >= 0) {
#pragma unroll
          for (int v = 0; v < M; ++v) rs[sp][v] = r[v];
        }
#pragma unroll 1
        for (int j = 0; j < i - 1; ++j) {
          const R c = dtR * tb.a[i][j];
          const int sj = tb.slot[j];
          if (sj >= 0 && c != R(0)) {
#pragma unroll
            for (int v = 0; v < M; ++v) w[v] += c * rs[sj][v];
          }
        }
      }
    }
    R uu[M], q[P], fn[M];
#pragma unroll
    for (int v = 0; v < M; ++v) uu[v] = u0[v] - w[v];
    EQ::pair_data(uu, q, pp);
    // face sums: of use at the two end nodes
    EQ::flux(0, q, fn, pp);
    EQ::cons_from_pair(q, uu, pp);
    if (i == 0) lam = EQ::wave_speed(0, q, pp);
    const R bi = tb.b[i];
#pragma unroll
    for (int v = 0; v < M; ++v) {
      U[v] += bi * uu[v];
      F[v] += bi * fn[v];
    }
    R qa[P], qb[P], f[M];
#pragma unroll
    for (int c = 0; c < P; ++c) {
      qa[c] = __shfl_sync(0xffffffffu, q[c], base + pa);
      qb[c] = __shfl_sync(0xffffffffu, q[c], base + pb);
    }
    EQ::two_point(0, qa, qb, f, pp);
    // (the inner nodes' own flux has coefficient zero: left out, not multiplied)
    const bool end = k == 0 || k == N;
#pragma unroll
    for (int v = 0; v < M; ++v) r[v] = end ? mulr(diag, fn[v]) : R(0);
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int v = 0; v < M; ++v) r[v] += (EQ::half(v) ? cB[j] : cA[j]) * __shfl_sync(0xffffffffu, f[v], src[j]);
  }
  if (!active || g > N) return;
#pragma unroll
  for (int v = 0; v < M; ++v) rbar[((size_t)v * E + e) * n + k] = rb[v] + tb.b[S - 1] * r[v];
  if (k == 0 || k == N) {
    R* dst = trace + trace_index<EQ, 1>(0, k ? 1 : 0, 0, 0, E, e);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      dst[(size_t)v * E] = U[v];
      dst[(size_t)(M + v) * E] = F[v];
    }
    dst[(size_t)(2 * M) * E] = lam;
  }
}

}  // namespace crk
