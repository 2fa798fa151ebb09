// cr_variant.cuh -- launchers of one (system, degree, precision) variant.
#pragma once
#include "cr_internal.h"
#include "crkfr_volume_lanes.cuh"
#include "crkfr_volume_pairs.cuh"

#include <algorithm>
#include <atomic>

namespace crk {

template <typename R> struct PP;
template <> struct PP<double> {
  static const PhysParams<double>& get(const LaunchCtx& c) { return c.pp64; }
  static const RefTab<double>& tab(const LaunchCtx& c) { return c.tb64; }
};
template <> struct PP<float> {
  static const PhysParams<float>& get(const LaunchCtx& c) { return c.pp32; }
  static const RefTab<float>& tab(const LaunchCtx& c) { return c.tb32; }
};

template <typename R> struct PPB;
template <> struct PPB<double> {
  static const PhysParams<double>& get(const BatchLaunch& b) { return b.pp64; }
  static const RefTab<double>& tab(const BatchLaunch& b) { return b.tb64; }
};
template <> struct PPB<float> {
  static const PhysParams<float>& get(const BatchLaunch& b) { return b.pp32; }
  static const RefTab<float>& tab(const BatchLaunch& b) { return b.tb32; }
};

constexpr int kOccDevices = 64;   // devices whose occupancies are kept

template <class EQ, int N, typename R>
struct Variant {
  using LL = LaneLayout<EQ, N, R>;
  using PL = PersistLayout<EQ, N, R>;
  using FL = FaceLaneLayout<EQ, N, R>;
  static_assert(PL::fits() && FL::fits(), "the lane layouts hold every variant");
  // Resident CTAs per SM of a persistent kernel on the current device, whose
  // shared-memory allowance set_smem has raised: asked for once per device (a call
  // costs several microseconds), by whichever thread comes first, since
  // all of them get the same answer.  0: not known yet.
  using OccCache = std::atomic<int>[kOccDevices];
  template <class K>
  static int occupancy_of(OccCache& cache, K k, int threads, size_t bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
    const bool known = dev >= 0 && dev < kOccDevices;
    int nb = known ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (nb == 0) {
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, threads, bytes);
      if (known) cache[dev].store(nb, std::memory_order_relaxed);
    }
    return nb;
  }
  template <int SH>
  static int vol_occupancy() {
    using PS = PersistLayout<EQ, N, R, SH>;
    static OccCache occ;
    return std::max(1, occupancy_of(occ, k_volume_lanes<EQ, N, R, SH>, PS::L::THREADS, PS::bytes()));
  }
  template <int SH>
  static cudaError_t volume_shape(const LaunchCtx& c, cudaStream_t s) {
    using PS = PersistLayout<EQ, N, R, SH>;
    const long long ntiles = (c.ma.E + PS::L::EPB - 1) / PS::L::EPB;
    const long long grid = std::min(ntiles, (long long)c.sms * vol_occupancy<SH>());
    k_volume_lanes<EQ, N, R, SH><<<(unsigned)grid, PS::L::THREADS, PS::bytes(), s>>>(
        c.u, (R*)c.rbar, (R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot);
    return cudaGetLastError();
  }
  // FP64: tiles of 8 or 16 elements (LaneLayout<.., 2>).  The FP64 pipe bounds the
  // launch, so its time is that of the SM with the most warps of work, and
  // smaller tiles spread a mesh more evenly.  Where they fill whole warps (2D N = 1, 3,
  // 5, 3D N = 1, 3) they are never more work and always taken; else where the
  // busiest SM has fewer warps.  us per step, default against small tiles: 2D Euler N = 3
  // 97x61 225 -> 171, 200^2 870 -> 850, N = 5 40x33 699 -> 505, 200^2 4492 -> 4265, GLM-MHD N = 3
  // 97x61 596 -> 378, 61x45 310 -> 295, TGV N = 3 8x9x11 361 -> 238, 22x20x19 1297 -> 1270; by the
  // rule: 2D N = 4 40x33 399 -> 324 (42 tiles, 5 warps against 3), 97x61 586 -> 548, but
  // 200^2 2344 against 2659 (45 warps against 51), TGV N = 2 8x9x11 211 -> 116, 22x20x19
  // 415 against 496.
  static constexpr bool kSmall = sizeof(R) == 8 && EQ::DIM > 1 && LaneLayout<EQ, N, R, 2>::EPB < LL::EPB;
  static constexpr bool kSmallOnly = kSmall && LaneLayout<EQ, N, R, 2>::THREADS % 32 == 0;
  // warps of work on the SM with the most tiles
  template <int SH>
  static long long warps_per_sm(const LaunchCtx& c) {
    using L = LaneLayout<EQ, N, R, SH>;
    const long long ntiles = (c.ma.E + L::EPB - 1) / L::EPB;
    return (ntiles + c.sms - 1) / c.sms * ((L::THREADS + 31) / 32);
  }
  // the form for a mesh: decides the launch and what cr_tuning_info reports
  static VolForm vol_form(const LaunchCtx& c) {
    if constexpr (kPairs) {
      if (c.ma.E <= kPairElems * c.sms) return VolForm::Pairs;
    }
    if constexpr (kSmallOnly) return VolForm::SmallTiles;
    if constexpr (kSmall) {
      if (warps_per_sm<2>(c) < warps_per_sm<0>(c)) return VolForm::SmallTiles;
    }
    return VolForm::Lanes;
  }
  static cudaError_t volume(const LaunchCtx& c, cudaStream_t s) {
    const VolForm form = vol_form(c);
    if constexpr (kPairs) {
      if (form == VolForm::Pairs) return volume_pairs(c, s);
    }
    if constexpr (kSmall) {
      if (kSmallOnly || form == VolForm::SmallTiles) return volume_shape<2>(c, s);
    }
    if constexpr (!kSmallOnly) return volume_shape<0>(c, s);
    return cudaErrorNotSupported;
  }
  // 1D, few elements: a lane per pair of nodes (k_volume_pairs).  The form with a
  // thread per element takes the same time from 1 to 32 elements per SM; the
  // pair form's grows beyond 8 to 16, and they meet at 35 to 80 elements per SM
  // (FP32 with the Kennedy-Gruber flux, the cheapest, at 20 to 35).
  static constexpr bool kPairs = EQ::DIM == 1 && !EQ::NC && EQ::VOL != VOL_CENTRAL && N >= 2;
  static constexpr long long kPairElems = sizeof(R) == 4 && EQ::VOL == VOL_KEP ? 16 : 24;
  static cudaError_t volume_pairs(const LaunchCtx& c, cudaStream_t s) {
    constexpr int EPB = PairLanes<EQ, N>::EPB;
    k_volume_pairs<EQ, N, R><<<(unsigned)((c.ma.E + EPB - 1) / EPB), 32, 0, s>>>(
        c.u, (R*)c.rbar, (R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot);
    return cudaGetLastError();
  }
  static cudaError_t volume_stage(const LaunchCtx& c, cudaStream_t s, const double* u_in, int first) {
    const long long ntiles = (c.ma.E + LL::EPB - 1) / LL::EPB;
    const long long grid = std::min(ntiles, (long long)c.sms * vol_stage_occupancy());
    k_volume_lanes_stage<EQ, N, R><<<(unsigned)grid, LL::THREADS, PL::bytes(), s>>>(
        u_in, (R*)c.rbar, (R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot, first);
    return cudaGetLastError();
  }
  static int vol_stage_occupancy() {
    static OccCache occ;
    return std::max(1, occupancy_of(occ, k_volume_lanes_stage<EQ, N, R>, LL::THREADS, PL::bytes()));
  }
  static unsigned face_tiles(const LaunchCtx& c) { return (unsigned)((c.ma.E + FL::EPB - 1) / FL::EPB); }
  static cudaError_t face_stage(const LaunchCtx& c, cudaStream_t s, int j, int ns) {
    const RkStage<R> rk{(R*)c.kbuf, j == ns - 1 ? c.u : c.ustage, j, ns};
    k_face_stage_lanes<EQ, N, R><<<face_tiles(c), FL::THREADS, FL::bytes(), s>>>(
        c.u, (const R*)c.rbar, (const R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot, rk);
    return cudaGetLastError();
  }
  // 1D: the update kernel with a thread per line (face_line) or per node
  // (face_lanes_tile).  us per step, EC flux, line against node.  FP32: N = 1 9000
  // elements 6.13 / 6.28, 131072 12.6 / 13.8; N = 3 9000 9.10 / 9.47, 131072 21.5 /
  // 23.0, 262144 33.6 / 35.3: always the line.  N = 2 64 5.73 / 5.97, 16000 7.31 /
  // 7.43; its lines of three have no 16-byte accesses, and from the
  // L2's capacity on a thread per node moves them better (262144 26.1 / 24.8).  N = 4 and 5 hold too much
  // per thread: N = 4 64 8.71 / 8.47, 30000 16.5 / 15.8, 262144 (face launch) 24.5 /
  // 18.9.  FP64, all degrees: N = 5 64 41.9 / 43.9, 2046 52.1 / 52.8; N = 4 30000
  // (face launch) 19.9 / 18.6, 65536 32.6 / 27.8.
  static bool face_by_line(const LaunchCtx& c) {
    if (EQ::DIM > 1) return false;
    if (sizeof(R) == 8) return c.ma.E <= 96LL * c.sms;
    return N == 1 || N == 3 || (N == 2 && c.ma.E <= 1024LL * c.sms);
  }
  static constexpr bool kBatched = EQ::DIM == 2 && !EQ::NC;
  static_assert(!kBatched || (LL::EPB == 32 && FL::EPB == 32), "the work list holds 32-element tiles");
  static cudaError_t face_update(const LaunchCtx& c, cudaStream_t s) {
    if constexpr (EQ::DIM == 1) {
      if (!c.out.reset && face_by_line(c)) {
        k_face_update_line<EQ, N, R><<<face_tiles(c), FL::THREADS, 0, s>>>(
            c.u, (const R*)c.rbar, (const R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot);
        return cudaGetLastError();
      }
    }
    if (c.out.reset)
      k_face_update_lanes_out<EQ, N, R><<<face_tiles(c), FL::THREADS, FL::bytes(), s>>>(
          c.u, (const R*)c.rbar, (const R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot, c.out);
    else
      k_face_update_lanes<EQ, N, R><<<face_tiles(c), FL::THREADS, FL::bytes(), s>>>(
          c.u, (const R*)c.rbar, (const R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot);
    return cudaGetLastError();
  }
  static constexpr bool kVolInd = !EQ::NC && sizeof(R) == 4;
  static cudaError_t volume_ind(const LaunchCtx& c, cudaStream_t s) {
    if constexpr (kVolInd) {
      static OccCache occ;
      const int per_sm = std::max(1, occupancy_of(occ, k_volume_lanes_ind<EQ, N, R>, LL::THREADS, PL::bytes()));
      const long long ntiles = (c.ma.E + LL::EPB - 1) / LL::EPB;
      const long long grid = std::min(ntiles, (long long)c.sms * per_sm);
      k_volume_lanes_ind<EQ, N, R><<<(unsigned)grid, LL::THREADS, PL::bytes(), s>>>(
          c.u, (R*)c.rbar, (R*)c.trace, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c), c.slot, c.araw, c.tcount, c.lt);
      return cudaGetLastError();
    }
    return cudaErrorNotSupported;
  }
  static cudaError_t alpha_smooth(const LaunchCtx& c, cudaStream_t s) {
    if constexpr (kVolInd) {
      k_alpha_fix<EQ, N><<<(unsigned)((c.ma.E + 127) / 128), 128, 0, s>>>(c.u, c.araw, c.ma, c.lt);
      k_alpha_smooth<EQ::DIM><<<(unsigned)((c.ma.E + 255) / 256), 256, 0, s>>>(c.araw, c.alpha, c.touched, c.tlist,
                                                                              c.tcount, c.ma);
      return cudaGetLastError();
    }
    return cudaErrorNotSupported;
  }
  // FP64: the raw coefficients, then the smoothing pass (FP32: volume_ind, alpha_smooth)
  static cudaError_t alpha(const LaunchCtx& c, cudaStream_t s) {
    if constexpr (!EQ::NC && !kVolInd) {
      constexpr int T = AlphaRawLayout<EQ, N>::THREADS;
      const unsigned grid = (unsigned)((c.ma.E + T - 1) / T);
      k_alpha_raw<EQ, N><<<grid, T, 0, s>>>(c.u, c.araw, c.tcount, c.ma, c.lt);
      k_alpha_smooth<EQ::DIM><<<(unsigned)((c.ma.E + 255) / 256), 256, 0, s>>>(c.araw, c.alpha, c.touched, c.tlist,
                                                                              c.tcount, c.ma);
      return cudaGetLastError();
    }
    return cudaErrorNotSupported;
  }
  // the limited face / update part: the lane kernel for the elements the
  // limiter does not touch, the per-node limited kernel for the others
  static cudaError_t face_limited(const LaunchCtx& c, cudaStream_t s) {
    if constexpr (!EQ::NC) {
      k_face_update_lanes_clean<EQ, N, R><<<face_tiles(c), FL::THREADS, FL::bytes(), s>>>(
          c.u, c.u_next, (const R*)c.rbar, (const R*)c.trace, c.touched, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c),
          c.slot);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
      // their number is known on the device only: a grid of four CTAs per SM
      // strides over the touched elements' nodes
      const long long total = c.ma.E * LL::NP;
      const unsigned grid = (unsigned)std::min((total + 255) / 256, 4LL * c.sms);
      k_face_update_limited<EQ, N, R><<<grid, 256, 0, s>>>(c.u, c.u_next, (const R*)c.rbar, (const R*)c.trace, c.alpha,
                                                           c.tlist, c.tcount, c.st, c.ma, PP<R>::get(c), PP<R>::tab(c),
                                                           c.lt, c.slot);
      return cudaGetLastError();
    }
    return cudaErrorNotSupported;
  }
  using FU = FusedLayout<EQ, N, R>;
  static constexpr bool kFused = FU::fits() && !EQ::NC && LL::EPB == 32;
  static int fused_occupancy() {
    if constexpr (kFused) {
      static OccCache occ;
      return occupancy_of(occ, k_step_fused<EQ, N, R>, LL::THREADS, FU::bytes());
    }
    return 0;
  }
  static cudaError_t step_fused(const LaunchCtx& c, cudaStream_t s, int phase) {
    if constexpr (kFused) {
      const int occ = fused_occupancy();
      if (occ < 1) return cudaErrorInvalidConfiguration;
      const long long ntiles = (c.ma.E + LL::EPB - 1) / LL::EPB;
      // cooperative: every CTA resident, so the bounded readiness waits end
      const long long grid = std::min(ntiles, (long long)c.sms * occ);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)grid);
      cfg.blockDim = dim3(LL::THREADS);
      cfg.dynamicSmemBytes = FU::bytes();
      cfg.stream = s;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      return cudaLaunchKernelEx(&cfg, k_step_fused<EQ, N, R>, c.u, (R*)c.rbar, (R*)c.trace, c.st, c.flags, c.ma,
                                PP<R>::get(c), PP<R>::tab(c), phase);
    }
    return cudaErrorNotSupported;
  }
  static cudaError_t lambda(const LaunchCtx& c, cudaStream_t s) {
    const long long total = c.ma.E * LL::NP;
    const unsigned grid = (unsigned)((total + 255) / 256);
    k_lambda<EQ, N, R><<<grid, 256, 0, s>>>(c.u, c.st, c.ma, c.slot, c.out.reset);
    return cudaGetLastError();
  }
  static cudaError_t totals(const LaunchCtx& c, cudaStream_t s) {
    const long long total = c.ma.E * LL::NP;
    const unsigned grid = (unsigned)((total + 255) / 256);
    k_totals<EQ, N><<<grid, 256, 0, s>>>(c.u, c.totals_part, c.ma, c.tb64);
    return cudaGetLastError();
  }
  template <class K>
  static cudaError_t allow(K k, size_t bytes) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  }
  // dynamic shared memory of every kernel of the variant
  static cudaError_t set_smem() {
    cudaError_t e = cudaSuccess;
    if constexpr (!kSmallOnly) e = allow(k_volume_lanes<EQ, N, R>, PL::bytes());
    if constexpr (kSmall) {
      if (e == cudaSuccess) e = allow(k_volume_lanes<EQ, N, R, 2>, PersistLayout<EQ, N, R, 2>::bytes());
    }
    if (e == cudaSuccess) e = allow(k_volume_lanes_stage<EQ, N, R>, PL::bytes());
    if constexpr (kVolInd) {
      if (e == cudaSuccess) e = allow(k_volume_lanes_ind<EQ, N, R>, PL::bytes());
    }
    if (e == cudaSuccess) e = allow(k_face_update_lanes<EQ, N, R>, FL::bytes());
    if (e == cudaSuccess) e = allow(k_face_update_lanes_out<EQ, N, R>, FL::bytes());
    if (e == cudaSuccess) e = allow(k_face_stage_lanes<EQ, N, R>, FL::bytes());
    if constexpr (!EQ::NC) {
      if (e == cudaSuccess) e = allow(k_face_update_lanes_clean<EQ, N, R>, FL::bytes());
    }
    if constexpr (kBatched) {
      if (e == cudaSuccess) e = allow(k_volume_batched<EQ, N, R, 0>, PL::bytes());
      if (e == cudaSuccess) e = allow(k_volume_batched<EQ, N, R, 1>, PL::bytes());
      if (e == cudaSuccess) e = allow(k_face_batched<EQ, N, R>, FL::bytes());
    }
    if constexpr (kFused) {
      if (e == cudaSuccess) e = allow(k_step_fused<EQ, N, R>, FU::bytes());
    }
    return e;
  }
  static cudaError_t vol_batched(const BatchLaunch& b, cudaStream_t s) {
    if constexpr (kBatched) {
      if (b.shape == 1)
        k_volume_batched<EQ, N, R, 1><<<b.grid, LL::THREADS, PL::bytes(), s>>>(
            b.solves, b.tiles, b.ntiles, PPB<R>::get(b), PPB<R>::tab(b), b.slot);
      else
        k_volume_batched<EQ, N, R, 0><<<b.grid, LL::THREADS, PL::bytes(), s>>>(
            b.solves, b.tiles, b.ntiles, PPB<R>::get(b), PPB<R>::tab(b), b.slot);
      return cudaGetLastError();
    }
    return cudaErrorNotSupported;
  }
  static cudaError_t face_batched(const BatchLaunch& b, cudaStream_t s) {
    if constexpr (kBatched) {
      k_face_batched<EQ, N, R><<<b.grid, FL::THREADS, FL::bytes(), s>>>(b.solves, b.tiles, b.ntiles, PPB<R>::get(b),
                                                                        PPB<R>::tab(b), b.slot);
      return cudaGetLastError();
    }
    return cudaErrorNotSupported;
  }
  static int occupancy(int which, int shape) {
    int nb = 0;
    if constexpr (kBatched) {
      if (which == 0) {
        auto k = shape == 1 ? k_volume_batched<EQ, N, R, 1> : k_volume_batched<EQ, N, R, 0>;
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PL::bytes());
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, LL::THREADS, PL::bytes());
      } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_face_batched<EQ, N, R>, FL::THREADS, FL::bytes());
      }
    }
    return nb;
  }
  static void fill(VariantOps* o) {
    o->vol_batched = kBatched ? &vol_batched : nullptr;
    o->face_batched = kBatched ? &face_batched : nullptr;
    o->occupancy = kBatched ? &occupancy : nullptr;
    o->vol_shapes = kBatched ? 2 : 0;
    o->threads_vol = LL::THREADS;
    o->threads_face = FL::THREADS;
    o->M = EQ::M;
    o->NP = LL::NP;
    o->NF = LL::NF;
    o->C = trace_comps<EQ>();
    o->ncs_per_elem = EQ::NCS ? ncs_values_per_elem<EQ, N>() : 0;
    o->dim = EQ::DIM;
    o->vol_form = &vol_form;
    o->lane_elems = LL::EPB;
    o->small_elems = LaneLayout<EQ, N, R, 2>::EPB;
    if constexpr (kPairs) o->pair_elems = PairLanes<EQ, N>::EPB;
    else o->pair_elems = 0;
    o->face_by_line = &face_by_line;
    o->real_bytes = sizeof(R);
    o->volume = &volume;
    o->face_update = &face_update;
    o->volume_stage = &volume_stage;
    o->face_stage = &face_stage;
    o->lambda = &lambda;
    o->step_fused = kFused ? &step_fused : nullptr;
    o->alpha = EQ::NC || kVolInd ? nullptr : &alpha;
    o->face_limited = EQ::NC ? nullptr : &face_limited;
    o->volume_ind = kVolInd ? &volume_ind : nullptr;
    o->alpha_smooth = kVolInd ? &alpha_smooth : nullptr;
    o->totals = &totals;
    o->set_smem = &set_smem;
  }
};

template <class EQ, typename R>
bool fill_ops(int N, VariantOps* o) {
  switch (N) {
    case 1: Variant<EQ, 1, R>::fill(o); return true;
    case 2: Variant<EQ, 2, R>::fill(o); return true;
    case 3: Variant<EQ, 3, R>::fill(o); return true;
    case 4: Variant<EQ, 4, R>::fill(o); return true;
    case 5: Variant<EQ, 5, R>::fill(o); return true;
  }
  return false;
}

}  // namespace crk
