// cr_noalloc.cu -- cr_step_noalloc: one cRKFR step that allocates no memory.
//
// Some callers cannot allocate device memory when they advance a solve: an
// application whose memory pool (for example a framework's caching allocator)
// has already reserved the device, or a host loop that must not stall other
// streams, which cudaMalloc/cudaFree can do by synchronising the device.  For
// them this entry point runs the same volume and face/update kernels as
// cr_step, with every scratch buffer (stage residual sums, face traces and
// the step record with its CFL reduction) carved out of one file-scope
// __device__ array of CR_NOALLOC_SCRATCH_BYTES.  The caller passes the input
// and output states; nothing is allocated or freed.
//
// The array exists once per device that loads the library and lives until the
// process exits.  All calls on a device share it and it keeps the last call's
// contents, so calls that overlap on the GPU (on different streams, or from
// several threads) race; the step record is clean at the start of every
// call (the face kernel zeroes the CFL slot its step has read, the first
// kernel drops a timeout; a call whose launches failed makes the next one clear
// it whole).  Its non-physical bit, which this entry point does not report, stays
// once it is set.  The array's device address is looked up on the first call on each
// device and kept for the life of the process; cudaDeviceReset destroys the
// context that address belongs to, so a process that resets a device must
// not call this entry point on that device afterwards.
#include <cuda_runtime.h>

#include <atomic>
#include <cstring>
#include <mutex>

#include "../../include/cr.h"
#include "cr_internal.h"

namespace crk {

static __device__ __align__(256) unsigned char g_noalloc_scratch[CR_NOALLOC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_mutex;
void* g_scratch_ptr[kMaxDevices] = {nullptr};
std::atomic<bool> g_dirty[kMaxDevices];   // the record may hold a failed call's values

// The variant's kernels get their shared memory allowance on the first call per
// device (a dozen runtime calls otherwise, of each call's host time).
using SetSmem = cudaError_t (*)();
constexpr int kMaxVariants = 128;   // variants per process: at most 110
SetSmem g_ready[kMaxDevices][kMaxVariants];
int g_nready[kMaxDevices];

cudaError_t prepare_variant(int dev, SetSmem f) {
  std::lock_guard<std::mutex> lock(g_mutex);
  for (int k = 0; k < g_nready[dev]; ++k)
    if (g_ready[dev][k] == f) return cudaSuccess;
  const cudaError_t e = f();
  if (e == cudaSuccess && g_nready[dev] < kMaxVariants) g_ready[dev][g_nready[dev]++] = f;
  return e;
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Device address of the scratch array on the current device; looked up once
// per device (the host-side symbol is only a stand-in, never a device address).
cudaError_t scratch_address(int dev, void** out) {
  std::lock_guard<std::mutex> lock(g_mutex);
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

int to_status(cudaError_t e) {
  if (e == cudaSuccess) return CR_OK;
  if (e == cudaErrorNoKernelImageForDevice || e == cudaErrorInvalidDevice || e == cudaErrorNoDevice)
    return CR_ENODEV;
  return CR_ECUDA;
}

bool desc_ok(const cr_mesh_desc& d) {
  if (d.eq != CR_EULER && d.eq != CR_GLM_MHD) return false;
  if (d.dim < 1 || d.dim > 3 || d.degree_N < 1 || d.degree_N > 5) return false;
  if (d.eq == CR_GLM_MHD && (d.dim != 2 || d.vol == CR_VOL_KEP)) return false;
  if (d.vol < 0 || d.vol > 2 || d.surf != CR_SURF_RUSANOV) return false;
  if (d.prec != CR_FP64 && d.prec != CR_FP32_PAIRFLUX) return false;
  if (d.scheme != CR_SCHEME_CRKFR || d.ncflux != CR_NCFLUX_REDUCED || d.limiter != CR_LIMITER_NONE) return false;
  if (!(d.gamma > 1.0) || !(d.cfl > 0.0) || !(d.dt_fixed >= 0.0) || !(d.c_h >= 0.0)) return false;   // NaN fails
  for (int k = 0; k < d.dim; ++k)
    if (d.cells[k] < 1 || !(d.hi[k] > d.lo[k])) return false;
  return true;
}

}  // namespace
}  // namespace crk

using namespace crk;

extern "C" int cr_step_noalloc(const cr_mesh_desc* desc, const double* u_in, double* u_out, double* dt_out,
                               void* cuda_stream) {
  if (!desc || !u_in || !u_out || !desc_ok(*desc)) return CR_EINVAL;
  const cr_mesh_desc& d = *desc;
  VariantOps o;
  if (!get_ops(d.eq, d.dim, d.prec, d.vol, d.degree_N, &o)) return CR_EINVAL;
  long long E = 1;
  for (int k = 0; k < d.dim; ++k) E *= d.cells[k];
  const long long nodes = E * o.NP;
  // scratch layout: step record | rbar | face traces
  const size_t off_rbar = align256(sizeof(DevState));
  const size_t off_trace = off_rbar + align256(o.real_bytes * (size_t)o.M * nodes);
  const size_t need = off_trace + align256(o.real_bytes * (size_t)o.dim * 2 * o.C * (E * o.NF));
  if (need > (size_t)CR_NOALLOC_SCRATCH_BYTES) return CR_ETOOLARGE;

  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return to_status(e);
  unsigned char* base = nullptr;
  e = scratch_address(dev, (void**)&base);
  if (e != cudaSuccess) return to_status(e);
  cudaStream_t s = (cudaStream_t)cuda_stream;

  LaunchCtx lc;
  fill_launch_ctx(d, &lc);
  // u^n is read where it is; u^{n+1} goes to u_out (in place if they are one)
  lc.u = const_cast<double*>(u_in);
  lc.st = (DevState*)base;
  lc.rbar = base + off_rbar;
  lc.trace = base + off_trace;
  lc.out = FaceOut{u_out == u_in ? nullptr : u_out, dt_out, 1};
  lc.ma.tma_ok = tma_ok_for(u_in, E, o.NP);

  // Three launches: the CFL reduction of u^n (slot 0), volume, face / update (with
  // dt and the clean-up); a copy of the state, a clear of the record and a copy of
  // dt besides were half of a small step.  64^2, N = 3, FP32: 62 -> 37 us a call.
  if ((e = prepare_variant(dev, o.set_smem)) != cudaSuccess) return to_status(e);
  if (g_dirty[dev].exchange(true) && (e = cudaMemsetAsync(lc.st, 0, sizeof(DevState), s)) != cudaSuccess)
    return to_status(e);
  lc.slot = 0;
  if ((e = o.lambda(lc, s)) != cudaSuccess) return to_status(e);
  if ((e = o.volume(lc, s)) != cudaSuccess) return to_status(e);
  if ((e = o.face_update(lc, s)) != cudaSuccess) return to_status(e);
  g_dirty[dev] = false;
  return CR_OK;
}
