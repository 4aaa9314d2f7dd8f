// C ABI of the demag convolution + exchange/LLG/RK4 library (declarations and contracts in
// include/gbdemag.h). Host side: argument checks, planning, device buffers, the kernel
// spectrum upload and the launch sequences of Eq. 1 (Sec. II) and of the RK4 time step.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "gbdemag.h"
#include "gbd_fft.cuh"
#include "gbd_kernels.cuh"
#include "gbd_plan.h"

static thread_local std::string g_err;

static gbd_status fail(gbd_status s, const std::string& msg) {
  g_err = msg;
  return s;
}

static gbd_status cuda_fail(cudaError_t e, const char* where) {
  return fail(GBD_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

struct gbd_mesh {
  gbd_mesh_desc d;
  gbd::Plan p;
  int device = -1;
  float2* S = nullptr;      // x spectrum [3][nz][Hx][ny]
  float2* T = nullptr;      // 3D y spectrum [3][nz][Hx][Py] (ny > 1 and nz > 1)
  void* K = nullptr;        // packed kernel spectrum
  float* acc = nullptr;     // RK4 state: k-sum and two stage buffers, each [3][N]
  float* bufA = nullptr;
  float* bufB = nullptr;
  float2* tw = nullptr;     // twiddle levels, 2 GBD_TW_LEN entries
  unsigned* status = nullptr;   // device status word (GBD_DEV_*), the 16 bytes after the twiddles
  unsigned stage_extra = 0;     // test hook GBD_TEST_WAIT_TIMEOUT (RowArgs::stage_extra)
  // demag history for extrapolation at RK4 sub-steps: 5 slots of [3][N], allocated on the
  // first gbd_llg_step_ex with GBD_STEP_EXTRAP; hist_head = newest slot
  float* hist = nullptr;
  int hist_count = 0, hist_head = 0;
  double hist_dt = 0.0;
  unsigned version = 0;     // bumped when launch arguments change (params, tuning): batch graphs re-capture
  // RKF5(6) stepping (allocated on first use): 8 stage slopes [3][N] each, the step's result
  // and the error word
  float* rk_k = nullptr;
  float* rk_m = nullptr;
  unsigned* rk_err = nullptr;
  // device-controlled run (gbd_llg_run_rkf56 without extrapolation): the control block and the
  // instantiated loop graph, built for the array rkf_key_m at parameter version rkf_key_version
  gbd::RkfCtl* rk_ctl = nullptr;
  cudaGraphExec_t rkf_exec = nullptr;
  const float* rkf_key_m = nullptr;
  unsigned rkf_key_version = 0;
  // demag history of RKF5(6) with extrapolation: 6 slots of [3][N]; rk_ring holds the slots of
  // the accepted step starts, newest first (rk_count valid), rk_ring_t their times relative to
  // the current time; rk_pend receives the field of the step being tried
  float* rk_hist = nullptr;
  int rk_ring[5] = {0, 1, 2, 3, 4};
  double rk_ring_t[5] = {0, 0, 0, 0, 0};
  int rk_count = 0, rk_pend = 5;
  bool kernel_set = false;
  // optional per-launch timing: events[2i], events[2i+1] bracket launch i of class cls[i]
  int timing = 0;           // GBD_TIMING_EVENTS | GBD_TIMING_NVTX
  std::vector<cudaEvent_t> events;
  std::vector<int> cls;
  size_t used = 0;
  // the last work each stream was given for this mesh (recorded after every call that enqueues
  // work outside a stream capture, and after batch graph launches); gbd_mesh_destroy orders the
  // frees after these
  std::vector<std::pair<cudaStream_t, cudaEvent_t>> done;
};

// Runs f() (which enqueues one kernel on st); with GBD_TIMING_EVENTS it brackets the launch with
// CUDA events, with GBD_TIMING_NVTX with an NVTX range named after the pass class.
static const char* const kPassName[GBD_NPASS] = {"row_fwd", "row_inv", "row_rk", "film_conv",
                                                 "y_fwd", "z_conv", "y_inv", "extrap_stage"};
template <class F>
static void timed_events(gbd_mesh* m, int pass, cudaStream_t st, F f) {
  if (m->used + 2 > m->events.size()) {
    size_t grow = m->events.size() < 256 ? 256 : m->events.size();
    for (size_t i = 0; i < grow; ++i) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) {
        f();
        return;
      }
      m->events.push_back(e);
    }
  }
  cudaEventRecord(m->events[m->used], st);
  f();
  cudaEventRecord(m->events[m->used + 1], st);
  m->cls.push_back(pass);
  m->used += 2;
}
template <class F>
static void timed(gbd_mesh* m, int pass, cudaStream_t st, F f) {
  if (!m->timing) {
    f();
    return;
  }
  if (m->timing & GBD_TIMING_NVTX) nvtxRangePushA(kPassName[pass]);
  if (m->timing & GBD_TIMING_EVENTS)
    timed_events(m, pass, st, f);
  else
    f();
  if (m->timing & GBD_TIMING_NVTX) nvtxRangePop();
}

namespace gbd {

static int pow2_at_least(long long v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

// The smallest mixed length L (kMixedLens) with L >= v, or 0.
static int mixed_at_least(long long v) {
  for (int L : kMixedLens)
    if (L >= v) return L;
  return 0;
}

bool make_plan(int nx, int ny, int nz, int per, bool mixed, Plan& p, const char** why) {
  if (nx < 1 || ny < 1 || nz < 1) {
    *why = "mesh sizes must be >= 1";
    return false;
  }
  const int n[3] = {nx, ny, nz};
  for (int d = 0; d < 3; ++d)
    if ((per >> d & 1) && (n[d] & (n[d] - 1)) != 0) {
      *why = "a periodic axis needs a power-of-two number of cells";
      return false;
    }
  if ((per & 1) && nx < 2) {
    *why = "a periodic x axis needs nx >= 2";
    return false;
  }
  if (((per & 2) && ny == 2) || ((per & 4) && nz == 2)) {
    *why = "a periodic y or z axis needs 1 or at least 4 cells";
    return false;
  }
  p.nx = nx;
  p.ny = ny;
  p.nz = nz;
  p.N = (long long)nx * ny * nz;
  p.per = per;
  // periodic: the period itself (circular convolution); otherwise zero padded
  p.Px = (per & 1) ? nx : (nx == 1 ? 2 : pow2_at_least(2LL * nx - 1));
  p.Py = (per & 2) ? ny : (ny == 1 ? 1 : pow2_at_least(2LL * ny - 1));
  if (mixed && !(per & 1) && nx > 1) {
    const int lx = mixed_at_least(nx);   // 2 Lx >= 2 nx - 1
    if (lx && 2 * lx < p.Px) p.Px = 2 * lx;
  }
  if (mixed && !(per & 2) && ny > 1) {
    const int ly = mixed_at_least(2LL * ny - 1);
    if (ly && ly < p.Py) p.Py = ly;
  }
  p.Pz = (per & 4) ? nz : (nz == 1 ? 1 : pow2_at_least(2LL * nz - 1));
  p.ox = (per & 1) ? nx / 2 + 1 : nx;
  p.oy = (per & 2) ? ny / 2 + 1 : ny;
  p.oz = (per & 4) ? nz / 2 + 1 : nz;
  if (p.Px > kMaxPadX || p.Py > kMaxPad || p.Pz > kMaxPad) {
    *why = "mesh too large: supported nx <= 4096, ny <= 2048, nz <= 2048";
    return false;
  }
  p.Lx = p.Px / 2;
  p.Hx = p.Lx + 1;
  p.Ky = p.Py / 2 + 1;
  p.Kz = p.Pz / 2 + 1;
  p.film = (nz == 1);
  // block shapes (the kernels are compiled for these per transform length)
  p.RB = row_rb(p.Lx, p.var_row);
  p.Cf = film_cols(p.Py, p.var_film);
  p.Cy = ypass_lines(p.Py, p.var_y);
  p.Wz = zconv_cols(p.Pz, p.var_z);
  p.bytes_S = (size_t)3 * nz * p.Hx * ny * sizeof(float2);
  p.bytes_T = (!p.film && ny > 1) ? (size_t)3 * nz * p.Hx * p.Py * sizeof(float2) : 0;
  p.bytes_K = p.film ? (size_t)p.Hx * p.Ky * sizeof(float4) : (size_t)p.Hx * p.Ky * p.Kz * 6 * sizeof(float);
  p.bytes_state = (size_t)3 * 3 * p.N * sizeof(float);
  p.bytes_tw = (size_t)(GBD_TW_TOTAL + 2) * sizeof(float2);   // + the 16-byte device status word
  return true;
}

}  // namespace gbd

constexpr int kMaxImages = 10000;

static gbd_status check_desc(const gbd_mesh_desc* d, gbd::Plan& p) {
  if (!d) return fail(GBD_EINVAL, "desc is NULL");
  const char* why = nullptr;
  if (d->nx < 1 || d->ny < 1 || d->nz < 1) return fail(GBD_EINVAL, "mesh sizes must be >= 1");
  if (!(d->dx > 0 && d->dy > 0 && d->dz > 0) || !std::isfinite(d->dx * d->dy * d->dz))
    return fail(GBD_EINVAL, "cell sizes must be finite and > 0");
  if (!(d->Ms > 0) || !std::isfinite(d->Ms)) return fail(GBD_EINVAL, "Ms must be finite and > 0");
  if (!(d->A_ex >= 0) || !std::isfinite(d->A_ex)) return fail(GBD_EINVAL, "A_ex must be finite and >= 0");
  if (!(d->alpha >= 0) || !std::isfinite(d->alpha)) return fail(GBD_EINVAL, "alpha must be finite and >= 0");
  if (!(d->gamma >= 0) || !std::isfinite(d->gamma)) return fail(GBD_EINVAL, "gamma must be finite and >= 0");
  for (int i = 0; i < 3; ++i)
    if (!std::isfinite(d->Hext[i])) return fail(GBD_EINVAL, "Hext must be finite");
  if (d->precision != GBD_FP32 && d->precision != GBD_SPLIT_BF16 && d->precision != GBD_SPLIT_FP16)
    return fail(GBD_EINVAL, "precision must be GBD_FP32, GBD_SPLIT_BF16 or GBD_SPLIT_FP16");
  if (d->flags & ~(unsigned)(GBD_FLAG_PBC_X | GBD_FLAG_PBC_Y | GBD_FLAG_PBC_Z | GBD_FLAG_POW2_PAD))
    return fail(GBD_EINVAL, "unknown flags");
  const int per = (int)(d->flags & 7u);
  if (per && (d->pbc_images < 1 || d->pbc_images > kMaxImages))
    return fail(GBD_EINVAL, "pbc_images must be in [1, " + std::to_string(kMaxImages) + "] with a periodic axis");
  // lengths 3 * 2^k and 5 * 2^k have FP32 kernels only
  const bool mixed = d->precision == GBD_FP32 && !(d->flags & GBD_FLAG_POW2_PAD);
  if (!gbd::make_plan(d->nx, d->ny, d->nz, per, mixed, p, &why)) return fail(GBD_EUNSUPPORTED, why);
  p.images = per ? d->pbc_images : 0;
  p.prec = (d->precision == GBD_SPLIT_BF16) ? 1 : (d->precision == GBD_SPLIT_FP16) ? 2 : 0;
  return GBD_OK;
}

static bool ptr_ok(const void* p) { return p && (reinterpret_cast<uintptr_t>(p) % 4 == 0); }

static gbd_status check_device(const gbd_mesh* m) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev != m->device) return fail(GBD_ECUDA, "current device differs from the mesh's device");
  e = cudaPeekAtLastError();
  if (e != cudaSuccess) return cuda_fail(e, "pending CUDA error");
  return GBD_OK;
}

// Device memory of meshes comes from the device's stream-ordered pool (cudaMallocAsync /
// cudaFreeAsync) on a library stream per device, so that creating or destroying a mesh never
// waits for the whole device (cudaMalloc / cudaFree do): an allocation is made on the library
// stream and that stream is synchronized before the memory is handed out; a free is ordered
// after the mesh's own recorded work and returns at once.
static cudaStream_t lib_stream(int dev) {
  static std::mutex mu;
  static cudaStream_t streams[64] = {nullptr};
  if (dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!streams[dev] && cudaStreamCreateWithFlags(&streams[dev], cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    streams[dev] = nullptr;
  }
  return streams[dev];
}

// Allocates `bytes` for a mesh on device dev and waits until the memory is usable by any stream.
static cudaError_t mesh_alloc(int dev, void** ptr, size_t bytes) {
  cudaStream_t ls = lib_stream(dev);
  cudaError_t e = cudaMallocAsync(ptr, bytes, ls);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ls);
  return e;
}

static void free_mesh_buffers(gbd_mesh* m) {
  cudaStream_t ls = lib_stream(m->device);
  for (auto& d : m->done) {
    cudaStreamWaitEvent(ls, d.second, 0);
    cudaEventDestroy(d.second);
  }
  m->done.clear();
  if (m->rkf_exec) cudaGraphExecDestroy(m->rkf_exec);   // never running here: its call waited for it
  m->rkf_exec = nullptr;
  void* bufs[] = {m->S, m->T, m->K, m->acc, m->bufA, m->bufB, m->tw, m->hist, m->rk_k, m->rk_m, m->rk_err, m->rk_hist,
                  m->rk_ctl};
  for (void* b : bufs)
    if (b) cudaFreeAsync(b, ls);
  m->hist = nullptr;
  m->rk_hist = nullptr;
  m->rk_k = m->rk_m = nullptr;
  m->rk_err = nullptr;
  m->rk_ctl = nullptr;
  m->S = m->T = nullptr;
  m->K = nullptr;
  m->acc = m->bufA = m->bufB = nullptr;
  m->tw = nullptr;
  m->status = nullptr;
}

// Records the end of the work just enqueued for m on st (not inside a stream capture: captured
// work is run by the caller's graph, which the caller finishes before destroying the mesh).
static void mark_done(gbd_mesh* m, cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return;
  }
  for (auto& d : m->done)
    if (d.first == st) {
      cudaEventRecord(d.second, st);
      return;
    }
  cudaEvent_t ev;
  if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  cudaEventRecord(ev, st);
  m->done.emplace_back(st, ev);
}

// Twiddle levels: exp(-2 pi i m / N) at index tw_base(N) + m for m < N and N = 1, 2, 4, ...,
// GBD_TW_LEN, N = 3, 6, ..., GBD_TW3_MAX and N = 5, 10, ..., GBD_TW5_MAX, FP64 on the host, rounded
// to FP32 (the split DFT-16 fragment tables between them are written on the device). The same for
// every mesh: computed once per process (80,000 sines and cosines, most of a mesh's creation time).
static const std::vector<float2>& twiddle_levels() {
  static const std::vector<float2> table = [] {
    std::vector<float2> tw(GBD_TW_TOTAL, make_float2(1.f, 0.f));
    auto level = [&](int N) {
      for (int k = 0; k < N; ++k) {
        const double ang = -2.0 * 3.14159265358979323846264338327950288 * (double)k / N;
        tw[gbd::tw_base(N) + k] = make_float2((float)std::cos(ang), (float)std::sin(ang));
      }
    };
    for (int N = 1; N <= GBD_TW_LEN; N *= 2) level(N);
    for (int N = 3; N <= GBD_TW3_MAX; N *= 2) level(N);
    for (int N = 5; N <= GBD_TW5_MAX; N *= 2) level(N);
    return tw;
  }();
  return table;
}

// ---- launch sequences ------------------------------------------------------------------------

// Tile variant of an x-row launch: the transform-only launches (forward, or inverse to H_d) and
// the launches with an epilogue are tuned separately.
static int row_var(const gbd_mesh* m, int mode) {
  return (mode == gbd::ROW_FWD || mode == gbd::ROW_H) ? m->p.var_row_io : m->p.var_row;
}

static gbd::RowArgs row_args(const gbd_mesh* m) {
  const gbd::Plan& p = m->p;
  const gbd_mesh_desc& d = m->d;
  gbd::RowArgs a;
  std::memset(&a, 0, sizeof(a));
  a.nx = p.nx;
  a.ny = p.ny;
  a.nz = p.nz;
  a.rows = p.ny * p.nz;
  a.N = p.N;
  a.S = m->S;
  a.status = m->status;
  a.stage_extra = m->stage_extra;
  const double mu0 = 4.0e-7 * 3.14159265358979323846;
  const double lex = 2.0 * d.A_ex / (mu0 * d.Ms);
  a.cx = p.nx > 1 ? (float)(lex / (d.dx * d.dx)) : 0.f;
  a.cy = p.ny > 1 ? (float)(lex / (d.dy * d.dy)) : 0.f;
  a.cz = p.nz > 1 ? (float)(lex / (d.dz * d.dz)) : 0.f;
  a.hx = (float)d.Hext[0];
  a.hy = (float)d.Hext[1];
  a.hz = (float)d.Hext[2];
  const double gam = d.gamma > 0 ? d.gamma : 2.212761569e5;
  a.geff = (float)(gam / (1.0 + d.alpha * d.alpha));
  a.alpha = (float)d.alpha;
  a.hscale = (float)d.Ms;
  a.per = p.per;
  return a;
}

static gbd::ColArgs col_args(const gbd_mesh* m) {
  const gbd::Plan& p = m->p;
  gbd::ColArgs a;
  std::memset(&a, 0, sizeof(a));
  a.Hx = p.Hx;
  a.ny = p.ny;
  a.nz = p.nz;
  a.Py = p.Py;
  a.Pz = p.Pz;
  return a;
}

// The whole convolution along y and z in one launch (gbd_small.cu).
static bool conv_in_one(const gbd::Plan& p) {
  const bool fp32 = p.film ? gbd::stage_prec(p.prec, p.Py, true) == 0
                           : gbd::stage_prec(p.prec, p.Py, false) == 0 && gbd::stage_prec(p.prec, p.Pz, true) == 0;
  return fp32 && gbd::small_conv_ok(p.Hx, p.Py, p.Pz, p.nz, p.per);
}

// Strides of the z convolution on T [3][nz][Hx][Py], or, when ny = 1, on S [3][nz][Hx].
static void z_strides(const gbd::Plan& p, gbd::ColArgs& a) {
  a.Pyq = p.ny > 1 ? p.Py : 1;
  a.Q = (long long)p.Hx * a.Pyq;
}

// Middle of Eq. 1: everything between the forward and the inverse x transforms, on the spectra S
// and T. A 3D convolution that runs in one launch is split into its passes, the same arithmetic,
// while events time the launches by pass.
static void enqueue_conv(gbd_mesh* m, float2* S, float2* T, cudaStream_t st) {
  const gbd::Plan& p = m->p;
  gbd::ColArgs a = col_args(m);
  const bool one = conv_in_one(p);
  if (p.film) {
    a.dst = S;
    a.Kf = static_cast<const float4*>(m->K);
    timed(m, GBD_PASS_FILM_CONV, st, [&] {
      if (one)
        gbd::launch_small_conv(a, S, nullptr, 7, m->tw, st);
      else
        gbd::launch_film_conv(p.var_film, p.prec, a, m->tw, st);
    });
    return;
  }
  a.K3 = static_cast<const float2*>(m->K);
  if (one) {
    if (m->timing & GBD_TIMING_EVENTS) {
      timed(m, GBD_PASS_Y_FWD, st, [&] { gbd::launch_small_conv(a, S, T, 1, m->tw, st); });
      timed(m, GBD_PASS_Z_CONV, st, [&] { gbd::launch_small_conv(a, S, T, 2, m->tw, st); });
      timed(m, GBD_PASS_Y_INV, st, [&] { gbd::launch_small_conv(a, S, T, 4, m->tw, st); });
    } else {
      timed(m, GBD_PASS_Z_CONV, st, [&] { gbd::launch_small_conv(a, S, T, 7, m->tw, st); });
    }
    return;
  }
  if (p.ny > 1) {
    a.lines_total = 3LL * p.nz * p.Hx;
    a.src = S;
    a.dst = T;
    timed(m, GBD_PASS_Y_FWD, st, [&] { gbd::launch_y_fwd(p.var_y, p.prec, a, m->tw, st); });
    a.dst = T;
    z_strides(p, a);
    timed(m, GBD_PASS_Z_CONV, st, [&] { gbd::launch_z_conv(p.var_z, p.prec, a, m->tw, st); });
    a.src = T;
    a.dst = S;
    timed(m, GBD_PASS_Y_INV, st, [&] { gbd::launch_y_inv(p.var_y, p.prec, a, m->tw, st); });
  } else {
    a.dst = S;
    z_strides(p, a);
    timed(m, GBD_PASS_Z_CONV, st, [&] { gbd::launch_z_conv(p.var_z, p.prec, a, m->tw, st); });
  }
}

static gbd_status after_launch(const char* where) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, where);
  return GBD_OK;
}

// ---- C ABI -----------------------------------------------------------------------------------

extern "C" {

const char* gbd_last_error(void) { return g_err.c_str(); }

gbd_status gbd_plan_dims(const gbd_mesh_desc* desc, int out[6]) {
  gbd::Plan p;
  gbd_status s = check_desc(desc, p);
  if (s != GBD_OK) return s;
  if (!out) return fail(GBD_EINVAL, "out is NULL");
  out[0] = p.Px;
  out[1] = p.Py;
  out[2] = p.Pz;
  out[3] = p.Hx;
  out[4] = p.Ky;
  out[5] = p.Kz;
  return GBD_OK;
}

gbd_status gbd_mesh_bytes(const gbd_mesh_desc* desc, size_t* out) {
  gbd::Plan p;
  gbd_status s = check_desc(desc, p);
  if (s != GBD_OK) return s;
  if (!out) return fail(GBD_EINVAL, "out is NULL");
  *out = p.total_bytes();
  return GBD_OK;
}

gbd_status gbd_tensor_at(const gbd_mesh_desc* desc, int X, int Y, int Z, double out[6]) {
  if (!desc || !out) return fail(GBD_EINVAL, "NULL argument");
  if (!(desc->dx > 0 && desc->dy > 0 && desc->dz > 0)) return fail(GBD_EINVAL, "cell sizes must be > 0");
  gbdt::tensor_at(X, Y, Z, desc->dx, desc->dy, desc->dz, out);
  return GBD_OK;
}

gbd_status gbd_kernel_spectrum_host(const gbd_mesh_desc* desc, double* out, size_t count) {
  gbd::Plan p;
  gbd_status s = check_desc(desc, p);
  if (s != GBD_OK) return s;
  const size_t need = (size_t)6 * p.Kz * p.Ky * p.Hx;
  if (!out || count != need) return fail(GBD_EINVAL, "out is NULL or count != 6*Kz*Ky*Hx");
  std::vector<double> spec;
  if (!gbdt::kernel_spectrum(p, desc->dx, desc->dy, desc->dz, spec)) return fail(GBD_ENOMEM, "host allocation failed");
  std::memcpy(out, spec.data(), need * sizeof(double));
  return GBD_OK;
}

static gbd_status spectrum_of_tensor(const gbd::Plan& p, const double* N6, std::vector<double>& spec);

gbd_status gbd_kernel_spectrum_from_tensor_host(const gbd_mesh_desc* desc, const double* N6, double* out,
                                                size_t count) {
  gbd::Plan p;
  gbd_status s = check_desc(desc, p);
  if (s != GBD_OK) return s;
  const size_t need = (size_t)6 * p.Kz * p.Ky * p.Hx;
  if (!out || count != need) return fail(GBD_EINVAL, "out is NULL or count != 6*Kz*Ky*Hx");
  std::vector<double> spec;
  s = spectrum_of_tensor(p, N6, spec);
  if (s != GBD_OK) return s;
  std::memcpy(out, spec.data(), need * sizeof(double));
  return GBD_OK;
}

gbd_status gbd_mesh_create(const gbd_mesh_desc* desc, gbd_mesh** out) {
  if (!out) return fail(GBD_EINVAL, "out is NULL");
  *out = nullptr;
  gbd::Plan p;
  gbd_status s = check_desc(desc, p);
  if (s != GBD_OK) return s;
  gbd_mesh* m = new (std::nothrow) gbd_mesh();
  if (!m) return fail(GBD_ENOMEM, "host allocation failed");
  m->d = *desc;
  m->p = p;
  cudaError_t e = cudaGetDevice(&m->device);
  if (e != cudaSuccess) {
    delete m;
    return cuda_fail(e, "cudaGetDevice");
  }
  struct {
    void** ptr;
    size_t bytes;
  } allocs[] = {{(void**)&m->S, p.bytes_S},      {(void**)&m->T, p.bytes_T},
                {(void**)&m->K, p.bytes_K},      {(void**)&m->acc, p.bytes_state / 3},
                {(void**)&m->bufA, p.bytes_state / 3}, {(void**)&m->bufB, p.bytes_state / 3},
                {(void**)&m->tw, p.bytes_tw}};
  // test hook: GBD_TEST_FAIL_ALLOC=k makes the k-th device allocation below report
  // out-of-memory without calling cudaMalloc (exercises the clean-up path)
  const char* fail_env = std::getenv("GBD_TEST_FAIL_ALLOC");
  const int fail_at = fail_env ? std::atoi(fail_env) : 0;
  int nalloc = 0;
  for (auto& al : allocs) {
    if (al.bytes == 0) continue;
    e = (++nalloc == fail_at) ? cudaErrorMemoryAllocation : mesh_alloc(m->device, al.ptr, al.bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      free_mesh_buffers(m);
      cudaStreamSynchronize(lib_stream(m->device));   // the pool gives the memory back at this point
      delete m;
      return fail(e == cudaErrorMemoryAllocation ? GBD_ENOMEM : GBD_ECUDA,
                  std::string("cudaMallocAsync: ") + cudaGetErrorString(e));
    }
  }
  const std::vector<float2>& tw = twiddle_levels();
  cudaStream_t ls = lib_stream(m->device);
  m->status = reinterpret_cast<unsigned*>(m->tw + GBD_TW_TOTAL);
  // test hook: GBD_TEST_WAIT_TIMEOUT=1 makes this mesh's staged RK-stage copies expect 16 bytes
  // more than they deliver, so the kernels' bounded waits run out (exercises the timeout path)
  const char* wait_env = std::getenv("GBD_TEST_WAIT_TIMEOUT");
  m->stage_extra = (wait_env && std::atoi(wait_env) != 0) ? 16u : 0u;
  e = cudaMemsetAsync(m->status, 0, 16, ls);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice, ls);
  if (e == cudaSuccess) {
    gbd::launch_dft16_frags(m->tw + 2 * GBD_TW_LEN, ls);
    e = cudaStreamSynchronize(ls);
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    free_mesh_buffers(m);
    delete m;
    return cuda_fail(e, "cudaMemcpy twiddles");
  }
  // shared-memory attributes of this mesh's kernels (both tile variants), set now so that
  // later launches, also inside a stream capture, need no configuration call
  gbd::prepare_small();
  bool have = gbd::prepare_row(p.Lx, p.prec);
  if (p.film) {
    have = have && gbd::prepare_film_conv(p.Py, p.prec);
  } else {
    have = have && gbd::prepare_z_conv(p.Pz, p.prec);
    if (p.ny > 1) have = have && gbd::prepare_y_passes(p.Py, p.prec);
  }
  if (!have) {
    free_mesh_buffers(m);
    delete m;
    return fail(GBD_EUNSUPPORTED, "no kernel instantiated for these transform lengths");
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    free_mesh_buffers(m);
    delete m;
    return cuda_fail(e, "kernel attributes");
  }
  *out = m;
  return GBD_OK;
}

gbd_status gbd_mesh_set_timing(gbd_mesh* m, int enable) {
  if (!m) return fail(GBD_EINVAL, "mesh is NULL");
  m->timing = enable & (GBD_TIMING_EVENTS | GBD_TIMING_NVTX);
  if (enable != 0 && m->timing == 0) m->timing = GBD_TIMING_EVENTS;
  return GBD_OK;
}

gbd_status gbd_mesh_read_timing(gbd_mesh* m, double* ms, long long* launches) {
  if (!m || !ms || !launches) return fail(GBD_EINVAL, "NULL argument");
  for (int i = 0; i < GBD_NPASS; ++i) {
    ms[i] = 0.0;
    launches[i] = 0;
  }
  for (size_t i = 0; i < m->cls.size(); ++i) {
    cudaError_t e = cudaEventSynchronize(m->events[2 * i + 1]);
    float t = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, m->events[2 * i], m->events[2 * i + 1]);
    if (e != cudaSuccess) return cuda_fail(e, "gbd_mesh_read_timing");
    ms[m->cls[i]] += t;
    launches[m->cls[i]] += 1;
  }
  m->cls.clear();
  m->used = 0;
  return GBD_OK;
}

gbd_status gbd_mesh_set_params(gbd_mesh* m, const double Hext[3], double alpha) {
  if (!m) return fail(GBD_EINVAL, "mesh is NULL");
  if (Hext && !(std::isfinite(Hext[0]) && std::isfinite(Hext[1]) && std::isfinite(Hext[2])))
    return fail(GBD_EINVAL, "Hext must be finite");
  if (!std::isfinite(alpha)) return fail(GBD_EINVAL, "alpha must be finite (negative keeps the damping)");
  if (Hext)
    for (int c = 0; c < 3; ++c) m->d.Hext[c] = Hext[c];
  if (alpha >= 0) m->d.alpha = alpha;
  ++m->version;
  return GBD_OK;
}

gbd_status gbd_mesh_device_status(gbd_mesh* m, void* stream) {
  if (!m) return fail(GBD_EINVAL, "mesh is NULL");
  gbd_status s = check_device(m);
  if (s != GBD_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  unsigned h = 0;
  cudaError_t e = cudaMemcpyAsync(&h, m->status, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->status, 0, sizeof(h), st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "device status");
  if (h & GBD_DEV_WAIT_TIMEOUT) return fail(GBD_ETIMEOUT, "a kernel's wait for its staged copies gave up");
  return GBD_OK;
}

gbd_status gbd_mesh_destroy(gbd_mesh* m) {
  if (!m) return GBD_OK;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != m->device) cudaSetDevice(m->device);
  for (cudaEvent_t e : m->events) cudaEventDestroy(e);
  free_mesh_buffers(m);   // ordered after the mesh's recorded work; the host does not wait
  if (prev != m->device && prev >= 0) cudaSetDevice(prev);
  delete m;
  return GBD_OK;
}

// Host cache of packed FP32 kernel spectra keyed by geometry (mesh size and cell), so meshes
// of a geometry seen before skip the FP64 tensor and its transform. Least recently used
// entries are dropped beyond GBD_KERNEL_CACHE_BYTES (environment, default 4 GiB).
namespace {
struct GeoKey {
  int nx, ny, nz;
  double dx, dy, dz;
  int per, images;   // periodic axes and images per side
  int Px, Py, Pz;    // padded lengths (the spectrum is sampled on them)
  bool operator<(const GeoKey& o) const {
    if (Px != o.Px) return Px < o.Px;
    if (Py != o.Py) return Py < o.Py;
    if (Pz != o.Pz) return Pz < o.Pz;
    if (nx != o.nx) return nx < o.nx;
    if (ny != o.ny) return ny < o.ny;
    if (nz != o.nz) return nz < o.nz;
    if (dx != o.dx) return dx < o.dx;
    if (dy != o.dy) return dy < o.dy;
    if (dz != o.dz) return dz < o.dz;
    if (per != o.per) return per < o.per;
    return images < o.images;
  }
};
struct SpecEntry {
  std::shared_ptr<const std::vector<float>> data;
  unsigned long long last_use = 0;
};
std::mutex g_spec_mu;
std::map<GeoKey, SpecEntry> g_spec;
unsigned long long g_spec_clock = 0;

size_t spec_cache_limit() {
  const char* v = std::getenv("GBD_KERNEL_CACHE_BYTES");
  if (v && *v) return (size_t)std::strtoull(v, nullptr, 10);
  return (size_t)4 << 30;
}

std::shared_ptr<const std::vector<float>> spec_cache_get(const GeoKey& k) {
  std::lock_guard<std::mutex> lock(g_spec_mu);
  auto it = g_spec.find(k);
  if (it == g_spec.end()) return nullptr;
  it->second.last_use = ++g_spec_clock;
  return it->second.data;
}

void spec_cache_put(const GeoKey& k, std::shared_ptr<const std::vector<float>> d) {
  std::lock_guard<std::mutex> lock(g_spec_mu);
  g_spec[k] = SpecEntry{d, ++g_spec_clock};
  const size_t limit = spec_cache_limit();
  for (;;) {
    size_t total = 0;
    auto oldest = g_spec.end();
    for (auto it = g_spec.begin(); it != g_spec.end(); ++it) {
      total += it->second.data->size() * sizeof(float);
      if (oldest == g_spec.end() || it->second.last_use < oldest->second.last_use) oldest = it;
    }
    if (total <= limit || g_spec.size() <= 1) break;
    g_spec.erase(oldest);
  }
}
}  // namespace

// Packs the FP64 spectrum [6][Kz][Ky][Hx] into the device layout, uploads it on st and waits;
// a geometry key puts the packed copy into the host cache.
static gbd_status upload_spectrum(gbd_mesh* m, const std::vector<double>& spec, cudaStream_t st, const GeoKey* key) {
  const gbd::Plan& p = m->p;
  const size_t plane = (size_t)p.Ky * p.Hx;
  const size_t comp = (size_t)p.Kz * plane;
  auto packed_ptr = std::make_shared<std::vector<float>>();
  std::vector<float>& packed = *packed_ptr;
  try {
    packed.resize(p.bytes_K / sizeof(float));
  } catch (...) {
    return fail(GBD_ENOMEM, "host allocation failed");
  }
  if (p.film) {
    // [kx][ky] x (xx, yy, zz, xy)
    for (int kx = 0; kx < p.Hx; ++kx)
      for (int ky = 0; ky < p.Ky; ++ky)
        for (int c = 0; c < 4; ++c)
          packed[((size_t)kx * p.Ky + ky) * 4 + c] = (float)spec[c * comp + (size_t)ky * p.Hx + kx];
  } else {
    // [kz][pair][kx][ky] x (xx, yy), (zz, xy), (xz, yz): the z convolution's lanes take consecutive
    // (kx, ky) columns at one kz, so each of its loads reads consecutive 8-byte entries
    for (int kz = 0; kz < p.Kz; ++kz)
      for (int i = 0; i < 3; ++i)
        for (int kx = 0; kx < p.Hx; ++kx)
          for (int ky = 0; ky < p.Ky; ++ky)
            for (int c = 0; c < 2; ++c)
              packed[((((size_t)kz * 3 + i) * p.Hx + kx) * p.Ky + ky) * 2 + c] =
                  (float)spec[(2 * i + c) * comp + (size_t)kz * plane + (size_t)ky * p.Hx + kx];
  }
  cudaError_t e = cudaMemcpyAsync(m->K, packed.data(), p.bytes_K, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "kernel upload");
  if (key) spec_cache_put(*key, packed_ptr);
  m->kernel_set = true;
  return GBD_OK;
}

gbd_status gbd_set_kernel(gbd_mesh* m, void* stream) {
  if (!m) return fail(GBD_EINVAL, "mesh is NULL");
  gbd_status s = check_device(m);
  if (s != GBD_OK) return s;
  const gbd::Plan& p = m->p;
  const GeoKey key{p.nx, p.ny, p.nz, m->d.dx, m->d.dy, m->d.dz, p.per, p.images, p.Px, p.Py, p.Pz};
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (auto hit = spec_cache_get(key)) {
    cudaError_t e = cudaMemcpyAsync(m->K, hit->data(), p.bytes_K, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "kernel upload");
    m->kernel_set = true;
    return GBD_OK;
  }
  std::vector<double> spec;
  if (!gbdt::kernel_spectrum(p, m->d.dx, m->d.dy, m->d.dz, spec)) return fail(GBD_ENOMEM, "host allocation failed");
  return upload_spectrum(m, spec, st, &key);
}

// Spectrum of a caller tensor [6][Gz][Gy][Gx] (see gbd_set_kernel_tensor).
static gbd_status spectrum_of_tensor(const gbd::Plan& p, const double* N6, std::vector<double>& spec) {
  if (!N6) return fail(GBD_EINVAL, "tensor is NULL");
  std::vector<double> oct;
  const int r = gbdt::octant_from_full(p, N6, oct, GBD_TENSOR_SYM_TOL);
  if (r < 0) return fail(GBD_ENOMEM, "host allocation failed");
  if (r > 0)
    return fail(GBD_EINVAL, "tensor has a non-finite value or lacks the demag parities (xx, yy, zz even; "
                            "xy odd in X, Y; xz odd in X, Z; yz odd in Y, Z)");
  if (!gbdt::spectrum_from_octant(p, oct, spec)) return fail(GBD_ENOMEM, "host allocation failed");
  return GBD_OK;
}

gbd_status gbd_set_kernel_tensor(gbd_mesh* m, const double* N6, void* stream) {
  if (!m) return fail(GBD_EINVAL, "mesh is NULL");
  gbd_status s = check_device(m);
  if (s != GBD_OK) return s;
  std::vector<double> spec;
  s = spectrum_of_tensor(m->p, N6, spec);
  if (s != GBD_OK) return s;
  return upload_spectrum(m, spec, static_cast<cudaStream_t>(stream), nullptr);
}

static gbd_status ready(gbd_mesh* m) {
  if (!m) return fail(GBD_EINVAL, "mesh is NULL");
  if (!m->kernel_set) return fail(GBD_ESTATE, "gbd_set_kernel has not been called on this mesh");
  return check_device(m);
}

gbd_status gbd_demag(gbd_mesh* m, const float* M, float* H, void* stream) {
  gbd_status s = ready(m);
  if (s != GBD_OK) return s;
  if (!ptr_ok(M) || !ptr_ok(H)) return fail(GBD_EINVAL, "M and H must be non-NULL, 4-byte aligned device pointers");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  gbd::RowArgs a = row_args(m);
  a.in = M;
  a.mode = gbd::ROW_FWD;
  a.fwd_after = 1;
  timed(m, GBD_PASS_ROW_FWD, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
  enqueue_conv(m, m->S, m->T, st);
  a.hscale = 1.f;
  a.out = H;
  a.mode = gbd::ROW_H;
  a.fwd_after = 0;
  timed(m, GBD_PASS_ROW_INV, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
  mark_done(m, st);
  return after_launch("gbd_demag");
}

static gbd_status field_like(gbd_mesh* m, const float* mm, float* out, int mode, void* stream, const char* name) {
  gbd_status s = ready(m);
  if (s != GBD_OK) return s;
  if (!ptr_ok(mm) || !ptr_ok(out)) return fail(GBD_EINVAL, "m and out must be non-NULL, 4-byte aligned device pointers");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  gbd::RowArgs a = row_args(m);
  a.in = mm;
  a.mode = gbd::ROW_FWD;
  a.fwd_after = 1;
  timed(m, GBD_PASS_ROW_FWD, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
  enqueue_conv(m, m->S, m->T, st);
  a.ms = mm;
  a.out = out;
  a.mode = mode;
  a.fwd_after = 0;
  timed(m, GBD_PASS_ROW_INV, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
  mark_done(m, st);
  return after_launch(name);
}

gbd_status gbd_effective_field(gbd_mesh* m, const float* mm, float* H, void* stream) {
  return field_like(m, mm, H, gbd::ROW_HEFF, stream, "gbd_effective_field");
}

gbd_status gbd_llg_rhs(gbd_mesh* m, const float* mm, float* dmdt, void* stream) {
  return field_like(m, mm, dmdt, gbd::ROW_RHS, stream, "gbd_llg_rhs");
}

// Lagrange weights of the quartic through the step starts t_n, t_n - dt, ..., t_n - 4 dt,
// evaluated at t_n + c dt.
static void extrap_weights(double c, float w[5]) {
  for (int k = 0; k < 5; ++k) {
    double num = 1.0, den = 1.0;
    for (int j = 0; j < 5; ++j)
      if (j != k) {
        num *= c + j;
        den *= (double)(j - k);
      }
    w[k] = (float)(num / den);
  }
}

// Allocates the mesh's extrapolation history on first use (never inside a stream capture).
static gbd_status ensure_history(gbd_mesh* m) {
  if (m->hist) return GBD_OK;
  cudaError_t e = mesh_alloc(m->device, (void**)&m->hist, (size_t)5 * 3 * m->p.N * sizeof(float));
  if (e != cudaSuccess) {
    cudaGetLastError();
    m->hist = nullptr;
    return fail(e == cudaErrorMemoryAllocation ? GBD_ENOMEM : GBD_ECUDA, "demag history allocation");
  }
  m->hist_count = 0;
  return GBD_OK;
}

// The launch sequence of gbd_llg_step_ex on st (timed per launch when the mesh's timing is on).
// Advances the mesh's extrapolation history state as the launches will; with GBD_STEP_EXTRAP
// the history must exist.
static void enqueue_llg_ex(gbd_mesh* m, float* mm, int nsteps, double dt, unsigned flags, cudaStream_t st) {
  if (nsteps <= 0) return;
  const bool extrap = (flags & GBD_STEP_EXTRAP) != 0;
  const long long n3 = 3 * m->p.N;
  if (extrap) {
    if (!(flags & GBD_STEP_CONTINUE) || dt != m->hist_dt) m->hist_count = 0;
    m->hist_dt = dt;
  }
  float w_half[5], w_one[5];
  extrap_weights(0.5, w_half);
  extrap_weights(1.0, w_one);
  gbd::RowArgs a = row_args(m);
  a.dt = (float)dt;
  a.in = mm;
  a.mode = gbd::ROW_FWD;
  a.fwd_after = 1;
  timed(m, GBD_PASS_ROW_FWD, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
  a.m0 = mm;
  a.m0_out = mm;
  a.acc = m->acc;
  for (int step = 0; step < nsteps; ++step) {
    const bool last = (step == nsteps - 1);
    // stage inputs: m -> A -> B -> A -> m
    const float* ms[4] = {mm, m->bufA, m->bufB, m->bufA};
    float* mn[4] = {m->bufA, m->bufB, m->bufA, nullptr};
    // with four earlier step-start fields in the history, this step's stages 2-4 extrapolate
    const bool warm = extrap && m->hist_count >= 4;
    for (int stage = 0; stage < 4; ++stage) {
      a.ms = ms[stage];
      a.mnext = mn[stage];
      a.mode = gbd::ROW_RK1 + stage;
      a.extrap = 0;
      a.hrec = nullptr;
      if (stage == 0 && extrap) {
        m->hist_head = (m->hist_head + 1) % 5;
        a.hrec = m->hist + (size_t)m->hist_head * n3;
        if (m->hist_count < 5) ++m->hist_count;
      }
      a.hx0 = a.hx1 = nullptr;
      if (warm && stage == 1) {
        // stage 2 reads the five fields once for all three stages: it keeps its own, at t + dt/2, for
        // stage 3 in the x spectrum's buffer, free until stage 4's forward transform (at least 12 bytes
        // per cell), and stage 4's, at t + dt, in place of the oldest field, which the next step's first
        // stage replaces
        a.extrap = 1;
        a.nh = 5;
        for (int k = 0; k < 5; ++k) {
          a.hw[k] = w_half[k];
          a.hw1[k] = w_one[k];
          a.hist[k] = m->hist + (size_t)((m->hist_head - k + 5) % 5) * n3;
        }
        a.hx0 = reinterpret_cast<float*>(m->S);
        a.hx1 = m->hist + (size_t)((m->hist_head + 1) % 5) * n3;
      } else if (warm && stage > 1) {
        a.extrap = 1;
        a.nh = 1;
        a.hw[0] = 1.f;
        a.hist[0] = stage == 2 ? reinterpret_cast<const float*>(m->S) : m->hist + (size_t)((m->hist_head + 1) % 5) * n3;
        for (int k = 1; k < 5; ++k) a.hist[k] = nullptr;
      } else {
        enqueue_conv(m, m->S, m->T, st);
      }
      // the next stage needs this stage's forward transform unless it extrapolates
      const bool next_exact = stage == 3 ? !last : !warm;
      a.fwd_after = next_exact ? 1 : 0;
      if (a.extrap && !a.fwd_after)
        timed(m, GBD_PASS_EXTRAP, st, [&] { gbd::launch_extrap_stage(a, st); });
      else
        timed(m, GBD_PASS_ROW_RK, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
    }
  }
}

gbd_status gbd_llg_step_ex(gbd_mesh* m, float* mm, int nsteps, double dt, unsigned flags, void* stream) {
  gbd_status s = ready(m);
  if (s != GBD_OK) return s;
  if (!ptr_ok(mm)) return fail(GBD_EINVAL, "m must be a non-NULL, 4-byte aligned device pointer");
  if (nsteps < 0) return fail(GBD_EINVAL, "nsteps must be >= 0");
  if (!(dt > 0) || !std::isfinite(dt)) return fail(GBD_EINVAL, "dt must be finite and > 0");
  if (flags & ~(unsigned)(GBD_STEP_EXTRAP | GBD_STEP_CONTINUE)) return fail(GBD_EINVAL, "unknown flags");
  if (nsteps == 0) return GBD_OK;
  if (flags & GBD_STEP_EXTRAP) {
    s = ensure_history(m);
    if (s != GBD_OK) return s;
  }
  enqueue_llg_ex(m, mm, nsteps, dt, flags, static_cast<cudaStream_t>(stream));
  mark_done(m, static_cast<cudaStream_t>(stream));
  return after_launch("gbd_llg_step");
}

// ---- adaptive RKF5(6) (Sec. III) -------------------------------------------------------------
// Fehlberg's eight-stage RK5(6) pair: rows a_(i+1),j of the stage matrix, fifth-order weights
// b5 (the step's result) and sixth-order weights b6 (the error estimate).
static const double kRkfA[8][7] = {
    {0, 0, 0, 0, 0, 0, 0},
    {1.0 / 6, 0, 0, 0, 0, 0, 0},
    {4.0 / 75, 16.0 / 75, 0, 0, 0, 0, 0},
    {5.0 / 6, -8.0 / 3, 5.0 / 2, 0, 0, 0, 0},
    {-8.0 / 5, 144.0 / 25, -4.0, 16.0 / 25, 0, 0, 0},
    {361.0 / 320, -18.0 / 5, 407.0 / 128, -11.0 / 80, 55.0 / 128, 0, 0},
    {-11.0 / 640, 0, 11.0 / 256, -11.0 / 160, 11.0 / 256, 0, 0},
    {93.0 / 640, -18.0 / 5, 803.0 / 256, -11.0 / 160, 99.0 / 256, 0, 1.0}};
static const double kRkfB5[8] = {31.0 / 384, 0, 1125.0 / 2816, 9.0 / 32, 125.0 / 768, 5.0 / 66, 0, 0};
static const double kRkfB6[8] = {7.0 / 1408, 0, 1125.0 / 2816, 9.0 / 32, 125.0 / 768, 0, 5.0 / 66, 5.0 / 66};
static const double kRkfC[8] = {0, 1.0 / 6, 4.0 / 15, 2.0 / 3, 4.0 / 5, 1.0, 0, 1.0};
static const double kRkfSafety = 0.9, kRkfFacMin = 0.2, kRkfFacMax = 5.0;

// An accepted step of size h: with extrapolation the pending field becomes the newest history
// entry (at relative time 0 before the shift), the oldest slot becomes the next pending one,
// and every recorded time moves back by h.
static void rkf_accept(gbd_mesh* m, double h, bool extrap) {
  if (!extrap) return;
  const int freed = m->rk_ring[4];
  for (int q = 4; q > 0; --q) {
    m->rk_ring[q] = m->rk_ring[q - 1];
    m->rk_ring_t[q] = m->rk_ring_t[q - 1] - h;
  }
  m->rk_ring[0] = m->rk_pend;
  m->rk_ring_t[0] = -h;
  m->rk_pend = freed;
  if (m->rk_count < 5) ++m->rk_count;
}

static gbd_status ensure_rkf_history(gbd_mesh* m) {
  if (m->rk_hist) return GBD_OK;
  cudaError_t e = mesh_alloc(m->device, (void**)&m->rk_hist, (size_t)6 * 3 * m->p.N * sizeof(float));
  if (e != cudaSuccess) {
    cudaGetLastError();
    m->rk_hist = nullptr;
    return fail(e == cudaErrorMemoryAllocation ? GBD_ENOMEM : GBD_ECUDA, "RKF5(6) demag history allocation");
  }
  m->rk_count = 0;
  return GBD_OK;
}

static gbd_status ensure_rkf(gbd_mesh* m) {
  if (m->rk_k) return GBD_OK;
  const size_t n3 = (size_t)3 * m->p.N;
  cudaError_t e = mesh_alloc(m->device, (void**)&m->rk_k, 8 * n3 * sizeof(float));
  if (e == cudaSuccess) e = mesh_alloc(m->device, (void**)&m->rk_m, n3 * sizeof(float));
  if (e == cudaSuccess) e = mesh_alloc(m->device, (void**)&m->rk_err, sizeof(unsigned));
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaStream_t ls = lib_stream(m->device);
    if (m->rk_k) cudaFreeAsync(m->rk_k, ls);
    if (m->rk_m) cudaFreeAsync(m->rk_m, ls);
    if (m->rk_err) cudaFreeAsync(m->rk_err, ls);
    cudaStreamSynchronize(ls);
    m->rk_k = m->rk_m = nullptr;
    m->rk_err = nullptr;
    return fail(e == cudaErrorMemoryAllocation ? GBD_ENOMEM : GBD_ECUDA, "RKF5(6) buffer allocation");
  }
  return GBD_OK;
}

// Enqueues one RKF5(6) attempt of size h from mm on st: the normalized fifth-order result into
// m->rk_m and the largest error norm |sum_i (b6_i - b5_i) k_i| (float bits) into *err_word, which
// must be zero beforehand. With hdev the step size is read on the device (*hdev, FP32; h is not
// used) and there is no extrapolation.
static void rkf_enqueue_attempt(gbd_mesh* m, const float* mm, double h, const float* hdev, unsigned* err_word,
                                cudaStream_t st, bool extrap) {
  const size_t n3 = (size_t)3 * m->p.N;
  float* k[8];
  for (int i = 0; i < 8; ++i) k[i] = m->rk_k + i * n3;
  // with five accepted step starts recorded, stages 2-8 take the quintic through them and this
  // step's stage-1 field (recorded into the pending slot) instead of a convolution
  const bool warm = extrap && m->rk_count >= 5;
  double nodes[6] = {0.0};
  const float* hsrc[6] = {nullptr};
  if (extrap) {
    hsrc[0] = m->rk_hist + (size_t)m->rk_pend * n3;
    for (int q = 0; q < 5; ++q) {
      nodes[q + 1] = m->rk_ring_t[q];
      hsrc[q + 1] = m->rk_hist + (size_t)m->rk_ring[q] * n3;
    }
  }
  const double hk = hdev ? 1.0 : h;   // factor folded into the weights on the host
  gbd::RowArgs a = row_args(m);
  a.in = mm;
  a.mode = gbd::ROW_FWD;
  a.fwd_after = 1;
  timed(m, GBD_PASS_ROW_FWD, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
  float* stage_in[2] = {m->bufA, m->bufB};
  const float* ms = mm;
  for (int i = 0; i < 8; ++i) {
    a.mode = gbd::ROW_RKG;
    a.ms = ms;
    a.m0 = mm;
    a.kout = k[i];
    a.nk = i;
    a.hdev = hdev;
    for (int j = 0; j < i; ++j) a.kin[j] = k[j];
    a.hrec = (extrap && i == 0) ? m->rk_hist + (size_t)m->rk_pend * n3 : nullptr;
    a.extrap = 0;
    a.nh = 0;
    if (warm && i > 0) {
      a.extrap = 1;
      a.nh = 6;
      const double c = kRkfC[i] * h;
      for (int q = 0; q < 6; ++q) {
        double num = 1.0, den = 1.0;
        for (int r = 0; r < 6; ++r)
          if (r != q) {
            num *= c - nodes[r];
            den *= nodes[q] - nodes[r];
          }
        a.hw[q] = (float)(num / den);
        a.hist[q] = hsrc[q];
      }
    }
    if (i < 7) {
      for (int j = 0; j <= i; ++j) a.kw[j] = (float)(hk * kRkfA[i + 1][j]);
      a.mnext = stage_in[i % 2];
    } else {
      a.mnext = nullptr;
    }
    // the next stage needs this stage's forward transform only when it convolves
    a.fwd_after = (i < 7 && !warm) ? 1 : 0;
    if (a.extrap) {
      timed(m, GBD_PASS_EXTRAP, st, [&] { gbd::launch_extrap_stage(a, st); });
    } else {
      enqueue_conv(m, m->S, m->T, st);
      timed(m, GBD_PASS_ROW_RK, st, [&] { gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st); });
    }
    ms = a.mnext;
  }
  gbd::RkfArgs f;
  std::memset(&f, 0, sizeof(f));
  f.N = m->p.N;
  f.m = mm;
  for (int i = 0; i < 8; ++i) {
    f.k[i] = k[i];
    f.b5dt[i] = (float)(hk * kRkfB5[i]);
    f.db[i] = (float)(kRkfB6[i] - kRkfB5[i]);
  }
  f.out = m->rk_m;
  f.err_max = err_word;
  f.hdev = hdev;
  gbd::launch_rkf_final(f, st);
}

// One RKF5(6) step of size h from mm: the normalized fifth-order result into m->rk_m and the
// error estimate h max_cells |sum_i (b6_i - b5_i) k_i| into *err (waits for the stream).
static gbd_status rkf_step(gbd_mesh* m, const float* mm, double h, cudaStream_t st, double* err, bool extrap) {
  cudaError_t e = cudaMemsetAsync(m->rk_err, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return cuda_fail(e, "RKF5(6) step");
  rkf_enqueue_attempt(m, mm, h, nullptr, m->rk_err, st, extrap);
  unsigned err_word = 0;
  e = cudaMemcpyAsync(&err_word, m->rk_err, sizeof(unsigned), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "RKF5(6) step");
  float ef;
  std::memcpy(&ef, &err_word, sizeof(float));
  *err = h * (double)ef;
  return GBD_OK;
}

// gbd_llg_run_rkf56 without extrapolation: the whole adaptive run as one CUDA graph whose
// conditional WHILE node repeats [attempt, step control, copy if accepted] until t_end or
// max_steps, so the host neither waits nor launches between steps. The instantiated graph is
// kept in the mesh for the magnetization array it was built on (and rebuilt after a parameter
// or tuning change).
static gbd_status rkf_run_device(gbd_mesh* m, float* mm, double t_end, double* dt, double tol, int max_steps,
                                 int* accepted, int* rejected, cudaStream_t st) {
  if (!m->rk_ctl) {
    cudaError_t e = mesh_alloc(m->device, (void**)&m->rk_ctl, sizeof(gbd::RkfCtl));
    if (e != cudaSuccess) {
      cudaGetLastError();
      m->rk_ctl = nullptr;
      return fail(e == cudaErrorMemoryAllocation ? GBD_ENOMEM : GBD_ECUDA, "RKF5(6) control block allocation");
    }
  }
  if (!m->rkf_exec || m->rkf_key_m != mm || m->rkf_key_version != m->version) {
    if (m->rkf_exec) {
      cudaGraphExecDestroy(m->rkf_exec);
      m->rkf_exec = nullptr;
    }
    cudaGraph_t g = nullptr;
    cudaStream_t cs = nullptr;
    cudaGraphConditionalHandle cond;
    cudaError_t e = cudaGraphCreate(&g, 0);
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault);
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = cond;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    if (e == cudaSuccess) e = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
      cudaGraph_t body = np.conditional.phGraph_out[0];
      e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        const int tmp = m->timing;
        m->timing = 0;   // no timing events inside the graph
        rkf_enqueue_attempt(m, mm, 0.0, &m->rk_ctl->hf, &m->rk_ctl->err, cs, false);
        m->timing = tmp;
        gbd::launch_rkf_control(m->rk_ctl, cond, kRkfSafety, kRkfFacMin, kRkfFacMax, cs);
        gbd::launch_rkf_accept(m->rk_ctl, m->rk_m, mm, 3 * m->p.N, cs);
        e = cudaStreamEndCapture(cs, &body);
      }
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&m->rkf_exec, g, 0);
    if (cs) cudaStreamDestroy(cs);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      cudaGetLastError();
      m->rkf_exec = nullptr;
      return cuda_fail(e, "gbd_llg_run_rkf56: graph");
    }
    m->rkf_key_m = mm;
    m->rkf_key_version = m->version;
  }
  gbd::RkfCtl c;
  std::memset(&c, 0, sizeof(c));
  c.t_end = t_end;
  c.tol = tol;
  c.h = std::min(*dt, t_end);
  c.h_next = *dt;
  c.hf = (float)c.h;
  c.max_steps = max_steps;
  cudaError_t e = cudaSuccess;
  if (t_end > 0.0) {
    e = cudaMemcpyAsync(m->rk_ctl, &c, sizeof(c), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaGraphLaunch(m->rkf_exec, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&c, m->rk_ctl, sizeof(c), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) return cuda_fail(e, "gbd_llg_run_rkf56");
  *dt = c.h_next;
  if (accepted) *accepted = c.acc;
  if (rejected) *rejected = c.rej;
  mark_done(m, st);
  return after_launch("gbd_llg_run_rkf56");
}

// Validates RKF flags, allocates what they need and resets the history unless continued.
static gbd_status rkf_prepare(gbd_mesh* m, unsigned flags) {
  if (flags & ~(unsigned)(GBD_STEP_EXTRAP | GBD_STEP_CONTINUE)) return fail(GBD_EINVAL, "unknown flags");
  gbd_status s = ensure_rkf(m);
  if (s != GBD_OK) return s;
  if (flags & GBD_STEP_EXTRAP) {
    s = ensure_rkf_history(m);
    if (s != GBD_OK) return s;
    if (!(flags & GBD_STEP_CONTINUE)) m->rk_count = 0;
  }
  return GBD_OK;
}

gbd_status gbd_llg_rkf56_step(gbd_mesh* m, float* mm, double dt, double* err, unsigned flags, void* stream) {
  gbd_status s = ready(m);
  if (s != GBD_OK) return s;
  if (!ptr_ok(mm) || !err) return fail(GBD_EINVAL, "m must be a 4-byte aligned device pointer and err non-NULL");
  if (!(dt > 0) || !std::isfinite(dt)) return fail(GBD_EINVAL, "dt must be finite and > 0");
  s = rkf_prepare(m, flags);
  if (s != GBD_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const bool extrap = (flags & GBD_STEP_EXTRAP) != 0;
  s = rkf_step(m, mm, dt, st, err, extrap);
  if (s != GBD_OK) return s;
  rkf_accept(m, dt, extrap);
  cudaError_t e = cudaMemcpyAsync(mm, m->rk_m, (size_t)3 * m->p.N * sizeof(float), cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return cuda_fail(e, "gbd_llg_rkf56_step");
  mark_done(m, st);
  return after_launch("gbd_llg_rkf56_step");
}

gbd_status gbd_llg_run_rkf56(gbd_mesh* m, float* mm, double t_end, double* dt, double tol, int max_steps,
                             int* accepted, int* rejected, unsigned flags, void* stream) {
  gbd_status s = ready(m);
  if (s != GBD_OK) return s;
  if (!ptr_ok(mm) || !dt) return fail(GBD_EINVAL, "m must be a 4-byte aligned device pointer and dt non-NULL");
  if (!(t_end >= 0) || !std::isfinite(t_end)) return fail(GBD_EINVAL, "t_end must be finite and >= 0");
  if (!(*dt > 0) || !std::isfinite(*dt)) return fail(GBD_EINVAL, "*dt must be finite and > 0");
  if (!(tol > 0) || !std::isfinite(tol)) return fail(GBD_EINVAL, "tol must be finite and > 0");
  if (max_steps < 1) return fail(GBD_EINVAL, "max_steps must be >= 1");
  s = rkf_prepare(m, flags);
  if (s != GBD_OK) return s;
  const bool extrap = (flags & GBD_STEP_EXTRAP) != 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (!extrap && !m->timing) return rkf_run_device(m, mm, t_end, dt, tol, max_steps, accepted, rejected, st);
  const size_t bytes = (size_t)3 * m->p.N * sizeof(float);
  double t = 0.0, h_next = *dt;
  int acc = 0, rej = 0;
  while (t < t_end && acc + rej < max_steps) {
    const double h = std::min(h_next, t_end - t);
    double err = 0.0;
    s = rkf_step(m, mm, h, st, &err, extrap);
    if (s != GBD_OK) return s;
    const double fac = err == 0.0 ? kRkfFacMax
                                  : std::min(kRkfFacMax, std::max(kRkfFacMin, kRkfSafety * std::pow(tol / err, 1.0 / 6.0)));
    h_next = h * fac;
    if (err <= tol) {
      cudaError_t e = cudaMemcpyAsync(mm, m->rk_m, bytes, cudaMemcpyDeviceToDevice, st);
      if (e != cudaSuccess) return cuda_fail(e, "gbd_llg_run_rkf56");
      rkf_accept(m, h, extrap);
      t += h;
      ++acc;
    } else {
      ++rej;
    }
  }
  *dt = h_next;
  if (accepted) *accepted = acc;
  if (rejected) *rejected = rej;
  mark_done(m, st);
  return after_launch("gbd_llg_run_rkf56");
}

gbd_status gbd_llg_step(gbd_mesh* m, float* mm, int nsteps, double dt, void* stream) {
  return gbd_llg_step_ex(m, mm, nsteps, dt, 0u, stream);
}

// ---- integrator state (checkpoint / resume) ---------------------------------------------------
// Host image: a fixed header, then the RK4 demag history (5 slots of [3][N] float32) if the
// mesh has one, then the RKF5(6) history (6 slots) if it has one. The header records the mesh
// shape and periodic axes, so an image only loads into a mesh whose slots have its layout.
struct StateHeader {
  char magic[8];            // "GBDSTAT2"
  long long N;              // cells
  int nx, ny, nz, per;      // mesh shape and periodic axes of the saved mesh
  int has_hist, hist_count, hist_head, has_rk;
  double hist_dt;
  int rk_ring[5];
  int rk_count, rk_pend;
  double rk_ring_t[5];
};
static const char kStateMagic[8] = {'G', 'B', 'D', 'S', 'T', 'A', 'T', '2'};

static size_t state_bytes(const gbd_mesh* m) {
  const size_t slot = (size_t)3 * m->p.N * sizeof(float);
  return sizeof(StateHeader) + (m->hist ? 5 * slot : 0) + (m->rk_hist ? 6 * slot : 0);
}

gbd_status gbd_mesh_state_bytes(const gbd_mesh* m, size_t* out) {
  if (!m || !out) return fail(GBD_EINVAL, "mesh or out is NULL");
  *out = state_bytes(m);
  return GBD_OK;
}

gbd_status gbd_mesh_get_state(gbd_mesh* m, void* host, size_t bytes, void* stream) {
  if (!m || !host) return fail(GBD_EINVAL, "mesh or buffer is NULL");
  gbd_status s = check_device(m);
  if (s != GBD_OK) return s;
  if (bytes < state_bytes(m)) return fail(GBD_EINVAL, "buffer smaller than gbd_mesh_state_bytes");
  StateHeader h;
  std::memset(&h, 0, sizeof(h));
  std::memcpy(h.magic, kStateMagic, sizeof(kStateMagic));
  h.N = m->p.N;
  h.nx = m->p.nx;
  h.ny = m->p.ny;
  h.nz = m->p.nz;
  h.per = m->p.per;
  h.has_hist = m->hist != nullptr;
  h.hist_count = m->hist_count;
  h.hist_head = m->hist_head;
  h.hist_dt = m->hist_dt;
  h.has_rk = m->rk_hist != nullptr;
  for (int i = 0; i < 5; ++i) {
    h.rk_ring[i] = m->rk_ring[i];
    h.rk_ring_t[i] = m->rk_ring_t[i];
  }
  h.rk_count = m->rk_count;
  h.rk_pend = m->rk_pend;
  char* out = static_cast<char*>(host);
  std::memcpy(out, &h, sizeof(h));
  out += sizeof(h);
  const size_t slot = (size_t)3 * m->p.N * sizeof(float);
  cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  if (e == cudaSuccess && m->hist) {
    e = cudaMemcpy(out, m->hist, 5 * slot, cudaMemcpyDeviceToHost);
    out += 5 * slot;
  }
  if (e == cudaSuccess && m->rk_hist) e = cudaMemcpy(out, m->rk_hist, 6 * slot, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "gbd_mesh_get_state");
  return GBD_OK;
}

gbd_status gbd_mesh_set_state(gbd_mesh* m, const void* host, size_t bytes, void* stream) {
  if (!m || !host) return fail(GBD_EINVAL, "mesh or buffer is NULL");
  gbd_status s = check_device(m);
  if (s != GBD_OK) return s;
  StateHeader h;
  if (bytes < sizeof(h)) return fail(GBD_EINVAL, "buffer shorter than a state header");
  std::memcpy(&h, host, sizeof(h));
  const size_t slot = (size_t)3 * m->p.N * sizeof(float);
  const bool ring_ok = h.rk_count >= 0 && h.rk_count <= 5 && h.rk_pend >= 0 && h.rk_pend < 6 &&
                       std::all_of(h.rk_ring, h.rk_ring + 5, [](int v) { return v >= 0 && v < 6; });
  if (std::memcmp(h.magic, kStateMagic, sizeof(kStateMagic)) != 0 || h.N != m->p.N || h.nx != m->p.nx ||
      h.ny != m->p.ny || h.nz != m->p.nz || h.per != m->p.per || h.hist_count < 0 || h.hist_count > 5 ||
      h.hist_head < 0 || h.hist_head >= 5 || !ring_ok)
    return fail(GBD_EINVAL, "not a state image of a mesh of this shape and periodicity");
  if (bytes != sizeof(h) + (h.has_hist ? 5 * slot : 0) + (h.has_rk ? 6 * slot : 0))
    return fail(GBD_EINVAL, "state image size does not match its header");
  if (h.has_hist && (s = ensure_history(m)) != GBD_OK) return s;
  if (h.has_rk && (s = ensure_rkf_history(m)) != GBD_OK) return s;
  const char* in = static_cast<const char*>(host) + sizeof(h);
  cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  if (e == cudaSuccess && h.has_hist) {
    e = cudaMemcpy(m->hist, in, 5 * slot, cudaMemcpyHostToDevice);
    in += 5 * slot;
  }
  if (e == cudaSuccess && h.has_rk) e = cudaMemcpy(m->rk_hist, in, 6 * slot, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    // the device histories may be partly overwritten: the next extrapolated step restarts them
    m->hist_count = 0;
    m->rk_count = 0;
    ++m->version;
    return cuda_fail(e, "gbd_mesh_set_state");
  }
  m->hist_count = h.has_hist ? h.hist_count : 0;
  m->hist_head = h.hist_head;
  m->hist_dt = h.hist_dt;
  for (int i = 0; i < 5; ++i) {
    m->rk_ring[i] = h.rk_ring[i];
    m->rk_ring_t[i] = h.rk_ring_t[i];
  }
  m->rk_count = h.has_rk ? h.rk_count : 0;
  m->rk_pend = h.rk_pend;
  ++m->version;   // batch graphs keyed on the history state re-capture
  return GBD_OK;
}

}  // extern "C"

// ---- allocation-free demag -------------------------------------------------------------------
//
// Scratch for gbd_demag_noalloc: the x spectrum and, for 3D meshes, the y spectrum of one
// demag evaluation live in this file-scope device array instead of the mesh's buffers.
// Every GPU that loads the library holds it (GBD_NOALLOC_MAX_BYTES) until the process exits.
// Host code cannot use the symbol as a device address: its device address is looked up once
// per device with cudaGetSymbolAddress, with that device current, and passed to the kernels.
static __device__ __align__(256) unsigned char g_noalloc_scratch[GBD_NOALLOC_MAX_BYTES];

namespace {
constexpr int kNoallocMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_addr[kNoallocMaxDevices] = {nullptr};

}  // namespace

extern "C" gbd_status gbd_demag_noalloc(gbd_mesh* m, const float* M, float* H, void* stream) {
  gbd_status s = ready(m);
  if (s != GBD_OK) return s;
  if (!ptr_ok(M) || !ptr_ok(H)) return fail(GBD_EINVAL, "M and H must be non-NULL, 4-byte aligned device pointers");
  const gbd::Plan& p = m->p;
  const size_t s_bytes = (p.bytes_S + 255) / 256 * 256;
  const size_t need = s_bytes + p.bytes_T;
  if (need > (size_t)GBD_NOALLOC_MAX_BYTES)
    return fail(GBD_EBUDGET, "gbd_demag_noalloc: this mesh needs " + std::to_string(need) +
                                 " bytes of scratch, more than the static maximum of " +
                                 std::to_string((size_t)GBD_NOALLOC_MAX_BYTES));
  int dev = m->device;
  if (dev < 0 || dev >= kNoallocMaxDevices) return fail(GBD_EUNSUPPORTED, "gbd_demag_noalloc: device ordinal out of range");
  void* base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
      void* ptr = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
      if (e != cudaSuccess || !ptr) return cuda_fail(e, "gbd_demag_noalloc: cudaGetSymbolAddress");
      g_noalloc_addr[dev] = ptr;
    }
    base = g_noalloc_addr[dev];
  }
  float2* S = static_cast<float2*>(base);
  float2* T = p.bytes_T ? reinterpret_cast<float2*>(static_cast<unsigned char*>(base) + s_bytes) : nullptr;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  gbd::RowArgs a = row_args(m);
  a.S = S;
  a.in = M;
  a.mode = gbd::ROW_FWD;
  a.fwd_after = 1;
  gbd::launch_row(p.Lx, row_var(m, a.mode), p.prec, a, m->tw, st);
  const int tmp = m->timing;
  m->timing = 0;   // this call is not traced
  enqueue_conv(m, S, T, st);
  m->timing = tmp;
  a.hscale = 1.f;
  a.out = H;
  a.mode = gbd::ROW_H;
  a.fwd_after = 0;
  gbd::launch_row(p.Lx, row_var(m, a.mode), p.prec, a, m->tw, st);
  mark_done(m, st);
  return after_launch("gbd_demag_noalloc");
}

// ---- tile-shape autotuner --------------------------------------------------------------------
//
// Each kernel family has two tile shapes (lines per block; gbd_kernels.cuh). They compute the
// same numbers -- every line's transform and every cell's update is independent of how lines
// are grouped into blocks -- so the choice only changes speed. gbd_mesh_autotune times both
// shapes of each pass whose launches on this mesh have them, on the mesh's own (zeroed) buffers, keeps the faster one,
// and caches the choice by mesh size and device: in the process, and in the text file named
// by GBD_AUTOTUNE_CACHE when that is set (lines "gbd<generation> nx ny nz device Px Py precision var_row
// var_film var_y var_z pow2 var_row_io"). A choice holds for the kernels it was timed on: lines of
// another generation, and the lines without one that older versions wrote, are passed over. For a mesh planned with 3 * 2^k / 5 * 2^k lengths it also times the
// power-of-two plan of the same mesh and moves the mesh onto it when that is faster (pow2 = 1).

namespace {
struct TuneKey {
  int nx, ny, nz, dev, Px, Py, prec;
  bool operator<(const TuneKey& o) const {
    if (Px != o.Px) return Px < o.Px;
    if (Py != o.Py) return Py < o.Py;
    if (prec != o.prec) return prec < o.prec;
    if (nx != o.nx) return nx < o.nx;
    if (ny != o.ny) return ny < o.ny;
    if (nz != o.nz) return nz < o.nz;
    return dev < o.dev;
  }
};
std::mutex g_tune_mu;
std::map<TuneKey, std::array<int, 6>> g_tune;   // variants (row, film, y, z), power-of-two padding, row (transforms only)
bool g_tune_file_read = false;
// Raised whenever a variant number comes to mean another tile or kernel, or the kernels that a mesh
// runs change (without it: y variants 0 and 1 the other way round).
constexpr int kTuneGeneration = 2;

const char* tune_file() {
  const char* p = std::getenv("GBD_AUTOTUNE_CACHE");
  return (p && *p) ? p : nullptr;
}

void read_tune_file_locked() {
  if (g_tune_file_read) return;
  g_tune_file_read = true;
  const char* path = tune_file();
  if (!path) return;
  FILE* f = std::fopen(path, "r");
  if (!f) return;
  char line[256];
  while (std::fgets(line, sizeof line, f)) {
    int gen = 0;
    TuneKey k;
    std::array<int, 6> v;
    if (std::sscanf(line, "gbd%d %d %d %d %d %d %d %d %d %d %d %d %d %d", &gen, &k.nx, &k.ny, &k.nz, &k.dev, &k.Px, &k.Py,
                    &k.prec, &v[0], &v[1], &v[2], &v[3], &v[4], &v[5]) != 14 || gen != kTuneGeneration)
      continue;
    bool ok = (v[4] == 0 || v[4] == 1) && v[5] >= 0 && v[5] <= 3;
    for (int i = 0; i < 4; ++i) ok = ok && (v[i] == 0 || v[i] == 1 || (i == 0 && (v[i] == 2 || v[i] == 3)));
    if (ok) g_tune[k] = v;
  }
  std::fclose(f);
}

void append_tune_file_locked(const TuneKey& k, const std::array<int, 6>& v) {
  const char* path = tune_file();
  if (!path) return;
  FILE* f = std::fopen(path, "a");
  if (!f) return;
  std::fprintf(f, "gbd%d %d %d %d %d %d %d %d %d %d %d %d %d %d\n", kTuneGeneration, k.nx, k.ny, k.nz, k.dev, k.Px, k.Py,
               k.prec, v[0], v[1], v[2], v[3], v[4], v[5]);
  std::fclose(f);
}

template <class A>
void apply_tuning(gbd_mesh* m, const A& v) {
  gbd::Plan& p = m->p;
  p.var_row = v[0];
  p.var_row_io = v.size() > 5 ? v[5] : v[0];
  p.var_film = v[1];
  p.var_y = v[2];
  p.var_z = v[3];
  p.RB = gbd::row_rb(p.Lx, p.var_row);
  p.Cf = gbd::film_cols(p.Py, p.var_film);
  p.Cy = gbd::ypass_lines(p.Py, p.var_y);
  p.Wz = gbd::zconv_cols(p.Pz, p.var_z);
  ++m->version;
}

// Mean device time in ms of one launch made by f(variant), over `reps` launches after one
// untimed launch.
template <class F>
cudaError_t time_variant(cudaStream_t st, int reps, F f, float* ms) {
  cudaEvent_t e0, e1;
  cudaError_t e = cudaEventCreate(&e0);
  if (e != cudaSuccess) return e;
  e = cudaEventCreate(&e1);
  if (e != cudaSuccess) {
    cudaEventDestroy(e0);
    return e;
  }
  f();
  cudaEventRecord(e0, st);
  for (int i = 0; i < reps; ++i) f();
  cudaEventRecord(e1, st);
  e = cudaEventSynchronize(e1);
  float t = 0.f;
  if (e == cudaSuccess) e = cudaEventElapsedTime(&t, e0, e1);
  *ms = t / reps;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (e == cudaSuccess) e = cudaGetLastError();
  return e;
}
}  // namespace

namespace {
// The mesh is planned with a 3 * 2^k or 5 * 2^k length that a power-of-two plan would replace.
bool can_pad_pow2(const gbd_mesh* m) {
  return m->p.prec == 0 && !(m->d.flags & GBD_FLAG_POW2_PAD) && (gbd::mixed_len(m->p.Lx) || gbd::mixed_len(m->p.Py));
}

// Mean device time of one demag evaluation's passes (forward x, convolution, inverse x) on the
// mesh's own buffers (zeroed by the caller).
cudaError_t time_demag_passes(gbd_mesh* m, cudaStream_t st, float* ms) {
  gbd::RowArgs a = row_args(m);
  return time_variant(st, 5, [&] {
    a.in = m->bufA;
    a.mode = gbd::ROW_FWD;
    a.fwd_after = 1;
    gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st);
    enqueue_conv(m, m->S, m->T, st);
    a.out = m->bufB;
    a.mode = gbd::ROW_H;
    a.fwd_after = 0;
    gbd::launch_row(m->p.Lx, row_var(m, a.mode), m->p.prec, a, m->tw, st);
  }, ms);
}

// No tracing while the autotuner times: traced launches would be counted, and the convolution split
// into its passes.
struct Untraced {
  gbd_mesh* m;
  int timing;
  explicit Untraced(gbd_mesh* mesh) : m(mesh), timing(mesh->timing) { m->timing = 0; }
  ~Untraced() { m->timing = timing; }
};

// A scratch copy of m planned on powers of two (kernel spectrum zero: for timing only), tuned.
gbd_status make_pow2_twin(gbd_mesh* m, void* stream, gbd_mesh** out) {
  gbd_mesh_desc d2 = m->d;
  d2.flags |= GBD_FLAG_POW2_PAD;
  gbd_status s = gbd_mesh_create(&d2, out);
  if (s != GBD_OK) return s;
  gbd_mesh* t = *out;
  cudaError_t e = cudaMemsetAsync(t->K, 0, t->p.bytes_K, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) {
    gbd_mesh_destroy(t);
    return cuda_fail(e, "gbd_mesh_autotune: power-of-two plan");
  }
  t->kernel_set = true;
  s = gbd_mesh_autotune(t, stream);
  if (s != GBD_OK) gbd_mesh_destroy(t);
  return s;
}

gbd_status pow2_is_faster(gbd_mesh* m, void* stream, int* pow2) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  gbd_mesh* twin = nullptr;
  gbd_status s = make_pow2_twin(m, stream, &twin);
  if (s != GBD_OK) return s;
  float t_cur = 0.f, t_pow2 = 0.f;
  cudaError_t e = time_demag_passes(m, st, &t_cur);
  if (e == cudaSuccess) e = time_demag_passes(twin, st, &t_pow2);
  gbd_mesh_destroy(twin);
  if (e != cudaSuccess) return cuda_fail(e, "gbd_mesh_autotune: padded length");
  *pow2 = t_pow2 < 0.98f * t_cur ? 1 : 0;   // keep the shorter lengths unless clearly slower
  return GBD_OK;
}

// Moves m onto its power-of-two plan: new spectrum buffers and twiddles from a tuned twin, the
// kernel spectrum recomputed for the new lengths; the old buffers are freed after m's work.
gbd_status move_to_pow2(gbd_mesh* m, void* stream) {
  gbd_mesh* twin = nullptr;
  gbd_status s = make_pow2_twin(m, stream, &twin);
  if (s != GBD_OK) return s;
  for (auto& d : m->done) cudaEventSynchronize(d.second);
  std::swap(m->p, twin->p);
  std::swap(m->S, twin->S);
  std::swap(m->T, twin->T);
  std::swap(m->K, twin->K);
  std::swap(m->tw, twin->tw);
  std::swap(m->status, twin->status);   // the status word lies behind the twiddles
  m->d.flags |= GBD_FLAG_POW2_PAD;
  ++m->version;
  gbd_mesh_destroy(twin);
  return gbd_set_kernel(m, stream);
}
}  // namespace

extern "C" gbd_status gbd_mesh_plan_dims(const gbd_mesh* m, int out[6]) {
  if (!m || !out) return fail(GBD_EINVAL, "NULL argument");
  out[0] = m->p.Px;
  out[1] = m->p.Py;
  out[2] = m->p.Pz;
  out[3] = m->p.Hx;
  out[4] = m->p.Ky;
  out[5] = m->p.Kz;
  return GBD_OK;
}

extern "C" gbd_status gbd_mesh_get_tuning(const gbd_mesh* m, int out[4]) {
  if (!m || !out) return fail(GBD_EINVAL, "NULL argument");
  out[0] = m->p.var_row;
  out[1] = m->p.var_film;
  out[2] = m->p.var_y;
  out[3] = m->p.var_z;
  return GBD_OK;
}

extern "C" gbd_status gbd_mesh_set_tuning(gbd_mesh* m, const int in[4]) {
  if (!m || !in) return fail(GBD_EINVAL, "NULL argument");
  std::array<int, 4> v;
  for (int i = 0; i < 4; ++i) {
    if (in[i] != 0 && in[i] != 1 && !(i == 0 && (in[i] == 2 || in[i] == 3)))
      return fail(GBD_EINVAL, "tile variants are 0 or 1 (row: 0 to 3)");
    v[i] = in[i];
  }
  apply_tuning(m, v);
  return GBD_OK;
}

extern "C" gbd_status gbd_mesh_autotune(gbd_mesh* m, void* stream) {
  gbd_status s = ready(m);
  if (s != GBD_OK) return s;
  const gbd::Plan& p = m->p;
  const TuneKey key{p.nx, p.ny, p.nz, m->device, p.Px, p.Py, p.prec};
  {
    std::unique_lock<std::mutex> lock(g_tune_mu);
    read_tune_file_locked();
    auto it = g_tune.find(key);
    if (it != g_tune.end()) {
      const std::array<int, 6> v = it->second;
      lock.unlock();
      apply_tuning(m, v);
      if (v[4] == 1 && can_pad_pow2(m)) return move_to_pow2(m, stream);
      return GBD_OK;
    }
  }
  const Untraced untraced(m);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // zeroed buffers keep every timed pass finite
  cudaError_t e = cudaSuccess;
  if (p.bytes_S) e = cudaMemsetAsync(m->S, 0, p.bytes_S, st);
  if (e == cudaSuccess && p.bytes_T) e = cudaMemsetAsync(m->T, 0, p.bytes_T, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->acc, 0, p.bytes_state / 3, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->bufA, 0, p.bytes_state / 3, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->bufB, 0, p.bytes_state / 3, st);
  if (e != cudaSuccess) return cuda_fail(e, "gbd_mesh_autotune: memset");
  const int reps = 20;
  std::array<int, 4> best = {p.var_row, p.var_film, p.var_y, p.var_z};
  auto pick = [&](int slot, auto launch_v, int nvar = 2) -> cudaError_t {
    float t[4];
    for (int v = 0; v < nvar; ++v) {
      cudaError_t ee = time_variant(st, reps, [&] { launch_v(v); }, &t[v]);
      if (ee != cudaSuccess) return ee;
    }
    // keep the default unless another shape is faster by more than 2 %
    const int def = best[slot];
    int b = def;
    for (int v = 0; v < nvar; ++v)
      if (t[v] < 0.98f * t[def] && t[v] < t[b]) b = v;
    best[slot] = b;
    return cudaSuccess;
  };
  // x rows: an RK4 middle stage with the next forward transform, on zeroed state, after its convolution
  // (launched alone, back to back, the rows find their spectrum in other caches and start on empty SMs:
  // the choice lost up to a quarter of a step)
  gbd::RowArgs ra = row_args(m);
  ra.dt = 1e-13f;
  ra.ms = m->bufA;
  ra.m0 = m->bufB;
  ra.mnext = m->bufB;
  ra.acc = m->acc;
  ra.mode = gbd::ROW_RK2;
  ra.fwd_after = 1;
  const bool rows_vary = gbd::row_has_variants(p.Lx, p.prec, ra.rows);
  if (rows_vary)
    e = pick(0, [&](int v) {
      enqueue_conv(m, m->S, m->T, st);
      gbd::launch_row(p.Lx, v, p.prec, ra, m->tw, st);
    }, p.prec == 0 ? 4 : 2);
  // the transform-only x-row launches, around the convolution: a forward transform and an inverse one to H_d
  int best_io = p.var_row_io;
  if (e == cudaSuccess && rows_vary) {
    gbd::RowArgs fa = row_args(m), ia = row_args(m);
    fa.in = m->bufA;
    fa.mode = gbd::ROW_FWD;
    fa.fwd_after = 1;
    ia.out = m->bufB;
    ia.mode = gbd::ROW_H;
    float t[3];
    const int nv = p.prec == 0 ? 3 : 2;
    for (int v = 0; v < nv && e == cudaSuccess; ++v)
      e = time_variant(st, reps, [&] {
        gbd::launch_row(p.Lx, v, p.prec, fa, m->tw, st);
        enqueue_conv(m, m->S, m->T, st);
        gbd::launch_row(p.Lx, v, p.prec, ia, m->tw, st);
      }, &t[v]);
    if (e == cudaSuccess) {
      int b = best_io;
      for (int v = 0; v < nv; ++v)
        if (t[v] < 0.98f * t[best_io] && t[v] < t[b]) b = v;
      best_io = b;
    }
  }
  gbd::ColArgs ca = col_args(m);
  if (conv_in_one(p)) {
    // one kernel, no variants
  } else if (e == cudaSuccess && p.film) {
    ca.dst = m->S;
    ca.Kf = static_cast<const float4*>(m->K);
    e = pick(1, [&](int v) { gbd::launch_film_conv(v, p.prec, ca, m->tw, st); });
  } else if (e == cudaSuccess) {
    ca.K3 = static_cast<const float2*>(m->K);
    if (p.ny > 1) {
      ca.lines_total = 3LL * p.nz * p.Hx;
      ca.src = m->S;
      ca.dst = m->T;
      e = pick(2, [&](int v) {
        gbd::launch_y_fwd(v, p.prec, ca, m->tw, st);
        gbd::ColArgs cb = ca;
        cb.src = m->T;
        cb.dst = m->S;
        gbd::launch_y_inv(v, p.prec, cb, m->tw, st);
      });
      ca.dst = m->T;
    } else {
      ca.dst = m->S;
    }
    z_strides(p, ca);
    if (e == cudaSuccess) e = pick(3, [&](int v) { gbd::launch_z_conv(v, p.prec, ca, m->tw, st); });
  }
  if (e != cudaSuccess) return cuda_fail(e, "gbd_mesh_autotune");
  apply_tuning(m, std::array<int, 6>{best[0], best[1], best[2], best[3], 0, best_io});
  // padded length: against the same mesh on power-of-two lengths
  int pow2 = 0;
  if (can_pad_pow2(m)) {
    s = pow2_is_faster(m, stream, &pow2);
    if (s != GBD_OK) return s;
  }
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    if (g_tune.find(key) == g_tune.end()) {
      const std::array<int, 6> v = {best[0], best[1], best[2], best[3], pow2, best_io};
      g_tune[key] = v;
      append_tune_file_locked(key, v);
    }
  }
  return pow2 ? move_to_pow2(m, stream) : GBD_OK;
}

// ---- batched meshes: one CUDA graph per run ------------------------------------------------
//
// A batch advances many independent meshes. Each mesh's launch sequence (the same as
// gbd_llg_step's) is a chain on one of up to kBatchBranches branch streams; the chains are
// captured into one CUDA graph behind a fork event and joined back into the caller's stream,
// so the GPU runs kernels of different meshes side by side and the host makes one graph
// launch per run. The instantiated graph is cached with its arguments (state pointers,
// step counts, time steps) and relaunched while they repeat.

struct gbd_batch {
  std::vector<gbd_mesh*> meshes;
  int device = -1;
  cudaStream_t origin = nullptr;  // capture and launch stream (the legacy default stream cannot be captured)
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  std::vector<cudaStream_t> branches;
  cudaEvent_t fork = nullptr;
  std::vector<cudaEvent_t> join;
  std::vector<float*> key_m;
  std::vector<int> key_steps;
  std::vector<double> key_dt;
  std::vector<unsigned> key_version;
  std::vector<unsigned> key_flags;
  // extrapolation history state of each mesh before the captured run (part of the key) and
  // after it (restored on every replay, which advances the history exactly as the capture did)
  std::vector<std::array<double, 3>> key_hist, post_hist;
  cudaGraphExec_t exec = nullptr;
};

namespace {
constexpr int kBatchBranches = 32;

// gbd_llg_step's launch sequence for one mesh on one stream (no timing events).
// gbd_llg_step_ex's launch sequence for one mesh on one stream, without timing events.
void enqueue_llg(gbd_mesh* m, float* mm, int nsteps, double dt, unsigned flags, cudaStream_t st) {
  const int tmp = m->timing;
  m->timing = 0;
  enqueue_llg_ex(m, mm, nsteps, dt, flags, st);
  m->timing = tmp;
}

void destroy_batch(gbd_batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  for (cudaStream_t s : b->branches) cudaStreamDestroy(s);
  for (cudaEvent_t e : b->join) cudaEventDestroy(e);
  if (b->fork) cudaEventDestroy(b->fork);
  if (b->ev_in) cudaEventDestroy(b->ev_in);
  if (b->ev_out) cudaEventDestroy(b->ev_out);
  if (b->origin) cudaStreamDestroy(b->origin);
  delete b;
}
}  // namespace

extern "C" gbd_status gbd_batch_create(gbd_mesh* const* meshes, int count, gbd_batch** out) {
  if (!out) return fail(GBD_EINVAL, "out is NULL");
  *out = nullptr;
  if (!meshes || count < 1) return fail(GBD_EINVAL, "meshes must be a non-empty array");
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  for (int i = 0; i < count; ++i) {
    if (!meshes[i]) return fail(GBD_EINVAL, "meshes[" + std::to_string(i) + "] is NULL");
    if (!meshes[i]->kernel_set) return fail(GBD_ESTATE, "gbd_set_kernel has not been called on meshes[" + std::to_string(i) + "]");
    if (meshes[i]->device != dev) return fail(GBD_EINVAL, "all meshes must live on the current device");
    for (int j = 0; j < i; ++j)
      if (meshes[j] == meshes[i]) return fail(GBD_EINVAL, "a mesh appears twice in the batch");
  }
  gbd_batch* b = new (std::nothrow) gbd_batch();
  if (!b) return fail(GBD_ENOMEM, "host allocation failed");
  b->meshes.assign(meshes, meshes + count);
  b->device = dev;
  const int nb = count < kBatchBranches ? count : kBatchBranches;
  e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->origin, cudaStreamNonBlocking);
  for (int i = 0; i < nb && e == cudaSuccess; ++i) {
    cudaStream_t s;
    cudaEvent_t j;
    e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e != cudaSuccess) break;
    b->branches.push_back(s);
    e = cudaEventCreateWithFlags(&j, cudaEventDisableTiming);
    if (e != cudaSuccess) break;
    b->join.push_back(j);
  }
  if (e != cudaSuccess) {
    destroy_batch(b);
    return cuda_fail(e, "gbd_batch_create");
  }
  *out = b;
  return GBD_OK;
}

static std::array<double, 3> hist_state(const gbd_mesh* m) {
  return {(double)m->hist_head, (double)m->hist_count, m->hist_dt};
}

static void set_hist_state(gbd_mesh* m, const std::array<double, 3>& h) {
  m->hist_head = (int)h[0];
  m->hist_count = (int)h[1];
  m->hist_dt = h[2];
}

extern "C" gbd_status gbd_batch_run_ex(gbd_batch* b, float* const* m, const int* nsteps, const double* dt,
                                       const unsigned* flags, void* stream) {
  if (!b || !m || !nsteps || !dt) return fail(GBD_EINVAL, "NULL argument");
  const int n = (int)b->meshes.size();
  std::vector<unsigned> fl(n, 0u);
  for (int i = 0; i < n; ++i) {
    if (!ptr_ok(m[i])) return fail(GBD_EINVAL, "m[" + std::to_string(i) + "] must be a non-NULL, 4-byte aligned device pointer");
    if (nsteps[i] < 0) return fail(GBD_EINVAL, "nsteps must be >= 0");
    if (!(dt[i] > 0) || !std::isfinite(dt[i])) return fail(GBD_EINVAL, "dt must be finite and > 0");
    if (flags) fl[i] = flags[i];
    if (fl[i] & ~(unsigned)(GBD_STEP_EXTRAP | GBD_STEP_CONTINUE)) return fail(GBD_EINVAL, "unknown flags");
  }
  gbd_status s = check_device(b->meshes[0]);
  if (s != GBD_OK) return s;
  for (int i = 0; i < n; ++i)
    if ((fl[i] & GBD_STEP_EXTRAP) && nsteps[i] > 0) {
      s = ensure_history(b->meshes[i]);
      if (s != GBD_OK) return s;
    }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaStream_t og = b->origin;
  std::vector<unsigned> version(n);
  std::vector<std::array<double, 3>> pre(n);
  for (int i = 0; i < n; ++i) {
    version[i] = b->meshes[i]->version;
    pre[i] = hist_state(b->meshes[i]);
  }
  const bool same = b->exec && b->key_m == std::vector<float*>(m, m + n) &&
                    b->key_steps == std::vector<int>(nsteps, nsteps + n) &&
                    b->key_dt == std::vector<double>(dt, dt + n) && b->key_version == version &&
                    b->key_flags == fl && b->key_hist == pre;
  if (same) {
    for (int i = 0; i < n; ++i) set_hist_state(b->meshes[i], b->post_hist[i]);
  } else {
    if (b->exec) {
      cudaGraphExecDestroy(b->exec);
      b->exec = nullptr;
    }
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(og, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(e, "gbd_batch_run: begin capture");
    cudaEventRecord(b->fork, og);
    const int nb = (int)b->branches.size();
    for (int j = 0; j < nb; ++j) cudaStreamWaitEvent(b->branches[j], b->fork, 0);
    for (int i = 0; i < n; ++i) enqueue_llg(b->meshes[i], m[i], nsteps[i], dt[i], fl[i], b->branches[i % nb]);
    for (int j = 0; j < nb; ++j) {
      cudaEventRecord(b->join[j], b->branches[j]);
      cudaStreamWaitEvent(og, b->join[j], 0);
    }
    e = cudaStreamEndCapture(og, &graph);
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
      b->exec = nullptr;
      cudaGetLastError();
      for (int i = 0; i < n; ++i) set_hist_state(b->meshes[i], pre[i]);
      return cuda_fail(e, "gbd_batch_run: graph capture");
    }
    b->key_m.assign(m, m + n);
    b->key_steps.assign(nsteps, nsteps + n);
    b->key_dt.assign(dt, dt + n);
    b->key_version = version;
    b->key_flags = fl;
    b->key_hist = pre;
    b->post_hist.resize(n);
    for (int i = 0; i < n; ++i) b->post_hist[i] = hist_state(b->meshes[i]);
  }
  // order the graph after the caller's earlier work on `stream`, and later work after it
  cudaEventRecord(b->ev_in, st);
  cudaStreamWaitEvent(og, b->ev_in, 0);
  cudaError_t e = cudaGraphLaunch(b->exec, og);
  if (e != cudaSuccess) return cuda_fail(e, "gbd_batch_run: graph launch");
  cudaEventRecord(b->ev_out, og);
  cudaStreamWaitEvent(st, b->ev_out, 0);
  for (gbd_mesh* mesh : b->meshes) mark_done(mesh, og);
  return after_launch("gbd_batch_run");
}

extern "C" gbd_status gbd_batch_run(gbd_batch* b, float* const* m, const int* nsteps, const double* dt, void* stream) {
  return gbd_batch_run_ex(b, m, nsteps, dt, nullptr, stream);
}

extern "C" gbd_status gbd_batch_destroy(gbd_batch* b) {
  if (!b) return GBD_OK;
  // the batch's last graph launch must have finished before its executable graph goes; the
  // rest of the device keeps running
  if (b->ev_out) cudaEventSynchronize(b->ev_out);
  destroy_batch(b);
  return GBD_OK;
}
