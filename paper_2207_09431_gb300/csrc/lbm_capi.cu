// Host side of the C ABI declared in include/lbm.h: parameter validation,
// arena carving, initial conditions (Sec. 4.2, Eq. 42), the step loop, field
// readback, observables post-processing (Sec. 4.1-4.2) and checkpoints.
#include <cuda_runtime.h>
#include <unistd.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "lbm.h"
#include "lbm_kernels.h"

#include "lbm_internal.h"

// Writes a byte into every page of the caller's array that the copies below are to fill.  A page
// of a new array is mapped when something first writes to it, and where that is the GPU's copy
// (through the address translation it shares with a Grace host) the faults cost it far more than
// they cost the CPU, and at times stall it.  lbm_get_field into new memory without and with this
// (GB300): the first g of 128 x 128 1.2 to 3.8 against 0.13 ms, g of 1024 x 1024 5.6 (36 in some
// processes) against 3.4 ms, of 1500 x 1500 7.4 (23) against 7.1 ms; into memory in use no difference.
static void map_pages(double *dst, size_t values) {
  static const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  volatile char *p = reinterpret_cast<volatile char *>(dst), *const end = p + values * sizeof(double);
  while (p < end) {
    *p = 0;
    p += page - reinterpret_cast<uintptr_t>(p) % page;
  }
}

// Small fields are converted on the host from the FP32 planes as they are stored: planes of up to
// 8192 floats together, populations of up to 2560 nodes in planes of up to 4096.  Above, the loop costs more than a launch and twice the
// bytes; below, us per lbm_get_field on the host and on the device (GB300, Grace host): tau 64 x 40
// 15.4 and 18.6, 64 x 128 16.8 and 19.1, 100 x 200 18.2 and 19.4 but u_x 34.8 and 33.0; g 16 x 16 17
// and 43, 64 x 40 43 and 45, 60 x 60 51 and 46.
constexpr size_t kHostPlanes = 8192, kHostPopulations = 2560;
static cudaError_t staged_on_host(lbm_handle *h, const float *src, size_t floats) {
  h->stage.resize(floats);
  const cudaError_t e = cudaMemcpyAsync(h->stage.data(), src, floats * sizeof(float), cudaMemcpyDeviceToHost, h->stream);
  return e == cudaSuccess ? cudaStreamSynchronize(h->stream) : e;
}

// Fields go to the host as dense doubles, converted on the device in the spare
// population buffer (free between steps; four dense planes of doubles fit) and copied
// straight into the caller's array.
static cudaError_t download_planes(lbm_handle *h, const float *src, double *dst, int nplanes, int kind = lbm::kPlane) {
  const size_t N = (size_t)h->prm.nx * h->prm.ny;
  if (kind == lbm::kPlane && nplanes * h->plane_floats() <= kHostPlanes) {
    cudaError_t e = staged_on_host(h, src, nplanes * h->plane_floats());
    for (int q = 0; q < nplanes && e == cudaSuccess; ++q)
      for (int y = 0; y < h->prm.ny; ++y) {
        const float *row = h->stage.data() + q * h->plane_floats() + (size_t)y * h->dp.pitch;
        std::copy(row, row + h->prm.nx, dst + (q * (size_t)h->prm.ny + y) * h->prm.nx);
      }
    return e;
  }
  double *dense = reinterpret_cast<double *>(h->g[1 - h->cur]);
  cudaError_t e = lbm::launch_planes_to_f64(h->dp, h->prm.rho, src, kind, nplanes, dense, h->stream);
  map_pages(dst, nplanes * N);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(dst, dense, nplanes * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  return e;
}

// The nq planes of a device population array, plane after plane.
static cudaError_t download_pops(lbm_handle *h, const float *src, double *dst, int nq, bool g16) {
  const size_t N = (size_t)h->prm.nx * h->prm.ny;
  if (!g16 && N <= kHostPopulations && h->plane_floats() <= 4096) {
    cudaError_t e = staged_on_host(h, src, nq * h->plane_floats());
    for (int q = 0; q < nq && e == cudaSuccess; ++q)
      for (int y = 0; y < h->prm.ny; ++y)
        for (int x = 0; x < h->prm.nx; ++x)
          *dst++ = h->stage[lbm::pop_index((long long)y * h->dp.pitch + x, q, nq)];
    return e;
  }
  double *dense = reinterpret_cast<double *>(h->g[1 - h->cur]);
  cudaError_t e = cudaSuccess;
  for (int q0 = 0; q0 < nq && e == cudaSuccess; q0 += 4) {
    const int q1 = std::min(nq, q0 + 4);
    e = lbm::launch_pops_to_f64(h->dp, src, q0, q1, nq, g16, dense, h->stream);
    map_pages(dst + q0 * N, (q1 - q0) * N);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(dst + q0 * N, dense, (q1 - q0) * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  return e;
}

extern "C" {

int lbm_version(void) { return kVersion; }

size_t lbm_required_bytes(const lbm_params *p) {
  if (validate(p)) return 0;
  return layout_of(*p).total;
}

// The copy stream and its events for the overlapped upload of lbm_set_fields, on handles with C of
// 32 MB and more and chunks of at least 16 rows (the equilibria read two rows beyond their own).  A
// copy from pageable memory returns when it is done, and 4 to 16 small copies, events and launches
// cost more than they hide in smaller fields.  Whole and in chunks, us (GB300): C pageable 200 x 400
// 30 and 72, 2048 x 4096 547 and 601; C, p and u pageable 200 x 400 75 and 203; C page-locked 200 x
// 400 22 and 35, 1024 x 2048 135 and 133, 2048 x 4096 467 and 419.  Created with the handle: a
// process's first one takes 0.2 ms, half of such an upload.
static void create_upload_stream(lbm_handle *h) {
  const size_t bytes = (size_t)(h->prm.ncomp - 1) * h->prm.nx * h->prm.ny * sizeof(double);
  if (bytes < ((size_t)32 << 20) || h->prm.ny < 16 * lbm_handle::kUploadChunks) return;
  bool ok = true;
  for (auto &ev : h->upload_ev) ok = ok && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) == cudaSuccess;
  if (!ok || cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking) != cudaSuccess) {
    h->copy_stream = nullptr;  // fields go up whole
    cudaGetLastError();
  }
}

lbm_status lbm_create(const lbm_params *p, void *dev_arena, size_t arena_bytes, void *cuda_stream,
                      lbm_handle **out) {
  if (!out) return LBM_E_INVAL;
  *out = nullptr;
  if (validate(p)) return LBM_E_INVAL;
  if (!dev_arena || ((uintptr_t)dev_arena % kAlign) != 0) return LBM_E_INVAL;
  Layout L = layout_of(*p);
  if (arena_bytes < L.total) return LBM_E_NOMEM;
  lbm_handle *h = new (std::nothrow) lbm_handle();
  if (!h) return LBM_E_NOMEM;
  h->prm = *p;
  h->dp = dev_params(*p);
  h->L = L;
  h->stream = (cudaStream_t)cuda_stream;
  h->arena = (char *)dev_arena;
  const size_t pf = L.plane_bytes / sizeof(float);
  const int nh = p->ncomp - 1;
  for (int b = 0; b < 2; ++b) {
    h->g[b] = (float *)(h->arena + L.g) + (size_t)b * 9 * pf;
    h->h[b] = (float *)(h->arena + L.h) + (size_t)b * (p->collapse_h ? 1 : 9) * nh * pf;
    h->tau[b] = (float *)(h->arena + L.tau) + (size_t)b * pf;
  }
  h->C = (float *)(h->arena + L.C);
  h->mu = (float *)(h->arena + L.mu);
  h->p = (float *)(h->arena + L.p);
  h->ux = (float *)(h->arena + L.ux);
  h->uy = (float *)(h->arena + L.uy);
  h->shear = (float *)(h->arena + L.shear);
  h->SV = (float *)(h->arena + L.SV);
  h->acc = (double *)(h->arena + L.small);
  h->ext = (int *)(h->acc + 16);
  h->err = (unsigned *)(h->ext + 8);
  // plane stride used by the kernels must match the arena planes
  h->dp.plane = (long long)pf;
  h->cur = 0;
  h->variant = h->fused() ? lbm::fused_default_variant(h->dp) : 0;
  h->initialized = false;
  h->step = 0;
  h->have_prev = false;
  cudaError_t e = cudaMemsetAsync(h->arena, 0, L.total, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    delete h;
    return LBM_E_CUDA;
  }
  create_upload_stream(h);
  *out = h;
  return LBM_OK;
}

// Whether lbm_set_fields overlaps the upload with the initial equilibria: all fields in page-locked
// memory, a handle that has the streams for it, and a stream that is not being captured.
static bool upload_overlappable(lbm_handle *h, const double *C, const double *const f[3]) {
  if (!h->copy_stream) return false;
  for (const double *p : {C, f[0], f[1], f[2]}) {
    cudaPointerAttributes a{};
    if (!p) continue;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
      cudaGetLastError();  // not CUDA's memory: nothing else asks for this error
      return false;
    }
    if (a.type != cudaMemoryTypeHost) return false;
  }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  return cudaStreamIsCapturing(h->stream, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone;
}

// FP64 fields on the device, dense: C in the spare population buffer g[1] (free
// until the first step), p, ux and uy in the scratch planes mu .. uy, which lie next
// to each other (six FP32 planes hold three of doubles).
struct StagedFields {
  double *C, *f[3];
  explicit StagedFields(const lbm_handle *h) : C(reinterpret_cast<double *>(h->g[1])) {
    for (int q = 0; q < 3; ++q) f[q] = reinterpret_cast<double *>(reinterpret_cast<char *>(h->mu) + 2 * q * h->L.plane_bytes);
  }
};

// Equilibria of rows [y0, y1) into buffer 0 from the staged fields.
static cudaError_t init_rows(lbm_handle *h, const StagedFields &st, const bool given[3], int y0, int y1) {
  return lbm::launch_init_rows(h->dp, st.C, given[0] ? st.f[0] : nullptr, given[1] ? st.f[1] : nullptr,
                               given[2] ? st.f[2] : nullptr, h->g[0], h->h[0], h->tau[0], y0, y1, h->stream);
}

// The fields go up in row chunks on the copy stream; the handle's stream computes the
// equilibria of the rows whose two-row neighbourhood has arrived (those of the first
// chunk last under periodic y, where they read the last rows).  Same node values as
// one upload.
static cudaError_t upload_and_init_overlapped(lbm_handle *h, const StagedFields &st, const double *C,
                                              const double *const f[3], const bool given[3]) {
  constexpr int n = lbm_handle::kUploadChunks;
  const int nh = h->prm.ncomp - 1, nx = h->prm.nx, ny = h->prm.ny, rows = (ny + n - 1) / n;
  const bool per = h->prm.periodic_y != 0;
  // the staging buffers are free once the work before on the stream is done
  cudaError_t e = cudaEventRecord(h->upload_ev[n], h->stream);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(h->copy_stream, h->upload_ev[n], 0);
  for (int c = 0; c < n && e == cudaSuccess; ++c) {
    const int y0 = c * rows, y1 = std::min(ny, y0 + rows);
    const size_t bytes = (size_t)(y1 - y0) * nx * sizeof(double);
    for (int q = 0; q < nh && e == cudaSuccess; ++q) {
      const size_t off = ((size_t)q * ny + y0) * nx;
      e = cudaMemcpyAsync(st.C + off, C + off, bytes, cudaMemcpyHostToDevice, h->copy_stream);
    }
    for (int q = 0; q < 3 && e == cudaSuccess; ++q)
      if (given[q])
        e = cudaMemcpyAsync(st.f[q] + (size_t)y0 * nx, f[q] + (size_t)y0 * nx, bytes, cudaMemcpyHostToDevice,
                            h->copy_stream);
    if (e == cudaSuccess) e = cudaEventRecord(h->upload_ev[c], h->copy_stream);
  }
  for (int c = 0; c < n && e == cudaSuccess; ++c) {
    e = cudaStreamWaitEvent(h->stream, h->upload_ev[c], 0);
    if (e == cudaSuccess && c >= 1 && (c >= 2 || !per)) e = init_rows(h, st, given, (c - 1) * rows, c * rows);
  }
  if (e == cudaSuccess) e = init_rows(h, st, given, (n - 1) * rows, ny);
  if (e == cudaSuccess && per) e = init_rows(h, st, given, 0, rows);
  return e;
}

// The state that the staged fields (or those still to be uploaded) have become.
static lbm_status fields_set(lbm_handle *h, cudaError_t e) {
  const cudaError_t done = cudaStreamSynchronize(h->stream);
  if (e == cudaSuccess) e = done;
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_set_fields");
  h->cur = 0;
  h->initialized = true;
  h->step = 0;
  h->have_prev = false;
  h->last_error.clear();
  return LBM_OK;
}

lbm_status lbm_set_fields(lbm_handle *h, const double *C, const double *p, const double *ux, const double *uy) {
  if (!h) return LBM_E_INVAL;
  if (!C) return h->fail(LBM_E_INVAL, "C is NULL");
  const int nh = h->prm.ncomp - 1;
  const StagedFields st(h);
  const double *const f[3] = {p, ux, uy};
  const bool given[3] = {p != nullptr, ux != nullptr, uy != nullptr};
  if (upload_overlappable(h, C, f)) return fields_set(h, upload_and_init_overlapped(h, st, C, f, given));
  const size_t bytes = (size_t)h->prm.nx * h->prm.ny * sizeof(double);
  cudaError_t e = cudaMemcpyAsync(st.C, C, nh * bytes, cudaMemcpyHostToDevice, h->stream);
  for (int q = 0; q < 3 && e == cudaSuccess; ++q)
    if (given[q]) e = cudaMemcpyAsync(st.f[q], f[q], bytes, cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess) e = init_rows(h, st, given, 0, h->prm.ny);
  return fields_set(h, e);
}

lbm_status lbm_init_bubbles(lbm_handle *h, const lbm_bubble *bubbles, int nb, unsigned long long seed,
                            double noise_amp) {
  if (!h) return LBM_E_INVAL;
  if (nb < 0 || (nb > 0 && !bubbles)) return h->fail(LBM_E_INVAL, "bad bubble list");
  const int nh = h->prm.ncomp - 1;
  bool used[2] = {false, false};
  for (int b = 0; b < nb; ++b) {
    const int c = bubbles[b].comp;
    if (c < 2 || c > 3 || (nh == 1 && c != 3)) return h->fail(LBM_E_INVAL, "disc component must be 3 (or 2 with ncomp 3)");
    used[c - 2] = true;
  }
  const StagedFields st(h);
  cudaError_t e = cudaSuccess;
  for (int b0 = 0; (b0 < nb || b0 == 0) && e == cudaSuccess; b0 += lbm::kDiscs) {
    lbm::DiscGroup d{};
    d.count = std::min(nb - b0, lbm::kDiscs);
    std::copy(bubbles + b0, bubbles + b0 + d.count, d.disc);
    d.first = b0 == 0;
    d.last = b0 + lbm::kDiscs >= nb;
    d.seed = seed;
    for (int c = 0; c < 2; ++c) d.noise[c] = used[c] ? noise_amp : 0.0;
    e = lbm::launch_discs(h->dp, h->prm.xi, d, st.C, h->stream);
  }
  const bool given[3] = {false, false, false};
  if (e == cudaSuccess) e = init_rows(h, st, given, 0, h->prm.ny);
  return fields_set(h, e);
}

lbm_status lbm_step(lbm_handle *h, long long nsteps) {
  if (!h) return LBM_E_INVAL;
  if (!h->initialized) return h->fail(LBM_E_STATE, "lbm_step before initial fields");
  if (nsteps < 0) return h->fail(LBM_E_INVAL, "nsteps < 0");
  cudaError_t e = cudaMemsetAsync(h->err, 0, sizeof(unsigned), h->stream);
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_step memset");
  long long t = 0;
  // Runs of 16 and of 4 steps are replayed from captured graphs (on a
  // created stream; capture needs one).  The last step writes the diagnostics and is
  // launched directly; a first run with a new configuration is too, so that
  // its kernels are configured outside the capture.  A graph starts from one of the two
  // buffers, and a call that comes with the state in the other one takes a direct step
  // first: with a graph per buffer, captured where the first direct step had led, a
  // program of equal even runs captured anew on every call (64 steps of 64 x 128:
  // 333 -> 279 us, GB300).  A launch from the host takes some 6 us, longer than a step of a
  // lattice of up to about 150 x 300 nodes (3.6 to 6.4 us), whose last 15 steps therefore go
  // in fours (279 -> 254 us).  With larger ones the host is ahead of the device, and the fours
  // save the wider gaps between direct launches, some 1.8 us each (64 steps of three
  // components 256 x 256 604 -> 585 us); they are captured while the device is busy with the sixteens.
  // Without sixteens before them a capture costs as much as the launches of two runs, so a handle
  // captures the fours on its second missed run (first call of a new handle of 64 x 128, 5 and 8 steps:
  // 64 and 77 us with a capture, 52 and 69 without).
  const bool capturable = h->stream != nullptr && h->stream != cudaStreamLegacy && h->stream != cudaStreamPerThread;
  const bool small = (long long)h->prm.nx * h->prm.ny <= lbm_handle::kSmallNodes;
  for (auto &sg : h->graphs) {
    const bool captured = sg.exec && sg.variant == h->variant;
    if (!capturable || nsteps - 1 - t < sg.steps) continue;
    if (!captured && sg.steps < lbm_handle::kStepGraph && t == 0) {
      if (!small) continue;
      sg.missed += (int)std::min<long long>((nsteps - 1) / sg.steps, 2);
      if (sg.missed < 2) continue;
    }
    if (captured ? sg.from != h->cur : t == 0) {
      h->launch_step(false, nullptr);
      ++t;
    }
    if (!captured) {
      const int c = h->cur;
      if (sg.exec) cudaGraphExecDestroy(sg.exec);
      sg.exec = nullptr;
      cudaGraph_t g = nullptr;
      e = cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal);
      for (int k = 0; k < sg.steps && e == cudaSuccess; ++k) {
        h->launch_step(false, nullptr);
        e = cudaGetLastError();
      }
      cudaError_t ec = cudaStreamEndCapture(h->stream, &g);
      if (e == cudaSuccess) e = ec;
      if (e == cudaSuccess) e = cudaGraphInstantiate(&sg.exec, g, 0);
      if (g) cudaGraphDestroy(g);
      h->cur = c;  // an even number of captured steps returns to the same buffer
      if (e != cudaSuccess) {
        sg.exec = nullptr;
        return h->cuda_fail(e, "lbm_step graph capture");
      }
      sg.variant = h->variant;
      sg.from = c;
      sg.missed = 0;
    }
    for (; nsteps - 1 - t >= sg.steps && e == cudaSuccess; t += sg.steps) e = cudaGraphLaunch(sg.exec, h->stream);
    if (e != cudaSuccess) return h->cuda_fail(e, "lbm_step graph launch");
  }
  for (; t < nsteps; ++t) h->launch_step(t == nsteps - 1, nullptr);
  e = cudaGetLastError();
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_step launch");
  unsigned flag = 0;
  e = cudaMemcpyAsync(&flag, h->err, sizeof(unsigned), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_step");
  h->step += nsteps;
  if (flag) return h->fail(LBM_E_DIVERGED, "non-finite rho, p, u or tau during lbm_step");
  return LBM_OK;
}

// FP32 populations of the current state: the state itself, or (FP16 storage)
// their decoded copy in the spare buffer.
static const float *fp32_populations(lbm_handle *h, cudaError_t *e) {
  if (!h->dp.g16) return h->g[h->cur];
  *e = lbm::launch_g16_decode(h->dp, h->g[h->cur], h->g[1 - h->cur], h->stream);
  return h->g[1 - h->cur];
}

static lbm_status compute_macros(lbm_handle *h) {
  lbm::StepBuffers B = h->buffers(h->cur);
  cudaError_t e = cudaSuccess;
  B.g_in = fp32_populations(h, &e);
  if (e != cudaSuccess) return h->cuda_fail(e, "FP16 decode");
  lbm::launch_macros(h->dp, B, h->stream);
  e = cudaGetLastError();
  if (e != cudaSuccess) return h->cuda_fail(e, "macro kernels");
  return LBM_OK;
}

lbm_status lbm_postprocess(const lbm_params *p, const double raw[15], lbm_obs *o) {
  if (!p || !raw || !o) return LBM_E_INVAL;
  std::memset(o, 0, sizeof(*o));
  for (int i = 0; i < 15; ++i) o->raw[i] = raw[i];
  for (int i = 0; i < 3; ++i) {
    o->mass[i] = raw[i];
    o->mass_thr[i] = raw[3 + i];
  }
  const int gc = (p->gas_comp == 2 || p->gas_comp == 3) ? p->gas_comp : 3;
  const double rho_l = p->rho[0], rho_g = p->rho[gc - 1];
  const double sigma = gc == 3 ? p->sigma13 : p->sigma12;
  const double g = p->gravity;
  const double n = p->powerlaw ? p->pl_n : 1.0;
  const double k = p->powerlaw ? p->pl_k : rho_l * p->tau[0] / 3.0;
  const double A = raw[6];
  const double nan = std::nan("");
  o->area = A;
  if (A > 0) {
    o->centroid[0] = raw[7] / A;  // Eq. 44
    o->centroid[1] = raw[8] / A;
    o->velocity[0] = raw[9] / A;  // Eq. 43
    o->velocity[1] = raw[10] / A;
  } else {
    o->centroid[0] = o->centroid[1] = o->velocity[0] = o->velocity[1] = nan;
  }
  const double U = o->velocity[1];
  o->rise_velocity = U;
  const double d = A > 0 ? 2.0 * std::sqrt(A / M_PI) : nan;  // area-equivalent diameter
  o->d_eq = d;
  o->aspect_E = raw[11] >= 0 ? (raw[14] - raw[13] + 1.0) / (raw[12] - raw[11] + 1.0) : nan;
  o->drag_coefficient = (A > 0 && U != 0 && g != 0) ? 4.0 * d * g * (rho_l - rho_g) / (3.0 * rho_l * U * U) : nan;
  o->Re = A > 0 ? rho_l * std::pow(std::fabs(U), 2.0 - n) * std::pow(d, n) / k : nan;  // Eq. 38
  o->Eo = A > 0 ? (rho_l - rho_g) * g * d * d / sigma : nan;                             // Eq. 40
  o->Mo = (A > 0 && U != 0)
              ? g * (rho_l - rho_g) / (rho_l * rho_l * sigma * sigma * sigma) *
                    std::pow(k * std::pow(std::fabs(U) / d, n - 1.0), 4.0)
              : nan;  // Eq. 39
  return LBM_OK;
}

lbm_status lbm_observables(lbm_handle *h, lbm_obs *out) {
  if (!h || !out) return LBM_E_INVAL;
  if (!h->initialized) return h->fail(LBM_E_STATE, "observables before initial fields");
  // straight from the state, in its stored form; the sums and the extents lie
  // next to each other (one clear, one copy back)
  struct {
    double acc[16];
    int ext[8];
  } sums;
  static_assert(sizeof(sums) == 16 * sizeof(double) + 8 * sizeof(int), "as the arena holds them");
  cudaError_t e = cudaMemsetAsync(h->acc, 0, sizeof(sums), h->stream);
  if (e == cudaSuccess)
    e = lbm::launch_observe(h->dp, h->fused_buffers(h->cur, false), h->prm.gas_comp, h->acc, h->ext, h->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&sums, h->acc, sizeof(sums), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return h->cuda_fail(e, "observables");
  double raw[15];
  for (int i = 0; i < 11; ++i) raw[i] = sums.acc[i];
  const bool any = sums.ext[0] > 0;
  raw[11] = any ? h->prm.nx - sums.ext[0] : -1.0;
  raw[12] = any ? sums.ext[1] - 1 : -1.0;
  raw[13] = any ? h->prm.ny - sums.ext[2] : -1.0;
  raw[14] = any ? sums.ext[3] - 1 : -1.0;
  lbm_postprocess(&h->prm, raw, out);
  out->step = h->step;
  // centroid y at the first call plus the trapezoidal integral of the rise velocity
  if (!h->have_prev) {
    h->y_int = out->centroid[1];
    h->have_prev = true;
  } else {
    h->y_int += 0.5 * (h->prev_v + out->rise_velocity) * (double)(h->step - h->prev_step);
  }
  h->prev_step = h->step;
  h->prev_v = out->rise_velocity;
  out->y_integrated = h->y_int;
  return LBM_OK;
}

lbm_status lbm_get_field(lbm_handle *h, int id, double *out, size_t n) {
  if (!h || !out) return LBM_E_INVAL;
  if (!h->initialized) return h->fail(LBM_E_STATE, "get_field before initial fields");
  const int nh = h->prm.ncomp - 1;
  const size_t N = (size_t)h->prm.nx * h->prm.ny;
  size_t need;
  switch (id) {
    case LBM_FIELD_G: need = 9 * N; break;
    case LBM_FIELD_H: need = (size_t)9 * nh * N; break;
    case LBM_FIELD_SV: need = (size_t)nh * N; break;
    case LBM_FIELD_C1: case LBM_FIELD_C2: case LBM_FIELD_C3: case LBM_FIELD_RHO: case LBM_FIELD_P:
    case LBM_FIELD_UX: case LBM_FIELD_UY: case LBM_FIELD_TAU: case LBM_FIELD_MU1: case LBM_FIELD_MU2:
    case LBM_FIELD_MU3: case LBM_FIELD_SHEAR: need = N; break;
    default: return h->fail(LBM_E_INVAL, "unknown field id");
  }
  if (n < need) return h->fail(LBM_E_INVAL, "output buffer too small");
  const size_t pf = h->L.plane_bytes / sizeof(float);
  // C_i (the state itself in the C forms)
  auto c_planes = [&]() -> const float * {
    const lbm::StepBuffers B = h->buffers(h->cur);
    if (B.h_in) lbm::launch_moments(h->dp, B.h_in, B.C, h->stream);
    return B.C;
  };
  cudaError_t e = cudaSuccess;
  switch (id) {
    case LBM_FIELD_G: e = download_pops(h, h->g[h->cur], out, 9, h->dp.g16); break;
    case LBM_FIELD_H:
      if (h->prm.collapse_h) return h->fail(LBM_E_STATE, "the collapsed state form stores no h populations");
      e = download_pops(h, h->h[h->cur], out, 9 * nh, false);
      break;
    case LBM_FIELD_TAU: e = download_planes(h, h->tau[h->cur], out, 1); break;
    case LBM_FIELD_SHEAR: e = download_planes(h, h->shear, out, 1); break;
    case LBM_FIELD_SV: e = download_planes(h, h->SV, out, nh); break;
    case LBM_FIELD_C1: e = download_planes(h, c_planes(), out, 1); break;
    case LBM_FIELD_C2:
      if (nh == 2) e = download_planes(h, c_planes() + pf, out, 1);
      else std::memset(out, 0, N * sizeof(double));
      break;
    case LBM_FIELD_C3: e = download_planes(h, c_planes(), out, 1, lbm::kThird); break;
    case LBM_FIELD_RHO: e = download_planes(h, c_planes(), out, 1, lbm::kDensity); break;
    default: {
      const lbm_status st = compute_macros(h);
      if (st != LBM_OK) return st;
      const float *src = id == LBM_FIELD_P    ? h->p
                         : id == LBM_FIELD_UX ? h->ux
                         : id == LBM_FIELD_UY ? h->uy
                                              : h->mu + (size_t)(id - LBM_FIELD_MU1) * pf;
      e = download_planes(h, src, out, 1);
    }
  }
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_get_field");
  return LBM_OK;
}

lbm_status lbm_save(lbm_handle *h, const char *path) {
  if (!h || !path) return LBM_E_INVAL;
  if (!h->initialized) return h->fail(LBM_E_STATE, "save before initial fields");
  const int nh = h->prm.ncomp - 1;
  const size_t pf = h->L.plane_bytes / sizeof(float);
  const int hp = (h->prm.collapse_h ? 1 : 9) * nh;
  const int nplanes = 9 + hp + 1;
  std::vector<float> buf((size_t)nplanes * pf);
  cudaError_t e = cudaMemcpyAsync(buf.data(), h->g[h->cur], 9 * pf * sizeof(float), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(buf.data() + 9 * pf, h->h[h->cur], hp * pf * sizeof(float), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(buf.data() + (size_t)(9 + hp) * pf, h->tau[h->cur], pf * sizeof(float),
                        cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_save");
  FILE *f = std::fopen(path, "wb");
  if (!f) return h->fail(LBM_E_IO, std::string("cannot open ") + path);
  long long hdr[2] = {h->step, (long long)buf.size()};
  bool ok = std::fwrite(kMagic, 1, 8, f) == 8 && std::fwrite(&h->prm, sizeof(lbm_params), 1, f) == 1 &&
            std::fwrite(hdr, sizeof(hdr), 1, f) == 1 &&
            std::fwrite(buf.data(), sizeof(float), buf.size(), f) == buf.size();
  ok = (std::fclose(f) == 0) && ok;
  if (!ok) return h->fail(LBM_E_IO, "short write");
  return LBM_OK;
}

lbm_status lbm_load(lbm_handle *h, const char *path) {
  if (!h || !path) return LBM_E_INVAL;
  FILE *f = std::fopen(path, "rb");
  if (!f) return h->fail(LBM_E_IO, std::string("cannot open ") + path);
  char magic[8];
  lbm_params prm;
  long long hdr[2];
  const int nh = h->prm.ncomp - 1;
  const size_t pf = h->L.plane_bytes / sizeof(float);
  const int hp = (h->prm.collapse_h ? 1 : 9) * nh;
  const size_t count = (size_t)(9 + hp + 1) * pf;
  bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, kMagic, 8) == 0 &&
            std::fread(&prm, sizeof(prm), 1, f) == 1 && std::fread(hdr, sizeof(hdr), 1, f) == 1;
  if (ok && (std::memcmp(&prm, &h->prm, sizeof(prm)) != 0 || hdr[1] != (long long)count)) {
    std::fclose(f);
    return h->fail(LBM_E_INVAL, "checkpoint parameters differ from the handle's");
  }
  std::vector<float> buf(count);
  ok = ok && std::fread(buf.data(), sizeof(float), count, f) == count;
  std::fclose(f);
  if (!ok) return h->fail(LBM_E_IO, "truncated or foreign checkpoint");
  cudaError_t e = cudaMemcpyAsync(h->g[0], buf.data(), 9 * pf * sizeof(float), cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->h[0], buf.data() + 9 * pf, hp * pf * sizeof(float), cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h->tau[0], buf.data() + (size_t)(9 + hp) * pf, pf * sizeof(float),
                        cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_load");
  h->cur = 0;
  h->step = hdr[0];
  h->initialized = true;
  h->have_prev = false;
  return LBM_OK;
}

int lbm_kernels_per_step(const lbm_handle *h) { return h ? h->kernels_per_step() : 0; }

const char *lbm_kernel_name(const lbm_handle *h, int i) {
  static const char *open_ends[lbm::kSplitKernels] = {"k_fields_step", "k_collide_step"};
  static const char *periodic_x[lbm::kSplitKernels] = {"k_fields_step", "k_collide_push"};
  if (!h || i < 0 || i >= h->kernels_per_step()) return "";
  if (!h->fused()) return h->dp.open_x ? open_ends[i] : periodic_x[i];
  lbm_handle *m = const_cast<lbm_handle *>(h);
  const bool sweep = h->variant < lbm::sweep_variant_count(h->dp);
  m->kname = std::string(sweep ? "k_step_sweep[" : "k_step_fused[") + lbm::fused_variant_name(h->dp, h->variant) + "]";
  return m->kname.c_str();
}

int lbm_kernel_config_count(const lbm_handle *h) {
  if (!h) return 0;
  return h->fused() ? lbm::fused_variant_count(h->dp) : 1;
}

lbm_status lbm_set_kernel_config(lbm_handle *h, int config) {
  if (!h) return LBM_E_INVAL;
  if (config < 0 || config >= lbm_kernel_config_count(h)) return h->fail(LBM_E_INVAL, "no such kernel configuration");
  h->variant = h->fused() ? config : 0;
  return LBM_OK;
}

lbm_status lbm_autotune(lbm_handle *h, int reps, int *chosen) {
  if (!h || reps < 1) return LBM_E_INVAL;
  if (!h->initialized) return h->fail(LBM_E_STATE, "autotune before initial fields");
  if (!h->fused()) {
    if (chosen) *chosen = 0;
    return LBM_OK;
  }
  const int nv = lbm::fused_variant_count(h->dp);
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return h->fail(LBM_E_CUDA, "cudaEventCreate");
  // every candidate runs from the current state into the spare buffer; the
  // state itself is not advanced
  const lbm::FusedBuffers B = h->fused_buffers(h->cur, false);
  int best = -1;
  float best_ms = 0.f;
  cudaError_t err = cudaSuccess;
  for (int v = 0; v < nv && err == cudaSuccess; ++v) {
    if (!lbm::fused_variant_timed(h->dp, v)) continue;
    err = lbm::launch_fused_step(h->dp, B, h->stream, v);  // warm-up and attribute set-up
    if (err != cudaSuccess) break;
    cudaEventRecord(e0, h->stream);
    for (int r = 0; r < reps; ++r) lbm::launch_fused_step(h->dp, B, h->stream, v);
    cudaEventRecord(e1, h->stream);
    err = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
    if (err == cudaSuccess && (best < 0 || ms < best_ms)) {
      best = v;
      best_ms = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (err != cudaSuccess) return h->cuda_fail(err, "lbm_autotune");
  h->variant = best;
  if (chosen) *chosen = best;
  return LBM_OK;
}

lbm_status lbm_profile_step(lbm_handle *h, long long nsteps, double *ms_per_kernel, int nkernels) {
  if (!h || !ms_per_kernel || nsteps < 1) return LBM_E_INVAL;
  if (!h->initialized) return h->fail(LBM_E_STATE, "profile before initial fields");
  const int K = h->kernels_per_step();
  if (nkernels < K) return h->fail(LBM_E_INVAL, "ms_per_kernel too small");
  std::vector<cudaEvent_t> ev((size_t)(K + 1) * nsteps);
  for (auto &e : ev)
    if (cudaEventCreate(&e) != cudaSuccess) return h->fail(LBM_E_CUDA, "cudaEventCreate");
  for (long long t = 0; t < nsteps; ++t) h->launch_step(false, ev.data() + t * (K + 1));
  cudaError_t e = cudaStreamSynchronize(h->stream);
  for (int i = 0; i < K; ++i) ms_per_kernel[i] = 0.0;
  for (long long t = 0; t < nsteps && e == cudaSuccess; ++t)
    for (int i = 0; i < K; ++i) {
      float ms = 0.f;
      e = cudaEventElapsedTime(&ms, ev[t * (K + 1) + i], ev[t * (K + 1) + i + 1]);
      ms_per_kernel[i] += ms / (double)nsteps;
    }
  for (auto &x : ev) cudaEventDestroy(x);
  if (e != cudaSuccess) return h->cuda_fail(e, "lbm_profile_step");
  h->step += nsteps;
  return LBM_OK;
}

void lbm_destroy(lbm_handle *h) { delete h; }

const char *lbm_last_error(const lbm_handle *h) { return h ? h->last_error.c_str() : "NULL handle"; }

}  // extern "C"
