// Anisotropic acoustic (TTI) propagation for sm_103a.
//
// Sec. IV-B ("Anisotropic acoustic") and App. A (Eq. rot): two scalar fields
// p, q coupled through a rotated anisotropic Laplacian,
//     m p_tt + eta p_t = (1+2 eps) H_0 p + sqrt(1+2 delta) H_z q + s,
//     m q_tt + eta q_t = sqrt(1+2 delta) H_0 p + H_z q + s,
// H_z u = sum_ab n_a n_b D_ab u along the symmetry axis
// n = (sin t cos p, sin t sin p, cos t) (t the tilt, p the azimuth, per cell)
// and H_0 = Laplacian - H_z (the xbar and ybar directions of Eq. rot), D_aa
// the centred order-2R second-derivative weights and D_ab (a != b) the product
// of centred order-2R first-derivative weights along a and b: at space order
// 16 the 769-point stencil of the paper's TTI figure (the 49-point star and
// the 16 x 16 squares of the xy, xz and yz planes through the point).  Time
// stepping, damping layer (strength from the fastest speed v sqrt(1+2 eps)),
// zero ghost, source scaling and trilinear points as in the isotropic path;
// the source enters both fields, receivers interpolate p.
//
// Step kernel (2.5D, one point per thread, a CTA owning a 32-wide xy tile and
// a run of z planes; k_tti_q, fd_tti_q.cuh): p and q are stored interleaved,
// one float2 per cell, and run through the stencil as packed pairs.  Each
// plane enters once, by TMA, with an R-wide halo; its in-plane second
// derivatives and its first x and y differences are formed then, and every z
// sum (D_zz, D_xz, D_yz) runs over per-thread register queues, so shared
// memory holds only the entering plane, one plane of first y differences and
// the update's per-point tiles.  The model enters through six per-cell fields
// (dt^2 v^2 / h^2, 1 + 2 eps, sqrt(1 + 2 delta) and the axis n), computed
// once per model in double precision.  fd_tti_set_state and fd_tti_get_state
// convert between the caller's separate p and q arrays and the pairs.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "../../include/fd.h"
#include "fd_aux.h"
#include "fd_internal.h"
#include "fd_runtime.h"
#include "fd_tti_q.cuh"

namespace fd {
void fd_weights(int R, double* c);
double cfl_limit(const double* c, int R);
}  // namespace fd

using namespace fd;

struct fd_tti_s {
  fd_grid_desc d;
  int R = 1;
  int Nx = 0, Ny = 0, Nz = 0, pitch = 0;
  size_t ncell = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float2* u[2] = {nullptr, nullptr};  // (p, q): u[cur] at t_n, u[cur^1] at t_{n-1}
  // model on the padded grid: pairs (A, e2), (dl, nz), (nx, ny), field f at
  // coef + f * ncell
  float2* coef = nullptr;
  int cur = 0;
  bool model_set = false;
  double vmax = 0.0, cfl = 0.0;
  float bscale = 0.0f;
  double c[kMaxR + 1] = {}, d1[kMaxR + 1] = {};
  DevBuf inj, rec, stage_val, stage_rec, stage_in, scratch;
  DevBuf err;  // error word of the TMA kernel's bounded waits
  // tensor maps of the step kernel, per buffer
  CUtensorMap halo[2], tile[2], coef_map;
  long long spin_limit = 0;
  int ctas = 0;  // persistent CTAs of a step (0: not known yet)
  int n_inj = 0, n_rec = 0;
  bool profiling = false;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  double step_ms = 0.0;
  long long steps_timed = 0;
};

namespace {

constexpr size_t kStageBytes = size_t(32) << 20;  // staging of states not on the device

struct TtiInj {
  long long off;
  int x, y, z;
  float w;  // trilinear weight / h
  int col;
};

struct TtiRec {
  long long off[8];
  float w[8];
};

__device__ __forceinline__ int depth(int g, int nbl, int n) {
  int d = nbl - g;
  const int e = g - (n + nbl - 1);
  d = d > e ? d : e;
  return d > 0 ? d : 0;
}

// Model fields on the padded, pitched grid (edge replication into the layer),
// in double, rounded once: A = dt^2 v^2 / h^2, 1 + 2 eps, sqrt(1 + 2 delta),
// n = (sin t cos p, sin t sin p, cos t).
__global__ void k_tti_coef(const float* __restrict__ vp, const float* __restrict__ eps,
                           const float* __restrict__ del, const float* __restrict__ th,
                           const float* __restrict__ ph, int nx, int ny, int nz, int nbl,
                           int Nx, int Ny, int pitch, size_t ncell, double dt2_h2,
                           float2* __restrict__ coef) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y, z = blockIdx.z;
  if (x >= pitch) return;
  const size_t o = (static_cast<size_t>(z) * Ny + y) * pitch + x;
  if (x >= Nx) {
    for (int f = 0; f < 3; ++f) coef[f * ncell + o] = make_float2(0.f, 0.f);
    return;
  }
  const int px = min(max(x - nbl, 0), nx - 1);
  const int py = min(max(y - nbl, 0), ny - 1);
  const int pz = min(max(z - nbl, 0), nz - 1);
  const size_t i = (static_cast<size_t>(pz) * ny + py) * nx + px;
  const double v = vp[i], t = th[i], p = ph[i];
  coef[o] = make_float2(static_cast<float>(dt2_h2 * v * v),
                        static_cast<float>(1.0 + 2.0 * static_cast<double>(eps[i])));
  coef[ncell + o] =
      make_float2(static_cast<float>(sqrt(1.0 + 2.0 * static_cast<double>(del[i]))),
                  static_cast<float>(cos(t)));
  coef[2 * ncell + o] =
      make_float2(static_cast<float>(sin(t) * cos(p)), static_cast<float>(sin(t) * sin(p)));
}

// max of v sqrt(1+2 eps) (bits of a non-negative float) and the count of
// invalid cells (v not positive, 1+2eps or 1+2delta not positive, anything
// not finite).
__global__ void k_tti_stats(const float* __restrict__ vp, const float* __restrict__ eps,
                            const float* __restrict__ del, const float* __restrict__ th,
                            const float* __restrict__ ph, size_t n, unsigned int* out) {
  float hi = 0.f;
  int bad = 0;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const float v = vp[i], e = eps[i], d = del[i];
    if (!(v > 0.f) || !isfinite(v) || !(1.f + 2.f * e > 0.f) || !isfinite(e) ||
        !(1.f + 2.f * d > 0.f) || !isfinite(d) || !isfinite(th[i]) || !isfinite(ph[i])) {
      ++bad;
      continue;
    }
    hi = fmaxf(hi, v * sqrtf(1.f + 2.f * e));
  }
  for (int o = 16; o > 0; o >>= 1) {
    hi = fmaxf(hi, __shfl_down_sync(0xffffffffu, hi, o));
    bad += __shfl_down_sync(0xffffffffu, bad, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(out, __float_as_uint(hi));
    if (bad) atomicAdd(out + 1, static_cast<unsigned int>(bad));
  }
}

// The points between two steps, on u = (p, q)^n: first the sources of the step
// that made u,
//   p, q at each source node += A w q(t_{n-1}) / (h (1 + b))
// (s^n = w q / h^3 scaled by dt^2 v^2 and the damping division of the update;
// val null: none), then the receivers, rec[n][r] = sum_k w_k p[off_k] (out null:
// none).  Both in one launch take one block, so that the receivers see the sources.
constexpr int kPointThreads = 512, kPointsAtOnce = 4096;
__global__ void __launch_bounds__(kPointThreads)
    k_tti_points(const TtiInj* __restrict__ inj, int ninj, const float* __restrict__ val,
                 const float2* __restrict__ coef, float bscale, int nbl, int nx, int ny, int nz,
                 float2* u, const TtiRec* __restrict__ recs, int nrec, float* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  if (val) {
    for (int i = blockIdx.x * kPointThreads + threadIdx.x; i < ninj;
         i += gridDim.x * kPointThreads) {
      const TtiInj e = inj[i];
      const int dx = depth(e.x, nbl, nx), dy = depth(e.y, nbl, ny), dz = depth(e.z, nbl, nz);
      const float b = bscale * static_cast<float>(dx * dx + dy * dy + dz * dz);
      const float s = coef[e.off].x * e.w * val[e.col] / (1.f + b);
      atomicAdd(&u[e.off].x, s);
      atomicAdd(&u[e.off].y, s);
    }
    __threadfence();
    __syncthreads();
  }
  if (out) {
    for (int r = blockIdx.x * kPointThreads + threadIdx.x; r < nrec;
         r += gridDim.x * kPointThreads) {
      const TtiRec e = recs[r];
      float acc = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k)  // (L2: where the atomics went)
        acc = fmaf(e.w[k], __ldcg(&u[e.off[k]].x), acc);
      out[r] = acc;
    }
  }
}

// Rows [row0, row0 + rows) of the padded grid (row = z Ny + y) between the
// (p, q) pairs and a dense array of one of the two fields (f = 0: p, 1: q)
// that starts at row row0.
__global__ void k_tti_field(float2* __restrict__ u, float* __restrict__ dense, int Nx, int pitch,
                            size_t row0, int f, int to_user) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= Nx) return;
  float* cell = reinterpret_cast<float*>(u + (row0 + blockIdx.y) * pitch + x) + f;
  float* user = dense + static_cast<size_t>(blockIdx.y) * Nx + x;
  if (to_user)
    *user = *cell;
  else
    *cell = *user;
}

// The same for both fields at once.  A field alone reads or writes half of each
// 32-byte sector of the pairs.  set_state and get_state of four arrays on the device
// at 240^3, us: 196 and 190 with the separate wavefields of the former kernel, 263
// one field at a time, 139 by pairs.
__global__ void k_tti_pairs(float2* u, float* p, float* q, int Nx, int pitch, size_t row0,
                            int to_user) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= Nx) return;
  float2* cell = u + (row0 + blockIdx.y) * pitch + x;
  const size_t i = static_cast<size_t>(blockIdx.y) * Nx + x;
  if (to_user) {
    const float2 v = *cell;
    p[i] = v.x;
    q[i] = v.y;
  } else {
    *cell = make_float2(p[i], q[i]);
  }
}

// Launches one step on the resident CTAs (*ctas, found by the first call).
template <int R>
cudaError_t launch_q(const tti::QMaps& M, const tti::QArgs& qa, int* ctas, bool pdl,
                     cudaStream_t s) {
  if (*ctas == 0) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (!e) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (!e)
      e = cudaFuncSetAttribute(tti::k_tti_q<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(tti::QGeom<R>::SMEM));
    if (!e)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, tti::k_tti_q<R>, tti::kQT,
                                                        tti::QGeom<R>::SMEM);
    if (e) return e;
    // at least R planes per share: each run of planes first enters 2R
    const long long units = (long long)qa.cols * qa.Nz;
    *ctas = int(std::max<long long>(
        1, std::min<long long>((long long)std::max(per, 1) * sms, units / R)));
  }
  return launch_step(tti::k_tti_q<R>, dim3(*ctas), tti::kQT, tti::QGeom<R>::SMEM, pdl, s, M, qa);
}

cudaError_t launch_q_r(int R, const tti::QMaps& M, const tti::QArgs& qa, int* ctas, bool pdl,
                       cudaStream_t s) {
  count_launch();
  switch (R) {
    case 1: return launch_q<1>(M, qa, ctas, pdl, s);
    case 2: return launch_q<2>(M, qa, ctas, pdl, s);
    case 3: return launch_q<3>(M, qa, ctas, pdl, s);
    case 4: return launch_q<4>(M, qa, ctas, pdl, s);
    case 5: return launch_q<5>(M, qa, ctas, pdl, s);
    case 6: return launch_q<6>(M, qa, ctas, pdl, s);
    case 7: return launch_q<7>(M, qa, ctas, pdl, s);
    case 8: return launch_q<8>(M, qa, ctas, pdl, s);
  }
  return cudaErrorInvalidValue;
}

// Centred first-derivative weights of order 2R:
// d_j = (-1)^(j+1) (R!)^2 / (j (R-j)! (R+j)!), d_0 = 0.
void first_weights(int R, double* d) {
  d[0] = 0.0;
  for (int j = 1; j <= R; ++j) {
    double ratio = 1.0;  // (R!)^2 / ((R-j)! (R+j)!)
    for (int k = 1; k <= j; ++k) ratio *= double(R - k + 1) / double(R + k);
    d[j] = ((j & 1) ? 1.0 : -1.0) * ratio / double(j);
  }
}

fd_status stage(fd_tti t, DevBuf& buf, const float* p, size_t n, size_t off_floats,
                const float** out) {
  if (is_device_ptr(p)) {
    *out = p;
    return FD_OK;
  }
  cudaError_t e = cudaMemcpyAsync(static_cast<float*>(buf.p) + off_floats, p, n * sizeof(float),
                                  cudaMemcpyHostToDevice, t->stream);
  if (e) return cuda_fail(e, "host to device copy");
  *out = static_cast<const float*>(buf.p) + off_floats;
  return FD_OK;
}

fd_status locate(fd_tti t, const float* xyz, int i0[3], double f[3]) {
  const int n[3] = {t->d.nx, t->d.ny, t->d.nz};
  for (int a = 0; a < 3; ++a) {
    const double s = double(xyz[a]) / t->d.h;
    if (!(s >= 0.0) || s > double(n[a] - 1))
      return fail(FD_ERR_ARG, "point (%g, %g, %g) outside the physical box", xyz[0], xyz[1],
                  xyz[2]);
    const double fl = floor(s);
    i0[a] = int(fl) + t->d.nbl;
    f[a] = s - fl;
  }
  return FD_OK;
}

size_t offset(fd_tti t, int x, int y, int z) {
  return (size_t(z) * t->Ny + y) * t->pitch + x;
}

fd_status tables(fd_tti t, const fd_points* src, const fd_points* rec) {
  std::vector<TtiInj> inj;
  std::vector<TtiRec> recs;
  const int N[3] = {t->Nx, t->Ny, t->Nz};
  for (int p = 0; p < (src ? src->n : 0); ++p) {
    int i0[3];
    double f[3];
    fd_status st = locate(t, src->xyz + 3 * p, i0, f);
    if (st) return st;
    for (int c = 0; c < 8; ++c) {
      int node[3];
      double w = 1.0;
      for (int a = 0; a < 3; ++a) {
        const int hi = (c >> a) & 1;
        node[a] = i0[a] + hi;
        w *= hi ? f[a] : 1.0 - f[a];
      }
      if (w == 0.0 || node[0] >= N[0] || node[1] >= N[1] || node[2] >= N[2]) continue;
      inj.push_back({(long long)offset(t, node[0], node[1], node[2]), node[0], node[1], node[2],
                     float(w / t->d.h), p});
    }
  }
  for (int p = 0; p < (rec ? rec->n : 0); ++p) {
    int i0[3];
    double f[3];
    fd_status st = locate(t, rec->xyz + 3 * p, i0, f);
    if (st) return st;
    TtiRec e;
    for (int c = 0; c < 8; ++c) {
      int node[3];
      double w = 1.0;
      for (int a = 0; a < 3; ++a) {
        const int hi = (c >> a) & 1;
        node[a] = i0[a] + hi;
        w *= hi ? f[a] : 1.0 - f[a];
      }
      const bool ok = node[0] < N[0] && node[1] < N[1] && node[2] < N[2];
      e.off[c] = ok ? (long long)offset(t, node[0], node[1], node[2]) : 0;
      e.w[c] = ok ? float(w) : 0.f;
    }
    recs.push_back(e);
  }
  cudaError_t e = t->inj.ensure(std::max<size_t>(inj.size() * sizeof(TtiInj), 16));
  if (!e) e = t->rec.ensure(std::max<size_t>(recs.size() * sizeof(TtiRec), 16));
  if (!e && !inj.empty())
    e = cudaMemcpyAsync(t->inj.p, inj.data(), inj.size() * sizeof(TtiInj),
                        cudaMemcpyHostToDevice, t->stream);
  if (!e && !recs.empty())
    e = cudaMemcpyAsync(t->rec.p, recs.data(), recs.size() * sizeof(TtiRec),
                        cudaMemcpyHostToDevice, t->stream);
  if (!e) e = cudaStreamSynchronize(t->stream);
  if (e) return cuda_fail(e, "point tables");
  t->n_inj = int(inj.size());
  t->n_rec = int(recs.size());
  return FD_OK;
}

// One field of a state (f = 0: p, 1: q) between its pairs and a dense padded
// array of the caller: memory of the grid's own device directly, host memory and
// that of other devices through a staging buffer in pieces of whole rows.
fd_status copy_state(fd_tti t, float2* dev, int f, void* user, bool to_user) {
  const size_t rows = size_t(t->Ny) * t->Nz;
  const bool on_device = is_local_ptr(user, t->d.device);
  const size_t row_bytes = size_t(t->Nx) * 4;
  const size_t most = 65535;  // rows of one launch
  const size_t piece =
      std::min(on_device ? most : std::max<size_t>(1, std::min(most, kStageBytes / row_bytes)),
               rows);
  cudaError_t e;
  if (!on_device && (e = t->stage_in.ensure(piece * row_bytes)))
    return cuda_fail(e, "state staging");
  for (size_t r = 0; r < rows; r += piece) {
    const size_t n = std::min(piece, rows - r);
    char* u = static_cast<char*>(user) + r * row_bytes;
    float* dense = static_cast<float*>(on_device ? static_cast<void*>(u) : t->stage_in.p);
    if (!on_device && !to_user) {
      e = cudaMemcpyAsync(dense, u, n * row_bytes, cudaMemcpyDefault, t->stream);
      if (e) return cuda_fail(e, "wavefield copy");
    }
    k_tti_field<<<dim3((t->Nx + 127) / 128, unsigned(n)), 128, 0, t->stream>>>(
        dev, dense, t->Nx, t->pitch, r, f, to_user ? 1 : 0);
    count_launch();
    if ((e = cudaGetLastError())) return cuda_fail(e, "wavefield copy");
    if (!on_device && to_user) {
      e = cudaMemcpyAsync(u, dense, n * row_bytes, cudaMemcpyDefault, t->stream);
      if (e) return cuda_fail(e, "wavefield copy");
    }
  }
  return FD_OK;
}

// The caller's arrays p_prev, p, q_prev, q (null: left alone) from or to the state:
// both fields of a time level together where a kernel can address both arrays, each
// array in turn otherwise, or if one array is given twice (the last one counts).
fd_status copy_states(fd_tti t, float* const user[4], bool to_user) {
  bool twice = false;
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < i; ++j) twice = twice || (user[i] && user[i] == user[j]);
  bool done[4] = {false, false, false, false};
  const size_t rows = size_t(t->Ny) * t->Nz, most = 65535;  // rows of one launch
  for (int k = 0; k < 2 && !twice; ++k) {
    float *p = user[k], *q = user[k + 2];
    if (!is_local_ptr(p, t->d.device) || !is_local_ptr(q, t->d.device)) continue;
    for (size_t r = 0; r < rows; r += most) {
      k_tti_pairs<<<dim3((t->Nx + 127) / 128, unsigned(std::min(most, rows - r))), 128, 0,
                    t->stream>>>(t->u[k ? t->cur : t->cur ^ 1], p + r * t->Nx, q + r * t->Nx,
                                 t->Nx, t->pitch, r, to_user ? 1 : 0);
      count_launch();
      cudaError_t e = cudaGetLastError();
      if (e) return cuda_fail(e, "wavefield copy");
    }
    done[k] = done[k + 2] = true;
  }
  for (int i = 0; i < 4; ++i) {
    if (!user[i] || done[i]) continue;
    fd_status st = copy_state(t, t->u[(i & 1) ? t->cur : t->cur ^ 1], i >> 1, user[i], to_user);
    if (st) return st;
  }
  cudaError_t e = cudaStreamSynchronize(t->stream);
  return e ? cuda_fail(e, "wavefield copy") : FD_OK;
}

fd_status propagate(fd_tti t, int n0, int nsteps, const fd_points* src, const float* wavelet,
                    const fd_points* rec, float* rec_out) {
  if (!t->model_set) return fail(FD_ERR_STATE, "fd_tti_set_model has not been called");
  if (n0 < 0 || nsteps < 0) return fail(FD_ERR_ARG, "negative step range");
  const int nsrc = src ? src->n : 0, nrec = rec ? rec->n : 0;
  if ((nsrc && (!src->xyz || !wavelet)) || (nrec && (!rec->xyz || !rec_out)))
    return fail(FD_ERR_ARG, "points given without their data array");
  fd_status st = tables(t, src, rec);
  if (st) return st;
  cudaError_t e;
  const float* dval = nullptr;
  if (nsrc) {
    const size_t n = size_t(n0 + nsteps) * nsrc;
    if (!is_device_ptr(wavelet) && (e = t->stage_val.ensure(n * 4))) return cuda_fail(e, "staging");
    if ((st = stage(t, t->stage_val, wavelet, n, 0, &dval))) return st;
  }
  float* drec = nullptr;
  if (nrec) {
    if (is_device_ptr(rec_out)) {
      drec = rec_out;
    } else {
      if ((e = t->stage_rec.ensure(size_t(nsteps) * nrec * 4))) return cuda_fail(e, "staging");
      drec = static_cast<float*>(t->stage_rec.p);
    }
  }
  tti::QArgs qa;
  memset(&qa, 0, sizeof(qa));
  qa.err = static_cast<int*>(t->err.p);
  qa.Nx = t->Nx;
  qa.Ny = t->Ny;
  qa.Nz = t->Nz;
  qa.pitch = t->pitch;
  qa.nbl = t->d.nbl;
  qa.nx = t->d.nx;
  qa.ny = t->d.ny;
  qa.nz = t->d.nz;
  qa.spin_limit = t->spin_limit;
  qa.bscale = t->bscale;
  for (int j = 0; j <= kMaxR; ++j) {
    qa.c[j].x = qa.c[j].y = j <= t->R ? float(t->c[j]) : 0.f;
    qa.d[j].x = qa.d[j].y = j <= t->R ? float(t->d1[j]) : 0.f;
  }
  // the centre weight that the FP32 weights c_j need, as hi + lo
  double c0 = 0.0;
  for (int j = 1; j <= t->R; ++j) c0 -= 2.0 * qa.c[j].x;
  qa.c[0].x = qa.c[0].y = float(c0);
  qa.c0lo.x = qa.c0lo.y = float(c0 - qa.c[0].x);
  qa.cols_y = (t->Ny + tti::kQY - 1) / tti::kQY;
  qa.cols = qa.cols_y * ((t->Nx + tti::kQX - 1) / tti::kQX);
  if (t->profiling) cudaEventRecord(t->ev0, t->stream);
  // Launches of short steps may start before the one ahead has finished.  us a step
  // without / with it, at M padded cells:
  //   SO 4   1.0 M 25.2 / 21.9   3.4 M  47.6 / 44.5    5.8 M  69.3 / 70.8   8.0 M   94 / 102
  //   SO 8   1.0 M 34.6 / 30.7   3.9 M  68.9 / 66.4    5.8 M  93.3 / 93.6  37.9 M  469 / 499
  //   SO 10  2.2 M 59.8 / 55.1   4.1 M  76.5 / 73.5   15.6 M 234.8 / 239.4 27.0 M  401 / 415
  //   SO 12  2.2 M 68.6 / 64.8   4.1 M  89.4 / 87.1    9.3 M 179.5 / 183.3 27.0 M  464 / 476
  //   SO 14  1.0 M 48.6 / 43.6   4.1 M  99.0 / 94.2   15.6 M 310.1 / 305.2 63.8 M 1207 / 1202
  //   SO 16  1.0 M 54.5 / 48.8   4.1 M 108.1 / 103.6  19.7 M 433.2 / 428.9 63.8 M 1330 / 1326
  // CTAs that start where an earlier one ends break up the waves of neighbouring
  // columns, which share halos in L2; with the two CTAs per SM of SO 14 and 16 that
  // costs less than the launch's latency at every size up to those 64 M.
  const bool early =
      (long long)t->Nx * t->Ny * t->Nz <= (t->R >= 7 ? 64000000LL : 4000000LL);
  // sources of step `s` (-1: none) and receivers of the field it made, on u;
  // many of them in two launches of several blocks
  auto points = [&](int s, float2* u, bool first) -> cudaError_t {
    const bool inj = t->n_inj && s >= 0, rec = nrec && s + 1 < nsteps;
    const float* val = inj ? dval + size_t(n0 + s) * nsrc : nullptr;
    float* out = rec ? drec + size_t(s + 1) * nrec : nullptr;
    auto launch = [&](int blocks, const float* v, float* o) {
      count_launch();
      return launch_step(k_tti_points, dim3(blocks), kPointThreads, 0, early && !first, t->stream,
                         static_cast<const TtiInj*>(t->inj.p), t->n_inj, v, t->coef, t->bscale,
                         t->d.nbl, t->d.nx, t->d.ny, t->d.nz, u,
                         static_cast<const TtiRec*>(t->rec.p), nrec, o);
    };
    auto blocks = [](int n) { return (n + kPointThreads - 1) / kPointThreads; };
    if (!inj && !rec) return cudaSuccess;
    if (t->n_inj <= kPointsAtOnce && nrec <= kPointsAtOnce) return launch(1, val, out);
    cudaError_t er = inj ? launch(blocks(t->n_inj), val, nullptr) : cudaSuccess;
    if (!er && rec) er = launch(blocks(nrec), nullptr, out);
    return er;
  };
  if ((e = points(-1, t->u[t->cur], true))) return cuda_fail(e, "TTI points launch");
  for (int s = 0; s < nsteps; ++s) {
    const int cur = t->cur;
    tti::QMaps M;
    M.halo = t->halo[cur];
    M.prev = t->tile[cur ^ 1];
    M.coef = t->coef_map;
    qa.out = t->u[cur ^ 1];
    if ((e = launch_q_r(t->R, M, qa, &t->ctas, early && s > 0, t->stream)))
      return cuda_fail(e, "TTI step launch");
    if ((e = points(s, t->u[cur ^ 1], false))) return cuda_fail(e, "TTI points launch");
    t->cur = cur ^ 1;
  }
  if (t->profiling) {
    cudaEventRecord(t->ev1, t->stream);
    if ((e = cudaEventSynchronize(t->ev1))) return cuda_fail(e, "profiling event");
    float ms = 0.f;
    cudaEventElapsedTime(&ms, t->ev0, t->ev1);
    t->step_ms += ms;
    t->steps_timed += nsteps;
  }
  if ((e = cudaGetLastError())) return cuda_fail(e, "TTI launch");
  if (nrec) {
    int bad = 0;
    e = count_nonfinite(drec, size_t(nsteps) * nrec, reinterpret_cast<int*>(t->scratch.p), &bad,
                        t->stream);
    if (e) return cuda_fail(e, "finite check");
    if (bad) return fail(FD_ERR_NONFINITE, "%d receiver samples are NaN or Inf", bad);
    if (drec != rec_out && nsteps > 0) {
      e = cudaMemcpyAsync(rec_out, drec, size_t(nsteps) * nrec * 4, cudaMemcpyDeviceToHost,
                          t->stream);
      if (e) return cuda_fail(e, "device to host copy");
    }
  }
  e = cudaStreamSynchronize(t->stream);
  if (e) return cuda_fail(e, "stream synchronize");
  if (nsteps > 0) {
    int flag = 0;
    e = cudaMemcpyAsync(&flag, t->err.p, sizeof(flag), cudaMemcpyDeviceToHost, t->stream);
    if (!e) e = cudaStreamSynchronize(t->stream);
    if (e) return cuda_fail(e, "error word");
    if (flag) {
      cudaMemsetAsync(t->err.p, 0, sizeof(int), t->stream);
      cudaStreamSynchronize(t->stream);
      return fail(FD_ERR_TIMEOUT, "a bounded wait of the TTI step ran out");
    }
  }
  return FD_OK;
}

}  // namespace

extern "C" {

fd_status fd_tti_create(const fd_grid_desc* d, fd_tti* out) {
  clear_error();
  if (!d || !out) return fail(FD_ERR_ARG, "null argument");
  *out = nullptr;
  if (d->nx < 1 || d->ny < 1 || d->nz < 1) return fail(FD_ERR_ARG, "grid sizes must be positive");
  if (!(d->h > 0.0) || !(d->dt > 0.0)) return fail(FD_ERR_ARG, "h and dt must be positive");
  if (d->space_order < 2 || d->space_order > 16 || (d->space_order & 1))
    return fail(FD_ERR_ARG, "space_order must be even, 2..16");
  if (d->nbl < 0 || d->nt < 0) return fail(FD_ERR_ARG, "nbl and nt must be >= 0");
  const long long Nx = d->nx + 2LL * d->nbl, Ny = d->ny + 2LL * d->nbl, Nz = d->nz + 2LL * d->nbl;
  if (Nx > (1 << 24) || Ny > 65535 || Nz > 65535) return fail(FD_ERR_ARG, "padded grid too large");
  cudaError_t e = cudaSetDevice(d->device);
  if (e) return cuda_fail(e, "cudaSetDevice");
  fd_tti t = new fd_tti_s();
  t->d = *d;
  t->R = d->space_order / 2;
  t->Nx = int(Nx);
  t->Ny = int(Ny);
  t->Nz = int(Nz);
  t->pitch = int((Nx + 31) / 32 * 32);
  t->ncell = size_t(t->pitch) * t->Ny * t->Nz;
  fd_weights(t->R, t->c);
  first_weights(t->R, t->d1);
  t->cfl = cfl_limit(t->c, t->R);
  fd_status st = FD_OK;
  if (d->stream) {
    t->stream = static_cast<cudaStream_t>(d->stream);
  } else {
    e = cudaStreamCreateWithFlags(&t->stream, cudaStreamDefault);
    if (e) st = cuda_fail(e, "stream create");
    t->own_stream = true;
  }
  for (int b = 0; b < 2 && !st; ++b) {
    e = dev_alloc(reinterpret_cast<void**>(&t->u[b]), t->ncell * sizeof(float2));
    if (e) st = cuda_fail(e, "wavefield allocation");
  }
  if (!st) {
    e = dev_alloc(reinterpret_cast<void**>(&t->coef), 3 * t->ncell * sizeof(float2));
    if (!e) e = t->scratch.ensure(64);
    if (!e) e = t->err.ensure(16);
    if (!e) e = cudaMemsetAsync(t->err.p, 0, 16, t->stream);
    if (e) st = cuda_fail(e, "model allocation");
  }
  t->spin_limit = default_spin_limit();
  if (!st) {
    // tensor maps of the step kernel: staged planes with the x halo rounded
    // up to two cells and R rows, per-point tiles (rows of pairs are rows of
    // twice as many floats), the model
    const int W = tti::kQX + 2 * tti::q_halo_x(t->R);
    for (int b = 0; b < 2 && !st; ++b) {
      const float* u = reinterpret_cast<const float*>(t->u[b]);
      st = make_map(&t->halo[b], u, 2 * t->Nx, t->Ny, t->Nz, 2 * t->pitch, 2 * W, tti::kQY + 2 * t->R);
      if (!st)
        st = make_map(&t->tile[b], u, 2 * t->Nx, t->Ny, t->Nz, 2 * t->pitch, 2 * tti::kQX, tti::kQY);
    }
    if (!st)
      st = make_map(&t->coef_map, reinterpret_cast<const float*>(t->coef), 2 * t->Nx, t->Ny,
                    3 * t->Nz, 2 * t->pitch, 2 * tti::kQX, tti::kQY);
  }
  if (!st) {
    for (int b = 0; b < 2 && !e; ++b)
      e = cudaMemsetAsync(t->u[b], 0, t->ncell * sizeof(float2), t->stream);
    if (!e) e = cudaMemsetAsync(t->coef, 0, 3 * t->ncell * sizeof(float2), t->stream);
    if (!e) e = cudaEventCreate(&t->ev0);
    if (!e) e = cudaEventCreate(&t->ev1);
    if (!e) e = cudaStreamSynchronize(t->stream);
    if (e) st = cuda_fail(e, "grid initialisation");
  }
  if (st) {
    fd_tti_destroy(t);
    return st;
  }
  *out = t;
  return FD_OK;
}

fd_status fd_tti_destroy(fd_tti t) {
  if (!t) return FD_OK;
  cudaSetDevice(t->d.device);
  if (t->stream) cudaStreamSynchronize(t->stream);
  for (int b = 0; b < 2; ++b)
    if (t->u[b]) cudaFree(t->u[b]);
  if (t->coef) cudaFree(t->coef);
  for (DevBuf* b : {&t->inj, &t->rec, &t->stage_val, &t->stage_rec, &t->stage_in, &t->scratch,
                    &t->err})
    b->release();
  if (t->ev0) cudaEventDestroy(t->ev0);
  if (t->ev1) cudaEventDestroy(t->ev1);
  if (t->own_stream && t->stream) cudaStreamDestroy(t->stream);
  delete t;
  return FD_OK;
}

fd_status fd_tti_set_model(fd_tti t, const float* vp, const float* epsilon, const float* delta,
                           const float* theta, const float* phi) {
  clear_error();
  if (!t || !vp || !epsilon || !delta || !theta || !phi) return fail(FD_ERR_ARG, "null argument");
  cudaSetDevice(t->d.device);
  const size_t np = size_t(t->d.nx) * t->d.ny * t->d.nz;
  const float* in[5] = {vp, epsilon, delta, theta, phi};
  const float* dev[5];
  bool host = false;
  for (int f = 0; f < 5; ++f) host |= !is_device_ptr(in[f]);
  cudaError_t e;
  if (host && (e = t->stage_in.ensure(5 * np * 4))) return cuda_fail(e, "model staging");
  for (int f = 0; f < 5; ++f) {
    fd_status st = stage(t, t->stage_in, in[f], np, size_t(f) * np, &dev[f]);
    if (st) return st;
  }
  // the staging copy of host arrays is only needed inside this call: freed
  // on every return, after the work that reads it has finished
  struct Release {
    DevBuf& b;
    cudaStream_t s;
    ~Release() {
      if (b.p) cudaStreamSynchronize(s);
      b.release();
    }
  } release_staging{t->stage_in, t->stream};
  unsigned int h[2] = {0, 0};
  unsigned int* s = static_cast<unsigned int*>(t->scratch.p);
  e = cudaMemsetAsync(s, 0, 8, t->stream);
  if (!e) {
    k_tti_stats<<<1024, 256, 0, t->stream>>>(dev[0], dev[1], dev[2], dev[3], dev[4], np, s);
    count_launch();
    e = cudaGetLastError();
  }
  if (!e) e = cudaMemcpyAsync(h, s, 8, cudaMemcpyDeviceToHost, t->stream);
  if (!e) e = cudaStreamSynchronize(t->stream);
  if (e) return cuda_fail(e, "model statistics");
  if (h[1]) return fail(FD_ERR_ARG, "%u model cells are invalid", h[1]);
  float vmax;
  memcpy(&vmax, &h[0], 4);
  const double courant = double(vmax) * t->d.dt / t->d.h;
  if (courant > t->cfl)
    return fail(FD_ERR_UNSTABLE, "v_max sqrt(1+2 eps) dt / h = %.4f exceeds the limit %.4f",
                courant, t->cfl);
  dim3 grid((t->pitch + 127) / 128, t->Ny, t->Nz);
  k_tti_coef<<<grid, 128, 0, t->stream>>>(dev[0], dev[1], dev[2], dev[3], dev[4], t->d.nx,
                                          t->d.ny, t->d.nz, t->d.nbl, t->Nx, t->Ny, t->pitch,
                                          t->ncell, t->d.dt * t->d.dt / (t->d.h * t->d.h), t->coef);
  count_launch();
  if ((e = cudaGetLastError())) return cuda_fail(e, "model set-up");
  t->vmax = vmax;
  if (t->d.nbl > 0) {
    const double gmax = 3.0 * double(vmax) * log(1000.0) / (2.0 * t->d.nbl * t->d.h);
    t->bscale = float(gmax * t->d.dt / 2.0 / (double(t->d.nbl) * t->d.nbl));
  } else {
    t->bscale = 0.f;
  }
  for (int b = 0; b < 2 && !e; ++b)
    e = cudaMemsetAsync(t->u[b], 0, t->ncell * sizeof(float2), t->stream);
  if (!e) e = cudaStreamSynchronize(t->stream);
  if (e) return cuda_fail(e, "model set-up");
  t->cur = 0;
  t->model_set = true;
  return FD_OK;
}

fd_status fd_tti_forward(fd_tti t, const fd_points* src, const float* wavelet,
                         const fd_points* rec, float* rec_out) {
  clear_error();
  if (!t) return fail(FD_ERR_ARG, "null grid");
  cudaSetDevice(t->d.device);
  for (int b = 0; b < 2; ++b) {
    cudaError_t e = cudaMemsetAsync(t->u[b], 0, t->ncell * sizeof(float2), t->stream);
    if (e) return cuda_fail(e, "wavefield reset");
  }
  t->cur = 0;
  return propagate(t, 0, t->d.nt, src, wavelet, rec, rec_out);
}

fd_status fd_tti_propagate(fd_tti t, int32_t n0, int32_t nsteps, const fd_points* src,
                           const float* wavelet, const fd_points* rec, float* rec_out) {
  clear_error();
  if (!t) return fail(FD_ERR_ARG, "null grid");
  cudaSetDevice(t->d.device);
  return propagate(t, n0, nsteps, src, wavelet, rec, rec_out);
}

fd_status fd_tti_set_state(fd_tti t, const float* p_prev, const float* p, const float* q_prev,
                           const float* q) {
  clear_error();
  if (!t) return fail(FD_ERR_ARG, "null grid");
  cudaSetDevice(t->d.device);
  float* const in[4] = {const_cast<float*>(p_prev), const_cast<float*>(p),
                        const_cast<float*>(q_prev), const_cast<float*>(q)};
  return copy_states(t, in, false);
}

fd_status fd_tti_get_state(fd_tti t, float* p_prev, float* p, float* q_prev, float* q) {
  clear_error();
  if (!t) return fail(FD_ERR_ARG, "null grid");
  cudaSetDevice(t->d.device);
  float* const out[4] = {p_prev, p, q_prev, q};
  return copy_states(t, out, true);
}

fd_status fd_tti_set_profiling(fd_tti t, int32_t enabled) {
  clear_error();
  if (!t) return fail(FD_ERR_ARG, "null grid");
  t->profiling = enabled != 0;
  if (t->profiling) {
    t->step_ms = 0.0;
    t->steps_timed = 0;
  }
  return FD_OK;
}

fd_status fd_tti_get_info(fd_tti t, fd_grid_info* info) {
  clear_error();
  if (!t || !info) return fail(FD_ERR_ARG, "null argument");
  memset(info, 0, sizeof(*info));
  info->nx_pad = t->Nx;
  info->ny_pad = t->Ny;
  info->nz_pad = t->Nz;
  info->pitch = t->pitch;
  info->tile_x = tti::kQX;
  info->tile_y = tti::kQY;
  info->v_max = t->vmax;
  info->cfl_limit = t->cfl;
  info->launches = fd_launch_count();
  info->step_ms = t->step_ms;
  info->steps_timed = t->steps_timed;
  return FD_OK;
}

}  // extern "C"
