// Small helper kernels of libfd.so: model set-up, reductions, gradient fold.
#include <math.h>
#include <string.h>

#include "fd_aux.h"

namespace fd {

namespace {

// Smallest and largest velocity of a model and its count of bad values.  Bound by
// memory: four loads of a thread are in flight, on up to eight blocks per SM.  The
// maxima of a block go to the words in one atomic each (one per thread queued 2.6e5
// of them on each word; one per warp and two blocks per SM left too few loads in
// flight for large models).  fd_set_model of 64^3 / 256^3 / 512^3 cells, us: with one
// atomic per thread and 1024 blocks 63 / 328 / 1772, with one per warp and two blocks
// per SM 54 / 387 / 2316, now 52 / 303 / 1634.
constexpr int kStatThreads = 256, kStatLoads = 4;
__global__ void __launch_bounds__(kStatThreads)
    k_model_stats(const float* __restrict__ data, size_t n, int kind, unsigned int* vmin_bits,
                  unsigned int* vmax_bits, int* bad) {
  // positive floats order like their bit patterns
  unsigned lo = 0x7f800000u, hi = 0u, nbad = 0u;
  auto take = [&](float x) {
    if (!(x > 0.0f) || !isfinite(x)) {
      ++nbad;
      return;
    }
    const unsigned v = __float_as_uint(kind == 0 ? x : 1.0f / sqrtf(x));
    lo = min(lo, v);
    hi = max(hi, v);
  };
  const size_t step = (size_t)gridDim.x * kStatThreads;
  size_t i = blockIdx.x * (size_t)kStatThreads + threadIdx.x;
  for (; i + (kStatLoads - 1) * step < n; i += kStatLoads * step) {
    float x[kStatLoads];
#pragma unroll
    for (int k = 0; k < kStatLoads; ++k) x[k] = data[i + k * step];
#pragma unroll
    for (int k = 0; k < kStatLoads; ++k) take(x[k]);
  }
  for (; i < n; i += step) take(data[i]);
  __shared__ unsigned s_lo[kStatThreads / 32], s_hi[kStatThreads / 32], s_bad[kStatThreads / 32];
  __syncwarp();
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  nbad = __reduce_add_sync(0xffffffffu, nbad);
  if ((threadIdx.x & 31) == 0) {
    s_lo[threadIdx.x >> 5] = lo;
    s_hi[threadIdx.x >> 5] = hi;
    s_bad[threadIdx.x >> 5] = nbad;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < kStatThreads / 32; ++w) {
    lo = min(lo, s_lo[w]);
    hi = max(hi, s_hi[w]);
    nbad += s_bad[w];
  }
  if (nbad) atomicAdd(bad, static_cast<int>(nbad));
  if (hi) {
    atomicMin(vmin_bits, lo);
    atomicMax(vmax_bits, hi);
  }
}

// A = dt^2 / (m h^2) on every padded cell, the model edge-replicated into the
// layer.  Computed in double, rounded once to float.
__global__ void k_model_to_A(const float* __restrict__ data, int kind, int nx,
                             int ny, int nz, int nbl, int Nx, int Ny, int Nz,
                             int pitch, double dt2_h2, float* __restrict__ A) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  const int z = blockIdx.z;
  if (x >= pitch) return;
  float* row = A + ((size_t)z * Ny + y) * pitch;
  if (x >= Nx) {
    row[x] = 0.0f;
    return;
  }
  const int px = min(max(x - nbl, 0), nx - 1);
  const int py = min(max(y - nbl, 0), ny - 1);
  const int pz = min(max(z - nbl, 0), nz - 1);
  const double val = data[((size_t)pz * ny + py) * nx + px];
  const double a = kind == 0 ? dt2_h2 * val * val : dt2_h2 / val;
  row[x] = (float)a;
}

__global__ void k_count_nonfinite(const float* __restrict__ x, size_t n, int* cnt) {
  int c = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    c += isfinite(x[i]) ? 0 : 1;
  if (c) atomicAdd(cnt, c);
}

__global__ void k_residual(const float* __restrict__ rec, const float* __restrict__ obs,
                           float* __restrict__ r, size_t n, double* loss) {
  double acc = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const float d = rec[i] - obs[i];
    r[i] = d;
    acc += 0.5 * (double)d * (double)d;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0 && acc != 0.0) atomicAdd(loss, acc);
}

// Physical gradient: each physical cell sums the padded cells that replicate
// it (only cells on the faces of the physical box have more than one).
__global__ void k_fold_grad(const float* __restrict__ gpad, int nx, int ny, int nz,
                            int nbl, int Nx, int Ny, int Nz, int pitch,
                            float* __restrict__ gphys) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  const int z = blockIdx.z;
  const int xa = x == 0 ? 0 : x + nbl, xb = x == nx - 1 ? Nx - 1 : x + nbl;
  const int ya = y == 0 ? 0 : y + nbl, yb = y == ny - 1 ? Ny - 1 : y + nbl;
  const int za = z == 0 ? 0 : z + nbl, zb = z == nz - 1 ? Nz - 1 : z + nbl;
  double acc = 0.0;
  // the columns of an x end (nbl + 1 cells or more per row) over the lanes of
  // its warp, rows in turn: a corner alone sums (nbl + 1)^3 cells
  const bool end = x < nx && xb > xa;
  for (unsigned todo = __ballot_sync(0xffffffffu, end); todo; todo &= todo - 1) {
    const int src = __ffs(todo) - 1, lane = threadIdx.x & 31;
    const int a = __shfl_sync(0xffffffffu, xa, src), w = __shfl_sync(0xffffffffu, xb, src) - a + 1;
    const int rows = yb - ya + 1;
    double part = 0.0;
    for (int k = za; k <= zb; ++k)
      for (int e = lane; e < rows * w; e += 32)
        part += gpad[((size_t)k * Ny + ya + e / w) * pitch + a + e % w];
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == src) acc = part;
  }
  if (x >= nx) return;
  if (!end)
    for (int k = za; k <= zb; ++k)
      for (int j = ya; j <= yb; ++j) acc += gpad[((size_t)k * Ny + j) * pitch + xa];
  gphys[((size_t)z * ny + y) * nx + x] = (float)acc;
}

__global__ void k_pad_coef(const float* __restrict__ phys, int R, int nx, int ny, int nz,
                           int nbl, int Nx, int Ny, int Nz, int pitch, size_t ncell,
                           float* __restrict__ coef) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y;
  const int z = blockIdx.z;
  if (x >= Nx) return;
  const int px = min(max(x - nbl, 0), nx - 1);
  const int py = min(max(y - nbl, 0), ny - 1);
  const int pz = min(max(z - nbl, 0), nz - 1);
  const size_t src = (((size_t)pz * ny + py) * nx + px) * R;
  const size_t dst = ((size_t)z * Ny + y) * pitch + x;
  for (int j = 0; j < R; ++j) coef[j * ncell + dst] = phys[src + j];
}

// The TMA unit reads tensor maps through a proxy of its own and may hold what an
// address held before its map was refreshed (another tile, or an adjoint segment's
// checkpoint), so each refreshed map is fenced once, on every SM: the shared memory
// of a block admits one per SM.  Everything later on the stream lies behind these
// fences.  Fencing in the step kernels instead costs each CTA several fences: once per
// run 15 us on 83 x 69 x 430 bricks, and in each launch 0.5 us a step on 84^3 and 5 us
// on 149 x 128 x 103; maps passed as kernel parameters, which need no fence, cost 1 us a
// step in launches outside graphs, as each brings them at an address no SM has seen.
constexpr int kAcquireSmem = 120 * 1024;
__global__ void k_acquire_maps(const unsigned char* maps, size_t stride, int groups, int per) {
  for (int i = threadIdx.x; i < groups * per; i += blockDim.x)
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(
                     maps + i / per * stride + size_t(i % per) * 128)
                 : "memory");
}

}  // namespace

cudaError_t acquire_maps(const void* maps, size_t stride, int groups, int per, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_acquire_maps, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kAcquireSmem);
  if (e != cudaSuccess) return e;
  k_acquire_maps<<<sms, 32, kAcquireSmem, s>>>(static_cast<const unsigned char*>(maps), stride,
                                               groups, per);
  count_launch();
  return cudaGetLastError();
}

cudaError_t pad_coefficients(const float* phys, int R, int nx, int ny, int nz, int nbl, int Nx,
                             int Ny, int Nz, int pitch, size_t ncell, float* coef,
                             cudaStream_t s) {
  dim3 grid((Nx + 127) / 128, Ny, Nz);
  k_pad_coef<<<grid, 128, 0, s>>>(phys, R, nx, ny, nz, nbl, Nx, Ny, Nz, pitch, ncell, coef);
  count_launch();
  return cudaGetLastError();
}

cudaError_t model_stats(const float* data, size_t n, int kind, float* vmin,
                        float* vmax, int* nbad, unsigned int* scratch,
                        cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // scratch: [vmin_bits, vmax_bits, bad]
  unsigned int init[3] = {0x7f800000u, 0u, 0u};
  e = cudaMemcpyAsync(scratch, init, sizeof(init), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  const size_t want = (n + kStatThreads * kStatLoads - 1) / (kStatThreads * kStatLoads);
  const int blocks = int(want < 1 ? 1 : (want < size_t(8) * sms ? want : size_t(8) * sms));
  k_model_stats<<<blocks, kStatThreads, 0, s>>>(data, n, kind, scratch, scratch + 1,
                                                reinterpret_cast<int*>(scratch + 2));
  count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  unsigned int out[3];
  e = cudaMemcpyAsync(out, scratch, sizeof(out), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
  memcpy(vmin, &out[0], sizeof(float));
  memcpy(vmax, &out[1], sizeof(float));
  *nbad = static_cast<int>(out[2]);
  return cudaSuccess;
}

cudaError_t model_to_A(const float* data, int kind, int nx, int ny, int nz, int nbl,
                       int Nx, int Ny, int Nz, int pitch, double dt2_h2, float* A,
                       cudaStream_t s) {
  dim3 grid((pitch + 127) / 128, Ny, Nz);
  k_model_to_A<<<grid, 128, 0, s>>>(data, kind, nx, ny, nz, nbl, Nx, Ny, Nz, pitch,
                                    dt2_h2, A);
  count_launch();
  return cudaGetLastError();
}

cudaError_t count_nonfinite_async(const float* x, size_t n, int* dcnt, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(dcnt, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  if (n) {
    k_count_nonfinite<<<256, 256, 0, s>>>(x, n, dcnt);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t count_nonfinite(const float* x, size_t n, int* dcnt, int* hcnt,
                            cudaStream_t s) {
  cudaError_t e = count_nonfinite_async(x, n, dcnt, s);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(hcnt, dcnt, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  return cudaStreamSynchronize(s);
}

cudaError_t residual(const float* rec, const float* obs, float* r, size_t n,
                     double* dloss, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(dloss, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  if (n) {
    k_residual<<<256, 256, 0, s>>>(rec, obs, r, n, dloss);
    count_launch();
  }
  return cudaGetLastError();
}

cudaError_t fold_grad(const float* gpad, int nx, int ny, int nz, int nbl, int Nx,
                      int Ny, int Nz, int pitch, float* gphys, cudaStream_t s) {
  dim3 grid((nx + 127) / 128, ny, nz);
  k_fold_grad<<<grid, 128, 0, s>>>(gpad, nx, ny, nz, nbl, Nx, Ny, Nz, pitch, gphys);
  count_launch();
  return cudaGetLastError();
}

}  // namespace fd
