// Learned stencil coefficients: a 4 -> 64 -> 64 -> 8 network (FP32) that maps
// local, scale-free inputs to space-order-8 weights, with hand-written
// inference, training (fused forward + loss + backward) and Adam kernels, and
// the sampling kernels that turn fine-grid runs of the propagator into
// training samples.  The paper has no learned component; the construction
// follows the learned-discretisation idea of Bar-Sinai et al. (PNAS 2019).
//
// Inputs per cell: x = [v dt / h, h / 10 m, dt / 1 ms, f / 10 Hz].
// Outputs o_1..o_8 -> s_j = (o_j + o_{j+4}) / 2, c_j = cT_j (1 + tanh(s_j)/2),
// c_0 = -2 sum_j c_j (symmetric, zero row sum; an all-zero output layer gives
// the Taylor weights cT).  Sample: x[4], T[4] (T_j = sum of the six neighbours
// at distance j minus 6 u), target y, weight w; prediction p = sum_j c_j T_j;
// loss L = (1/n) sum w (p - y)^2.
// Parameters (5000 floats): W1[64][4] b1[64] W2[64][64] b2[64] W3[8][64] b3[8].
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "fd_aux.h"
#include "fd_mlp.h"
#include "fd_runtime.h"
#include "fd_step.cuh"

using namespace fd;

namespace {

constexpr int H = 64, NIN = 4, NOUT = 8, RL = 4;
constexpr int OW1 = 0, OB1 = OW1 + H * NIN, OW2 = OB1 + H, OB2 = OW2 + H * H,
              OW3 = OB2 + H, OB3 = OW3 + NOUT * H, NPARAM = OB3 + NOUT;
static_assert(NPARAM == FD_MLP_NPARAM, "parameter layout");
constexpr int SAMPLE = FD_MLP_SAMPLE;  // x[4] T[4] y w

struct TaylorC {
  float c[RL + 1];
};

// ---------------------------------------------------------------------------
// One block works on chunks of S = 64 samples with 256 threads as register
// tiles: thread (sg, ug) = (tid / 16, tid % 16) holds samples 4 sg .. 4 sg + 3
// by units 4 ug .. 4 ug + 3, and the three 64 x 64 x 64 contractions (z2 = W2 h1,
// dh1 = W2^T dz2, dW2 = dz2^T h1) run over two float4 shared loads per 16 FMAs.
// Everything that belongs to a tile's own points (h2, the output layer, dz2, dz1
// and the gradients of W1, W3 and the biases) stays in registers; the sixteen
// lanes that share four samples sit in one half warp, so the output layer's
// sums over units are shuffles.
//
// What bounds it: shared-memory reads (two 128-bit loads per 16 FMAs; the FMAs
// alone, 14 336 per sample forward and backward, would take 23 us of the 60 us
// below).  One thread per sample, the former layout, read one shared word per
// FMA and kept four warps per SM; here 16 warps per SM share each operand.
// Loss and gradient of 65 536 samples: 196 -> 83 us a call, of which the kernel
// 60 us.
//
// Only s_j = (o_j + o_{j+4}) / 2 enters the coefficients, so o_j + o_{j+4} is
// one sum and dL/do_j = dL/do_{j+4} is formed once.  (Adding the two weight rows
// beforehand would round each weight the same way for every sample, which
// showed in the error of loss and gradient.)
// ---------------------------------------------------------------------------
constexpr int S = 64;         // samples per chunk
constexpr int NTHR = 256;     // threads per block
constexpr int NSUB = 8;       // samples per warp: the unit in which work is dealt out

// Offsets (floats) of the block's shared memory: parameters, then (gradient
// only) W2 as stored, the activation tiles and two staged sample chunks.
constexpr int SM_W1 = 0, SM_B1 = SM_W1 + 4 * H, SM_B2 = SM_B1 + H, SM_W3 = SM_B2 + H,
              SM_B3 = SM_W3 + NOUT * H, SM_W2T = SM_B3 + NOUT, SM_H1T = SM_W2T + H * H,
              SM_W2 = SM_H1T + H * S, SM_H1 = SM_W2 + H * H, SM_D2 = SM_H1 + S * H,
              SM_D2T = SM_D2 + S * H, SM_SMP = SM_D2T + H * S,
              SM_GRAD = SM_SMP + 2 * S * SAMPLE;
static_assert(SM_W2T % 4 == 0 && SM_SMP % 4 == 0, "float4 tiles");

// Float4 block of the transposed tiles [unit][sample]: the sample blocks of a
// row are permuted by the row's unit group, so that sixteen unit groups
// writing the same sample block touch different banks.
__device__ __forceinline__ int tblk(int row, int sg) { return row * S + 4 * (sg ^ ((row >> 2) & 15)); }

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ float at4(const float4& v, int i) {
  return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

// Parameters into shared memory: W1, W3, biases, W2 transposed (W2T[i][k]) and, to keep, W2 as stored.
template <int T>
__device__ __forceinline__ void load_params(float* sm, const float* __restrict__ p, bool keep) {
  for (int i = threadIdx.x; i < 4 * H; i += T) {
    sm[SM_W1 + i] = p[OW1 + i];
    sm[SM_W3 + i] = p[OW3 + i];
    sm[SM_W3 + RL * H + i] = p[OW3 + RL * H + i];
  }
  for (int i = threadIdx.x; i < H; i += T) {
    sm[SM_B1 + i] = p[OB1 + i];
    sm[SM_B2 + i] = p[OB2 + i];
  }
  if (threadIdx.x < NOUT) sm[SM_B3 + threadIdx.x] = p[OB3 + threadIdx.x];
  // W2 by 4 x 4 blocks, transposed in registers
  static_assert(OW2 % 4 == 0, "float4 rows of W2");
#pragma unroll
  for (int e = threadIdx.x; e < H * H / 16; e += T) {
    const int kb = e & 15, ub = e >> 4;
    float4 w[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      w[r] = *reinterpret_cast<const float4*>(p + OW2 + (4 * kb + r) * H + 4 * ub);
      if (keep) *reinterpret_cast<float4*>(sm + SM_W2 + (4 * kb + r) * H + 4 * ub) = w[r];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
      st4(sm + SM_W2T + (4 * ub + r) * H + 4 * kb, at4(w[0], r), at4(w[1], r), at4(w[2], r),
          at4(w[3], r));
  }
}

// acc[s][u] += a_s b_u
__device__ __forceinline__ void outer4(float (&acc)[4][4], const float4& a, const float4& b) {
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[s][u] = fmaf(at4(a, s), at4(b, u), acc[s][u]);
}

// First layer of the thread's tile: h1 = relu(W1 x + b1) for its four samples
// and units, into the transposed tile.
__device__ __forceinline__ void layer1(float* sm, int sg, int ug, const float (&x)[4][NIN],
                                       float (&h1)[4][4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float4 w = ld4(sm + SM_W1 + 4 * (4 * ug + u));
    const float b = sm[SM_B1 + 4 * ug + u];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      float z = b;
#pragma unroll
      for (int c = 0; c < NIN; ++c) z = fmaf(at4(w, c), x[s][c], z);
      h1[s][u] = fmaxf(z, 0.0f);
    }
    st4(sm + SM_H1T + tblk(4 * ug + u, sg), h1[0][u], h1[1][u], h1[2][u], h1[3][u]);
  }
}

// acc[s][u] += sum_r T[r][sample s] W[r][unit u] over the 64 rows r of a
// transposed tile T and of W.
__device__ __forceinline__ void contract(const float* T, const float* W, int sg, int ug,
                                         float (&acc)[4][4]) {
#pragma unroll 4
  for (int r4 = 0; r4 < H / 4; ++r4) {
    const float* t = T + 4 * r4 * S + 4 * (sg ^ r4);
    const float* w = W + 4 * r4 * H + 4 * ug;
#pragma unroll
    for (int r = 0; r < 4; ++r) outer4(acc, ld4(t + r * S), ld4(w + r * H));
  }
}

// Second layer and output of the thread's tile: h2 (kept) and, in lane
// (sample 4 sg + (ug >> 2), output j = ug & 3), s_j = (o_j + o_{j+4}) / 2.
__device__ __forceinline__ float layer2_out(const float* sm, int sg, int ug, float (&h2)[4][4]) {
  const float4 b2 = ld4(sm + SM_B2 + 4 * ug);
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int u = 0; u < 4; ++u) h2[s][u] = at4(b2, u);
  contract(sm + SM_H1T, sm + SM_W2T, sg, ug, h2);
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int u = 0; u < 4; ++u) h2[s][u] = fmaxf(h2[s][u], 0.0f);
  // sums over units, reduced and scattered over the half warp: lane bits 3 and 2
  // end with the sample, bits 1 and 0 with the output
  auto fold = [&](float lo, float hi, int m) {
    const bool up = (ug & m) != 0;
    return (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, m);
  };
  float v[RL];
#pragma unroll
  for (int j = 0; j < RL; ++j) {
    const float4 w = ld4(sm + SM_W3 + j * H + 4 * ug);
    const float4 w4 = ld4(sm + SM_W3 + (j + RL) * H + 4 * ug);
    float z[4];  // this thread's share, per sample
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      z[s] = 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) z[s] = fmaf(at4(w4, u), h2[s][u], fmaf(at4(w, u), h2[s][u], z[s]));
    }
    v[j] = fold(fold(z[0], z[2], 8), fold(z[1], z[3], 8), 4);
  }
  const float o = fold(fold(v[0], v[2], 2), fold(v[1], v[3], 2), 1);
  return 0.5f * (o + (sm[SM_B3 + (ug & 3)] + sm[SM_B3 + RL + (ug & 3)]));
}

// ---------------------------------------------------------------------------
// inference: coefficients of feature rows (coef[n][4]), or of every padded cell
// of a grid, where x0 = v dt / h = sqrt(A) because A = dt^2 v^2 / h^2 and
// coefficient field j lies at coef + j * n (columns x >= Nx get the Taylor
// weights).
//
// A chunk of 128 samples on 128 threads as 8 x 8 register tiles: thread
// (sg, ug) = (tid / 8, tid % 8) holds samples 8 sg .. 8 sg + 7 by units 4 ug ..
// 4 ug + 3 and 32 + 4 ug .. 35 + 4 ug, so that a step reads four 128-bit words
// per 64 FMAs, half as many as a 4 x 4 tile (there is no gradient to keep in
// registers here; with it, 8 x 8 tiles leave eight warps per SM, and k_mlp_grad
// took 70 us instead of 60).  230 x 213 x 181 cells: 2.25 -> 1.9 ms against 4 x 4
// tiles, 1.1 ms of it FMAs.
// ---------------------------------------------------------------------------
constexpr int CS = 128, CTHR = 128;  // samples per chunk, threads
constexpr int SM_CH1T = SM_W2T + H * H, SM_COEF = SM_CH1T + H * CS;

// Float4 block h (of two) of sample group sg in row `row` of the [unit][sample]
// tile, permuted so that eight unit groups writing it touch all banks.
__device__ __forceinline__ int cblk(int row, int sg, int h) {
  return row * CS + 4 * ((2 * sg + h) ^ ((row >> 2) & 7));
}

template <bool GRID>
__global__ void __launch_bounds__(CTHR, 4)
    k_mlp_coef(const float* __restrict__ params, const float* __restrict__ in, size_t n, int pitch,
               int Nx, float x1, float x2, float x3, TaylorC t, float* __restrict__ coef) {
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, sg = tid >> 3, ug = tid & 7;
  load_params<CTHR>(sm, params, false);
  __syncthreads();
  const size_t step = size_t(gridDim.x) * CS;
  const int xstep = GRID ? int(step % pitch) : 0;
  size_t base = size_t(blockIdx.x) * CS;
  int col = GRID ? int((base + tid) % pitch) : 0;  // of the lane's own cell
  for (; base < n; base += step) {
    float x[8][NIN];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const size_t i = base + 8 * sg + s;
      if (GRID) {
        x[s][0] = i < n ? sqrtf(in[i]) : 0.f;
        x[s][1] = x1;
        x[s][2] = x2;
        x[s][3] = x3;
      } else {
#pragma unroll
        for (int c = 0; c < NIN; ++c) x[s][c] = i < n ? in[i * NIN + c] : 0.f;
      }
    }
    __syncwarp();  // a warp's samples are written and read by the warp alone
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = (u >> 2) * 32 + 4 * ug + (u & 3);
      const float4 w = ld4(sm + SM_W1 + 4 * k);
      const float b = sm[SM_B1 + k];
      float h[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        float z = b;
#pragma unroll
        for (int c = 0; c < NIN; ++c) z = fmaf(at4(w, c), x[s][c], z);
        h[s] = fmaxf(z, 0.0f);
      }
      st4(sm + SM_CH1T + cblk(k, sg, 0), h[0], h[1], h[2], h[3]);
      st4(sm + SM_CH1T + cblk(k, sg, 1), h[4], h[5], h[6], h[7]);
    }
    __syncwarp();
    float h2[8][8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int s = 0; s < 8; ++s) h2[s][u] = sm[SM_B2 + (u >> 2) * 32 + 4 * ug + (u & 3)];
#pragma unroll 2
    for (int r4 = 0; r4 < H / 4; ++r4) {
      const float* t0 = sm + SM_CH1T + cblk(4 * r4, sg, 0);
      const float* t1 = sm + SM_CH1T + cblk(4 * r4, sg, 1);
      const float* w = sm + SM_W2T + 4 * r4 * H + 4 * ug;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 a[2] = {ld4(t0 + r * CS), ld4(t1 + r * CS)};
        const float4 b[2] = {ld4(w + r * H), ld4(w + r * H + 32)};
#pragma unroll
        for (int s = 0; s < 8; ++s)
#pragma unroll
          for (int u = 0; u < 8; ++u)
            h2[s][u] = fmaf(at4(a[s >> 2], s & 3), at4(b[u >> 2], u & 3), h2[s][u]);
      }
    }
    // sums over units, reduced and scattered over the eight lanes: lane ug ends
    // with the outputs of sample 8 sg + ug
    auto fold = [&](float lo, float hi, int m) {
      const bool up = (ug & m) != 0;
      return (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, m);
    };
#pragma unroll
    for (int s = 0; s < 8; ++s)
#pragma unroll
      for (int u = 0; u < 8; ++u) h2[s][u] = fmaxf(h2[s][u], 0.0f);
    const size_t i = base + tid;
#pragma unroll
    for (int j = 0; j < RL; ++j) {
      float z[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) z[s] = 0.f;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const float4 w = ld4(sm + SM_W3 + j * H + 32 * hf + 4 * ug);
        const float4 w4 = ld4(sm + SM_W3 + (j + RL) * H + 32 * hf + 4 * ug);
#pragma unroll
        for (int s = 0; s < 8; ++s)
#pragma unroll
          for (int u = 0; u < 4; ++u)
            z[s] = fmaf(at4(w4, u), h2[s][4 * hf + u], fmaf(at4(w, u), h2[s][4 * hf + u], z[s]));
      }
      const float o = fold(fold(fold(z[0], z[4], 4), fold(z[2], z[6], 4), 2),
                           fold(fold(z[1], z[5], 4), fold(z[3], z[7], 4), 2), 1);
      const float sj = 0.5f * (o + (sm[SM_B3 + j] + sm[SM_B3 + RL + j]));
      if (i < n) {
        const float c = t.c[j + 1] * (1.0f + 0.5f * tanhf(sj));
        if (GRID)
          coef[j * n + i] = col < Nx ? c : t.c[j + 1];
        else
          coef[i * RL + j] = c;
      }
    }
    if (GRID) {
      col += xstep;
      if (col >= pitch) col -= pitch;
    }
  }
}

// ---------------------------------------------------------------------------
// training: fused forward, loss and backward.  Block b of B takes the NSUB-sample
// units [b U / B, (b + 1) U / B) of the U units in chunks of S; warps whose
// samples lie beyond the last chunk's end skip it.  The gradient of W2 (64 x 64)
// is accumulated in the register tile, all others per tile; a block leaves its
// sums, NPARAM floats, in part[block] and its warps' losses in lpart[block], and
// k_mlp_sum adds the blocks up.
// ---------------------------------------------------------------------------
constexpr int NWARP = NTHR / 32;
__device__ __forceinline__ void put4(float* p, const float4& v) {
  *reinterpret_cast<float4*>(p) = v;
}

__global__ void __launch_bounds__(NTHR, 2)
    k_mlp_grad(const float* __restrict__ params, const float* __restrict__ samples, int n,
               float inv_n, TaylorC t, float* __restrict__ part, double* __restrict__ lpart) {
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, sg = tid >> 4, ug = tid & 15, j = ug & 3;
  float* grad = part + size_t(blockIdx.x) * NPARAM;
  pdl_trigger();
  const long long units = (static_cast<long long>(n) + NSUB - 1) / NSUB;
  const long long lo = units * blockIdx.x / gridDim.x * NSUB;
  long long hi = units * (blockIdx.x + 1) / gridDim.x * NSUB;
  if (hi > n) hi = n;
  constexpr int NST = (S * SAMPLE + NTHR - 1) / NTHR;  // staged floats per thread
  auto fetch = [&](long long base, float (&r)[NST]) {
#pragma unroll
    for (int q = 0; q < NST; ++q) {
      const int e = tid + q * NTHR;
      const bool ok = e < S * SAMPLE && base * SAMPLE + e < hi * SAMPLE;
      r[q] = ok ? samples[base * SAMPLE + e] : 0.f;
    }
  };
  auto stage = [&](int buf, const float (&r)[NST]) {
#pragma unroll
    for (int q = 0; q < NST; ++q) {
      const int e = tid + q * NTHR;
      if (e < S * SAMPLE) sm[SM_SMP + buf * S * SAMPLE + e] = r[q];
    }
  };
  float nxt[NST];
  fetch(lo, nxt);
  load_params<NTHR>(sm, params, true);
  const float tc = t.c[j + 1];
  float a1[4][4], a2[4][4], a3[4][4], ab1[4], ab2[4], ab3 = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    ab1[q] = ab2[q] = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) a1[q][r] = a2[q][r] = a3[q][r] = 0.f;
  }
  double lsum = 0.0;
  stage(0, nxt);
  __syncthreads();

  int buf = 0;
  for (long long base = lo; base < hi; base += S, buf ^= 1) {
    const int nv = hi - base < S ? static_cast<int>(hi - base) : S;
    const bool more = base + S < hi;
    if (more) fetch(base + S, nxt);
    const float* smp = sm + SM_SMP + buf * S * SAMPLE;
    const bool live = (tid >> 5) * NSUB < nv;  // uniform in a warp
    unsigned m1 = 0;                           // h1 > 0, bit 4 s + u
    if (live) {
      float x[4][NIN], h1[4][4];
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < NIN; ++c) x[s][c] = smp[(4 * sg + s) * SAMPLE + c];
      layer1(sm, sg, ug, x, h1);
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        st4(sm + SM_H1 + (4 * sg + s) * H + 4 * ug, h1[s][0], h1[s][1], h1[s][2], h1[s][3]);
#pragma unroll
        for (int u = 0; u < 4; ++u) m1 |= h1[s][u] > 0.f ? 1u << (4 * s + u) : 0u;
      }
      // a warp's samples of the transposed tiles are read by the warp alone
      __syncwarp();
      float h2[4][4];
      const float sj = layer2_out(sm, sg, ug, h2);
      // loss and dL/do_j (= dL/do_{j+4}) of sample 4 sg + (ug >> 2)
      const float* own = smp + (4 * sg + (ug >> 2)) * SAMPLE;
      const float T = own[NIN + j], y = own[NIN + RL], w = own[NIN + RL + 1];
      const float th = tanhf(sj);
      float p = tc * (1.0f + 0.5f * th) * T;
      p += __shfl_xor_sync(0xffffffffu, p, 1);
      p += __shfl_xor_sync(0xffffffffu, p, 2);
      const float r = p - y;
      if (j == 0) lsum += double(w) * double(r) * double(r);
      const float dp = 2.0f * w * r * inv_n;
      const float dout = 0.5f * (dp * T * tc * 0.5f * (1.0f - th * th));
      ab3 += dout;
      // dz2 and the gradients of W3 and b2
      float dz[4][4];
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int u = 0; u < 4; ++u) dz[s][u] = 0.f;
#pragma unroll
      for (int jj = 0; jj < RL; ++jj) {
        const float4 w3 = ld4(sm + SM_W3 + jj * H + 4 * ug);
        const float4 w34 = ld4(sm + SM_W3 + (jj + RL) * H + 4 * ug);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float d = __shfl_sync(0xffffffffu, dout, 4 * s + jj, 16);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            dz[s][u] = fmaf(at4(w34, u), d, fmaf(at4(w3, u), d, dz[s][u]));
            a3[jj][u] = fmaf(d, h2[s][u], a3[jj][u]);
          }
        }
      }
#pragma unroll
      for (int s = 0; s < 4; ++s) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          dz[s][u] = h2[s][u] > 0.f ? dz[s][u] : 0.f;
          ab2[u] += dz[s][u];
        }
        st4(sm + SM_D2 + (4 * sg + s) * H + 4 * ug, dz[s][0], dz[s][1], dz[s][2], dz[s][3]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        st4(sm + SM_D2T + tblk(4 * ug + u, sg), dz[0][u], dz[1][u], dz[2][u], dz[3][u]);
      __syncwarp();
      // dz1 and the gradients of W1 and b1
      float d1[4][4];
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int u = 0; u < 4; ++u) d1[s][u] = 0.f;
      contract(sm + SM_D2T, sm + SM_W2, sg, ug, d1);
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        float xs[NIN];
#pragma unroll
        for (int c = 0; c < NIN; ++c) xs[c] = smp[(4 * sg + s) * SAMPLE + c];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float d = (m1 >> (4 * s + u)) & 1u ? d1[s][u] : 0.f;
          ab1[u] += d;
#pragma unroll
          for (int c = 0; c < NIN; ++c) a1[u][c] = fmaf(d, xs[c], a1[u][c]);
        }
      }
    }
    __syncthreads();
    // dW2 over the chunk's samples, in units of a warp's samples (those beyond
    // the end within a unit carry w = 0, so dz2 = 0)
    {
      const int nr = (nv + NSUB - 1) / NSUB * NSUB;
      const float* D = sm + SM_D2 + 4 * sg;
      const float* Hs = sm + SM_H1 + 4 * ug;
      for (int s = 0; s < nr; s += NSUB)
#pragma unroll
        for (int q = 0; q < NSUB; ++q) outer4(a2, ld4(D + (s + q) * H), ld4(Hs + (s + q) * H));
    }
    if (more) stage(buf ^ 1, nxt);
    __syncthreads();
  }

  // dW2[4 sg + q][4 ug ..]
#pragma unroll
  for (int q = 0; q < 4; ++q)
    put4(grad + OW2 + (4 * sg + q) * H + 4 * ug, make_float4(a2[q][0], a2[q][1], a2[q][2], a2[q][3]));
  // the others: sums over the sixteen sample groups through shared memory
  // (the activation tiles are free now), as 161 float4 entries [entry][sg]
  float* R = sm + SM_W2T;
  constexpr int E1 = 64, EB1 = 128, EB2 = 144, EB3 = 160, NE = 161;
  static_assert(NE * 64 <= SM_GRAD - SM_W2T, "reduction scratch");
  auto put = [&](int e, float a, float b, float c, float d) { st4(R + e * 64 + 4 * sg, a, b, c, d); };
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    put(q * 16 + ug, a3[q][0], a3[q][1], a3[q][2], a3[q][3]);
    put(E1 + 4 * ug + q, a1[q][0], a1[q][1], a1[q][2], a1[q][3]);
  }
  put(EB1 + ug, ab1[0], ab1[1], ab1[2], ab1[3]);
  put(EB2 + ug, ab2[0], ab2[1], ab2[2], ab2[3]);
  ab3 += __shfl_xor_sync(0xffffffffu, ab3, 4);
  ab3 += __shfl_xor_sync(0xffffffffu, ab3, 8);
  if (ug < 4) R[EB3 * 64 + 4 * sg + ug] = ab3;
  __syncthreads();
  if (tid < NE) {
    float4 v = ld4(R + tid * 64);
    for (int q = 1; q < 16; ++q) {
      const float4 o = ld4(R + tid * 64 + 4 * q);
      v.x += o.x;
      v.y += o.y;
      v.z += o.z;
      v.w += o.w;
    }
    if (tid < E1) {  // rows j and j + 4 of W3 share their gradient
      put4(grad + OW3 + 4 * tid, v);
      put4(grad + OW3 + RL * H + 4 * tid, v);
    } else if (tid < EB1) {
      put4(grad + OW1 + 4 * (tid - E1), v);
    } else if (tid < EB2) {
      put4(grad + OB1 + 4 * (tid - EB1), v);
    } else if (tid < EB3) {
      put4(grad + OB2 + 4 * (tid - EB2), v);
    } else {
      put4(grad + OB3, v);
      put4(grad + OB3 + RL, v);
    }
  }
  for (int off = 16; off > 0; off >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, off);
  if ((tid & 31) == 0) lpart[blockIdx.x * NWARP + (tid >> 5)] = lsum * double(inv_n);
}

// Sums of the blocks' gradients and losses.  Block b sums words [32 b, 32 b + 32)
// of the gradient (8 threads side by side on a float4 each, 32 rows of blocks at
// a time, 5 rows ahead), the last block the losses.  Every sum is kept as hi + lo (Knuth's
// two-sum, whose error term is exact), so that it adds one rounding whatever the
// number of blocks.  Adding each block's sums to the words in global memory rounds
// once per block: relative error of the gradient against FP64, mean of four to six
// seeds, 1050 / 65 536 samples: 1.9e-7 / 2.5e-7 so, 0.95e-7 / 1.8e-7 with one block
// of 128 samples per SM, 0.56e-7 / 0.55e-7 with this sum.  The call takes no longer than
// with the additions: they cost the training kernel what this launch costs behind it.  FP64 sums would be as exact;
// this GPU does about 2 of them per SM and clock.
constexpr int SW = 8, SR = 32;  // float4 words and rows of a block
__device__ __forceinline__ void two_sum(float& hi, float& lo, float v) {
  const float s = __fadd_rn(hi, v), b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(v, b)));
  hi = s;
}

__global__ void __launch_bounds__(SW* SR)
    k_mlp_sum(const float* __restrict__ part, const double* __restrict__ lpart, int blocks,
              float* __restrict__ grad, double* __restrict__ loss) {
  const int tid = threadIdx.x;
  pdl_wait();
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double warp[SW * SR / 32];
    double v = 0.0;
    for (int i = tid; i < blocks * NWARP; i += SW * SR) v += lpart[i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((tid & 31) == 0) warp[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
      for (int i = 1; i < SW * SR / 32; ++i) v += warp[i];
      *loss = v;
    }
    return;
  }
  __shared__ float hi_of[SR / 4][4 * SW], lo_of[SR / 4][4 * SW];
  const int q = tid % SW, row = tid / SW;
  const int w = (blockIdx.x * SW + q) * 4;
  float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
  if (w < NPARAM) {
    constexpr int kAhead = 5;  // loads in flight: 304 blocks are two rounds
    for (int b = row; b < blocks; b += kAhead * SR) {
      float4 v[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k)
        v[k] = b + k * SR < blocks ? ld4(part + size_t(b + k * SR) * NPARAM + w)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < kAhead; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i) two_sum(hi[i], lo[i], at4(v[k], i));
    }
  }
  // the warp's four rows, then the warps
#pragma unroll
  for (int o = SW; o < 32; o *= 2)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float l = __shfl_xor_sync(0xffffffffu, lo[i], o);
      two_sum(hi[i], lo[i], __shfl_xor_sync(0xffffffffu, hi[i], o));
      lo[i] = __fadd_rn(lo[i], l);
    }
  if ((row & 3) == 0) {
    st4(&hi_of[row / 4][4 * q], hi[0], hi[1], hi[2], hi[3]);
    st4(&lo_of[row / 4][4 * q], lo[0], lo[1], lo[2], lo[3]);
  }
  __syncthreads();
  if (tid >= 4 * SW || blockIdx.x * 4 * SW + tid >= NPARAM) return;
  float h = 0.f, l = 0.f;
#pragma unroll
  for (int r = 0; r < SR / 4; ++r) {
    two_sum(h, l, hi_of[r][tid]);
    l = __fadd_rn(l, lo_of[r][tid]);
  }
  // (an overflow or a NaN leaves its mark in h; the error term is then NaN)
  grad[blockIdx.x * 4 * SW + tid] = isfinite(h) ? __fadd_rn(h, l) : h;
}

// Adam (Kingma & Ba, ICLR 2015) with bias correction; step t >= 1.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Stencil values of sampled cells: out[n][1 + 6 rad] = centre, then for
// j = 1..rad the neighbours at -j s and +j s along x, y and z (s = stride);
// cells are padded (x, y, z) indices, outside the grid reads as 0.
__global__ void k_sample_stencil(const float* __restrict__ u, int Nx, int Ny, int Nz, int pitch,
                                 const int* __restrict__ cells, int n, int stride, int rad,
                                 float* __restrict__ out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int x = cells[3 * s], y = cells[3 * s + 1], z = cells[3 * s + 2];
  auto at = [&](int xx, int yy, int zz) -> float {
    if (xx < 0 || yy < 0 || zz < 0 || xx >= Nx || yy >= Ny || zz >= Nz) return 0.0f;
    return u[(size_t(zz) * Ny + yy) * pitch + xx];
  };
  const int w = 1 + 6 * rad;
  float* o = out + size_t(s) * w;
  o[0] = at(x, y, z);
  for (int j = 1; j <= rad; ++j) {
    const int d = j * stride;
    o[6 * (j - 1) + 1] = at(x - d, y, z);
    o[6 * (j - 1) + 2] = at(x + d, y, z);
    o[6 * (j - 1) + 3] = at(x, y - d, z);
    o[6 * (j - 1) + 4] = at(x, y + d, z);
    o[6 * (j - 1) + 5] = at(x, y, z - d);
    o[6 * (j - 1) + 6] = at(x, y, z + d);
  }
}

// Training samples from three stencil snapshots at coarse times t-dt, t,
// t+dt: T_j = sum of the six values at distance j - 6 u, target
// y = (u+ - 2u + u-) / C^2 with C = v dt / h, so that the coarse update
// u+ = 2u - u- + C^2 sum_j c_j T_j reproduces the fine solution; weight
// w = 1 / (scale + mean of the squared stencil values).
__global__ void k_make_samples(const float* __restrict__ prev, const float* __restrict__ cur,
                               const float* __restrict__ next, const float* __restrict__ vel,
                               int n, float h, float dt, float f, float scale,
                               float* __restrict__ out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int w = 1 + 6 * RL;
  const float* c = cur + size_t(s) * w;
  const float u = c[0];
  float* o = out + size_t(s) * SAMPLE;
  const float C = vel[s] * dt / h;
  o[0] = C;
  o[1] = h / 10.0f;
  o[2] = dt / 1.0f;
  o[3] = f / 10.0f;
  float ms = u * u;
  for (int j = 1; j <= RL; ++j) {
    float sum = 0.f;
    for (int q = 1; q <= 6; ++q) {
      const float v = c[6 * (j - 1) + q];
      sum += v;
      ms += v * v;
    }
    o[NIN + j - 1] = sum - 6.0f * u;
  }
  o[NIN + RL] = (next[size_t(s) * w] - 2.0f * u + prev[size_t(s) * w]) / (C * C);
  o[NIN + RL + 1] = 1.0f / (scale + ms / float(w));
}

TaylorC taylor_c() {
  TaylorC t;
  double c[RL + 1], sum = 0.0;
  for (int j = 1; j <= RL; ++j) {
    double ratio = 1.0;
    for (int k = 1; k <= j; ++k) ratio *= double(RL - k + 1) / double(RL + k);
    c[j] = ((j & 1) ? 2.0 : -2.0) * ratio / (double(j) * j);
    sum += c[j];
  }
  c[0] = -2.0 * sum;
  for (int j = 0; j <= RL; ++j) t.c[j] = float(c[j]);
  return t;
}

// The inference kernels' dynamic shared memory, above the default limit.
fd_status coef_attr() {
  cudaError_t e = cudaFuncSetAttribute(k_mlp_coef<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(SM_COEF * sizeof(float)));
  if (!e)
    e = cudaFuncSetAttribute(k_mlp_coef<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(SM_COEF * sizeof(float)));
  return e ? cuda_fail(e, "kernel attribute") : FD_OK;
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

}  // namespace

// gradient and, behind it, the loss: one read for both
constexpr size_t GRAD_BYTES = NPARAM * 4 + sizeof(double);
static_assert(NPARAM * 4 % sizeof(double) == 0, "loss alignment");

struct fd_mlp_s {
  int device = 0;
  cudaStream_t stream = nullptr;
  void* mem = nullptr;  // one allocation for all of the following
  float* p = nullptr;   // params
  float* g = nullptr;   // gradient
  float* m = nullptr;   // Adam first moment
  float* v = nullptr;   // Adam second moment
  double* loss = nullptr;  // behind the gradient
  double* lpart = nullptr;  // losses and gradient sums of the training kernel's blocks,
  float* part = nullptr;    // for as many blocks as it launches at most
  int most_blocks = 0;
  std::vector<float> host;  // image of gradient and loss
  int t = 0;               // Adam step count
  DevBuf stage, stage2;
};

namespace fd {

fd_status mlp_grid_coefficients(fd_mlp net, const float* A, size_t ncell, int pitch, int Nx,
                                double h, double dt, double f_hz, float* coef,
                                cudaStream_t s) {
  const TaylorC t = taylor_c();
  const fd_status st = coef_attr();
  if (st) return st;
  const int grid =
      int(std::max<size_t>(1, std::min<size_t>(size_t(sm_count()) * 4, (ncell + CS - 1) / CS)));
  k_mlp_coef<true><<<grid, CTHR, SM_COEF * sizeof(float), s>>>(
      net->p, A, ncell, pitch, Nx, float(h / 10.0), float(dt / 1.0), float(f_hz / 10.0), t, coef);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e) return cuda_fail(e, "learned coefficient inference");
  return FD_OK;
}

}  // namespace fd

extern "C" {

fd_status fd_mlp_create(int32_t device, const float* params, fd_mlp* out) {
  clear_error();
  if (!out) return fail(FD_ERR_ARG, "null argument");
  *out = nullptr;
  cudaError_t e = cudaSetDevice(device);
  if (e) return cuda_fail(e, "cudaSetDevice");
  fd_mlp net = new fd_mlp_s();
  net->device = device;
  fd_status st = FD_OK;
  e = cudaStreamCreateWithFlags(&net->stream, cudaStreamDefault);  // see fd_create_grid
  float** bufs[4] = {&net->p, &net->g, &net->m, &net->v};
  constexpr size_t kField = (GRAD_BYTES + 255) / 256 * 256;
  net->most_blocks = 2 * std::max(1, sm_count());  // two per SM
  if (!e)
    e = dev_alloc(&net->mem, 4 * kField + size_t(net->most_blocks) *
                                              (NPARAM * 4 + NWARP * sizeof(double)));
  if (!e) {
    char* q = static_cast<char*>(net->mem);
    for (int i = 0; i < 4; ++i, q += kField) *bufs[i] = reinterpret_cast<float*>(q);
    net->lpart = reinterpret_cast<double*>(q);
    net->part = reinterpret_cast<float*>(net->lpart + size_t(net->most_blocks) * NWARP);
    net->loss = reinterpret_cast<double*>(net->g + NPARAM);
    net->host.resize(GRAD_BYTES / sizeof(float));
    for (int i = 0; i < 4 && !e; ++i) e = cudaMemsetAsync(*bufs[i], 0, NPARAM * 4, net->stream);
    if (!e && params) e = cudaMemcpyAsync(net->p, params, NPARAM * 4, cudaMemcpyDefault,
                                          net->stream);
    if (!e) e = cudaStreamSynchronize(net->stream);
  }
  if (e) st = cuda_fail(e, "network allocation");
  if (st) {
    fd_mlp_destroy(net);
    return st;
  }
  *out = net;
  return FD_OK;
}

fd_status fd_mlp_destroy(fd_mlp net) {
  if (!net) return FD_OK;
  cudaSetDevice(net->device);
  if (net->stream) cudaStreamSynchronize(net->stream);
  if (net->mem) cudaFree(net->mem);
  net->stage.release();
  net->stage2.release();
  if (net->stream) cudaStreamDestroy(net->stream);
  delete net;
  return FD_OK;
}

fd_status fd_mlp_get_params(fd_mlp net, float* out) {
  clear_error();
  if (!net || !out) return fail(FD_ERR_ARG, "null argument");
  cudaSetDevice(net->device);
  cudaError_t e = cudaMemcpyAsync(out, net->p, NPARAM * 4, cudaMemcpyDefault, net->stream);
  if (!e) e = cudaStreamSynchronize(net->stream);
  if (e) return cuda_fail(e, "parameter read");
  return FD_OK;
}

fd_status fd_mlp_set_params(fd_mlp net, const float* in) {
  clear_error();
  if (!net || !in) return fail(FD_ERR_ARG, "null argument");
  cudaSetDevice(net->device);
  cudaError_t e = cudaMemcpyAsync(net->p, in, NPARAM * 4, cudaMemcpyDefault, net->stream);
  if (!e) e = cudaMemsetAsync(net->m, 0, NPARAM * 4, net->stream);
  if (!e) e = cudaMemsetAsync(net->v, 0, NPARAM * 4, net->stream);
  if (!e) e = cudaStreamSynchronize(net->stream);
  if (e) return cuda_fail(e, "parameter write");
  net->t = 0;
  return FD_OK;
}

static fd_status mlp_grad_device(fd_mlp net, int64_t n, const float* dsamples) {
  cudaError_t e = cudaSuccess;
  if (n == 0) {
    e = cudaMemsetAsync(net->g, 0, GRAD_BYTES, net->stream);
    return e ? cuda_fail(e, "gradient reset") : FD_OK;
  }
  static bool attr = false;
  if (!attr) {
    e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(SM_GRAD * sizeof(float)));
    if (e) return cuda_fail(e, "kernel attribute");
    attr = true;
  }
  // One block per SM up to four chunks each: its eight warps take a chunk's units
  // side by side, and every block is one more row to sum.  Two per SM beyond (us a
  // call, one / two: 2009 samples 43.5 / 54.6, 8192 46.2 / 55.9, 20 000 58.2 / 68.4,
  // 36 000 71.5 / 72.9, 65 536 93.2 / 92.4, 300 000 289 / 254).  A small batch is
  // spread one warp's samples per block.
  const int sms = net->most_blocks / 2;
  const int most = n <= int64_t(4) * S * sms ? sms : 2 * sms;
  const int blocks = int(std::min<int64_t>(most, (n + NSUB - 1) / NSUB));
  k_mlp_grad<<<blocks, NTHR, SM_GRAD * sizeof(float), net->stream>>>(
      net->p, dsamples, int(n), float(1.0 / double(n)), taylor_c(), net->part, net->lpart);
  count_launch(2);
  e = cudaGetLastError();
  // (may start while the last blocks of the training kernel run: it waits itself)
  if (!e)
    e = launch_step(k_mlp_sum, dim3((NPARAM + 4 * SW - 1) / (4 * SW) + 1), SW * SR, 0, true,
                    net->stream, static_cast<const float*>(net->part),
                    static_cast<const double*>(net->lpart), blocks, net->g, net->loss);
  if (e) return cuda_fail(e, "training kernel");
  return FD_OK;
}

// Loss and (grad not null) gradient of the last mlp_grad_device to the caller.
static fd_status mlp_grad_read(fd_mlp net, double* loss, float* grad) {
  cudaError_t e = cudaSuccess;
  const bool dev = grad && is_device_ptr(grad);
  if (dev) e = cudaMemcpyAsync(grad, net->g, NPARAM * 4, cudaMemcpyDeviceToDevice, net->stream);
  if (!e && (loss || (grad && !dev)))
    e = cudaMemcpyAsync(net->host.data(), net->g, GRAD_BYTES, cudaMemcpyDeviceToHost, net->stream);
  if (!e) e = cudaStreamSynchronize(net->stream);
  if (e) return cuda_fail(e, "gradient read");
  if (loss) memcpy(loss, net->host.data() + NPARAM, sizeof(double));
  if (grad && !dev) memcpy(grad, net->host.data(), NPARAM * 4);
  return FD_OK;
}

fd_status fd_mlp_loss_grad(fd_mlp net, int64_t n, const float* samples, double* loss,
                           float* grad_out) {
  clear_error();
  if (!net || (n > 0 && !samples)) return fail(FD_ERR_ARG, "null argument");
  if (n < 0 || n > INT32_MAX) return fail(FD_ERR_ARG, "bad sample count");
  cudaSetDevice(net->device);
  const float* d = samples;
  if (n > 0 && !is_device_ptr(samples)) {
    cudaError_t e = net->stage.ensure(size_t(n) * SAMPLE * 4);
    if (!e) e = cudaMemcpyAsync(net->stage.p, samples, size_t(n) * SAMPLE * 4,
                                cudaMemcpyHostToDevice, net->stream);
    if (e) return cuda_fail(e, "sample upload");
    d = static_cast<const float*>(net->stage.p);
  }
  fd_status st = mlp_grad_device(net, n, d);
  if (st || (!loss && !grad_out)) return st;
  return mlp_grad_read(net, loss, grad_out);
}

static fd_status adam_device(fd_mlp net, float lr) {
  net->t += 1;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = float(1.0 - pow(0.9, net->t)), c2 = float(1.0 - pow(0.999, net->t));
  k_adam<<<(NPARAM + 255) / 256, 256, 0, net->stream>>>(net->p, net->g, net->m, net->v, NPARAM,
                                                       lr, b1, b2, eps, c1, c2);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e) return cuda_fail(e, "adam");
  return FD_OK;
}

fd_status fd_mlp_adam_step(fd_mlp net, float lr) {
  clear_error();
  if (!net || !(lr > 0.f)) return fail(FD_ERR_ARG, "bad argument");
  cudaSetDevice(net->device);
  fd_status st = adam_device(net, lr);
  if (st) return st;
  cudaError_t e = cudaStreamSynchronize(net->stream);
  if (e) return cuda_fail(e, "adam");
  return FD_OK;
}

fd_status fd_mlp_train(fd_mlp net, int64_t n, const float* samples, int32_t epochs,
                       int32_t batch, float lr, double* loss_out) {
  clear_error();
  if (!net || !samples || n <= 0 || epochs < 0 || batch <= 0 || !(lr > 0.f))
    return fail(FD_ERR_ARG, "bad argument");
  cudaSetDevice(net->device);
  const float* d = samples;
  if (!is_device_ptr(samples)) {
    cudaError_t e = net->stage.ensure(size_t(n) * SAMPLE * 4);
    if (!e) e = cudaMemcpyAsync(net->stage.p, samples, size_t(n) * SAMPLE * 4,
                                cudaMemcpyHostToDevice, net->stream);
    if (e) return cuda_fail(e, "sample upload");
    d = static_cast<const float*>(net->stage.p);
  }
  fd_status st;
  for (int ep = 0; ep < epochs; ++ep) {
    for (int64_t b0 = 0; b0 < n; b0 += batch) {
      const int64_t nb = std::min<int64_t>(batch, n - b0);
      if ((st = mlp_grad_device(net, nb, d + size_t(b0) * SAMPLE))) return st;
      if ((st = adam_device(net, lr))) return st;
    }
  }
  if (loss_out) {
    // loss of the whole set with the final parameters
    double total = 0.0;
    for (int64_t b0 = 0; b0 < n; b0 += (int64_t(1) << 24)) {
      const int64_t nb = std::min<int64_t>(int64_t(1) << 24, n - b0);
      double l = 0.0;
      if ((st = mlp_grad_device(net, nb, d + size_t(b0) * SAMPLE))) return st;
      if ((st = mlp_grad_read(net, &l, nullptr))) return st;
      total += l * double(nb);
    }
    *loss_out = total / double(n);
  }
  cudaError_t e = cudaStreamSynchronize(net->stream);
  if (e) return cuda_fail(e, "training");
  return FD_OK;
}

fd_status fd_mlp_coefficients(fd_mlp net, int64_t n, const float* features, float* coef_out) {
  clear_error();
  if (!net || (n > 0 && (!features || !coef_out))) return fail(FD_ERR_ARG, "null argument");
  cudaSetDevice(net->device);
  if (n == 0) return FD_OK;
  const float* fin = features;
  float* cout = coef_out;
  cudaError_t e = cudaSuccess;
  if (!is_device_ptr(features)) {
    e = net->stage.ensure(size_t(n) * NIN * 4);
    if (!e) e = cudaMemcpyAsync(net->stage.p, features, size_t(n) * NIN * 4,
                                cudaMemcpyHostToDevice, net->stream);
    fin = static_cast<const float*>(net->stage.p);
  }
  const bool host_out = !is_device_ptr(coef_out);
  if (!e && host_out) {
    e = net->stage2.ensure(size_t(n) * RL * 4);
    cout = static_cast<float*>(net->stage2.p);
  }
  if (e) return cuda_fail(e, "staging");
  const fd_status st = coef_attr();
  if (st) return st;
  const int grid = int(std::min<int64_t>(sm_count() * 4, (n + CS - 1) / CS));
  k_mlp_coef<false><<<grid, CTHR, SM_COEF * sizeof(float), net->stream>>>(
      net->p, fin, size_t(n), 1, 1, 0.f, 0.f, 0.f, taylor_c(), cout);
  count_launch();
  if ((e = cudaGetLastError())) return cuda_fail(e, "inference");
  if (host_out)
    e = cudaMemcpyAsync(coef_out, cout, size_t(n) * RL * 4, cudaMemcpyDeviceToHost, net->stream);
  if (!e) e = cudaStreamSynchronize(net->stream);
  if (e) return cuda_fail(e, "inference");
  return FD_OK;
}

fd_status fd_sample_stencil(fd_grid g, int32_t n, const int32_t* cells, int32_t stride,
                            int32_t radius, float* out) {
  clear_error();
  if (!g || (n > 0 && (!cells || !out)) || n < 0 || stride < 1 || radius < 0 || radius > 8)
    return fail(FD_ERR_ARG, "bad argument");
  if (n == 0) return FD_OK;
  cudaSetDevice(g->d.device);
  const size_t w = 1 + 6 * size_t(radius);
  cudaError_t e = g->stage_aux.ensure(size_t(n) * 3 * 4 + 256 + size_t(n) * w * 4);
  if (e) return cuda_fail(e, "staging");
  int* dcells = static_cast<int*>(g->stage_aux.p);
  float* dout = reinterpret_cast<float*>(static_cast<char*>(g->stage_aux.p) +
                                         ((size_t(n) * 12 + 255) / 256) * 256);
  e = cudaMemcpyAsync(dcells, cells, size_t(n) * 12, cudaMemcpyDefault, g->stream);
  if (e) return cuda_fail(e, "cell upload");
  float* target = is_device_ptr(out) ? out : dout;
  k_sample_stencil<<<(n + 127) / 128, 128, 0, g->stream>>>(g->F.u[g->F.cur], g->Nx, g->Ny, g->Nz,
                                                          g->pitch, dcells, n, stride, radius,
                                                          target);
  count_launch();
  if ((e = cudaGetLastError())) return cuda_fail(e, "stencil sampling");
  if (target != out)
    e = cudaMemcpyAsync(out, target, size_t(n) * w * 4, cudaMemcpyDeviceToHost, g->stream);
  if (!e) e = cudaStreamSynchronize(g->stream);
  if (e) return cuda_fail(e, "stencil sampling");
  return FD_OK;
}

fd_status fd_mlp_make_samples(int32_t n, const float* prev, const float* cur, const float* next,
                              const float* vel, double h, double dt, double f_hz, double scale,
                              float* out) {
  clear_error();
  if (n < 0 || (n > 0 && (!prev || !cur || !next || !vel || !out)))
    return fail(FD_ERR_ARG, "bad argument");
  if (n == 0) return FD_OK;
  for (const void* p : {(const void*)prev, (const void*)cur, (const void*)next,
                        (const void*)vel, (const void*)out})
    if (!is_device_ptr(p)) return fail(FD_ERR_ARG, "fd_mlp_make_samples takes device arrays");
  k_make_samples<<<(n + 127) / 128, 128>>>(prev, cur, next, vel, n, float(h), float(dt),
                                           float(f_hz), float(scale), out);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (!e) e = cudaDeviceSynchronize();
  if (e) return cuda_fail(e, "sample assembly");
  return FD_OK;
}

}  // extern "C"
