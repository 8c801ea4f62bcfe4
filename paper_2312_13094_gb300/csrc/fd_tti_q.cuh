// TTI step with register queues and TMA staging (included by fd_tti.cu;
// Sec. IV-B and App. A, Eq. rot).
//
// The two wavefields are stored interleaved, float2 (p, q) per cell, and every
// stencil operation runs on the pair as one packed f32x2 instruction: both
// fields take the same weights, so no lane ever needs a neighbour's half.
// One point per thread, one warp per tile row, a CTA streaming runs of z planes.
// Every derivative is split by what it needs:
//  * the in-plane terms of a plane need only that plane, so they are formed
//    once, when the plane enters (p = k + R for output plane k): D_xx, D_yy,
//    the first differences dx and dy, and D_xy as the x difference of dy.
//    dy of the tile and of R columns on each side goes through shared memory
//    (two buffers); the halo costs 2R columns on 32, where differences of dx
//    rows would cost 2R rows on the tile's 4.  With the axis (nx, ny) of the
//    entering plane they are folded at once into what the update needs,
//    D_xx p + D_yy p and the in-plane part of H_z of both fields, which wait R
//    planes in register queues (three floats per plane instead of six);
//  * the z terms D_zz, D_xz and D_yz are sums over planes k-R .. k+R of the
//    thread's own (p, q), dx and dy, which live in register queues of 2R+1
//    entries.
// Shared memory holds a ring of four slots, each with one entering plane, its
// halo and its (nx, ny), and the update's per-point values of the output plane
// 2R planes behind (the model and the previous p and q; L2 evict-first), all
// TMA tiles on one mbarrier, and the dy scratch.  The z loop runs four planes
// per trip, so that a slot's addresses are constants of the code and three of
// four planes rename the queues instead of shifting them.  Loads outside the
// grid are zero-filled by the TMA unit (the zero ghost).
//
// A launch is persistent.  The tile columns are numbered along y first.  While
// there are G of them left for the G CTAs, each CTA streams one whole column,
// in step with its neighbours, whose halos it then finds in L2; the rest is
// cut into G equal contiguous shares of (column, plane) units.
//
// What bounds it (ncu, 336^3 at SO 8): shared-memory reads and latency; the
// shared-memory pipe is 66 % busy, issue 59 %, DRAM 63 % of the copy rate at 1.12 x
// the 48 B per point.  The scalar kernel with separate fields that this replaced
// executed 523 instructions per point at SO 8 and 902 at SO 16, this one 280 and
// 422: 100 steps of 336^3 at SO 8 80.7 -> 46.9 ms (80.9 Gpts/s), 60 steps of
// 243 x 181 x 207 at SO 16 31.6 -> 12.9 ms (42.3 Gpts/s).  Equal shares of all
// columns instead of whole waves read 1.67 x the bytes (50.5 ms).
//
// Every mbarrier wait is bounded.  A thread whose wait runs out records an
// error and stops waiting (its later waits return at once), the producer stops
// issuing, and the CTA leaves at the end of the run after a bounded wait for
// its copies in flight.
#pragma once

#include <type_traits>

#include "fd_step.cuh"

namespace fd {
namespace tti {

// Tile and threads: one warp per row of 32 cells, four rows.  Small CTAs keep
// the per-plane barrier among four warps; eight rows (less halo per tile, half
// the CTAs) measured 47.7 against 45.9 ms for 100 steps of 336^3 at SO 8, and
// 14.2 against 13.3 ms for 60 steps of 243 x 181 x 207 at SO 16.
constexpr int kQX = 32, kQY = 4, kQT = kQX * kQY;
constexpr int kQS = 4;  // ring slots = planes per loop trip

// Resident CTAs per SM that the launch bounds ask for.  The queues take
// 6(2R+1) + 3(R+1) registers.  100 steps of 336^3 (ms): SO 4 with 6 / 5 CTAs
// 33.0 / 34.2; SO 10 with 3 / 2 52.8 / 64.8; SO 12 with 3 / 2 62.6 / 69.8.
constexpr int q_ctas(int R) { return R <= 2 ? 6 : (R <= 4 ? 4 : (R <= 6 ? 3 : 2)); }
// x halo of a staged tile: R rounded up to 2 cells (16-byte aligned TMA x coordinate)
constexpr int q_halo_x(int R) { return (R + 1) / 2 * 2; }

template <int R>
struct QGeom {
  static constexpr int RX = q_halo_x(R);
  static constexpr int W = kQX + 2 * RX, H = kQY + 2 * R;
  // dy of a row's 2R halo cells: HL groups of HP lanes of the row's warp share
  // the terms of the cells (HT each); a half warp's loads then hit all banks.
  // At R = 3 four groups (one term each) fit too, and gain nothing over two: us a
  // step, two / four, 190^3 85.8 / 85.9, 296^3 278.7 / 281.3.
  static constexpr int HP = R == 1 ? 2 : (R == 2 ? 4 : (R <= 4 ? 8 : 16));
  static constexpr int HL = R == 4 ? 4 : (R >= 2 ? 2 : 1);
  static constexpr int HT = (R + HL - 1) / HL;
  static_assert(HP * HL <= 32 && HP >= 2 * R, "one warp per row");
  static constexpr uint32_t UBYTES = W * H * 8;
  static constexpr uint32_t TBYTES = kQT * 8;  // a tile of pairs
  // a slot: the plane, its (nx, ny); the output plane's (A, e2), (dl, nz), (nx, ny), previous
  // (p, q)
  static constexpr uint32_t OFF_N = (UBYTES + 127) / 128 * 128;
  static constexpr uint32_t OFF_C = OFF_N + TBYTES;
  static constexpr uint32_t OFF_P = OFF_C + 3 * TBYTES;
  static constexpr uint32_t SLOT = OFF_P + TBYTES;
  static constexpr uint32_t DP = (W * kQY * 8 + 127) / 128 * 128;
  static constexpr uint32_t OFF_D = kQS * SLOT;  // dy scratch, two buffers
  static constexpr uint32_t OFF_BAR = OFF_D + 2 * DP;
  static constexpr uint32_t SMEM = OFF_BAR + 8 * kQS + 128;  // + alignment slack
};

struct QMaps {
  CUtensorMap halo;  // (p, q)^n: W x H boxes of cells
  CUtensorMap prev;  // (p, q)^{n-1}: tiles of cells
  CUtensorMap coef;  // (A, e2), (dl, nz), (nx, ny) stacked along z: tiles of cells
};

struct QArgs {
  float2* out;  // (p, q)^{n-1} in, (p, q)^{n+1} out (in place)
  int* err;     // set on an expired wait
  int Nx, Ny, Nz, pitch;
  int nbl, nx, ny, nz;
  int cols_y, cols;  // tile columns in y, and in all
  long long spin_limit;
  float bscale;
  float2 c[kMaxR + 1];  // each weight twice, one per half of a pair
  float2 c0lo;          // the centre weight is c[0] + c0lo
  float2 d[kMaxR + 1];
};

__device__ __forceinline__ int qdepth(int g, int nbl, int n) {
  int d = nbl - g;
  const int e = g - (n + nbl - 1);
  d = d > e ? d : e;
  return d > 0 ? d : 0;
}

template <int N, class T>
__device__ __forceinline__ void qpush(T (&q)[N], T v) {
#pragma unroll
  for (int i = 0; i < N - 1; ++i) q[i] = q[i + 1];
  q[N - 1] = v;
}

__device__ __forceinline__ float2 lds2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}

__device__ __forceinline__ void sts2(uint32_t a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }

// a - b, rounded as a subtraction (the product by -1 is exact)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}

template <int R>
__global__ void __launch_bounds__(kQT, q_ctas(R))
    k_tti_q(const __grid_constant__ QMaps M, const __grid_constant__ QArgs a) {
  using G = QGeom<R>;
  extern __shared__ unsigned char qsm_raw[];
  // aligned by an offset from the shared array, so the address space is kept
  unsigned char* qsm =
      qsm_raw + ((128u - (static_cast<uint32_t>(__cvta_generic_to_shared(qsm_raw)) & 127u)) &
                 127u);
  const uint32_t sbase = smem_u32(qsm);
  const uint32_t bar0 = sbase + G::OFF_BAR;
  const int tid = threadIdx.x, tx = tid % kQX, ty = tid / kQX;
  // own cell in a staged plane, in the dy scratch and in a tile
  const uint32_t cown = sbase + 8u * ((ty + R) * G::W + tx + G::RX);
  const uint32_t cd = sbase + G::OFF_D + 8u * (ty * G::W + tx + G::RX);
  const uint32_t ctile = sbase + 8u * tid;
  // dy of the row's halo cells: lane tx takes terms j = hj + 1, hj + 1 + HL, ..
  // of halo cell hc (weight 0 beyond R and for lanes without a cell)
  const int hc = min(tx % G::HP, 2 * R - 1), hj = min(tx / G::HP, G::HL - 1);
  const int hcol = hc < R ? hc - R : kQX + hc - R;  // tile column
  const uint32_t chalo = sbase + 8u * ((ty + R) * G::W + hcol + G::RX);
  const uint32_t chd = sbase + G::OFF_D + 8u * (ty * G::W + hcol + G::RX);
  const bool hwrite = tx < 2 * R;  // (its terms' other groups: lanes tx + HP, ..)
  float hd[G::HT];
#pragma unroll
  for (int m = 0; m < G::HT; ++m) {
    hd[m] = 0.f;
#pragma unroll
    for (int j = 1; j <= R; ++j)
      if (j == hj + 1 + m * G::HL) hd[m] = a.d[j].x;
  }
  const uint32_t hstep = 8u * G::W * (hj + 1);  // row offset of the first term

  // this CTA's share of the last, partial wave of columns
  const int waves = a.cols / gridDim.x, rest = a.cols - waves * gridDim.x;
  const long long units = static_cast<long long>(rest) * a.Nz;
  long long pos = units * blockIdx.x / gridDim.x;
  const long long hi = units * (blockIdx.x + 1) / gridDim.x;
  bool bad = false;
  long long limit = a.spin_limit;
  pdl_trigger();
  pdl_wait();

  for (int w = 0; w < waves || pos < hi; ++w) {
    int col = w * gridDim.x + blockIdx.x, z0 = 0, z1 = a.Nz;
    if (w >= waves) {
      col = waves * gridDim.x + static_cast<int>(pos / a.Nz);
      z0 = static_cast<int>(pos % a.Nz);
      z1 = static_cast<int>(min(static_cast<long long>(a.Nz), z0 + (hi - pos)));
      pos += z1 - z0;
    }
    const int x0 = col / a.cols_y * kQX, y0 = col % a.cols_y * kQY;
    const int nout = z1 - z0, nin = nout + 2 * R;  // entering planes z0-R .. z1+R-1

    if (tid == 0) {
      for (int s = 0; s < kQS; ++s) mbar_init(bar0 + 8 * s, 1);
      fence_mbar_init();
    }
    __syncthreads();

    // producer (thread 0): entering plane i (z = z0-R+i) into slot i mod 4,
    // with the per-point values of output plane i - 2R
    int next = 0;
    auto issue = [&](int i, int s) {
      if (i >= nin || bad) return;
      next = i + 1;
      const uint32_t bar = bar0 + 8 * s, dst = sbase + s * G::SLOT;
      const int z = z0 - R + i;
      // the axis of planes that are output planes of this run
      const bool axis = i >= R && i < R + nout, outp = i >= 2 * R;
      mbar_expect_tx(bar, G::UBYTES + ((axis ? 1 : 0) + (outp ? 4 : 0)) * G::TBYTES);
      tma_load_3d(dst, &M.halo, 2 * (x0 - G::RX), y0 - R, z, bar);
      if (axis) tma_load_3d(dst + G::OFF_N, &M.coef, 2 * x0, y0, z + 2 * a.Nz, bar);
      if (outp) {
#pragma unroll
        for (int f = 0; f < 3; ++f)
          tma_load_3d_stream(dst + G::OFF_C + f * G::TBYTES, &M.coef, 2 * x0, y0,
                             z - R + f * a.Nz, bar);
        tma_load_3d_stream(dst + G::OFF_P, &M.prev, 2 * x0, y0, z - R, bar);
      }
    };
    if (tid == 0)
      for (int i = 0; i < kQS; ++i) issue(i, i);

    // register queues: own (p, q), dx, dy of planes k-R .. k+R (centre at R);
    // the in-plane H_z of both fields and D_xx p + D_yy p of planes k .. k+R
    // (centre at 0)
    float2 qu[2 * R + 1], qdx[2 * R + 1], qdy[2 * R + 1], qh[R + 1];
    float ql[R + 1];
#pragma unroll
    for (int i = 0; i < 2 * R + 1; ++i) qu[i] = qdx[i] = qdy[i] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < R + 1; ++i) {
      qh[i] = make_float2(0.f, 0.f);
      ql[i] = 0.f;
    }

    const int gx = x0 + tx, gy = y0 + ty;
    const bool inside = gx < a.Nx && gy < a.Ny;
    const int dxv = qdepth(gx, a.nbl, a.nx), dyv = qdepth(gy, a.nbl, a.ny);
    float2* po = a.out + (static_cast<size_t>(z0) * a.Ny + gy) * a.pitch + gx;
    const size_t plane = static_cast<size_t>(a.Ny) * a.pitch;
    // damping of the current output plane: 1 - b and 1 / (1 + b), formed again
    // only when the plane's depth in the layer changes
    int dz_of = -1;
    float omb = 1.f, binv = 1.f;

    // plane i, staged in slot s, enters: its first differences and (planes that
    // will be output planes) in-plane terms go into the queues; one barrier
    float2 zz, xz, yz;  // z sums of the output plane
    // the second derivatives' centre term: -2 sum_j c_j of the FP32 weights, as
    // two FP32 numbers, so that a constant field has none (one FP32 centre
    // weight leaves a row sum of ~1e-7, which adds up over the steps)
    auto centre = [&](float2 u) { return __ffma2_rn(a.c[0], u, __fmul2_rn(a.c0lo, u)); };
    auto enter = [&](int i, int s, auto inplane, auto zpart) {
      constexpr bool kIn = decltype(inplane)::value;
      if (!mbar_wait(bar0 + 8 * s, (i / kQS) & 1, limit)) {
        bad = true;
        limit = 0;
      }
      // the z sums but for their last term, which enters with this plane:
      // independent work in the shadow of the loads below (4 % at SO 8 and 16)
      if (decltype(zpart)::value) {
        zz = centre(qu[R + 1]);
        xz = yz = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 1; j < R; ++j) {
          zz = __ffma2_rn(a.c[j], __fadd2_rn(qu[R + 1 + j], qu[R + 1 - j]), zz);
          xz = __ffma2_rn(a.d[j], sub2(qdx[R + 1 + j], qdx[R + 1 - j]), xz);
          yz = __ffma2_rn(a.d[j], sub2(qdy[R + 1 + j], qdy[R + 1 - j]), yz);
        }
      }
      const uint32_t P = cown + s * G::SLOT;
      const uint32_t D = cd + (s & 1) * G::DP;
      const float2 u0 = lds2(P);
      float2 xx = kIn ? centre(u0) : make_float2(0.f, 0.f), yy = xx;
      float2 dx = make_float2(0.f, 0.f), dy = dx, hxy = dx, nn = dx;
#pragma unroll
      for (int j = 1; j <= R; ++j) {
        const float2 xp = lds2(P + 8 * j), xm = lds2(P - 8 * j);
        if (kIn) xx = __ffma2_rn(a.c[j], __fadd2_rn(xp, xm), xx);
        dx = __ffma2_rn(a.d[j], sub2(xp, xm), dx);
      }
#pragma unroll
      for (int j = 1; j <= R; ++j) {
        const float2 yp = lds2(P + 8 * j * G::W), ym = lds2(P - 8 * j * G::W);
        if (kIn) yy = __ffma2_rn(a.c[j], __fadd2_rn(yp, ym), yy);
        dy = __ffma2_rn(a.d[j], sub2(yp, ym), dy);
      }
      if (kIn) {
        sts2(D, dy);
        float2 e = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < G::HT; ++m) {
          // terms beyond R (R not a multiple of HL) read the last one again
          const uint32_t o = (m + 1) * G::HL <= R || hj + 1 + m * G::HL <= R
                                 ? hstep + 8u * G::W * G::HL * m
                                 : 8u * G::W * R;
          const uint32_t h = chalo + s * G::SLOT;
          e = __ffma2_rn(dup2(hd[m]), sub2(lds2(h + o), lds2(h - o)), e);
        }
#pragma unroll
        for (int o = G::HP; o < G::HP * G::HL; o *= 2)
          e = __fadd2_rn(e, make_float2(__shfl_xor_sync(0xffffffffu, e.x, o),
                                        __shfl_xor_sync(0xffffffffu, e.y, o)));
        if (hwrite) sts2(chd + (s & 1) * G::DP, e);
        nn = lds2(ctile + s * G::SLOT + G::OFF_N);
        hxy = __ffma2_rn(dup2(nn.x * nn.x), xx, __fmul2_rn(dup2(nn.y * nn.y), yy));
      }
      __syncthreads();
      if (kIn) {
        float2 xy = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 1; j <= R; ++j)
          xy = __ffma2_rn(a.d[j], sub2(lds2(D + 8 * j), lds2(D - 8 * j)), xy);
        hxy = __ffma2_rn(dup2(2.f * nn.x * nn.y), xy, hxy);
        qpush(qh, hxy);
        qpush(ql, xx.x + yy.x);
      }
      qpush(qu, u0);
      qpush(qdx, dx);
      qpush(qdy, dy);
    };

    // planes below the first output plane, then those up to its own R-th
    // neighbour; a slot is refilled one plane later, when the next barrier
    // shows that every thread is past it
#pragma unroll 1
    for (int i = 0; i < R; ++i) {
      enter(i, i % kQS, std::false_type(), std::false_type());
      if (tid == 0) issue(i + kQS, i % kQS);
    }
#pragma unroll 1
    for (int i = R; i < 2 * R; ++i) {
      enter(i, i % kQS, std::true_type(), std::false_type());
      if (tid == 0) issue(i + kQS, i % kQS);
    }

    // The slot of output plane k also holds its per-point values, read after
    // the plane's barrier: it is refilled behind the next plane's barrier.
    for (int k0 = 0; k0 < nout; k0 += kQS) {
#pragma unroll
      for (int t = 0; t < kQS; ++t) {
        const int k = k0 + t;
        if (k >= nout) goto done;
        {
          constexpr int kFirst = 2 * R % kQS;
          const int s = (kFirst + t) % kQS;
          // the last R planes of a run are entered for their z terms only;
          // their axis is not loaded, and what is formed from it is not used
          enter(k + 2 * R, s, std::true_type(), std::true_type());
          if (tid == 0 && k > 0) issue(k + 2 * R - 1 + kQS, (s + kQS - 1) % kQS);
          const int dz = qdepth(z0 + k, a.nbl, a.nz);
          if (dz != dz_of) {
            dz_of = dz;
            const float b = a.bscale * static_cast<float>(dxv * dxv + dyv * dyv + dz * dz);
            omb = 1.f - b;
            binv = 1.f / (1.f + b);  // exactly 1 outside the layer
          }
          const uint32_t T = ctile + s * G::SLOT;
          const float2 ae = lds2(T + G::OFF_C);                  // A, e2
          const float2 dn = lds2(T + G::OFF_C + G::TBYTES);      // dl, nz
          const float2 nn = lds2(T + G::OFF_C + 2 * G::TBYTES);  // nx, ny
          const float2 um = lds2(T + G::OFF_P), uc = qu[R];
          zz = __ffma2_rn(a.c[R], __fadd2_rn(qu[2 * R], qu[0]), zz);
          xz = __ffma2_rn(a.d[R], sub2(qdx[2 * R], qdx[0]), xz);
          yz = __ffma2_rn(a.d[R], sub2(qdy[2 * R], qdy[0]), yz);
          // H_z of both fields, then H_0 p = Laplacian - H_z
          const float nz = dn.y, nz2 = 2.f * nz, dl = dn.x;
          float2 hz = __ffma2_rn(dup2(nz * nz), zz, qh[0]);
          hz = __ffma2_rn(dup2(nz2 * nn.x), xz, hz);
          hz = __ffma2_rn(dup2(nz2 * nn.y), yz, hz);
          const float h0 = (ql[0] + zz.x) - hz.x;
          const float2 r = make_float2(fmaf(ae.y, h0, dl * hz.y), fmaf(dl, h0, hz.y));
          // (1+b) u+ = 2u - (1-b) u- + A r as an increment of u,
          //   u+ = u + ((1-b) (u - u-) + A r) / (1+b):
          // u - u- is exact or nearly so, and the rounding of the terms and of
          // the reciprocal is relative to the increment, not to u.  Rounding
          // 2u - u- at the size of u was a third to a half of the error against
          // FP64 (60 steps of 110 x 90 x 100 at SO 16, FP32 emulated term by term:
          // 4.3e-7 to 5.1e-7 of 5.7e-7 to 1.1e-6; the final rounding the rest).
          const float2 inc = __ffma2_rn(dup2(ae.x), r, __fmul2_rn(dup2(omb), sub2(uc, um)));
          if (inside) *po = __ffma2_rn(inc, dup2(binv), uc);
          po += plane;
        }
      }
    }
  done:
    // every issued copy has been waited for, but where a wait ran out: there
    // the producer waits (bounded) for its copies in flight
    if (bad) atomicOr(a.err, 1);
    if (tid == 0 && bad)
      for (int i = max(0, next - kQS); i < next; ++i)
        mbar_wait(bar0 + 8 * (i % kQS), (i / kQS) & 1, a.spin_limit);
    // release the barriers for the next run
    if (__syncthreads_or(bad)) return;
    if (tid == 0)
      for (int s = 0; s < kQS; ++s) mbar_inval(bar0 + 8 * s);
  }
}

}  // namespace tti
}  // namespace fd
