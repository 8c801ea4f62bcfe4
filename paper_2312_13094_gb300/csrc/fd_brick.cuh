// Step kernel of small grids: one CTA per brick of the grid (included by
// fd_step_inst.cuh).
//
// The streaming sweep (fd_step.cuh) walks z plane by plane: every plane waits
// for its copy, and a CTA-wide barrier orders the reuse of its ring slot.  A
// grid whose columns give the GPU only a few planes per CTA is bound by that
// chain, not by memory.  Here a CTA takes 32 x 8 x 8 points, brings
// everything they read (the brick of u^n with its halo, u^{n-1} and A) into
// shared memory at once, one TMA tile load per plane issued by as many lanes,
// and waits once; its threads then compute two or four planes each without
// another barrier.  The halo is read (8 + 2R)^2 (32 + 2RX) / 2048 times instead
// of (8 + 2R) (32 + 2RX) / 256, from L2, where such a grid lives.
//
// The arithmetic of a point is that of the sweep (lap4_packed, update4_inner,
// update4_layer, receivers, sources in list order), so both give the same bits.
#pragma once

#include "fd_step.cuh"

namespace fd {

template <int R, int MODE>
struct BrickCfg {
  // ZT planes per thread: four, or two where shared memory admits few CTAs and
  // each needs more warps
  static constexpr int TX = 8, TY = 8, ZB = 8, ZT = R <= 4 ? 4 : 2, ZG = ZB / ZT;
  static constexpr int NT = TX * TY * ZG;
  static constexpr int RX = ((R + 3) / 4) * 4;
  static constexpr int BX = 4 * TX, BY = TY;
  static constexpr int W = BX + 2 * RX, H = BY + 2 * R, NP = ZB + 2 * R;
  static constexpr uint32_t UBYTES = W * H * 4;
  static constexpr uint32_t UPITCH = (UBYTES + 127) / 128 * 128;
  static constexpr uint32_t TBYTES = BX * BY * 4;  // a multiple of 128
  static constexpr uint32_t OFF_P = NP * UPITCH;
  static constexpr uint32_t OFF_A = OFF_P + ZB * TBYTES;
  static constexpr int NC = MODE == kModePerCell ? R : 0;  // coefficient fields
  static constexpr uint32_t OFF_C = OFF_A + ZB * TBYTES;   // [field][plane]
  static constexpr uint32_t OFF_T = OFF_C + NC * ZB * TBYTES;
  // the weight table of kModeTable
  static constexpr uint32_t OFF_BAR = OFF_T + (MODE == kModeTable ? 2 * kTableNodes * 16 : 0);
  static constexpr uint32_t SMEM = OFF_BAR + 8 + 128;  // + alignment slack
  // resident CTAs per SM (shared memory: 228 KB, 1 KB of it per CTA reserved)
  static constexpr int CTAS =
      R <= 3 ? 4 : (R == 4 && MODE != kModePerCell ? 3 : (R <= 7 ? 2 : 1));
  static_assert(CTAS * (SMEM + 1024) <= 228 * 1024, "resident CTAs");
  static_assert(TBYTES % 128 == 0, "tile pitch");
};

__device__ __forceinline__ void prefetch_map(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}

template <int R, int MODE>
__global__ void __launch_bounds__(BrickCfg<R, MODE>::NT, BrickCfg<R, MODE>::CTAS)
    brick_kernel(const ShotDesc* __restrict__ shot, const __grid_constant__ StepOverride ov) {
  using C = BrickCfg<R, MODE>;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 127u) & ~127u;
  float4* tab = reinterpret_cast<float4*>(smem_raw + (sbase - smem_u32(smem_raw)) + C::OFF_T);
  const uint32_t bar = sbase + C::OFF_BAR;
  const int tid = threadIdx.x, tx = tid % C::TX, ty = tid / C::TX % C::TY,
            zg = tid / (C::TX * C::TY);
  const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY, zb = blockIdx.z * C::ZB;
  const StepArgs& a = shot->args;
  const int cur = ov.cur;
  pdl_trigger();
  if (tid < 3)  // the tensor maps, fetched while the step ahead still runs
    prefetch_map(tid == 0 ? &shot->halo[cur] : (tid == 1 ? &shot->tile[cur ^ 1] : &shot->A));
  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    mbar_expect_tx(bar, C::NP * C::UBYTES + (2 + C::NC) * C::ZB * C::TBYTES);
  }
  if (MODE == kModeTable)  // (written before the first step)
    for (int i = tid; i < 2 * a.tab_nodes; i += C::NT) tab[i] = a.table[i];
  __syncthreads();
  // the copies over the lanes of warp 0: A and the coefficients, which no step
  // writes, before the step ahead has finished, the wavefields after it
  if (tid < C::ZB)
    tma_load_3d(sbase + C::OFF_A + tid * C::TBYTES, &shot->A, x0, y0, zb + tid, bar);
  if (tid < 32) {
#pragma unroll
    for (int c = tid; c < C::NC * C::ZB; c += 32)  // field j sits j * Nz planes further
      tma_load_3d(sbase + C::OFF_C + c * C::TBYTES, &shot->C, x0, y0,
                  zb + c % C::ZB + c / C::ZB * a.Nz, bar);
  }
  pdl_wait();
  if (tid < 32) {
#pragma unroll
    for (int c = tid; c < C::NP + C::ZB; c += 32) {
      if (c < C::NP) {
        const int z = zb - R + c;
        if (ov.debug_skip_plane < 0 || z != ov.debug_skip_plane)
          tma_load_3d(sbase + c * C::UPITCH, &shot->halo[cur], x0 - C::RX, y0 - R, z, bar);
      } else {
        const int i = c - C::NP;
        tma_load_3d(sbase + C::OFF_P + i * C::TBYTES, &shot->tile[cur ^ 1], x0, y0, zb + i, bar);
      }
    }
  }

  const int Nz = a.Nz, zend = min(zb + C::ZB, Nz), k0 = zb + C::ZT * zg;
  const int gx = x0 + 4 * tx, gy = y0 + ty;
  const bool in_grid = gx < a.xend && gy < a.yend;
  const size_t plane = static_cast<size_t>(a.Ny) * a.pitch;
  const size_t off = static_cast<size_t>(k0) * plane + static_cast<size_t>(gy) * a.pitch + gx;
  float* __restrict__ out = shot->u[cur ^ 1];
  float4 ein[MODE == kModeAdjoint ? C::ZT : 1], gr[MODE == kModeAdjoint ? C::ZT : 1];
  if (MODE == kModeAdjoint) {
#pragma unroll
    for (int p = 0; p < C::ZT; ++p) {
      if (in_grid && k0 + p < zend) {
        ein[p] = __ldg(reinterpret_cast<const float4*>(ov.e_in + off + p * plane));
        gr[p] = *reinterpret_cast<const float4*>(a.grad + off + p * plane);
      }
    }
  }
  // the tile's sources from plane k0 on (sorted by z), and its receivers
  const int tile = blockIdx.y * a.tiles_x + blockIdx.x;
  int ip = 0, iend = 0, rp = 0, rend = 0;
  if (a.inj_start) {
    ip = a.inj_start[tile];
    iend = a.inj_start[tile + 1];
    if (ip < iend && a.inj[iend - 1].z < k0) ip = iend;
    while (ip < iend && a.inj[ip].z < k0) ++ip;
  }
  if (a.rec_start) {
    rp = a.rec_start[tile];
    rend = a.rec_start[tile + 1];
  }
  // the layer, as in the sweep: planes [zf_lo, zf_hi) of the tile have b = 0
  // everywhere and no point outside the grid
  const int dyv = sponge_depth(gy, a.nbl, a.ny);
  float dxx[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const int d = sponge_depth(gx + l, a.nbl, a.nx);
    dxx[l] = static_cast<float>(d * d + dyv * dyv);
  }
  const bool no_sponge = a.bscale == 0.0f;
  const bool inner_xy = x0 >= a.nbl && x0 + C::BX <= a.nbl + a.nx && y0 >= a.nbl &&
                        y0 + C::BY <= a.nbl + a.ny;
  const bool full = x0 + C::BX <= a.xend && y0 + C::BY <= a.yend;
  const bool flat = full && (no_sponge || inner_xy);
  const int zf_lo = no_sponge ? 0 : a.nbl, zf_hi = no_sponge ? Nz : a.nbl + a.nz;
  const bool ok[4] = {gx < a.xend, gx + 1 < a.xend, gx + 2 < a.xend, gx + 3 < a.xend};

  // once a wait of this run has failed, its later launches do nothing; the word
  // is read while the copies are on their way, and they are waited for either way
  const bool failed = *reinterpret_cast<volatile const int*>(a.err) != 0;
  // every thread waits, so that each sees the copies; on expiry (the copies
  // of this CTA have then had the whole limit to land) the CTA records it
  if (!mbar_wait(bar, 0, ov.spin_limit)) {
    atomicOr(a.err, 1);
    return;
  }
  if (failed) return;

  const uint32_t crow = 4u * ((ty + R) * C::W + 4 * tx + C::RX);
  const uint32_t own = sbase + C::ZT * zg * C::UPITCH + crow;  // plane k0 - R
  const uint32_t ctile = 4u * (ty * C::BX + 4 * tx) + C::ZT * zg * C::TBYTES;
  float4 q[C::ZT + 2 * R];
#pragma unroll
  for (int j = 0; j < C::ZT + 2 * R; ++j) q[j] = lds4(own + j * C::UPITCH);
  constexpr int NROW4 = 2 * C::RX / 4 + 1;
#pragma unroll
  for (int p = 0; p < C::ZT; ++p) {
    const int k = k0 + p;
    if (k >= zend) break;
    const uint32_t P = own + (p + R) * C::UPITCH;
    const float4 uc = q[p + R];
    float xr[4 * NROW4];
#pragma unroll
    for (int m = 0; m < NROW4; ++m) {
      const float4 v = (m == NROW4 / 2) ? uc : lds4(P + 16 * (m - NROW4 / 2));
      xr[4 * m + 0] = v.x;
      xr[4 * m + 1] = v.y;
      xr[4 * m + 2] = v.z;
      xr[4 * m + 3] = v.w;
    }
    float lap[4];
    auto yn = [&](int jj, float4& ym, float4& yp) {
      ym = lds4(P - 4 * jj * C::W);
      yp = lds4(P + 4 * jj * C::W);
    };
    auto zn = [&](int o) -> float4 { return q[p + R + o]; };
    if (MODE == kModePerCell || MODE == kModeTable) {
      float2 dj[R][2];
      diffs4<R, C::RX>(xr, yn, zn, dj);
      if (MODE == kModePerCell)
        weigh_cells<R>(
            dj,
            [&](int jj) {
              return lds4(sbase + C::OFF_C + ((jj - 1) * C::ZB + p) * C::TBYTES + ctile);
            },
            lap);
      else
        weigh_table<R>(dj, lds4(sbase + C::OFF_A + ctile + p * C::TBYTES), tab, a.tab_lo,
                       a.tab_inv, a.tab_nodes, lap);
    } else {
      lap4_packed<R, C::RX>(xr, yn, zn, ov.c, ov.c[0], ov.c[kMaxR + 1], lap);
    }
    float src[4] = {0.f, 0.f, 0.f, 0.f};
    while (ip < iend) {
      const InjEntry e = a.inj[ip];
      if (e.z != k) break;
      if (e.ly == ty && (e.lx >> 2) == tx) {
        const float val = e.w * a.inj_val[static_cast<size_t>(ov.inj_row) * a.inj_ncol + e.col];
#pragma unroll
        for (int l = 0; l < 4; ++l) src[l] += ((e.lx & 3) == l) ? val : 0.f;
      }
      ++ip;
    }
    const float4 up = lds4(sbase + C::OFF_P + ctile + p * C::TBYTES);
    const float4 Av = lds4(sbase + C::OFF_A + ctile + p * C::TBYTES);
    float res[4], ev[4];
    if (flat && k >= zf_lo && k < zf_hi) {
      update4_inner(lap, src, uc, up, Av, res, ev);
    } else {
      const int dz = sponge_depth(k, a.nbl, a.nz);
      update4_layer(lap, src, uc, up, Av, dxx, static_cast<float>(dz * dz), a.bscale, ok, res, ev);
    }
    if (in_grid) {
      const size_t o = off + p * plane;
      *reinterpret_cast<float4*>(out + o) = make_float4(res[0], res[1], res[2], res[3]);
      if (MODE == kModeStoreE) st_stream(ov.e_out + o, ev[0], ev[1], ev[2], ev[3]);
      if (MODE == kModeAdjoint) {
        float4 g = gr[p];
        g.x -= uc.x * ein[p].x * a.inv_dt2;
        g.y -= uc.y * ein[p].y * a.inv_dt2;
        g.z -= uc.z * ein[p].z * a.inv_dt2;
        g.w -= uc.w * ein[p].w * a.inv_dt2;
        *reinterpret_cast<float4*>(a.grad + o) = g;
      }
    }
  }

  // receivers whose floor node lies in the brick's planes (k and k + 1 are
  // both staged)
  for (int e = rp + tid; e < rend; e += C::NT) {
    const RecEntry r = a.recs[e];
    if (r.z < zb || r.z >= zend) continue;
    const uint32_t o = 4u * ((r.ly + R) * C::W + r.lx + C::RX);
    const uint32_t P0 = sbase + (r.z - zb + R) * C::UPITCH, P1 = P0 + C::UPITCH;
    constexpr uint32_t W4 = 4u * C::W;
    const float gx0 = 1.0f - r.fx, gy0 = 1.0f - r.fy;
    const float p0 = gy0 * (gx0 * lds1(P0 + o) + r.fx * lds1(P0 + o + 4)) +
                     r.fy * (gx0 * lds1(P0 + o + W4) + r.fx * lds1(P0 + o + W4 + 4));
    const float p1 = gy0 * (gx0 * lds1(P1 + o) + r.fx * lds1(P1 + o + 4)) +
                     r.fy * (gx0 * lds1(P1 + o + W4) + r.fx * lds1(P1 + o + W4 + 4));
    a.rec_out[static_cast<size_t>(ov.rec_row) * a.rec_ncol + r.col] =
        (1.0f - r.fz) * p0 + r.fz * p1;
  }
}

}  // namespace fd
