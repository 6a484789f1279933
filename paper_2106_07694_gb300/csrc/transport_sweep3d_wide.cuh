// 3D FP32 transport with four adjacent x columns per thread: one SSP-RK3 stage of the
// WENO5 + diffusion + settling update of c (steps a4..a8) as a tiled sweep along the
// vertical axis z.  The scheme variants and the sugar scalar are compile-time forms of the
// same kernel.
//
// A CTA of kV3x x kV3y threads owns a tile of 4 kV3x x kV3y (x, y) columns and a segment
// of z levels and sweeps it upward.  At level k:
//  - the x-split fluxes of the tile rows with a four-column halo quad on each side, the
//    y-split fluxes of the tile columns with a three-row halo below and above, and c on
//    both, are staged in shared memory as float4 quads (loaded one level ahead; one buffer,
//    refilled between two barriers, so that four CTAs fit an SM);
//  - a thread reconstructs the left x faces of its four columns (first and second
//    differences of the split fluxes shared between the four faces) and the lower y face
//    of each of them; the x face right of its last column is its neighbour's first one,
//    the y face above is the lower face of the thread above; the faces right of the tile's
//    last column and above its top row come from the staged halo, by the first two warps
//    (computed for the whole segment before the sweep, from global memory, they were nine
//    trips to L2 before the first level and a tenth of the kernel);
//  - the upper z face of each column comes from a private ring of the z-split fluxes of
//    levels k-2 .. k+3, filled three levels ahead; the lower z face is carried.
// Every face is computed once with the arithmetic of face_flux_x, so c is
// bitwise that of the one-column kernel.
//
// Bound by instruction issue with 16 warps an SM (128 registers, 44.6 KB of shared memory a
// CTA).  256 x 256 x 512: 391 / 388 / 411 us a stage, 476 / 476 / 491 with the edge faces ahead
// of the sweep and the first loads one after the other.
//
// Walls: ghost levels -2, -1, nz, nz+1 reflect c (even) and the fluid velocity (odd, Vs
// unchanged); the floor face carries -Vs c(0), the lid 0 (the floor deposit is folded by
// its own kernel in 3D).
#pragma once
#include "common.cuh"
#include "weno.cuh"
#include "transport_sweep3d.cuh"       // Sweep3dParams
#include "transport_stage2d_wide.cuh"  // scheme_split, x_faces, column_faces

namespace lw {

constexpr int kV3x = 8;                 // threads along x (4 columns each)
constexpr int kV3y = 16;                // threads along y
constexpr int kV3T = kV3x * kV3y;       // threads per CTA
constexpr int kV3W = 4 * kV3x;          // tile width in columns
constexpr int kV3Qx = kV3x + 2;         // staged quads per row (tile and one halo quad per side)
constexpr int kV3Ry = kV3y + 6;         // staged rows of the y stencil (three-row halo per side)
constexpr int kV3maxH = 32;             // longest z segment

struct Sweep3dWideSmem {
  float4 xp[kV3y][kV3Qx];   // x-split h+/alpha of the tile rows
  float4 xm[kV3y][kV3Qx];
  float4 yp[kV3Ry][kV3x];   // y-split h+/alpha of the tile columns (rows -3 .. kV3y + 2)
  float4 ym[kV3Ry][kV3x];
  float4 c[kV3Ry][kV3Qx];   // stage input c (rows -3 .. kV3y + 2, quads -1 .. kV3x)
  float4 zp[6][kV3T];          // z-split ring of each thread's four columns
  float4 zm[6][kV3T];
  float fx[2][kV3y][kV3x + 1];     // first left x face of each thread (+ the tile's right edge)
  float4 fy[2][kV3y + 1][kV3x];    // lower y faces of each thread's columns (+ the tile's top edge)
};

// SUGAR, SCHEME: as in the 2D kernel (stage2d_wide_body).
template <int STAGE, bool SUGAR = false, int SCHEME = 0>
__device__ __forceinline__ void sweep3d_wide_body(Sweep3dWideSmem& S, const Args<float>& a, const Sweep3dParams& sp) {
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kV3x + tx;
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int x0 = blockIdx.x * kV3W, y0 = blockIdx.y * kV3y;
  const int z0 = blockIdx.z * sp.H, z1 = min(nz, z0 + sp.H);
  const int xl = x0 + 4 * tx, yl = y0 + ty;
  const bool out = xl < nx && yl < ny;
  const unsigned X = (unsigned)(xl % nx), Y = (unsigned)(yl % ny);
  const unsigned plane = (unsigned)nx * (unsigned)ny, n = (unsigned)a.n;
  const unsigned col = Y * (unsigned)nx + X;
  const float ia = a.inv_alpha, vs_a = a.vs * a.inv_alpha, alpha = a.alpha, kd = a.kappa * a.inv_alpha;
  const float* __restrict__ cin = sp.cin;
  const float* __restrict__ ux = a.u;
  const float* __restrict__ uy = a.u + n;
  const float* __restrict__ uz = a.u + 2 * n;

  // staging positions: the cross of tile rows x [quads -1 .. kV3x] and rows [-3 .. kV3y+2]
  // x tile quads (the corners are not needed); each thread takes up to two
  constexpr int kPos = kV3y * kV3Qx + 6 * kV3x;  // tile rows (with x halo) + the 6 halo rows
  constexpr int kSl = (kPos + kV3T - 1) / kV3T;
  int sl_r[kSl], sl_q[kSl];  // staged row (0 .. kV3Ry-1) and quad (0 .. kV3Qx-1)
  unsigned sl_off[kSl];
  bool sl_on[kSl], sl_x[kSl], sl_y[kSl];
#pragma unroll
  for (int s = 0; s < kSl; ++s) {
    const int j = tid + s * kV3T;
    int r, q;
    if (j < kV3y * kV3Qx) {  // a tile row, any quad
      r = 3 + j / kV3Qx;
      q = j % kV3Qx;
    } else {  // a halo row, a tile quad
      const int h = j - kV3y * kV3Qx;
      const int hr = h / kV3x;  // 0..5: rows -3, -2, -1, kV3y, kV3y + 1, kV3y + 2
      r = hr < 3 ? hr : kV3y + hr;
      q = 1 + h % kV3x;
    }
    sl_on[s] = j < kPos;
    sl_r[s] = r;
    sl_q[s] = q;
    sl_x[s] = r >= 3 && r < 3 + kV3y;
    sl_y[s] = q >= 1 && q <= kV3x;
    const int gx = ((x0 - 4 + 4 * q) % nx + nx) % nx, gy = ((y0 - 3 + r) % ny + ny) % ny;
    sl_off[s] = (unsigned)gy * (unsigned)nx + (unsigned)gx;
  }
  float4 pc[kSl], pu[kSl], pv[kSl];
  auto fetch_tile = [&](int l) {
    const unsigned lv = (unsigned)l * plane;
#pragma unroll
    for (int s = 0; s < kSl; ++s) {
      if (sl_on[s]) {
        pc[s] = LoadNC::v4(cin + lv + sl_off[s]);
        if (sl_x[s]) pu[s] = LoadNC::v4(ux + lv + sl_off[s]);
        if (sl_y[s]) pv[s] = LoadNC::v4(uy + lv + sl_off[s]);
      }
    }
  };
  auto stage_tile = [&]() {
#pragma unroll
    for (int s = 0; s < kSl; ++s) {
      if (sl_on[s]) {
        const float4 c = pc[s];
        S.c[sl_r[s]][sl_q[s]] = c;
        if (sl_x[s]) {
          const float4 u = pu[s];
          float4 p, m;
          scheme_split<SCHEME>(c.x, u.x * ia, p.x, m.x);
          scheme_split<SCHEME>(c.y, u.y * ia, p.y, m.y);
          scheme_split<SCHEME>(c.z, u.z * ia, p.z, m.z);
          scheme_split<SCHEME>(c.w, u.w * ia, p.w, m.w);
          S.xp[sl_r[s] - 3][sl_q[s]] = p;
          S.xm[sl_r[s] - 3][sl_q[s]] = m;
        }
        if (sl_y[s]) {
          const float4 u = pv[s];
          float4 p, m;
          scheme_split<SCHEME>(c.x, u.x * ia, p.x, m.x);
          scheme_split<SCHEME>(c.y, u.y * ia, p.y, m.y);
          scheme_split<SCHEME>(c.z, u.z * ia, p.z, m.z);
          scheme_split<SCHEME>(c.w, u.w * ia, p.w, m.w);
          S.yp[sl_r[s]][sl_q[s] - 1] = p;
          S.ym[sl_r[s]][sl_q[s] - 1] = m;
        }
      }
    }
  };

  // own columns, ring level l (ghost levels reflect: c even, u_z odd); levels past the
  // ones any face reads are clamped into the lattice and never used
  float4 Rc, Ru, Rs = make_float4(0.f, 0.f, 0.f, 0.f);
  bool Rg = false;
  auto fetch_r = [&](int l) {
    Rg = l < 0 || l >= nz;
    int lr = l < 0 ? -1 - l : (l >= nz ? 2 * nz - 1 - l : l);
    lr = max(0, min(nz - 1, lr));
    const unsigned k3 = (unsigned)lr * plane + col;
    Rc = LoadNC::v4(cin + k3);
    Ru = LoadNC::v4(uz + k3);
    if (SUGAR) Rs = LoadNC::v4(a.S + k3);
  };
  auto put_r = [&](int slot) {
    const float s = Rg ? -ia : ia;
    float4 p, m;
    auto vsa = [&](float S_) { return SUGAR ? vs_a * fmaf(-a.ks, S_, 1.f) : vs_a; };
    scheme_split<SCHEME>(Rc.x, fmaf(Ru.x, s, -vsa(Rs.x)), p.x, m.x);
    scheme_split<SCHEME>(Rc.y, fmaf(Ru.y, s, -vsa(Rs.y)), p.y, m.y);
    scheme_split<SCHEME>(Rc.z, fmaf(Ru.z, s, -vsa(Rs.z)), p.z, m.z);
    scheme_split<SCHEME>(Rc.w, fmaf(Ru.w, s, -vsa(Rs.w)), p.w, m.w);
    S.zp[slot][tid] = p;
    S.zm[slot][tid] = m;
  };

  const int kb = z0 == 0 ? 0 : z0 - 1;  // first level: z0, or the priming level below it
  int ring[6];                          // slots of levels k-2 .. k+3
  {
    // first loads: level kb of the tile and the six ring levels, all in flight together
    float4 rc[6], ru[6], rs[6];
    bool rg[6];
    fetch_tile(kb);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      fetch_r(kb - 2 + j);
      rc[j] = Rc;
      ru[j] = Ru;
      if (SUGAR) rs[j] = Rs;
      rg[j] = Rg;
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      ring[j] = j;
      Rc = rc[j];
      Ru = ru[j];
      if (SUGAR) Rs = rs[j];
      Rg = rg[j];
      put_r(j);
    }
  }
  fetch_r(kb + 4);
  stage_tile();
  fetch_tile(kb + 1);  // kb + 1 <= z0 < nz
  float4 cn = make_float4(0.f, 0.f, 0.f, 0.f);
  if (STAGE > 1) cn = LoadNC::v4(a.c + (unsigned)kb * plane + col);
  float4 carry = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();

  for (int k = kb; k < z1; ++k) {
    const int b = k & 1;  // face exchange buffers
    const bool prime = k < z0;
    const float4 cq = S.c[3 + ty][1 + tx];  // c of level k at this thread's columns

    float fxq[4] = {0.f, 0.f, 0.f, 0.f};
    float4 fyl = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!prime) {
      // left x faces of the four columns (shared differences, as in the 2D kernel)
      {
        const float4 p0 = S.xp[ty][tx], p1 = S.xp[ty][tx + 1], p2 = S.xp[ty][tx + 2];
        const float4 m0 = S.xm[ty][tx], m1 = S.xm[ty][tx + 1], m2 = S.xm[ty][tx + 2];
        const float c0w = S.c[3 + ty][tx].w;
        x_faces<SCHEME>(p0, p1, p2, m0, m1, m2, c0w, cq, kd, fxq);
        S.fx[b][ty][tx] = fxq[0];
      }
      // lower y face of each column: y-split rows ty-3 .. ty+2 (staged rows ty .. ty+5)
      {
        float4 P[6], M[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          P[q] = S.yp[ty + q][tx];
          M[q] = S.ym[ty + q][tx];
        }
        const float4 cb = S.c[2 + ty][1 + tx];  // c of the row below
        fyl = column_faces<SCHEME>(P, M, kd, cb, cq);
        S.fy[b][ty][tx] = fyl;
      }
      // the tile's top y faces (warp 0, a column each) and right x faces (warp 1, a row each)
      if (tid < kV3W) {
        const float* P = reinterpret_cast<const float*>(&S.yp[kV3y][0]) + tid;
        const float* M = reinterpret_cast<const float*>(&S.ym[kV3y][0]) + tid;
        const float* C = reinterpret_cast<const float*>(&S.c[kV3y + 2][1]) + tid;
        float p[6], m[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          p[q] = P[q * kV3W];
          m[q] = M[q * kV3W];
        }
        reinterpret_cast<float*>(&S.fy[b][kV3y][0])[tid] = face_flux_scheme<SCHEME>(p, m, kd, C[0], C[4 * kV3Qx]);
      } else if (tid < kV3W + kV3y) {
        const int r = tid - kV3W;
        const float* P = reinterpret_cast<const float*>(&S.xp[r][0]) + kV3W + 1;  // column kV3W - 3
        const float* M = reinterpret_cast<const float*>(&S.xm[r][0]) + kV3W + 1;
        const float* C = reinterpret_cast<const float*>(&S.c[3 + r][0]) + kV3W + 3;
        float p[6], m[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          p[q] = P[q];
          m[q] = M[q];
        }
        S.fx[b][r][kV3x] = face_flux_scheme<SCHEME>(p, m, kd, C[0], C[1]);
      }
    }

    __syncthreads();
    // one staging buffer: level k + 1 replaces level k once every face has read it
    if (k + 1 < nz) stage_tile();
    if (k + 1 < z1 && k + 2 < nz) fetch_tile(k + 2);
    __syncthreads();

    // upper z face of each column from the ring (the lid face carries nothing); c of
    // level k + 1 at the own columns was staged before the barrier
    float fup[4] = {0.f, 0.f, 0.f, 0.f};
    if (k != nz - 1) {
      const float4 cnext = S.c[3 + ty][1 + tx];
      float4 P[6], M[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        P[q] = S.zp[ring[q]][tid];
        M[q] = S.zm[ring[q]][tid];
      }
      const float4 fu = column_faces<SCHEME>(P, M, kd, cq, cnext);
      fup[0] = fu.x;
      fup[1] = fu.y;
      fup[2] = fu.z;
      fup[3] = fu.w;
    }
    // ring: level k + 4 replaces level k - 2; fetch level k + 5
    put_r(ring[0]);
    fetch_r(k + 5);
    {
      const int r0 = ring[0];
#pragma unroll
      for (int j = 0; j < 5; ++j) ring[j] = ring[j + 1];
      ring[5] = r0;
    }

    // ---- divergence and the Shu-Osher combination of this stage
    if (!prime) {
      const float fr[4] = {fxq[1], fxq[2], fxq[3], S.fx[b][ty][tx + 1]};
      const float4 fyu = S.fy[b][ty + 1][tx];
      const float fyl4[4] = {fyl.x, fyl.y, fyl.z, fyl.w}, fyu4[4] = {fyu.x, fyu.y, fyu.z, fyu.w};
      const float ch[4] = {cq.x, cq.y, cq.z, cq.w};
      const float cnv[4] = {cn.x, cn.y, cn.z, cn.w};
      const float cy[4] = {carry.x, carry.y, carry.z, carry.w};
      float v[4], Lk[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) Lk[j] = fxq[j] - fr[j] + fyl4[j] - fyu4[j] + cy[j] - fup[j];
      if (k == 0) {  // the floor level's settling outflow (its lower face, carry, is 0)
        float vsf[4] = {a.vs, a.vs, a.vs, a.vs};
        if (SUGAR) {
          const float4 s0 = LoadNC::v4(a.S + col);
          vsf[0] *= fmaf(-a.ks, s0.x, 1.f);
          vsf[1] *= fmaf(-a.ks, s0.y, 1.f);
          vsf[2] *= fmaf(-a.ks, s0.z, 1.f);
          vsf[3] *= fmaf(-a.ks, s0.w, 1.f);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = rk_combine_floor<STAGE>(ch[j], Lk[j], alpha, cnv[j], vsf[j]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = rk_combine<STAGE>(ch[j], Lk[j], alpha, cnv[j]);
      }
      if (out) {
        *reinterpret_cast<float4*>(sp.cout + (unsigned)k * plane + col) = make_float4(v[0], v[1], v[2], v[3]);
        if (STAGE == 3)
          report_status(a.status, !(isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]) && isfinite(v[3])));
      }
    }
    carry = make_float4(fup[0], fup[1], fup[2], fup[3]);
    if (STAGE > 1 && k + 1 < z1) cn = LoadNC::v4(a.c + (unsigned)(k + 1) * plane + col);
  }
}

template <int STAGE, bool SUGAR = false, int SCHEME = 0>
__global__ void __launch_bounds__(kV3T, 4) rk_sweep3d_wide_kernel(Args<float> a, Sweep3dParams sp) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  sweep3d_wide_body<STAGE, SUGAR, SCHEME>(*reinterpret_cast<Sweep3dWideSmem*>(smem_raw), a, sp);
}

using Sweep3dKernel = void (*)(Args<float>, Sweep3dParams);

// The stage kernel of the handle's sugar and transport scheme (runtime fields).
template <int STAGE>
inline Sweep3dKernel sweep3d_wide_entry(bool sugar, int scheme) {
  switch (scheme) {
    case kSchemeWeno3:
      return sugar ? rk_sweep3d_wide_kernel<STAGE, true, kSchemeWeno3> : rk_sweep3d_wide_kernel<STAGE, false, kSchemeWeno3>;
    case kSchemeSignSplit:
      return sugar ? rk_sweep3d_wide_kernel<STAGE, true, kSchemeSignSplit>
                   : rk_sweep3d_wide_kernel<STAGE, false, kSchemeSignSplit>;
    case kSchemeWeno3 | kSchemeSignSplit:
      return sugar ? rk_sweep3d_wide_kernel<STAGE, true, kSchemeWeno3 | kSchemeSignSplit>
                   : rk_sweep3d_wide_kernel<STAGE, false, kSchemeWeno3 | kSchemeSignSplit>;
    default:
      return sugar ? rk_sweep3d_wide_kernel<STAGE, true> : rk_sweep3d_wide_kernel<STAGE>;
  }
}

inline size_t sweep3d_wide_smem() { return sizeof(Sweep3dWideSmem); }

inline cudaError_t sweep3d_wide_prepare(bool sugar, int scheme) {
  const int bytes = (int)sizeof(Sweep3dWideSmem);
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(sweep3d_wide_entry<1>(sugar, scheme), at, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep3d_wide_entry<2>(sugar, scheme), at, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep3d_wide_entry<3>(sugar, scheme), at, bytes);
  return e;
}

// Levels per segment of the four-column kernel: the height that minimises launch waves x
// (H + 2) for the resident CTA count, as for the 2D kernel; capped at kV3maxH.
inline int sweep3d_wide_rows(int nx, int ny, int nz, int sm_count, int per_sm, int override_rows) {
  if (override_rows > 0) return min(min(override_rows, nz), kV3maxH);
  const long long tiles = (long long)((nx + kV3W - 1) / kV3W) * ((ny + kV3y - 1) / kV3y);
  const long long slots = (long long)max(1, per_sm) * max(1, sm_count);
  int best = min(2, nz);
  double best_cost = 1e300;
  for (int H = 2; H <= kV3maxH; ++H) {
    const long long ctas = tiles * ((nz + H - 1) / H);
    const long long waves = (ctas + slots - 1) / slots;
    const double cost = (double)waves * (H + 2) - 1e-6 * (double)ctas / (double)(waves * slots);
    if (cost < best_cost) {
      best_cost = cost;
      best = H;
    }
    if (H >= nz) break;
  }
  return min(best, nz);
}

template <int STAGE>
inline cudaError_t launch_sweep3d_wide(const Args<float>& a, const float* cin, float* cout, int H, cudaStream_t s) {
  Sweep3dParams sp;
  sp.cin = cin;
  sp.cout = cout;
  sp.H = H;
  sp.ghost_shift = 2.f * a.vs * a.inv_alpha;
  const dim3 grid((a.nx + kV3W - 1) / kV3W, (a.ny + kV3y - 1) / kV3y, (a.nz + H - 1) / H);
  sweep3d_wide_entry<STAGE>(a.S != nullptr, a.scheme)<<<grid, dim3(kV3x, kV3y), sizeof(Sweep3dWideSmem), s>>>(a, sp);
  return cudaGetLastError();
}

}  // namespace lw
