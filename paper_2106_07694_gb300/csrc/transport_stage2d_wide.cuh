// 2D FP32 transport with four adjacent columns per thread: one SSP-RK3 stage of the
// WENO5 + diffusion + settling update of c (steps a4..a8; the stage-3 kernel also folds
// the floor deposit, a9).  The scheme variants and the sugar scalar are compile-time
// forms of the same kernel; against one column per thread, which shares no differences between
// faces, their steps take 122 -> 88 us (sugar, 1024 x 2048), 129 -> 92 (WENO3, 1536 x 2048) and
// 136 -> 103 (sign split).
//
// A CTA of kWT threads owns a strip of kWW = 4 kWT columns and a segment of rows and
// sweeps it upward.  At row k:
//  - the x-split fluxes and c of row k+1 on the strip plus one four-column halo quad on
//    each side are staged in shared memory as float4 quads, double-buffered by row
//    parity and loaded one row ahead, so the row needs a single barrier;
//  - each thread reconstructs the left x faces of its four columns from three quads of
//    h+/alpha, three of h-/alpha and two of c, sharing the first and second differences
//    of the split fluxes between the four faces; the right face of its last column is
//    its neighbour's first face, and for the strip's last column it is computed for the
//    whole segment before the sweep;
//  - the upper y face of each of its columns comes from a private ring of the y-split
//    fluxes of rows k-2 .. k+3 (one float4 per row and split half), filled three rows
//    ahead; the lower y face is carried from the previous row;
//  - stages 2 and 3 also combine with c^n at the node, copied two rows ahead by cp.async
//    into a three-row ring in shared memory (no registers held while it is in flight).
// Every face is computed once, with the arithmetic of face_flux_x, so
// the faces and the updated c are bitwise those of the one-column kernel.
//
// Bound by instruction issue with 12 warps an SM (128-133 registers, six CTAs; a cap that lets
// seven or eight in costs more in moves than they give, 280 -> 290 us a step).  2048 x 4096:
// 61.4 / 62.4 / 65.6 us a stage, 65.7 / 67.4 / 69.4 with the longer form of the reconstruction
// (weno.cuh) and the first loads one after the other.
#pragma once
#include "common.cuh"
#include "weno.cuh"
#include "transport_stage2d.cuh"  // Stage2dParams

namespace lw {

constexpr int kWq = 4;           // columns per thread (one float4)
constexpr int kWT = 64;          // threads per CTA
constexpr int kWW = kWq * kWT;   // columns per strip
constexpr int kWQ = kWT + 2;     // staged quads per row: the strip and one halo quad per side
constexpr int kWring = 6;        // y ring rows (k-2 .. k+3)
constexpr int kWmaxH = 64;       // longest row segment (its strip-edge faces are held in smem)
constexpr int kWminB = 1;        // CTAs per SM the register allocation must allow

struct StageWideSmem {
  float4 xp[2][kWQ];  // x-split h+/alpha of the staged row, by row parity
  float4 xm[2][kWQ];  // x-split h-/alpha
  float4 xc[2][kWQ];  // stage input c
  float4 yp[kWring][kWT];  // y-split ring of each thread's four columns
  float4 ym[kWring][kWT];
  float fx[2][kWT + 1];  // first left x face of each thread (+ the strip's right edge), by row parity
  float edge[kWmaxH];    // the strip's right-edge x face for each row of the segment
  float4 cn[3][kWT];     // stages 2, 3: c^n of rows k .. k+2 at each thread's columns (cp.async ring)
  double red[kWT / 32];
  bool last;
};

// Sum over eight neighbouring lanes (32 columns), valid in the first of each eight.
__device__ __forceinline__ double tile_group_sum(double v) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Lax-Friedrichs split of one node: p = h+/alpha, m = h-/alpha with h = c/2, w = u/alpha.
__device__ __forceinline__ void lf_split(float c, float w, float& p, float& m) {
  const float h = 0.5f * c;
  p = fmaf(w, h, h);
  m = fmaf(w, h, -h);
}

// The pair a scheme stages at one node from c and w / alpha: the Lax-Friedrichs halves, or
// for the sign split w c / alpha and w / alpha (face_flux_scheme).
template <int SCHEME>
__device__ __forceinline__ void scheme_split(float c, float w, float& p, float& m) {
  if (SCHEME & kSchemeSignSplit) {
    p = w * c;
    m = w;
  } else {
    lf_split(c, w, p, m);
  }
}

// Left x faces (divided by alpha) of four adjacent columns x .. x+3 from the staged quads of
// columns x-4 .. x+7 (p, m: the scheme's pair), c of column x-1 and of the four: the first and
// second differences are shared between the faces.
template <int SCHEME>
__device__ __forceinline__ void x_faces(const float4& p0, const float4& p1, const float4& p2, const float4& m0,
                                        const float4& m1, const float4& m2, float c0w, const float4& cq, float kd,
                                        float (&fxq)[4]) {
  const float C[5] = {c0w, cq.x, cq.y, cq.z, cq.w};  // c at columns x-1 .. x+3
  if constexpr (SCHEME == 0) {
    const float P[8] = {p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w, p2.x};  // h+ at columns x-3 .. x+4
    const float M[8] = {m0.z, m0.w, m1.x, m1.y, m1.z, m1.w, m2.x, m2.y};  // h- at columns x-2 .. x+5
    float D[7], E[7], SD[6], SE[6];
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      D[j] = P[j + 1] - P[j];
      E[j] = M[j + 1] - M[j];
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      SD[j] = D[j + 1] - D[j];
      SE[j] = E[j + 1] - E[j];
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {  // face between columns x - 1 + f and x + f
      const Recon<float> hp = weno5_recon(D[f], D[f + 1], D[f + 2], D[f + 3], SD[f], SD[f + 1], SD[f + 2]);
      const Recon<float> hm = weno5_recon(-E[f + 3], -E[f + 2], -E[f + 1], -E[f], SE[f + 2], SE[f + 1], SE[f]);
      fxq[f] = fmaf(kd, C[f] - C[f + 1], recon_sum(hp, P[f + 2], hm, M[f + 2]));
    }
  } else if constexpr (SCHEME == kSchemeWeno3) {  // three values a half: h+ at x-2 .. x+3, h- at x-1 .. x+4
    const float P[6] = {p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
    const float M[6] = {m0.w, m1.x, m1.y, m1.z, m1.w, m2.x};
    float D[5], E[5], A[5], B[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      D[j] = P[j + 1] - P[j];
      E[j] = M[j + 1] - M[j];
      A[j] = weno3_smooth(D[j]);
      B[j] = weno3_smooth(E[j]);
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const Recon<float> hp = weno3_recon(D[f], D[f + 1], A[f], A[f + 1]);
      const Recon<float> hm = weno3_recon(-E[f + 1], -E[f], B[f + 1], B[f]);
      fxq[f] = fmaf(kd, C[f] - C[f + 1], recon_sum(hp, P[f + 1], hm, M[f + 1]));
    }
  } else {  // sign split: w c at columns x-3 .. x+5, w at x-1 .. x+3
    const float P[9] = {p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w, p2.x, p2.y};
    const float W[5] = {m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float p[6] = {P[f], P[f + 1], P[f + 2], P[f + 3], P[f + 4], P[f + 5]};
      const float m[6] = {0.f, 0.f, W[f], W[f + 1], 0.f, 0.f};
      fxq[f] = face_flux_scheme<SCHEME>(p, m, kd, C[f], C[f + 1]);
    }
  }
}

// Faces between the third and fourth of six stacked rows, of four columns: P[q], M[q] the
// staged pairs of row q, cl and cr c of rows 2 and 3.
template <int SCHEME>
__device__ __forceinline__ float4 column_faces(const float4 (&P)[6], const float4 (&M)[6], float kd, const float4& cl,
                                               const float4& cr) {
  auto face = [&](auto get, float l, float r) {
    float p[6], m[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      p[q] = get(P[q]);
      m[q] = get(M[q]);
    }
    return face_flux_scheme<SCHEME>(p, m, kd, l, r);
  };
  return make_float4(face([](const float4& v) { return v.x; }, cl.x, cr.x),
                     face([](const float4& v) { return v.y; }, cl.y, cr.y),
                     face([](const float4& v) { return v.z; }, cl.z, cr.z),
                     face([](const float4& v) { return v.w; }, cl.w, cr.w));
}

// SUGAR: the settling velocity of a node is Vs (1 - ks S).  SCHEME: transport-scheme variant
// bits (face_flux_scheme).  LD: the global-load policy (LoadPlain for a launch of its own, LoadL2
// inside a kernel whose earlier phases wrote the fields).
template <int STAGE, bool SUGAR = false, int SCHEME = 0, class LD = LoadPlain>
__device__ __forceinline__ void stage2d_wide_body(StageWideSmem& S, const Args<float>& a, const Stage2dParams& sp,
                                                  int bx, int by, int strips) {
  const int t = threadIdx.x;
  const int nx = a.nx, ny = a.ny;
  const int x0 = bx * kWW;
  const int y0 = by * sp.H, y1 = min(ny, y0 + sp.H);
  const int xl = x0 + kWq * t;  // first column of this thread (past a ragged strip end: wrapped)
  const bool out = xl < nx;
  const unsigned X = (unsigned)(xl % nx);
  const float ia = a.inv_alpha, vs_a = a.vs * a.inv_alpha, alpha = a.alpha, kd = a.kappa * a.inv_alpha;
  const float* cin = sp.cin;
  const float* ux = a.u;
  const float* uy = a.u + a.n;

  // halo quads of the staged row: thread 0 the quad left of the strip, thread 1 the one right of it
  const bool halo = t < 2;
  const int hslot = t == 0 ? 0 : kWQ - 1;
  const unsigned hX = (unsigned)(t == 0 ? ((x0 - kWq) % nx + nx) % nx : (x0 + kWW) % nx);

  float4 Xc, Xu, Hc = make_float4(0.f, 0.f, 0.f, 0.f), Hu = Hc;
  auto fetch_x = [&](int r) {
    const unsigned row = (unsigned)r * (unsigned)nx;
    Xc = LD::v4(cin + row + X);
    Xu = LD::v4(ux + row + X);
    if (halo) {
      Hc = LD::v4(cin + row + hX);
      Hu = LD::v4(ux + row + hX);
    }
  };
  auto put_quad = [&](int b, int q, const float4& c, const float4& u) {
    float4 p, m;
    scheme_split<SCHEME>(c.x, u.x * ia, p.x, m.x);
    scheme_split<SCHEME>(c.y, u.y * ia, p.y, m.y);
    scheme_split<SCHEME>(c.z, u.z * ia, p.z, m.z);
    scheme_split<SCHEME>(c.w, u.w * ia, p.w, m.w);
    S.xp[b][q] = p;
    S.xm[b][q] = m;
    S.xc[b][q] = c;
  };
  auto stage_x = [&](int b) {
    put_quad(b, t + 1, Xc, Xu);
    if (halo) put_quad(b, hslot, Hc, Hu);
  };

  // own columns, ring row l (ghost rows reflect: c even, u_y odd); rows past the ones any
  // face reads are clamped into the lattice and never used
  float4 Rc, Ru, Rs = make_float4(0.f, 0.f, 0.f, 0.f);
  bool Rg = false;
  auto fetch_r = [&](int l) {
    Rg = l < 0 || l >= ny;
    int lr = l < 0 ? -1 - l : (l >= ny ? 2 * ny - 1 - l : l);
    lr = max(0, min(ny - 1, lr));
    const unsigned row = (unsigned)lr * (unsigned)nx;
    Rc = LD::v4(cin + row + X);
    Ru = LD::v4(uy + row + X);
    if (SUGAR) Rs = LD::v4(a.S + row + X);
  };
  // ring entries are addressed by byte offset (slot * kWT + t) * 16, rotated as the sweep advances
  auto ring_at = [&](float4 (*arr)[kWT], unsigned off) -> float4& {
    return *reinterpret_cast<float4*>(reinterpret_cast<char*>(&arr[0][0]) + off);
  };
  auto put_r = [&](unsigned off) {
    const float s = Rg ? -ia : ia;
    float4 p, m;
    auto vsa = [&](float S_) { return SUGAR ? vs_a * fmaf(-a.ks, S_, 1.f) : vs_a; };
    scheme_split<SCHEME>(Rc.x, fmaf(Ru.x, s, -vsa(Rs.x)), p.x, m.x);
    scheme_split<SCHEME>(Rc.y, fmaf(Ru.y, s, -vsa(Rs.y)), p.y, m.y);
    scheme_split<SCHEME>(Rc.z, fmaf(Ru.z, s, -vsa(Rs.z)), p.z, m.z);
    scheme_split<SCHEME>(Rc.w, fmaf(Ru.w, s, -vsa(Rs.w)), p.w, m.w);
    ring_at(S.yp, off) = p;
    ring_at(S.ym, off) = m;
  };

  const int kb = y0 == 0 ? 0 : y0 - 1;  // first row: y0, or the priming row below it
  // first loads: the six ring rows and row kb, all in flight together (one after the other
  // they cost a trip to memory each: the 256 x 512 step 20.4 -> 18.6 us, 1024 x 2048 84.0 -> 80.1)
  float4 rc[kWring], ru[kWring], rs[kWring];
  bool rg[kWring];
#pragma unroll
  for (int j = 0; j < kWring; ++j) {
    fetch_r(kb - 2 + j);
    rc[j] = Rc;
    ru[j] = Ru;
    if (SUGAR) rs[j] = Rs;
    rg[j] = Rg;
  }
  fetch_x(kb);

  // right-edge x face of every row of the segment (full strips; a ragged strip's last
  // column takes the first face of the next, wrapped, thread)
  for (int r = t; r < y1 - y0; r += kWT) {
    float e = 0.f;
    if (x0 + kWW <= nx) {
      const unsigned row = (unsigned)(y0 + r) * (unsigned)nx;
      float P[6], M[6], C[6];
#pragma unroll
      for (int o = 0; o < 6; ++o) {
        const unsigned col = (unsigned)wrap_inc(x0 + kWW - 3 + o, nx);
        C[o] = LD::s(cin + row + col);
        scheme_split<SCHEME>(C[o], LD::s(ux + row + col) * ia, P[o], M[o]);
      }
      e = face_flux_scheme<SCHEME>(P, M, kd, C[2], C[3]);
    }
    S.edge[r] = e;
  }

  unsigned ring[kWring];  // rows k-2 .. k+3
#pragma unroll
  for (int j = 0; j < kWring; ++j) {
    ring[j] = (unsigned)((j * kWT + t) * sizeof(float4));
    Rc = rc[j];
    Ru = ru[j];
    if (SUGAR) Rs = rs[j];
    Rg = rg[j];
    put_r(ring[j]);
  }
  fetch_r(kb + 4);
  stage_x(kb & 1);
  fetch_x(kb + 1);  // kb + 1 <= y0 < ny
  // stages 2, 3: c^n of this thread's columns, copied two rows ahead into a three-row ring
  // (each thread reads back only its own copies: a wait per thread, no barrier)
  auto fetch_cn = [&](int r) {
    if (STAGE > 1 && r < y1) cp_async16(&S.cn[r % 3][t], a.c + (unsigned)r * (unsigned)nx + X);
    if (STAGE > 1) cp_async_commit();
  };
  fetch_cn(kb);
  fetch_cn(kb + 1);
  float4 carry = make_float4(0.f, 0.f, 0.f, 0.f);
  double dep = 0.0;  // stage 3, floor row: this thread's Vs-free deposit term
  __syncthreads();

  for (int k = kb; k < y1; ++k) {
    const int b = k & 1;
    const bool prime = k < y0;
    // ---- stage row k + 1 into the other buffer, fetch row k + 2
    const float4 cnext = Xc;  // c of row k + 1 at this thread's columns
    if (k + 1 < y1) stage_x(b ^ 1);
    if (k + 1 < y1 && k + 2 < ny) fetch_x(k + 2);
    const float4 cq = S.xc[b][t + 1];  // c of row k at this thread's columns

    // ---- left x faces of this thread's four columns
    float fxq[4] = {0.f, 0.f, 0.f, 0.f};
    if (!prime) {
      const float4 p0 = S.xp[b][t], p1 = S.xp[b][t + 1], p2 = S.xp[b][t + 2];
      const float4 m0 = S.xm[b][t], m1 = S.xm[b][t + 1], m2 = S.xm[b][t + 2];
      const float c0w = S.xc[b][t].w;
      x_faces<SCHEME>(p0, p1, p2, m0, m1, m2, c0w, cq, kd, fxq);
      S.fx[b][t] = fxq[0];
      if (t == kWT - 1) S.fx[b][kWT] = S.edge[k - y0];
    }

    // ---- upper y face of each column (the lid face carries nothing)
    float fup[4] = {0.f, 0.f, 0.f, 0.f};
    if (k != ny - 1) {
      float4 P[6], M[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        P[q] = ring_at(S.yp, ring[q]);
        M[q] = ring_at(S.ym, ring[q]);
      }
      const float4 fu = column_faces<SCHEME>(P, M, kd, cq, cnext);
      fup[0] = fu.x;
      fup[1] = fu.y;
      fup[2] = fu.z;
      fup[3] = fu.w;
    }
    // ---- ring: row k + 4 replaces row k - 2; fetch row k + 5
    put_r(ring[0]);
    fetch_r(k + 5);
    {
      const unsigned r0 = ring[0];
#pragma unroll
      for (int j = 0; j < kWring - 1; ++j) ring[j] = ring[j + 1];
      ring[kWring - 1] = r0;
    }
    __syncthreads();

    // ---- divergence and the Shu-Osher combination of this stage
    float4 cn = make_float4(0.f, 0.f, 0.f, 0.f);
    if (STAGE > 1) {
      cp_async_wait<1>();  // row k landed (row k + 1 may still fly)
      cn = S.cn[k % 3][t];
    }
    if (!prime) {
      const float fr[4] = {fxq[1], fxq[2], fxq[3], S.fx[b][t + 1]};
      const float ch[4] = {cq.x, cq.y, cq.z, cq.w};
      const float cnv[4] = {cn.x, cn.y, cn.z, cn.w};
      const float cy[4] = {carry.x, carry.y, carry.z, carry.w};
      float v[4], Lk[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) Lk[j] = fxq[j] - fr[j] + (cy[j] - fup[j]);
      float vsf[4] = {a.vs, a.vs, a.vs, a.vs};
      if (k == 0) {  // the floor row's settling outflow (its lower face, carry, is 0)
        if (SUGAR) {
          const float4 s0 = LD::v4(a.S + X);
          vsf[0] *= fmaf(-a.ks, s0.x, 1.f);
          vsf[1] *= fmaf(-a.ks, s0.y, 1.f);
          vsf[2] *= fmaf(-a.ks, s0.z, 1.f);
          vsf[3] *= fmaf(-a.ks, s0.w, 1.f);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
          v[j] = rk_combine_floor<STAGE>(ch[j], Lk[j], alpha, cnv[j], vsf[j]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = rk_combine<STAGE>(ch[j], Lk[j], alpha, cnv[j]);
      }
      if (out) {
        *reinterpret_cast<float4*>(sp.cout + (unsigned)k * (unsigned)nx + X) = make_float4(v[0], v[1], v[2], v[3]);
        if (STAGE == 3) {
          report_status(a.status, !(isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]) && isfinite(v[3])));
          if (k == 0) {  // RK3 b-weights of the floor flux: c^n/6 + c1/6 + 2 c2/3
            const float4 c1 = LD::v4(a.c1 + X);
            const float c1v[4] = {c1.x, c1.y, c1.z, c1.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const double b_ = fma((double)cnv[j] + (double)c1v[j], 1.0 / 6.0, (double)ch[j] * (2.0 / 3.0));
              dep += SUGAR ? b_ * (double)vsf[j] : b_;  // with sugar Vs(S) per node, else Vs once at the fold
            }
          }
        }
      }
    }
    carry = make_float4(fup[0], fup[1], fup[2], fup[3]);
    fetch_cn(k + 2);
  }
  if (STAGE > 1) cp_async_wait<0>();

  // stage 3: the CTAs holding the floor row fold the deposit of this step (FP64, fixed
  // order: warp shuffles, then a warp of the last CTA folds the per-CTA partials)
  if (STAGE == 3 && y0 == 0) {
    double v = tile_group_sum(dep);
    v += __shfl_down_sync(0xffffffffu, v, 8);
    v += __shfl_down_sync(0xffffffffu, v, 16);
    if ((t & 31) == 0) S.red[t >> 5] = v;
    __syncthreads();
    if (t == 0) {
      double s2 = 0.0;
      for (int w = 0; w < kWT / 32; ++w) s2 += S.red[w];
      if (!SUGAR) s2 *= (double)a.vs;
      S.last = false;
      if (strips == 1) {  // nothing to wait for: no fence and ticket
        *reinterpret_cast<volatile double*>(a.scalars) += s2;
      } else {
        a.partials[bx] = s2;
        __threadfence();
        S.last = atomicAdd(a.ticket, 1u) == (unsigned)strips - 1;
      }
    }
    __syncthreads();
    if (S.last && t < 32) {
      __threadfence();
      const double prev = *reinterpret_cast<volatile double*>(a.scalars);  // written by earlier steps
      const double tot = fold_partials(a.partials, strips);
      if (t == 0) {
        a.scalars[0] = prev + tot;
        *a.ticket = 0u;
      }
    }
  }
}

template <int STAGE, bool SUGAR = false, int SCHEME = 0>
__global__ void __launch_bounds__(kWT, kWminB) rk_stage2d_wide_kernel(Args<float> a, Stage2dParams sp) {
  after_previous();
  __shared__ __align__(16) StageWideSmem S;
  stage2d_wide_body<STAGE, SUGAR, SCHEME>(S, a, sp, blockIdx.x, blockIdx.y, gridDim.x);
}

using StageWideKernel = void (*)(Args<float>, Stage2dParams);

// The stage kernel of the handle's sugar and transport scheme (runtime fields).
template <int STAGE>
inline StageWideKernel stage2d_wide_entry(bool sugar, int scheme) {
  switch (scheme) {
    case kSchemeWeno3:
      return sugar ? rk_stage2d_wide_kernel<STAGE, true, kSchemeWeno3> : rk_stage2d_wide_kernel<STAGE, false, kSchemeWeno3>;
    case kSchemeSignSplit:
      return sugar ? rk_stage2d_wide_kernel<STAGE, true, kSchemeSignSplit>
                   : rk_stage2d_wide_kernel<STAGE, false, kSchemeSignSplit>;
    case kSchemeWeno3 | kSchemeSignSplit:
      return sugar ? rk_stage2d_wide_kernel<STAGE, true, kSchemeWeno3 | kSchemeSignSplit>
                   : rk_stage2d_wide_kernel<STAGE, false, kSchemeWeno3 | kSchemeSignSplit>;
    default:
      return sugar ? rk_stage2d_wide_kernel<STAGE, true> : rk_stage2d_wide_kernel<STAGE>;
  }
}

// Rows per segment of the four-column kernel.  The CTAs of a launch run in waves of
// sm_count x per_sm (the CTAs the SMs hold at once), and a CTA's time grows with its rows
// plus about two rows of set-up (ring fill, priming row), so take the height that
// minimises waves x (H + 2); ties go to the fuller last wave.  Capped at kWmaxH.
inline int stage2d_wide_rows(int nx, int ny, int sm_count, int per_sm, int override_rows) {
  if (override_rows > 0) return min(min(override_rows, ny), kWmaxH);
  const long long strips = (nx + kWW - 1) / kWW;
  const long long slots = (long long)max(1, per_sm) * max(1, sm_count);
  int best = min(2, ny);
  double best_cost = 1e300;
  for (int H = 2; H <= kWmaxH; ++H) {
    const long long ctas = strips * ((ny + H - 1) / H);
    const long long waves = (ctas + slots - 1) / slots;
    const double cost = (double)waves * (H + 2) - 1e-6 * (double)ctas / (double)(waves * slots);
    if (cost < best_cost) {
      best_cost = cost;
      best = H;
    }
    if (H >= ny) break;
  }
  return min(best, ny);
}

template <int STAGE>
inline cudaError_t launch_stage2d_wide(const Args<float>& a, const float* cin, float* cout, int H, cudaStream_t s) {
  Stage2dParams sp;
  sp.cin = cin;
  sp.cout = cout;
  sp.H = H;
  const dim3 grid((a.nx + kWW - 1) / kWW, (a.ny + H - 1) / H);
  launch_dependent(stage2d_wide_entry<STAGE>(a.S != nullptr, a.scheme), grid, kWT, 0, s, a, sp);
  return cudaGetLastError();
}

}  // namespace lw
