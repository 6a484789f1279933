// FP32 adjoint of one SSP-RK3 stage of the transport on tiles: every face's flux derivatives
// and their sum over the nodes of its stencil in one pass, nothing recorded per face.
//
// With h+- = (w/alpha +- 1) c / 2 (divided by alpha) a face flux depends on the four
// differences of h+ over its stencil, the four of h- and the two centre values.  Summed over
// the faces, weighted with lamF (lambda of the node the flux enters less that of the one it
// leaves), the derivatives with respect to the differences give one value ED per difference
// and half, and the derivative with respect to h+ at node i is
//   GP_i = ED_{i-1} - ED_i + lamF(face whose h+ is centred on i),   likewise GM_i for h-;
// with them
//   d/dc_i = alpha/2 [GP_i (w_i/alpha + 1) + GM_i (w_i/alpha - 1)] + kappa (lamF_right - lamF_left)
//   d/dw_i = c_i/2 (GP_i + GM_i).
// So a face adds eight values instead of recording 24, and c and w enter once per node.
//
// A CTA owns kAx x kAy nodes.  It stages the split fluxes along y (tile columns, four-row halo
// above and below) and along x (tile rows, four-column halo on each side) and lambda; a thread
// then takes four consecutive faces of one column (or row), shares the differences between
// them, sums their contributions to seven differences in registers and leaves them in shared
// memory: four for the block of its own faces, three for the one below.  The halo's faces (two
// below, three above) are computed again by the neighbouring tile, 37 faces for 32 nodes.
// Then a thread gathers four nodes.  Ghost rows behind the walls are stencil nodes like any
// other (c even, u odd); their derivatives go to the nodes they mirror.
//
// Bound by instruction issue: about 75 FP32 operations and 4 reciprocals a reconstruction.
// Against a kernel that records each face's derivatives (24 fields, 50 MB through L2 a stage on
// 512 x 1024) and one that gathers them, the gradient of 100 steps there took 11.45 instead of
// 14.47 ms; with a tile's loads sent together and the forward steps it replays made faster it
// takes 9.2.  494-505 instructions a node and stage, 56-59 % of the issue slots while it runs.  The FP64 build keeps that pair (adjoint.cuh).
#pragma once
#include "common.cuh"
#include "weno.cuh"
#include "adjoint.cuh"

#include <type_traits>

namespace lw {

constexpr int kAx = 32, kAy = 32;        // tile (nodes)
constexpr int kAT = kAx * kAy / 4;       // threads: four nodes each
constexpr int kAg = kAx / 4 + 2;         // blocks of four faces along an axis, one halo block per side
static_assert(kAx == kAy && kAx == 32, "a warp is one block of a tile's columns");

struct AdjTileSmem {
  float lam[kAy + 8][kAx + 8];  // lambda of the stage output, scaled
  float px[kAy][kAx + 8];       // x-split h+/alpha, h-/alpha of the tile rows
  float mx[kAy][kAx + 8];
  float py[kAy + 8][kAx];       // y-split of the tile columns; later the y parts of d/dc and d/dw
  float my[kAy + 8][kAx];
  union {
    float y[2][kAg][8][kAx];         // ED by half, block, element (0..3 own block, 5..7 the block below), column
    float4 x[2][2][kAy][kAg];        // ED by half, own / below, row, block
  } ed;
  float vs_red[kAT];       // Vs terms of the threads, and of the floor nodes
  double vs_floor[kAx];
};

// Derivatives e[0..3] of a WENO5 face value with respect to its differences d1..d4 (upwind side
// first).  With beta_k, r_k as in weno5_recon, w_k the normalised weights and R = sum w_k r_k:
//   2 e_m = sum_k w_k dr_k/dd_m - 2 sum_k (r_k - R) w_k / (eps + beta_k) dbeta_k/dd_m.
__device__ __forceinline__ void weno5_diff_grad(float d1, float d2, float d3, float d4, float s0, float s1, float s2,
                                                float (&e)[4]) {
  const float eps = 0.75e-6f, g2 = 0.75f * d2, g3 = 0.75f * d3;
  const float i0 = rcp_approx(fmaf(g2, d2 + s0, fmaf(s0, s0, eps)));
  const float i1 = rcp_approx(fmaf(g2, d3, fmaf(s1, s1, eps)));
  const float i2 = rcp_approx(fmaf(g3, d3 - s2, fmaf(s2, s2, eps)));
  const float r0 = fmaf(2.f / 3.f, s0, d2), r1 = fmaf(2.f / 3.f, s1, d2), r2 = fmaf(-1.f / 3.f, s2, d3);
  const float a0 = i0 * i0, a1 = 6.f * (i1 * i1), a2 = 3.f * (i2 * i2);
  const float inv = rcp_approx(a0 + a1 + a2);
  const float w0 = a0 * inv, w1 = a1 * inv, w2 = a2 * inv;
  const float R = fmaf(w2, r2, fmaf(w1, r1, w0 * r0));
  const float q0 = (R - r0) * (w0 * i0), q1 = (R - r1) * (w1 * i1), q2 = (R - r2) * (w2 * i2);
  e[0] = fmaf(q0, fmaf(-2.75f, d2, 2.f * d1), (-1.f / 3.f) * w0);
  e[1] = fmaf(q0, fmaf(-2.75f, d1, 5.f * d2), fmaf(q1, fmaf(-1.25f, d3, 2.f * d2), fmaf(5.f / 6.f, w0, (1.f / 6.f) * w1)));
  e[2] = fmaf(q2, fmaf(-2.75f, d4, 5.f * d3), fmaf(q1, fmaf(-1.25f, d2, 2.f * d3), fmaf(2.f / 3.f, w2, (1.f / 3.f) * w1)));
  e[3] = fmaf(q2, fmaf(-2.75f, d3, 2.f * d4), (-1.f / 6.f) * w2);
}

// Faces F0 .. F1-1 of a block of four: P = h+ at the eight nodes from three below the block's
// first face's upper node, M = h- from two below it; lamF of the faces.  Adds to the seven
// differences of P (from node -3 on) and of M (from node -2 on).
template <int F0, int F1>
__device__ __forceinline__ void block_faces(const float (&P)[8], const float (&M)[8], const float (&lamF)[4],
                                            float (&accP)[7], float (&accM)[7]) {
  float D[7], E[7], SD[6], SE[6];
#pragma unroll
  for (int j = 0; j < 7; ++j) {
    D[j] = P[j + 1] - P[j];
    E[j] = M[j + 1] - M[j];
    accP[j] = accM[j] = 0.f;
  }
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    SD[j] = D[j + 1] - D[j];
    SE[j] = E[j + 1] - E[j];
  }
#pragma unroll
  for (int f = F0; f < F1; ++f) {
    float e[4];
    weno5_diff_grad(D[f], D[f + 1], D[f + 2], D[f + 3], SD[f], SD[f + 1], SD[f + 2], e);
#pragma unroll
    for (int m = 0; m < 4; ++m) accP[f + m] = fmaf(lamF[f], e[m], accP[f + m]);
    weno5_diff_grad(-E[f + 3], -E[f + 2], -E[f + 1], -E[f], SE[f + 2], SE[f + 1], SE[f], e);
#pragma unroll
    for (int m = 0; m < 4; ++m) accM[f + 3 - m] = fmaf(-lamF[f], e[m], accM[f + 3 - m]);
  }
}

// GP, GM of node i (tile-local, -2 .. kAy + 1) of a column: sums of the two blocks' shares.
__device__ __forceinline__ float column_ed(const AdjTileSmem& S, int half, int j, int col) {
  const int b = (j + 4) >> 2, e = j & 3;
  float v = S.ed.y[half][b][e][col];
  if (e > 0 && b + 1 < kAg) v += S.ed.y[half][b + 1][4 + e][col];
  return v;
}

// (hi, lo) += (h, l): the rounding error of hi + h (Knuth's two-sum) is kept in lo, so a sum of
// FP32 terms that cancel is held to about 2^-47 of their size without the narrow FP64 pipe.
__device__ __forceinline__ void add_pair(float& hi, float& lo, float h, float l) {
  const float s = hi + h, b = s - hi;
  lo += l + ((hi - (s - b)) + (h - b));
  hi = s;
}

// One stage backwards (STAGE 3, 2, 1: lambda of c', c2, c1 scaled by 2/3, 1/4, 1):
//   STAGE 3: lc2 = lamL + L^T lamL, lambda(u) written
//   STAGE 2: lc1 = lamL + L^T lamL, lambda(u) accumulated
//   STAGE 1: lc = 1/3 mu + 3/4 lc2 + lamL + L^T lamL, lambda(u) accumulated
// with the deposit's floor terms and the floor face; the Vs terms (w = +-u - Vs on vertical
// faces, the floor face -Vs c_0 and the deposit's weights) go to this CTA's partial.
template <int STAGE>
__global__ void __launch_bounds__(kAT, 4) adj_stage_kernel(Args<float> a, AdjFields<float> f) {
  after_previous();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  AdjTileSmem& S = *reinterpret_cast<AdjTileSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nx = a.nx, ny = a.ny;
  const int x0 = blockIdx.x * kAx, y0 = blockIdx.y * kAy;
  const unsigned n = (unsigned)a.n;
  const float* cs = STAGE == 3 ? a.c2 : (STAGE == 2 ? a.c1 : a.c);
  const float* lsrc = STAGE == 3 ? f.mu : (STAGE == 2 ? f.lc2 : f.lc1);
  const float* ux = a.u;
  const float* uy = a.u + n;
  // lambda of the stage output, scaled: 2/3 mu, 1/4 lc2, lc1.  The first is mu - mu/3, the transpose of
  // the forward's s + (c - s)/3: with 1/3 and 2/3 each rounded to FP32 lambda grew by 3e-8 a step
  // (gradient of 100 steps on 200 x 160: 1.3e-6 relative L2 off, 2.0e-7 to 2.8e-7 so).
  auto scaled = [](float l) { return STAGE == 3 ? fmaf(-1.f / 3.f, l, l) : (STAGE == 2 ? 0.25f * l : l); };
  const float alpha = a.alpha, ia = a.inv_alpha, kappa = a.kappa, vs = a.vs;

  // ---- stage the tile and its halo cross
  constexpr int kQ = kAx / 4 + 2, kPos = (kAy + 8) * kQ;
  constexpr int kRounds = (kPos + kAT - 1) / kAT;
  Quad<float> Lc[kRounds], Ll[kRounds], Lx[kRounds], Ly[kRounds];
#pragma unroll
  for (int k = 0; k < kRounds; ++k) {  // all loads in flight together
    const int p = tid + k * kAT, row = p / kQ, q = p % kQ;
    const bool in_row = row >= 4 && row < kAy + 4, in_col = q >= 1 && q <= kAx / 4;
    if (p >= kPos || (!in_row && !in_col)) continue;
    const int gr = y0 - 4 + row;
    int lr = gr < 0 ? -1 - gr : (gr >= ny ? 2 * ny - 1 - gr : gr);
    lr = max(0, min(ny - 1, lr));  // rows past the ghosts that a face reads: any value
    int gx = x0 - 4 + 4 * q;
    gx = gx < 0 ? gx + nx : gx;
    while (gx >= nx) gx -= nx;
    const unsigned node = (unsigned)lr * (unsigned)nx + (unsigned)gx;
    Lc[k] = load_quad(cs + node);
    Ll[k] = load_quad(lsrc + node);
    if (in_row) Lx[k] = load_quad(ux + node);
    if (in_col) Ly[k] = load_quad(uy + node);
  }
#pragma unroll
  for (int k = 0; k < kRounds; ++k) {
    const int p = tid + k * kAT, row = p / kQ, q = p % kQ;
    const bool in_row = row >= 4 && row < kAy + 4, in_col = q >= 1 && q <= kAx / 4;
    if (p >= kPos || (!in_row && !in_col)) continue;
    const int gr = y0 - 4 + row;
    const bool ghost = gr < 0 || gr >= ny;
    const Quad<float> c = Lc[k];
    Quad<float> P, M;
#pragma unroll
    for (int j = 0; j < 4; ++j) P.v[j] = scaled(Ll[k].v[j]);
    *reinterpret_cast<Quad<float>*>(&S.lam[row][4 * q]) = P;
    if (in_row) {
      const Quad<float> u = Lx[k];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float h = 0.5f * c.v[j], w = u.v[j] * ia;
        P.v[j] = fmaf(w, h, h);
        M.v[j] = fmaf(w, h, -h);
      }
      *reinterpret_cast<Quad<float>*>(&S.px[row - 4][4 * q]) = P;
      *reinterpret_cast<Quad<float>*>(&S.mx[row - 4][4 * q]) = M;
    }
    if (in_col) {
      const Quad<float> u = Ly[k];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float h = 0.5f * c.v[j], w = ((ghost ? -u.v[j] : u.v[j]) - vs) * ia;
        P.v[j] = fmaf(w, h, h);
        M.v[j] = fmaf(w, h, -h);
      }
      *reinterpret_cast<Quad<float>*>(&S.py[row][4 * (q - 1)]) = P;
      *reinterpret_cast<Quad<float>*>(&S.my[row][4 * (q - 1)]) = M;
    }
  }
  __syncthreads();

  // ---- y faces: a block of four lower faces (rows 4 g .. 4 g + 3) of one column; face r lies
  // between rows r - 1 and r and exists for 1 <= y0 + r <= ny - 1
  auto lam_y = [&](int r, int col) {
    const int fr = y0 + r;
    return fr >= 1 && fr <= ny - 1 ? S.lam[r + 4][col + 4] - S.lam[r + 3][col + 4] : 0.f;
  };
  auto y_block = [&](auto f0, auto f1, int g, int col) {
    constexpr int F0 = decltype(f0)::value, F1 = decltype(f1)::value;
    float P[8], M[8], lamF[4], accP[7], accM[7];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      // rows past the staged halo (of faces that are not computed): any staged row
      P[j] = S.py[min(max(4 * g + 1 + j, 0), kAy + 7)][col];
      M[j] = S.my[min(max(4 * g + 2 + j, 0), kAy + 7)][col];
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) lamF[m] = m >= F0 && m < F1 ? lam_y(4 * g + m, col) : 0.f;
    block_faces<F0, F1>(P, M, lamF, accP, accM);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      S.ed.y[0][g + 1][j][col] = accP[3 + j];
      S.ed.y[1][g + 1][j][col] = accM[3 + j];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      S.ed.y[0][g + 1][5 + j][col] = accP[j];
      S.ed.y[1][g + 1][5 + j][col] = accM[j];
    }
  };
  using I0 = std::integral_constant<int, 0>;
  using I2 = std::integral_constant<int, 2>;
  using I3 = std::integral_constant<int, 3>;
  using I4 = std::integral_constant<int, 4>;
  y_block(I0(), I4(), warp, lane);
  if (warp == 0) y_block(I2(), I4(), -1, lane);
  if (warp == 1) y_block(I0(), I3(), kAy / 4, lane);
  // c and u_y of this thread's four rows, on their way during the barrier
  float yc[4], yu[4];
  const int ycol = x0 + lane < nx ? x0 + lane : (x0 + lane) % nx;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const unsigned node = (unsigned)min(y0 + 4 * warp + j, ny - 1) * (unsigned)nx + (unsigned)ycol;
    yc[j] = cs[node];
    yu[j] = uy[node];
  }
  __syncthreads();

  // ---- y part of the tile's nodes: four rows of one column
  {
    float vs_acc = 0.f;
    const int col = lane, r0 = 4 * warp;
    const bool own = x0 + col < nx;
    float lamF[5], edP[5], edM[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      lamF[j] = lam_y(r0 + j, col);
      edP[j] = column_ed(S, 0, r0 - 1 + j, col);
      edM[j] = column_ed(S, 1, r0 - 2 + j, col);  // M's differences are stored one lower
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + j, y = y0 + r;
      float gc = 0.f, gw = 0.f;
      if (y < ny) {
        const float c = yc[j], u = yu[j];
        const float GP = edP[j] - edP[j + 1] + lamF[j + 1], GM = edM[j] - edM[j + 1] + lamF[j];
        const float wa = (u - vs) * ia, hc = 0.5f * c;
        gc = fmaf(0.5f * alpha, fmaf(GP, wa + 1.f, GM * (wa - 1.f)), kappa * (lamF[j + 1] - lamF[j]));
        gw = hc * (GP + GM);
        float vw = gw;
        if (y <= 1 || y >= ny - 2) {  // the ghost rows that mirror this one (both walls if ny is small)
#pragma unroll
          for (int side = 0; side < 2; ++side) {
            if (side == 0 ? y > 1 : y < ny - 2) continue;
            const int i = (side == 0 ? -1 - y : 2 * ny - 1 - y) - y0;
            const float gp = column_ed(S, 0, i - 1, col) - column_ed(S, 0, i, col);
            const float gm = column_ed(S, 1, i - 2, col) - column_ed(S, 1, i - 1, col);
            const float wg = (-u - vs) * ia, g = hc * (gp + gm);
            gc = fmaf(0.5f * alpha, fmaf(gp, wg + 1.f, gm * (wg - 1.f)), gc);
            gw -= g;
            vw += g;
          }
        }
        if (own) vs_acc -= vw;
      }
      S.py[r][col] = gc;
      S.my[r][col] = gw;
    }
    S.vs_red[tid] = vs_acc;
    if (y0 == 0 && warp == 0)
      S.vs_floor[col] = own ? (double)yc[0] * ((STAGE == 3 ? 2.0 / 3.0 : 1.0 / 6.0) - (double)S.lam[4][col + 4]) : 0.0;
  }
  __syncthreads();

  // ---- x faces: a block of four left faces (columns 4 g .. 4 g + 3) of one row
  auto x_block = [&](auto f0, auto f1, int g, int row) {
    constexpr int F0 = decltype(f0)::value, F1 = decltype(f1)::value;
    float lamF[4], accP[7], accM[7];
    // quads past the staged halo (of faces that are not computed): any staged quad
    const int q0 = max(4 * g, 0), q2 = min(4 * g + 8, kAx + 4);
    auto quad = [&](const float (&r)[kAx + 8], int at) { return *reinterpret_cast<const float4*>(&r[at]); };
    const float4 p0 = quad(S.px[row], q0), p1 = quad(S.px[row], 4 * g + 4), p2 = quad(S.px[row], q2);
    const float4 m0 = quad(S.mx[row], q0), m1 = quad(S.mx[row], 4 * g + 4), m2 = quad(S.mx[row], q2);
    const float P[8] = {p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w, p2.x};
    const float M[8] = {m0.z, m0.w, m1.x, m1.y, m1.z, m1.w, m2.x, m2.y};
#pragma unroll
    for (int m = 0; m < 4; ++m)
      lamF[m] = m >= F0 && m < F1 ? S.lam[row + 4][4 * g + m + 4] - S.lam[row + 4][4 * g + m + 3] : 0.f;
    block_faces<F0, F1>(P, M, lamF, accP, accM);
    S.ed.x[0][0][row][g + 1] = make_float4(accP[3], accP[4], accP[5], accP[6]);
    S.ed.x[0][1][row][g + 1] = make_float4(0.f, accP[0], accP[1], accP[2]);
    S.ed.x[1][0][row][g + 1] = make_float4(accM[3], accM[4], accM[5], accM[6]);
    S.ed.x[1][1][row][g + 1] = make_float4(0.f, accM[0], accM[1], accM[2]);
  };
  const int q = tid & 7, row = tid >> 3;
  x_block(I0(), I4(), q, row);
  if (warp == 2) x_block(I2(), I4(), -1, lane);
  if (warp == 3) x_block(I0(), I3(), kAx / 4, lane);
  // the fields of this thread's four nodes, on their way during the barrier
  const int y = y0 + row, xl = x0 + 4 * q;
  const bool own = y < ny && xl < nx;
  const unsigned node = (unsigned)y * (unsigned)nx + (unsigned)xl;
  Quad<float> c{}, u{}, mu{}, l2{}, ox{}, oy{};
  if (own) {
    c = load_quad(cs + node);
    u = load_quad(ux + node);
    if (STAGE == 1) {
      mu = load_quad(f.mu + node);
      l2 = load_quad(f.lc2 + node);
    }
    if (STAGE < 3) {
      ox = load_quad(f.lam_u + node);
      oy = load_quad(f.lam_u + n + node);
    }
  }
  __syncthreads();

  // ---- the tile's nodes: four columns of one row
  {
    if (own) {
      auto sum4 = [](const float4& p, const float4& r) { return make_float4(p.x + r.x, p.y + r.y, p.z + r.z, p.w + r.w); };
      float edP[5], edM[5], lamF[5];
      {
        const float4 lo = sum4(S.ed.x[0][0][row][q], S.ed.x[0][1][row][q + 1]);
        const float4 hi = sum4(S.ed.x[0][0][row][q + 1], S.ed.x[0][1][row][q + 2]);
        edP[0] = lo.w;
        edP[1] = hi.x;
        edP[2] = hi.y;
        edP[3] = hi.z;
        edP[4] = hi.w;
      }
      {
        const float4 lo = sum4(S.ed.x[1][0][row][q], S.ed.x[1][1][row][q + 1]);
        const float4 hi = sum4(S.ed.x[1][0][row][q + 1], S.ed.x[1][1][row][q + 2]);
        edM[0] = lo.z;
        edM[1] = lo.w;
        edM[2] = hi.x;
        edM[3] = hi.y;
        edM[4] = hi.z;
      }
#pragma unroll
      for (int j = 0; j < 5; ++j) lamF[j] = S.lam[row + 4][4 * q + j + 4] - S.lam[row + 4][4 * q + j + 3];
      Quad<float> v, gx, gy;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float GP = edP[j] - edP[j + 1] + lamF[j + 1], GM = edM[j] - edM[j + 1] + lamF[j];
        const float wa = u.v[j] * ia, lam = S.lam[row + 4][4 * q + j + 4];
        const float gc = fmaf(0.5f * alpha, fmaf(GP, wa + 1.f, GM * (wa - 1.f)), kappa * (lamF[j + 1] - lamF[j]));
        v.v[j] = lam + (gc + S.py[row][4 * q + j]);
        if (y == 0) v.v[j] += (STAGE == 3 ? 2.f / 3.f : 1.f / 6.f) * vs - vs * lam;  // deposit weight, floor face
        gx.v[j] = (0.5f * c.v[j]) * (GP + GM);
        gy.v[j] = S.my[row][4 * q + j];
      }
      if (STAGE == 1) {
#pragma unroll
        for (int j = 0; j < 4; ++j) v.v[j] += fmaf(1.f / 3.f, mu.v[j], 0.75f * l2.v[j]);
      }
      if (STAGE < 3) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          gx.v[j] += ox.v[j];
          gy.v[j] += oy.v[j];
        }
      }
      *reinterpret_cast<Quad<float>*>((STAGE == 3 ? f.lc2 : (STAGE == 2 ? f.lc1 : f.lc)) + node) = v;
      *reinterpret_cast<Quad<float>*>(f.lam_u + node) = gx;
      *reinterpret_cast<Quad<float>*>(f.lam_u + n + node) = gy;
    }
  }

  // ---- this CTA's Vs terms (written before the last two barriers), by one warp.  Gradient of 100
  // steps on 512 x 1024 through autograd: 9.53 ms with a warp's sums in plain FP32, 9.61 so, 10.03
  // with all of them in FP64
  if (warp == 0) {
    float hi = S.vs_red[lane], lo = 0.f;
#pragma unroll
    for (int w = 1; w < kAT / 32; ++w) add_pair(hi, lo, S.vs_red[w * 32 + lane], 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      add_pair(hi, lo, __shfl_down_sync(0xffffffffu, hi, o), __shfl_down_sync(0xffffffffu, lo, o));
    double floor_sum = 0.0;
    if (y0 == 0) {
      floor_sum = S.vs_floor[lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) floor_sum += __shfl_down_sync(0xffffffffu, floor_sum, o);
    }
    if (lane == 0)  // own slot, fixed order over steps
      f.vs_part[blockIdx.y * gridDim.x + blockIdx.x] += ((double)hi + (double)lo) + floor_sum;
  }
}

inline cudaError_t adj_stage_prepare() {
  const int bytes = (int)sizeof(AdjTileSmem);
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(adj_stage_kernel<1>, at, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(adj_stage_kernel<2>, at, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(adj_stage_kernel<3>, at, bytes);
  return e;
}

template <int STAGE>
inline void launch_adj_stage(const Args<float>& a, const AdjFields<float>& f, cudaStream_t s) {
  const dim3 grid((a.nx + kAx - 1) / kAx, (a.ny + kAy - 1) / kAy);
  launch_dependent(adj_stage_kernel<STAGE>, grid, kAT, sizeof(AdjTileSmem), s, a, f);
}

}  // namespace lw
