// 2D FP32 transport on tiles: one SSP-RK3 stage of the WENO5 + diffusion + settling update of
// c (steps a4..a8; the stage-3 kernel also folds the floor deposit, a9), with the scheme
// variants and the sugar scalar as compile-time forms.
//
// A CTA owns kTX x kTY nodes.  It stages the split fluxes along x (tile rows, a four-column halo
// on each side), along y (tile columns, a three-row halo below and above) and c on the cross,
// all loads in flight at once; a thread then computes the lower y faces of four consecutive
// rows of one column and the left x faces of four consecutive columns of one row, sharing the
// first and second differences of the split fluxes between the four faces in both directions.
// A block's fifth face is its neighbour's first (shared memory in y, a shuffle in x); the faces
// on the tile's right and top edges are computed once more by the next tile.
// Ghost rows behind the walls reflect c (even) and u_y (odd); the lid and floor faces carry
// nothing here and the floor row's settling outflow is taken off in the combination.
// The arithmetic and its order are those of the row-sweep kernels, the fold of the deposit
// included, so c and the deposit are bitwise those of the four-column one.
//
// Against that kernel a tile has no serial chain of rows: 32 warps an SM at 54-61 registers
// instead of 12 at 133, and no priming row or half-filled wave on a small lattice; it pays with
// halos split twice (213-220 instructions a node and stage instead of 191-207).  Bound by
// instruction issue where the fields sit in L2 (68-69 % of the slots on 1024 x 2048; on 512 x 1024,
// less than a wave, 52 %; the rest waits for a tile's first loads and at its barriers).
// Whole steps, four-column kernel -> tiles, the deposit folded in the same step by both:
// 128 x 256 15.0 -> 13.4 us, 512 x 1024 32.3 -> 24.2, 1260 x 701 41.3 -> 35.8, 1024 x 2048
// 80.7 -> 76.3 (with the fold left to the next step and dependent launches 10.5, 21.5, 34.3 and
// 74.8; larger ones at kTileMaxNodes).  Tiles of
// 64 x 16, 32 x 32 and 64 x 32 nodes were 1-5 % slower on most sizes.
#pragma once
#include "common.cuh"
#include "weno.cuh"
#include "transport_stage2d.cuh"       // Stage2dParams
#include "transport_stage2d_wide.cuh"  // scheme_split, x_faces

namespace lw {

constexpr int kTX = 32, kTY = 16;      // tile (nodes)
constexpr int kTT = kTX * kTY / 4;     // threads
// Largest lattice that runs on tiles: its populations (36 bytes a node) and fields stay in L2
// (129 MB) up to about here; beyond, a tile's start waits for HBM and the row sweep, which loads a
// row ahead, is the faster one.  Steps with both kernels as they are (late fold on tiles, dependent
// launches on both), us, tiles against the row sweep:
//            1536 x 2048     1792 x 2048     2048 x 2048     2048 x 3072     2048 x 4096
//            (3.1 M nodes)   (3.7 M)         (4.2 M)         (6.3 M)         (8.4 M)
//   plain    110.4  115.0    128.1  130.1    145.8  145.3    220.4  212.4    287.9  278.3
//   sugar    121.7  124.2    142.1  140.7    163.0  157.3    245.6  231.2    320.6  303.2
//   WENO3     89.1   91.2    103.5  103.3    118.3  116.2    184.0  173.3    241.2  227.0
//   sign      98.9  101.0    114.7  113.9    131.2  127.8    200.5  186.5    261.7  243.7
constexpr long long kTileMaxNodes = 3500000;

struct Tile2dSmem {
  float px[kTY][kTX + 8];      // the scheme's pair along x, columns -4 .. kTX + 3
  float mx[kTY][kTX + 8];
  float py[kTY + 6][kTX];      // along y, rows -3 .. kTY + 2; later the y divergence of row r in py[r]
  float my[kTY + 6][kTX];
  float c[kTY + 6][kTX + 8];   // stage input c on the cross
  float fy[kTY / 4 + 1][kTX];  // first lower y face of each block of four rows (+ the tile's top edge)
  float fx[kTY];             // right edge x face of each row
};

template <int STAGE, bool SUGAR = false, int SCHEME = 0>
__global__ void __launch_bounds__(kTT, 1024 / kTT) rk_tile2d_kernel(Args<float> a, Stage2dParams sp) {
  after_previous();
  constexpr int TX = kTX, TY = kTY, T = kTT;
  __shared__ __align__(16) Tile2dSmem S;
  const int tid = threadIdx.x;
  const int nx = a.nx, ny = a.ny;
  // the first stage's first row of blocks folds the deposit of the step before
  const int by = (int)blockIdx.y - (STAGE == 1 && a.late_count > 0 ? 1 : 0);
  if (STAGE == 1 && by < 0) {
    if (blockIdx.x == 0 && tid < 32) fold_late_deposit(a);
    return;
  }
  const int x0 = blockIdx.x * TX, y0 = by * TY;
  const float ia = a.inv_alpha, vs_a = a.vs * a.inv_alpha, alpha = a.alpha, kd = a.kappa * a.inv_alpha;
  const float* cin = sp.cin;
  const float* ux = a.u;
  const float* uy = a.u + a.n;

  // ---- stage the tile and its halo cross
  constexpr int kQ = TX / 4 + 2, kPos = (TY + 6) * kQ;
#pragma unroll
  for (int p0 = 0; p0 < kPos; p0 += T) {
    const int p = p0 + tid;
    const int r = p / kQ, q = p - r * kQ;
    const bool in_row = r >= 3 && r < TY + 3, in_col = q >= 1 && q <= TX / 4;
    if (p < kPos && (in_row || in_col)) {
      const int gr = y0 - 3 + r;
      const bool ghost = gr < 0 || gr >= ny;
      int lr = gr < 0 ? -1 - gr : (gr >= ny ? 2 * ny - 1 - gr : gr);
      lr = max(0, min(ny - 1, lr));  // rows past the ghosts that a face reads: any value
      int gx = x0 - 4 + 4 * q;
      gx = gx < 0 ? gx + nx : gx;
      while (gx >= nx) gx -= nx;
      const unsigned node = (unsigned)lr * (unsigned)nx + (unsigned)gx;
      const float4 c = LoadPlain::v4(cin + node);
      float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u, s = u;
      if (in_row) u = LoadPlain::v4(ux + node);
      if (in_col) v = LoadPlain::v4(uy + node);
      if (SUGAR && in_col) s = LoadPlain::v4(a.S + node);
      *reinterpret_cast<float4*>(&S.c[r][4 * q]) = c;
      float4 P, M;
      if (in_row) {
        scheme_split<SCHEME>(c.x, u.x * ia, P.x, M.x);
        scheme_split<SCHEME>(c.y, u.y * ia, P.y, M.y);
        scheme_split<SCHEME>(c.z, u.z * ia, P.z, M.z);
        scheme_split<SCHEME>(c.w, u.w * ia, P.w, M.w);
        *reinterpret_cast<float4*>(&S.px[r - 3][4 * q]) = P;
        *reinterpret_cast<float4*>(&S.mx[r - 3][4 * q]) = M;
      }
      if (in_col) {
        const float sg = ghost ? -ia : ia;
        auto vsa = [&](float S_) { return SUGAR ? vs_a * fmaf(-a.ks, S_, 1.f) : vs_a; };
        scheme_split<SCHEME>(c.x, fmaf(v.x, sg, -vsa(s.x)), P.x, M.x);
        scheme_split<SCHEME>(c.y, fmaf(v.y, sg, -vsa(s.y)), P.y, M.y);
        scheme_split<SCHEME>(c.z, fmaf(v.z, sg, -vsa(s.z)), P.z, M.z);
        scheme_split<SCHEME>(c.w, fmaf(v.w, sg, -vsa(s.w)), P.w, M.w);
        *reinterpret_cast<float4*>(&S.py[r][4 * (q - 1)]) = P;
        *reinterpret_cast<float4*>(&S.my[r][4 * (q - 1)]) = M;
      }
    }
  }
  __syncthreads();

  // ---- lower y faces of rows 4 g .. 4 g + 3 of a column (none at the floor and the lid)
  const int col = tid % TX, g = tid / TX;
  float fyq[4];
  {
    const float* P = &S.py[4 * g][col];
    const float* M = &S.my[4 * g][col];
    const float* C = &S.c[4 * g + 2][col + 4];
    const float4 p0 = make_float4(0.f, P[0], P[TX], P[2 * TX]), p1 = make_float4(P[3 * TX], P[4 * TX], P[5 * TX], P[6 * TX]);
    const float4 p2 = make_float4(P[7 * TX], P[8 * TX], 0.f, 0.f);
    const float4 m0 = make_float4(0.f, 0.f, M[TX], M[2 * TX]), m1 = make_float4(M[3 * TX], M[4 * TX], M[5 * TX], M[6 * TX]);
    const float4 m2 = make_float4(M[7 * TX], M[8 * TX], 0.f, 0.f);
    constexpr int W = TX + 8;
    x_faces<SCHEME>(p0, p1, p2, m0, m1, m2, C[0], make_float4(C[W], C[2 * W], C[3 * W], C[4 * W]), kd, fyq);
    if (y0 == 0 && g == 0) fyq[0] = 0.f;
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (y0 + 4 * g + m == ny) fyq[m] = 0.f;
    S.fy[g][col] = fyq[0];
  }
  // the tile's top y faces and right x faces
  if (tid < TX) {
    float p[6], m[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      p[q] = S.py[TY + q][tid];
      m[q] = S.my[TY + q][tid];
    }
    const float f = face_flux_scheme<SCHEME>(p, m, kd, S.c[TY + 2][tid + 4], S.c[TY + 3][tid + 4]);
    S.fy[TY / 4][tid] = y0 + TY == ny ? 0.f : f;
  } else if (tid < TX + TY) {
    const int r = tid - TX;
    float p[6], m[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      p[q] = S.px[r][TX + 1 + q];
      m[q] = S.mx[r][TX + 1 + q];
    }
    S.fx[r] = face_flux_scheme<SCHEME>(p, m, kd, S.c[r + 3][TX + 3], S.c[r + 3][TX + 4]);
  }
  __syncthreads();

  // ---- y divergence of the block's rows (into the py rows, no longer read)
  {
    const float fup[4] = {fyq[1], fyq[2], fyq[3], S.fy[g + 1][col]};
#pragma unroll
    for (int m = 0; m < 4; ++m) S.py[4 * g + m][col] = fyq[m] - fup[m];
  }

  // ---- left x faces of four columns of a row
  constexpr int kRow = TX / 4;  // threads per row
  const int row = tid / kRow, q = tid % kRow;
  const int y = y0 + row, xl = x0 + 4 * q;
  const bool out = y < ny && xl < nx;
  const unsigned node = (unsigned)y * (unsigned)nx + (unsigned)xl;
  float4 cn = make_float4(0.f, 0.f, 0.f, 0.f);
  if (STAGE > 1 && out) cn = LoadPlain::v4(a.c + node);
  float fxq[4], fr;
  float4 cq;
  {
    auto quad = [&](const float* r, int at) { return *reinterpret_cast<const float4*>(r + at); };
    const float* P = &S.px[row][4 * q];
    const float* M = &S.mx[row][4 * q];
    cq = quad(&S.c[row + 3][4 * q], 4);
    x_faces<SCHEME>(quad(P, 0), quad(P, 4), quad(P, 8), quad(M, 0), quad(M, 4), quad(M, 8), S.c[row + 3][4 * q + 3], cq,
                    kd, fxq);
    fr = __shfl_down_sync(0xffffffffu, fxq[0], 1);
    if (q == kRow - 1) fr = S.fx[row];
  }
  __syncthreads();

  // ---- divergence and the Shu-Osher combination of this stage
  double dep = 0.0;  // stage 3, floor row: this thread's deposit term
  if (out) {
    const float4 dy = *reinterpret_cast<const float4*>(&S.py[row][4 * q]);
    const float frq[4] = {fxq[1], fxq[2], fxq[3], fr};
    const float ch[4] = {cq.x, cq.y, cq.z, cq.w}, cnv[4] = {cn.x, cn.y, cn.z, cn.w}, dyv[4] = {dy.x, dy.y, dy.z, dy.w};
    float v[4], Lk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) Lk[j] = fxq[j] - frq[j] + dyv[j];
    float vsf[4] = {a.vs, a.vs, a.vs, a.vs};
    if (y == 0) {  // the floor row's settling outflow
      if (SUGAR) {
        const float4 s0 = LoadPlain::v4(a.S + xl);
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
    *reinterpret_cast<float4*>(sp.cout + node) = make_float4(v[0], v[1], v[2], v[3]);
    if (STAGE == 3) {
      report_status(a.status, !(isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]) && isfinite(v[3])));
      if (y == 0) {  // RK3 b-weights of the floor flux: c^n/6 + c1/6 + 2 c2/3
        const float4 c1 = LoadPlain::v4(a.c1 + xl);
        const float c1v[4] = {c1.x, c1.y, c1.z, c1.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const double b = fma((double)cnv[j] + (double)c1v[j], 1.0 / 6.0, (double)ch[j] * (2.0 / 3.0));
          dep += SUGAR ? b * (double)vsf[j] : b;  // with sugar Vs(S) per node, else Vs once at the fold
        }
      }
    }
  }

  // stage 3: the floor tiles (their floor row is in the first eight threads) leave the deposit of
  // this step for the next kernel, or fold it: FP64, in the order of the four-column kernel
  if (STAGE == 3 && y0 == 0 && tid < 32) {
    const double v = tile_group_sum(dep);
    if (a.late_count > 0) {
      if (tid == 0) a.partials[kLateOffset + blockIdx.x] = v;
      return;
    }
    const int tiles = gridDim.x;
    int last = 0;
    if (tid == 0) {
      a.partials[blockIdx.x] = v;
      __threadfence();
      last = atomicAdd(a.ticket, 1u) == (unsigned)tiles - 1;
    }
    if (__shfl_sync(0xffffffffu, last, 0)) {
      __threadfence();
      const double prev = *reinterpret_cast<volatile double*>(a.scalars);  // written by earlier steps
      const double tot = fold_tile_partials(a.partials, tiles, SUGAR ? 1.0 : (double)a.vs);
      if (tid == 0) {
        a.scalars[0] = prev + tot;
        *a.ticket = 0u;
      }
    }
  }
}

// The stage kernel of the handle's sugar and transport scheme (runtime fields).
template <int STAGE>
inline StageWideKernel tile2d_entry(bool sugar, int scheme) {
  switch (scheme) {
    case kSchemeWeno3:
      return sugar ? rk_tile2d_kernel<STAGE, true, kSchemeWeno3> : rk_tile2d_kernel<STAGE, false, kSchemeWeno3>;
    case kSchemeSignSplit:
      return sugar ? rk_tile2d_kernel<STAGE, true, kSchemeSignSplit> : rk_tile2d_kernel<STAGE, false, kSchemeSignSplit>;
    case kSchemeWeno3 | kSchemeSignSplit:
      return sugar ? rk_tile2d_kernel<STAGE, true, kSchemeWeno3 | kSchemeSignSplit>
                   : rk_tile2d_kernel<STAGE, false, kSchemeWeno3 | kSchemeSignSplit>;
    default:
      return sugar ? rk_tile2d_kernel<STAGE, true> : rk_tile2d_kernel<STAGE>;
  }
}

inline bool tile2d_use(int nx, int ny) {
  return (long long)nx * ny <= kTileMaxNodes && (nx + kTX - 1) / kTX <= kMaxReduceBlocks;
}

template <int STAGE>
inline cudaError_t launch_tile2d(const Args<float>& a, const float* cin, float* cout, cudaStream_t s) {
  Stage2dParams sp;
  sp.cin = cin;
  sp.cout = cout;
  sp.H = kTY;
  const dim3 grid((a.nx + kTX - 1) / kTX, (a.ny + kTY - 1) / kTY + (STAGE == 1 && a.late_count > 0 ? 1 : 0));
  launch_dependent(tile2d_entry<STAGE>(a.S != nullptr, a.scheme), grid, kTT, 0, s, a, sp);
  return cudaGetLastError();
}

}  // namespace lw
