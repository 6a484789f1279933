// Shared device-side argument block and small helpers of the lbm_wenoc kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lw {

// Status bits ORed by kernels into the device status word.
constexpr unsigned kStatusUnstable = 1u;  // non-finite value or |u_d| > u_cap
constexpr unsigned kStatusTimeout = 2u;   // a bounded wait gave up

template <typename T>
struct Args {
  T* g;    // populations stored as g_i = f_i - w_i, SoA: g[i*n + node]
  T* c;    // concentration c^n (updated in place by the last RK stage)
  T* c1;   // RK stage 1 field
  T* c2;   // RK stage 2 field
  T* u;    // transport velocity of the current step, u[d*n + node]
  double* partials;  // per-block FP64 partial sums (fixed-order reductions)
  double* scalars;   // [0] deposit, [1] reduction result
  unsigned* status;  // status word
  unsigned* ticket;  // last-block ticket of the reductions
  int nx, ny, nz;    // extents (nz = 1 in 2D)
  long long n;       // nodes
  int walls;         // 1 = no-slip floor and lid, 0 = periodic vertical
  T omega;           // 1/tau
  T guo;             // 1 - 1/(2 tau)
  T A;               // gravity * density_contrast
  T bf[3];           // body force
  T vs;              // settling velocity
  T kappa;           // diffusivity
  T alpha;           // Lax-Friedrichs split speed
  T inv_alpha;
  T u_cap;
  // sugar (the paper's density-altering scalar), null S when off
  const T* S;  // S of step n
  T* S2;       // S of step n + 1
  T gS;        // gravity * sugar_contrast (S*): force -gS S (1 - phi0 c) along the vertical
  T phi0;      // particle volume fraction at c = 1
  T ks;        // settling velocity Vs (1 - ks S)
  T Ds;        // sugar diffusivity
  int scheme;  // flux variant bits (kSchemeWeno3, kSchemeSignSplit); 0 = WENO5, Lax-Friedrichs
  int late_count;  // deposit folded late (fold_late_deposit): partials a step's last stage leaves; 0 = it folds them
};

// Global-load policies.  LoadPlain is an ordinary load, for a kernel that may have been started
// before the one ahead of it ended (launch_dependent): it reads what that one wrote, so the
// read-only path is closed to it, and so is __restrict__ on its pointers, by which the compiler
// may choose that path for an ordinary load.  LoadNC reads through the non-coherent (read-only)
// path, for data no thread writes while the kernel runs.  LoadL2 reads at L2 (ld.global.cg: no L1
// line is kept), for a kernel that reads what other CTAs wrote earlier in the same launch, after a
// grid barrier.
struct LoadNC {
  static __device__ __forceinline__ float s(const float* p) { return __ldg(p); }
  static __device__ __forceinline__ double s(const double* p) { return __ldg(p); }
  static __device__ __forceinline__ float4 v4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
};
struct LoadL2 {
  static __device__ __forceinline__ float s(const float* p) { return __ldcg(p); }
  static __device__ __forceinline__ double s(const double* p) { return __ldcg(p); }
  static __device__ __forceinline__ float4 v4(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
};
struct LoadPlain {
  static __device__ __forceinline__ float s(const float* p) { return *p; }
  static __device__ __forceinline__ double s(const double* p) { return *p; }
  static __device__ __forceinline__ float4 v4(const float* p) { return *reinterpret_cast<const float4*>(p); }
};

// Four adjacent values (nx is a multiple of four and every field starts on a 256-byte line),
// moved as one or two 16-byte accesses.
template <typename T>
struct alignas(4 * sizeof(T)) Quad {
  T v[4];
};
template <typename T>
__device__ __forceinline__ Quad<T> load_quad(const T* p) { return *reinterpret_cast<const Quad<T>*>(p); }

constexpr int kSchemeWeno3 = 1;
constexpr int kSchemeSignSplit = 2;

// Settling velocity at node m: Vs, or Vs (1 - ks S_m) with sugar.
template <typename T>
__device__ __forceinline__ T settling_at(const Args<T>& a, long long m) {
  return a.S ? a.vs * (T(1) - a.ks * a.S[m]) : a.vs;
}

// Asynchronous 16-byte global -> shared copy at L2 (cp.async.cg: no L1 line, so it also
// sees what other SMs wrote earlier in the same launch); groups of copies are committed
// and waited for per thread.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Programmatic dependent launch: a kernel launched by launch_dependent() has its launch and
// its CTAs' start processed while the one before it on the stream drains; after_previous(),
// its first statement, waits until that one has ended and its writes are visible, so no
// global memory is touched early.  Nothing triggers the next launch before a CTA's end: with
// the trigger at a kernel's start the next grids' waiting CTAs took the slots unevenly (the
// 128 x 256 FP64 step went from 97 to 259 us); without it a launch costs about 0.25 us less.
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                    const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// fused multiply-add of the kernel's precision (fmaf for FP32, fma for FP64)
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ int wrap_dec(int a, int n) { return a < 0 ? a + n : a; }
__device__ __forceinline__ int wrap_inc(int a, int n) { return a >= n ? a - n : a; }
__device__ __forceinline__ int wrap_any(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

template <typename T>
__device__ __forceinline__ bool finite_val(T v) { return isfinite(v); }

// Sum of n FP64 partials written by other CTAs, by one whole warp in a fixed order (valid in
// lane 0).  One thread that adds them in turn waits for a trip to L2 for each (sixteen took
// 12 us), so up to eight are loaded together, and more are dealt to the lanes (l, l + 32, ...)
// and folded by a shuffle tree, whose five FP64 steps cost about 1 us.
__device__ __forceinline__ double fold_partials(const double* partials, int n) {
  const volatile double* vp = partials;
  double s = 0.0;
  if (n <= 8) {
    double v[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) v[b] = b < n ? vp[b] : 0.0;
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if (b < n) s += v[b];
    return s;
  }
  for (int b = (int)(threadIdx.x & 31); b < n; b += 32) s += vp[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  return s;
}

// The deposit's sums.  The four-column kernel adds the terms of 32 columns (eight threads), then
// pairs of those groups twice (a warp), then its two warps, times Vs: a strip of 256 columns;
// then the strips (fold_partials).  A tile holds one group; this fold, by a whole warp, rebuilds
// the strips (valid in lane 0).
__device__ __forceinline__ double fold_tile_partials(const double* partials, int tiles, double scale) {
  const volatile double* vp = partials;
  const int lane = threadIdx.x & 31, strips = (tiles + 7) / 8;
  auto strip = [&](int b) {
    double g[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) g[j] = 8 * b + j < tiles ? vp[8 * b + j] : 0.0;
    return (((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]))) * scale;
  };
  double s = 0.0;
  if (strips <= 8) {
    const double p = lane < strips ? strip(lane) : 0.0;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const double v = __shfl_sync(0xffffffffu, p, b);
      if (b < strips) s += v;
    }
    return s;
  }
  for (int b = lane; b < strips; b += 32) s += strip(b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  return s;
}

// Tile handles leave the fold of a step's deposit to the next kernel that can take it: the next
// step's first stage (a block of its own, started first), or late_deposit_kernel before the
// deposit is read.  The last stage then ends with one store a tile instead of a fence, a ticket
// and a fold on its critical path (a step on 128 x 256 13.4 -> 11.3 us).  In the fluid kernel
// the extra row of blocks cost more than that on lattices beyond L2 (108 -> 114 us on 2048 x 4096
// in front of the lattice, 110 behind it).  The partials have a place of their own behind the
// ones of the reductions that fold at once, and are zero before the first step and after
// late_deposit_kernel, so adding them is always right.
constexpr int kLateOffset = 512, kLateMax = 512;
template <typename T>
__device__ __forceinline__ void fold_late_deposit(const Args<T>& a) {
  const double* p = a.partials + kLateOffset;
  const double prev = *reinterpret_cast<const volatile double*>(a.scalars);
  const double tot = fold_tile_partials(p, a.late_count, a.S ? 1.0 : (double)a.vs);
  if ((threadIdx.x & 31) == 0) a.scalars[0] = prev + tot;
}

// Flag a bad value once per warp (no trap, no assert: the host reads the word).
__device__ __forceinline__ unsigned lane_id() {
  unsigned l;
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(l));
  return l;
}

__device__ __forceinline__ void report_status(unsigned* status, bool bad) {
  unsigned m = __ballot_sync(__activemask(), bad);
  if (m != 0u && lane_id() == (unsigned)(__ffs(m) - 1)) atomicOr(status, kStatusUnstable);
}

}  // namespace lw
