// 2D heat with the plan left to the library: overlapped tiles.
//
// A block takes a window of WX x WY points (WX = 64 columns, WY = 8 L rows),
// advances it kk <= G steps and writes the points at least G from the window's
// edge, which no wrong value has reached; the state goes from one array to the
// other and back.  A step has one level here where the swept rule has three
// (bridges, growing and shrinking squares), all lanes work in every level, and
// the shape is fixed at compile time: a thread owns L consecutive points of one
// column, keeps them in registers, reads its west and east neighbours (and
// one point above and below its run) from shared memory and stores its points
// for its neighbours: 3 shared-memory accesses a point instead of 6 and no index
// arithmetic.  The price is the ghost points, (WX WY) / ((WX - 2G)(WY - 2G))
// updates a point.  Ghosts beyond a mirror wall hold their mirror point's value and
// stay its image, because the update is symmetric in x and in y, bit for bit.
//
// Bound: FP32, shared-memory instructions (3 a point at one a cycle and SM); FP64,
// integer issue.  Measured against the swept passes with no plan set: 1024^2
// FP32, 500 steps, 3.50 -> 0.75 ms; 768 x 512 FP64 insulated, 300 steps, 2.52 ->
// 1.44 ms; with all five operations on the FP64 pipe 2.07 ms.  Periodic FP64, 300 steps, noisy field / hot spot on
// zeros / a field of subnormals (FP64 alone): 768 x 512 1.47 / 1.69 / 2.2 ms (swept passes 2.12), 1024^2 3.41 / 3.75 /
// 5.0 (4.32).
#pragma once
#include "kernels2d.cuh"

namespace swept2d {

struct Tile2d {
  int L = 0, G = 0;  // rows per thread (0: not used), ghost width = steps per launch
};

constexpr int kTileWX = 64, kTileBands = 8;

// the point of [0, n) that position x of the unbounded line stands for
__device__ __forceinline__ int64_t tile2d_point(int64_t x, int64_t n, int bc) {
  if (x >= 0 && x < n) return x;
  if (bc == 0) return swept::wrap_n(x, n);
  const int64_t r = swept::wrap_n(x, 2 * n);
  return r < n ? r : 2 * n - 1 - r;
}

// one column run: v[i] <- its update, from the rows' west and east values (stride
// kTileWX) and the run's neighbours above and below
template <typename T, int L>
__device__ __forceinline__ void tile2d_run_fp(const T* w, const T* e, T up, T down, T (&v)[L], const Heat2dK<T>& k) {
  T below = up;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    const T sx = add_rn(w[i * kTileWX], e[i * kTileWX]);
    const T sy = add_rn(below, i == L - 1 ? down : v[i + 1 < L ? i + 1 : i]);
    below = v[i];
    v[i] = fma_rn(k.fo, add_rn(sx, sy), mul_rn(k.c1, v[i]));
  }
}
// In FP64 the three sums run on the integer pipes (fixadd.cuh), two of a point's
// five operations on the FP64 pipe; a warp with a run outside their range (magnitudes more than 2^24
// apart, a subnormal, -0, ...) takes the FP64 instructions, which cost it the same for one lane as for all.
// The range is looked at before any sum, so such a warp pays for one form only, and the multiply-adds of a
// point start while the sums of the next are formed; zeros, which a field may be full of, are looked at again and
// stay with the integers.  What is left are sums that cancel to 2^-26 of their operands: those lanes do
// their run again from the values in shared memory (`own`), behind a branch the compiler cannot turn into
// predicated instructions: those would hold the pipe as long as ones that run.
template <typename T, int L>
__device__ __forceinline__ void tile2d_run(const T* own, const T* w, const T* e, T up, T down, T (&v)[L],
                                           const Heat2dK<T>& k) {
  if constexpr (sizeof(T) == 8) {
    int E;
    bool in = swept::fix::cross_scale<L, kTileWX>(w, e, up, down, v, E);
    if (!__all_sync(0xffffffffu, in)) in = swept::fix::cross_scale_zeros<L, kTileWX>(w, e, up, down, v, E);
    if (__all_sync(0xffffffffu, in)) {
      T s[L];
      bool ok = true;
      swept::fix::cross_at<L, kTileWX>(w, e, up, down, v, s, E, ok);
#pragma unroll
      for (int i = 0; i < L; ++i) v[i] = fma_rn(k.fo, s[i], mul_rn(k.c1, v[i]));
      int redo = ok ? 0 : 1;
      asm volatile("" : "+r"(redo));
      for (; redo > 0; --redo) {
        asm volatile("" ::: "memory");
#pragma unroll
        for (int i = 0; i < L; ++i) v[i] = own[i * kTileWX];
        tile2d_run_fp<T, L>(w, e, up, down, v, k);
      }
      return;
    }
  }
  tile2d_run_fp<T, L>(w, e, up, down, v, k);
}

template <typename T, int L>
__global__ void __launch_bounds__(kTileWX* kTileBands) k_tile2d(int64_t nx, int64_t ny, int bc, Heat2dK<T> k,
                                                                const T* __restrict__ in, T* __restrict__ out, int G,
                                                                int kk) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int WY = kTileBands * L, ST = kTileWX, SIZE = ST * WY;
  T* sm = reinterpret_cast<T*>(smraw);
  const int col = (int)threadIdx.x % kTileWX, r0 = (int)threadIdx.x / kTileWX * L;
  const int64_t gx = (int64_t)blockIdx.x * (kTileWX - 2 * G) - G + col;
  const int64_t gy = (int64_t)blockIdx.y * (WY - 2 * G) - G + r0;
  const int64_t px = tile2d_point(gx, nx, bc);
  T v[L];
  const int at = r0 * ST + col;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    const int64_t p = tile2d_point(gy + i, ny, bc) * nx + px;
    v[i] = dbg::in_range(p, nx * ny, dbg::STATE) ? in[p] : T(0);
    sm[at + i * ST] = v[i];
  }
  // a point at the window's edge takes itself for the neighbour outside: wrong, as it
  // would be with any value, but of its own size, which keeps the integer sums in range
  const int west = col == 0 ? 0 : -1, east = col == kTileWX - 1 ? 0 : 1;
  __syncthreads();
  for (int t = 0; t < kk; ++t) {
    const T* a = sm + (t & 1) * SIZE;
    T* b = sm + ((t & 1) ^ 1) * SIZE;
    const T up = r0 == 0 ? v[0] : a[at - ST], down = r0 + L == WY ? v[L - 1] : a[at + L * ST];
    tile2d_run<T, L>(a + at, a + at + west, a + at + east, up, down, v, k);
    if (t + 1 < kk) {
#pragma unroll
      for (int i = 0; i < L; ++i) b[at + i * ST] = v[i];
      __syncthreads();
    }
  }
  if (col >= G && col < kTileWX - G && gx < nx) {
#pragma unroll
    for (int i = 0; i < L; ++i)
      if (r0 + i >= G && r0 + i < WY - G && gy + i < ny) out[(gy + i) * nx + gx] = v[i];
  }
}

template <typename T>
constexpr size_t tile2d_smem(int L) {
  return (size_t)2 * kTileWX * kTileBands * L * sizeof(T);
}

}  // namespace swept2d
