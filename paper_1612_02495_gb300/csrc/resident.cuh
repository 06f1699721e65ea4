// Small grids of the scalar schemes, with the plan left to the library: the
// whole grid stays in the registers of one thread-block cluster for the whole
// solve.
//
// On a grid of a few thousand points a pass of the swept rule is a chain of 2h
// dependent tiers between launches, and a tier costs its latency, not its
// work.  Here every point advances one sub-timestep per tier (one tier a
// sub-timestep where the swept rule has two: one growing, one shrinking).  A
// warp keeps O consecutive points of its own and G = (32 P - O) / 2 points of
// its neighbours on each side, P points a lane; the neighbour values of a tier
// come by shuffle.  The outermost R points of the window become wrong with each
// tier, so after K <= G / R tiers the warps trade: each writes its own points
// to a board in shared memory and reads its ghost points from its neighbours'
// boards (distributed shared memory when they are in another block of the
// cluster).  Boards are double buffered, so one barrier a trade is enough.
// Periodic ghosts wrap; the mirror wall of the insulated heat equation needs no
// code in the tiers, as a ghost point beyond it holds its mirror point's value
// and the update is symmetric in its neighbours, bit for bit.
//
// Bound: latency.  One tier is a shuffle (24 cycles) and a dependent update, or,
// in FP64, 64 cycles of the FP64 pipe per instruction and lane point, which is
// why FP64 grids are spread over up to 16 SMs with one point a lane.
#pragma once
#include <cooperative_groups.h>

#include "debug_check.cuh"
#include "ops.cuh"
#include "swept_geom.cuh"

namespace swept {

// the point a position x of the unbounded line stands for
__device__ __forceinline__ int resident_point(int x, int N, int bc) {
  if (bc == 0) {
    const int r = x % N;
    return r < 0 ? r + N : r;
  }
  int r = x % (2 * N);
  if (r < 0) r += 2 * N;
  return r < N ? r : 2 * N - 1 - r;
}

template <typename T, class Op, int STAGE, int P>
__device__ __forceinline__ void resident_tier(const T (&src)[P], T (&dst)[P], const typename Op::K& k) {
  constexpr int R = Op::R;
  T w[P + 2 * R];
#pragma unroll
  for (int d = 0; d < R; ++d) {
    const int kl = (R - d + P - 1) / P, kr = 1 + d / P;
    w[d] = __shfl_up_sync(0xffffffffu, src[d - R + kl * P], kl);
    w[R + P + d] = __shfl_down_sync(0xffffffffu, src[d - (kr - 1) * P], kr);
  }
#pragma unroll
  for (int i = 0; i < P; ++i) w[R + i] = src[i];
#pragma unroll
  for (int i = 0; i < P; ++i) dst[i] = Op::template point_fp<STAGE>(&w[i], dst[i], k);
}

// O: points a warp owns; K: tiers between trades (a multiple of the stage count)
template <typename T, class Op, int P>
__global__ void __launch_bounds__(512) k_resident(int N, int bc, typename Op::K k, T* u, int64_t n_sub, int O, int K) {
  extern __shared__ __align__(16) unsigned char smraw[];
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  T* board = reinterpret_cast<T*>(smraw);  // two buffers of the block's own points
  const bool one_block = cluster.num_blocks() == 1;
  const int nw = (int)(blockDim.x >> 5), warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31u);
  const int per_block = nw * O;
  const int own0 = ((int)cluster.block_rank() * nw + warp) * O;
  const int x0 = own0 - (32 * P - O) / 2 + lane * P;
  T a[P], b[P];
  const T* ghost[P];  // where a point of another warp is read at a trade; null for the warp's own points
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const int x = x0 + i, p = resident_point(x, N, bc);
    const int rank = p / per_block;
    const bool own = x >= own0 && x < own0 + O && x < N;
    ghost[i] = own ? nullptr : cluster.map_shared_rank(board, rank) + (p - rank * per_block);
    a[i] = dbg::in_range(p, N, dbg::STATE) ? __ldcg(u + p) : T(0);
    b[i] = a[i];
  }
  int buf = 0;
  for (int64_t done = 0;;) {
    const int kk = (int)(n_sub - done < K ? n_sub - done : K);
    int t = 0;
    for (; t + 2 <= kk; t += 2) {
      resident_tier<T, Op, 0, P>(a, b, k);
      resident_tier<T, Op, Op::S == 1 ? 0 : 1, P>(b, a, k);
    }
    if (t < kk) {  // one-stage schemes only: n_sub is a multiple of the stage count, and so is K
      resident_tier<T, Op, 0, P>(a, b, k);
#pragma unroll
      for (int i = 0; i < P; ++i) a[i] = b[i];
    }
    done += kk;
    if (done >= n_sub) break;
    T* mine = board + buf * per_block + warp * O - own0 + x0;
#pragma unroll
    for (int i = 0; i < P; ++i)
      if (!ghost[i] && dbg::in_range(x0 + i - own0, O, dbg::WINDOW)) mine[i] = a[i];
    if (one_block)
      __syncthreads();
    else
      cluster.sync();
#pragma unroll
    for (int i = 0; i < P; ++i)
      if (ghost[i]) a[i] = ghost[i][buf * per_block];
    buf ^= 1;
  }
  // no write before every warp has read its start; no exit before a neighbour has read this block's board
  if (one_block)
    __syncthreads();
  else
    cluster.sync();
#pragma unroll
  for (int i = 0; i < P; ++i)
    if (!ghost[i] && dbg::in_range(x0 + i, N, dbg::STATE)) u[x0 + i] = a[i];
}

}  // namespace swept
