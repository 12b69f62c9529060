// Latency form of the plain rod's time step: overlapping warp tiles.
//
// The block, cluster and grid kernels (corde_step.cuh, corde_cluster.cu) exchange boundary
// data at 2 + n_iters barriers a step.  Here a rod is cut into tiles of one warp, PER
// elements per lane.  A tile also steps G lanes of each neighbouring tile's elements
// (ghosts), so inside a step all exchanges are warp shuffles.  A ghost misses its outer
// neighbour: the force phase spoils one element from the tile's edge inward, each constraint
// iteration two more, 2 n_iters + 1 a step.  G lanes hold 24 (PER 4) or 22 (PER 2)
// elements, so the paper's ten iterations fit, and one exchange of the ghosts' state per
// step, with one barrier (on a grid: a wait for the two neighbours), replaces the twelve.  Fewer iterations allow several steps per
// exchange; more need velocity exchanges within the step.
//
// Every element takes the arithmetic of the <ARITH, *> layout of the block kernels, in
// the same order (ARITH elements per thread there: the layout decides the order in which
// an element's force contributions are added and the form of the impulses), so the results
// are the same bit for bit, whichever kernel runs.
#include <climits>

#include "corde_tile.cuh"

namespace corde {
namespace {

// MAXT threads per SM bound the registers: 256 for the lone warps of a long chain, 512 to fill an
// SM with rods of one warp.
template <int PER, int ARITH, int SYNC, int MAXT = 32 * kTileMaxWarps>
__global__ void __launch_bounds__(MAXT, 1)
tile_step_kernel(const RodDev* __restrict__ rods, const int* __restrict__ work, float4* __restrict__ x4,
                 float4* __restrict__ v4, float4* __restrict__ q4, float4* __restrict__ o4,
                 const float4* __restrict__ u4, const float4* __restrict__ k4, const float4* __restrict__ drive,
                 int n_steps, float4* __restrict__ traj, int64_t n_elem, int C, float4* __restrict__ gh,
                 float4* __restrict__ pos_out, CkptDev ckpt) {
  using T = Tile<PER>;
  extern __shared__ float4 smem[];
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  const int rid = work[blockIdx.x / C];
  const RodDev R = rods[rid];
  // the work list and the rod constants are only written with the host waiting, so they are
  // read before the wait for the stream's previous kernel (0.03 us a step of ten-step launches)
  if constexpr (!tile_on_grid(SYNC)) pdl_begin();
  const int K = T::count(R.n);
  const int k = (blockIdx.x % C) * W + (threadIdx.x >> 5);  // this warp's tile
  const bool active = k < K;  // warps beyond the rod only take part in the barriers
  TileRod<PER, ARITH> rod(R, lane, active ? (k * T::O + lane) * PER : R.n, x4, v4, q4, o4, u4, k4);
  TileLink<PER, SYNC, SYNC == kTileGrid ? T::kGridBuf : T::kBuf> link(k, K, W, lane, (R.n + PER - 1) / PER, smem, gh);
  float3 v_drive = zero3(), w_drive = zero3();
  if (drive != nullptr) {
    v_drive = f3(drive[2 * rid]);
    w_drive = f3(drive[2 * rid + 1]);
  }
  auto exchange = [&]() {
    float4 a[T::SLOTS];
    rod.pack(a);
    if (link.trade(a)) rod.unpack(a);
  };
  auto exchange_v = [&]() {
    float4 a[T::VSLOTS];
    rod.pack_v(a);
    if (link.trade(a)) rod.unpack_v(a);
  };

  // ---- steps between two exchanges, and iterations between two velocity exchanges when a
  // step has more than the ghosts allow: x spoilt elements become x + 1 in the force phase
  // and (x rounded up to even) + 1 in an iteration
  const bool inext = (R.flags & F_INEXT) != 0;
  const int n_iters = inext ? R.n_iters : 0;
  constexpr int kChunk = (T::B - 1) / 2;
  int steps_per = 1;
  if (n_iters <= kChunk) {
    int x = 0, s = 0;
    while (s < n_steps) {
      int y = x + 1;
      if (n_iters > 0) y = (y + (y & 1)) + 2 * n_iters - 1;
      if (y > T::B) break;
      x = y;
      ++s;
    }
    steps_per = s;
  }

  const float inv_dt = 1.f / R.dt;
  auto iteration = [&](auto tube_on) {
    rod.distance_iteration();
    if constexpr (decltype(tube_on)::value) {
#pragma unroll
      for (int e = 0; e < PER; ++e)
        if (rod.e0 + e < rod.n) tube_contact(rod.r[e], rod.v[e], rod.w[e], R, R.dt, inv_dt);
    }
  };
  int since = 0;
  for (int step = 0; step < n_steps; ++step) {
    if (K > 1 && since == steps_per) {
      exchange();
      since = 0;
    }
    ++since;
    if (ckpt.ckpt != nullptr && link.owned && step % ckpt.every == 0)
      put_checkpoint<PER>(ckpt, step, R, rod.e0, n_elem, rod.r, rod.v, rod.q, rod.om, rod.w);
    if (active) rod.forces(v_drive, w_drive);
    if (inext) {
      if (n_iters <= kChunk || K == 1) {
        if (active) {
          if (R.flags & F_TUBE) {
            for (int it = 0; it < n_iters; ++it) iteration(std::true_type());
          } else {
            // a lone warp hides no instruction fetch: ten iterations as one block of code at two
            // elements per lane (2.11 against 2.14 us/step unrolled twice, 512 nodes), five at
            // four, where ten miss the instruction cache (2.96 / 3.00 / 3.22 at 5 / 2 / 10, 5000)
            constexpr int kUnroll = PER == 2 ? 10 : 5;
#pragma unroll kUnroll
            for (int it = 0; it < n_iters; ++it) iteration(std::false_type());
          }
        }
      } else {
        for (int it0 = 0; it0 < n_iters; it0 += kChunk) {
          if (it0 > 0) exchange_v();
          if (active) {
            const int m = min(kChunk, n_iters - it0);
            if (R.flags & F_TUBE) {
              for (int it = 0; it < m; ++it) iteration(std::true_type());
            } else {
              for (int it = 0; it < m; ++it) iteration(std::false_type());
            }
          }
        }
      }
    }
    rod.positions();
    if (traj != nullptr && link.owned) {
#pragma unroll
      for (int e = 0; e < PER; ++e)
        if (rod.e0 + e < rod.n)
          traj[(int64_t)step * n_elem + R.off + rod.e0 + e] = make_float4(rod.r[e].x, rod.r[e].y, rod.r[e].z, rod.w[e]);
    }
  }

  // every tile has loaded its ghosts' elements, and read its neighbours' last buffers, before
  // any state is overwritten or any block leaves
  // (a grid sync has no limit of its own: every block is resident and every wait before it ends)
  if (K > 1) link.barrier();
  link.leave(k, lane);
  if constexpr (SYNC == kTileGrid) {
    // what a wait that ran out let through is anywhere in the rod: nothing of this launch stands
    if (K > 1 && link.ran_out()) {
      rod.spoil();
      if (traj != nullptr && link.owned) {
        const float nan = __int_as_float(0x7fffffff);
        for (int step = 0; step < n_steps; ++step)
#pragma unroll
          for (int e = 0; e < PER; ++e)
            if (rod.e0 + e < rod.n) traj[(int64_t)step * n_elem + R.off + rod.e0 + e] = make_float4(nan, nan, nan, rod.w[e]);
      }
    }
  }
  if (link.owned) rod.store(x4, v4, q4, o4, pos_out);
}

using TileFn = void (*)(const RodDev*, const int*, float4*, float4*, float4*, float4*, const float4*, const float4*,
                        const float4*, int, float4*, int64_t, int, float4*, float4*, CkptDev);

template <int PER, int ARITH>
TileFn tile_fn_t(const TilePlan& p) {
  if constexpr (PER == 4)
    if (p.grid) return tile_step_kernel<PER, ARITH, kTileGrid>;
  return p.blocks > 1 ? tile_step_kernel<PER, ARITH, kTileCluster> : tile_step_kernel<PER, ARITH, kTileBlock>;
}
TileFn tile_fn(const TilePlan& p) {
  if (p.full && p.grid && p.warps >= 1 && p.warps <= 2 * kTileMaxWarps && p.per == 4)
    return p.arith == 4 ? tile_step_kernel<4, 4, kTileGridSync, 512> : tile_step_kernel<4, 2, kTileGridSync, 512>;
  if (p.warps < 1 || p.warps > kTileMaxWarps) return nullptr;
  if (p.full) {
    if (p.blocks != 1 || p.warps != 1 || p.per != 2) return nullptr;
    return p.arith == 4 ? tile_step_kernel<2, 4, kTileBlock, 512> : tile_step_kernel<2, 2, kTileBlock, 512>;
  }
  if (p.per == 4 && p.arith == 4) return tile_fn_t<4, 4>(p);
  if (p.per == 4 && p.arith == 2) return tile_fn_t<4, 2>(p);
  if (p.per == 2 && p.arith == 4) return tile_fn_t<2, 4>(p);
  if (p.per == 2 && p.arith == 2) return tile_fn_t<2, 2>(p);
  return nullptr;
}
int tile_smem(const TilePlan& p, int warps) {
  return p.grid || (p.blocks == 1 && warps == 1) ? 0
                                                 : 2 * warps * (p.per == 4 ? Tile<4>::kBuf : Tile<2>::kBuf) * (int)sizeof(float4);
}

}  // namespace

int prepare_cluster(const void* fn, const TilePlan& p, int smem_max, int smem) {
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
  if (e == cudaSuccess && p.blocks > 8) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  int n = INT_MAX;
  if (e == cudaSuccess && p.blocks > 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.blocks);
    cfg.blockDim = dim3(32 * p.warps);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
  }
  if (e == cudaSuccess) return n;
  cudaGetLastError();
  return 0;
}

int tile_count(int per, int n) { return per == 4 ? Tile<4>::count(n) : Tile<2>::count(n); }
int64_t tile_halo_bytes(int per, int n) {
  const int64_t buf = per == 4 ? Tile<4>::kGridBuf : Tile<2>::kGridBuf;
  return (2 * tile_count(per, n) * buf + 1) * (int64_t)sizeof(float4);  // and the tail
}
unsigned* tile_tail(float4* gh, int per, int n) {
  return reinterpret_cast<unsigned*>(gh + tile_halo_bytes(per, n) / sizeof(float4) - 1);
}

int prepare_tile(const TilePlan& p) {
  const TileFn fn = tile_fn(p);
  if (fn == nullptr) return 0;
  if (!p.grid) return prepare_cluster(reinterpret_cast<const void*>(fn), p, tile_smem(p, kTileMaxWarps), tile_smem(p, p.warps));
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * p.warps, 0) != cudaSuccess) cudaGetLastError();
  return per_sm > 0 ? 1 : 0;  // (a block per SM: the plan has no more)
}

cudaError_t launch_tile(const StepArgs& a, int n_rods, const TilePlan& p, cudaStream_t s) {
  const TileFn fn = tile_fn(p);
  if (fn == nullptr) return cudaErrorInvalidValue;
  const dim3 grid(n_rods * p.blocks), block(32 * p.warps);
  if (!p.grid)
    return launch_kernel(fn, grid, block, tile_smem(p, p.warps), s, a.pdl, p.blocks > 1 ? p.blocks : 0, a.rods, a.work, a.x4,
                         a.v4, a.q4, a.o4, a.u4, a.k4, a.drive, a.n_steps, a.traj, a.n_elem, p.blocks, a.grid_halo,
                         a.pos_out, CkptDev{a.ckpt, a.ckpt_every});
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, a.rods, a.work, a.x4, a.v4, a.q4, a.o4, a.u4, a.k4, a.drive, a.n_steps, a.traj,
                            a.n_elem, p.blocks, a.grid_halo, a.pos_out, CkptDev{a.ckpt, a.ckpt_every});
}

}  // namespace corde
