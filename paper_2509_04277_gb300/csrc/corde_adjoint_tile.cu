// Latency form of the adjoint (corde_adjoint.cu) for few rods: overlapping warp tiles (corde_tile.cu)
// over several SMs per rod.
//
// Two kernels.  The checkpoint segments of a rollout do not depend on one another, so the first
// steps all of them forward at once, each on a cluster of its own, and keeps every step's state and
// the velocities before each of its half-sweeps.  The second walks the steps backwards: a warp
// holds two elements per lane, so the reverse sweeps exchange by shuffles, and the tiles exchange
// their ghosts' adjoints once a step.  An iteration spoils two elements from a tile's edge inward and
// the force phase one: 21 of the 22 ghosts for the paper's ten iterations.  The arithmetic
// is the block kernels' (reverse_step is theirs), so the gradients are the same bit for bit.
//
// 256 nodes x 200 steps, 20 steps a segment, one rod: 753 us, against 0.90 ms pipelined over two blocks
// and 1.17 ms in one.  What bounds it is the chain of a step: about 2300 instructions of a
// lone warp per SM partition, three cycles each.
#include "corde_reverse.cuh"
#include "corde_tile.cuh"

namespace corde {
namespace {

using T = Tile<2>;

// The records of a step of rod `slot`: [2 rec_iters][3][npad] floats, by element.
__device__ __forceinline__ int64_t rec_offset(const AdjointTileArgs& a, int step, int slot) {
  return ((int64_t)step * a.n_rods + slot) * (2 * a.rec_iters) * 3 * a.npad;
}

// Steps segment b % n_seg of rod b / n_seg (b the cluster's index) forward from its checkpoint.
__global__ void __launch_bounds__(32 * kTileMaxWarps, 1) tile_record_kernel(AdjointTileArgs a) {
  extern __shared__ float4 smem[];
  const int n_seg = (a.n_steps + a.ckpt_every - 1) / a.ckpt_every;
  const int b = blockIdx.x / a.blocks, seg = b % n_seg, slot = b / n_seg;
  const int rid = a.work[slot];
  const RodDev R = a.rods[rid];
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  const int K = T::count(R.n), k = (blockIdx.x % a.blocks) * W + (threadIdx.x >> 5);
  const bool active = k < K;
  const int64_t E = a.n_elem;
  const float4* ck = a.ckpt + (int64_t)seg * 4 * E;
  TileRod<2, 2> rod(R, lane, active ? (k * T::O + lane) * 2 : R.n, ck, ck + E, ck + 2 * E, ck + 3 * E, a.u4, a.k4);
  TileLink<2, kTileCluster, T::kBuf> link(k, K, W, lane, (R.n + 1) / 2, smem, nullptr);
  float3 v_drive = zero3(), w_drive = zero3();
  if (a.drive != nullptr) {
    v_drive = f3(a.drive[2 * rid]);
    w_drive = f3(a.drive[2 * rid + 1]);
  }
  // lanes beyond the rod's end write their zeros too: the reverse pass reads whole windows, and an
  // absent constraint times zero has to be zero
  const bool keeps = link.owned;
  const int t0 = seg * a.ckpt_every, cnt = min(a.ckpt_every, a.n_steps - t0);
  const int n_iters = (R.flags & F_INEXT) ? R.n_iters : 0;
  auto put_state = [&](int step) {
    float4* st = a.states + (int64_t)step * 4 * E + R.off + rod.e0;
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (keeps && rod.e0 + e < rod.n) {
        st[e] = make_float4(rod.r[e].x, rod.r[e].y, rod.r[e].z, rod.w[e]);
        st[2 * E + e] = rod.q[e];
        st[3 * E + e] = make_float4(rod.om[e].x, rod.om[e].y, rod.om[e].z, 0.f);
      }
  };
  auto put_record = [&](float* rec, int i) {
    if (!keeps) return;
    float2* f = reinterpret_cast<float2*>(rec + (int64_t)i * 3 * a.npad + rod.e0);
    f[0] = make_float2(rod.v[0].x, rod.v[1].x);
    f[a.npad / 2] = make_float2(rod.v[0].y, rod.v[1].y);
    f[a.npad] = make_float2(rod.v[0].z, rod.v[1].z);
  };
  for (int s = 0; s < cnt; ++s) {
    if (K > 1 && s > 0) {
      float4 x[T::SLOTS];
      rod.pack(x);
      if (link.trade(x)) rod.unpack(x);
    }
    put_state(t0 + s);
    if (active) {
      rod.forces(v_drive, w_drive);
      float* rec = a.rec + rec_offset(a, t0 + s, slot);
      for (int it = 0; it < n_iters; ++it) {
        put_record(rec, 2 * it);
        rod.even_sweep();
        put_record(rec, 2 * it + 1);
        rod.odd_sweep();
      }
    }
    rod.positions();
  }
  if (t0 + cnt == a.n_steps) put_state(a.n_steps);
  link.barrier();  // no block leaves while a neighbour still reads its buffers
}

// A lane's place in its tile (see reverse_step): neighbours by shuffles; rows of 64 floats of the
// tile's record window in shared memory.
struct WarpNet {
  static constexpr bool kShared = true;  // a shuffle more on the chain, a constraint less per iteration
  static constexpr int kUnroll = 5;      // 753 us; 777 at two, 835 at one and at ten (below)
  const int lane, e0_;
  const float4 (&u_)[2];
  const float4 (&k_)[2];
  const float* rows;
  __device__ __forceinline__ int e0() const { return e0_; }
  __device__ __forceinline__ bool has_next() const { return lane < 31; }
  __device__ __forceinline__ bool has_prev() const { return lane > 0; }
  __device__ __forceinline__ float4 u(int e) const { return u_[e]; }
  __device__ __forceinline__ float4 k(int e) const { return k_[e]; }
  __device__ __forceinline__ float3 rec(int slot, int e) const {
    const float2* p = reinterpret_cast<const float2*>(rows + slot * 192) + lane;
    return e == 0 ? f3(p[0].x, p[32].x, p[64].x) : f3(p[0].y, p[32].y, p[64].y);
  }
  __device__ __forceinline__ float3 rec_next(int slot) const {
    const float* p = rows + slot * 192 + min(2 * lane + 2, 63);
    return f3(p[0], p[64], p[128]);
  }
  __device__ __forceinline__ float3 from_prev(float3 a) const {
    const float3 p = up3(a);
    return has_prev() ? p : zero3();
  }
  __device__ __forceinline__ void swap_velocities(float3 first, float3 last, float3& next, float3& prev) const {
    next = down3(first);
    prev = zero3();  // (kShared: not needed)
  }
  __device__ __forceinline__ void swap_forces(float3 a, float3 b, float3& an, float3& bn) const {
    an = down3(a);
    bn = down3(b);
    if (!has_next()) an = bn = zero3();
  }
  __device__ __forceinline__ void swap_carries(float3 a, float4 b, float3& ap, float4& bp) const {
    ap = up3(a);
    bp = make_float4(__shfl_up_sync(0xffffffffu, b.x, 1), __shfl_up_sync(0xffffffffu, b.y, 1),
                     __shfl_up_sync(0xffffffffu, b.z, 1), __shfl_up_sync(0xffffffffu, b.w, 1));
  }
};

__global__ void __launch_bounds__(32 * kTileMaxWarps, 1) tile_adjoint_kernel(AdjointTileArgs a) {
  extern __shared__ float4 smem[];
  const int slot = blockIdx.x / a.blocks;
  const int rid = a.work[slot];
  const RodDev R = a.rods[rid];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int K = T::count(R.n), k = (blockIdx.x % a.blocks) * W + wid;
  const bool active = k < K;
  const int e0 = active ? (k * T::O + lane) * 2 : R.n;
  const int64_t E = a.n_elem;
  TileLink<2, kTileCluster, T::kBuf> link(k, K, W, lane, (R.n + 1) / 2, smem, nullptr);
  const int n_iters = (R.flags & F_INEXT) ? R.n_iters : 0;
  const int n_rows = 2 * a.rec_iters * 3;
  float* rows = reinterpret_cast<float*>(smem + 2 * W * T::kBuf) + (size_t)wid * 2 * n_rows * 64;  // two steps' windows
  // copies step s's record window of the tile: 16 bytes per lane, two rows at a time
  auto fetch = [&](int s) {
    const float* src = a.rec + rec_offset(a, s, slot) + k * T::O * 2 + (lane >> 4) * a.npad + (lane & 15) * 4;
    float* dst = rows + (size_t)(s & 1) * n_rows * 64 + lane * 4;
    for (int p = 0; p < n_iters * 3; ++p, src += 2 * a.npad, dst += 128)
      cp_async16(reinterpret_cast<float4*>(dst), reinterpret_cast<const float4*>(src));
    cp_async_commit();
  };
  float4 u[2], kk[2];
  float3 rb[2], vb[2], ob[2], Kb[2], ub[2];
  float4 qb[2], nq[2];
  float3 nom[2];
  // the state before a step and the loss gradient after it, loaded one step ahead
  float4 px[2], pq[2], po[2], pg[2];
  auto prefetch = [&](int s) {
    const float4* st = a.states + (int64_t)s * 4 * E + R.off + e0;
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (e0 + e < R.n) {
        px[e] = st[e];
        pq[e] = st[2 * E + e];
        po[e] = st[3 * E + e];
        if (a.dLdpos != nullptr) pg[e] = a.dLdpos[(int64_t)s * E + R.off + e0 + e];
      }
  };
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    rb[e] = vb[e] = ob[e] = Kb[e] = ub[e] = nom[e] = zero3();
    qb[e] = u[e] = kk[e] = px[e] = po[e] = pg[e] = zero4();
    nq[e] = pq[e] = make_float4(0.f, 0.f, 0.f, 1.f);
    if (e0 + e < R.n) {
      u[e] = a.u4[R.off + e0 + e];
      kk[e] = a.k4[R.off + e0 + e];
      const float4* st = a.states + (int64_t)a.n_steps * 4 * E + R.off + e0 + e;
      nq[e] = st[2 * E];
      nom[e] = f3(st[3 * E]);
    }
  }
  const StepCache<2> sc{};  // (used by the compact layout only)
  if (active) {
    fetch(a.n_steps - 1);
    prefetch(a.n_steps - 1);
  }
  for (int s = a.n_steps - 1; s >= 0; --s) {
    if (active) {
      float3 r[2], om[2], om1[2];
      float4 q[2], qo[2];
      float w[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        r[e] = f3(px[e]);
        w[e] = px[e].w;
        q[e] = pq[e];
        om[e] = f3(po[e]);
        if (a.dLdpos != nullptr && e0 + e < R.n) rb[e] += f3(pg[e]);  // loss gradient after this step
        qo[e] = nq[e];
        om1[e] = nom[e];
        nq[e] = q[e];
        nom[e] = om[e];
      }
      cp_async_wait_all();
      __syncwarp();
      if (s > 0) {
        fetch(s - 1);
        prefetch(s - 1);
      }
      StepNeighbours nb;
      nb.r_next = down3(r[0]);
      nb.w_next = __shfl_down_sync(0xffffffffu, w[0], 1);
      nb.r_prev = up3(r[1]);
      nb.w_prev = __shfl_up_sync(0xffffffffu, w[1], 1);
      nb.q_next = make_float4(__shfl_down_sync(0xffffffffu, q[0].x, 1), __shfl_down_sync(0xffffffffu, q[0].y, 1),
                              __shfl_down_sync(0xffffffffu, q[0].z, 1), __shfl_down_sync(0xffffffffu, q[0].w, 1));
      WarpNet net{lane, e0, u, kk, rows + (size_t)(s & 1) * n_rows * 64};
      reverse_step<false>(R, net, r, q, om, w, om1, qo, nb, sc, rb, vb, qb, ob, Kb, ub);
    }
    if (K > 1 && s > 0) {
      float4 x[T::SLOTS];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        x[3 * e] = make_float4(rb[e].x, rb[e].y, rb[e].z, vb[e].x);
        x[3 * e + 1] = make_float4(vb[e].y, vb[e].z, ob[e].x, ob[e].y);
        x[3 * e + 2] = qb[e];
      }
      x[6] = make_float4(ob[0].z, ob[1].z, 0.f, 0.f);
      if (link.trade(x)) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          rb[e] = f3(x[3 * e]);
          vb[e] = f3(x[3 * e].w, x[3 * e + 1].x, x[3 * e + 1].y);
          ob[e] = f3(x[3 * e + 1].z, x[3 * e + 1].w, e == 0 ? x[6].x : x[6].y);
          qb[e] = x[3 * e + 2];
        }
      }
    }
  }
  link.barrier();  // no block leaves while a neighbour still reads its buffers
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int i = e0 + e;
    if (link.owned && i < R.n) {
      const int64_t o = R.off + i;
      if (a.dpos0) a.dpos0[o] = make_float4(rb[e].x, rb[e].y, rb[e].z, 0.f);
      if (a.dvel0) a.dvel0[o] = make_float4(vb[e].x, vb[e].y, vb[e].z, 0.f);
      if (a.dquat0) a.dquat0[o] = qb[e];
      if (a.domega0) a.domega0[o] = make_float4(ob[e].x, ob[e].y, ob[e].z, 0.f);
      if (a.dK) a.dK[o] = make_float4(Kb[e].x, Kb[e].y, Kb[e].z, 0.f);
      if (a.duhat) a.duhat[o] = make_float4(ub[e].x, ub[e].y, ub[e].z, 0.f);
    }
  }
}

}  // namespace

int adjoint_tile_npad(int n) { return 2 * T::O * (T::count(n) - 1) + 64; }

cudaError_t launch_adjoint_tile(const AdjointTileArgs& a, int warps, cudaStream_t s) {
  if (warps < 1 || warps > kTileMaxWarps || a.rec_iters > kAdjointTileIters) return cudaErrorInvalidValue;
  const int n_seg = (a.n_steps + a.ckpt_every - 1) / a.ckpt_every;
  const int link = 2 * warps * T::kBuf * (int)sizeof(float4);
  const int rows = warps * 2 * (2 * a.rec_iters * 3) * 64 * (int)sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(tile_record_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, link);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tile_adjoint_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, link + rows);
  if (e == cudaSuccess)
    e = launch_kernel(tile_record_kernel, dim3(a.n_rods * n_seg * a.blocks), dim3(32 * warps), link, s, 0, a.blocks, a);
  if (e == cudaSuccess)
    e = launch_kernel(tile_adjoint_kernel, dim3(a.n_rods * a.blocks), dim3(32 * warps), link + rows, s, 0, a.blocks, a);
  return e;
}

}  // namespace corde
