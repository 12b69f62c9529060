// Building blocks of the tile kernels (corde_tile.cu, corde_pair_tile.cu): the part of a rod that
// one warp steps, PER elements per lane, and the exchange of ghosts between a rod's tiles.
#pragma once

#include <cooperative_groups.h>
#include <type_traits>

#include "corde_step.cuh"
#include "corde_variants.cuh"

namespace corde {

template <int PER>
struct Tile {
  static constexpr int G = PER == 4 ? 6 : 11;  // ghost lanes on each side
  static constexpr int O = 32 - 2 * G;         // lanes a tile owns (the rod's ends own their G too)
  static constexpr int B = PER * G;            // elements an exchange makes valid on each side
  static constexpr int SLOTS = PER == 4 ? 13 : 7;    // float4 of a lane's state: 13 floats per element
  static constexpr int VSLOTS = (3 * PER + 3) / 4;   // float4 of its velocities
  static constexpr int kBuf = SLOTS * 32;            // float4 of a tile's exchange buffer
  static constexpr int kGridBuf = (4 * SLOTS + 2) / 3 * 32;  // the same on a grid: three floats and a stamp
  // tiles of Q lanes' worth of elements
  __host__ __device__ static int count_lanes(int Q) { return Q <= 32 ? 1 : (Q - 32 + O - 1) / O + 1; }
  // tiles of a rod of n nodes
  __host__ __device__ static int count(int n) { return count_lanes((n + PER - 1) / PER); }
};

__device__ __forceinline__ float3 down3(float3 a) {
  return f3(__shfl_down_sync(0xffffffffu, a.x, 1), __shfl_down_sync(0xffffffffu, a.y, 1),
            __shfl_down_sync(0xffffffffu, a.z, 1));
}
__device__ __forceinline__ float3 up3(float3 a) {
  return f3(__shfl_up_sync(0xffffffffu, a.x, 1), __shfl_up_sync(0xffffffffu, a.y, 1),
            __shfl_up_sync(0xffffffffu, a.z, 1));
}
// Predicted offset of a constraint and its reciprocal length.
__device__ __forceinline__ float3 offset_of(float3 e, float3 va, float3 vb, float dt, float& il) {
  const float3 d = f3(__fmaf_rn(dt, __fsub_rn(vb.x, va.x), e.x), __fmaf_rn(dt, __fsub_rn(vb.y, va.y), e.y),
                      __fmaf_rn(dt, __fsub_rn(vb.z, va.z), e.z));
  il = rsqrtf(__fmaf_rn(d.x, d.x, __fmaf_rn(d.y, d.y, __fmul_rn(d.z, d.z))));
  return d;
}

// A warp's part of a rod: elements e0 ... e0 + PER - 1 of each lane (e0 >= n: none), stepped with
// the arithmetic of the <ARITH, *> layout.
template <int PER, int ARITH>
struct TileRod {
  static constexpr bool FOLD = StepCache<ARITH>::kFold;
  const RodDev R;
  const int lane, e0, n;
  float3 r[PER], v[PER], om[PER], uh[PER], kk[PER];
  float4 q[PER];
  float w[PER];
  // launch constants of the constraints: segment s joins elements s and s + 1; the last one
  // reaches into the next lane, and the lane's first element also ends the previous lane's last
  // one (index PER)
  float inv[PER + 1], ca[PER + 1], la[PER + 1], cb[PER + 1], lb[PER + 1];
  float3 e_seg[PER], e_left;  // the step's segment vectors

  __device__ __forceinline__ TileRod(const RodDev& R_, int lane_, int e0_, const float4* __restrict__ x4,
                                     const float4* __restrict__ v4, const float4* __restrict__ q4,
                                     const float4* __restrict__ o4, const float4* __restrict__ u4,
                                     const float4* __restrict__ k4)
      : R(R_), lane(lane_), e0(e0_), n(R_.n) {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int i = e0 + e;
      r[e] = v[e] = om[e] = uh[e] = kk[e] = zero3();
      q[e] = make_float4(0.f, 0.f, 0.f, 1.f);
      w[e] = 0.f;
      if (i < n) {
        const float4 a = x4[R.off + i];
        r[e] = f3(a);
        w[e] = a.w;
        v[e] = f3(v4[R.off + i]);
        if (i <= n - 2) q[e] = q4[R.off + i];  // (what the arrays hold beyond the last frame and joint is not read)
        om[e] = f3(o4[R.off + i]);
        if (i <= n - 3) {  // (an absent joint has K = 0 and so no torques)
          uh[e] = f3(u4[R.off + i]);
          kk[e] = f3(k4[R.off + i]);
        }
      }
    }
    const float w_next = __shfl_down_sync(0xffffffffu, w[0], 1), w_prev = __shfl_up_sync(0xffffffffu, w[PER - 1], 1);
#pragma unroll
    for (int s = 0; s <= PER; ++s) {
      const int j = s < PER ? e0 + s : e0 - 1;  // the segment's index in the rod
      const float wa = s < PER ? w[s % PER] : w_prev, wb = s + 1 < PER ? w[(s + 1) % PER] : (s < PER ? w_next : w[0]);
      const bool here = s < PER - 1 || (s == PER - 1 ? lane < 31 : lane > 0 && j >= 0);
      inv[s] = inv_dt_wsum(here && j + 1 <= n - 1, wa, wb, R.dt);
      ca[s] = wa * inv[s];
      cb[s] = wb * inv[s];
      la[s] = R.l0 * ca[s];
      lb[s] = R.l0 * cb[s];
    }
    e_left = zero3();
  }

  // one distance constraint of the lane; segments PER - 1 and PER belong half to the
  // neighbouring lanes, which compute the same impulse for their own half
  __device__ __forceinline__ void constrain(int s, float3 es, float3 va, float3 vb, float3* pa, float3* pb) const {
    float il;
    const float3 d = offset_of(es, va, vb, R.dt, il);
    if constexpr (FOLD) {
      if (pa != nullptr) {
        const float sa = -__fmaf_rn(la[s], il, -ca[s]);
        *pa = f3(__fmaf_rn(sa, d.x, va.x), __fmaf_rn(sa, d.y, va.y), __fmaf_rn(sa, d.z, va.z));
      }
      if (pb != nullptr) {
        const float sb = __fmaf_rn(lb[s], il, -cb[s]);
        *pb = f3(__fmaf_rn(sb, d.x, vb.x), __fmaf_rn(sb, d.y, vb.y), __fmaf_rn(sb, d.z, vb.z));
      }
    } else {
      const float sc = __fmul_rn(__fmaf_rn(R.l0, il, -1.f), inv[s]);
      const float3 gi = f3(__fmul_rn(sc, d.x), __fmul_rn(sc, d.y), __fmul_rn(sc, d.z));
      if (pa != nullptr) {
        const float wa = w[s % PER];
        *pa = f3(__fmaf_rn(-wa, gi.x, va.x), __fmaf_rn(-wa, gi.y, va.y), __fmaf_rn(-wa, gi.z, va.z));
      }
      if (pb != nullptr) {
        const float wb = s < PER ? w[(s + 1) % PER] : w[0];
        *pb = f3(__fmaf_rn(wb, gi.x, vb.x), __fmaf_rn(wb, gi.y, vb.y), __fmaf_rn(wb, gi.z, vb.z));
      }
    }
  }

  // Forces, their integration into the velocities, the frames, and the constraint geometry.
  __device__ __forceinline__ void forces(float3 v_drive, float3 w_drive) {
    const bool inext = (R.flags & F_INEXT) != 0, clamp = (R.flags & F_CLAMP) != 0;
    const float dt = R.dt, half_dt = 0.5f * dt;
    // ---- elastic forces and torques
    float3 F[PER], tau[PER];
    const float3 r_next = down3(r[0]), r_prev = up3(r[PER - 1]);
    const float4 q_next = make_float4(__shfl_down_sync(0xffffffffu, q[0].x, 1), __shfl_down_sync(0xffffffffu, q[0].y, 1),
                                      __shfl_down_sync(0xffffffffu, q[0].z, 1), __shfl_down_sync(0xffffffffu, q[0].w, 1));
    // each element's joint and segment, all computed before any is added up
    float3 ta[PER], tb[PER], fa[PER], fb[PER], t_body[PER];
    float lk[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const float4 qb = e + 1 < PER ? q[(e + 1) % PER] : q_next;
      const float3 rb = e + 1 < PER ? r[(e + 1) % PER] : r_next;
      joint_torques(q[e], qb, make_float4(uh[e].x, uh[e].y, uh[e].z, 0.f), make_float4(kk[e].x, kk[e].y, kk[e].z, 0.f),
                    R.two_over_l, ta[e], tb[e]);
      segment_forces(r[e], rb, q[e], R, e0 + e <= n - 2, !inext, fa[e], fb[e], t_body[e], lk[e]);
    }
    float3 Fi = up3(fb[PER - 1]), Ti = up3(tb[PER - 1]);  // from the previous lane's last element
    if (lane == 0) Fi = Ti = zero3();
    // The layout's order: an element that starts one of its threads takes the previous element's
    // contribution after its own, the others before (at ARITH > PER two lanes make a thread).
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const float3 f = e == 0 ? Fi : fb[(e + PER - 1) % PER], c = e == 0 ? Ti : tb[(e + PER - 1) % PER];
      const bool after = ARITH <= PER ? e % ARITH == 0 : e == 0 && ((e0 >> 1) & 1) == 0;
      auto pick = [](bool p, float3 x) { return f3(p ? x.x : 0.f, p ? x.y : 0.f, p ? x.z : 0.f); };
      F[e] = add_rn(add_rn(pick(!after, f), fa[e]), pick(after, f));
      tau[e] = add_rn(add_penalty_torque(add_rn(pick(!after, c), ta[e]), lk[e], t_body[e]), pick(after, c));
    }

    // ---- constraint geometry
#pragma unroll
    for (int s = 0; s < PER; ++s)
      e_seg[s] = safe_segment(inv[s], segment_vector(r[s], s + 1 < PER ? r[(s + 1) % PER] : r_next), R.l0);
    e_left = safe_segment(inv[PER], segment_vector(r_prev, r[0]), R.l0);

    // ---- force integration and frames
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int i = e0 + e;
      integrate_node(R, w[e], F[e], v[e]);
      integrate_frame(R, (i <= n - 2) && !(clamp && i == 0), tau[e], om[e]);
    }
    if (clamp && e0 == 0) {
      v[0] = v_drive;
      om[0] = w_drive;
    }
#pragma unroll
    for (int e = 0; e < PER; ++e) update_frame(half_dt, e0 + e <= n - 2, om[e], q[e]);
  }

  // One iteration of the distance constraints, red-black.
  __device__ __forceinline__ void even_sweep() {
#pragma unroll
    for (int s = 0; s < PER; s += 2) constrain(s, e_seg[s], v[s], v[s + 1], &v[s], &v[s + 1]);
  }
  __device__ __forceinline__ void odd_sweep() {
    const float3 vn = down3(v[0]), vp = up3(v[PER - 1]);
#pragma unroll
    for (int s = 1; s + 1 < PER; s += 2) constrain(s, e_seg[s], v[s], v[s + 1], &v[s], &v[s + 1]);
    float3 v_last, v_first;
    constrain(PER - 1, e_seg[PER - 1], v[PER - 1], vn, &v_last, nullptr);
    constrain(PER, e_left, vp, v[0], nullptr, &v_first);
    v[PER - 1] = v_last;
    v[0] = v_first;
  }
  __device__ __forceinline__ void distance_iteration() {
    even_sweep();
    odd_sweep();
  }

  __device__ __forceinline__ void positions() {
#pragma unroll
    for (int e = 0; e < PER; ++e) r[e] += R.dt * v[e];
  }

  // the lane's state as float4, and back
  __device__ __forceinline__ void pack(float4* a) const {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      a[3 * e] = make_float4(r[e].x, r[e].y, r[e].z, v[e].x);
      a[3 * e + 1] = make_float4(v[e].y, v[e].z, om[e].x, om[e].y);
      a[3 * e + 2] = q[e];
    }
    a[3 * PER] = make_float4(om[0].z, om[1].z, om[PER - 2].z, om[PER - 1].z);
  }
  __device__ __forceinline__ void unpack(const float4* a) {
    const float oz[4] = {a[3 * PER].x, a[3 * PER].y, a[3 * PER].z, a[3 * PER].w};
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      r[e] = f3(a[3 * e]);
      v[e] = f3(a[3 * e].w, a[3 * e + 1].x, a[3 * e + 1].y);
      q[e] = a[3 * e + 2];
      om[e] = f3(a[3 * e + 1].z, a[3 * e + 1].w, oz[e]);
    }
  }
  __device__ __forceinline__ void pack_v(float4* a) const {
    constexpr int VS = Tile<PER>::VSLOTS;
    float f[4 * VS];
    f[4 * VS - 1] = f[4 * VS - 2] = 0.f;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      f[3 * e] = v[e].x;
      f[3 * e + 1] = v[e].y;
      f[3 * e + 2] = v[e].z;
    }
#pragma unroll
    for (int s = 0; s < VS; ++s) a[s] = make_float4(f[4 * s], f[4 * s + 1], f[4 * s + 2], f[4 * s + 3]);
  }
  __device__ __forceinline__ void unpack_v(const float4* a) {
    constexpr int VS = Tile<PER>::VSLOTS;
    float f[4 * VS];
#pragma unroll
    for (int s = 0; s < VS; ++s) {
      f[4 * s] = a[s].x;
      f[4 * s + 1] = a[s].y;
      f[4 * s + 2] = a[s].z;
      f[4 * s + 3] = a[s].w;
    }
#pragma unroll
    for (int e = 0; e < PER; ++e) v[e] = f3(f[3 * e], f[3 * e + 1], f[3 * e + 2]);
  }

  // a state that no one takes for a result
  __device__ __forceinline__ void spoil() {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const float nan = __int_as_float(0x7fffffff);
      r[e] = v[e] = om[e] = f3(nan, nan, nan);
      q[e] = make_float4(nan, nan, nan, nan);
    }
  }

  __device__ __forceinline__ void store(float4* __restrict__ x4, float4* __restrict__ v4, float4* __restrict__ q4,
                                        float4* __restrict__ o4, float4* __restrict__ pos_out) const {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int i = e0 + e;
      if (i < n) {
        x4[R.off + i] = make_float4(r[e].x, r[e].y, r[e].z, w[e]);
        v4[R.off + i] = make_float4(v[e].x, v[e].y, v[e].z, 0.f);
        if (i <= n - 2) q4[R.off + i] = q[e];
        o4[R.off + i] = make_float4(om[e].x, om[e].y, om[e].z, 0.f);
        if (pos_out != nullptr) pos_out[R.off + i] = make_float4(r[e].x, r[e].y, r[e].z, w[e]);
      }
    }
  }
};

// How a rod's tiles exchange: the block's shared memory and barrier; the shared memory of a
// cluster's blocks and its barrier; global memory and a grid sync.
// kTileGrid: neighbours wait for each other by polling the data (a step of 16384 / 65536 nodes 3.31 /
// 4.51 us, 3.92 / 5.02 with a grid barrier between writing and reading; polling one slot and then reading all
// 3.65 / 4.53).  kTileGridSync: the barrier, with more than eight warps per SM, where the loop's
// registers spill (131072 nodes 7.01 us against 7.63).
enum TileSync { kTileBlock, kTileCluster, kTileGrid, kTileGridSync };
__host__ __device__ constexpr bool tile_on_grid(int sync) { return sync == kTileGrid || sync == kTileGridSync; }

// 16 bytes of three floats and a stamp in L2, written and read as one: a reader that finds the
// stamp has the floats, so neighbours need no barrier and no fence between data and flag.
__device__ __forceinline__ void put_stamped(float4* p, float x, float y, float z, unsigned stamp) {
  asm volatile(
      "{ .reg .b128 t; .reg .b64 lo, hi; mov.b64 lo, {%1, %2}; mov.b64 hi, {%3, %4}; mov.b128 t, {lo, hi};\n\t"
      "st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)),
      "r"(__float_as_uint(z)), "r"(stamp)
      : "memory");
}
__device__ __forceinline__ unsigned get_stamped(const float4* p, float& x, float& y, float& z) {
  unsigned a, b, c, stamp;
  asm volatile(
      "{ .reg .b128 t; .reg .b64 lo, hi; ld.relaxed.gpu.global.b128 t, [%4];\n\t"
      "mov.b128 {lo, hi}, t; mov.b64 {%0, %1}, lo; mov.b64 {%2, %3}, hi; }"
      : "=r"(a), "=r"(b), "=r"(c), "=r"(stamp)
      : "l"(p)
      : "memory");
  x = __uint_as_float(a);
  y = __uint_as_float(b);
  z = __uint_as_float(c);
  return stamp;
}
// Behind a grid's exchange buffers: the stamp of its last exchange, the launch in which a wait ran out
// (launch_id; 0: none), and the polls after which a wait gives up.
enum TileTail { kTailStamp, kTailLost, kTailLimit };

// A warp's place among the K tiles of a rod (or pair): tile k holds lanes k O ... k O + 31 of it.
// BUF: float4 of a tile's exchange buffer, of which there are two, used in turn.
template <int PER, int SYNC, int BUF>
struct TileLink {
  bool owned;               // the tile owns the lane's elements
  float4* mine;             // where the lane publishes
  const float4* theirs;     // where a ghost lane's owner publishes (NULL: not a ghost)
  int64_t stride;           // from one buffer to the other
  int parity = 0;
  // grids: the stamp of the last exchange (it goes on from launch to launch, kept behind the buffers); this
  // launch's id (from the stamp it began with), the polls of a wait, and whether one of the tile's has given up
  unsigned* tail = nullptr;
  unsigned stamp = 0, launch_id = 0, limit = 0;
  bool lost = false;

  // Q: lanes of the whole rod; smem: the block's buffers, or gh: the grid's
  __device__ __forceinline__ TileLink(int k, int K, int W, int lane, int Q, float4* smem, float4* gh) {
    using T = Tile<PER>;
    const bool active = k < K;
    const int g = k * T::O + lane, wid = threadIdx.x >> 5;
    owned = active && (k == 0 || lane >= T::G) && (k == K - 1 || lane < 32 - T::G);
    mine = tile_on_grid(SYNC) ? gh + (int64_t)k * BUF + lane : smem + wid * BUF + lane;
    stride = (int64_t)(tile_on_grid(SYNC) ? K : W) * BUF;
    theirs = nullptr;
    if constexpr (SYNC == kTileGrid) {
      tail = reinterpret_cast<unsigned*>(gh + 2 * stride);
      stamp = __ldcg(tail + kTailStamp);
      limit = __ldcg(tail + kTailLimit);
      launch_id = 2 * stamp + 1;  // (a launch in which a wait can run out moves the stamp)
    }
    if (active && !owned && g < Q) {
      const int ok = min(max((g - T::G) / T::O, 0), K - 1);  // the tile that owns lane g
      const int ol = g - ok * T::O;
      if constexpr (tile_on_grid(SYNC)) {
        theirs = gh + (int64_t)ok * BUF + ol;
      } else if constexpr (SYNC == kTileCluster) {
        theirs = cooperative_groups::this_cluster().map_shared_rank(smem + (ok % W) * BUF + ol, ok / W);
      } else {
        theirs = smem + ok * BUF + ol;
      }
    }
  }
  __device__ __forceinline__ void barrier() const {
    if constexpr (tile_on_grid(SYNC)) {
      cooperative_groups::this_grid().sync();
    } else if constexpr (SYNC == kTileCluster) {
      cooperative_groups::this_cluster().sync();
    } else {
      __syncthreads();
    }
  }
  // the barrier of an exchange: it orders the tiles' shared-memory buffers (global memory on a grid of many warps)
  // and nothing else.  The full cluster barrier also waits for a block's global accesses in
  // flight, the adjoint's prefetches above all.
  // A tile's reads of a neighbour's buffer are not ordered by it: the release is that of the block's own shared
  // memory, and the arrive is relaxed.  They are complete all the same, since whatever a ghost lane reads in one
  // exchange goes into the step's arithmetic (forces, sweeps, positions, the reverse step), whose results the
  // warp stores into its own buffer before the next meet, and the neighbour rewrites the buffer that was read only
  // after that one.  An exchange of values that are not used before the next one would need a full barrier.
  __device__ __forceinline__ void meet() const {
    if constexpr (SYNC == kTileCluster) {
      asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
      asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
      barrier();
    }
  }
  // ghost lanes receive the N float4 of the lane that owns their elements (true for them)
  template <int N>
  __device__ __forceinline__ bool trade(float4 (&a)[N]) {
    if constexpr (SYNC == kTileGrid) return trade_stamped(a);
    static_assert(SYNC == kTileGrid || N * 32 <= BUF, "exchange buffer");
    if (owned) {
      float4* m = mine + parity * stride;
#pragma unroll
      for (int s = 0; s < N; ++s) {
        if constexpr (SYNC == kTileGridSync) __stcg(m + s * 32, a[s]);
        else m[s * 32] = a[s];
      }
    }
    meet();
    if (theirs != nullptr) {
      const float4* p = theirs + parity * stride;
#pragma unroll
      for (int s = 0; s < N; ++s) {
        if constexpr (SYNC == kTileGridSync) a[s] = __ldcg(p + s * 32);
        else a[s] = p[s * 32];
      }
    }
    parity ^= 1;
    return theirs != nullptr;
  }
  // On a grid a tile waits for its two neighbours only, by polling the data itself.  A tile
  // publishes exchange i only after it has read its neighbours' exchange i - 1, and they published
  // that after they had read its exchange i - 2: two buffers suffice.  Nothing else orders these accesses:
  // they are relaxed, and the vote orders no memory.  Within a warp the reads come first because the vote needs
  // every lane's stamps (a slot's stamp and floats are one access); between warps a slot read too late
  // would carry a newer stamp, which the loop does not take.
  template <int N>
  __device__ __forceinline__ bool trade_stamped(float4 (&a)[N]) {
    constexpr int M = (4 * N + 2) / 3;
    float f[3 * M];
    f[3 * M - 1] = f[3 * M - 2] = 0.f;
#pragma unroll
    for (int s = 0; s < N; ++s) {
      f[4 * s] = a[s].x;
      f[4 * s + 1] = a[s].y;
      f[4 * s + 2] = a[s].z;
      f[4 * s + 3] = a[s].w;
    }
    ++stamp;
    if (owned) {
      float4* m = mine + parity * stride;
#pragma unroll
      for (int s = 0; s < M; ++s) put_stamped(m + s * 32, f[3 * s], f[3 * s + 1], f[3 * s + 2], stamp);
    }
    const float4* p = theirs + parity * stride;
    for (unsigned tries = 0;; ++tries) {
      unsigned other = 0;
      if (theirs != nullptr) {
#pragma unroll
        for (int s = 0; s < M; ++s) other |= get_stamped(p + s * 32, f[3 * s], f[3 * s + 1], f[3 * s + 2]) ^ stamp;
      }
      if (__all_sync(0xffffffffu, other == 0)) break;
      // A wait that runs out marks the launch, and so ends every other wait: a tile that no longer waits runs ahead,
      // so its neighbours would each wait for the whole limit, one after the other.
      if (lost) break;
      if (tries >= limit) {
        lost = true;
        if ((threadIdx.x & 31) == 0) __stcg(tail + kTailLost, launch_id);
        break;
      }
      if ((tries & 255) == 255 && __any_sync(0xffffffffu, ran_out())) {
        lost = true;
        break;
      }
    }
#pragma unroll
    for (int s = 0; s < N; ++s) a[s] = make_float4(f[4 * s], f[4 * s + 1], f[4 * s + 2], f[4 * s + 3]);
    parity ^= 1;
    return theirs != nullptr;
  }
  // whether a wait of this launch has run out, on whichever tile (all see it after the launch's last barrier)
  __device__ __forceinline__ bool ran_out() const { return __ldcg(tail + kTailLost) == launch_id; }
  // after the launch's last barrier: the stamps go on from here
  __device__ __forceinline__ void leave(int k, int lane) const {
    if (SYNC == kTileGrid && k == 0 && lane == 0) tail[kTailStamp] = stamp;
  }
};

}  // namespace corde
