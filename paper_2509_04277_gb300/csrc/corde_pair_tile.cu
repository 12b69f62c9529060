// Latency form of the catheter/guidewire pair (corde_pair.cu): warp tiles that hold both rods.
//
// A lane holds two elements of the outer and two of the inner rod, the inner ones shifted
// by the binding offset so that an inner element's binding point lies on the lane's outer
// elements or on those of one neighbouring lane.  All exchanges of an iteration (the distance
// sweeps of both rods and the two binding colors) are then warp shuffles, where the block
// kernel needs a barrier per distance sweep and three for the binding; the ghosts are
// exchanged across the tiles once or twice a step.  The arithmetic and its order are the block
// kernel's, so the results are the same bit for bit.
//
// With k0 = floor(beta), inner element i binds to the outer elements i + k0 and i + k0 + 1.  Even k0:
// the lane's first inner element binds to the lane's two outer elements (color 0), its second
// to the lane's second and the next lane's first (color 1).  Odd k0: the first binds to the
// previous lane's second and the lane's first (color 0), the second to the lane's two.
// Elements spoilt from a tile's edge: one in the force phase, then two per iteration (four
// for two-way binding with even k0, whose across color follows its in-lane color); the counts
// come from stepping the dependencies of every phase.  22 ghosts hold ten (five) iterations.
#include "corde_tile.cuh"

namespace corde {
namespace {

constexpr int kPairBuf = 2 * Tile<2>::SLOTS * 32;

// TWO_WAY: some pair of the launch binds both ways (the others' outer shares are then zero).
template <int ARITH, bool TWO_WAY>
__global__ void __launch_bounds__(32 * kTileMaxWarps, 1)
pair_tile_kernel(const RodDev* __restrict__ rods, const int4* __restrict__ pairs, float4* __restrict__ x4,
                 float4* __restrict__ v4, float4* __restrict__ q4, float4* __restrict__ o4, const float4* __restrict__ u4,
                 const float4* __restrict__ k4, const float4* __restrict__ drive, int n_steps, int C,
                 float4* __restrict__ pos_out) {
  using T = Tile<2>;
  using Rod = TileRod<2, ARITH>;
  extern __shared__ float4 smem[];
  const int4 pr = pairs[blockIdx.x / C];  // (outer rod, inner rod, mode, 0)
  const int mode = pr.z;
  const RodDev Ro = rods[pr.x], Ri = rods[pr.y];
  pdl_begin();
  const int lane = threadIdx.x & 31, W = blockDim.x >> 5;
  float3 vd_o = zero3(), wd_o = zero3(), vd_i = zero3(), wd_i = zero3();
  float beta = 0.f;
  if (drive != nullptr) {
    vd_o = f3(drive[2 * pr.x]);
    wd_o = f3(drive[2 * pr.x + 1]);
    const float4 d = drive[2 * pr.y];
    vd_i = f3(d);
    beta = d.w;
    wd_i = f3(drive[2 * pr.y + 1]);
  }
  const float a = beta - floorf(beta), b = 1.f - a;
  // an offset beyond the outer rod binds nothing: the nearest such offset gives the window
  const int k0 = min(max((int)floorf(beta), -(Ri.n + 2)), Ro.n + 2);
  const bool odd = (k0 & 1) != 0;

  // ---- the tiles' window over both rods, in lanes of two outer elements: lane P holds the outer
  // elements 2 P, 2 P + 1 and the inner elements 2 (P - h), 2 (P - h) + 1
  const int h = (k0 + (odd ? 1 : 0)) / 2;  // (k0 + odd is even: exact)
  const int Qo = (Ro.n + 1) / 2, Qi = (Ri.n + 1) / 2;
  const int P0 = min(0, h), Q = max(Qo, Qi + h) - P0;
  const int K = T::count_lanes(Q);
  const int k = (blockIdx.x % C) * W + (threadIdx.x >> 5);
  const bool active = k < K;
  const int P = P0 + k * T::O + lane;
  Rod ro(Ro, lane, active && P >= 0 && P < Qo ? 2 * P : Ro.n + 1, x4, v4, q4, o4, u4, k4);
  Rod ri(Ri, lane, active && P - h >= 0 && P - h < Qi ? 2 * (P - h) : Ri.n + 1, x4, v4, q4, o4, u4, k4);
  TileLink<2, kTileCluster, kPairBuf> link(k, K, W, lane, Q, smem, nullptr);
  const float dt = Ri.dt;  // (the rods share it)

  auto exchange = [&]() {
    float4 s[2 * T::SLOTS];
    ro.pack(s);
    ri.pack(s + T::SLOTS);
    if (link.trade(s)) {
      ro.unpack(s);
      ri.unpack(s + T::SLOTS);
    }
  };
  auto exchange_v = [&]() {
    float4 s[2 * T::VSLOTS];
    ro.pack_v(s);
    ri.pack_v(s + T::VSLOTS);
    if (link.trade(s)) {
      ro.unpack_v(s);
      ri.unpack_v(s + T::VSLOTS);
    }
  };

  // the binding point between two outer elements, rounded as the block kernel's code is fused
  auto mix = [&](float x, float x1) { return __fmaf_rn(a, x1, __fmul_rn(b, x)); };
  // per step: the inner elements' offsets from their binding points, -1 / (dt w_eff) (0: not
  // bound), and the outer elements' shares (see PairHook)
  float3 rp[2];
  float inv[2], sk[2], sk1[2];
  auto binding_geometry = [&]() {
    // the outer element beyond the lane that the across color needs: the next lane's first (even
    // k0) or the previous lane's last (odd)
    const float3 rx = odd ? up3(ro.r[1]) : down3(ro.r[0]);
    const float wx = odd ? __shfl_up_sync(0xffffffffu, ro.w[1], 1) : __shfl_down_sync(0xffffffffu, ro.w[0], 1);
    const bool edge = lane == (odd ? 0 : 31);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const bool across = odd ? e == 0 : e == 1;
      const float3 rk = across ? (odd ? rx : ro.r[1]) : ro.r[0];
      const float3 rk1 = across ? (odd ? ro.r[0] : rx) : ro.r[1];
      const float wok = across ? (odd ? wx : ro.w[1]) : ro.w[0];
      const float wok1 = across ? (odd ? ro.w[0] : wx) : ro.w[1];
      const int i = ri.e0 + e, kn = i + k0;
      inv[e] = 0.f;
      rp[e] = zero3();
      sk[e] = sk1[e] = 0.f;
      if (i >= ri.n || kn < 0 || kn > ro.n - 2 || (across && edge)) continue;
      const float wk = mode == 2 ? wok : 0.f, wk1 = mode == 2 ? wok1 : 0.f;
      const float weff = __fmaf_rn(__fmul_rn(a, a), wk1, __fmaf_rn(__fmul_rn(b, b), wk, ri.w[e]));
      if (!(weff > 0.f)) continue;
      rp[e] = f3(__fsub_rn(ri.r[e].x, mix(rk.x, rk1.x)), __fsub_rn(ri.r[e].y, mix(rk.y, rk1.y)),
                 __fsub_rn(ri.r[e].z, mix(rk.z, rk1.z)));
      inv[e] = -1.f / (dt * weff);
      sk[e] = b * wk;
      sk1[e] = a * wk1;
    }
  };
  // one inner element's binding to outer velocities vk, vk1: the element and (two-way) both move;
  // branch-free, an unbound element (inv = 0) leaves all as they are
  auto bind = [&](int e, float3& vk, float3& vk1) {
    auto lambda = [&](float rpc, float ve, float x, float x1) {
      return __fmul_rn(inv[e], __fmaf_rn(dt, __fsub_rn(ve, mix(x, x1)), rpc));
    };
    const float3 lam = f3(lambda(rp[e].x, ri.v[e].x, vk.x, vk1.x), lambda(rp[e].y, ri.v[e].y, vk.y, vk1.y),
                          lambda(rp[e].z, ri.v[e].z, vk.z, vk1.z));
    const bool on = inv[e] != 0.f;
    auto move = [&](float3& v, float s) {
      v = f3(on ? __fmaf_rn(s, lam.x, v.x) : v.x, on ? __fmaf_rn(s, lam.y, v.y) : v.y, on ? __fmaf_rn(s, lam.z, v.z) : v.z);
    };
    move(ri.v[e], ri.w[e]);
    if constexpr (TWO_WAY) {
      move(vk, -sk[e]);
      move(vk1, -sk1[e]);
    }
  };
  // the across color's outer element comes from the neighbouring lane and goes back (an unbound
  // element sends it back unchanged); the tile's last lane in that direction keeps its own
  auto binding = [&]() {
    if (odd) {
      float3 vx = up3(ro.v[1]);
      bind(0, vx, ro.v[0]);
      if constexpr (TWO_WAY) {
        const float3 back = down3(vx);
        if (lane < 31) ro.v[1] = back;
      }
      bind(1, ro.v[0], ro.v[1]);
    } else {
      bind(0, ro.v[0], ro.v[1]);
      float3 vx = down3(ro.v[0]);
      bind(1, ro.v[1], vx);
      if constexpr (TWO_WAY) {
        const float3 back = up3(vx);
        if (lane > 0) ro.v[0] = back;
      }
    }
  };

  const int n_iters = Ro.n_iters;
  const int chunk = mode == 2 && !odd ? 5 : 10;
  for (int step = 0; step < n_steps; ++step) {
    if (K > 1 && step > 0) exchange();
    if (active) {
      ro.forces(vd_o, wd_o);
      ri.forces(vd_i, wd_i);
      if (mode != 0) binding_geometry();
    }
    for (int it0 = 0; it0 < n_iters; it0 += chunk) {
      if (K > 1 && it0 > 0) exchange_v();
      if (active) {
        const int m = min(chunk, n_iters - it0);
        for (int it = 0; it < m; ++it) {
          ro.distance_iteration();
          ri.distance_iteration();
          if (mode != 0) binding();
        }
      }
    }
    ro.positions();
    ri.positions();
  }
  link.barrier();
  if (link.owned) {
    ro.store(x4, v4, q4, o4, pos_out);
    ri.store(x4, v4, q4, o4, pos_out);
  }
}

}  // namespace

// Tiles of the widest window over two rods of at most n nodes (one just beyond the other).
int pair_tile_count(int n) { return Tile<2>::count_lanes(2 * ((n + 1) / 2) + 4); }

using PairTileFn = void (*)(const RodDev*, const int4*, float4*, float4*, float4*, float4*, const float4*, const float4*,
                            const float4*, int, int, float4*);
static PairTileFn pair_tile_fn(const TilePlan& p, bool two_way) {
  if (p.arith == 4) return two_way ? pair_tile_kernel<4, true> : pair_tile_kernel<4, false>;
  return two_way ? pair_tile_kernel<2, true> : pair_tile_kernel<2, false>;
}

int prepare_pair_tile(const TilePlan& p, bool two_way) {
  constexpr int kWarpSmem = 2 * kPairBuf * (int)sizeof(float4);
  return prepare_cluster(reinterpret_cast<const void*>(pair_tile_fn(p, two_way)), p, kTileMaxWarps * kWarpSmem,
                         p.warps * kWarpSmem);
}

cudaError_t launch_pair_tile(const StepArgs& a, const int4* pairs, int n_pairs, const TilePlan& p, bool two_way,
                             cudaStream_t s) {
  if (p.warps < 1 || p.warps > kTileMaxWarps) return cudaErrorInvalidValue;
  const int smem = 2 * p.warps * kPairBuf * (int)sizeof(float4);
  return launch_kernel(pair_tile_fn(p, two_way), dim3(n_pairs * p.blocks), dim3(32 * p.warps), smem, s, a.pdl, p.blocks,
                       a.rods, pairs, a.x4, a.v4, a.q4, a.o4, a.u4, a.k4, a.drive, a.n_steps, p.blocks, a.pos_out);
}

}  // namespace corde
