// Latency form of the plain rod's time step: overlapping warp tiles.
//
// The block, cluster and grid kernels (corde_step.cuh, corde_cluster.cu) exchange boundary
// data at 2 + n_iters barriers a step.  Here a rod is cut into tiles of one warp, PER
// elements per lane.  A tile also steps G lanes of each neighbouring tile's elements
// (ghosts), so inside a step all exchanges are warp shuffles.  A ghost misses its outer
// neighbour: the force phase spoils one element from the tile's edge inward, each constraint
// iteration two more, 2 n_iters + 1 a step.  G lanes hold 24 (PER 4) or 22 (PER 2)
// elements, so the paper's ten iterations fit, and one exchange of the ghosts' state per
// step, with one barrier, replaces the twelve.  Fewer iterations allow several steps per
// exchange; more need velocity exchanges within the step.
//
// Every element takes the arithmetic of the <ARITH, *> layout of the block kernels, in
// the same order (ARITH elements per thread there: the layout decides the order in which
// an element's force contributions are added and the form of the impulses), so the results
// are the same bit for bit, whichever kernel runs.
#include <cooperative_groups.h>
#include <type_traits>

#include "corde_step.cuh"
#include "corde_variants.cuh"

namespace corde {
namespace {

template <int PER>
struct Tile {
  static constexpr int G = PER == 4 ? 6 : 11;  // ghost lanes on each side
  static constexpr int O = 32 - 2 * G;         // lanes a tile owns (the rod's ends own their G too)
  static constexpr int B = PER * G;            // elements an exchange makes valid on each side
  static constexpr int SLOTS = PER == 4 ? 13 : 7;    // float4 of a lane's state: 13 floats per element
  static constexpr int VSLOTS = (3 * PER + 3) / 4;   // float4 of its velocities
  static constexpr int kBuf = SLOTS * 32;            // float4 of a tile's exchange buffer
  // tiles of a rod of n nodes
  __host__ __device__ static int count(int n) {
    const int Q = (n + PER - 1) / PER;
    return Q <= 32 ? 1 : (Q - 32 + O - 1) / O + 1;
  }
};

__device__ __forceinline__ float3 down3(float3 a) {
  return f3(__shfl_down_sync(0xffffffffu, a.x, 1), __shfl_down_sync(0xffffffffu, a.y, 1),
            __shfl_down_sync(0xffffffffu, a.z, 1));
}
__device__ __forceinline__ float3 up3(float3 a) {
  return f3(__shfl_up_sync(0xffffffffu, a.x, 1), __shfl_up_sync(0xffffffffu, a.y, 1),
            __shfl_up_sync(0xffffffffu, a.z, 1));
}
__device__ __forceinline__ float3 add_rn(float3 a, float3 b) {
  return f3(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z));
}

// Where a tile's ghosts come from: barrier and buffers of the rod's tiles.
enum TileSync { kTileBlock, kTileCluster, kTileGrid };

// Predicted offset of a constraint and its reciprocal length.
__device__ __forceinline__ float3 offset_of(float3 e, float3 va, float3 vb, float dt, float& il) {
  const float3 d = f3(__fmaf_rn(dt, __fsub_rn(vb.x, va.x), e.x), __fmaf_rn(dt, __fsub_rn(vb.y, va.y), e.y),
                      __fmaf_rn(dt, __fsub_rn(vb.z, va.z), e.z));
  il = rsqrtf(__fmaf_rn(d.x, d.x, __fmaf_rn(d.y, d.y, __fmul_rn(d.z, d.z))));
  return d;
}

template <int PER, int ARITH, int SYNC>
__global__ void __launch_bounds__(32 * kTileMaxWarps, 1)
tile_step_kernel(const RodDev* __restrict__ rods, const int* __restrict__ work, float4* __restrict__ x4,
                 float4* __restrict__ v4, float4* __restrict__ q4, float4* __restrict__ o4,
                 const float4* __restrict__ u4, const float4* __restrict__ k4, const float4* __restrict__ drive,
                 int n_steps, float4* __restrict__ traj, int64_t n_elem, int C, float4* __restrict__ gh,
                 float4* __restrict__ pos_out) {
  using T = Tile<PER>;
  constexpr bool FOLD = StepCache<ARITH>::kFold;
  constexpr int G = T::G, O = T::O;
  extern __shared__ float4 smem[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int c = blockIdx.x % C;
  const int rid = work[blockIdx.x / C];
  const RodDev R = rods[rid];
  // the work list and the rod constants are only written with the host waiting, so they are
  // read before the wait for the stream's previous kernel (0.03 us a step of ten-step launches)
  if constexpr (SYNC != kTileGrid) pdl_begin();
  const int n = R.n;
  const int K = T::count(n), Q = (n + PER - 1) / PER;
  const int k = c * W + wid;    // this warp's tile
  const bool active = k < K;    // warps beyond the rod only take part in the barriers
  const int g = k * O + lane;   // lane of the rod: elements g PER ... g PER + PER - 1
  const int e0 = g * PER;
  const bool owned = active && (k == 0 || lane >= G) && (k == K - 1 || lane < 32 - G);
  const bool inext = (R.flags & F_INEXT) != 0;
  const bool clamp = (R.flags & F_CLAMP) != 0;
  const float dt = R.dt, half_dt = 0.5f * dt, l0 = R.l0;

  // ---- load
  float3 r[PER], v[PER], om[PER], uh[PER], kk[PER];
  float4 q[PER];
  float w[PER];
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    const int i = e0 + e;
    r[e] = v[e] = om[e] = uh[e] = kk[e] = zero3();
    q[e] = make_float4(0.f, 0.f, 0.f, 1.f);
    w[e] = 0.f;
    if (active && i < n) {
      const float4 a = x4[R.off + i];
      r[e] = f3(a);
      w[e] = a.w;
      v[e] = f3(v4[R.off + i]);
      q[e] = q4[R.off + i];
      om[e] = f3(o4[R.off + i]);
      uh[e] = f3(u4[R.off + i]);
      kk[e] = f3(k4[R.off + i]);
    }
  }
  float3 v_drive = zero3(), w_drive = zero3();
  if (drive != nullptr) {
    v_drive = f3(drive[2 * rid]);
    w_drive = f3(drive[2 * rid + 1]);
  }

  // ---- where this lane publishes its state, and where a ghost lane reads its owner's
  float4* mine = nullptr;
  const float4* theirs = nullptr;
  int64_t buf_stride = 0;  // from an exchange's buffer to the next one's (two, in turn)
  if constexpr (SYNC == kTileGrid) {
    buf_stride = (int64_t)K * T::kBuf;
    mine = gh + (int64_t)k * T::kBuf + lane;
  } else {
    buf_stride = (int64_t)W * T::kBuf;
    mine = smem + wid * T::kBuf + lane;
  }
  if (active && !owned && g < Q) {
    const int ok = min(max((g - G) / O, 0), K - 1);  // the tile that owns lane g
    const int ol = g - ok * O;
    if constexpr (SYNC == kTileGrid) {
      theirs = gh + (int64_t)ok * T::kBuf + ol;
    } else if constexpr (SYNC == kTileCluster) {
      theirs = cooperative_groups::this_cluster().map_shared_rank(smem + (ok % W) * T::kBuf + ol, ok / W);
    } else {
      theirs = smem + ok * T::kBuf + ol;
    }
  }
  auto barrier = [&]() {
    if constexpr (SYNC == kTileGrid) {
      cooperative_groups::this_grid().sync();
    } else if constexpr (SYNC == kTileCluster) {
      cooperative_groups::this_cluster().sync();
    } else {
      __syncthreads();
    }
  };
  auto put = [&](float4* p, float4 a) {
    if constexpr (SYNC == kTileGrid) __stcg(p, a);
    else *p = a;
  };
  auto get = [&](const float4* p) {
    if constexpr (SYNC == kTileGrid) return __ldcg(p);
    else return *p;
  };
  int parity = 0;
  // the ghosts' whole state, from the lanes that own their elements
  auto exchange = [&]() {
    float4* m = mine + parity * buf_stride;
    if (owned) {
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        put(m + (3 * e) * 32, make_float4(r[e].x, r[e].y, r[e].z, v[e].x));
        put(m + (3 * e + 1) * 32, make_float4(v[e].y, v[e].z, om[e].x, om[e].y));
        put(m + (3 * e + 2) * 32, q[e]);
      }
      put(m + 3 * PER * 32, make_float4(om[0].z, om[1].z, om[PER - 2].z, om[PER - 1].z));
    }
    barrier();
    if (theirs != nullptr) {
      const float4* s = theirs + parity * buf_stride;
      const float4 z = get(s + 3 * PER * 32);
      const float oz[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        const float4 a = get(s + (3 * e) * 32), b = get(s + (3 * e + 1) * 32);
        q[e] = get(s + (3 * e + 2) * 32);
        r[e] = f3(a);
        v[e] = f3(a.w, b.x, b.y);
        om[e] = f3(b.z, b.w, oz[e]);
      }
    }
    parity ^= 1;
  };
  // the ghosts' velocities (between constraint iterations)
  auto exchange_v = [&]() {
    float4* m = mine + parity * buf_stride;
    float a[4 * T::VSLOTS];
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      a[3 * e] = v[e].x;
      a[3 * e + 1] = v[e].y;
      a[3 * e + 2] = v[e].z;
    }
    if constexpr (3 * PER < 4 * T::VSLOTS) a[4 * T::VSLOTS - 1] = a[4 * T::VSLOTS - 2] = 0.f;
    if (owned) {
#pragma unroll
      for (int s = 0; s < T::VSLOTS; ++s) put(m + s * 32, make_float4(a[4 * s], a[4 * s + 1], a[4 * s + 2], a[4 * s + 3]));
    }
    barrier();
    if (theirs != nullptr) {
      const float4* p = theirs + parity * buf_stride;
#pragma unroll
      for (int s = 0; s < T::VSLOTS; ++s) {
        const float4 b = get(p + s * 32);
        a[4 * s] = b.x;
        a[4 * s + 1] = b.y;
        a[4 * s + 2] = b.z;
        a[4 * s + 3] = b.w;
      }
#pragma unroll
      for (int e = 0; e < PER; ++e) v[e] = f3(a[3 * e], a[3 * e + 1], a[3 * e + 2]);
    }
    parity ^= 1;
  };

  // ---- launch constants of the constraints: segment s joins elements s and s + 1; the last
  // one reaches into the next lane, and the lane's first element also ends the previous
  // lane's last one (index PER)
  const float w_next = __shfl_down_sync(0xffffffffu, w[0], 1), w_prev = __shfl_up_sync(0xffffffffu, w[PER - 1], 1);
  float inv[PER + 1], ca[PER + 1], la[PER + 1], cb[PER + 1], lb[PER + 1];
#pragma unroll
  for (int s = 0; s <= PER; ++s) {
    const int j = s < PER ? e0 + s : e0 - 1;  // the segment's index in the rod
    const float wa = s < PER ? w[s % PER] : w_prev, wb = s + 1 < PER ? w[(s + 1) % PER] : (s < PER ? w_next : w[0]);
    const bool here = s < PER - 1 || (s == PER - 1 ? lane < 31 : lane > 0);
    inv[s] = inv_dt_wsum(active && here && j + 1 <= n - 1, wa, wb, dt);
    ca[s] = wa * inv[s];
    cb[s] = wb * inv[s];
    la[s] = l0 * ca[s];
    lb[s] = l0 * cb[s];
  }
  // one distance constraint of the lane; segments PER - 1 and PER belong half to the
  // neighbouring lanes, which compute the same impulse for their own half
  auto constrain = [&](int s, float3 es, float3 va, float3 vb, float3* pa, float3* pb) {
    float il;
    const float3 d = offset_of(es, va, vb, dt, il);
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
      const float sc = __fmul_rn(__fmaf_rn(l0, il, -1.f), inv[s]);
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
  };

  // ---- steps between two exchanges, and iterations between two velocity exchanges when a
  // step has more than the ghosts allow: x spoilt elements become x + 1 in the force phase
  // and (x rounded up to even) + 1 in an iteration
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

  int since = 0;
  for (int step = 0; step < n_steps; ++step) {
    if (K > 1 && since == steps_per) {
      exchange();
      since = 0;
    }
    ++since;
    float3 e_seg[PER], e_left = zero3();
    if (active) {
      // ---- elastic forces and torques
      float3 F[PER], tau[PER], Fc[PER + 1], Tc[PER + 1];
#pragma unroll
      for (int e = 0; e < PER; ++e) F[e] = tau[e] = zero3();
#pragma unroll
      for (int e = 0; e <= PER; ++e) Fc[e] = Tc[e] = zero3();
      const float3 r_next = down3(r[0]), r_prev = up3(r[PER - 1]);
      const float4 q_next = make_float4(__shfl_down_sync(0xffffffffu, q[0].x, 1), __shfl_down_sync(0xffffffffu, q[0].y, 1),
                                        __shfl_down_sync(0xffffffffu, q[0].z, 1), __shfl_down_sync(0xffffffffu, q[0].w, 1));
      auto joint_and_segment = [&](int e, float4 qb, float3 rb) {
        const int j = e0 + e;
        const bool carry = (e + 1) % (ARITH < PER ? ARITH : PER) == 0;  // to another lane, or a thread boundary of the layout
        if (j <= n - 3) {
          float3 ta, tb;
          joint_torques(q[e], qb, make_float4(uh[e].x, uh[e].y, uh[e].z, 0.f), make_float4(kk[e].x, kk[e].y, kk[e].z, 0.f),
                        R.two_over_l, ta, tb);
          tau[e] += ta;
          if (!carry) {
            tau[(e + 1) % PER] += tb;
          } else {
            Tc[e + 1] = tb;
          }
        }
        if (j <= n - 2) {
          float3 fa, fb, tq;
          segment_forces(r[e], rb, q[e], R, !inext, fa, fb, tq);
          F[e] += fa;
          tau[e] += tq;
          if (!carry) {
            F[(e + 1) % PER] += fb;
          } else {
            Fc[e + 1] = fb;
          }
        }
      };
      if constexpr (ARITH <= PER) {
#pragma unroll
        for (int e = 0; e < PER; ++e)
          joint_and_segment(e, e + 1 < PER ? q[(e + 1) % PER] : q_next, e + 1 < PER ? r[(e + 1) % PER] : r_next);
        Fc[0] = up3(Fc[PER]);
        Tc[0] = up3(Tc[PER]);
        if (lane == 0) Fc[0] = Tc[0] = zero3();
      } else {
        // two lanes make a thread of the <4, *> layout: the first element of the second lane
        // takes the previous element's contribution before its own, the first lane's after
        static_assert(ARITH <= PER || (PER == 2 && ARITH == 4), "tile layouts");
        float3 ta = zero3(), fa = zero3(), fb, tq, tb = zero3();
        if (e0 <= n - 3)
          joint_torques(q[0], q[1], make_float4(uh[0].x, uh[0].y, uh[0].z, 0.f), make_float4(kk[0].x, kk[0].y, kk[0].z, 0.f),
                        R.two_over_l, ta, tau[1]);
        if (e0 <= n - 2) {
          segment_forces(r[0], r[1], q[0], R, !inext, fa, fb, tq, &tb);
          F[1] += fb;
        }
        joint_and_segment(1, q_next, r_next);
        float3 Fi = up3(Fc[2]), Ti = up3(Tc[2]);
        if (lane == 0) Fi = Ti = zero3();
        if (lane & 1) {
          F[0] = Fi;
          tau[0] = Ti;
        } else {
          Fc[0] = Fi;
          Tc[0] = Ti;
        }
        F[0] = add_rn(F[0], fa);
        tau[0] = add_rn(tau[0], ta);
        // the penalty torque as the layouts fuse it (segment_forces' tq scaled and added)
        tau[0] = f3(__fmaf_rn(-R.lKp, tb.y, tau[0].x), __fmaf_rn(R.lKp, tb.x, tau[0].y), tau[0].z);
      }

      // ---- constraint geometry
#pragma unroll
      for (int s = 0; s < PER; ++s)
        e_seg[s] = safe_segment(inv[s], segment_vector(r[s], s + 1 < PER ? r[(s + 1) % PER] : r_next), l0);
      e_left = safe_segment(inv[PER], segment_vector(r_prev, r[0]), l0);

      // ---- force integration
      auto integrate = [&](int e) {
        const int i = e0 + e;
        if (w[e] > 0.f) {
          const float3 a = f3(w[e] * F[e].x + R.gx, w[e] * F[e].y + R.gy, w[e] * F[e].z + R.gz);
          v[e] = R.damp * (v[e] + dt * a);
        }
        const bool frame_dynamic = (i <= n - 2) && !(clamp && i == 0);
        if (frame_dynamic) {
          const float3 o = om[e];
          const float3 Jw = f3(R.J1 * o.x, R.J1 * o.y, R.J3 * o.z);
          const float3 rhs = tau[e] - cross3(o, Jw);
          const float3 on = f3(o.x + dt * R.Jinv1 * rhs.x, o.y + dt * R.Jinv1 * rhs.y, o.z + dt * R.Jinv3 * rhs.z);
          om[e] = R.damp * on;
        }
      };
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        if (e % ARITH == 0) {  // (zero for a second lane of ARITH > PER)
          F[e] = add_rn(F[e], Fc[e]);
          tau[e] = add_rn(tau[e], Tc[e]);
        }
        integrate(e);
      }
      if (clamp && e0 == 0) {
        v[0] = v_drive;
        om[0] = w_drive;
      }
      // ---- frames
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        if (e0 + e <= n - 2) {
          const float4 a = q[e];
          const float3 o = om[e];
          const float dx = a.w * o.x + a.y * o.z - a.z * o.y;
          const float dy = a.w * o.y + a.z * o.x - a.x * o.z;
          const float dz = a.w * o.z + a.x * o.y - a.y * o.x;
          const float dwq = -(a.x * o.x + a.y * o.y + a.z * o.z);
          const float4 b = make_float4(a.x + half_dt * dx, a.y + half_dt * dy, a.z + half_dt * dz, a.w + half_dt * dwq);
          const float il = rsqrtf(b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w);
          q[e] = make_float4(b.x * il, b.y * il, b.z * il, b.w * il);
        }
      }
    }

    // ---- distance-constraint iterations, red-black
    if (inext) {
      const float inv_dt = 1.f / dt;
      auto iteration = [&](auto tube_on) {
#pragma unroll
        for (int s = 0; s < PER; s += 2) constrain(s, e_seg[s], v[s], v[s + 1], &v[s], &v[s + 1]);
        const float3 vn = down3(v[0]), vp = up3(v[PER - 1]);
#pragma unroll
        for (int s = 1; s + 1 < PER; s += 2) constrain(s, e_seg[s], v[s], v[s + 1], &v[s], &v[s + 1]);
        float3 v_last, v_first;
        constrain(PER - 1, e_seg[PER - 1], v[PER - 1], vn, &v_last, nullptr);
        constrain(PER, e_left, vp, v[0], nullptr, &v_first);
        v[PER - 1] = v_last;
        v[0] = v_first;
        if constexpr (decltype(tube_on)::value) {
#pragma unroll
          for (int e = 0; e < PER; ++e)
            if (e0 + e < n) tube_contact(r[e], v[e], w[e], R, dt, inv_dt);
        }
      };
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
#pragma unroll
    for (int e = 0; e < PER; ++e) r[e] += dt * v[e];
    if (traj != nullptr && owned) {
#pragma unroll
      for (int e = 0; e < PER; ++e)
        if (e0 + e < n) traj[(int64_t)step * n_elem + R.off + e0 + e] = make_float4(r[e].x, r[e].y, r[e].z, w[e]);
    }
  }

  // every tile has loaded its ghosts' elements, and read its neighbours' last buffers, before
  // any state is overwritten or any block leaves
  if (K > 1) barrier();
  if (owned) {
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const int i = e0 + e;
      if (i < n) {
        x4[R.off + i] = make_float4(r[e].x, r[e].y, r[e].z, w[e]);
        v4[R.off + i] = make_float4(v[e].x, v[e].y, v[e].z, 0.f);
        q4[R.off + i] = q[e];
        o4[R.off + i] = make_float4(om[e].x, om[e].y, om[e].z, 0.f);
        if (pos_out != nullptr) pos_out[R.off + i] = make_float4(r[e].x, r[e].y, r[e].z, w[e]);
      }
    }
  }
}

using TileFn = void (*)(const RodDev*, const int*, float4*, float4*, float4*, float4*, const float4*, const float4*,
                        const float4*, int, float4*, int64_t, int, float4*, float4*);

template <int PER, int ARITH>
TileFn tile_fn_t(const TilePlan& p) {
  if (p.grid) return tile_step_kernel<PER, ARITH, kTileGrid>;
  return p.blocks > 1 ? tile_step_kernel<PER, ARITH, kTileCluster> : tile_step_kernel<PER, ARITH, kTileBlock>;
}
TileFn tile_fn(const TilePlan& p) {
  if (p.warps < 1 || p.warps > kTileMaxWarps) return nullptr;
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

int tile_count(int per, int n) { return per == 4 ? Tile<4>::count(n) : Tile<2>::count(n); }
int64_t tile_halo_bytes(int per, int n) {
  return (int64_t)2 * tile_count(per, n) * (per == 4 ? Tile<4>::kBuf : Tile<2>::kBuf) * (int64_t)sizeof(float4);
}

cudaError_t prepare_tile(const TilePlan& p) {
  const TileFn fn = tile_fn(p);
  if (fn == nullptr) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  if (!p.grid) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem(p, kTileMaxWarps));
  if (e == cudaSuccess && p.blocks > 8 && !p.grid)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

cudaError_t launch_tile(const StepArgs& a, int n_rods, const TilePlan& p, cudaStream_t s) {
  const TileFn fn = tile_fn(p);
  if (fn == nullptr) return cudaErrorInvalidValue;
  const dim3 grid(n_rods * p.blocks), block(32 * p.warps);
  if (!p.grid)
    return launch_kernel(fn, grid, block, tile_smem(p, p.warps), s, a.pdl, p.blocks > 1 ? p.blocks : 0, a.rods, a.work, a.x4,
                         a.v4, a.q4, a.o4, a.u4, a.k4, a.drive, a.n_steps, a.traj, a.n_elem, p.blocks, a.grid_halo,
                         a.pos_out);
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
                            a.n_elem, p.blocks, a.grid_halo, a.pos_out);
}

}  // namespace corde
