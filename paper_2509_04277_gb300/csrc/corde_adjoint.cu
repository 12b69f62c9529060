// Hand-written adjoint of the multi-step rollout (reverse-mode differentiation through
// the step of Fig. 5), with checkpoint-and-recompute.
//
// One thread block per rod, two elements per thread (the step kernel's <2, NT> layout).
// The forward rollout (rod_rollout) stores a checkpoint every K steps.  The reverse
// kernel walks the segments backwards.  For each segment it runs the K steps forward
// from the checkpoint, keeping the states and (record mode) the velocities the
// constraint half-sweeps start from in scratch memory; in recompute mode each step is
// run once more just before its reverse, its velocity records in shared memory.  Then,
// for each step (last to first), it applies the transposed Jacobian of the step:
//   r' = r + dt v2, q' = normalize(q + dt/2 q (x) (0, omega1))       (position update)
//   v2 = P(r, v1): 2 n_iters half-sweeps of distance impulses          (constraints)
//   v1 = damp (v + dt (w F + g)), omega1 = damp (omega + dt J^-1 (tau - omega x J omega))
//   F, tau = elastic forces / torques of Eq. 2, 3, 8 (second derivatives of the energies)
// Gradients flow to the initial positions and velocities and, accumulated over all
// steps, to the per-joint stiffness (K1, K2, K3) and intrinsic Darboux vectors u-hat.
#include "corde_reverse.cuh"
#include "corde_variants.cuh"

namespace corde {
namespace {

// A thread's place in a block of NT (see reverse_step): neighbours through shared memory and block
// barriers; sweep_v holds the step's records (rec_put).
template <int NT>
struct BlockNet {
  static constexpr bool kShared = false;  // (one exchange less on the chain)
  static constexpr int kUnroll = 2;       // iterations per block of code
  const int t, tn, tp;
  const float4 *par_u, *par_k;
  float4* halo;
  int& xc;
  const float4* sweep_v;
  __device__ __forceinline__ int e0() const { return 2 * t; }
  __device__ __forceinline__ bool has_next() const { return t + 1 < NT; }
  __device__ __forceinline__ bool has_prev() const { return t > 0; }
  __device__ __forceinline__ float4 u(int e) const { return par_u[e * NT + t]; }
  __device__ __forceinline__ float4 k(int e) const { return par_k[e * NT + t]; }
  __device__ __forceinline__ float3 rec(int slot, int e) const { return rec_get<2, NT>(sweep_v, slot, e, t); }
  // (in-range neighbour slots at the ends)
  __device__ __forceinline__ float3 rec_next(int slot) const { return rec_get<2, NT>(sweep_v, slot, 0, tn); }
  __device__ __forceinline__ float3 rec_prev(int slot) const { return rec_get<2, NT>(sweep_v, slot, 1, tp); }
  __device__ __forceinline__ float4* buffer() {
    float4* hb = halo + (xc & 1) * kHaloSlots * NT;
    ++xc;
    return hb;
  }
  __device__ __forceinline__ void swap_velocities(float3 first, float3 last, float3& next, float3& prev) {
    const BlockHalo<NT, NT> H{t};
    float4* hb = buffer();
    H.put3(hb, 0, first);
    H.put3(hb, 1, last);
    block_sync<NT>();
    next = H.sweep_next(hb);
    prev = H.sweep_prev(hb);
  }
  // the next thread's a and b
  __device__ __forceinline__ void swap_forces(float3 a, float3 b, float3& an, float3& bn) {
    float4* hb = buffer();
    hb[t] = make_float4(a.x, a.y, a.z, 0.f);
    hb[NT + t] = make_float4(b.x, b.y, b.z, 0.f);
    block_sync<NT>();
    an = bn = zero3();
    if (has_next()) {
      an = f3(hb[t + 1]);
      bn = f3(hb[NT + t + 1]);
    }
  }
  // the previous thread's a and b
  __device__ __forceinline__ void swap_carries(float3 a, float4 b, float3& ap, float4& bp) {
    float4* hb = buffer();
    hb[t] = make_float4(a.x, a.y, a.z, 0.f);
    hb[NT + t] = b;
    block_sync<NT>();
    ap = zero3();
    bp = zero4();
    if (has_prev()) {
      ap = f3(hb[t - 1]);
      bp = hb[NT + t - 1];
    }
  }
};

// Reverse pass over the whole rollout of one rod per block.  MODE 0: recompute every
// step before its reverse; 1: record mode with one sweep buffer (a step's records are
// copied in after the step before it is reversed); 2: record mode with two buffers (the
// copy overlaps the reverse of the step before).  PIPE (record mode, two buffers, full
// layout): each rod has a cluster of two blocks; the first records the segments, the
// second reverses them one segment behind, so that the recording of segment k - 1 runs
// while segment k is reversed (segment scratch in two sets, by segment parity; one
// cluster barrier per segment).
template <int NT, int MODE, bool COMPACT, bool PIPE = false>
__global__ void __launch_bounds__(NT)
adjoint_kernel(AdjointArgs a) {
  static_assert(!PIPE || (MODE == 2 && !COMPACT), "the pipelined form records the full layout");
  constexpr bool RECORD = MODE > 0;
  constexpr int STORE = COMPACT ? 2 : 1;  // step_body's record layout
  constexpr int NBUF = MODE == 2 ? 2 : 1;
  constexpr int EPT = 2;
  static_assert((3 * EPT * NT) % 4 == 0, "a record slot is a whole number of 16-byte pieces");
  extern __shared__ float4 smem[];
  float4* par_u = smem;
  float4* par_k = smem + EPT * NT;
  float4* halo = smem + 2 * EPT * NT;
  float4* sweep_v = halo + 2 * kHaloSlots * NT;
  // float4 per (step, block) record: 1 + n_iters (compact) or 2 n_iters slots of 3 EPT NT
  // floats (rec_put)
  const int64_t rec_stride = (int64_t)(COMPACT ? a.rec_iters + 1 : 2 * a.rec_iters) * 3 * EPT * NT / 4;

  const int rod_slot = PIPE ? (int)blockIdx.x / 2 : (int)blockIdx.x;  // the rod's place in the launch
  const int n_slots = PIPE ? (int)gridDim.x / 2 : (int)gridDim.x;
  const int role = PIPE ? (int)(blockIdx.x & 1) : 0;  // PIPE: 0 records, 1 reverses (the cluster rank)
  const int rid = a.work[rod_slot];
  const RodDev R = a.rods[rid];
  const int t = threadIdx.x;
  const int e0 = t * EPT;
  const int64_t E = a.n_elem;
  float3 v_drive = zero3(), w_drive = zero3();
  if (a.drive != nullptr) {
    v_drive = f3(a.drive[2 * rid]);
    w_drive = f3(a.drive[2 * rid + 1]);
  }

  float3 r[EPT], v[EPT], om[EPT];
  float4 q[EPT];
  float w[EPT];
  float3 rb[EPT], vb[EPT], ob[EPT], Kb[EPT], ub[EPT];
  float4 qb[EPT];
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    rb[e] = vb[e] = ob[e] = Kb[e] = ub[e] = zero3();
    qb[e] = zero4();
  }
  const BlockHalo<NT, NT> H{t};
  int xc = 0;
  StepCache<EPT> sc;  // launch constants of the step (filled on the first step)
  const int n_seg = (a.n_steps + a.ckpt_every - 1) / a.ckpt_every;
  bool params_loaded = false;
  // segment scratch: states 0 .. K and the velocity records of segment seg (two sets by
  // segment parity with PIPE)
  auto seg_base = [&](int seg) {
    return a.seg_states + (PIPE ? (int64_t)(seg & 1) * (a.ckpt_every + 1) * 4 * E : (int64_t)0);
  };
  auto rec_at = [&](int seg, int s) {
    return a.sweep_rec + ((int64_t)(PIPE ? (seg & 1) * a.ckpt_every : 0) + s) * n_slots * rec_stride +
           (int64_t)rod_slot * rec_stride;
  };
  // copies step s's record into a shared buffer: 16-byte pieces spread over the block
  // (a barrier orders them before any thread's reads; a block or cluster barrier orders
  // the recording pass's stores before them)
  auto fetch = [&](int seg, int s, float4* dst) {
    const float4* src = rec_at(seg, s);
    const int slots = R.n_iters > 0 ? (COMPACT ? R.n_iters + 1 : 2 * R.n_iters) : 0;
    const int n16 = slots * 3 * EPT * NT / 4;
    for (int k = t; k < n16; k += NT) cp_async16(dst + k, src + k);
    cp_async_commit();
  };
  // rounds: without PIPE round j records (or recomputes) segment n_seg - 1 - j and then
  // reverses it; with PIPE round j records segment n_seg - 1 - j (first block) while the
  // second block reverses segment n_seg - j
  const int n_round = PIPE ? n_seg + 1 : n_seg;
  for (int j = 0; j < n_round; ++j) {
    const int rec_seg = n_seg - 1 - j;
    const int rev_seg = PIPE ? n_seg - j : rec_seg;
    const bool do_rec = rec_seg >= 0 && role == 0;
    const bool do_rev = rev_seg >= 0 && rev_seg < n_seg && (!PIPE || role == 1);
    if (do_rec || !params_loaded) {
      // the recording (or recomputing) block loads the segment's checkpoint; a reversing
      // block only the inverse masses and joint parameters, once
      const int ls = do_rec ? rec_seg : n_seg - 1;
      const float4* ck = a.ckpt + (int64_t)ls * 4 * E;
      load_rod<EPT, NT>(R, t, t, ck, ck + E, ck + 2 * E, ck + 3 * E, a.u4, a.k4, r, v, q, om, w,
                        params_loaded ? nullptr : par_u, par_k);
      params_loaded = true;
    }
    if (do_rec) {
      const int cnt = min(a.ckpt_every, a.n_steps - rec_seg * a.ckpt_every);
      auto put_state = [&](int s) {
        float4* st = seg_base(rec_seg) + (int64_t)s * 4 * E + R.off;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
          if (e0 + e < R.n) {
            st[e0 + e] = make_float4(r[e].x, r[e].y, r[e].z, w[e]);
            if constexpr (!RECORD) st[E + e0 + e] = make_float4(v[e].x, v[e].y, v[e].z, 0.f);  // record mode reads none
            st[2 * E + e0 + e] = q[e];
            st[3 * E + e0 + e] = make_float4(om[e].x, om[e].y, om[e].z, 0.f);
          }
        }
      };
      if constexpr (RECORD) {
        // forward over the segment, keeping states 0 .. cnt and the velocity records
        for (int s = 0; s < cnt; ++s) {
          put_state(s);
          StepNeighbours nb;
          step_body<EPT, NT, STORE>(R, H, r, v, q, om, w, par_u, par_k, halo, xc, sc, v_drive, w_drive,
                                    rec_at(rec_seg, s), &nb);
        }
        put_state(cnt);
      } else {
        // recompute the segment's states into scratch
        for (int s = 0; s < cnt; ++s) {
          put_state(s);
          if (s + 1 < cnt)
            step_body<EPT, NT, 0>(R, H, r, v, q, om, w, par_u, par_k, halo, xc, sc, v_drive, w_drive, nullptr,
                                  nullptr);
        }
      }
    }
    if (!do_rev) {
      if constexpr (PIPE) cooperative_groups::this_cluster().sync();
      continue;
    }
    const int seg = rev_seg;
    const int t0 = seg * a.ckpt_every;
    const int cnt = min(a.ckpt_every, a.n_steps - t0);
    if constexpr (RECORD) {
      // the recording pass's stores are visible here: a block barrier follows each step's
      // records within step_body, or (PIPE) the cluster barrier ended the round that wrote
      // them
      fetch(seg, cnt - 1, sweep_v + ((cnt - 1) % NBUF) * rec_stride);
    }
    // reverse the segment's steps
    if constexpr (RECORD) {
      // Each step's inputs are loaded one step ahead, while the step before is reversed:
      // the state before it, its neighbour data and the loss gradient after it.  The frame
      // and angular velocity after step s are the state before step s + 1.  The segment
      // states are read from L2 (ld.cg): with PIPE another SM wrote them.
      float3 pr[EPT], pom[EPT], pg[EPT];
      float4 pq[EPT], pn0, pn1, pn2;
      float4 nq[EPT];
      float3 nom[EPT];
      auto prefetch = [&](int s) {
        const float4* st = seg_base(seg) + (int64_t)s * 4 * E + R.off;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
          pg[e] = zero3();
          if (e0 + e < R.n) {
            pr[e] = f3(__ldcg(st + e0 + e));
            pq[e] = __ldcg(st + 2 * E + e0 + e);
            pom[e] = f3(__ldcg(st + 3 * E + e0 + e));
            if (a.dLdpos != nullptr) pg[e] = f3(a.dLdpos[(int64_t)(t0 + s) * E + R.off + e0 + e]);
          }
        }
        // the neighbour data of the step: the neighbouring threads' nodes in the same state
        // (read where the constraint or joint exists; an in-range node elsewhere)
        const int in = min(e0 + EPT, R.n - 1), ip = min(max(e0 - 1, 0), R.n - 1);
        pn0 = __ldcg(st + in);
        pn1 = __ldcg(st + ip);
        pn2 = __ldcg(st + 2 * E + in);
      };
      {
        const float4* sn = seg_base(seg) + (int64_t)cnt * 4 * E + R.off;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
          nq[e] = q[e];
          nom[e] = om[e];
          if (e0 + e < R.n) {
            nq[e] = __ldcg(sn + 2 * E + e0 + e);
            nom[e] = f3(__ldcg(sn + 3 * E + e0 + e));
          }
        }
      }
      prefetch(cnt - 1);
      for (int s = cnt - 1; s >= 0; --s) {
        float3 r_in[EPT], om_in[EPT];
        float4 q_in[EPT];
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
          if (e0 + e < R.n) {
            r[e] = pr[e];
            q[e] = pq[e];
            om[e] = pom[e];
          }
          r_in[e] = r[e];
          q_in[e] = q[e];
          om_in[e] = om[e];
          if (a.dLdpos != nullptr && e0 + e < R.n) rb[e] += pg[e];  // loss gradient after this step
          if (e0 + e < R.n) {
            q[e] = nq[e];
            om[e] = nom[e];
          }
          nq[e] = q_in[e];
          nom[e] = om_in[e];
        }
        StepNeighbours nb;
        nb.r_next = f3(pn0);
        nb.w_next = pn0.w;
        nb.r_prev = f3(pn1);
        nb.w_prev = pn1.w;
        nb.q_next = pn2;
        // step s's sweeps (threads read their neighbours' entries too); with two buffers the
        // copy of step s - 1's starts once every thread is done with the buffer it reuses
        // (step s + 1's), with one buffer once every thread is done with step s's
        cp_async_wait_all();
        block_sync<NT>();
        if (s > 0) {
          if constexpr (NBUF == 2) fetch(seg, s - 1, sweep_v + ((s - 1) & 1) * rec_stride);
          prefetch(s - 1);
        }
        BlockNet<NT> net{t, min(t + 1, NT - 1), max(t - 1, 0), par_u, par_k, halo, xc, sweep_v + (s % NBUF) * rec_stride};
        reverse_step<COMPACT>(R, net, r_in, q_in, om_in, w, om, q, nb, sc, rb, vb, qb, ob, Kb, ub);
        if constexpr (NBUF == 1) {
          if (s > 0) {
            block_sync<NT>();
            fetch(seg, s - 1, sweep_v);
          }
        }
      }
    } else {
      // each step's state and loss gradient loaded one step ahead, as in record mode
      float3 pr[EPT], pv[EPT], pom[EPT], pg[EPT];
      float4 pq[EPT];
      auto prefetch = [&](int s) {
        const float4* st = seg_base(seg) + (int64_t)s * 4 * E + R.off;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
          pg[e] = zero3();
          if (e0 + e < R.n) {
            pr[e] = f3(st[e0 + e]);
            pv[e] = f3(st[E + e0 + e]);
            pq[e] = st[2 * E + e0 + e];
            pom[e] = f3(st[3 * E + e0 + e]);
            if (a.dLdpos != nullptr) pg[e] = f3(a.dLdpos[(int64_t)(t0 + s) * E + R.off + e0 + e]);
          }
        }
      };
      prefetch(cnt - 1);
      for (int s = cnt - 1; s >= 0; --s) {
        float3 r_in[EPT], om_in[EPT], g_s[EPT];
        float4 q_in[EPT];
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
          if (e0 + e < R.n) {
            r[e] = pr[e];
            v[e] = pv[e];
            q[e] = pq[e];
            om[e] = pom[e];
          }
          r_in[e] = r[e];
          q_in[e] = q[e];
          om_in[e] = om[e];
          g_s[e] = pg[e];
        }
        if (s > 0) prefetch(s - 1);
        StepNeighbours nb;
        step_body<EPT, NT, STORE>(R, H, r, v, q, om, w, par_u, par_k, halo, xc, sc, v_drive, w_drive, sweep_v, &nb);
        // loss gradient with respect to the positions after this step
        if (a.dLdpos != nullptr) {
#pragma unroll
          for (int e = 0; e < EPT; ++e)
            if (e0 + e < R.n) rb[e] += g_s[e];
        }
        BlockNet<NT> net{t, min(t + 1, NT - 1), max(t - 1, 0), par_u, par_k, halo, xc, sweep_v};
        reverse_step<COMPACT>(R, net, r_in, q_in, om_in, w, om, q, nb, sc, rb, vb, qb, ob, Kb, ub);
      }
    }
    if constexpr (PIPE) cooperative_groups::this_cluster().sync();  // end of the round
  }
  if (PIPE && role == 0) return;  // the recording block holds no gradients
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    const int i = e0 + e;
    if (i < R.n) {
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

using AdjointFn = void (*)(AdjointArgs);
template <int NT>
AdjointFn adjoint_fn_nt(int mode, bool compact) {
  switch (mode) {
    case 0: return compact ? adjoint_kernel<NT, 0, true> : adjoint_kernel<NT, 0, false>;
    case 1: return compact ? adjoint_kernel<NT, 1, true> : adjoint_kernel<NT, 1, false>;
    case 2: return compact ? adjoint_kernel<NT, 2, true> : adjoint_kernel<NT, 2, false>;
    default: return nullptr;
  }
}
// The reverse kernel of `nt` threads in `mode`, with the compact record layout or not
// (nullptr for a thread count that does not exist).
AdjointFn adjoint_fn(int nt, int mode, bool compact) {
  switch (nt) {
    case 32: return adjoint_fn_nt<32>(mode, compact);
    case 64: return adjoint_fn_nt<64>(mode, compact);
    case 128: return adjoint_fn_nt<128>(mode, compact);
    case 256: return adjoint_fn_nt<256>(mode, compact);
    default: return nullptr;
  }
}

// The pipelined reverse kernel (record mode, two buffers, full layout) of `nt` threads.
AdjointFn adjoint_pipe_fn(int nt) {
  switch (nt) {
    case 32: return adjoint_kernel<32, 2, false, true>;
    case 64: return adjoint_kernel<64, 2, false, true>;
    case 128: return adjoint_kernel<128, 2, false, true>;
    case 256: return adjoint_kernel<256, 2, false, true>;
    default: return nullptr;
  }
}

}  // namespace

int adjoint_smem_bytes(int nt, int n_iters, int mode, bool compact) {
  const int ept = 2;
  const int it = n_iters > 0 ? n_iters : 1;
  const int sweep = (compact ? it + 1 : 2 * it) * 3 * ept * nt / 4;  // record slots of one step, in float4
  return (2 * ept * nt + 2 * kHaloSlots * nt + (mode == 2 ? 2 : 1) * sweep) * (int)sizeof(float4);
}

cudaError_t adjoint_occupancy(int nt, int mode, bool compact, int smem, int* blocks) {
  const AdjointFn fn = adjoint_fn(nt, mode, compact);
  if (fn == nullptr) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, fn, nt, (size_t)smem);
}

cudaError_t preload_adjoint(int nt) {
  for (int c = 0; c < 2; ++c) {
    const AdjointFn fn = adjoint_fn(nt, 0, c != 0);
    if (fn == nullptr) return cudaErrorInvalidValue;
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, fn);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_adjoint(int nt, int mode, bool compact, const AdjointArgs& a, int n_blocks, int smem,
                           cudaStream_t s) {
  if ((mode > 0) != (a.sweep_rec != nullptr)) return cudaErrorInvalidValue;
  const AdjointFn fn = adjoint_fn(nt, mode, compact);
  if (fn == nullptr) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  fn<<<n_blocks, nt, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_pipe(int nt, const AdjointArgs& a, int n_rods, int smem, cudaStream_t s) {
  if (a.sweep_rec == nullptr) return cudaErrorInvalidValue;
  const AdjointFn fn = adjoint_pipe_fn(nt);
  if (fn == nullptr) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * n_rods);
  cfg.blockDim = dim3(nt);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, a);
}

}  // namespace corde
