// The transposed time step (reverse mode), shared by the block kernels (corde_adjoint.cu) and the
// tile kernel (corde_adjoint_tile.cu).
#pragma once

#include "corde_step.cuh"

namespace corde {

__device__ __forceinline__ float4 qmul4(float4 a, float4 b) {
  return make_float4(a.w * b.x + a.x * b.w + a.y * b.z - a.z * b.y, a.w * b.y - a.x * b.z + a.y * b.w + a.z * b.x,
                     a.w * b.z + a.x * b.y - a.y * b.x + a.z * b.w, a.w * b.w - a.x * b.x - a.y * b.y - a.z * b.z);
}
__device__ __forceinline__ float4 pure(float3 v) { return make_float4(v.x, v.y, v.z, 0.f); }
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 scale4(float s, float4 a) { return make_float4(s * a.x, s * a.y, s * a.z, s * a.w); }
__device__ __forceinline__ float dot4(float4 a, float4 b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }
__device__ __forceinline__ float4 zero4() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// VJP of joint_torques: given the adjoints of (ta, tb), the adjoints of qa, qb, K, u-hat.
__device__ __forceinline__ void joint_torques_vjp(float4 qa, float4 qb, float4 uh, float4 K, float two_over_l,
                                                  float3 ta_bar, float3 tb_bar, float4& qa_bar, float4& qb_bar,
                                                  float3& K_bar, float3& uh_bar) {
  const float dw = dot4(qa, qb);
  const float3 dv = im_conj_mul(qa, qb);
  const float3 u = two_over_l * dv;
  const float3 du = f3(u.x - uh.x, u.y - uh.y, u.z - uh.z);
  const float3 m = f3(2.f * K.x * du.x, 2.f * K.y * du.y, 2.f * K.z * du.z);
  const float3 cv_bar = 0.5f * (ta_bar + tb_bar);
  const float3 diff = ta_bar - tb_bar;
  const float dw_bar = 0.5f * dot3(m, diff);
  const float3 m_bar = 0.5f * dw * diff + cross3(cv_bar, dv);
  float3 dv_bar = cross3(m, cv_bar);
  K_bar = f3(2.f * du.x * m_bar.x, 2.f * du.y * m_bar.y, 2.f * du.z * m_bar.z);
  const float3 u_bar = f3(2.f * K.x * m_bar.x, 2.f * K.y * m_bar.y, 2.f * K.z * m_bar.z);
  uh_bar = -u_bar;
  dv_bar += two_over_l * u_bar;
  // dv = Im(conj(qa) (x) qb): d/dqb = qa (x) (0, .), d/dqa = -qb (x) (0, .); dw = qa . qb
  qa_bar = add4(scale4(dw_bar, qb), scale4(-1.f, qmul4(qb, pure(dv_bar))));
  qb_bar = add4(scale4(dw_bar, qa), qmul4(qa, pure(dv_bar)));
}

// VJP of rotate_inv(q, v) = v + 2 u x (u x v - w v) (u, w: vector and real part of q).
__device__ __forceinline__ void rotate_inv_vjp(float4 q, float3 v, float3 o_bar, float3& v_bar, float4& q_bar) {
  const float3 u = f3(q.x, q.y, q.z);
  const float3 s = cross3(u, v) - q.w * v;
  const float3 z_bar = 2.f * o_bar;
  float3 u_bar = cross3(s, z_bar);
  const float3 s_bar = cross3(z_bar, u);
  u_bar += cross3(v, s_bar);
  v_bar = o_bar + cross3(s_bar, u) - q.w * s_bar;
  q_bar = make_float4(u_bar.x, u_bar.y, u_bar.z, -dot3(v, s_bar));
}

// VJP of director3.
__device__ __forceinline__ float4 director3_vjp(float4 q, float3 a) {
  return make_float4(2.f * (q.z * a.x - q.w * a.y) - 4.f * q.x * a.z, 2.f * (q.w * a.x + q.z * a.y) - 4.f * q.y * a.z,
                     2.f * (q.x * a.x + q.y * a.y), 2.f * (q.y * a.x - q.x * a.y));
}

// VJP of segment_forces.
__device__ __forceinline__ void segment_forces_vjp(float3 ra, float3 rb, float4 q, const RodDev& R, bool extensible,
                                                   float3 fa_bar, float3 fb_bar, float3 tq_bar, float3& ra_bar,
                                                   float3& rb_bar, float4& q_bar) {
  const float3 e = rb - ra;
  const float ee = dot3(e, e);
  const float il = rsqrtf(ee);
  const float3 t = il * e;
  const float3 d3 = director3(q);
  const float c = dot3(t, d3);
  const float k = R.lKp;
  const float3 f_bar = fb_bar - fa_bar;
  const float3 g = d3 - c * t;
  float il_bar = k * dot3(g, f_bar);
  float3 d3_bar = (k * il) * f_bar;
  const float c_bar = -k * il * dot3(t, f_bar);
  float3 t_bar = (-k * il * c) * f_bar;
  t_bar += c_bar * d3;
  d3_bar += c_bar * t;
  float ee_bar = 0.f;
  if (extensible) {
    const float len = ee * il;
    const float3 fs_bar = fa_bar - fb_bar;
    t_bar += (R.Ks * (len * R.inv_l0 - 1.f)) * fs_bar;
    const float len_bar = R.Ks * R.inv_l0 * dot3(t, fs_bar);
    ee_bar += il * len_bar;
    il_bar += ee * len_bar;
  }
  // torque l0 Kp (-t_b.y, t_b.x, 0), t_b = R(q)^T t
  const float3 tb_bar = f3(k * tq_bar.y, -k * tq_bar.x, 0.f);
  float3 t_bar2;
  float4 q_bar_rot;
  rotate_inv_vjp(q, t, tb_bar, t_bar2, q_bar_rot);
  t_bar += t_bar2;
  q_bar = add4(q_bar_rot, director3_vjp(q, d3_bar));
  // t = il e, il = ee^(-1/2), ee = e . e
  float3 e_bar = il * t_bar;
  il_bar += dot3(e, t_bar);
  ee_bar += -0.5f * il * il * il * il_bar;
  e_bar += (2.f * ee_bar) * e;
  ra_bar = -e_bar;
  rb_bar = e_bar;
}

// Asynchronous 16-byte global -> shared copies (completed by cp_async_wait_all).
__device__ __forceinline__ void cp_async16(float4* dst_smem, const float4* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Adjoint of one distance constraint (pre-update velocities va, vb): with g = s d and
// dg/dd = M = -(1/(dt W)) [(1 - l0/L) I + (l0/L) n n^T], d_bar = M (-wa va_bar + wb vb_bar);
// the caller applies va_bar -= dt d_bar, vb_bar += dt d_bar, ra_bar -= d_bar, rb_bar += d_bar.
// In two parts: the geometry (direction n and l0/L of the predicted segment) depends only
// on the recorded velocities, so it is computed before the exchange of the adjoint velocities;
// inv = -1/(dt W) is constant over a step, and 0 for a constraint that does not exist (the
// returned d_bar is then 0).
struct VjpGeo {
  float3 n;
  float rho;
};
__device__ __forceinline__ float vjp_inv(bool exists, float wa, float wb, float dt) {
  return (exists && wa + wb > 0.f) ? -__frcp_rn(__fmul_rn(dt, wa + wb)) : 0.f;
}
// e = r_b - r_a, a safe vector where the constraint does not exist (see vjp_segment)
__device__ __forceinline__ VjpGeo vjp_geo(float3 e, float3 va, float3 vb, float l0, float dt) {
  const float3 d = f3(__fmaf_rn(dt, __fsub_rn(vb.x, va.x), e.x), __fmaf_rn(dt, __fsub_rn(vb.y, va.y), e.y),
                      __fmaf_rn(dt, __fsub_rn(vb.z, va.z), e.z));
  const float dd = __fmaf_rn(d.x, d.x, __fmaf_rn(d.y, d.y, __fmul_rn(d.z, d.z)));
  const float il = rsqrtf(dd);
  return VjpGeo{il * d, l0 * il};
}
// The safe vector is long against any dt v, so that the predicted segment cannot vanish.
__device__ __forceinline__ float3 vjp_segment(float inv, float3 ra, float3 rb) {
  return inv != 0.f ? segment_vector(ra, rb) : f3(0.f, 0.f, 1e6f);
}
__device__ __forceinline__ float3 vjp_apply(const VjpGeo& G, float inv, float wa, float wb, float3 va_bar,
                                            float3 vb_bar) {
  const float3 g_bar = f3(__fmaf_rn(wb, vb_bar.x, -__fmul_rn(wa, va_bar.x)),
                          __fmaf_rn(wb, vb_bar.y, -__fmul_rn(wa, va_bar.y)),
                          __fmaf_rn(wb, vb_bar.z, -__fmul_rn(wa, va_bar.z)));
  return inv * ((1.f - G.rho) * g_bar + (G.rho * dot3(G.n, g_bar)) * G.n);
}

// One step of the reverse pass over a thread's two elements.  Net gives the thread's place in the
// rod (first element e0, neighbours), its joint parameters, the step's velocity records (of the
// thread's own elements, the next thread's first and the previous one's last; in the layout
// step_body writes with STORE == 2, COMPACT, or STORE == 1) and the exchanges with the neighbours.
// Net::kShared: the adjoint of the constraint to the previous thread comes from that thread, which
// computes it as its right one, instead of being computed on both sides.
template <bool COMPACT, class Net>
__device__ __forceinline__ void reverse_step(const RodDev& R, Net& net, const float3 (&r)[2], const float4 (&q)[2],
                                             const float3 (&om)[2], const float (&w)[2], const float3 (&om1)[2],
                                             const float4 (&qo)[2], const StepNeighbours& nb, const StepCache<2>& sc,
                                             float3 (&rb)[2], float3 (&vb)[2], float4 (&qb)[2], float3 (&ob)[2],
                                             float3 (&Kb)[2], float3 (&ub)[2]) {
  constexpr int EPT = 2;
  const int e0 = net.e0();
  const int n = R.n;
  const bool inext = (R.flags & F_INEXT) != 0;
  const bool clamp = (R.flags & F_CLAMP) != 0;
  const float dt = R.dt;
  const float half_dt = 0.5f * dt;

  // ---- position update: r' = r + dt v2, q' = normalize(q + dt/2 q (x) (0, omega1))
  float3 vb2[EPT], ob1[EPT];
  float4 qbi[EPT];
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    const int i = e0 + e;
    vb2[e] = vb[e] + dt * rb[e];
    ob1[e] = ob[e];
    qbi[e] = zero4();
    if (i <= n - 2) {
      const float4 a = q[e];
      const float3 o = om1[e];
      const float dx = a.w * o.x + a.y * o.z - a.z * o.y;
      const float dy = a.w * o.y + a.z * o.x - a.x * o.z;
      const float dz = a.w * o.z + a.x * o.y - a.y * o.x;
      const float dwq = -(a.x * o.x + a.y * o.y + a.z * o.z);
      const float4 p = make_float4(a.x + half_dt * dx, a.y + half_dt * dy, a.z + half_dt * dz, a.w + half_dt * dwq);
      const float inv = rsqrtf(dot4(p, p));
      const float4 pb = scale4(inv, add4(qb[e], scale4(-dot4(qo[e], qb[e]), qo[e])));
      qbi[e] = add4(pb, scale4(half_dt, qmul4(pb, make_float4(-o.x, -o.y, -o.z, 0.f))));
      ob1[e] += half_dt * im_conj_mul(a, pb);
    }
  }

  // ---- constraint half-sweeps in reverse order (odd, then even, last iteration first)
  if (inext) {
    // -1 / (dt W) of every constraint the thread touches (constant over the step)
    const float inv_e = vjp_inv(e0 + 1 <= n - 1, w[0], w[1], dt);
    const float inv_r = vjp_inv(net.has_next() && e0 + EPT <= n - 1, w[EPT - 1], nb.w_next, dt);
    const float inv_l = Net::kShared ? 0.f : vjp_inv(net.has_prev() && e0 <= n - 1, nb.w_prev, w[0], dt);
    // the segment vectors (positions are fixed during the sweeps), once per step
    const float3 s_r = vjp_segment(inv_r, r[EPT - 1], nb.r_next), s_e = vjp_segment(inv_e, r[0], r[1]);
    const float3 s_l = Net::kShared ? zero3() : vjp_segment(inv_l, nb.r_prev, r[0]);
    // the forward's boundary segment vectors
    const float3 e_r = safe_segment(sc.i_right, segment_vector(r[EPT - 1], nb.r_next), R.l0);
    const float3 e_l = safe_segment(sc.i_left, segment_vector(nb.r_prev, r[0]), R.l0);
    const Vec3x2 e_bnd{make_float2(e_r.x, e_l.x), make_float2(e_r.y, e_l.y), make_float2(e_r.z, e_l.z)};
    constexpr int kUnroll = Net::kUnroll;
#pragma unroll kUnroll
    for (int it = R.n_iters - 1; it >= 0; --it) {
      // geometry of this iteration's constraints, from the recorded velocities
      const int so = COMPACT ? 1 + it : 2 * it + 1;  // record slot before the odd half-sweep
      // the velocities before the even half-sweep: recorded; in the compact layout only for
      // the first iteration, and for a later one the odd half-sweep of the iteration before
      // repeated on its recorded input (the forward's own arithmetic, so the same values)
      float3 ve[EPT];
      {
        // slot 2 it; compact: slot 0, or the record before the previous odd half-sweep
        const int sp = COMPACT ? it : 2 * it;
#pragma unroll
        for (int e = 0; e < EPT; ++e) ve[e] = net.rec(sp, e);
        if constexpr (COMPACT) {
          if (it > 0) {
            const float3 vn = net.has_next() ? net.rec_next(sp) : zero3();
            const float3 vp = net.has_prev() ? net.rec_prev(sp) : zero3();
            boundary_apply(e_bnd, sc.l_bnd, sc.c_bnd, dt, vn, vp, ve[EPT - 1], ve[0]);
          }
        }
      }
      const VjpGeo g_r = vjp_geo(s_r, net.rec(so, EPT - 1), net.rec_next(so), R.l0, dt);
      VjpGeo g_l;
      if constexpr (!Net::kShared) g_l = vjp_geo(s_l, net.rec_prev(so), net.rec(so, 0), R.l0, dt);
      const VjpGeo g_e = vjp_geo(s_e, ve[0], ve[1], R.l0, dt);
      // exchange of the adjoint velocities of the first and last element
      float3 vn_bar, vp_bar;  // (finite where there is no neighbour)
      net.swap_velocities(vb2[0], vb2[EPT - 1], vn_bar, vp_bar);
      const float3 db_r = vjp_apply(g_r, inv_r, w[EPT - 1], nb.w_next, vb2[EPT - 1], vn_bar);
      vb2[EPT - 1] -= dt * db_r;
      rb[EPT - 1] -= db_r;
      float3 db_l;
      if constexpr (Net::kShared) {
        db_l = net.from_prev(db_r);
      } else {
        db_l = vjp_apply(g_l, inv_l, nb.w_prev, w[0], vp_bar, vb2[0]);
      }
      vb2[0] += dt * db_l;
      rb[0] += db_l;
      {
        const float3 db = vjp_apply(g_e, inv_e, w[0], w[1], vb2[0], vb2[1]);
        vb2[0] -= dt * db;
        vb2[1] += dt * db;
        rb[0] -= db;
        rb[1] += db;
      }
    }
  }

  // ---- force integration: v1 = damp (v + dt (w F + g)), omega1 = damp (...)
  float3 Fb[EPT], Tb[EPT];
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    const int i = e0 + e;
    if (w[e] > 0.f) {
      Fb[e] = (R.damp * dt * w[e]) * vb2[e];
      vb[e] = R.damp * vb2[e];
    } else {
      Fb[e] = zero3();
      vb[e] = zero3();
    }
    const bool frame_dynamic = (i <= n - 2) && !(clamp && i == 0);
    if (frame_dynamic) {
      const float3 b = f3(R.Jinv1 * ob1[e].x, R.Jinv1 * ob1[e].y, R.Jinv3 * ob1[e].z);
      Tb[e] = (R.damp * dt) * b;
      const float3 o = om[e];
      const float3 Jw = f3(R.J1 * o.x, R.J1 * o.y, R.J3 * o.z);
      const float3 oxb = cross3(o, b);
      const float3 Joxb = f3(R.J1 * oxb.x, R.J1 * oxb.y, R.J3 * oxb.z);
      ob[e] = R.damp * (ob1[e] + dt * (Joxb - cross3(Jw, b)));
    } else {
      Tb[e] = zero3();
      ob[e] = zero3();
    }
  }

  // ---- elastic forces and torques (transposed)
  float3 Fb_next, Tb_next;
  net.swap_forces(Fb[0], Tb[0], Fb_next, Tb_next);
  float3 r_carry = zero3();
  float4 q_carry = zero4();
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    const int j = e0 + e;
    const float4 qn = (e + 1 < EPT) ? q[(e + 1) % EPT] : nb.q_next;
    const float3 rn = (e + 1 < EPT) ? r[(e + 1) % EPT] : nb.r_next;
    if (j <= n - 3) {
      const float3 tbar_b = (e + 1 < EPT) ? Tb[(e + 1) % EPT] : Tb_next;
      float4 qa_bar, qn_bar;
      float3 K_bar, uh_bar;
      joint_torques_vjp(q[e], qn, net.u(e), net.k(e), R.two_over_l, Tb[e], tbar_b, qa_bar, qn_bar,
                        K_bar, uh_bar);
      qbi[e] = add4(qbi[e], qa_bar);
      if (e + 1 < EPT) {
        qbi[(e + 1) % EPT] = add4(qbi[(e + 1) % EPT], qn_bar);
      } else {
        q_carry = qn_bar;
      }
      Kb[e] += K_bar;
      ub[e] += uh_bar;
    }
    if (j <= n - 2) {
      const float3 fbar_b = (e + 1 < EPT) ? Fb[(e + 1) % EPT] : Fb_next;
      float3 ra_bar, rn_bar;
      float4 q_bar;
      segment_forces_vjp(r[e], rn, q[e], R, !inext, Fb[e], fbar_b, Tb[e], ra_bar, rn_bar, q_bar);
      rb[e] += ra_bar;
      if (e + 1 < EPT) {
        rb[(e + 1) % EPT] += rn_bar;
      } else {
        r_carry = rn_bar;
      }
      qbi[e] = add4(qbi[e], q_bar);
    }
  }
  float3 r_from;
  float4 q_from;
  net.swap_carries(r_carry, q_carry, r_from, q_from);
  if (net.has_prev()) {
    rb[0] += r_from;
    qbi[0] = add4(qbi[0], q_from);
  }
#pragma unroll
  for (int e = 0; e < EPT; ++e) qb[e] = qbi[e];
}


}  // namespace corde
