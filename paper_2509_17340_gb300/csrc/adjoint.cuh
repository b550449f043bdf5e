// Gradient of the Stage I cost S(1) of a noise-free rollout with respect to
// its T x 4 controls, by reverse mode (adjoint) through the rollout.  Not a
// step of the paper: it serves the gradient refinement of the updated nominals
// before Stage II and the cost-and-gradient entry point.
//
// Every recurrence over the steps is a scan, one step per lane (thread).  In the
// cost-and-gradient kernel:
// Forward: rollout_by_scans' prefix products and sums.  Backward, with
// L_{k+1} = dS/dx_{k+1} (the state terms at x_{k+1} plus what flows back from
// later steps):
//   position  Lp_{k+1} = sum_{i >= k} gp_i
//   velocity  Lv_{k+1} = sum_{i >= k} (gv_i + h Lp_{i+2})
//   attitude  the step is q_{k+1} = q_k (x) m_k / |q_k (x) m_k|, m_k from u_k
//     alone.  Its transposed Jacobian maps l to ((P l) / |y|) (x) conj(m_k), P
//     the projection off q_{k+1} and |y| = |m_k| for a unit q_k.  Multiplied
//     by conj(q_k) on the right this is (P l) (x) conj(q_{k+1}): the vector
//     part of l (x) conj(q), the adjoint in world axes, passes through a step
//     unchanged, and the scalar part is what P removes.  So
//     tau_{k+1} = vec(Lq_{k+1} (x) conj(q_{k+1})) is a suffix sum too: of the
//     attitude state terms and of what each step's translation contributes.
// Then dS/du_k of every step in parallel.
#pragma once

#include "device.cuh"
#include "internal.h"

namespace aero {

__device__ __forceinline__ State state_load(const float* d) {
  State x;
#pragma unroll
  for (int i = 0; i < 3; ++i) x.p[i] = d[i];
#pragma unroll
  for (int i = 0; i < 4; ++i) x.q[i] = d[3 + i];
#pragma unroll
  for (int i = 0; i < 3; ++i) x.v[i] = d[7 + i];
  return x;
}

// Stage I state terms at the post-step state x against guide sample (gx, gy,
// gz), given its nearest-point squared distance d2 and nearest point; the
// form the rollout kernels use.  kGrad: the gradient into gs[10] (overwritten).
template <bool kGrad>
__device__ __forceinline__ float state_terms(const State& x, float gx, float gy, float gz,
                                             float d2, float4 nearest, const CostParams& cp,
                                             float dmax2, float* gs) {
  const float ex = x.p[0] - gx, ey = x.p[1] - gy, ez = x.p[2] - gz;
  const float et = norm3f(ex, ey, ez);
  const float px = x.p[0] - cp.goal_rel[0], py = x.p[1] - cp.goal_rel[1], pz = x.p[2] - cp.goal_rel[2];
  const float np = norm3f(px, py, pz);
  const float vx = x.v[0] - cp.v_goal[0], vy = x.v[1] - cp.v_goal[1], vz = x.v[2] - cp.v_goal[2];
  const float nv = norm3f(vx, vy, vz);
  const float* q = x.q;
  const float* qg = cp.q_goal;
  const float r1 = -q[0] * qg[1] + q[1] * qg[0] - q[2] * qg[3] + q[3] * qg[2];
  const float r2 = -q[0] * qg[2] + q[1] * qg[3] + q[2] * qg[0] - q[3] * qg[1];
  const float r3 = -q[0] * qg[3] - q[1] * qg[2] + q[2] * qg[1] + q[3] * qg[0];
  const float nr = fast_sqrt(r1 * r1 + r2 * r2 + r3 * r3);
  const float jc = jcol_from_d2(d2, cp, dmax2);
  const float c = cp.Q_track * et + cp.Q_vnorm * (x.v[0] * x.v[0] + x.v[1] * x.v[1] + x.v[2] * x.v[2]) +
                  cp.Q_p * np + cp.Q_v * nv + cp.Q_q * 2.8284271247461903f * nr + jc;
  if (kGrad) {
#pragma unroll
    for (int i = 0; i < 10; ++i) gs[i] = 0.0f;
    if (et > 0.0f) {
      const float s = cp.Q_track / et;
      gs[0] += s * ex; gs[1] += s * ey; gs[2] += s * ez;
    }
    if (np > 0.0f) {
      const float s = cp.Q_p / np;
      gs[0] += s * px; gs[1] += s * py; gs[2] += s * pz;
    }
    gs[7] += 2.0f * cp.Q_vnorm * x.v[0];
    gs[8] += 2.0f * cp.Q_vnorm * x.v[1];
    gs[9] += 2.0f * cp.Q_vnorm * x.v[2];
    if (nv > 0.0f) {
      const float s = cp.Q_v / nv;
      gs[7] += s * vx; gs[8] += s * vy; gs[9] += s * vz;
    }
    if (nr > 0.0f) {
      // d r / d q: r1 (-g1, g0, -g3, g2), r2 (-g2, g3, g0, -g1), r3 (-g3, -g2, g1, g0)
      const float s = cp.Q_q * 2.8284271247461903f / nr;
      const float a = s * r1, b = s * r2, e = s * r3;
      gs[3] += -a * qg[1] - b * qg[2] - e * qg[3];
      gs[4] += a * qg[0] + b * qg[3] - e * qg[2];
      gs[5] += -a * qg[3] + b * qg[0] + e * qg[1];
      gs[6] += a * qg[2] - b * qg[1] + e * qg[0];
    }
    if (d2 < dmax2) {
      const float d = fast_sqrt(d2);  // as jcol_from_d2 takes it: the same branch of J_col
      if (d >= cp.d_min && d > 0.0f) {
        const float s = -cp.a_col * jc / d;
        gs[0] += s * (x.p[0] - nearest.x);
        gs[1] += s * (x.p[1] - nearest.y);
        gs[2] += s * (x.p[2] - nearest.z);
      }
    }
  }
  return c;
}

// One step's adjoint: from the start attitude q, the control u and the adjoints
// lp, lv of the step's end position and velocity, the parts that do not need
// the end attitude's adjoint; step_adjoint_controls adds that one.  With
// a = q (x) [0, w/2], hh = h^2 |w|^2 / 4 and the RK4 stage attitudes q_i =
// alpha_i q + beta_i a of the closed-form step (see rk4_step), the position and
// velocity increments are sums of r(q_i) = R(q_i) e3 / 2, so the adjoint of q_i
// is r'(q_i)^T w_i with w_1 = Wp + Wv, w_2 = w_3 = Wp + 2 Wv, w_4 = Wv (Wp, Wv: lp
// and lv times the increments' factors): four 4-vectors instead of a reverse
// sweep over the four stage states.
struct StepAdjoint {
  float ga[4];  // adjoint of a
  float ghh;    // adjoint of hh
  float gF;     // adjoint of the thrust
};

// r'(q)^T w, r(q) = (xz + wy, yz - wx, 1/2 - x^2 - y^2).
__device__ __forceinline__ void r_vjp(const float* q, const float* w, float* g) {
  g[0] = w[0] * q[2] - w[1] * q[1];
  g[1] = w[0] * q[3] - w[1] * q[0] - 2.0f * w[2] * q[1];
  g[2] = w[0] * q[0] + w[1] * q[3] - 2.0f * w[2] * q[2];
  g[3] = w[0] * q[1] + w[1] * q[2];
}

__device__ __forceinline__ float dot4(const float* a, const float* b) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2] + a[3] * b[3];
}

// a = q (x) [0, w/2] and hh of a step.
__device__ __forceinline__ float step_a(const float* q, float4 u, float h, float* a) {
  const float hx = 0.5f * u.y, hy = 0.5f * u.z, hz = 0.5f * u.w;
  a[0] = -q[1] * hx - q[2] * hy - q[3] * hz;
  a[1] = q[0] * hx + q[2] * hz - q[3] * hy;
  a[2] = q[0] * hy - q[1] * hz + q[3] * hx;
  a[3] = q[0] * hz + q[1] * hy - q[2] * hx;
  return h * h * (hx * hx + hy * hy + hz * hz);
}

// Vector part of l (x) conj(q).
__device__ __forceinline__ float3 vec_mul_conj(const float* l, const float* q) {
  return make_float3(-l[0] * q[1] + l[1] * q[0] - l[2] * q[3] + l[3] * q[2],
                     -l[0] * q[2] + l[1] * q[3] + l[2] * q[0] - l[3] * q[1],
                     -l[0] * q[3] - l[1] * q[2] + l[2] * q[1] + l[3] * q[0]);
}

// The translation's part of the step's adjoint into s; returns what it adds to
// tau of the step's start state.
__device__ __forceinline__ float3 step_adjoint_translation(const float* q, float4 u, const DynParams& dp,
                                                           float3 lp, float3 lv, StepAdjoint& s) {
  const float h = dp.dt;
  float a[4];
  const float hh = step_a(q, u, h, a);
  const float c3 = 1.0f - 0.25f * hh, c4 = 1.0f - 0.5f * hh, hb = 0.5f * h, h4 = h * c3;
  float q2[4], q3[4], q4[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    q2[i] = q[i] + hb * a[i];
    q3[i] = c3 * q[i] + hb * a[i];
    q4[i] = c4 * q[i] + h4 * a[i];
  }
  const float kp = h * h * (1.0f / 3.0f) * dp.inv_mass, kv = h * (1.0f / 3.0f) * dp.inv_mass;
  const float P[3] = {kp * lp.x, kp * lp.y, kp * lp.z}, V[3] = {kv * lv.x, kv * lv.y, kv * lv.z};
  float w1[3], w2[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    w1[i] = P[i] + V[i];
    w2[i] = w1[i] + V[i];
  }
  // the thrust's adjoint: w_i . r(q_i) summed (the factors hold 1/m, not F/m)
  auto r_dot = [](const float* w, const float* z) {
    float rx, ry, rz;
    r_e3_half(z[0], z[1], z[2], z[3], rx, ry, rz);
    return w[0] * rx + w[1] * ry + w[2] * rz;
  };
  s.gF = r_dot(w1, q) + r_dot(w2, q2) + r_dot(w2, q3) + r_dot(V, q4);
  float g1[4], g2[4], g3[4], g4[4], gq[4];
  r_vjp(q, w1, g1);
  r_vjp(q2, w2, g2);
  r_vjp(q3, w2, g3);
  r_vjp(q4, V, g4);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    g1[i] *= u.x;
    g2[i] *= u.x;
    g3[i] *= u.x;
    g4[i] *= u.x;
    s.ga[i] = hb * (g2[i] + g3[i]) + h4 * g4[i];
    gq[i] = g1[i] + g2[i] + c3 * g3[i] + c4 * g4[i];
  }
  s.ghh = -0.25f * (dot4(g3, q) + h * dot4(g4, a)) - 0.5f * dot4(g4, q);
  // through a = q (x) [0, w/2]: ga (x) [0, -w/2]
  float at[4];
  step_a(s.ga, make_float4(0.f, -u.y, -u.z, -u.w), h, at);
#pragma unroll
  for (int i = 0; i < 4; ++i) gq[i] += at[i];
  return vec_mul_conj(gq, q);
}

// dS/du of the step from the translation's part s and tau of its end state.
__device__ __forceinline__ float4 step_adjoint_controls(const float* q, float4 u, const DynParams& dp,
                                                        const StepAdjoint& s, float3 tau) {
  const float h = dp.dt;
  float a[4], y[4];
  const float hh = step_a(q, u, h, a);
  const float cq = 1.0f - 0.5f * hh + hh * hh * (1.0f / 24.0f);
  const float ca = h * (1.0f - hh * (1.0f / 6.0f));
#pragma unroll
  for (int i = 0; i < 4; ++i) y[i] = cq * q[i] + ca * a[i];
  // the adjoint of y: (tau (x) q_{k+1}) / |y|, q_{k+1} = y / |y|
  const float inv2 = __frcp_rn(dot4(y, y));
  const float tx = tau.x * inv2, ty = tau.y * inv2, tz = tau.z * inv2;
  const float l[4] = {-tx * y[1] - ty * y[2] - tz * y[3], tx * y[0] + ty * y[3] - tz * y[2],
                      -tx * y[3] + ty * y[0] + tz * y[1], tx * y[2] - ty * y[1] + tz * y[0]};
  const float ghh = s.ghh + (hh * (1.0f / 12.0f) - 0.5f) * dot4(l, q) - h * (1.0f / 6.0f) * dot4(l, a);
  float g[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) g[i] = s.ga[i] + ca * l[i];
  // w_c = 2 (w/2)_c; hh = h^2 |w/2|^2
  const float k = 0.5f * h * h * ghh;
  return make_float4(s.gF,
                     0.5f * (-g[0] * q[1] + g[1] * q[0] + g[2] * q[3] - g[3] * q[2]) + k * u.y,
                     0.5f * (-g[0] * q[2] - g[1] * q[3] + g[2] * q[0] + g[3] * q[1]) + k * u.z,
                     0.5f * (-g[0] * q[3] + g[1] * q[2] - g[2] * q[1] + g[3] * q[0]) + k * u.w);
}

// The control terms' part of dS/du_t added to a: Q_c |u_t|^2 (t <= T-2) and
// Q_cd |u_t - u_{t-1}|^2 (1 <= t <= T-2).
__device__ __forceinline__ float4 control_terms_grad(float4 a, const float4* u, int t, int T,
                                                     const CostParams& cp) {
  const float4 ut = u[t];
  if (t <= T - 2) {
    a.x += 2.0f * cp.Q_c * ut.x; a.y += 2.0f * cp.Q_c * ut.y;
    a.z += 2.0f * cp.Q_c * ut.z; a.w += 2.0f * cp.Q_c * ut.w;
  }
  if (t >= 1 && t <= T - 2) {
    const float4 b = u[t - 1];
    a.x += 2.0f * cp.Q_cd * (ut.x - b.x); a.y += 2.0f * cp.Q_cd * (ut.y - b.y);
    a.z += 2.0f * cp.Q_cd * (ut.z - b.z); a.w += 2.0f * cp.Q_cd * (ut.w - b.w);
  }
  if (t + 1 <= T - 2) {
    const float4 c = u[t + 1];
    a.x -= 2.0f * cp.Q_cd * (c.x - ut.x); a.y -= 2.0f * cp.Q_cd * (c.y - ut.y);
    a.z -= 2.0f * cp.Q_cd * (c.z - ut.z); a.w -= 2.0f * cp.Q_cd * (c.w - ut.w);
  }
  return a;
}

// ---------------------------------------------------------------------------
// Cost and gradient of one sequence by one warp.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float3 add3(float3 a, float3 b) {
  return make_float3(a.x + b.x, a.y + b.y, a.z + b.z);
}

__device__ __forceinline__ float3 shfl3(float3 v, int src) {
  return make_float3(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src),
                     __shfl_sync(0xffffffffu, v.z, src));
}

// Inclusive sums over the lanes up to this one (kUp) or from this one on.
template <bool kUp>
__device__ __forceinline__ float3 warp_scan3(float3 x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float a = kUp ? __shfl_up_sync(0xffffffffu, x.x, o) : __shfl_down_sync(0xffffffffu, x.x, o);
    const float b = kUp ? __shfl_up_sync(0xffffffffu, x.y, o) : __shfl_down_sync(0xffffffffu, x.y, o);
    const float c = kUp ? __shfl_up_sync(0xffffffffu, x.z, o) : __shfl_down_sync(0xffffffffu, x.z, o);
    if (kUp ? lane >= o : lane + o < 32) x = make_float3(x.x + a, x.y + b, x.z + c);
  }
  return x;
}

// The value of the lane before (kUp) or after this one; `edge` at the end.
template <bool kUp>
__device__ __forceinline__ float3 warp_next3(float3 x, float3 edge, int lane) {
  const float a = kUp ? __shfl_up_sync(0xffffffffu, x.x, 1) : __shfl_down_sync(0xffffffffu, x.x, 1);
  const float b = kUp ? __shfl_up_sync(0xffffffffu, x.y, 1) : __shfl_down_sync(0xffffffffu, x.y, 1);
  const float c = kUp ? __shfl_up_sync(0xffffffffu, x.z, 1) : __shfl_down_sync(0xffffffffu, x.z, 1);
  return lane == (kUp ? 0 : 31) ? edge : make_float3(a, b, c);
}

// Nearest collision point of every lane's query (all 32 lanes call it): the
// squared distance into d2 (d_max^2 when none is closer) and the point.  Lists
// of at most kOwnList entries are scanned by their own lane, longer ones by the
// whole warp in turn.  Among equidistant points the one of lowest item index
// wins (the collision set's order, as the oracle breaks ties), whatever the
// order of the entries in the cell's list.
constexpr int kOwnList = 8;

__device__ __forceinline__ void warp_nearest(const GridView& g, int2 r, float px, float py, float pz,
                                             float dmax2, int lane, float& d2_out, float4& near) {
  float best = dmax2;
  int bitem = 0x7fffffff;
  float4 bp = make_float4(0.f, 0.f, 0.f, 0.f);
  auto visit = [&](int e, float qx, float qy, float qz) {
    const float4 p = grid_point(g, e);
    const float d2 = dist2_to(p, qx, qy, qz);
    const int item = point_item(p);
    if (d2 < best || (d2 == best && d2 < dmax2 && item < bitem)) {
      best = d2;
      bitem = item;
      bp = p;
    }
  };
  const bool lng = r.y > kOwnList;
  unsigned pend = __ballot_sync(0xffffffffu, lng);
  while (pend) {
    const int L = __ffs(pend) - 1;
    pend &= pend - 1;
    const int first = __shfl_sync(0xffffffffu, r.x, L), n = __shfl_sync(0xffffffffu, r.y, L);
    const float qx = __shfl_sync(0xffffffffu, px, L), qy = __shfl_sync(0xffffffffu, py, L),
                qz = __shfl_sync(0xffffffffu, pz, L);
    // the lanes' own results wait in registers while they work for lane L
    const float kb = best;
    const int ki = bitem;
    const float4 kp = bp;
    best = dmax2;
    bitem = 0x7fffffff;
    bp = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = lane; i < n; i += 32) visit(first + i, qx, qy, qz);
    const unsigned bits = __float_as_uint(best);  // non-negative: ordered as its bits
    const unsigned m = __reduce_min_sync(0xffffffffu, bits);
    const unsigned mi = __reduce_min_sync(0xffffffffu, bits == m ? (unsigned)bitem : 0x7fffffffu);
    const int src = __ffs(__ballot_sync(0xffffffffu, bits == m && (unsigned)bitem == mi)) - 1;
    const float4 p = make_float4(__shfl_sync(0xffffffffu, bp.x, src), __shfl_sync(0xffffffffu, bp.y, src),
                                 __shfl_sync(0xffffffffu, bp.z, src), 0.f);
    best = lane == L ? __uint_as_float(m) : kb;
    bitem = lane == L ? (int)mi : ki;
    bp = lane == L ? p : kp;
  }
  if (!lng)
    for (int i = 0; i < r.y; ++i) visit(r.x + i, px, py, pz);
  d2_out = best;
  near = bp;
}

// Scratch of one warp in shared memory (floats), for horizon T: the controls T x 4,
// the attitudes q_0 .. q_T and, per step, the state-term gradients gp, gv
// and the attitude terms' part of tau.
__host__ __device__ constexpr size_t cost_grad_words(int T) { return 4 * (size_t)T + 4 * (size_t)(T + 1) + 9 * (size_t)T + 3 & ~(size_t)3; }

// S(1) of the noise-free rollout of U (global, T entries) from x0 and, with
// kGrad, dS/dU into G (global).  guide: T x 3 (global).  Called by all 32 lanes
// of one warp; returns S on every lane.
//
// 32 steps at a time, one per lane: the scans above with the last lane's
// state (forward) or the first lane's adjoints (backward) carried to the
// next 32.  A sequence of 40 steps with its gradient takes two rounds each way
// instead of 40 dependent RK4 steps forward and 40 again with their reverse
// sweeps backward, which every lane computed alike: 2048 such sequences
// 90.7 -> 14.8 us (bound by the latency of the scans' shuffles and of the
// candidate lists).
template <bool kGrad>
__device__ float warp_cost_grad(const float4* __restrict__ U, float4* __restrict__ G, const float* guide,
                                int T, const float* x0, const DynParams& dp, const CostParams& cp,
                                const GridView& grid, float* scratch, int lane) {
  const float dmax2 = cp.d_max * cp.d_max;
  const float h = dp.dt;
  float4* const su = reinterpret_cast<float4*>(scratch);
  float4* const sq = su + T;
  float* const sg = reinterpret_cast<float*>(sq + T + 1);  // [9][T]
  for (int t = lane; t < T; t += 32) su[t] = __ldg(U + t);
  float4 qc = make_float4(x0[3], x0[4], x0[5], x0[6]);  // the round's first state
  float3 pc = make_float3(x0[0], x0[1], x0[2]), vc = make_float3(x0[7], x0[8], x0[9]);
  if (kGrad && lane == 0) sq[0] = qc;
  __syncwarp();
  const int rounds = (T + 31) / 32;
  float S = 0.0f;
  for (int r = 0; r < rounds; ++r) {
    const int j = 32 * r + lane;
    const bool on = j < T;
    const float4 u = on ? su[j] : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 m = on ? attitude_factor(u, dp) : make_float4(1.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float4 y = shfl_up4(m, o);
      if (lane >= o) m = quat_mul4(y, m);
    }
    float4 q1 = quat_mul4(qc, m);
    const float inv = rsqrtf(q1.x * q1.x + q1.y * q1.y + q1.z * q1.z + q1.w * q1.w);
    q1 = make_float4(q1.x * inv, q1.y * inv, q1.z * inv, q1.w * inv);
    float4 q = shfl_up4(q1, 1);
    if (lane == 0) q = qc;
    const float qj[4] = {q.x, q.y, q.z, q.w};
    float inc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (on) rk4_translation_increments(qj, u, dp, inc);
    const float3 v1 = add3(vc, warp_scan3<true>(make_float3(inc[3], inc[4], inc[5]), lane));
    const float3 vj = warp_next3<true>(v1, vc, lane);
    const float3 p1 = add3(pc, warp_scan3<true>(make_float3(h * vj.x + inc[0], h * vj.y + inc[1],
                                                            h * vj.z + inc[2]), lane));
    float d2;
    float4 near;
    warp_nearest(grid, on ? cell_range(p1.x, p1.y, p1.z, grid) : make_int2(0, 0), p1.x, p1.y, p1.z,
                 dmax2, lane, d2, near);
    if (on) {
      State x;
      x.p[0] = p1.x; x.p[1] = p1.y; x.p[2] = p1.z;
      x.q[0] = q1.x; x.q[1] = q1.y; x.q[2] = q1.z; x.q[3] = q1.w;
      x.v[0] = v1.x; x.v[1] = v1.y; x.v[2] = v1.z;
      float gs[10];
      S += state_terms<kGrad>(x, guide[3 * j], guide[3 * j + 1], guide[3 * j + 2], d2, near, cp, dmax2, gs);
      if (kGrad) {
        sq[j + 1] = q1;
        const float3 t = vec_mul_conj(gs + 3, x.q);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          sg[i * T + j] = gs[i];
          sg[(3 + i) * T + j] = gs[7 + i];
        }
        sg[6 * T + j] = t.x;
        sg[7 * T + j] = t.y;
        sg[8 * T + j] = t.z;
      }
      // J_ctrl: Q_c |u_j|^2 (j <= T-2) and Q_cd |u_j - u_{j-1}|^2 (1 <= j <= T-2)
      if (j <= T - 2) {
        S += cp.Q_c * (u.x * u.x + u.y * u.y + u.z * u.z + u.w * u.w);
        if (j >= 1) {
          const float4 b = su[j - 1];
          const float dx = u.x - b.x, dy = u.y - b.y, dz = u.z - b.z, dw = u.w - b.w;
          S += cp.Q_cd * (dx * dx + dy * dy + dz * dz + dw * dw);
        }
      }
    }
    if (r + 1 < rounds) {
      qc = make_float4(__shfl_sync(0xffffffffu, q1.x, 31), __shfl_sync(0xffffffffu, q1.y, 31),
                       __shfl_sync(0xffffffffu, q1.z, 31), __shfl_sync(0xffffffffu, q1.w, 31));
      vc = shfl3(v1, 31);
      pc = shfl3(p1, 31);
    }
  }
  S = warp_sum(S);
  if constexpr (kGrad) {
    __syncwarp();
    const float3 zero = make_float3(0.f, 0.f, 0.f);
    float3 cp_p = zero, cp_v = zero, cp_t = zero;  // the later rounds' sums
    for (int r = rounds - 1; r >= 0; --r) {
      const int k = 32 * r + lane;
      const bool on = k < T;
      float3 gp = zero, gv = zero, tg = zero;
      float4 u = make_float4(0.f, 0.f, 0.f, 0.f), q4 = make_float4(1.f, 0.f, 0.f, 0.f);
      if (on) {
        gp = make_float3(sg[k], sg[T + k], sg[2 * T + k]);
        gv = make_float3(sg[3 * T + k], sg[4 * T + k], sg[5 * T + k]);
        tg = make_float3(sg[6 * T + k], sg[7 * T + k], sg[8 * T + k]);
        u = su[k];
        q4 = sq[k];
      }
      const float q[4] = {q4.x, q4.y, q4.z, q4.w};
      const float3 lp = add3(warp_scan3<false>(gp, lane), cp_p);  // Lp_{k+1}
      const float3 lp2 = warp_next3<false>(lp, cp_p, lane);       // Lp_{k+2}
      const float3 lv = add3(warp_scan3<false>(make_float3(gv.x + h * lp2.x, gv.y + h * lp2.y,
                                                           gv.z + h * lp2.z), lane), cp_v);
      StepAdjoint sa;
      float3 bt = step_adjoint_translation(q, u, dp, lp, lv, sa);
      if (!on) bt = zero;
      const float3 ts = add3(warp_scan3<false>(add3(tg, bt), lane), cp_t);  // tau_k without tg_{k-1}
      const float3 tau = add3(warp_next3<false>(ts, cp_t, lane), tg);       // tau_{k+1}
      if (on) G[k] = control_terms_grad(step_adjoint_controls(q, u, dp, sa, tau), su, k, T, cp);
      if (r > 0) {
        cp_p = shfl3(lp, 0);
        cp_v = shfl3(lv, 0);
        cp_t = shfl3(ts, 0);
      }
    }
  }
  return S;
}

// ---------------------------------------------------------------------------
// The RK4 step's stages and their reverse sweep (the refinement).
// ---------------------------------------------------------------------------
// xd = f(x, u) of the quadrotor model (Eq. dynamics) at a stage state.
__device__ __forceinline__ void dyn_f(const float* x, float4 u, const DynParams& dp, float* xd) {
  const float qw = x[3], qx = x[4], qy = x[5], qz = x[6];
  xd[0] = x[7]; xd[1] = x[8]; xd[2] = x[9];
  xd[3] = 0.5f * (-qx * u.y - qy * u.z - qz * u.w);
  xd[4] = 0.5f * (qw * u.y + qy * u.w - qz * u.z);
  xd[5] = 0.5f * (qw * u.z - qx * u.w + qz * u.y);
  xd[6] = 0.5f * (qw * u.w + qx * u.z - qy * u.y);
  float rx, ry, rz;
  r_e3(qw, qx, qy, qz, rx, ry, rz);
  const float f = u.x * dp.inv_mass;
  xd[7] = f * rx; xd[8] = f * ry; xd[9] = f * rz - dp.g;
}

// w^T df/dx added to gx, w^T df/du added to gu, at stage state x.
__device__ __forceinline__ void dyn_vjp(const float* x, float4 u, const DynParams& dp,
                                        const float* w, float* gx, float* gu) {
  const float qw = x[3], qx = x[4], qy = x[5], qz = x[6];
  const float ox = u.y, oy = u.z, oz = u.w;
  gx[7] += w[0]; gx[8] += w[1]; gx[9] += w[2];
  const float W0 = 0.5f * w[3], W1 = 0.5f * w[4], W2 = 0.5f * w[5], W3 = 0.5f * w[6];
  gx[3] += W1 * ox + W2 * oy + W3 * oz;
  gx[4] += -W0 * ox - W2 * oz + W3 * oy;
  gx[5] += -W0 * oy + W1 * oz - W3 * ox;
  gx[6] += -W0 * oz - W1 * oy + W2 * ox;
  gu[1] += -W0 * qx + W1 * qw + W2 * qz - W3 * qy;
  gu[2] += -W0 * qy - W1 * qz + W2 * qw + W3 * qx;
  gu[3] += -W0 * qz + W1 * qy - W2 * qx + W3 * qw;
  const float V0 = w[7], V1 = w[8], V2 = w[9];
  float rx, ry, rz;
  r_e3(qw, qx, qy, qz, rx, ry, rz);
  gu[0] += (V0 * rx + V1 * ry + V2 * rz) * dp.inv_mass;
  const float s = u.x * dp.inv_mass;
  gx[3] += s * (2.0f * qy * V0 - 2.0f * qx * V1);
  gx[4] += s * (2.0f * qz * V0 - 2.0f * qw * V1 - 4.0f * qx * V2);
  gx[5] += s * (2.0f * qw * V0 + 2.0f * qz * V1 - 4.0f * qy * V2);
  gx[6] += s * (2.0f * qx * V0 + 2.0f * qy * V1);
}

// The stage states of one RK4 step from x with control u (Eq. dynamics):
// t2 = x + h/2 k1, t3 = x + h/2 k2, t4 = x + h k3, and the quaternion before
// renormalisation y = q + h/6 (k1 + 2 k2 + 2 k3 + k4) (quaternion part).
__device__ __forceinline__ void rk4_stages(const float* x, float4 u, const DynParams& dp, float* t2,
                                           float* t3, float* t4, float* y) {
  const float h = dp.dt;
  float k1[10], k2[10], k3[10], k4[10];
  dyn_f(x, u, dp, k1);
#pragma unroll
  for (int i = 0; i < 10; ++i) t2[i] = x[i] + 0.5f * h * k1[i];
  dyn_f(t2, u, dp, k2);
#pragma unroll
  for (int i = 0; i < 10; ++i) t3[i] = x[i] + 0.5f * h * k2[i];
  dyn_f(t3, u, dp, k3);
#pragma unroll
  for (int i = 0; i < 10; ++i) t4[i] = x[i] + h * k3[i];
  dyn_f(t4, u, dp, k4);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    y[i] = x[3 + i] + h * (1.0f / 6.0f) * (k1[3 + i] + 2.0f * k2[3 + i] + 2.0f * k3[3 + i] + k4[3 + i]);
}

// Reverse of one RK4 step given its stage states: lam holds dS/dx_{j+1} on
// entry and dS/dx_j on return; gu gets dS/du_j from the dynamics.  Through the
// renormalisation q+ = y/|y| (projection (I - q+ q+^T)/|y|), then the four
// stages in reverse.
__device__ __forceinline__ void rk4_vjp_stages(const float* x, const float* t2, const float* t3,
                                               const float* t4, const float* y, float4 u,
                                               const DynParams& dp, float* lam, float* gu) {
  const float h = dp.dt;
  const float inv = rsqrtf(y[0] * y[0] + y[1] * y[1] + y[2] * y[2] + y[3] * y[3]);
  const float dot = (y[0] * lam[3] + y[1] * lam[4] + y[2] * lam[5] + y[3] * lam[6]) * inv;
  float ly[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) ly[i] = lam[i];
#pragma unroll
  for (int i = 0; i < 4; ++i) ly[3 + i] = (lam[3 + i] - y[i] * inv * dot) * inv;
  float l1[10], l2[10], l3[10], l4[10], lt[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    lam[i] = ly[i];
    l1[i] = h * (1.0f / 6.0f) * ly[i];
    l2[i] = h * (1.0f / 3.0f) * ly[i];
    l3[i] = l2[i];
    l4[i] = l1[i];
  }
#pragma unroll
  for (int i = 0; i < 10; ++i) lt[i] = 0.0f;
  dyn_vjp(t4, u, dp, l4, lt, gu);
#pragma unroll
  for (int i = 0; i < 10; ++i) { lam[i] += lt[i]; l3[i] += h * lt[i]; lt[i] = 0.0f; }
  dyn_vjp(t3, u, dp, l3, lt, gu);
#pragma unroll
  for (int i = 0; i < 10; ++i) { lam[i] += lt[i]; l2[i] += 0.5f * h * lt[i]; lt[i] = 0.0f; }
  dyn_vjp(t2, u, dp, l2, lt, gu);
#pragma unroll
  for (int i = 0; i < 10; ++i) { lam[i] += lt[i]; l1[i] += 0.5f * h * lt[i]; }
  dyn_vjp(x, u, dp, l1, lam, gu);
}

// ---------------------------------------------------------------------------
// Gradient refinement by a whole CTA (the update kernels): the forward
// states by scans over the steps (rollout_by_scans); the backward pass split
// by dependence (suffix sums for the position and velocity adjoints, the 4x4
// attitude recurrence as a scan of affine maps over four warps, the vector-Jacobian
// products of every step in parallel); everything else over the CTA: the stage states of every
// step, the nearest point of every
// state (candidate lists cut into items of kRefItem entries; a 64-bit atomic
// minimum of (squared distance bits, item index) keeps the lowest item among
// equidistant points, the collision set's order), the state terms and their
// gradients, the control terms and the clamped step.  It keeps the stages' reverse
// sweep and the affine attitude recurrence, not warp_cost_grad's sums: five steps
// of 0.05 on gradients of up to 1e6 magnify a change of rounding (the refined nominals
// moved by up to 1e-5 of their norm, past their error against 64 bits on some
// inputs) and the sums saved 10 us of 74.
// ---------------------------------------------------------------------------
constexpr int kRefItem = 8;

struct RefineScratch {
  float4* tot;               // warps: scan totals of the forward rollout
  float4* g;                 // T: dS/du
  unsigned long long* key;   // T: (bits(d2) << 32) | item of the nearest point of x_{j+1}
  int2* qrange;              // T: candidate range of each listed query
  int2* scan;                // warps: block-scan totals
  float* xs;                 // (T + 1) x 10: states x_0 .. x_T
  float* st;                 // T x 34: stage states t2, t3, t4 and y of step j
  float* gs;                 // T x 10: state-term gradients at x_{j+1}
  int* qitem;                // T + 1: first item of each listed query
  int* qslot;                // T: step of each listed query
  float* afm;                // 4 x 20: the attitude adjoint scan's warp compositions
};

__host__ __device__ constexpr size_t refine_smem_bytes(int T, int warps) {
  return 16 * (size_t)warps + 16 * (size_t)T + 8 * (size_t)T + 8 * (size_t)T + 8 * (size_t)warps +
         4 * (size_t)(T + 1) * 10 + 4 * (size_t)T * 34 + 4 * (size_t)T * 10 + 4 * (size_t)(T + 1) +
         4 * (size_t)T + 4 * 80;
}

__device__ __forceinline__ RefineScratch refine_layout(unsigned char* base, int T, int warps) {
  RefineScratch r;
  r.tot = reinterpret_cast<float4*>(base);
  r.g = r.tot + warps;
  r.key = reinterpret_cast<unsigned long long*>(r.g + T);
  r.qrange = reinterpret_cast<int2*>(r.key + T);
  r.scan = r.qrange + T;
  r.xs = reinterpret_cast<float*>(r.scan + warps);
  r.st = r.xs + (size_t)(T + 1) * 10;
  r.gs = r.st + (size_t)T * 34;
  r.qitem = reinterpret_cast<int*>(r.gs + (size_t)T * 10);
  r.qslot = r.qitem + T + 1;
  r.afm = reinterpret_cast<float*>(r.qslot + T);
  return r;
}


// `steps` clamped gradient steps u <- clamp(u - alpha dS/du) on the nominal u
// (shared, T <= kThreads entries), by all kThreads threads of the CTA.
// kEither: the grid's entries may be the points themselves (grid_point).
template <int kThreads, bool kEither>
__device__ void block_refine(float4* u, const float* guide, int T, const float* x0,
                             const DynParams& dp, const CostParams& cp, const GridView& grid,
                             const float* umin, const float* umax, int steps, float alpha,
                             const RefineScratch& rs) {
  const int tid = threadIdx.x;
  const float dmax2 = cp.d_max * cp.d_max;
  const unsigned long long none =
      ((unsigned long long)__float_as_uint(dmax2) << 32) | 0xffffffffull;
  for (int r = 0; r < steps; ++r) {
    // forward: the states x_0 .. x_T, by scans over the steps
    rollout_by_scans<kThreads / 32>(u, T, x0, dp, rs.xs, rs.tot);
    // step tid: its stage states and the candidate range of x_{tid+1}
    int2 rg = make_int2(0, 0);
    if (tid < T) {
      float* stj = rs.st + (size_t)tid * 34;
      rk4_stages(rs.xs + tid * 10, u[tid], dp, stj, stj + 10, stj + 20, stj + 30);
      rs.key[tid] = none;
      const float* x1 = rs.xs + (tid + 1) * 10;
      rg = cell_range(x1[0], x1[1], x1[2], grid);
    }
    int2 total;
    const int2 off = block_scan2<kThreads / 32>(
        rg.y > 0 ? make_int2(1, (rg.y + kRefItem - 1) / kRefItem) : make_int2(0, 0), rs.scan, total);
    if (rg.y > 0) {
      rs.qitem[off.x] = off.y;
      rs.qrange[off.x] = rg;
      rs.qslot[off.x] = tid;
    }
    __syncthreads();
    // every item of entries of a listed query: its (squared distance, item index)
    // pair of lowest (distance, item) into the query's minimum
    for (int it = tid; it < total.y; it += kThreads) {
      const int lo = item_owner(rs.qitem, total.x, it);
      const int2 q = rs.qrange[lo];
      const int j = rs.qslot[lo];
      const int first = (it - rs.qitem[lo]) * kRefItem;
      const int n = q.y - first < kRefItem ? q.y - first : kRefItem;
      if (!AERO_CHECK(j < T && first >= 0 && n > 0 && q.x >= 0, kChkQuery)) continue;
      const float* x1 = rs.xs + (j + 1) * 10;
      float best = dmax2;
      int bitem = -1;
      for (int c = 0; c < n; ++c) {
        const float4 p = grid_point<kEither>(grid, q.x + first + c);
        const float d2 = dist2_to(p, x1[0], x1[1], x1[2]);
        const int item = point_item(p);
        if (d2 < best || (d2 == best && bitem >= 0 && item < bitem)) {
          best = d2;
          bitem = item;
        }
      }
      if (bitem >= 0)
        atomicMin(rs.key + j, ((unsigned long long)__float_as_uint(best) << 32) | (unsigned)bitem);
    }
    __syncthreads();
    // state-term gradients at x_{tid+1}
    if (tid < T) {
      const unsigned long long kk = rs.key[tid];
      const float d2 = __uint_as_float((unsigned)(kk >> 32));
      const unsigned bi = (unsigned)kk;
      const float4 nearest = bi == 0xffffffffu ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldg(grid.pts + bi);
      state_terms<true>(state_load(rs.xs + (tid + 1) * 10), guide[3 * tid], guide[3 * tid + 1],
                        guide[3 * tid + 2], d2, nearest, cp, dmax2, rs.gs + tid * 10);
    }
    __syncthreads();
    // backward.  With L_{k+1} = dS/dx_{k+1} (the state terms at x_{k+1} plus
    // what flows back from later steps), L_{k+1} = gs[k] + J_{k+1}^T L_{k+2},
    // J the step Jacobian.  Positions feed only positions and velocities only
    // positions and velocities, so the position and velocity parts are
    // suffix sums: Lp_{k+1} = sum_{i >= k} gs_p[i], Lv_{k+1} = sum_{i >= k}
    // (gs_v[i] + h Lp_{i+2}).  The attitude part is the linear recurrence
    // Lq_{k+1} = gs_q[k] + b_{k+1} + A_{k+1}^T Lq_{k+2}: b the attitude part of
    // J^T (Lp, 0, Lv) (the step's vector-Jacobian product, in parallel), A the
    // 4x4 attitude Jacobian, whose transpose is applied in closed form: the
    // unnormalised y = q (x) m, so A^T l = ((l - yh (yh . l)) / |y|) (x) conj(m),
    // yh = y / |y|; its affine maps are composed by a scan.  Then every step's dS/du_k
    // is the control part of J_k^T L_{k+1}, in parallel.
    {
      const float h = dp.dt;
      // (a) the suffix sums, thread t taking step k = T - 1 - t
      const int k = T - 1 - tid;
      const bool on = tid < T;
      const float* g = rs.gs + (on ? k : 0) * 10;
      const float3 gp = on ? make_float3(g[0], g[1], g[2]) : make_float3(0.f, 0.f, 0.f);
      const float3 gv = on ? make_float3(g[7], g[8], g[9]) : make_float3(0.f, 0.f, 0.f);
      const float3 lp = block_sum_scan3<kThreads / 32>(gp, rs.tot);
      const float3 lp2 = make_float3(lp.x - gp.x, lp.y - gp.y, lp.z - gp.z);  // Lp_{k+2}
      const float3 lv = block_sum_scan3<kThreads / 32>(
          make_float3(gv.x + h * lp2.x, gv.y + h * lp2.y, gv.z + h * lp2.z), rs.tot);
      if (on) {
        float* L = rs.gs + k * 10;
        L[0] = lp.x; L[1] = lp.y; L[2] = lp.z;
        L[7] = lv.x; L[8] = lv.y; L[9] = lv.z;
      }
      __syncthreads();
      // (b) b_k for every step k = tid, into rs.g
      if (tid < T) {
        const float* L = rs.gs + tid * 10;
        float lam[10] = {L[0], L[1], L[2], 0.f, 0.f, 0.f, 0.f, L[7], L[8], L[9]};
        float gu[4] = {0.f, 0.f, 0.f, 0.f};
        const float* stk = rs.st + (size_t)tid * 34;
        rk4_vjp_stages(rs.xs + tid * 10, stk, stk + 10, stk + 20, stk + 30, u[tid], dp, lam, gu);
        rs.g[tid] = make_float4(lam[3], lam[4], lam[5], lam[6]);
      }
      __syncthreads();
      // (c) the attitude recurrence Lq_k = C_k + A_{k+1}^T Lq_{k+1} (k = T-2
      // .. 0; C_k = gs_q[k] + b_{k+1}; Lq_{T-1} = gs_q[T-1]) is affine in Lq:
      // thread t = T-2-k holds the map x -> C_k + M x (M = A_{k+1}^T as a 4x4
      // matrix, its columns the images of the unit vectors), and an inclusive
      // scan composes the maps, later ones outside, so that thread t ends with
      // the composition that takes Lq_{T-1} to Lq_k.  T - 1 <= 127 maps: up to
      // four warps, each carrying the earlier warps' compositions.
      static_assert(kMaxT - 1 <= 128 && kThreads >= 128, "the attitude adjoint scan spans four warps");
      {
        const int kk = T - 2 - tid, wid = tid >> 5;
        const bool on = kk >= 0;
        float M[16], c[4];
#pragma unroll
        for (int i = 0; i < 16; ++i) M[i] = (i % 5 == 0) ? 1.0f : 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) c[i] = 0.0f;
        if (on) {
          const int j = kk + 1;  // A_j: the attitude Jacobian of step j
          const float* y = rs.st + (size_t)j * 34 + 30;
          const float inv = rsqrtf(y[0] * y[0] + y[1] * y[1] + y[2] * y[2] + y[3] * y[3]);
          const float4 m = rk4_attitude_coefs(u[j], dp);
          const float4 mc = make_float4(m.x, -m.y, -m.z, -m.w);
#pragma unroll
          for (int col = 0; col < 4; ++col) {
            // A_j^T e_col = ((e_col - yh (yh . e_col)) / |y|) (x) conj(m)
            const float d = y[col] * inv * inv;
            const float4 pl = make_float4(((col == 0 ? 1.f : 0.f) - y[0] * d) * inv,
                                          ((col == 1 ? 1.f : 0.f) - y[1] * d) * inv,
                                          ((col == 2 ? 1.f : 0.f) - y[2] * d) * inv,
                                          ((col == 3 ? 1.f : 0.f) - y[3] * d) * inv);
            const float4 at = quat_mul4(pl, mc);
            M[col] = at.x;
            M[4 + col] = at.y;
            M[8 + col] = at.z;
            M[12 + col] = at.w;
          }
          const float* Lk = rs.gs + kk * 10 + 3;
          const float4 b = rs.g[j];
          c[0] = Lk[0] + b.x;
          c[1] = Lk[1] + b.y;
          c[2] = Lk[2] + b.z;
          c[3] = Lk[3] + b.w;
        }
        // (M, c) o (M', c') = (M M', M c' + c)
        auto compose = [&](const float* M2, const float* c2) {
          float R[16], r[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              R[4 * i + q] = M[4 * i] * M2[q] + M[4 * i + 1] * M2[4 + q] + M[4 * i + 2] * M2[8 + q] +
                             M[4 * i + 3] * M2[12 + q];
            r[i] = M[4 * i] * c2[0] + M[4 * i + 1] * c2[1] + M[4 * i + 2] * c2[2] +
                   M[4 * i + 3] * c2[3] + c[i];
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) M[i] = R[i];
#pragma unroll
          for (int i = 0; i < 4; ++i) c[i] = r[i];
        };
        if (wid < 4) {
          const int lane = tid & 31;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            float M2[16], c2[4];
#pragma unroll
            for (int i = 0; i < 16; ++i) M2[i] = __shfl_up_sync(0xffffffffu, M[i], o);
#pragma unroll
            for (int i = 0; i < 4; ++i) c2[i] = __shfl_up_sync(0xffffffffu, c[i], o);
            if (lane >= o) compose(M2, c2);
          }
          if (lane == 31) {
#pragma unroll
            for (int i = 0; i < 16; ++i) rs.afm[20 * wid + i] = M[i];
#pragma unroll
            for (int i = 0; i < 4; ++i) rs.afm[20 * wid + 16 + i] = c[i];
          }
        }
        __syncthreads();
        if (on) {
          // the earlier warps' compositions, the latest one first (inside)
          for (int v = wid - 1; v >= 0; --v) {
            float M2[16], c2[4];
#pragma unroll
            for (int i = 0; i < 16; ++i) M2[i] = rs.afm[20 * v + i];
#pragma unroll
            for (int i = 0; i < 4; ++i) c2[i] = rs.afm[20 * v + 16 + i];
            compose(M2, c2);
          }
        }
        if (on) {
          const float* L = rs.gs + (T - 1) * 10 + 3;  // Lq_{T-1}
          const float l0 = L[0], l1 = L[1], l2 = L[2], l3 = L[3];
          float* Lk = rs.gs + kk * 10 + 3;
          float lo[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            lo[i] = M[4 * i] * l0 + M[4 * i + 1] * l1 + M[4 * i + 2] * l2 + M[4 * i + 3] * l3 + c[i];
#pragma unroll
          for (int i = 0; i < 4; ++i) Lk[i] = lo[i];
        }
      }
      __syncthreads();
      // (d) dS/du_k = the control part of J_k^T L_{k+1}
      if (tid < T) {
        float lam[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) lam[i] = rs.gs[tid * 10 + i];
        float gu[4] = {0.f, 0.f, 0.f, 0.f};
        const float* stk = rs.st + (size_t)tid * 34;
        rk4_vjp_stages(rs.xs + tid * 10, stk, stk + 10, stk + 20, stk + 30, u[tid], dp, lam, gu);
        rs.g[tid] = make_float4(gu[0], gu[1], gu[2], gu[3]);
      }
    }
    __syncthreads();
    // control terms, then the clamped step
    if (tid < T) rs.g[tid] = control_terms_grad(rs.g[tid], u, tid, T, cp);
    __syncthreads();
    if (tid < T) {
      const float4 a = u[tid], d = rs.g[tid];
      u[tid] = make_float4(fminf(fmaxf(a.x - alpha * d.x, umin[0]), umax[0]),
                           fminf(fmaxf(a.y - alpha * d.y, umin[1]), umax[1]),
                           fminf(fmaxf(a.z - alpha * d.z, umin[2]), umax[2]),
                           fminf(fmaxf(a.w - alpha * d.w, umin[3]), umax[3]));
    }
    __syncthreads();
  }
}

}  // namespace aero

