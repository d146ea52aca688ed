// Per-path adjoint in 3D, shared by the dense adjoint and the batched descent.
#pragma once

#include "drt_path3.cuh"

namespace drt {

// ------------------------------------------------------------ TX adjoint
// Reverse mode of path_power3 for the transmitter only (the gradient the antenna
// placement of Sec. VII needs): recompute the path, sweep the triangles once for
// each leg's visibility as (product of the non-zero factors, number of zero
// factors), then once more pushing each factor's adjoint into the path vertices;
// the vertex adjoints flow back through the leg lengths, the validity, the
// backtrace and the image chain to the transmitter.  A path with an exactly-zero
// factor has an exactly-zero gradient (a saturated smoothing), as in 2D.
struct LegTri {
  float x, y, X, t, ins, f;
  Smooth3 sx, sy, sd[3];
  float e0[3], e1[3];
};

template <int MODE>
__device__ __forceinline__ bool leg_tri(const float4& P, const float4* M, float3 a, float3 b,
                                        float alpha, LegTri& r) {
  r.x = dot3(P, a) - P.w;
  r.y = dot3(P, b) - P.w;
  r.sx = smooth3<MODE>(r.x, alpha);
  r.sy = smooth3<MODE>(r.y, alpha);
  r.X = fmaf(r.sx.s, r.sy.sb, r.sx.sb * r.sy.s);
  r.t = __fdividef(r.x, r.x - r.y);
  if (!(fabsf(r.t) <= 1e8f)) return false;
  r.ins = 1.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.e0[k] = dot3(M[k], a) - M[k].w;
    r.e1[k] = dot3(M[k], b) - M[k].w;
    r.sd[k] = smooth3<MODE>(fmaf(r.t, r.e1[k] - r.e0[k], r.e0[k]), alpha);
    r.ins *= r.sd[k].s;
  }
  if (MODE == MODE_SIGMOID) {
    // f = 1 - X ins as sums of non-negative terms (s + sb = 1 for each smoothed
    // value): 1 - X = s_x s_y + sb_x sb_y and 1 - ins = sb_0 + s_0 (sb_1 + s_1 sb_2),
    // so f = (1 - X) + X (1 - ins) keeps its relative accuracy where a triangle
    // nearly blocks the leg (1 - X ins there cancels to a few ulps of 1)
    const float omx = fmaf(r.sx.s, r.sy.s, r.sx.sb * r.sy.sb);
    const float omi = fmaf(r.sd[0].s, fmaf(r.sd[1].s, r.sd[2].sb, r.sd[1].sb), r.sd[0].sb);
    r.f = fmaf(r.X, omi, omx);
  } else {
    r.f = fmaf(-r.X, r.ins, 1.f);
  }
  return true;
}

// Per-triangle adjoint slots of the wall gradient (the four records' values):
// P = {n, c} in 0..3, M_k = {m_k, o_k} in 4 + 4k .. 7 + 4k.
constexpr int TRI_SLOTS = 16;

// Sums v[0..15] over the warp by recursive halving: lane l ends with the warp
// total of v[(l >> 1) & 15] (each total held by 2 lanes); 16 shuffles.
__device__ __forceinline__ float warp_reduce_scatter16(const float* v) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
  float a[8], b[4], c[2];
#pragma unroll
  for (int k = 0; k < 8; ++k)
    a[k] = (b4 ? v[k + 8] : v[k]) + __shfl_xor_sync(full, b4 ? v[k] : v[k + 8], 16);
#pragma unroll
  for (int k = 0; k < 4; ++k)
    b[k] = (b3 ? a[k + 4] : a[k]) + __shfl_xor_sync(full, b3 ? a[k] : a[k + 4], 8);
#pragma unroll
  for (int k = 0; k < 2; ++k)
    c[k] = (b2 ? b[k + 2] : b[k]) + __shfl_xor_sync(full, b2 ? b[k] : b[k + 2], 4);
  float d = (b1 ? c[1] : c[0]) + __shfl_xor_sync(full, b1 ? c[0] : c[1], 2);
  return d + __shfl_xor_sync(full, d, 1);
}

// Adds the warp's 16 adjoint slots of triangle w into the CTA table (the
// triangle is the same in every lane).
__device__ __forceinline__ void add_tri_adjoint(float* acc, int w, const float* v) {
  const float t = warp_reduce_scatter16(v);
  const int lane = threadIdx.x & 31;
  if ((lane & 1) == 0) atomicAdd(&acc[w * TRI_SLOTS + ((lane >> 1) & 15)], t);
}

__device__ __forceinline__ void axpy3(float a, float4 v, float3& acc) {
  acc.x = fmaf(a, v.x, acc.x);
  acc.y = fmaf(a, v.y, acc.y);
  acc.z = fmaf(a, v.z, acc.z);
}

// add_tri_adjoint where the triangle differs between the lanes (a batch of queued paths
// holds a few candidates): once per distinct triangle, the other lanes at 0.
__device__ __forceinline__ void add_tri_adjoints(float* acc, int w, const float* v) {
  unsigned todo = 0xffffffffu;
  while (todo) {
    const int wc = __shfl_sync(0xffffffffu, w, __ffs(todo) - 1);
    const bool same = w == wc;
    float x[TRI_SLOTS];
#pragma unroll
    for (int i = 0; i < TRI_SLOTS; ++i) x[i] = same ? v[i] : 0.f;
    add_tri_adjoint(acc, wc, x);
    todo &= ~__ballot_sync(0xffffffffu, same);
  }
}

// Forward values of one path, recomputed for its adjoint.
template <int K>
struct VjpPath3 {
  float3 I[K + 1];
  float dimg[K + 1];   // d = n . I_{j-1} - c of each image step
  float3 Q[K + 2];
  float ta[K + 1], tb[K + 1], tt[K + 1];
  float len[K + 1], L;
  float V[K + 1];
  bool degenerate;
};

template <int MODE, int K>
__device__ __forceinline__ void vjp3_recompute(const SmemTris& s, float3 tx, float3 rx, const Cand& cd,
                                               float alpha, VjpPath3<K>& R) {
  R.degenerate = false;
#pragma unroll
  for (int j = 1; j < K; ++j) R.degenerate |= one_plane(s.P[cd.w[j - 1]], s.P[cd.w[j]]);
  float3* I = R.I;
  float3* Q = R.Q;
  I[0] = tx;
  R.dimg[0] = 0.f;
#pragma unroll
  for (int j = 1; j <= K; ++j) {
    const float4 P = s.P[cd.w[j - 1]];
    R.dimg[j] = dot3(P, I[j - 1]) - P.w;
    const float d2 = 2.f * R.dimg[j];
    I[j] = make_float3(fmaf(-d2, P.x, I[j - 1].x), fmaf(-d2, P.y, I[j - 1].y),
                       fmaf(-d2, P.z, I[j - 1].z));
  }
  Q[0] = tx;
  Q[K + 1] = rx;
#pragma unroll
  for (int j = K; j >= 1; --j) {
    const float4 P = s.P[cd.w[j - 1]];
    R.ta[j] = dot3(P, I[j]) - P.w;
    R.tb[j] = dot3(P, Q[j + 1]) - P.w;
    float t = __fdiv_rn(R.tb[j], R.tb[j] - R.ta[j]);
    if (!(fabsf(t) <= 1e8f)) {
      R.degenerate = true;
      t = 0.f;
    }
    R.tt[j] = t;
    Q[j] = make_float3(fmaf(t, I[j].x - Q[j + 1].x, Q[j + 1].x),
                       fmaf(t, I[j].y - Q[j + 1].y, Q[j + 1].y),
                       fmaf(t, I[j].z - Q[j + 1].z, Q[j + 1].z));
  }
  R.L = 0.f;
#pragma unroll
  for (int j = 0; j <= K; ++j) {
    const float dx = Q[j + 1].x - Q[j].x, dy = Q[j + 1].y - Q[j].y, dz = Q[j + 1].z - Q[j].z;
    const float len2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    R.degenerate |= !(len2 > 0.f);
    R.len[j] = __fsqrt_rn(len2);
    R.L += R.len[j];
  }
  if (R.degenerate) R.L = 1.f;
#pragma unroll
  for (int j = 1; j <= K; ++j) {
    const int w = cd.w[j - 1];
    const float4 P = s.P[w];
    const Smooth3 sp = smooth3<MODE>(dot3(P, Q[j - 1]) - P.w, alpha);
    const Smooth3 sq = smooth3<MODE>(dot3(P, Q[j + 1]) - P.w, alpha);
    const float4 M0 = s.M0[w], M1 = s.M1[w], M2 = s.M2[w];
    const float in = smooth3<MODE>(dot3(M0, Q[j]) - M0.w, alpha).s *
                     smooth3<MODE>(dot3(M1, Q[j]) - M1.w, alpha).s *
                     smooth3<MODE>(dot3(M2, Q[j]) - M2.w, alpha).s;
    R.V[j] = in * fmaf(sp.s, sq.s, sp.sb * sq.sb);
  }
}

// Multiplies the visibility factors of triangles w0 .. w1 - 1 into nz (each leg's product);
// a factor of exactly 0 makes the path dead, as does a product of all of them below stop
// (checked every 8 triangles; 0: never).  The warp leaves once every path is dead.
template <int MODE, int K>
__device__ __forceinline__ void vjp3_factor_sweep(const SmemTris& s, int w0, int w1, const Cand& cd,
                                                  const VjpPath3<K>& R, float alpha, float stop,
                                                  float* nz, bool& dead) {
#pragma unroll
  for (int j = 0; j <= K; ++j) {   // one loop per leg, as vjp_factor_sweep
    const float4 Pa = s.P[j >= 1 ? cd.w[j >= 1 ? j - 1 : 0] : 0], Pb = s.P[j < K ? cd.w[j < K ? j : 0] : 0];
    float others = 1.f, v = nz[j];
#pragma unroll
    for (int i = 0; i <= K; ++i) others *= i == j ? 1.f : nz[i];
#pragma unroll(K == 0 ? 2 : 1)   // K == 0: see WALL_TURN
    for (int w = w0; w < w1; ++w) {
      if (((w - w0) & 7) == 0) {
        dead |= others * v < stop;
        if (__all_sync(0xffffffffu, dead)) return;
      }
      const float4 P = s.P[w];
      const float4 M[3] = {s.M0[w], s.M1[w], s.M2[w]};
      const bool cop = (j >= 1 && one_plane(P, Pa)) || (j < K && one_plane(P, Pb));
      LegTri r;
      const bool hit = leg_tri<MODE>(P, M, R.Q[j], R.Q[j + 1], alpha, r);
      if (hit && !cop) {
        dead |= r.f == 0.f;
        v *= r.f;
      }
    }
    nz[j] = v;
  }
}

// WG: also the adjoints of every triangle's records (plane {n, c}, edges
// {m_k, o_k}) into the CTA table acc [W][TRI_SLOTS], summed over the warp.
// vis: the legs' visibilities, none of them 0 in a lane of non-zero weight, when the
// caller has run sweep 1 itself (the walk below: lanes hold different candidates).
// Without it the caller's lanes hold different candidates too (WG is then false).
template <int MODE, int K, bool WG>
__device__ __forceinline__ void path_vjp3(const SmemTris& s, int W, float3 tx, float3 rx,
                                          const Cand& cd, float alpha, float gk, float g,
                                          float3& txb, float* acc, const float* vis = nullptr) {
  VjpPath3<K> R;
  vjp3_recompute<MODE, K>(s, tx, rx, cd, alpha, R);
  const bool degenerate = R.degenerate;
  const float3* I = R.I;
  const float3* Q = R.Q;
  const float *dimg = R.dimg, *ta = R.ta, *tb = R.tb, *tt = R.tt, *len = R.len, *V = R.V;
  const float L = R.L;
  if (degenerate) g = 0.f;
  bool dead = degenerate || g == 0.f;
#pragma unroll
  for (int j = 1; j <= K; ++j) dead |= (V[j] == 0.f);
  if (__all_sync(0xffffffffu, dead)) return;
  // sweep 1: each leg's visibility
  float nz[K + 1];
#pragma unroll
  for (int j = 0; j <= K; ++j) nz[j] = vis ? vis[j] : 1.f;
  if (!vis) vjp3_factor_sweep<MODE, K>(s, 0, W, cd, R, alpha, 0.f, nz, dead);
  if (__all_sync(0xffffffffu, dead)) return;
  // a path with a factor of exactly 0 has a gradient of exactly 0: weight 0
  if (dead) {
    g = 0.f;
#pragma unroll
    for (int j = 0; j <= K; ++j) nz[j] = 1.f;
  }
  // factor adjoints: p = C prod(F), C = Gamma^k / L^2, F = {V_1..V_K, vis_0..vis_K}
  constexpr int NF = 2 * K + 1;
  float F[NF];
#pragma unroll
  for (int j = 1; j <= K; ++j) F[j - 1] = V[j];
#pragma unroll
  for (int j = 0; j <= K; ++j) F[K + j] = nz[j];
  float pre[NF + 1], suf[NF + 1];
  pre[0] = 1.f;
#pragma unroll
  for (int i = 0; i < NF; ++i) pre[i + 1] = pre[i] * F[i];
  suf[NF] = 1.f;
#pragma unroll
  for (int i = NF - 1; i >= 0; --i) suf[i] = suf[i + 1] * F[i];
  const float C = __fdiv_rn(gk, L * L);
  const float p = C * pre[NF];
  const float gC = g * C;
  float Vb[K + 1], visb[K + 1];
#pragma unroll
  for (int j = 1; j <= K; ++j) Vb[j] = gC * pre[j - 1] * suf[j];
#pragma unroll
  for (int j = 0; j <= K; ++j) visb[j] = gC * pre[K + j] * suf[K + j + 1];
  const float Lb = -2.f * g * __fdiv_rn(p, L);
  float3 Qb[K + 2];
#pragma unroll
  for (int i = 0; i <= K + 1; ++i) Qb[i] = make_float3(0.f, 0.f, 0.f);
  // sweep 2: each factor f = 1 - X ins pushes its adjoint into the leg's end points
  // (and, WG, into the triangle's records: x = n . Q_j - c, y = n . Q_{j+1} - c,
  // delta_k = (1 - t) e0_k + t e1_k with e_k = m_k . Q - o_k)
#pragma unroll
  for (int j = 0; j <= K; ++j) {   // one loop per leg, as vjp_factor_sweep
    const float4 Pa = s.P[j >= 1 ? cd.w[j >= 1 ? j - 1 : 0] : 0], Pb = s.P[j < K ? cd.w[j < K ? j : 0] : 0];
    const float3 q0 = Q[j], q1 = Q[j + 1];
    float3 b0 = make_float3(0.f, 0.f, 0.f), b1 = b0;
#pragma unroll 1
    for (int w = 0; w < W; ++w) {
      const float4 P = s.P[w];
      const float4 M[3] = {s.M0[w], s.M1[w], s.M2[w]};
      const bool cop = (j >= 1 && one_plane(P, Pa)) || (j < K && one_plane(P, Pb));
      LegTri r;
      const bool hit = leg_tri<MODE>(P, M, q0, q1, alpha, r);
      // (a factor of 0 only in a lane of weight 0)
      const float fb = hit && !cop && r.f != 0.f ? visb[j] * __fdiv_rn(nz[j], r.f) : 0.f;
      // no adjoint where neither X nor its slopes, or neither the on-triangle factor nor
      // its slopes, differ from 0: most triangles leave a leg alone
      const bool any = fb != 0.f && (r.X != 0.f || r.sx.ds != 0.f || r.sy.ds != 0.f) &&
                       (r.ins != 0.f || r.sd[0].ds != 0.f || r.sd[1].ds != 0.f || r.sd[2].ds != 0.f);
      if (!__any_sync(0xffffffffu, any)) continue;
      float wa[TRI_SLOTS];
#pragma unroll
      for (int i = 0; i < TRI_SLOTS; ++i) wa[i] = 0.f;
      if (any) {
        const float Xb = -fb * r.ins, inb = -fb * r.X;
        float xb = Xb * r.sx.ds * (r.sy.sb - r.sy.s);
        float yb = Xb * r.sy.ds * (r.sx.sb - r.sx.s);
        float tbar = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float others = r.sd[(k + 1) % 3].s * r.sd[(k + 2) % 3].s;
          const float db = inb * r.sd[k].ds * others;
          const float d0 = db * (1.f - r.t), d1 = db * r.t;
          axpy3(d0, M[k], b0);
          axpy3(d1, M[k], b1);
          tbar = fmaf(db, r.e1[k] - r.e0[k], tbar);
          if (WG) {
            float* m = wa + 4 + 4 * k;
            m[0] = fmaf(d0, q0.x, d1 * q1.x);
            m[1] = fmaf(d0, q0.y, d1 * q1.y);
            m[2] = fmaf(d0, q0.z, d1 * q1.z);
            m[3] = -(d0 + d1);
          }
        }
        const float den = r.x - r.y;
        const float id2 = __frcp_rn(den * den);
        xb = fmaf(tbar * -r.y, id2, xb);
        yb = fmaf(tbar * r.x, id2, yb);
        axpy3(xb, P, b0);
        axpy3(yb, P, b1);
        if (WG) {
          wa[0] = fmaf(xb, q0.x, yb * q1.x);
          wa[1] = fmaf(xb, q0.y, yb * q1.y);
          wa[2] = fmaf(xb, q0.z, yb * q1.z);
          wa[3] = -(xb + yb);
        }
      }
      if (WG) add_tri_adjoint(acc, w, wa);
    }
    Qb[j] = make_float3(Qb[j].x + b0.x, Qb[j].y + b0.y, Qb[j].z + b0.z);
    Qb[j + 1] = make_float3(Qb[j + 1].x + b1.x, Qb[j + 1].y + b1.y, Qb[j + 1].z + b1.z);
  }
  // legs: L = sum |Q_{j+1} - Q_j|
#pragma unroll
  for (int j = 0; j <= K; ++j) {
    const float il = len[j] > 0.f ? __frcp_rn(len[j]) : 0.f;
    const float4 u = make_float4((Q[j + 1].x - Q[j].x) * il, (Q[j + 1].y - Q[j].y) * il,
                                 (Q[j + 1].z - Q[j].z) * il, 0.f);
    axpy3(Lb, u, Qb[j + 1]);
    axpy3(-Lb, u, Qb[j]);
  }
  // validity: on the triangle (three edge tests) and the same-side test
#pragma unroll
  for (int j = 1; j <= K; ++j) {
    const int w = cd.w[j - 1];
    const float4 P = s.P[w];
    const float4 M[3] = {s.M0[w], s.M1[w], s.M2[w]};
    const Smooth3 sp = smooth3<MODE>(dot3(P, Q[j - 1]) - P.w, alpha);
    const Smooth3 sq = smooth3<MODE>(dot3(P, Q[j + 1]) - P.w, alpha);
    const float S = fmaf(sp.s, sq.s, sp.sb * sq.sb);
    Smooth3 sdl[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) sdl[k] = smooth3<MODE>(dot3(M[k], Q[j]) - M[k].w, alpha);
    const float ins = sdl[0].s * sdl[1].s * sdl[2].s;
    const float insb = Vb[j] * S, Sb = Vb[j] * ins;
    float wa[TRI_SLOTS];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float dk = insb * sdl[k].ds * sdl[(k + 1) % 3].s * sdl[(k + 2) % 3].s;
      axpy3(dk, M[k], Qb[j]);
      wa[4 + 4 * k] = dk * Q[j].x;   // delta_k = m_k . Q_j - o_k
      wa[5 + 4 * k] = dk * Q[j].y;
      wa[6 + 4 * k] = dk * Q[j].z;
      wa[7 + 4 * k] = -dk;
    }
    const float pb = Sb * sp.ds * (sq.s - sq.sb), qb = Sb * sq.ds * (sp.s - sp.sb);
    axpy3(pb, P, Qb[j - 1]);
    axpy3(qb, P, Qb[j + 1]);
    if (WG) {   // p = n . Q_{j-1} - c, q = n . Q_{j+1} - c
      wa[0] = fmaf(pb, Q[j - 1].x, qb * Q[j + 1].x);
      wa[1] = fmaf(pb, Q[j - 1].y, qb * Q[j + 1].y);
      wa[2] = fmaf(pb, Q[j - 1].z, qb * Q[j + 1].z);
      wa[3] = -(pb + qb);
      add_tri_adjoints(acc, w, wa);
    }
  }
  // backtrace, reversed: Q_j = Q_{j+1} + t (I_j - Q_{j+1}), t = b / (b - a)
  float3 Ib[K + 1];
#pragma unroll
  for (int j = 0; j <= K; ++j) Ib[j] = make_float3(0.f, 0.f, 0.f);
#pragma unroll
  for (int j = 1; j <= K; ++j) {
    const float4 P = s.P[cd.w[j - 1]];
    const float t = tt[j];
    const float4 q = make_float4(Qb[j].x, Qb[j].y, Qb[j].z, 0.f);
    axpy3(1.f - t, q, Qb[j + 1]);
    axpy3(t, q, Ib[j]);
    const float tbar = fmaf(Qb[j].x, I[j].x - Q[j + 1].x,
                            fmaf(Qb[j].y, I[j].y - Q[j + 1].y, Qb[j].z * (I[j].z - Q[j + 1].z)));
    const float den = tb[j] - ta[j];
    const float id2 = (den != 0.f && !degenerate) ? __frcp_rn(den * den) : 0.f;
    const float abar = tbar * tb[j] * id2, bbar = -tbar * ta[j] * id2;
    axpy3(abar, P, Ib[j]);
    axpy3(bbar, P, Qb[j + 1]);
    if (WG) {   // a = n . I_j - c, b = n . Q_{j+1} - c
      float wa[TRI_SLOTS];
#pragma unroll
      for (int i = 4; i < TRI_SLOTS; ++i) wa[i] = 0.f;
      wa[0] = fmaf(abar, I[j].x, bbar * Q[j + 1].x);
      wa[1] = fmaf(abar, I[j].y, bbar * Q[j + 1].y);
      wa[2] = fmaf(abar, I[j].z, bbar * Q[j + 1].z);
      wa[3] = -(abar + bbar);
      add_tri_adjoints(acc, cd.w[j - 1], wa);
    }
  }
  // image chain, reversed: I_j = I_{j-1} - 2 d n, d = n . I_{j-1} - c
#pragma unroll
  for (int j = K; j >= 1; --j) {
    const float4 P = s.P[cd.w[j - 1]];
    const float dbar = -2.f * fmaf(Ib[j].x, P.x, fmaf(Ib[j].y, P.y, Ib[j].z * P.z));
    if (WG) {   // n_bar = -2 d I_bar_j + d_bar I_{j-1}, c_bar = -d_bar
      float wa[TRI_SLOTS];
#pragma unroll
      for (int i = 4; i < TRI_SLOTS; ++i) wa[i] = 0.f;
      wa[0] = fmaf(-2.f * dimg[j], Ib[j].x, dbar * I[j - 1].x);
      wa[1] = fmaf(-2.f * dimg[j], Ib[j].y, dbar * I[j - 1].y);
      wa[2] = fmaf(-2.f * dimg[j], Ib[j].z, dbar * I[j - 1].z);
      wa[3] = -dbar;
      add_tri_adjoints(acc, cd.w[j - 1], wa);
    }
    Ib[j - 1].x += fmaf(dbar, P.x, Ib[j].x);
    Ib[j - 1].y += fmaf(dbar, P.y, Ib[j].y);
    Ib[j - 1].z += fmaf(dbar, P.z, Ib[j].z);
  }
  txb.x += Qb[0].x + Ib[0].x;
  txb.y += Qb[0].y + Ib[0].y;
  txb.z += Qb[0].z + Ib[0].z;
}

// The dense 3D adjoint's walk (drt_vjp_walk.cuh's stages, one path per lane).  The
// sigmoid's paths below FLOOR_VJP of their receiver's floor are left out.
struct VjpQueue3 {
  uint2 e1[64], e2[64], e3[64];
  float4 v2[64], v3[64];
};

template <int MODE, int K, bool WG>
struct VjpWalk3 {
  const SmemTris& s;
  VjpQueue3& q;
  int W, w1;   // triangles, triangles of stage 1
  float3 tx;
  float alpha, gk;
  float3 rx;   // this lane's receiver, weight and floor
  float g, floor;
  float3& txb;
  float* acc;
  int h1 = 0, n1 = 0, h2 = 0, n2 = 0, h3 = 0, n3 = 0;

  __device__ __forceinline__ void push(uint2* e, float4* v, int head, int& n, bool take, uint2 x,
                                       const float* nz) {
    const unsigned b = __ballot_sync(0xffffffffu, take);
    if (take) {
      const int i = (head + n + __popc(b & ((1u << (threadIdx.x & 31)) - 1u))) & 63;
      e[i] = x;
      v[i] = make_float4(nz[0], K > 0 ? nz[K > 0 ? 1 : 0] : 0.f, K > 1 ? nz[K > 1 ? 2 : 0] : 0.f,
                         K > 2 ? nz[K > 2 ? 3 : 0] : 0.f);
    }
    n += __popc(b);
    __syncwarp();
  }
  __device__ __forceinline__ static void read(const float4& v, float* nz) {
    nz[0] = v.x;
    if (K > 0) nz[K > 0 ? 1 : 0] = v.y;
    if (K > 1) nz[K > 1 ? 2 : 0] = v.z;
    if (K > 2) nz[K > 2 ? 3 : 0] = v.w;
  }
  __device__ __forceinline__ float stop_at(const VjpPath3<K>& R, int r) const {
    const float f = __shfl_sync(0xffffffffu, floor, r);
    float V = gk;
#pragma unroll
    for (int j = 1; j <= K; ++j) V *= R.V[j];
    return MODE == MODE_SIGMOID && f > 0.f ? __fdividef(f * (R.L * R.L), V) : 0.f;
  }

  __device__ __forceinline__ void adjoint(int n) {
    const int lane = threadIdx.x & 31;
    const bool have = lane < n;
    const int i = (h3 + (have ? lane : 0)) & 63;
    const uint2 e = q.e3[i];
    float nz[K + 1];
    read(q.v3[i], nz);
    const int r = (int)(e.y >> 16);
    const float3 p = shfl3(rx, r);
    const float gr = __shfl_sync(0xffffffffu, g, r);
    path_vjp3<MODE, K, WG>(s, W, tx, p, entry_walls<K>(e), alpha, gk, have ? gr : 0.f, txb, acc, nz);
    h3 = (h3 + n) & 63;
    n3 -= n;
    __syncwarp();
  }

  // stage 1 (the first triangles, e1 -> e2) and stage 2 (the others, e2 -> e3)
  template <bool FIRST>
  __device__ __forceinline__ void factors(int n) {
    const int lane = threadIdx.x & 31;
    const bool have = lane < n;
    const int i = ((FIRST ? h1 : h2) + (have ? lane : 0)) & 63;
    const uint2 e = FIRST ? q.e1[i] : q.e2[i];
    float nz[K + 1];
    if (FIRST) {
#pragma unroll
      for (int j = 0; j <= K; ++j) nz[j] = 1.f;
    } else {
      read(q.v2[i], nz);
    }
    const Cand cd = entry_walls<K>(e);
    const int r = (int)(e.y >> 16);
    VjpPath3<K> R;
    vjp3_recompute<MODE, K>(s, tx, shfl3(rx, r), cd, alpha, R);
    const float stop = stop_at(R, r);
    bool dead = !have;
    vjp3_factor_sweep<MODE, K>(s, FIRST ? 0 : w1, FIRST ? w1 : W, cd, R, alpha, stop, nz, dead);
    if (FIRST) {
      h1 = (h1 + n) & 63;
      n1 -= n;
      push(q.e2, q.v2, h2, n2, !dead, e, nz);
    } else {
      float all = nz[0];
#pragma unroll
      for (int j = 1; j <= K; ++j) all *= nz[j];
      dead |= all < stop;
      h2 = (h2 + n) & 63;
      n2 -= n;
      push(q.e3, q.v3, h3, n3, !dead, e, nz);
    }
  }

  __device__ __forceinline__ void candidate(const Cand& cd) {
    const int lane = threadIdx.x & 31;
    VjpPath3<K> R;
    vjp3_recompute<MODE, K>(s, tx, rx, cd, alpha, R);
    bool take = !R.degenerate && g != 0.f;
    float V = fabsf(gk);
#pragma unroll
    for (int j = 1; j <= K; ++j) {
      take &= R.V[j] != 0.f;
      V *= R.V[j];
    }
    if (MODE == MODE_SIGMOID) take &= !(V < floor * (R.L * R.L));
    const unsigned b = __ballot_sync(0xffffffffu, take);
    if (!b) return;
    if (take) q.e1[(h1 + n1 + __popc(b & ((1u << lane) - 1u))) & 63] = entry_of(cd, lane);
    n1 += __popc(b);
    __syncwarp();
  }

  // as VjpWalk's
  __device__ __forceinline__ void work(bool end) {
    for (;;) {
      if (n3 >= 32 || (end && n3 && !n2 && !n1)) adjoint(min(n3, 32));
      else if (n2 >= 32 || (end && n2 && !n1)) factors<false>(min(n2, 32));
      else if (n1 >= 32 || (end && n1)) factors<true>(min(n1, 32));
      else break;
    }
  }

  template <class Stream>
  __device__ __forceinline__ void run(Stream& st) {
    for (;;) {
      Cand cd;
      const bool more = st.next(cd);
      if (more) candidate(cd);
      work(!more);
      if (!more) break;
    }
  }
};

template <int MODE, bool WG>
__device__ __forceinline__ void walk_vjp3(const SmemTris& s, int W, int K, float3 tx, float3 rx, float g,
                                          float alpha, const float* gk, long long n_cand, int c0,
                                          int nc, VjpQueue3& q, float3& txb, float* acc) {
  const float floor = FLOOR_VJP * receiver_floor3<MODE>(s, W, tx, rx, alpha, gk[1], n_cand);
  const TileFloor tf{MODE == MODE_SIGMOID ? warp_min(g != 0.f ? floor : INFINITY) : 0.f, gk, false};
  const Box3 box = tile_box3(rx, g != 0.f);
  const int w1 = max(W / 4, min(W, 8));
  const float m = zero_margin<MODE>(alpha);
  for_orders(W, K, c0, nc, [&](auto order, int lo, int n) {
    constexpr int KO = decltype(order)::value;
    auto reach = [&](const Cand& cd) { return tile_may_reach3<MODE, KO>(s, cd, tx, box, m, alpha, tf); };
    CandStream<KO, decltype(reach)> st{W, lo, n, reach};
    VjpWalk3<MODE, KO, WG> walk{s, q, W, w1, tx, alpha, gk[KO], rx, g, floor, txb, acc};
    walk.run(st);
  });
}

__device__ __forceinline__ float warp_sum3(float v) {
#pragma unroll
  for (int m = 16; m; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

}  // namespace drt
