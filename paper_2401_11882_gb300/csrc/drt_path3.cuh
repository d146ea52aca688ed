// Paths of the method in 3D (Sec. VI: the framework does not depend on the
// dimension): walls are triangles, lines become planes, and a point lies on an
// object when its three in-plane edge distances pass the smoothed comparison.
//
//   plane of triangle (A, B, C): unit normal n along (B - A) x (C - A), c = n . A,
//   d(p) = n . p - c; edge k (A->B, B->C, C->A): in-plane unit normal
//   m_k = n x e_k / |e_k| (pointing inside), delta_k(p) = m_k . p - m_k . (start of k);
//   image method and backtrace as in 2D with planes for lines;
//   validity of reflection j: prod_k s(delta_k(Q_j)) (s(p) s(q) + s(-p) s(-q));
//   obstruction of leg Q_j -> Q_{j+1} by triangle w (not one in the plane of a
//   triangle its end points lie on, which the leg meets only at that end point):
//   X(x, y) prod_k s(delta_k(P)), x, y the end points' plane distances and P
//   the point where the leg's line meets the plane, whose edge distances are the
//   end points' ones interpolated at t = x / (x - y) (delta_k is affine);
//   path power Gamma^k V vis / L^2, summed over the candidates;
//   two consecutive reflections on triangles of one plane make a degenerate path:
//   the leg between them has zero length, and in floating point its rounding-sized
//   length would make the path's power an arbitrary function of the rounding.
//   "One plane": normals parallel and offsets equal, both to 1e-5.
//
// Mapping as in drt_forward.cu: lanes are receivers, the candidate is
// warp-uniform, the triangles' plane and edge records sit in shared memory and
// are read as broadcasts; per triangle, the plane and edge distances of every
// path vertex are computed once and shared by the two legs meeting there.  Units
// of (32 receivers) x (a chunk of candidates), per-chunk partial sums added in
// chunk order: deterministic.
#pragma once

#include <cuda_runtime.h>

#include "drt_common.cuh"
#include "drt_internal.h"
#include "drt_path_queue.cuh"

namespace drt {

// Triangle records in shared memory, 4 float4 per triangle:
//   P  {nx, ny, nz, c}            plane: d(p) = n . p - c
//   Mk {mx, my, mz, o_k}, k=0..2  edge k: delta_k(p) = m_k . p - o_k
struct SmemTris {
  float4 *P, *M0, *M1, *M2;
};

__device__ __forceinline__ float dot3(float4 r, float3 p) {
  return fmaf(r.x, p.x, fmaf(r.y, p.y, r.z * p.z));
}

__device__ __forceinline__ void stage_tris(const float* __restrict__ tris, int W, SmemTris s) {
  for (int w = threadIdx.x; w < W; w += blockDim.x) {
    const float* t = tris + 9 * (size_t)w;
    const float3 a = make_float3(t[0], t[1], t[2]);
    const float3 b = make_float3(t[3], t[4], t[5]);
    const float3 c = make_float3(t[6], t[7], t[8]);
    const float3 e1 = make_float3(b.x - a.x, b.y - a.y, b.z - a.z);
    const float3 e2 = make_float3(c.x - a.x, c.y - a.y, c.z - a.z);
    float3 n = make_float3(fmaf(e1.y, e2.z, -e1.z * e2.y), fmaf(e1.z, e2.x, -e1.x * e2.z),
                           fmaf(e1.x, e2.y, -e1.y * e2.x));
    const float nl = __fsqrt_rn(fmaf(n.x, n.x, fmaf(n.y, n.y, n.z * n.z)));
    n = make_float3(__fdiv_rn(n.x, nl), __fdiv_rn(n.y, nl), __fdiv_rn(n.z, nl));
    const float4 P = make_float4(n.x, n.y, n.z, fmaf(n.x, a.x, fmaf(n.y, a.y, n.z * a.z)));
    s.P[w] = P;
    const float3 v[3] = {a, b, c};
    float4* M[3] = {s.M0, s.M1, s.M2};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float3 p = v[k], q = v[(k + 1) % 3];
      const float3 e = make_float3(q.x - p.x, q.y - p.y, q.z - p.z);
      float3 m = make_float3(fmaf(n.y, e.z, -n.z * e.y), fmaf(n.z, e.x, -n.x * e.z),
                             fmaf(n.x, e.y, -n.y * e.x));
      const float ml = __fsqrt_rn(fmaf(m.x, m.x, fmaf(m.y, m.y, m.z * m.z)));
      m = make_float3(__fdiv_rn(m.x, ml), __fdiv_rn(m.y, ml), __fdiv_rn(m.z, ml));
      M[k][w] = make_float4(m.x, m.y, m.z, fmaf(m.x, p.x, fmaf(m.y, p.y, m.z * p.z)));
    }
  }
}

// Triangles a and b lie in one plane (normals parallel, offsets equal, to 1e-5).
__device__ __forceinline__ bool one_plane(const float4& Pa, const float4& Pb) {
  const float nn = fmaf(Pa.x, Pb.x, fmaf(Pa.y, Pb.y, Pa.z * Pb.z));
  return fabsf(nn) >= 1.f - 1e-5f && fabsf(fmaf(-nn, Pb.w, Pa.w)) <= 1e-5f * (1.f + fabsf(Pa.w));
}

// Sigmoid obstruction of every leg by every triangle (the forward's loop; the
// adjoint keeps its own).  With e = 2^-|z| for the smoothed distances of a leg's
// end points to the triangle's plane, the straddle term is X = x1 / D1 with
// Ns = e_j + e_{j+1}, No = 1 + e_j e_{j+1}, D1 = Ns + No and x1 = Ns when both
// lie on one side, No otherwise (xb1 the other one), as in 2D.  The on-triangle
// factor at the crossing point is in = 1 / Pin with Pin = prod_k (1 + u_k),
// u_k = 2^-a_k for the three scaled in-plane edge distances a_k (u_k capped at
// 2^24, where s < 6e-8 already rounds the product); Pin - 1 is expanded as a sum
// of products of the u_k.  Then
//   1 - X in = (xb1 + x1 (1 - in)) / D1,   1 - in = (Pin - 1) / Pin,
// a sum of non-negative terms: a leg nearly blocked by a triangle keeps its
// relative accuracy, and one reciprocal gives the three edge factors (four MUFU
// operations per test and one per vertex, against seven and two for three
// separate sigmoids).  Numerators and D1 are multiplied up separately and folded
// into vis every 8 triangles (D1 <= 4).  stop: the warp leaves the loop once the product
// of each lane's leg visibilities is below it (0: never).
template <int K>
__device__ __forceinline__ void sigmoid_visibility3(const SmemTris& s, int W, const float3* Q,
                                                    const float4* Pr, float alpha, float* vis,
                                                    float stop) {
  const float kap = alpha * LOG2E;
  float vn[K + 1], vd[K + 1];
#pragma unroll
  for (int j = 0; j <= K; ++j) vn[j] = vd[j] = 1.f;
  for (int w0 = 0; w0 < W; w0 += 8) {
    const int w1 = min(w0 + 8, W);
#pragma unroll(K == 0 ? 2 : 1)   // K == 0: see WALL_TURN
    for (int w = w0; w < w1; ++w) {
      const float4 P = s.P[w], M0 = s.M0[w], M1 = s.M1[w], M2 = s.M2[w];
      bool cop[K + 2];   // w in the plane of reflection j's triangle
      cop[0] = cop[K + 1] = false;
#pragma unroll
      for (int j = 1; j <= K; ++j) cop[j] = one_plane(P, Pr[j]);
      float d[K + 2], ee[K + 2], e0[K + 2], e1[K + 2], e2[K + 2];
#pragma unroll
      for (int i = 0; i <= K + 1; ++i) {
        d[i] = dot3(P, Q[i]) - P.w;
        ee[i] = ex2_approx(-fabsf(d[i] * kap));
        e0[i] = (dot3(M0, Q[i]) - M0.w) * kap;
        e1[i] = (dot3(M1, Q[i]) - M1.w) * kap;
        e2[i] = (dot3(M2, Q[i]) - M2.w) * kap;
      }
#pragma unroll
      for (int j = 0; j <= K; ++j) {
        const float t = __fdividef(d[j], d[j] - d[j + 1]);
        // the leg's line misses the plane (or meets it absurdly far): not blocked
        const bool test = !(cop[j] || cop[j + 1]) && fabsf(t) <= 1e8f;
        const float ns = ee[j] + ee[j + 1];
        const float no = fmaf(ee[j], ee[j + 1], 1.f);
        const bool same = same_side(d[j], d[j + 1]);
        const float x1 = same ? ns : no, xb1 = same ? no : ns;
        const float u0 = ex2_approx(fminf(-fmaf(t, e0[j + 1] - e0[j], e0[j]), 24.f));
        const float u1 = ex2_approx(fminf(-fmaf(t, e1[j + 1] - e1[j], e1[j]), 24.f));
        const float u2 = ex2_approx(fminf(-fmaf(t, e2[j + 1] - e2[j], e2[j]), 24.f));
        const float a01 = fmaf(u0, u1, u0 + u1);
        const float pm1 = fmaf(u2, 1.f + a01, a01);
        const float omi = pm1 * rcp_approx(1.f + pm1);
        vn[j] *= test ? fmaf(x1, omi, xb1) : 1.f;
        vd[j] *= test ? ns + no : 1.f;
      }
    }
    float all = 1.f;
#pragma unroll
    for (int j = 0; j <= K; ++j) {
      vis[j] *= __fdividef(vn[j], vd[j]);
      vn[j] = vd[j] = 1.f;
      all *= vis[j];
    }
    if (__all_sync(0xffffffffu, all < stop)) break;
  }
}

// Receiver-dependent geometry of one path: vertices, length and validity.
template <int K>
struct Path3 {
  float3 Q[K + 2];
  float L, V;
  bool degenerate;
};

template <int MODE, int K>
__device__ __forceinline__ void path3_geometry(const SmemTris& s, float3 tx, float3 rx,
                                               const Cand& cd, float alpha, Path3<K>& g) {
  float3 I[K + 1];   // images
  I[0] = tx;
#pragma unroll
  for (int j = 1; j <= K; ++j) {
    const float4 P = s.P[cd.w[j - 1]];
    const float d2 = 2.f * (dot3(P, I[j - 1]) - P.w);
    I[j] = make_float3(fmaf(-d2, P.x, I[j - 1].x), fmaf(-d2, P.y, I[j - 1].y),
                       fmaf(-d2, P.z, I[j - 1].z));
  }
  // two consecutive reflections in one plane (two triangles of one flat face): the
  // leg between them has zero length, the path is degenerate
  g.degenerate = false;
#pragma unroll
  for (int j = 1; j < K; ++j) g.degenerate |= one_plane(s.P[cd.w[j - 1]], s.P[cd.w[j]]);
  // backtrace on the planes: Q_{K+1} = RX, Q_j = line(Q_{j+1}, I_j) x plane j
  float3* Q = g.Q;
  Q[0] = tx;
  Q[K + 1] = rx;
#pragma unroll
  for (int j = K; j >= 1; --j) {
    const float4 P = s.P[cd.w[j - 1]];
    const float a = dot3(P, I[j]) - P.w;
    const float b = dot3(P, Q[j + 1]) - P.w;
    float t = __fdividef(b, b - a);
    if (!(fabsf(t) <= 1e8f)) {
      g.degenerate = true;
      t = 0.f;
    }
    Q[j] = make_float3(fmaf(t, I[j].x - Q[j + 1].x, Q[j + 1].x),
                       fmaf(t, I[j].y - Q[j + 1].y, Q[j + 1].y),
                       fmaf(t, I[j].z - Q[j + 1].z, Q[j + 1].z));
  }
  g.L = 0.f;
#pragma unroll
  for (int j = 0; j <= K; ++j) {
    const float dx = Q[j + 1].x - Q[j].x, dy = Q[j + 1].y - Q[j].y, dz = Q[j + 1].z - Q[j].z;
    const float len2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    g.degenerate |= !(len2 > 0.f);
    g.L += __fsqrt_rn(len2);
  }
  // validity: on the triangle, and the neighbours on the same side of its plane
  g.V = 1.f;
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
    g.V *= in * fmaf(sp.s, sq.s, sp.sb * sq.sb);
  }
}

// Whether the path is 0 or below the receiver's floor whatever its legs meet (as
// path_negligible in 2D; the floor is 0 but for the sigmoid).
template <int MODE, int K>
__device__ __forceinline__ bool path3_negligible(const Path3<K>& g, float gk, float floor) {
  if (g.degenerate || g.V == 0.f) return true;
  return MODE == MODE_SIGMOID && g.V * fabsf(gk) < floor * (g.L * g.L);
}

// Power of one path of order K from its geometry (not degenerate): obstruction by every
// triangle of every leg, except the triangles in the plane of a triangle the leg's end
// points lie on (the leg meets that plane only there).  The warp leaves the loop once
// every lane's power is known to be 0, or below its floor.
template <int MODE, int K>
__device__ __forceinline__ float path3_power(const SmemTris& s, int W, const Path3<K>& g,
                                             const Cand& cd, float alpha, float gk, float floor) {
  const float3* Q = g.Q;
  float vis[K + 1];
#pragma unroll
  for (int j = 0; j <= K; ++j) vis[j] = 1.f;
  float4 Pr[K + 1];
#pragma unroll
  for (int j = 1; j <= K; ++j) Pr[j] = s.P[cd.w[j - 1]];
  if constexpr (MODE == MODE_SIGMOID) {
    const float stop = floor > 0.f ? __fdividef(floor * (g.L * g.L), g.V * gk) : 0.f;
    sigmoid_visibility3<K>(s, W, Q, Pr, alpha, vis, stop);
  } else {
#pragma unroll 1
    for (int w = 0; w < W; ++w) {
      if ((w & 7) == 0 && w > 0) {
        bool zero = false;
#pragma unroll
        for (int j = 0; j <= K; ++j) zero |= vis[j] == 0.f;
        if (__all_sync(0xffffffffu, zero)) break;
      }
      const float4 P = s.P[w], M0 = s.M0[w], M1 = s.M1[w], M2 = s.M2[w];
      bool cop[K + 2];   // w in the plane of reflection j's triangle
      cop[0] = cop[K + 1] = false;
#pragma unroll
      for (int j = 1; j <= K; ++j) cop[j] = one_plane(P, Pr[j]);
      float d[K + 2], e0[K + 2], e1[K + 2], e2[K + 2];
      Smooth3 sd[K + 2];
#pragma unroll
      for (int i = 0; i <= K + 1; ++i) {
        d[i] = dot3(P, Q[i]) - P.w;
        sd[i] = smooth3<MODE>(d[i], alpha);
        e0[i] = dot3(M0, Q[i]) - M0.w;
        e1[i] = dot3(M1, Q[i]) - M1.w;
        e2[i] = dot3(M2, Q[i]) - M2.w;
      }
#pragma unroll
      for (int j = 0; j <= K; ++j) {
        const float X = fmaf(sd[j].s, sd[j + 1].sb, sd[j].sb * sd[j + 1].s);
        const float den = d[j] - d[j + 1];
        const float t = __fdividef(d[j], den);
        const float in = smooth3<MODE>(fmaf(t, e0[j + 1] - e0[j], e0[j]), alpha).s *
                         smooth3<MODE>(fmaf(t, e1[j + 1] - e1[j], e1[j]), alpha).s *
                         smooth3<MODE>(fmaf(t, e2[j + 1] - e2[j], e2[j]), alpha).s;
        // the leg's line misses the plane (or meets it absurdly far): not blocked
        const bool test = !(cop[j] || cop[j + 1]) && fabsf(t) <= 1e8f;
        vis[j] = test ? fmaf(-X, in * vis[j], vis[j]) : vis[j];
      }
    }
  }
  float p = g.V * gk;
#pragma unroll
  for (int j = 0; j <= K; ++j) p *= vis[j];
  p = __fdividef(p, g.L * g.L);
  return fabsf(p) < floor ? 0.f : p;
}

// ---------------------------------------------------------------- the walk in 3D
// drt_path_queue.cuh's walk for triangles, one path per lane: candidates bounded over
// the tile's box, validity per receiver, obstruction on batches of 32 queued paths.
// Measured on the room (132 triangles, 4096 receivers, K = 2, hard sigmoid, GB300):
// forward and adjoint with the triangles 22.3 -> 12.5 ms (queues), 7.3 (one copy of each
// stage, one loop over the triangles per leg).
struct Box3 {
  float3 lo, hi;
};

__device__ __forceinline__ Box3 tile_box3(float3 q, bool live) {
  Box3 b;
  b.lo.x = warp_min(live ? q.x : INFINITY);
  b.lo.y = warp_min(live ? q.y : INFINITY);
  b.lo.z = warp_min(live ? q.z : INFINITY);
  b.hi.x = -warp_min(live ? -q.x : INFINITY);
  b.hi.y = -warp_min(live ? -q.y : INFINITY);
  b.hi.z = -warp_min(live ? -q.z : INFINITY);
  return b;
}

// false only when candidate cd is negligible for every receiver in the box (see
// tile_may_reach): the receivers' side of each reflection is held as the hull of the
// eight points the box's corners map to, and the reflection points' edge distances are
// ratios of affine functions of it as the 2D coordinate is.
template <int MODE, int K>
__device__ __forceinline__ bool tile_may_reach3(const SmemTris& s, const Cand& cd, float3 tx,
                                                const Box3& box, float m, float alpha,
                                                const TileFloor& tf) {
  if (K == 0 || !(m < 1e8f)) return true;
  constexpr float U = 6e-8f;
  float3 I[K + 1];
  I[0] = tx;
#pragma unroll
  for (int j = 1; j <= K; ++j) {
    const float4 P = s.P[cd.w[j - 1]];
    const float d2 = 2.f * (dot3(P, I[j - 1]) - P.w);
    I[j] = make_float3(fmaf(-d2, P.x, I[j - 1].x), fmaf(-d2, P.y, I[j - 1].y),
                       fmaf(-d2, P.z, I[j - 1].z));
  }
  if (MODE == MODE_SIGMOID && tf.floor > 0.f) {
    const float3 i = I[K];
    const float dx = fmaxf(fmaxf(box.lo.x - i.x, i.x - box.hi.x), 0.f);
    const float dy = fmaxf(fmaxf(box.lo.y - i.y, i.y - box.hi.y), 0.f);
    const float dz = fmaxf(fmaxf(box.lo.z - i.z, i.z - box.hi.z), 0.f);
    const float d2 = 0.999f * fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float mf = __fdividef(logf(__fdividef(tf.ck[K], tf.floor * d2)) + 1.f, alpha);
    if (mf < m) m = fmaxf(mf, 0.f);
  }
  float3 p[8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
    p[i] = make_float3(i & 1 ? box.hi.x : box.lo.x, i & 2 ? box.hi.y : box.lo.y,
                       i & 4 ? box.hi.z : box.lo.z);
  float dl = 0.f, nlo = 0.f, nhi = 0.f, ne = 0.f;
#pragma unroll
  for (int j = K; j >= 1; --j) {
    const int w = cd.w[j - 1];
    const float4 P = s.P[w];
    const float4 M[3] = {s.M0[w], s.M1[w], s.M2[w]};
    const float a = dot3(P, I[j]) - P.w;
    float S = 0.f, g = INFINITY, tmax = 0.f, blo = INFINITY, bhi = -INFINITY;
    float hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    bool pos = true, neg = true;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float b = dot3(P, p[i]) - P.w;
      const float den = b - a;
      const float t = __fdividef(b, den);
      pos &= den > 0.f;
      neg &= den < 0.f;
      g = fminf(g, fabsf(den));
      S = fmaxf(S, fabsf(p[i].x) + fabsf(p[i].y) + fabsf(p[i].z));
      tmax = fmaxf(tmax, fabsf(t));
      blo = fminf(blo, b);
      bhi = fmaxf(bhi, b);
      p[i] = make_float3(fmaf(t, I[j].x - p[i].x, p[i].x), fmaf(t, I[j].y - p[i].y, p[i].y),
                         fmaf(t, I[j].z - p[i].z, p[i].z));
#pragma unroll
      for (int k = 0; k < 3; ++k) hi[k] = fmaxf(hi[k], dot3(M[k], p[i]) - M[k].w);
    }
    S += fabsf(I[j].x) + fabsf(I[j].y) + fabsf(I[j].z) + fabsf(P.w) + fabsf(M[0].w) +
         fabsf(M[1].w) + fabsf(M[2].w);
    const float eb = fmaf(12.f * U, S, dl);
    if (!((pos || neg) && g > 64.f * eb && tmax < 1e6f && S < 1e8f)) return true;
    const float et = __fdividef(2.f * (eb + 2.f * tmax * eb), g) + 8.f * U * tmax;
    const float err = 2.f * (fmaf(dl, 1.f + tmax, et * S) + 48.f * U * S * (1.f + tmax));
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (hi[k] < -m - err) return false;   // off the triangle for every receiver
    // same side: the previous vertex (this reflection's hull) and the next of the wall after
    if (j < K) {
      const float4 H = s.P[cd.w[j]];
      float d0 = INFINITY, d1 = -INFINITY, T = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float d = dot3(H, p[i]) - H.w;
        d0 = fminf(d0, d);
        d1 = fmaxf(d1, d);
        T = fmaxf(T, fabsf(p[i].x) + fabsf(p[i].y) + fabsf(p[i].z));
      }
      const float e = m + ne + err + 12.f * U * (S + T + fabsf(H.w));
      if ((d1 < -e && nlo > e) || (d0 > e && nhi < -e)) return false;
    }
    if (j == 1) {
      const float d = dot3(P, tx) - P.w;
      const float e = m + eb + 12.f * U * (fabsf(tx.x) + fabsf(tx.y) + fabsf(tx.z));
      if ((d < -e && blo > e) || (d > e && bhi < -e)) return false;
    }
    nlo = blo;
    nhi = bhi;
    ne = eb;
    dl = err;
  }
  return true;
}

__device__ __forceinline__ float3 shfl3(float3 v, int src) {
  return make_float3(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src),
                     __shfl_sync(0xffffffffu, v.z, src));
}

// The receiver's floor: its line of sight's power times NEGLIGIBLE / number of candidates.
template <int MODE>
__device__ __forceinline__ float receiver_floor3(const SmemTris& s, int W, float3 tx, float3 rx,
                                                 float alpha, float gamma, long long n_cand) {
  if (MODE != MODE_SIGMOID || !has_floors(gamma, n_cand)) return 0.f;
  Cand cd;
  cd.k = 0;
#pragma unroll
  for (int j = 0; j < KMAX; ++j) cd.w[j] = -1;
  Path3<0> g;
  path3_geometry<MODE, 0>(s, tx, rx, cd, alpha, g);
  const float p = path3_power<MODE, 0>(s, W, g, cd, alpha, 1.f, 0.f);
  return !g.degenerate && p > 0.f ? p * (NEGLIGIBLE * __fdividef(1.f, (float)n_cand)) : 0.f;
}

// Per-warp queue of one order's paths (ring buffer) and the tile's sums.
struct WarpQueue3 {
  uint2 e[64];
  float acc[32];
};

template <int MODE, int K>
__device__ __forceinline__ void flush_paths3(const SmemTris& s, int W, float3 tx, float3 q, float floor,
                                             float alpha, float gk, WarpQueue3& wq, int head, int n) {
  const int lane = threadIdx.x & 31;
  bool rem = lane < n;
  const uint2 e = wq.e[(head + (rem ? lane : 0)) & 63];
  const int r = (int)(e.y >> 16);
  const Cand cd = entry_walls<K>(e);
  const float3 rx = shfl3(q, r);
  const float fl = __shfl_sync(0xffffffffu, floor, r);
  Path3<K> g;
  path3_geometry<MODE, K>(s, tx, rx, cd, alpha, g);
  const float v = path3_power<MODE, K>(s, W, g, cd, alpha, gk, fl);
  // queue order is candidate order: per round, each receiver's first remaining entry
  while (__any_sync(0xffffffffu, rem)) {
    const unsigned same = __match_any_sync(0xffffffffu, rem ? r : 32 + lane);
    if (rem && __ffs(same) - 1 == lane) {
      wq.acc[r] += v;
      rem = false;
    }
    __syncwarp();
  }
}

// The power of candidates c0 .. c0 + nc - 1 for this lane's receiver of the tile.
template <int MODE>
__device__ __forceinline__ float walk_valid_paths3(const SmemTris& s, int W, int K, float3 tx, float3 q,
                                                   bool live, float alpha, const float* gk,
                                                   long long n_cand, int c0, int nc,
                                                   WarpQueue3& wq) {
  const int lane = threadIdx.x & 31;
  const float floor = receiver_floor3<MODE>(s, W, tx, q, alpha, gk[1], n_cand);
  const TileFloor tf{MODE == MODE_SIGMOID ? warp_min(live ? floor : INFINITY) : 0.f, gk, false};
  __syncwarp();
  wq.acc[lane] = 0.f;
  __syncwarp();
  const Box3 box = tile_box3(q, live);
  const float m = zero_margin<MODE>(alpha);
  for_orders(W, K, c0, nc, [&](auto order, int lo, int count) {
    constexpr int KO = decltype(order)::value;
    auto reach = [&](const Cand& cd) { return tile_may_reach3<MODE, KO>(s, cd, tx, box, m, alpha, tf); };
    CandStream<KO, decltype(reach)> st{W, lo, count, reach};
    int head = 0, n = 0;
    for (;;) {
      Cand cd;
      const bool more = st.next(cd);
      if (more) {
        Path3<KO> g;
        path3_geometry<MODE, KO>(s, tx, q, cd, alpha, g);
        const bool take = live && !path3_negligible<MODE>(g, gk[KO], floor);
        const unsigned b = __ballot_sync(0xffffffffu, take);
        if (take) wq.e[(head + n + __popc(b & ((1u << lane) - 1u))) & 63] = entry_of(cd, lane);
        n += __popc(b);
        __syncwarp();
      }
      const int take = n >= 32 ? 32 : more ? 0 : n;
      if (take) {
        flush_paths3<MODE, KO>(s, W, tx, q, floor, alpha, gk[KO], wq, head, take);
        head = (head + take) & 63;
        n -= take;
      }
      if (!more) break;
    }
  });
  __syncwarp();
  return wq.acc[lane];
}

}  // namespace drt
