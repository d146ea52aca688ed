// Coherent field per receiver: Eq. 7 read as a sum of complex path fields,
//   E_r = sum over candidates of  prod_j C_j * V * vis * exp(-2 pi i L / lambda) / L,
// with the field normal to the scene plane, C_j the Fresnel reflection
// coefficient for that polarisation (TE) at the angle of incidence of the leg
// arriving at reflection j, or a constant amplitude coefficient, and the
// coherent power |E_r|^2.
//
// The geometry, validity and obstruction of each (receiver, candidate) are the
// forward pass's (path_geometry, leg_visibility): the obstruction loop is the
// cost and is unchanged.  Only the per-path epilogue differs: it recomputes the
// path length with correctly rounded leg lengths (the phase 2 pi L / lambda
// magnifies any error in L by L / lambda), takes 1/lambda as a float pair so
// the cycle count's only rounding is L's own, and reduces the cycle count to
// [-1/2, 1/2] before sincospi.  Work decomposition, determinism and the chunk
// reduction follow drt_forward.cu with (re, im) partial sums, including its two
// receivers per lane (packed FP32 obstruction loop) for the hard sigmoid and the
// sigmoid at alpha <= 1e4; the visibilities are the same, bit for bit, either way.
#include <cuda_runtime.h>

#include "drt_common.cuh"
#include "drt_internal.h"
#include "drt_path.cuh"
#include "drt_path_pair.cuh"
#include "drt_path_queue.cuh"

namespace drt {

namespace {

// Field (re, im) of one path from its geometry and its legs' visibilities.
template <int MODE, int K>
__device__ __forceinline__ float2 field_of_path(const SmemWalls& s, const FieldArgs& a,
                                                const PathGeom<MODE, K>& g, const float* vis,
                                                const Cand& cd) {
  // Only L needs correctly rounded arithmetic (the phase); the amplitude's factors
  // take the approximate reciprocal square root and division (a few ulps each,
  // far inside the amplitude's tolerance).
  float L = 0.f, coef = 1.f, amp = g.V;
#pragma unroll
  for (int j = 0; j <= K; ++j) {
    const float dx = g.Qx[j + 1] - g.Qx[j], dy = g.Qy[j + 1] - g.Qy[j];
    const float len2 = fmaf(dx, dx, dy * dy);
    L += __fsqrt_rn(len2);
    amp *= vis[j];
    if (j < K) {
      // leg j arrives at reflection j + 1 on wall w_{j+1}: cosine of incidence
      // |n . d| / |d| with n the wall's unit normal
      const float4 G = s.G[cd.w[j]];
      const float c = fminf(fabsf(fmaf(G.x, dx, G.y * dy)) * rsqrtf(len2), 1.f);
      float r = a.refl_amp;
      if (a.eps_r > 0.f) {
        const float x = fmaf(c, c, a.eps_r - 1.f);
        const float root = x > 0.f ? x * rsqrtf(x) : 0.f;
        const float den = c + root;
        r = den > 0.f ? __fdividef(c - root, den) : 0.f;   // den >= sqrt(eps_r - 1) > 0
      }
      coef *= r;
    }
  }
  // cycles L / lambda = L * (hi + lo): the product's rounding error is recovered
  // by an FMA, so the fractional part carries only L's own error
  const float p = L * a.inv_lambda_hi;
  const float e = fmaf(L, a.inv_lambda_hi, -p);
  const float frac = (p - rintf(p)) + fmaf(L, a.inv_lambda_lo, e);
  float sn, cs;
  sincospif(2.f * frac, &sn, &cs);
  const float m = __fdividef(amp * coef, L);
  return g.degenerate ? make_float2(0.f, 0.f) : make_float2(m * cs, -m * sn);
}

// The path's field, or 0 where its amplitude before the reflection coefficients' exact
// values (ck bounds their product) is below the receiver's floor.  keep: whether it is
// above share times the floor.
template <int MODE, int K>
__device__ __forceinline__ float2 field_above(const SmemWalls& s, const FieldArgs& a,
                                              const PathGeom<MODE, K>& g, const float* vis,
                                              const Cand& cd, bool none, float floor,
                                              float share = 1.f, bool* keep = nullptr) {
  const float2 f = field_of_path<MODE, K>(s, a, g, vis, cd);
  float amp = g.V * a.ck[K];
#pragma unroll
  for (int j = 0; j <= K; ++j) amp *= vis[j];
  if (keep) *keep = !(none || amp == 0.f || amp < share * floor * g.L);
  return none || amp < floor * g.L ? make_float2(0.f, 0.f) : f;
}

// Field of one path candidate of order K for this lane's receiver.
template <int MODE, int K, bool MASKED>
__device__ __forceinline__ float2 path_field(const SmemWalls& s, const FieldArgs& a, float2 tx,
                                             float2 rx, const Cand& cd, float floor,
                                             float* vis_out = nullptr) {
  float Ix[K + 1], Iy[K + 1];
  tx_images<K>(s, tx, cd, Ix, Iy);
  PathGeom<MODE, K> g;
  path_geometry<MODE, K>(s, Ix, Iy, tx, rx, cd, a.alpha, g);
  const bool none = path_negligible<MODE, true>(g, a.ck[K], floor);
  if (!vis_out && __all_sync(0xffffffffu, none)) return make_float2(0.f, 0.f);
  float vis[K + 1];
  const float min_div =
      leg_visibility<MODE, K, MASKED>(s, a.W, cd, g.Qx, g.Qy, g.mx, g.my, g.mc, vis);
  if constexpr (!MASKED && MODE != MODE_STEP) redo_masked<MODE, K>(s, a.W, cd, g, min_div, vis);
  if (vis_out) {
#pragma unroll
    for (int j = 0; j <= K; ++j) vis_out[j] = vis[j];
  }
  return field_above<MODE, K>(s, a, g, vis, cd, none, floor);
}

// Fields of two paths of order K per lane (hard sigmoid or sigmoid): the packed
// obstruction loop of path_power_pair.
// SAVED (the walk's saving evaluation): the floors passed are FLOOR_VJP of the sums'.
template <int MODE, int K, bool SAVED = false, int UNROLL = SIG_UNROLL>
__device__ __forceinline__ void path_field_pair(const SmemWalls& s, const SmemPairs& p,
                                                const FieldArgs& a, float2 tx, float2 rx0,
                                                const Cand& cd0, float floor0, float2 rx1,
                                                const Cand& cd1, float floor1, float2& f0,
                                                float2& f1, float2* vis_out = nullptr,
                                                bool* keep0 = nullptr, bool* keep1 = nullptr) {
  float Ix[K + 1], Iy[K + 1];
  PathGeom<MODE, K> g0, g1;
  tx_images<K>(s, tx, cd0, Ix, Iy);
  path_geometry<MODE, K>(s, Ix, Iy, tx, rx0, cd0, a.alpha, g0);
  tx_images<K>(s, tx, cd1, Ix, Iy);
  path_geometry<MODE, K>(s, Ix, Iy, tx, rx1, cd1, a.alpha, g1);
  float vis0[K + 1], vis1[K + 1];
  float2 stop = make_float2(0.f, 0.f);
  if (MODE == MODE_SIGMOID && (!vis_out || SAVED))
    stop = make_float2(stop_of<MODE, true>(g0, a.ck[K], floor0), stop_of<MODE, true>(g1, a.ck[K], floor1));
  path_visibility_pair<MODE, K, UNROLL>(s, p, a.W, g0, cd0, g1, cd1, vis0, vis1, stop);
  if (vis_out) {
#pragma unroll
    for (int j = 0; j <= K; ++j) vis_out[j] = f2(vis0[j], vis1[j]);
  }
  constexpr float SHARE = SAVED ? FLOOR_VJP : 1.f;
  f0 = field_above<MODE, K>(s, a, g0, vis0, cd0, path_negligible<MODE, true>(g0, a.ck[K], floor0),
                            floor0 * (1.f / SHARE), SHARE, keep0);
  f1 = field_above<MODE, K>(s, a, g1, vis1, cd1, path_negligible<MODE, true>(g1, a.ck[K], floor1),
                            floor1 * (1.f / SHARE), SHARE, keep1);
}

// Stage 3 of the walk (drt_path_queue.cuh): the fields of two queued paths per lane.
// SAVE: the visibilities of the paths that count for the adjoint are kept too.
template <int MODE, bool SAVE>
struct FieldEval {
  static constexpr bool FLOORS = MODE == MODE_SIGMOID, SAVES = SAVE;
  static constexpr float FLOOR = SAVE ? FLOOR_VJP : 1.f;
  const SmemWalls& s;
  const SmemPairs& p;
  const FieldArgs& a;
  float2 tx;
  const float* ck;
  SavedVis saved;
  template <int K, int UNROLL = SIG_UNROLL>
  __device__ __forceinline__ void operator()(const QueuedPath& q0, const QueuedPath& q1, float2& v0,
                                             float2& v1) const {
    // the sum takes what the plain field's takes; SAVE keeps the visibilities further down
    float2 vis[K + 1];
    bool keep0 = false, keep1 = false;
    path_field_pair<MODE, K, SAVE, UNROLL>(s, p, a, tx, q0.rx, q0.cd, q0.floor, q1.rx, q1.cd, q1.floor, v0,
                                   v1, SAVE ? vis : nullptr, &keep0, &keep1);
    if (SAVE) {
      float va[K + 1], vb[K + 1];
#pragma unroll
      for (int j = 0; j <= K; ++j) {
        va[j] = vis[j].x;
        vb[j] = vis[j].y;
      }
      if (keep0) saved.put<K>(q0, va);
      if (keep1) saved.put<K>(q1, vb);
    }
  }
};

template <int MODE, bool MASKED>
__device__ __forceinline__ float2 field_of(const SmemWalls& s, const FieldArgs& a, float2 tx,
                                           float2 q, const Cand& cd, float floor,
                                           float* vis_out) {
  switch (cd.k) {
    case 0: return path_field<MODE, 0, MASKED>(s, a, tx, q, cd, floor, vis_out);
    case 1: return path_field<MODE, 1, MASKED>(s, a, tx, q, cd, floor, vis_out);
    case 2: return path_field<MODE, 2, MASKED>(s, a, tx, q, cd, floor, vis_out);
    default: return path_field<MODE, 3, MASKED>(s, a, tx, q, cd, floor, vis_out);
  }
}

// One receiver per lane; a unit is (32 receivers) x (a chunk of candidates), as in
// the forward kernel, with one (re, im) partial sum per (chunk, receiver).  SAVE
// (sigmoid): every path's leg visibilities also go to a.saved, as drt_forward_save
// writes them (the same values: the same obstruction loops).
template <int MODE, bool SAVE = false>
__global__ void __launch_bounds__(256, MODE == MODE_SIGMOID ? 2 : 3) field_kernel(const FieldArgs a) {
  extern __shared__ float4 smem[];
  SmemWalls s{smem, smem + a.W, smem + 2 * a.W, smem + 3 * a.W};
  const float2 tx = make_float2(__ldg(a.tx), __ldg(a.tx + 1));
  stage_walls<MODE>(a.walls, a.W, tx, a.alpha, s);
  __syncthreads();

  const int lane = threadIdx.x & 31;
  const long long warps_per_cta = blockDim.x >> 5;
  const long long nwarps = (long long)gridDim.x * warps_per_cta;
  const bool masked = a.alpha > FAST_SKIP_MAX_ALPHA;
  for (long long u = (long long)blockIdx.x * warps_per_cta + (threadIdx.x >> 5); u < a.n_units;
       u = next_unit_of(a.unit_counter, u, nwarps, lane)) {
    const long long tile = u % a.n_tiles;
    const long long chunk = u / a.n_tiles;
    long long r = tile * 32 + lane;
    const bool live = r < a.R;
    if (!live) r = a.R - 1;
    const float2 q = __ldg(reinterpret_cast<const float2*>(a.rx) + r);
    const int c0 = (int)(chunk * a.chunk);
    const int nc = (int)(min(c0 + (long long)a.chunk, a.n_cand) - c0);
    float2 acc = make_float2(0.f, 0.f);
    const float floor =
        masked ? receiver_floor<MODE, true, true>(s, a.W, tx, q, a.alpha, a.ck[1], a.n_cand)
               : receiver_floor<MODE, true, false>(s, a.W, tx, q, a.alpha, a.ck[1], a.n_cand);
    auto add = [&](const Cand& cd, float* vo) {
      const float2 f = masked ? field_of<MODE, true>(s, a, tx, q, cd, floor, vo)
                              : field_of<MODE, false>(s, a, tx, q, cd, floor, vo);
      acc.x += f.x;
      acc.y += f.y;
    };
    if (SAVE) {
      float vbuf[KMAX + 1];   // the path's leg visibilities
      Cand cd = decode_candidate(c0, a.W, a.K);
      for (int i = 0; i < nc; ++i) {
        if (i > 0) next_candidate(cd, a.W);
#pragma unroll
        for (int j = 0; j <= KMAX; ++j) vbuf[j] = 0.f;
        add(cd, vbuf);
        if (live) {   // [n_cand][K + 1][R]
          float* dst = a.saved + (long long)(c0 + i) * (a.K + 1) * a.R + r;
          for (int j = 0; j <= cd.k; ++j) dst[j * a.R] = vbuf[j];
        }
      }
    } else {
      const TileFloor tf{MODE == MODE_SIGMOID ? warp_min(live ? floor : INFINITY) : 0.f, a.ck, true};
      for_reaching_candidates<MODE>(s, a.W, a.K, tx, tile_box(q, live, q, false), tf, a.alpha, c0, nc,
                                    [&](auto, const Cand& cd) { add(cd, nullptr); });
    }
    if (live) a.partial[chunk * a.R + r] = acc;
  }
}

// Hard sigmoid and sigmoid, two receivers per lane: lane l holds receivers l and
// l + 32 of its 64-receiver tile; the walls' paired records follow the four
// single-receiver arrays in shared memory.
template <int MODE, int SAVE = SAVE_NONE>
__global__ void __launch_bounds__(256, 2) field_pair_kernel(const FieldArgs a) {
  extern __shared__ float4 smem[];
  __shared__ WarpQueue<float2> queues[SAVE == SAVE_ALL ? 1 : 8];
  SmemWalls s{smem, smem + a.W, smem + 2 * a.W, smem + 3 * a.W};
  SmemPairs pr{smem + 4 * a.W, smem + 5 * a.W, smem + 6 * a.W, smem + 7 * a.W};
  const float2 tx = make_float2(__ldg(a.tx), __ldg(a.tx + 1));
  stage_walls<MODE>(a.walls, a.W, tx, a.alpha, s);
  __syncthreads();
  stage_pairs<MODE>(s, a.W, pr);
  __syncthreads();

  const int lane = threadIdx.x & 31;
  const long long warps_per_cta = blockDim.x >> 5;
  const long long nwarps = (long long)gridDim.x * warps_per_cta;
  for (long long u = (long long)blockIdx.x * warps_per_cta + (threadIdx.x >> 5); u < a.n_units;
       u = next_unit_of(a.unit_counter, u, nwarps, lane)) {
    const long long tile = u % a.n_tiles;
    const long long chunk = u / a.n_tiles;
    const long long r0 = tile * 64 + lane, r1 = r0 + 32;
    const bool live0 = r0 < a.R, live1 = r1 < a.R;
    const float2 q0 = __ldg(reinterpret_cast<const float2*>(a.rx) + (live0 ? r0 : a.R - 1));
    const float2 q1 = __ldg(reinterpret_cast<const float2*>(a.rx) + (live1 ? r1 : a.R - 1));
    const int c0 = (int)(chunk * a.chunk);
    const int nc = (int)(min(c0 + (long long)a.chunk, a.n_cand) - c0);
    float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
    if (SAVE == SAVE_ALL) {
      const float floor0 = receiver_floor<MODE, true, false>(s, a.W, tx, q0, a.alpha, a.ck[1], a.n_cand);
      const float floor1 = receiver_floor<MODE, true, false>(s, a.W, tx, q1, a.alpha, a.ck[1], a.n_cand);
      float2 vbuf[KMAX + 1];   // the paths' leg visibilities
      Cand cd = decode_candidate(c0, a.W, a.K);
      for (int i = 0; i < nc; ++i) {
        if (i > 0) next_candidate(cd, a.W);
#pragma unroll
        for (int j = 0; j <= KMAX; ++j) vbuf[j] = make_float2(0.f, 0.f);
        float2 f0, f1;
        switch (cd.k) {
          case 0: path_field_pair<MODE, 0, false, SIG_UNROLL_ALL>(s, pr, a, tx, q0, cd, floor0, q1, cd, floor1, f0, f1, vbuf); break;
          case 1: path_field_pair<MODE, 1, false, SIG_UNROLL_ALL>(s, pr, a, tx, q0, cd, floor0, q1, cd, floor1, f0, f1, vbuf); break;
          case 2: path_field_pair<MODE, 2, false, SIG_UNROLL_ALL>(s, pr, a, tx, q0, cd, floor0, q1, cd, floor1, f0, f1, vbuf); break;
          default: path_field_pair<MODE, 3, false, SIG_UNROLL_ALL>(s, pr, a, tx, q0, cd, floor0, q1, cd, floor1, f0, f1, vbuf); break;
        }
        acc0.x += f0.x;
        acc0.y += f0.y;
        acc1.x += f1.x;
        acc1.y += f1.y;
        // [n_cand][K + 1][R]
        float* dst = a.saved + (long long)(c0 + i) * (a.K + 1) * a.R;
        for (int j = 0; j <= cd.k; ++j) {
          if (live0) dst[j * a.R + r0] = vbuf[j].x;
          if (live1) dst[j * a.R + r1] = vbuf[j].y;
        }
      }
    } else {
      WarpQueue<float2>& wq = queues[threadIdx.x >> 5];
      walk_valid_paths<MODE, true>(s, a.W, a.K, tx, q0, live0, q1, live1, a.alpha, a.n_cand, c0, nc,
                                   wq, FieldEval<MODE, SAVE == SAVE_COUNTING>{
                                           s, pr, a, tx, a.ck,
                                           SavedVis{a.saved + tile * 64, a.R, a.W, a.K}});
      acc0 = wq.acc[lane];
      acc1 = wq.acc[lane + 32];
    }
    if (live0) a.partial[chunk * a.R + r0] = acc0;
    if (live1) a.partial[chunk * a.R + r1] = acc1;
  }
}

// field[r] = sum over chunks of partial[chunk][r], power[r] = |field[r]|^2: 8 threads per
// receiver add a slice of the chunks each, in chunk order, and the slices' sums are added
// in order (as reduce_chunks_kernel).
constexpr int REDUCE_SLICES = 8;
__global__ void __launch_bounds__(256) reduce_field_kernel(const float2* __restrict__ partial,
                                                           long long n_chunks, long long R,
                                                           float2* __restrict__ field,
                                                           float* __restrict__ power) {
  __shared__ float2 sums[REDUCE_SLICES][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const long long per = (n_chunks + REDUCE_SLICES - 1) / REDUCE_SLICES;
  const long long c0 = y * per, c1 = min(c0 + per, n_chunks);
  for (long long r0 = blockIdx.x * 32LL; r0 < R; r0 += gridDim.x * 32LL) {
    const long long r = r0 + x;
    float2 acc = make_float2(0.f, 0.f);
    if (r < R) {
#pragma unroll 8
      for (long long c = c0; c < c1; ++c) acc = value_sum(acc, __ldg(partial + c * R + r));
    }
    sums[y][x] = acc;
    __syncthreads();
    if (y == 0 && r < R) {
#pragma unroll
      for (int i = 1; i < REDUCE_SLICES; ++i) acc = value_sum(acc, sums[i][x]);
      field[r] = acc;
      if (power) power[r] = fmaf(acc.x, acc.x, acc.y * acc.y);
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_field(const FieldArgs& a, int mode, int ctas, int threads, cudaStream_t st) {
  const size_t smem = forward_smem_bytes(a.W, a.pairs);
  if (a.unit_counter && a.n_units > 0) {
    cudaError_t e = cudaMemsetAsync(a.unit_counter, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
  }
  const bool save = a.saved && mode == MODE_SIGMOID;
  if (a.n_units > 0 && a.pairs) {
    if (mode == MODE_SIGMOID && save && a.save_counting) {
      cudaError_t e = clear_saved(a.saved, a.n_cand, a.K, a.R, st);
      if (e != cudaSuccess) return e;
      field_pair_kernel<MODE_SIGMOID, SAVE_COUNTING><<<ctas, threads, smem, st>>>(a);
    } else if (mode == MODE_SIGMOID && save)
      field_pair_kernel<MODE_SIGMOID, SAVE_ALL><<<ctas, threads, smem, st>>>(a);
    else if (mode == MODE_SIGMOID)
      field_pair_kernel<MODE_SIGMOID><<<ctas, threads, smem, st>>>(a);
    else
      field_pair_kernel<MODE_HARD><<<ctas, threads, smem, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  } else if (a.n_units > 0) {
    switch (mode) {
      case MODE_SIGMOID:
        if (save)
          field_kernel<MODE_SIGMOID, true><<<ctas, threads, smem, st>>>(a);
        else
          field_kernel<MODE_SIGMOID><<<ctas, threads, smem, st>>>(a);
        break;
      case MODE_HARD: field_kernel<MODE_HARD><<<ctas, threads, smem, st>>>(a); break;
      default: field_kernel<MODE_STEP><<<ctas, threads, smem, st>>>(a); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (a.R > 0) {
    const long long nb = (a.R + 31) / 32;
    const int rb = (int)(nb < 16384 ? nb : 16384);
    reduce_field_kernel<<<rb, 256, 0, st>>>(a.partial, a.n_chunks, a.R, a.field, a.power);
  }
  return cudaGetLastError();
}

cudaError_t field_occupancy(int mode, bool pairs, int threads, int W, int* ctas_per_sm) {
  const size_t smem = forward_smem_bytes(W, pairs);
  if (pairs)
    return mode == MODE_SIGMOID
               ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                     ctas_per_sm, field_pair_kernel<MODE_SIGMOID>, threads, smem)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                     ctas_per_sm, field_pair_kernel<MODE_HARD>, threads, smem);
  switch (mode) {
    case MODE_SIGMOID:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, field_kernel<MODE_SIGMOID>,
                                                           threads, smem);
    case MODE_HARD:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, field_kernel<MODE_HARD>,
                                                           threads, smem);
    default:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, field_kernel<MODE_STEP>,
                                                           threads, smem);
  }
}

cudaError_t field_set_smem_limit(int W) {
  const int smem = (int)forward_smem_bytes(W, false);
  const int psmem = (int)forward_smem_bytes(W, true);
  cudaError_t e = cudaFuncSetAttribute(field_pair_kernel<MODE_HARD>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, psmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(field_pair_kernel<MODE_SIGMOID>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, psmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(field_pair_kernel<MODE_SIGMOID, SAVE_ALL>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, psmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(field_pair_kernel<MODE_SIGMOID, SAVE_COUNTING>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, psmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(field_kernel<MODE_SIGMOID>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(field_kernel<MODE_SIGMOID, true>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(field_kernel<MODE_HARD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(field_kernel<MODE_STEP>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

}  // namespace drt
