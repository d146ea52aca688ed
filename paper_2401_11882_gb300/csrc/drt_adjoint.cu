// Hand-written adjoint (reverse mode) of the forward pass: the vector-Jacobian
// product  sum_r g_r dP_r / d(tx, walls)  (Sec. III: gradient of the loss with
// respect to the scene parameters).
//
// Each (receiver, candidate) recomputes its image chain, reflection points, legs
// and validity, then runs two sweeps over the walls.  Sweep 1 rebuilds each
// leg's visibility; a path with a factor of exactly 0 has no gradient and stops
// there, so sweep 2 never divides by zero (for the sigmoid the forward can keep the
// visibilities instead, and the SAVED variants read them in place of sweep 1).  Sweep
// 2 recomputes each factor and pushes its adjoint into the vertices, the leg normals
// and the wall.  The vertex and leg adjoints then flow back through the leg lengths,
// the validity, the backtrace and the image chain to the transmitter.
//
// A unit is a tile of receivers x a chunk of candidates; warps take their units from
// a counter (work stealing) and store each unit's TX adjoint.  The hard sigmoid, the
// step and the sigmoid with the wall gradient (drt_adjoint_pair.cu) go through
// drt_vjp_walk.cuh, which queues the paths that have a gradient: their lanes hold
// queued paths.  In the sigmoid's other forms (without the wall gradient, or one
// receiver a lane) the lanes hold 32 receivers of one candidate at a time, and paths
// below FLOOR_VJP of the forward's floors are left out where a whole warp's are (128
// walls x 4096 receivers, GB300: transmitter only 99 -> 56 ms, one receiver a lane 94 ->
// 47).  Per-wall adjoints are summed over the warp with shuffles (only when a lane has a
// non-zero one), added into a per-CTA shared-memory table, and written per CTA; a last
// kernel adds the CTA tables in a fixed order, adds the units' TX adjoints in a fixed
// order, and chains the per-wall quantities (n, c, t0, len) back to the end points.
#include <cuda_runtime.h>

#include "drt_common.cuh"
#include "drt_internal.h"
#include "drt_path_vjp.cuh"
#include "drt_path_vjp_pair.cuh"
#include "drt_vjp_walk.cuh"

namespace drt {

namespace {

// SAVED: the sigmoid's leg visibilities come from a.saved (the forward's) instead
// of the first wall sweep.
// With the wall gradient two CTAs an SM are asked for: left to itself the compiler gave the
// sigmoid with saved visibilities 149 registers, one CTA (128 walls x 1024 receivers,
// K = 2, GB300: 25.0 ms, with two 16.8).
template <int MODE, bool WG, bool SAVED = false>
__global__ void __launch_bounds__(256, MODE == MODE_SIGMOID && !WG ? 0 : 2)
    vjp_kernel(const VjpArgs a) {
  extern __shared__ float4 smem[];
  __shared__ VjpQueue queues[MODE == MODE_SIGMOID ? 1 : 8];
  const float2 tx = make_float2(__ldg(a.tx), __ldg(a.tx + 1));
  VSmem s;
  s.G = smem;
  s.E = smem + a.W;
  s.T = smem + 2 * a.W;
  s.H = smem + 3 * a.W;
  s.acc = reinterpret_cast<float*>(smem + 4 * a.W);
  stage_walls<MODE>(a.walls, a.W, tx, a.alpha, SmemWalls{s.G, s.E, s.T, s.H});
  if (WG)
    for (int i = threadIdx.x; i < a.W * VJP_SLOTS; i += blockDim.x) s.acc[i] = 0.f;
  __syncthreads();

  const int lane = threadIdx.x & 31;
  const long long warps_per_cta = blockDim.x >> 5;
  const long long gwarp = (long long)blockIdx.x * warps_per_cta + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * warps_per_cta;
  for (long long u = gwarp; u < a.n_units; u = next_unit_of(a.unit_counter, u, nwarps, lane)) {
    const long long tile = u % a.n_tiles;
    const long long chunk = u / a.n_tiles;
    long long r = tile * 32 + lane;
    const bool live = r < a.R;
    if (!live) r = a.R - 1;
    const float g = live ? __ldg(a.grad_power + r) : 0.f;
    float ux = 0.f, uy = 0.f;
    if (!__all_sync(FULL, g == 0.f)) {
      const float2 q = __ldg(reinterpret_cast<const float2*>(a.rx) + r);
      const long long c0 = chunk * a.chunk;
      const long long c1 = min(c0 + (long long)a.chunk, a.n_cand);
      if constexpr (MODE != MODE_SIGMOID) {
        walk_vjp<MODE, WG, false>(s, a.W, a.K, tx, VjpRx{q, g, 0.f, 0.f}, live, a.alpha, a.gk,
                                  (int)c0, (int)(c1 - c0), queues[threadIdx.x >> 5], nullptr, ux, uy);
      } else {
        // paths below FLOOR_VJP of the forward's floor are left out: whole candidates by
        // the tile's bound, paths by their own values
        const SmemWalls sw{s.G, s.E, s.T, s.H};
        const float floor = FLOOR_VJP * receiver_floor<MODE, false, false>(sw, a.W, tx, q, a.alpha,
                                                                           a.gk[1], a.n_cand);
        const bool on = g != 0.f;
        const TileFloor tf{warp_min(on ? floor : INFINITY), a.gk, false};
        for_reaching_candidates<MODE>(
            sw, a.W, a.K, tx, tile_box(q, on, q, false), tf, a.alpha, (int)c0, (int)(c1 - c0),
            [&](auto order, const Cand& cd) {
              constexpr int KO = decltype(order)::value;
              // the forward's saved visibilities, [n_cand][K + 1][R] (or none)
              const float* sv = SAVED ? a.saved + candidate_index<KO>(cd, a.W) * (a.K + 1) * a.R + r
                                      : nullptr;
              path_vjp<MODE, KO, WG, true>(s, a.W, tx, q, cd, a.alpha, a.gk[KO], g, ux, uy, nullptr, sv,
                                           a.R, nullptr, __fdividef(floor, fmaxf(a.gk[KO], 1e-30f)));
            });
      }
    }
    unit_tx_done(a, u, lane, ux, uy);
  }
  if (WG) {
    __syncthreads();
    float* out = a.cta_walls + (size_t)blockIdx.x * a.W * VJP_SLOTS;
    for (int i = threadIdx.x; i < a.W * VJP_SLOTS; i += blockDim.x) out[i] = s.acc[i];
  }
}

// Adjoint of the min-power loss: loss = -P[argmin], so the gradient is
// -grad_loss * dP[argmin]/d(tx, walls) for one receiver.  A unit is a.chunk (1..32)
// consecutive candidates, as few as fill the chip's warps: the lanes test one
// candidate's validity each, then the warp takes the valid ones in turn with its lanes
// holding the walls (path_vjp_by_walls).  Bound by the latency of one path's chain.
// Measured (4097 sequences, 64 walls, GB300): 29 us with the sigmoid, against 91 us
// with 32 candidates per warp, each lane walking all walls.
template <int MODE, bool WG>
__global__ void __launch_bounds__(256) vjp_rx_kernel(const VjpArgs a) {
  extern __shared__ float4 smem[];
  const float2 tx = make_float2(__ldg(a.tx), __ldg(a.tx + 1));
  VSmem s;
  s.G = smem;
  s.E = smem + a.W;
  s.T = smem + 2 * a.W;
  s.H = smem + 3 * a.W;
  s.acc = reinterpret_cast<float*>(smem + 4 * a.W);
  stage_walls<MODE>(a.walls, a.W, tx, a.alpha, SmemWalls{s.G, s.E, s.T, s.H});
  if (WG)
    for (int i = threadIdx.x; i < a.W * VJP_SLOTS; i += blockDim.x) s.acc[i] = 0.f;
  __syncthreads();

  int ri = __ldg(a.rx_index);
  ri = ri < 0 ? 0 : (ri >= a.R ? (int)a.R - 1 : ri);
  const float2 q = __ldg(reinterpret_cast<const float2*>(a.rx) + ri);
  const float g = -(a.grad_loss ? __ldg(a.grad_loss) : 1.0f);
  const int lane = threadIdx.x & 31;
  const long long warps_per_cta = blockDim.x >> 5;
  const long long gwarp = (long long)blockIdx.x * warps_per_cta + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * warps_per_cta;
  float txb_x = 0.f, txb_y = 0.f;
  auto valid = [&](auto order, const Cand& cd) {
    constexpr int K = decltype(order)::value;
    VjpPath<K> P;
    vjp_recompute<MODE, K>(s, tx, q, cd, a.alpha, P);
    bool v = !P.degenerate;
#pragma unroll
    for (int j = 1; j <= K; ++j) v &= P.V[j] != 0.f;
    return v;
  };
  for (long long u = gwarp; u < a.n_units && g != 0.f; u += nwarps) {
    const long long c = u * a.chunk + lane;
    const bool in = lane < a.chunk && c < a.n_cand;
    const Cand mine = decode_candidate(in ? c : a.n_cand - 1, a.W, a.K);
    bool ok = in;
    switch (mine.k) {
      case 0: ok = ok && valid(Order<0>{}, mine); break;
      case 1: ok = ok && valid(Order<1>{}, mine); break;
      case 2: ok = ok && valid(Order<2>{}, mine); break;
      default: ok = ok && valid(Order<3>{}, mine); break;
    }
    unsigned todo = __ballot_sync(FULL, ok);
    while (todo) {
      const int i = __ffs(todo) - 1;
      todo &= todo - 1;
      Cand cd;
      cd.k = __shfl_sync(FULL, mine.k, i);
#pragma unroll
      for (int j = 0; j < KMAX; ++j) cd.w[j] = __shfl_sync(FULL, mine.w[j], i);
      switch (cd.k) {
        case 0: path_vjp_by_walls<MODE, 0, WG>(s, a.W, tx, q, cd, a.alpha, a.gk[0], g, txb_x, txb_y); break;
        case 1: path_vjp_by_walls<MODE, 1, WG>(s, a.W, tx, q, cd, a.alpha, a.gk[1], g, txb_x, txb_y); break;
        case 2: path_vjp_by_walls<MODE, 2, WG>(s, a.W, tx, q, cd, a.alpha, a.gk[2], g, txb_x, txb_y); break;
        default: path_vjp_by_walls<MODE, 3, WG>(s, a.W, tx, q, cd, a.alpha, a.gk[3], g, txb_x, txb_y); break;
      }
    }
  }
  if (lane == 0) {
    a.warp_tx[2 * gwarp] = txb_x;
    a.warp_tx[2 * gwarp + 1] = txb_y;
  }
  if (WG) {
    __syncthreads();
    float* out = a.cta_walls + (size_t)blockIdx.x * a.W * VJP_SLOTS;
    for (int i = threadIdx.x; i < a.W * VJP_SLOTS; i += blockDim.x) out[i] = s.acc[i];
  }
}

// Sums the per-CTA wall tables and the TX partials in a fixed order and chains
// (n, c, t0, len) back to the end points A, B of each wall:
//   u = (B - A)/|B - A|, n = (-u_y, u_x), c = n . A, t0 = u . A.
// Block w < W takes wall w, one warp per slot whose lanes stride over the CTAs; the
// last block takes the TX.  Bound by the latency of its loads: one thread per wall
// walking the CTA tables in one block took 200 us for 128 walls x 304 CTAs and 130k
// units.
constexpr int FINALIZE_THREADS = 32 * VJP_SLOTS;
__global__ void __launch_bounds__(FINALIZE_THREADS) vjp_finalize_kernel(const VjpArgs a, int n_ctas,
                                                                        int n_warps, int n_walls) {
  __shared__ float acc[VJP_SLOTS];
  __shared__ float sx[VJP_SLOTS], sy[VJP_SLOTS];
  const int lane = threadIdx.x & 31, slot = threadIdx.x >> 5;
  if ((int)blockIdx.x < n_walls) {
    const int w = blockIdx.x;
    float v = 0.f;
#pragma unroll 4
    for (int c = lane; c < n_ctas; c += 32)
      v += __ldg(a.cta_walls + ((size_t)c * a.W + w) * VJP_SLOTS + slot);
    v = warp_sum(v);
    if (lane == 0) acc[slot] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      const float4 ab = a.walls[w];
      const WallGeom g = wall_geometry(ab);
      const float nx = g.G.x, ny = g.G.y, len = g.G.w;
      const float ux = ny, uy = -nx;
      float nbx = acc[S_NX], nby = acc[S_NY];
      float Abx = acc[S_AX], Aby = acc[S_AY], Bbx = acc[S_BX], Bby = acc[S_BY];
      // c = n . A
      nbx = fmaf(acc[S_C], ab.x, nbx);
      nby = fmaf(acc[S_C], ab.y, nby);
      Abx = fmaf(acc[S_C], nx, Abx);
      Aby = fmaf(acc[S_C], ny, Aby);
      // t0 = u . A
      float ubx = acc[S_T0] * ab.x, uby = acc[S_T0] * ab.y;
      Abx = fmaf(acc[S_T0], ux, Abx);
      Aby = fmaf(acc[S_T0], uy, Aby);
      // n = (-u_y, u_x)
      ubx += nby;
      uby -= nbx;
      // u = e / len, len = |e|, e = B - A
      const float uu = fmaf(ubx, ux, uby * uy);
      const float ebx = fmaf(acc[S_LEN], ux, (ubx - uu * ux) / len);
      const float eby = fmaf(acc[S_LEN], uy, (uby - uu * uy) / len);
      Abx -= ebx;
      Aby -= eby;
      Bbx += ebx;
      Bby += eby;
      reinterpret_cast<float4*>(a.grad_walls)[w] = make_float4(Abx, Aby, Bbx, Bby);
    }
    return;
  }
  float x = 0.f, y = 0.f;
  // per-unit TX adjoints (the receiver-tile kernels) or per-warp ones
  const float* parts = a.unit_tx ? a.unit_tx : a.warp_tx;
  const long long n_parts = a.unit_tx ? a.n_units : n_warps;
#pragma unroll 4
  for (long long i = threadIdx.x; i < n_parts; i += FINALIZE_THREADS) {
    x += parts[2 * i];
    y += parts[2 * i + 1];
  }
  x = warp_sum(x);
  y = warp_sum(y);
  if (lane == 0) {
    sx[slot] = x;
    sy[slot] = y;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < VJP_SLOTS; ++i) {
      x += sx[i];
      y += sy[i];
    }
    a.grad_tx[0] = x;
    a.grad_tx[1] = y;
  }
}

template <int MODE, bool WG>
void launch_vjp_t(const VjpArgs& a, int ctas, int threads, size_t smem, cudaStream_t st) {
  if (a.rx_index)
    vjp_rx_kernel<MODE, WG><<<ctas, threads, smem, st>>>(a);
  else if (MODE == MODE_SIGMOID && a.saved)
    vjp_kernel<MODE, WG, true><<<ctas, threads, smem, st>>>(a);
  else
    vjp_kernel<MODE, WG><<<ctas, threads, smem, st>>>(a);
}

}  // namespace

cudaError_t launch_vjp_finalize(const VjpArgs& a, int ctas, int threads, cudaStream_t st) {
  const int n_walls = a.grad_walls ? a.W : 0;
  vjp_finalize_kernel<<<n_walls + 1, FINALIZE_THREADS, 0, st>>>(a, ctas, ctas * (threads / 32),
                                                                n_walls);
  return cudaGetLastError();
}

size_t vjp_smem_bytes(int W, bool wall_grad, bool pairs) {
  return (size_t)(pairs ? 9 : 4) * W * sizeof(float4) +
         (wall_grad ? (size_t)W * VJP_SLOTS * sizeof(float) : 0);
}

bool vjp_uses_pairs(int mode, int flags) {
  return mode == MODE_SIGMOID && !(flags & DRT_TILE_SINGLE_RX);
}

cudaError_t launch_vjp(const VjpArgs& a, int mode, int ctas, int threads, cudaStream_t st) {
  const bool wg = a.grad_walls != nullptr;
  const size_t smem = vjp_smem_bytes(a.W, wg, a.pairs && !a.rx_index && wg);
  if (!a.rx_index && a.unit_counter) {   // the receiver-tile kernels steal work
    cudaError_t e = cudaMemsetAsync(a.unit_counter, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
  }
  if (a.pairs && !a.rx_index && mode == MODE_SIGMOID && wg) {
    launch_vjp_pair(a, ctas, threads, smem, st);
  } else
  switch (mode * 2 + (wg ? 1 : 0)) {
    case MODE_SIGMOID * 2: launch_vjp_t<MODE_SIGMOID, false>(a, ctas, threads, smem, st); break;
    case MODE_SIGMOID * 2 + 1: launch_vjp_t<MODE_SIGMOID, true>(a, ctas, threads, smem, st); break;
    case MODE_HARD * 2: launch_vjp_t<MODE_HARD, false>(a, ctas, threads, smem, st); break;
    case MODE_HARD * 2 + 1: launch_vjp_t<MODE_HARD, true>(a, ctas, threads, smem, st); break;
    case MODE_STEP * 2: launch_vjp_t<MODE_STEP, false>(a, ctas, threads, smem, st); break;
    default: launch_vjp_t<MODE_STEP, true>(a, ctas, threads, smem, st); break;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_vjp_finalize(a, ctas, threads, st);
}

cudaError_t vjp_occupancy(int mode, bool wg, bool pairs, int threads, int W, int* ctas_per_sm) {
  const size_t smem = vjp_smem_bytes(W, wg, pairs);
  if (pairs && mode == MODE_SIGMOID && wg)
    return vjp_pair_occupancy(threads, smem, ctas_per_sm);
  switch (mode * 2 + (wg ? 1 : 0)) {
    case MODE_SIGMOID * 2:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, vjp_kernel<MODE_SIGMOID, false>, threads, smem);
    case MODE_SIGMOID * 2 + 1:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, vjp_kernel<MODE_SIGMOID, true>, threads, smem);
    case MODE_HARD * 2:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, vjp_kernel<MODE_HARD, false>, threads, smem);
    case MODE_HARD * 2 + 1:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, vjp_kernel<MODE_HARD, true>, threads, smem);
    case MODE_STEP * 2:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, vjp_kernel<MODE_STEP, false>, threads, smem);
    default:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, vjp_kernel<MODE_STEP, true>, threads, smem);
  }
}

cudaError_t vjp_set_smem_limit(int W) {
  const int s0 = (int)vjp_smem_bytes(W, false, false), s1 = (int)vjp_smem_bytes(W, true, false);
  cudaError_t e = cudaSuccess;
  e = vjp_pair_set_smem_limit((int)vjp_smem_bytes(W, true, true));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(vjp_kernel<MODE_SIGMOID, true, true>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, s1);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(vjp_kernel<MODE_SIGMOID, false, true>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, s0);
  if (e != cudaSuccess) return e;
#define DRT_SET(M, B, S)                                                                    \
  e = cudaFuncSetAttribute(vjp_kernel<M, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, S); \
  if (e != cudaSuccess) return e;                                                           \
  e = cudaFuncSetAttribute(vjp_rx_kernel<M, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, S); \
  if (e != cudaSuccess) return e;
  DRT_SET(MODE_SIGMOID, false, s0)
  DRT_SET(MODE_SIGMOID, true, s1)
  DRT_SET(MODE_HARD, false, s0)
  DRT_SET(MODE_HARD, true, s1)
  DRT_SET(MODE_STEP, false, s0)
  DRT_SET(MODE_STEP, true, s1)
#undef DRT_SET
  return field_vjp_set_smem_limit(s0, s1);
}

}  // namespace drt
