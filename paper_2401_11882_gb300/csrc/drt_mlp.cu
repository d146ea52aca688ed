// Surrogate MLP of the min-power objective over the transmitter position:
// Fourier features (32 frequencies: sin and cos of 2 pi B_j . x), four
// Linear(256) + SiLU layers and Linear(1); BF16 weights and activations, FP32
// accumulation, FP32 master weights trained with Adam.
//
// The dense layers are one GEMM kernel C = A . Bt^T (both operands stored
// K-contiguous) on the tensor cores (mma.sync m16n8k16 BF16 -> FP32, operands
// staged in shared memory and fed by ldmatrix), with three epilogues:
//   FWD: z = acc + bias; store z (FP32), h = SiLU(z) as BF16 row-major and
//        transposed (the transposed copy is the B operand of the weight gradient);
//   DH:  the GEMM is dH = dZ . W; store dZ_prev = dH * SiLU'(z_prev) (BF16, both layouts);
//   DW:  the GEMM is dW = dZ^T . H (K = batch); store FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <utility>

#include "drt.h"
#include "drt_internal.h"

namespace drt {
namespace mlp {

constexpr int NFREQ = DRT_MLP_FREQS;
constexpr int NFEAT = 2 * DRT_MLP_FREQS;
constexpr int WID = DRT_MLP_WIDTH;
constexpr int NL = DRT_MLP_LAYERS;

typedef __nv_bfloat16 bf16;

// Offsets (in floats) of each parameter block in the flat FP32 vector, and
// (in bf16 elements) of the shadow copies.
struct Layout {
  long long w[NL], b[NL], w5, b5, total;
  long long sw[NL], swt[NL], sw5, stotal;
  long long swc[NL];   // W_l in 256 x 32 K-chunks, each in the tensor-core smem layout
  int k[NL];
};

// K-chunk width of the chunked weight copy, and the byte offset of element
// (n, k) of a [256 x 32] chunk in the canonical no-swizzle K-major layout of the
// tcgen05 operands (8-row x 16-byte core matrices, four along K per 8-row group).
constexpr int WCHUNK_K = 32;
__host__ __device__ constexpr unsigned chunk_woff(int n, int k) {
  return (unsigned)((((n >> 3) * (WCHUNK_K / 8) + (k >> 3)) << 7) + ((n & 7) << 4) + ((k & 7) << 1));
}

__host__ __device__ inline Layout layout() {
  Layout L{};
  long long o = 0, so = 0;
  for (int l = 0; l < NL; ++l) {
    L.k[l] = (l == 0) ? NFEAT : WID;
    L.w[l] = o;
    o += (long long)WID * L.k[l];
    L.b[l] = o;
    o += WID;
    L.sw[l] = so;
    so += (long long)WID * L.k[l];
    L.swt[l] = so;
    so += (long long)WID * L.k[l];
  }
  L.w5 = o;
  o += WID;
  L.b5 = o;
  o += 1;
  L.total = o;
  L.sw5 = so;
  so += WID;
  for (int l = 0; l < NL; ++l) {
    L.swc[l] = so;
    so += (long long)WID * L.k[l];
  }
  L.stotal = so;
  return L;
}

enum : int { EPI_FWD = 0, EPI_DH = 1, EPI_DW = 2 };   // EPI_DW: the tcgen05 kernel's

struct GemmArgs {
  const bf16* A;
  int lda;
  const bf16* Bt;
  int ldb;
  int M, N, K;
  const float* bias;   // FWD
  float* Z;            // FWD: out [M][ldz]; DH: in (pre-activation of the layer below)
  int ldz;
  bf16* H;             // FWD: SiLU(z); DH: dZ  [M][ldh]
  int ldh;
  bf16* HT;            // transposed copy [N][ldht] (optional)
  int ldht;
  float* C;            // DW: out [M][ldc]; with split-K, partial z at C + z * M * ldc
  int ldc;
  int k_splits;        // DW: K is split into k_splits equal slices (blockIdx.z), >= 1
};

__device__ __forceinline__ void ldsm_x4(uint32_t* r, const void* smem_ptr) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem_ptr);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ float sigm(float z) { return 1.f / (1.f + expf(-z)); }

// C[M x N] = A[M x K] . Bt[N x K]^T; M, N and each K slice multiples of 64.
// One 64 x 64 tile per CTA of 4 warps (32 x 32 each).  At the training sizes (batch
// 4096, width 256) a layer is 0.5 GFLOP over 256 CTAs: bound by the latency of filling
// the tile, not by the tensor rate, so four 64-wide stages of both operands are in
// flight at once (cp.async; K = 256 is then loaded in one go).  16-bit outputs pass
// through the freed stages so that both layouts are written in 128-byte rows.  Measured
// per launch (batch 4096, 256 x 256, GB300): FWD 17.7 -> 9.7 us, DH 19.9 -> 12.8 us
// against one 32-wide stage loaded between barriers and element stores.
constexpr int GT = 64;            // tile edge and K stage
constexpr int G_STAGES = 4;
constexpr int G_LD = GT + 8;      // padded row (bf16): 144 bytes, conflict-free ldmatrix
constexpr int G_STAGE = 2 * GT * G_LD;   // bf16 per stage (A, then B)
constexpr int G_SMEM = G_STAGES * G_STAGE * (int)sizeof(bf16);

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem));
}

// acc = the tile's product over K in [kbeg, kend)
__device__ __forceinline__ void gemm_tile(const bf16* __restrict__ A, int lda,
                                          const bf16* __restrict__ Bt, int ldb, int m0, int n0,
                                          int kbeg, int kend, bf16* smem, float (*acc)[4][4]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 1, wn = warp & 1;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
  const int n_st = (kend - kbeg) / GT;
  auto fetch = [&](int st) {
    if (st < n_st) {
      bf16* As = smem + (st % G_STAGES) * G_STAGE;
      bf16* Bs = As + GT * G_LD;
      const int k0 = kbeg + st * GT;
#pragma unroll
      for (int i = tid; i < GT * GT / 8; i += 128) {
        const int r = i >> 3, c = (i & 7) * 8;
        cp_async16(As + r * G_LD + c, A + (size_t)(m0 + r) * lda + k0 + c);
        cp_async16(Bs + r * G_LD + c, Bt + (size_t)(n0 + r) * ldb + k0 + c);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  for (int st = 0; st < G_STAGES - 1; ++st) fetch(st);
  for (int st = 0; st < n_st; ++st) {
    fetch(st + G_STAGES - 1);
    asm volatile("cp.async.wait_group %0;\n" ::"n"(G_STAGES - 1));
    __syncthreads();
    const bf16* As = smem + (st % G_STAGES) * G_STAGE;
    const bf16* Bs = As + GT * G_LD;
#pragma unroll
    for (int kk = 0; kk < GT; kk += 16) {
      uint32_t a[2][4], b[4][2];
#pragma unroll
      for (int i = 0; i < 2; ++i)
        ldsm_x4(a[i], As + (wm * 32 + i * 16 + (lane % 16)) * G_LD + kk + (lane / 16) * 8);
#pragma unroll
      for (int jj = 0; jj < 2; ++jj) {
        uint32_t r[4];
        ldsm_x4(r, Bs + (wn * 32 + jj * 16 + (lane % 8) + (lane / 16) * 8) * G_LD + kk +
                       ((lane / 8) % 2) * 8);
        b[2 * jj][0] = r[0];
        b[2 * jj][1] = r[1];
        b[2 * jj + 1][0] = r[2];
        b[2 * jj + 1][1] = r[3];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j]);
    }
    __syncthreads();   // the stage may be refilled
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
  __syncthreads();
}

// Writes a 64-column row block of 16-bit values from shared memory, 16 bytes a thread.
__device__ __forceinline__ void store_rows(const bf16* tile, int rows, bf16* __restrict__ out,
                                           size_t ld, int threads) {
  for (int i = threadIdx.x; i < rows * (GT / 8); i += threads) {
    const int r = i >> 3, c = (i & 7) * 8;
    *reinterpret_cast<uint4*>(out + (size_t)r * ld + c) =
        *reinterpret_cast<const uint4*>(tile + r * G_LD + c);
  }
}

// First statement of every kernel of the training chain: lets the next kernel's blocks be
// scheduled as this one's drain, then waits for the kernel before this one (complete, its
// writes visible) ahead of any memory access.  A no-op in a plain launch.
__device__ __forceinline__ void chain_next() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int EPI>
__global__ void __launch_bounds__(128) gemm_nt_kernel(const GemmArgs g) {
  chain_next();
  extern __shared__ __align__(16) bf16 gsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = warp >> 1, wn = warp & 1;
  const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
  float acc[2][4][4];
  gemm_tile(g.A, g.lda, g.Bt, g.ldb, m0, n0, 0, g.K, gsm, acc);
  bf16* T = gsm;                  // the tile row-major, then transposed
  bf16* Tt = gsm + GT * G_LD;
  const int gq = lane >> 2, tq = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = wm * 32 + i * 16 + gq + h * 8, c = wn * 32 + j * 8 + 2 * tq;
        const float v0 = acc[i][j][2 * h], v1 = acc[i][j][2 * h + 1];
        const size_t zi = (size_t)(m0 + r) * g.ldz + n0 + c;
        bf16 o0, o1;
        if (EPI == EPI_FWD) {
          const float z0 = v0 + g.bias[n0 + c], z1 = v1 + g.bias[n0 + c + 1];
          if (g.Z) *reinterpret_cast<float2*>(g.Z + zi) = make_float2(z0, z1);
          o0 = __float2bfloat16(z0 * sigm(z0));
          o1 = __float2bfloat16(z1 * sigm(z1));
        } else {
          const float2 zp = *reinterpret_cast<const float2*>(g.Z + zi);
          const float s0 = sigm(zp.x), s1 = sigm(zp.y);
          o0 = __float2bfloat16(v0 * s0 * (1.f + zp.x * (1.f - s0)));
          o1 = __float2bfloat16(v1 * s1 * (1.f + zp.y * (1.f - s1)));
        }
        *reinterpret_cast<__nv_bfloat162*>(T + r * G_LD + c) = __nv_bfloat162(o0, o1);
        if (g.HT) {
          Tt[c * G_LD + r] = o0;
          Tt[(c + 1) * G_LD + r] = o1;
        }
      }
  __syncthreads();
  store_rows(T, GT, g.H + (size_t)m0 * g.ldh + n0, g.ldh, 128);
  if (g.HT) store_rows(Tt, GT, g.HT + (size_t)n0 * g.ldht + m0, g.ldht, 128);
}

// The weight gradients dW_l = dZ_l^T . H_l of all layers in one launch (each alone fills a
// third of the chip): blocks (layer's tile, K slice), FP32 partial sums per slice.
struct DwArgs {
  const bf16* dZT[NL];   // [256][B]
  const bf16* HT[NL];    // [K_l][B]
  float* part[NL];       // [splits][256][K_l]
  int k[NL];
  int B, splits;
};

__global__ void __launch_bounds__(128) dw_kernel(const DwArgs g) {
  chain_next();
  extern __shared__ __align__(16) bf16 gsm[];
  int t = blockIdx.x, l = 0;
  while (t >= (WID / GT) * (g.k[l] / GT)) {
    t -= (WID / GT) * (g.k[l] / GT);
    ++l;
  }
  const int nt = g.k[l] / GT, m0 = (t / nt) * GT, n0 = (t % nt) * GT, kz = g.B / g.splits;
  float acc[2][4][4];
  gemm_tile(g.dZT[l], g.B, g.HT[l], g.B, m0, n0, blockIdx.y * kz, (blockIdx.y + 1) * kz, gsm, acc);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = warp >> 1, wn = warp & 1, gq = lane >> 2, tq = lane & 3;
  float* C = g.part[l] + (size_t)blockIdx.y * WID * g.k[l];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = m0 + wm * 32 + i * 16 + gq + h * 8, c = n0 + wn * 32 + j * 8 + 2 * tq;
        *reinterpret_cast<float2*>(C + (size_t)r * g.k[l] + c) =
            make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
      }
}

// What is left of the gradient, in one launch.  Blocks by role: every weight = the sum of
// its K slices in order; the bias gradients (row sums of dZ_l^T) and w5's (rows of
// h_4^T weighted by dy), one warp per row; the loss and b5's gradient, the last block.
constexpr int ROW_PIECE = 2048;   // elements of a row in shared memory at a time

struct ReduceArgs {
  const float* part[NL];
  const bf16* dZT[NL];
  const bf16* H4T;
  const float *y, *t, *dy;
  int splits, B, weight_blocks, row_blocks;
  float *grad, *loss;
};

__global__ void __launch_bounds__(256) grad_reduce_kernel(const ReduceArgs a) {
  chain_next();
  const Layout L = layout();
  const int lane = threadIdx.x & 31;
  if ((int)blockIdx.x < a.weight_blocks) {
    long long i = (blockIdx.x * 256LL + threadIdx.x) * 4;   // 4 weights a thread
    int l = 0;
    while (l < NL && i >= (long long)WID * L.k[l]) {
      i -= (long long)WID * L.k[l];
      ++l;
    }
    if (l == NL) return;
    const long long n = (long long)WID * L.k[l];
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int z = 0; z < a.splits; ++z) {
      const float4 v = *reinterpret_cast<const float4*>(a.part[l] + (size_t)z * n + i);
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
    float* out = a.grad + L.w[l] + i;
    out[0] = s.x;
    out[1] = s.y;
    out[2] = s.z;
    out[3] = s.w;
    return;
  }
  if ((int)blockIdx.x < a.weight_blocks + a.row_blocks) {
    const int row = (blockIdx.x - a.weight_blocks) * 8 + (threadIdx.x >> 5);
    const int l = row / WID, r = row % WID;   // l == NL: w5
    const bf16* X = (l < NL ? a.dZT[l] : a.H4T) + (size_t)r * a.B;
    float s = 0.f;
    // Lane i adds elements i, i + 32, ... in order; the row comes through shared memory,
    // 16 bytes a lane and load with a whole piece in flight (B is a multiple of 64).
    __shared__ __align__(16) bf16 rows[8][ROW_PIECE];
    bf16* buf = rows[threadIdx.x >> 5];
    for (int c0 = 0; c0 < a.B; c0 += ROW_PIECE) {
      const int n = min(ROW_PIECE, a.B - c0);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < ROW_PIECE / 256; ++i) {
        const int c = (i * 32 + lane) * 8;
        if (c < n) *reinterpret_cast<uint4*>(buf + c) = *reinterpret_cast<const uint4*>(X + c0 + c);
      }
      __syncwarp();
#pragma unroll 16
      for (int c = lane; c < n; c += 32) {
        const float f = __bfloat162float(buf[c]);
        s = l < NL ? s + f : fmaf(f, a.dy[c0 + c], s);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) a.grad[(l < NL ? L.b[l] : L.w5) + r] = s;
    return;
  }
  // loss = mean (y - t)^2 and d loss / d b5 = sum dy, in a fixed order: 1024 strided sums,
  // four of them a thread, then a tree
  __shared__ float s1[256], s2[256];
  float e[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
  for (int b0 = 0; b0 < a.B; b0 += 1024) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int b = b0 + q * 256 + threadIdx.x;
      if (b < a.B) {
        const float d = a.y[b] - a.t[b];
        e[q] = fmaf(d, d, e[q]);
        c[q] += a.dy[b];
      }
    }
  }
  s1[threadIdx.x] = (e[0] + e[2]) + (e[1] + e[3]);
  s2[threadIdx.x] = (c[0] + c[2]) + (c[1] + c[3]);
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) {
      s1[threadIdx.x] += s1[threadIdx.x + o];
      s2[threadIdx.x] += s2[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    a.loss[0] = s1[0] / (float)a.B;
    a.grad[L.b5] = s2[0];
  }
}

// F[b] = (sin(2 pi B_j . x_b))_j, (cos(2 pi B_j . x_b))_j as BF16, row-major and transposed.
__global__ void fourier_kernel(const float* __restrict__ freqs, const float* __restrict__ x, int B,
                               bf16* __restrict__ F, bf16* __restrict__ FT) {
  chain_next();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B * NFREQ; i += gridDim.x * blockDim.x) {
    // with FT, neighbouring threads take neighbouring rows (its layout); else frequencies
    const int b = FT ? i % B : i / NFREQ, j = FT ? i / B : i % NFREQ;
    const float v = 2.f * fmaf(freqs[2 * j], x[2 * b], freqs[2 * j + 1] * x[2 * b + 1]);
    float sv, cv;
    sincospif(v, &sv, &cv);
    const bf16 s = __float2bfloat16(sv), c = __float2bfloat16(cv);
    F[(size_t)b * NFEAT + j] = s;
    F[(size_t)b * NFEAT + NFREQ + j] = c;
    if (FT) {
      FT[(size_t)j * B + b] = s;
      FT[(size_t)(NFREQ + j) * B + b] = c;
    }
  }
}

// y[b] = h4[b] . w5 + b5 (one warp per row).
__device__ __forceinline__ float out_row(const bf16* __restrict__ h, const bf16* __restrict__ w5,
                                         float b5) {
  const int lane = threadIdx.x & 31;
  float s = 0.f;
#pragma unroll
  for (int k = lane; k < WID; k += 32) s = fmaf(__bfloat162float(h[k]), __bfloat162float(w5[k]), s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s + b5;
}

__global__ void out_layer_kernel(const bf16* __restrict__ H4, const bf16* __restrict__ w5,
                                 const float* __restrict__ params, long long off_b5, int B,
                                 float* __restrict__ y) {
  const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long b = gw; b < B; b += nw) {
    const float yb = out_row(H4 + b * WID, w5, params[off_b5]);
    if ((threadIdx.x & 31) == 0) y[b] = yb;
  }
}

// The output layer and its backward for 32 rows per block: y, dy[b] = 2 (y[b] - t[b]) / B,
// dZ4[b][k] = dy[b] w5[k] SiLU'(z4[b][k]) (BF16, both layouts, the transposed one through
// shared memory in 64-byte rows).  Bound by the latency of a row's loads and its shuffle
// sum: 64 rows a block left 64 blocks on the chip at a batch of 4096.
constexpr int OUT_THREADS = 512, OUT_ROWS = 32, OUT_LD = OUT_ROWS + 8;
__global__ void __launch_bounds__(OUT_THREADS) out_train_kernel(
    const bf16* __restrict__ H4, const bf16* __restrict__ w5, const float* __restrict__ params,
    long long off_b5, const float* __restrict__ Z4, int B, const float* __restrict__ target,
    float* __restrict__ y, float* __restrict__ dy, bf16* __restrict__ dZ, bf16* __restrict__ dZT) {
  chain_next();
  __shared__ __align__(16) bf16 Tt[WID][OUT_LD];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long b0 = blockIdx.x * (long long)OUT_ROWS;
  for (int r = warp; r < OUT_ROWS; r += OUT_THREADS / 32) {
    const long long b = b0 + r;
    const float yb = out_row(H4 + b * WID, w5, params[off_b5]);
    const float d = 2.f * (yb - target[b]) / (float)B;
    if (lane == 0) {
      y[b] = yb;
      dy[b] = d;
    }
#pragma unroll
    for (int i = 0; i < WID / 64; ++i) {
      const int k = i * 64 + 2 * lane;
      const float2 z = *reinterpret_cast<const float2*>(Z4 + b * WID + k);
      const float s0 = sigm(z.x), s1 = sigm(z.y);
      const bf16 o0 = __float2bfloat16(d * __bfloat162float(w5[k]) * s0 * (1.f + z.x * (1.f - s0)));
      const bf16 o1 = __float2bfloat16(d * __bfloat162float(w5[k + 1]) * s1 * (1.f + z.y * (1.f - s1)));
      *reinterpret_cast<__nv_bfloat162*>(dZ + b * WID + k) = __nv_bfloat162(o0, o1);
      Tt[k][r] = o0;
      Tt[k + 1][r] = o1;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < WID * (OUT_ROWS / 8); i += OUT_THREADS) {
    const int r = i / (OUT_ROWS / 8), c = i % (OUT_ROWS / 8) * 8;
    *reinterpret_cast<uint4*>(dZT + b0 + (size_t)r * B + c) =
        *reinterpret_cast<const uint4*>(&Tt[r][c]);
  }
}

// Adam on the FP32 master vector; refreshes the BF16 shadows (W, W^T, w5).
// BF16 copies of parameter i (value v) in the shadow: W_l row-major, its
// transpose, its K-chunked tensor-core layout, and w5.
__device__ __forceinline__ void write_shadow(const Layout& L, bf16* __restrict__ shadow, long long i,
                                             float v) {
  for (int l = 0; l < NL; ++l) {
    const long long n_w = (long long)WID * L.k[l];
    if (i >= L.w[l] && i < L.w[l] + n_w) {
      const long long e = i - L.w[l];
      const int n = (int)(e / L.k[l]), k = (int)(e % L.k[l]);
      const bf16 b = __float2bfloat16(v);
      shadow[L.sw[l] + e] = b;
      shadow[L.swt[l] + (long long)k * WID + n] = b;
      shadow[L.swc[l] + (long long)(k / WCHUNK_K) * WID * WCHUNK_K +
             chunk_woff(n, k % WCHUNK_K) / 2] = b;
    }
  }
  if (i >= L.w5 && i < L.w5 + WID) shadow[L.sw5 + (i - L.w5)] = __float2bfloat16(v);
}

__global__ void adam_kernel(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, const int32_t* __restrict__ step, float lr,
                            float b1, float b2, float eps, bf16* __restrict__ shadow) {
  chain_next();
  const Layout L = layout();
  const int t = *step + 1;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < L.total;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = fmaf(b1, m[i], (1.f - b1) * gi);
    const float vi = fmaf(b2, v[i], (1.f - b2) * gi * gi);
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (shadow) write_shadow(L, shadow, i, pi);
  }
}

__global__ void shadow_kernel(const float* __restrict__ p, bf16* __restrict__ shadow) {
  const Layout L = layout();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < L.total;
       i += (long long)gridDim.x * blockDim.x)
    write_shadow(L, shadow, i, p[i]);
}

__global__ void increment_kernel(int32_t* step) {
  chain_next();
  if (threadIdx.x == 0 && blockIdx.x == 0) *step += 1;
}

}  // namespace mlp
}  // namespace drt

#include "drt_mlp_tc.cuh"
#include "drt_mlp_fused.cuh"

namespace drt {
namespace mlp {

// timeout flag of the tcgen05 kernels (device-global; read and cleared by drt_mlp_tc_status)
__device__ int g_tc_status;

}  // namespace mlp

// ------------------------------------------------------------------ host side
namespace {

using mlp::bf16;

struct MlpWs {
  bf16 *F, *FT, *H[DRT_MLP_LAYERS + 1], *HT[DRT_MLP_LAYERS + 1], *dZ[2], *dZT[DRT_MLP_LAYERS];
  float *Z[DRT_MLP_LAYERS], *y, *dy, *part[DRT_MLP_LAYERS];
  int splits;
  size_t bytes;
};

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

MlpWs carve(void* base, int B) {
  MlpWs w{};
  char* p = static_cast<char*>(base);
  size_t o = 0;
  auto take = [&](size_t n) {
    char* r = p ? p + o : nullptr;
    o = al256(o + n);
    return r;
  };
  const size_t hb = (size_t)B * mlp::WID * sizeof(bf16);
  w.F = reinterpret_cast<bf16*>(take((size_t)B * mlp::NFEAT * sizeof(bf16)));
  w.FT = reinterpret_cast<bf16*>(take((size_t)B * mlp::NFEAT * sizeof(bf16)));
  w.H[0] = w.F;
  w.HT[0] = w.FT;
  for (int l = 1; l <= mlp::NL; ++l) {
    w.H[l] = reinterpret_cast<bf16*>(take(hb));
    w.HT[l] = reinterpret_cast<bf16*>(take(hb));
  }
  for (int l = 0; l < mlp::NL; ++l) w.Z[l] = reinterpret_cast<float*>(take((size_t)B * mlp::WID * 4));
  w.y = reinterpret_cast<float*>(take((size_t)B * 4));
  w.dy = reinterpret_cast<float*>(take((size_t)B * 4));
  for (int i = 0; i < 2; ++i) w.dZ[i] = reinterpret_cast<bf16*>(take(hb));
  for (int l = 0; l < mlp::NL; ++l) w.dZT[l] = reinterpret_cast<bf16*>(take(hb));
  // weight gradients reduce over the batch: split it into slices of >= 256 rows
  w.splits = std::max(1, std::min(32, B / 256));
  while (w.splits > 1 && (B % (w.splits * 64))) --w.splits;
  for (int l = 0; l < mlp::NL; ++l)
    w.part[l] = reinterpret_cast<float*>(take((size_t)w.splits * mlp::WID * mlp::layout().k[l] * 4));
  w.bytes = o;
  return w;
}

// Which tensor-core path the dense layers use: 1 = tcgen05 (TMEM accumulator),
// 0 = mma.sync.  The tcgen05 path needs M a multiple of 128 and K of 64; other
// shapes take the mma.sync path.
std::atomic<int> g_tc_mode{1};
std::atomic<int> g_tc_skip_mma{0};
std::mutex g_tc_mu;
int* g_tc_status_ptr[64] = {};

// 72 KB of dynamic shared memory per CTA: the two 128 x 64 stages (or the FP32
// output tile) fit, and at most three CTAs (3 x 128 TMEM columns) share an SM.
constexpr int TC_SMEM = 72 * 1024;
static_assert(mlp::TcSmem<128>::BYTES <= TC_SMEM && mlp::TcSmem<64>::BYTES <= TC_SMEM, "smem");

int* tc_status_ptr() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(g_tc_mu);
  if (!g_tc_status_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, mlp::g_tc_status) != cudaSuccess) return nullptr;
    g_tc_status_ptr[dev] = static_cast<int*>(p);
    cudaFuncSetAttribute(mlp::tc_gemm_nt_kernel<mlp::EPI_FWD, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(mlp::tc_gemm_nt_kernel<mlp::EPI_DH, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(mlp::tc_gemm_nt_kernel<mlp::EPI_DW, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(mlp::tc_gemm_nt_kernel<mlp::EPI_FWD, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(mlp::tc_gemm_nt_kernel<mlp::EPI_DH, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(mlp::tc_gemm_nt_kernel<mlp::EPI_DW, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(mlp::tc_mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         mlp::FZ_SMEM);
  }
  return g_tc_status_ptr[dev];
}

// The mma.sync kernels' dynamic shared memory limit, raised once per device.
cudaError_t gemm_smem_limits() {
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_tc_mu);
  if (done[dev]) return cudaSuccess;
  constexpr auto LIMIT = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if ((e = cudaFuncSetAttribute(mlp::gemm_nt_kernel<mlp::EPI_FWD>, LIMIT, mlp::G_SMEM)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(mlp::gemm_nt_kernel<mlp::EPI_DH>, LIMIT, mlp::G_SMEM)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(mlp::dw_kernel, LIMIT, mlp::G_SMEM)) != cudaSuccess)
    return e;
  done[dev] = true;
  return cudaSuccess;
}

// whether a GEMM of this shape takes the tcgen05 kernel (mode 2)
bool gemm_uses_tc(int M, int N, int K) {
  return g_tc_mode.load() == 2 && M % mlp::TC_BM == 0 && K % mlp::TC_BK == 0 && N % 64 == 0 &&
         tc_status_ptr();
}

// Launch of a kernel that begins with chain_next(): its launch and block scheduling overlap
// the kernel before it on the stream.
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                           A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <int EPI>
cudaError_t gemm(const mlp::GemmArgs& g, cudaStream_t st) {
  // the training GEMMs take tcgen05 only in mode 2 (mode 1: the fused inference kernel)
  int* status = gemm_uses_tc(g.M, g.N, g.K) ? tc_status_ptr() : nullptr;
  if (status) {
    const int z = (EPI == mlp::EPI_DW && g.k_splits > 1) ? g.k_splits : 1;
    if (g.N % 128 == 0) {
      dim3 grid(g.N / 128, g.M / mlp::TC_BM, z);
      mlp::tc_gemm_nt_kernel<EPI, 128><<<grid, 128, TC_SMEM, st>>>(g, status, g_tc_skip_mma.load());
    } else {
      dim3 grid(g.N / 64, g.M / mlp::TC_BM, z);
      mlp::tc_gemm_nt_kernel<EPI, 64><<<grid, 128, TC_SMEM, st>>>(g, status, g_tc_skip_mma.load());
    }
    return cudaGetLastError();
  }
  if constexpr (EPI == mlp::EPI_DW) {
    return cudaErrorInvalidValue;   // dw_kernel takes the weight gradients of this path
  } else {
    cudaError_t e = gemm_smem_limits();
    if (e != cudaSuccess) return e;
    return launch_chained(mlp::gemm_nt_kernel<EPI>, dim3(g.N / mlp::GT, g.M / mlp::GT), 128,
                          mlp::G_SMEM, st, g);
  }
}

// the whole network for n rows in one kernel (any n)
cudaError_t launch_fused_forward(const float* params, const bf16* shadow, const float* freqs,
                                 const float* x, int n, float* y, int* status, cudaStream_t st) {
  const mlp::Layout L = mlp::layout();
  mlp::FusedArgs fa{};
  fa.params = params;
  fa.shadow = shadow;
  fa.freqs = freqs;
  fa.x = x;
  fa.y = y;
  fa.batch = n;
  for (int l = 0; l < mlp::NL; ++l) {
    fa.swc[l] = L.swc[l];
    fa.b[l] = L.b[l];
  }
  fa.sw5 = L.sw5;
  fa.b5 = L.b5;
  const int grid = (n + mlp::FZ_ROWS - 1) / mlp::FZ_ROWS;
  mlp::tc_mlp_forward_kernel<<<grid, mlp::FZ_THREADS, mlp::FZ_SMEM, st>>>(fa, status,
                                                                      g_tc_skip_mma.load());
  return cudaGetLastError();
}

// forward through the hidden layers; with_train keeps Z and the transposed copies
cudaError_t mlp_hidden_forward(const float* params, const bf16* shadow, const float* freqs,
                               const float* x, int B, const MlpWs& w, bool with_train,
                               cudaStream_t st) {
  const mlp::Layout L = mlp::layout();
  const int blocks = std::min(4096, (B * mlp::NFREQ + 255) / 256);
  cudaError_t e = launch_chained(mlp::fourier_kernel, dim3(blocks), 256, 0, st, freqs, x, B, w.F,
                                 with_train ? w.FT : nullptr);
  if (e != cudaSuccess) return e;
  for (int l = 0; l < mlp::NL; ++l) {
    mlp::GemmArgs g{};
    g.A = w.H[l];
    g.lda = L.k[l];
    g.Bt = shadow + L.sw[l];
    g.ldb = L.k[l];
    g.M = B;
    g.N = mlp::WID;
    g.K = L.k[l];
    g.bias = params + L.b[l];
    g.Z = with_train ? w.Z[l] : nullptr;   // pre-activations: only the backward pass reads them
    g.ldz = mlp::WID;
    g.H = w.H[l + 1];
    g.ldh = mlp::WID;
    g.HT = with_train ? w.HT[l + 1] : nullptr;
    g.ldht = B;
    if ((e = gemm<mlp::EPI_FWD>(g, st)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace
}  // namespace drt

using namespace drt;

namespace {
drt_status mlp_fail(drt_status st, const char* msg) {
  set_error_message(msg);
  return st;
}
bool a16(const void* p) { return p && (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
}  // namespace

extern "C" {

drt_status drt_mlp_sizes(int32_t batch, int64_t* n_params, size_t* shadow_bytes,
                         size_t* workspace_bytes) {
  const mlp::Layout L = mlp::layout();
  if (n_params) *n_params = L.total;
  if (shadow_bytes) *shadow_bytes = (size_t)L.stotal * sizeof(mlp::bf16);
  if (workspace_bytes) {
    if (batch < 64 || batch % 64) return mlp_fail(DRT_ERR_INVALID_ARG, "batch must be a positive multiple of 64");
    *workspace_bytes = carve(nullptr, batch).bytes;
  }
  return DRT_OK;
}

drt_status drt_mlp_shadow(const float* params, void* shadow, void* stream) {
  if (!params || !a16(shadow)) return mlp_fail(DRT_ERR_INVALID_ARG, "params / shadow (16-byte aligned)");
  mlp::shadow_kernel<<<256, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      params, static_cast<mlp::bf16*>(shadow));
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DRT_OK : mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
}

drt_status drt_mlp_forward(const float* params, const void* shadow, const float* freqs,
                           const float* x, int32_t batch, float* y, void* workspace,
                           size_t workspace_bytes, void* stream) {
  if (!params || !a16(shadow) || !freqs || !x || !y)
    return mlp_fail(DRT_ERR_INVALID_ARG, "NULL or misaligned pointer");
  if (batch < 64 || batch % 64) return mlp_fail(DRT_ERR_INVALID_ARG, "batch must be a positive multiple of 64");
  const MlpWs w = carve(workspace, batch);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < w.bytes)
    return mlp_fail(DRT_ERR_WORKSPACE, "MLP workspace too small or not 256-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const mlp::Layout L = mlp::layout();
  const mlp::bf16* sh = static_cast<const mlp::bf16*>(shadow);
  int* status = g_tc_mode.load() != 0 ? tc_status_ptr() : nullptr;
  if (status) {
    // tcgen05 path: the whole network in one kernel, activations on chip
    cudaError_t e = launch_fused_forward(params, sh, freqs, x, batch, y, status, st);
    return e == cudaSuccess ? DRT_OK : mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
  }
  cudaError_t e = mlp_hidden_forward(params, sh, freqs, x, batch, w, false, st);
  if (e == cudaSuccess) {
    mlp::out_layer_kernel<<<std::min(4096, (batch * 32 + 255) / 256), 256, 0, st>>>(
        w.H[mlp::NL], sh + L.sw5, params, L.b5, batch, y);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? DRT_OK : mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
}

drt_status drt_mlp_predict(const float* params, const void* shadow, const float* freqs,
                           const float* x, int32_t n, float* y, void* stream) {
  if (!params || !a16(shadow) || !freqs)
    return mlp_fail(DRT_ERR_INVALID_ARG, "NULL or misaligned pointer");
  if (n < 0) return mlp_fail(DRT_ERR_INVALID_ARG, "n < 0");
  if (n == 0) return DRT_OK;   // no rows: x and y may be NULL
  if (!x || !y) return mlp_fail(DRT_ERR_INVALID_ARG, "x or y is NULL");
  int* status = g_tc_mode.load() != 0 ? tc_status_ptr() : nullptr;
  if (!status) return mlp_fail(DRT_ERR_UNSUPPORTED, "drt_mlp_predict needs the tcgen05 path");
  const cudaError_t e = launch_fused_forward(params, static_cast<const mlp::bf16*>(shadow), freqs, x, n,
                                             y, status, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? DRT_OK : mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
}

drt_status drt_mlp_loss_grad(const float* params, const void* shadow, const float* freqs,
                             const float* x, const float* target, int32_t batch, float* loss,
                             float* grad, void* workspace, size_t workspace_bytes, void* stream) {
  if (!params || !a16(shadow) || !freqs || !x || !target || !loss || !grad)
    return mlp_fail(DRT_ERR_INVALID_ARG, "NULL or misaligned pointer");
  if (batch < 64 || batch % 64) return mlp_fail(DRT_ERR_INVALID_ARG, "batch must be a positive multiple of 64");
  const MlpWs w = carve(workspace, batch);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < w.bytes)
    return mlp_fail(DRT_ERR_WORKSPACE, "MLP workspace too small or not 256-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const mlp::Layout L = mlp::layout();
  const mlp::bf16* sh = static_cast<const mlp::bf16*>(shadow);
  const int B = batch;
  cudaError_t e = mlp_hidden_forward(params, sh, freqs, x, B, w, true, st);
  if (e != cudaSuccess) return mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
  e = launch_chained(mlp::out_train_kernel, dim3(B / mlp::OUT_ROWS), mlp::OUT_THREADS, 0, st,
                     w.H[mlp::NL], sh + L.sw5, params, L.b5, w.Z[mlp::NL - 1], B, target, w.y, w.dy,
                     w.dZ[0], w.dZT[mlp::NL - 1]);
  int cur = 0;
  for (int l = mlp::NL - 1; l > 0 && e == cudaSuccess; --l) {
    mlp::GemmArgs h{};
    h.A = w.dZ[cur];     // [B][256]
    h.lda = mlp::WID;
    h.Bt = sh + L.swt[l];   // W_l^T: [K_l][256]
    h.ldb = mlp::WID;
    h.M = B;
    h.N = L.k[l];
    h.K = mlp::WID;
    h.Z = w.Z[l - 1];
    h.ldz = mlp::WID;
    h.H = w.dZ[cur ^ 1];
    h.ldh = mlp::WID;
    h.HT = w.dZT[l - 1];
    h.ldht = B;
    e = gemm<mlp::EPI_DH>(h, st);
    cur ^= 1;
  }
  // the weight gradients need only the transposed copies, which every layer keeps
  bool tc = false;
  for (int l = 0; l < mlp::NL && e == cudaSuccess; ++l) {
    if (!gemm_uses_tc(mlp::WID, L.k[l], B)) continue;
    tc = true;
    mlp::GemmArgs g{};
    g.A = w.dZT[l];        // [256][B]
    g.lda = B;
    g.Bt = w.HT[l];        // [K_l][B]
    g.ldb = B;
    g.M = mlp::WID;
    g.N = L.k[l];
    g.K = B;
    g.C = w.part[l];
    g.ldc = L.k[l];
    g.k_splits = w.splits;
    e = gemm<mlp::EPI_DW>(g, st);
  }
  if (e != cudaSuccess) return mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
  mlp::ReduceArgs r{};
  if (!tc) {
    mlp::DwArgs d{};
    int tiles = 0;
    for (int l = 0; l < mlp::NL; ++l) {
      d.dZT[l] = w.dZT[l];
      d.HT[l] = w.HT[l];
      d.part[l] = w.part[l];
      d.k[l] = L.k[l];
      tiles += (mlp::WID / mlp::GT) * (L.k[l] / mlp::GT);
    }
    d.B = B;
    d.splits = w.splits;
    if ((e = gemm_smem_limits()) != cudaSuccess) return mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
    e = launch_chained(mlp::dw_kernel, dim3(tiles, w.splits), 128, mlp::G_SMEM, st, d);
    if (e != cudaSuccess) return mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
  }
  long long weights = 0;
  for (int l = 0; l < mlp::NL; ++l) {
    r.part[l] = w.part[l];
    r.dZT[l] = w.dZT[l];
    weights += (long long)mlp::WID * L.k[l];
  }
  r.H4T = w.HT[mlp::NL];
  r.y = w.y;
  r.t = target;
  r.dy = w.dy;
  r.splits = w.splits;
  r.B = B;
  r.weight_blocks = (int)((weights / 4 + 255) / 256);
  r.row_blocks = (mlp::NL + 1) * mlp::WID / 8;
  r.grad = grad;
  r.loss = loss;
  e = launch_chained(mlp::grad_reduce_kernel, dim3(r.weight_blocks + r.row_blocks + 1), 256, 0, st,
                     r);
  return e == cudaSuccess ? DRT_OK : mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
}

drt_status drt_mlp_set_tensor_core_path(int32_t use_tcgen05) {
  if (use_tcgen05 < 0 || use_tcgen05 > 2) return mlp_fail(DRT_ERR_INVALID_ARG, "use_tcgen05 must be 0, 1 or 2");
  g_tc_mode.store(use_tcgen05);
  return DRT_OK;
}

drt_status drt_mlp_test_skip_mma(int32_t skip) {
  g_tc_skip_mma.store(skip ? 1 : 0);
  return DRT_OK;
}

drt_status drt_mlp_tc_status(int32_t* timed_out) {
  if (!timed_out) return mlp_fail(DRT_ERR_INVALID_ARG, "NULL pointer");
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, mlp::g_tc_status, sizeof(int));
  if (e == cudaSuccess) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(mlp::g_tc_status, &zero, sizeof(int));
  }
  if (e != cudaSuccess) return mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
  *timed_out = v;
  return v ? DRT_ERR_TIMEOUT : DRT_OK;
}

drt_status drt_mlp_adam(float* params, float* m, float* v, const float* grad, int32_t* step,
                        float lr, float beta1, float beta2, float eps, void* shadow, void* stream) {
  if (!params || !m || !v || !grad || !step) return mlp_fail(DRT_ERR_INVALID_ARG, "NULL pointer");
  if (shadow && !a16(shadow)) return mlp_fail(DRT_ERR_INVALID_ARG, "shadow must be 16-byte aligned");
  if (!(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
    return mlp_fail(DRT_ERR_INVALID_ARG, "Adam hyper-parameters out of range");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = launch_chained(mlp::adam_kernel, dim3(256), 256, 0, st, params, m, v, grad, step, lr,
                                 beta1, beta2, eps, static_cast<mlp::bf16*>(shadow));
  if (e == cudaSuccess) e = launch_chained(mlp::increment_kernel, dim3(1), 32, 0, st, step);
  return e == cudaSuccess ? DRT_OK : mlp_fail(DRT_ERR_CUDA, cudaGetErrorString(e));
}

}  // extern "C"
