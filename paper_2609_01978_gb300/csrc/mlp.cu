// mlp.cu -- learned surrogate: a multilayer perceptron trained and evaluated by
// kernels written here (no counterpart in the paper; it learns the map from
// membrane-deformation parameters to the PSF and metrics that the CZT method
// computes, Sec. 7.2 / Sec. 9 name membrane deformation as the next input).
//
// Network: n_in -> hidden (x n_hidden_layers, SiLU) -> n_out (linear); loss =
// mean squared error over batch and outputs; optimiser AdamW (decoupled weight
// decay on weights, not biases).  Weights are kept as FP32 masters; every matrix
// product takes BF16 operands (weights, layer inputs, back-propagated errors)
// and accumulates in FP32 in tensor memory (tcgen05.mma kind::f16, M128 N64).
//
// Matrix products, all as C[M x N] = A[M x K] . B[N x K]^T with K contiguous:
//   forward  z_l   = h_{l-1} . W_l^T          (A = h, B = W)
//   backward dh    = g . W_l                  (A = g, B = W^T  kept transposed)
//            dW_l  = g^T . h_{l-1}            (A = g^T, B = h^T: transposed copies)
// At this network's sizes (batch 256, 512 hidden, 4114 outputs: 6.7 GFLOP of a
// training step, 3.5 us of the tensor rate) a step is bound by launches and by
// the length of each product's chain, so the products take 128 x 64 tiles with
// an eight-deep ring of loads, what follows a product (bias, SiLU and its
// derivative, the loss gradient, BF16 copies in both orders, column sums) is
// its epilogue, and a layer's two backward products share a launch.  Every
// product keeps one accumulation in K order: a split of the longest (dh of the
// output layer, K = 4160) was no slower to write but moves g in its last FP32
// bits, and with them the BF16 rounding of 3 % of g's values.  A launch overlaps
// the end of the one before.  Gradients of that batch: 46 launches, 1,154 us;
// fused 130; overlapped 111.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "fzp_internal.cuh"
#include "tc_ptx.cuh"

namespace fzp {
namespace {

using namespace tc;

constexpr int GM = 128, GN = 64, GK = 64;  // GEMM tile; K step = one 128-byte swizzle row
constexpr int GEMM_THREADS = 256;  // warps 0-3: columns 0-31 of the tile in the epilogue, 4-7: 32-63
constexpr int RING = 8, AHEAD = RING - 2;  // K steps loaded ahead (a slot rests one step, its MMAs in flight)
constexpr int STAGE_BYTES = (GM + GN) * GK * 2;
constexpr int GEMM_SMEM = 1024 + RING * STAGE_BYTES + 128;  // the epilogue's tile of g reuses the ring

__host__ __device__ inline int64_t pad64(int64_t x) { return (x + 63) / 64 * 64; }

// K-major, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t sdesc128(const void* p) {
  const uint64_t a = smem_u32(p);
  return ((a >> 4) & 0x3FFFull) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
constexpr uint32_t IDESC_G = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GN >> 3) << 17) | ((uint32_t)(GM >> 4) << 24);

__device__ __forceinline__ void mma_g(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
          dtmem),
      "l"(ad), "l"(bd), "r"(IDESC_G), "r"(acc)
      : "memory");
}

// 16 bytes global -> shared, or zeros (the address is not read then).
__device__ __forceinline__ void cp16(void* dst, const void* src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(live ? 16 : 0)
               : "memory");
}

__device__ __forceinline__ float sigm(float z) { return 1.f / (1.f + expf(-z)); }

// What follows a product.
enum Epi {
  EPI_HIDDEN = 0,  // z = acc + bias -> Z; h = silu(z) -> Hb (and, training, HTb)
  EPI_Y = 1,       // y = acc + bias -> C
  EPI_LOSS = 2,    // g = 2 (acc + bias - y) / (B n) -> Gb, GTb, column sums; loss
  EPI_DW = 3,      // C = acc (a layer's gradient, packed); the first tile column also adds the bias gradient up
  EPI_DH = 4       // g = acc silu'(z) -> Gb, GTb, column sums
};

struct Gemm {
  const __nv_bfloat16 *A, *B;
  int64_t lda, ldb;
  int M, N, K;         // K a multiple of 8
  int tiles_n, tiles;  // tiles along N, and all
  int epi;
  const float* bias;
  float* C;            // EPI_Y, EPI_DW
  int64_t ldc;
  float* Z;            // EPI_HIDDEN (written), EPI_DH (read)
  int64_t ldz;
  __nv_bfloat16 *rows, *cols;  // Hb / Gb and HTb / GTb (cols may be null)
  int64_t ldr, ldt;
  const float* y;      // EPI_LOSS
  double* lpart;       // EPI_LOSS: squared errors of each tile; EPI_DW of the first layer: to be totalled
  int nlpart;
  float* loss;         // EPI_DW of the first layer (may be null): the mean of the squared errors
  double loss_scale;
  float* sums;         // column sums per 128-row tile [tile][ld_sums]
  int64_t ld_sums;
  const float* bsums;  // EPI_DW: the column sums whose total is the bias gradient
  float* db;
  int nsums;
};

// Columns [c0, c0 + 32) of a row of g or h in BF16, row-major (64 bytes a
// thread) and transposed (a warp's 32 rows per column).  Columns from n on and
// rows from m on are zero in `v` / not stored.
__device__ __forceinline__ void store_bf16(const Gemm& p, const float (&v)[32], int r, int c0, bool row_live) {
  if (!row_live) return;
  uint32_t w[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    w[q] = *reinterpret_cast<const uint32_t*>(&t);
  }
  if (c0 < p.ldr) {
    uint4* o = reinterpret_cast<uint4*>(p.rows + (int64_t)r * p.ldr + c0);
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
  }
  if (p.cols) {
#pragma unroll
    for (int q = 0; q < 32; ++q)
      if (c0 + q < p.N) p.cols[(int64_t)(c0 + q) * p.ldt + r] = __float2bfloat16_rn(v[q]);
  }
}

// One tile of one of up to two products per CTA.
__global__ void __launch_bounds__(GEMM_THREADS) k_gemm(const Gemm g0, const Gemm g1, int n0_blocks, int* err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bar = reinterpret_cast<uint64_t*>(base + RING * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + RING);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar + RING + 1);
  const bool first = (int)blockIdx.x < n0_blocks;
  const Gemm& p = first ? g0 : g1;
  const int tile = first ? blockIdx.x : blockIdx.x - n0_blocks;
  const int m0 = tile / p.tiles_n * GM, n0 = tile % p.tiles_n * GN;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int q = 0; q < RING; ++q) mbar_init(&bar[q], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(GN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();
  const int nk = (p.K + GK - 1) / GK;
  // K step kb into its ring slot: 128 + 64 rows of 128 bytes, swizzled
  auto load = [&](int kb) {
    uint8_t* s = base + kb % RING * STAGE_BYTES;
    const int ch = tid & 7, gk = kb * GK + ch * 8;
#pragma unroll
    for (int q = 0; q < (GM + GN) / 32; ++q) {
      const int r = q * 32 + (tid >> 3);
      const bool isA = q < GM / 32;
      const int gr = isA ? m0 + r : n0 + r - GM;
      const bool live = gk < p.K && gr < (isA ? p.M : p.N);
      const __nv_bfloat16* src = isA ? p.A + (int64_t)gr * p.lda + gk : p.B + (int64_t)gr * p.ldb + gk;
      cp16(s + (r >> 3) * 1024 + (r & 7) * 128 + ((ch ^ (r & 7)) << 4), live ? src : (isA ? p.A : p.B), live);
    }
  };
#pragma unroll
  for (int q = 0; q < AHEAD; ++q) {
    if (q < nk) load(q);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  bool ok = true;
  for (int kb = 0; kb < nk; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
    fence_proxy_async();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      uint8_t* s = base + kb % RING * STAGE_BYTES;
      const uint64_t ad = sdesc128(s), bd = sdesc128(s + GM * GK * 2);
#pragma unroll
      for (int kk = 0; kk < GK / 16; ++kk)
        mma_g(tmem, ad + (uint64_t)((kk * 32) >> 4), bd + (uint64_t)((kk * 32) >> 4), (kb > 0 || kk > 0) ? 1u : 0u);
      mma_commit(&bar[kb % RING]);
    }
    // the slot of step kb - 2 is free once its MMAs are done
    if (kb + AHEAD < nk) {
      if (kb > 1) ok = mbar_wait(&bar[(kb - 2) % RING], (uint32_t)((kb - 2) / RING & 1), abort_flag, err, 200) && ok;
      load(kb + AHEAD);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  const int last = nk - 1;
  ok = mbar_wait(&bar[last % RING], (uint32_t)(last / RING & 1), abort_flag, err, 201) && ok;
  tc_fence_after();
  __syncthreads();  // every wait above has ended in all threads
  ok = ok && !*abort_flag;
  if (ok) {
    const int tr = tid & (GM - 1), r = m0 + tr;
    const bool row_live = r < p.M;
    float* tile_g = reinterpret_cast<float*>(base);  // [128][65] of g, for the column sums
    float lsum = 0.f;
    const float scale = 2.f / ((float)p.M * (float)p.N);
    {
      const int cc = (warp >> 2) * 32, c0 = n0 + cc;
      float v[32];
      tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cc, v);
      if (p.epi == EPI_HIDDEN) {
#pragma unroll
        for (int q = 0; q < 32; ++q) v[q] = c0 + q < p.N ? v[q] + p.bias[c0 + q] : 0.f;
        if (row_live && p.Z) {
#pragma unroll
          for (int q = 0; q < 8; ++q)  // the padding columns too (zeros)
            if (c0 + 4 * q < p.ldz)
              *reinterpret_cast<float4*>(p.Z + (int64_t)r * p.ldz + c0 + 4 * q) =
                  make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
#pragma unroll
        for (int q = 0; q < 32; ++q) v[q] = v[q] * sigm(v[q]);
        store_bf16(p, v, r, c0, row_live);
      } else if (p.epi == EPI_LOSS || p.epi == EPI_DH) {
        if (p.epi == EPI_LOSS) {
#pragma unroll
          for (int q = 0; q < 32; ++q) {
            float d = 0.f;
            if (row_live && c0 + q < p.N) d = v[q] + p.bias[c0 + q] - p.y[(int64_t)r * p.N + c0 + q];
            lsum += d * d;
            v[q] = scale * d;
          }
        } else {
#pragma unroll
          for (int q = 0; q < 32; ++q) {
            float d = 0.f;
            if (row_live && c0 + q < p.N) {
              const float zz = p.Z[(int64_t)r * p.ldz + c0 + q], sg = sigm(zz);
              d = v[q] * (sg * (1.f + zz * (1.f - sg)));
            }
            v[q] = d;
          }
        }
        store_bf16(p, v, r, c0, row_live);
#pragma unroll
        for (int q = 0; q < 32; ++q) tile_g[tr * 65 + cc + q] = v[q];
      } else {
        if (row_live) {
#pragma unroll
          for (int q = 0; q < 32; ++q)
            if (c0 + q < p.N) v[q] += p.epi == EPI_Y ? p.bias[c0 + q] : 0.f;
          float* C = p.C + (int64_t)r * p.ldc + c0;
          if ((p.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0 && c0 + 32 <= p.N) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
              *reinterpret_cast<float4*>(C + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          } else {
#pragma unroll
            for (int q = 0; q < 32; ++q)
              if (c0 + q < p.N) C[q] = v[q];
          }
        }
      }
    }
    if (p.epi == EPI_LOSS || p.epi == EPI_DH) {
      __syncthreads();
      if (tid < GN && n0 + tid < p.N) {
        float s = 0.f;
        for (int q = 0; q < GM; ++q) s += tile_g[q * 65 + tid];
        p.sums[(int64_t)(m0 / GM) * p.ld_sums + n0 + tid] = s;
      }
      if (p.epi == EPI_LOSS) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        float* part = tile_g + GM * 65;
        if (lane == 0) part[warp] = lsum;
        __syncthreads();
        if (tid == 0) {
          double t = 0.0;
          for (int q = 0; q < GEMM_THREADS / 32; ++q) t += (double)part[q];
          p.lpart[tile] = t;
        }
      }
    }
    if (p.epi == EPI_DW && p.loss && tile == 0 && warp == 7) {
      double t = 0.0;
      for (int q = lane; q < p.nlpart; q += 32) t += p.lpart[q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) *p.loss = (float)(t * p.loss_scale);
    }
    if (p.epi == EPI_DW && n0 == 0 && row_live && tid < GM) {
      float s = 0.f;
      for (int q = 0; q < p.nsums; ++q) s += p.bsums[(int64_t)q * p.ld_sums + r];
      p.db[r] = s;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(GN) : "memory");
  }
}

// The batch's inputs in BF16, row-major (zero padded) and, training, transposed.
__global__ void k_inputs(int64_t R, int64_t Cn, const float* x, __nv_bfloat16* rows, int64_t ldr, __nv_bfloat16* cols,
                         int64_t ldt) {
  pdl_trigger();
  const int64_t total = R * Cn;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t / Cn, c = t % Cn;
    const __nv_bfloat16 v = __float2bfloat16_rn(x[t]);
    rows[r * ldr + c] = v;
    if (cols) cols[c * ldt + r] = v;
  }
}

// AdamW on one layer's weights and biases (decay on the weights only), and the
// weights' BF16 copies: Wb [n_out][ld_in], WTb [n_in][ld_out].
__global__ void k_adamw(int64_t n_out, int64_t n_in, float* p, const float* g, float* m, float* v, float lr, float wd,
                        float b1, float b2, float eps, float c1, float c2, __nv_bfloat16* Wb, int64_t ld_in,
                        __nv_bfloat16* WTb, int64_t ld_out) {
  const int64_t nw = n_out * n_in, n = nw + n_out;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const float gg = g[t];
    const float mm = b1 * m[t] + (1.f - b1) * gg;
    const float vv = b2 * v[t] + (1.f - b2) * gg * gg;
    m[t] = mm;
    v[t] = vv;
    const float w = p[t], pw = w - lr * ((mm / c1) / (sqrtf(vv / c2) + eps) + (t < nw ? wd : 0.f) * w);
    p[t] = pw;
    if (t < nw) {
      const int64_t o = t / n_in, i = t % n_in;
      const __nv_bfloat16 b = __float2bfloat16_rn(pw);
      Wb[o * ld_in + i] = b;
      WTb[i * ld_out + o] = b;
    }
  }
}

// Weights W (FP32 [n_out][n_in], row-major, inside the flat vector) -> BF16
// copies Wb [n_out][ld_in] and WTb [n_in][ld_out].
__global__ void k_weights_bf16(int64_t n_out, int64_t n_in, const float* W, __nv_bfloat16* Wb, int64_t ld_in,
                               __nv_bfloat16* WTb, int64_t ld_out) {
  const int64_t total = n_out * n_in;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = t / n_in, i = t % n_in;
    const __nv_bfloat16 w = __float2bfloat16_rn(W[t]);
    Wb[o * ld_in + i] = w;
    WTb[i * ld_out + o] = w;
  }
}

__global__ void k_init_uniform(int64_t n, float* p, float scale, uint64_t seed) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)(t + 1);  // splitmix64
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    p[t] = scale * (2.f * (float)((z >> 40) * (1.0 / 16777216.0)) - 1.f);
  }
}

}  // namespace

struct Layer {
  int64_t n_in, n_out, ld_in, ld_out;  // ld: padded to 64
  int64_t off_w, off_b;                // offsets in the flat parameter vector
  __nv_bfloat16 *Wb = nullptr, *WTb = nullptr;
};

}  // namespace fzp

using namespace fzp;

struct fzp_surrogate_s {
  std::vector<Layer> L;
  int64_t max_batch = 0, n_params = 0, step = 0;
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  std::vector<float*> Z;             // pre-activations per layer [B][ld_out] FP32
  std::vector<__nv_bfloat16*> Hb;    // layer inputs, BF16 [B][ld_in]
  std::vector<__nv_bfloat16*> HTb;   // layer inputs transposed [ld_in... n_in][ldB]
  __nv_bfloat16 *Gb[2] = {}, *GTb[2] = {};  // g of a layer and of the one below it
  float* sums[2] = {};               // its column sums per 128 rows [tile][maxw]
  double* lpart = nullptr;           // squared errors of the output layer's tiles
  int64_t ldB = 0, maxw = 0;
  int* err = nullptr;
  std::vector<void*> allocs;
};

namespace {

unsigned blocks(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 4096); }

Gemm product(int64_t M, int64_t N, int64_t K, const __nv_bfloat16* A, int64_t lda, const __nv_bfloat16* B, int64_t ldb,
             int epi) {
  Gemm p{};
  p.A = A; p.B = B; p.lda = lda; p.ldb = ldb;
  p.M = (int)M; p.N = (int)N; p.K = (int)K;
  p.tiles_n = (int)((N + GN - 1) / GN);
  p.tiles = p.tiles_n * (int)((M + GM - 1) / GM);
  p.epi = epi;
  return p;
}

fzp_status run_gemm(fzp_surrogate_s& S, const Gemm& a, const Gemm* b, cudaStream_t s) {
  const int na = a.tiles, nb = b ? b->tiles : 0;
  FZP_CUDA_TRY(launch_after(k_gemm, dim3((unsigned)(na + nb)), dim3(GEMM_THREADS), GEMM_SMEM, s, a, b ? *b : a, na, S.err));
  return FZP_OK;
}

// Forward pass for a batch of B rows (x: FP32 [B][n_in0], contiguous).  y null:
// inference, the output to `out` (FP32 [B][n_out]).  Otherwise the tiles' squared
// errors, the output layer's g, and what the backward pass needs.
fzp_status forward(fzp_surrogate_s& S, const float* x, int64_t B, const float* y, float* out, cudaStream_t s) {
  const Layer& l0 = S.L[0];
  const bool train = y != nullptr;
  k_inputs<<<blocks(B * l0.n_in), 256, 0, s>>>(B, l0.n_in, x, S.Hb[0], l0.ld_in, train ? S.HTb[0] : nullptr, S.ldB);
  for (size_t l = 0; l < S.L.size(); ++l) {
    const Layer& ly = S.L[l];
    const bool top = l + 1 == S.L.size();
    Gemm p = product(B, ly.n_out, ly.ld_in, S.Hb[l], ly.ld_in, ly.Wb, ly.ld_in, !top ? EPI_HIDDEN : train ? EPI_LOSS : EPI_Y);
    p.bias = S.params + ly.off_b;
    if (!top) {
      p.Z = train ? S.Z[l] : nullptr;
      p.ldz = ly.ld_out;
      p.rows = S.Hb[l + 1];
      p.ldr = S.L[l + 1].ld_in;
      p.cols = train ? S.HTb[l + 1] : nullptr;
      p.ldt = S.ldB;
    } else if (train) {
      p.y = y;
      p.lpart = S.lpart;
      p.rows = S.Gb[0];
      p.ldr = S.maxw;
      p.cols = S.GTb[0];
      p.ldt = S.ldB;
      p.sums = S.sums[0];
      p.ld_sums = S.maxw;
    } else {
      p.C = out;
      p.ldc = ly.n_out;
    }
    const fzp_status st = run_gemm(S, p, nullptr, s);
    if (st != FZP_OK) return st;
  }
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

// Gradients into `grads` (flat, same layout as params) and the loss (if d_loss),
// after forward() on the same batch.  A layer's dW and dh run in one launch; g alternates between two
// buffers, as dh's epilogue writes the next one while dW still reads this one.
fzp_status backward(fzp_surrogate_s& S, int64_t B, float* grads, float* d_loss, cudaStream_t s) {
  const int nl = (int)S.L.size();
  for (int l = nl - 1, cur = 0; l >= 0; --l, cur ^= 1) {
    const Layer& ly = S.L[l];
    // dW = g^T h  (M = n_out, N = n_in, K = B; B is a multiple of 8, so the
    // 8-element loads never reach columns a larger earlier batch left behind)
    Gemm w = product(ly.n_out, ly.n_in, B, S.GTb[cur], S.ldB, S.HTb[l], S.ldB, EPI_DW);
    w.C = grads + ly.off_w;
    w.ldc = ly.n_in;
    w.bsums = S.sums[cur];
    w.ld_sums = S.maxw;
    w.nsums = (int)((B + GM - 1) / GM);
    w.db = grads + ly.off_b;
    if (l == 0) {
      const Layer& lo = S.L[nl - 1];
      w.loss = d_loss;
      w.lpart = S.lpart;
      w.nlpart = (int)(((B + GM - 1) / GM) * ((lo.n_out + GN - 1) / GN));
      w.loss_scale = 1.0 / ((double)B * (double)lo.n_out);
      return run_gemm(S, w, nullptr, s);
    }
    // dh = g W  (M = B, N = n_in, K = n_out), then g = dh silu'(z_{l-1})
    Gemm h = product(B, ly.n_in, ly.ld_out, S.Gb[cur], S.maxw, ly.WTb, ly.ld_out, EPI_DH);
    h.Z = S.Z[l - 1];
    h.ldz = S.L[l - 1].ld_out;
    h.rows = S.Gb[cur ^ 1];
    h.ldr = S.maxw;
    h.cols = S.GTb[cur ^ 1];
    h.ldt = S.ldB;
    h.sums = S.sums[cur ^ 1];
    h.ld_sums = S.maxw;
    const fzp_status st = run_gemm(S, h, &w, s);
    if (st != FZP_OK) return st;
  }
  return FZP_OK;
}

fzp_status refresh_weights(fzp_surrogate_s& S, cudaStream_t s) {
  for (const Layer& ly : S.L)
    k_weights_bf16<<<blocks(ly.n_out * ly.n_in), 256, 0, s>>>(ly.n_out, ly.n_in, S.params + ly.off_w, ly.Wb,
                                                              ly.ld_in, ly.WTb, ly.ld_out);
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status grad_all(fzp_surrogate_s& S, const float* x, const float* y, int64_t B, float* grads, float* d_loss,
                    cudaStream_t s) {
  const fzp_status st = forward(S, x, B, y, nullptr, s);
  return st == FZP_OK ? backward(S, B, grads, d_loss, s) : st;
}

void surrogate_release(fzp_surrogate_s* S) {
  if (!S) return;
  cudaDeviceSynchronize();
  for (void* p : S->allocs)
    if (p) cudaFree(p);
  delete S;
}

}  // namespace

extern "C" {

fzp_status fzp_surrogate_create(int n_in, int hidden, int n_hidden_layers, int n_out, int max_batch, uint64_t seed,
                                fzp_surrogate_t* out) {
  if (!out) return set_error(FZP_E_INVALID, "out is NULL");
  *out = nullptr;
  if (n_in < 1 || hidden < 1 || n_hidden_layers < 1 || n_out < 1 || max_batch < 1 || n_in > 65536 ||
      hidden > 65536 || n_out > 65536 || max_batch > 65536)
    return set_error(FZP_E_INVALID, "surrogate sizes must be in [1, 65536]");
  fzp_surrogate_s* S = new (std::nothrow) fzp_surrogate_s();
  if (!S) return set_error(FZP_E_OOM, "host allocation failed");
  std::vector<int64_t> dims;
  dims.push_back(n_in);
  for (int k = 0; k < n_hidden_layers; ++k) dims.push_back(hidden);
  dims.push_back(n_out);
  int64_t off = 0, maxw = 0;
  for (size_t l = 0; l + 1 < dims.size(); ++l) {
    Layer ly;
    ly.n_in = dims[l];
    ly.n_out = dims[l + 1];
    ly.ld_in = pad64(ly.n_in);
    ly.ld_out = pad64(ly.n_out);
    ly.off_w = off;
    off += ly.n_in * ly.n_out;
    ly.off_b = off;
    off += ly.n_out;
    maxw = std::max(maxw, std::max(ly.ld_in, ly.ld_out));
    S->L.push_back(ly);
  }
  S->n_params = off;
  S->max_batch = max_batch;
  S->ldB = pad64(max_batch);
  S->maxw = maxw;
  auto alloc = [&](size_t bytes) -> void* {
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) return nullptr;
    S->allocs.push_back(p);
    cudaMemset(p, 0, bytes);  // padding must read as zero
    return p;
  };
  bool ok = true;
  auto A = [&](size_t bytes) {
    void* p = alloc(bytes);
    ok = ok && p;
    return p;
  };
  S->params = (float*)A(sizeof(float) * off);
  S->grads = (float*)A(sizeof(float) * off);
  S->m = (float*)A(sizeof(float) * off);
  S->v = (float*)A(sizeof(float) * off);
  S->err = (int*)A(sizeof(int));
  for (Layer& ly : S->L) {
    ly.Wb = (__nv_bfloat16*)A(sizeof(__nv_bfloat16) * ly.n_out * ly.ld_in);
    ly.WTb = (__nv_bfloat16*)A(sizeof(__nv_bfloat16) * ly.n_in * ly.ld_out);
    S->Z.push_back((float*)A(sizeof(float) * max_batch * ly.ld_out));
    S->Hb.push_back((__nv_bfloat16*)A(sizeof(__nv_bfloat16) * max_batch * ly.ld_in));
    S->HTb.push_back((__nv_bfloat16*)A(sizeof(__nv_bfloat16) * ly.ld_in * S->ldB));
  }
  for (int q = 0; q < 2; ++q) {
    S->Gb[q] = (__nv_bfloat16*)A(sizeof(__nv_bfloat16) * max_batch * maxw);
    S->GTb[q] = (__nv_bfloat16*)A(sizeof(__nv_bfloat16) * maxw * S->ldB);
    S->sums[q] = (float*)A(sizeof(float) * (size_t)((max_batch + GM - 1) / GM) * maxw);
  }
  S->lpart = (double*)A(sizeof(double) * (size_t)(((max_batch + GM - 1) / GM) * ((S->L.back().n_out + GN - 1) / GN)));
  if (!ok) {
    cudaGetLastError();
    surrogate_release(S);
    return set_error(FZP_E_OOM, "surrogate allocation failed");
  }
  static std::atomic<uint64_t> attr{0};
  if (smem_attr_once((const void*)k_gemm, GEMM_SMEM, attr) != cudaSuccess) {
    surrogate_release(S);
    return set_error(FZP_E_CUDA, "cudaFuncSetAttribute(k_gemm)");
  }
  // weights ~ U(-1/sqrt(fan_in), 1/sqrt(fan_in)); biases zero
  for (const Layer& ly : S->L)
    k_init_uniform<<<blocks(ly.n_in * ly.n_out), 256>>>(ly.n_in * ly.n_out, S->params + ly.off_w,
                                                       1.f / sqrtf((float)ly.n_in), seed + (uint64_t)ly.off_w);
  fzp_status st = refresh_weights(*S, 0);
  if (st == FZP_OK && cudaDeviceSynchronize() != cudaSuccess) st = set_error(FZP_E_CUDA, "surrogate init failed");
  if (st != FZP_OK) {
    surrogate_release(S);
    return st;
  }
  *out = S;
  return FZP_OK;
}

size_t fzp_surrogate_param_count(fzp_surrogate_t S) { return S ? (size_t)S->n_params : 0; }

fzp_status fzp_surrogate_params(fzp_surrogate_t S, float* h_buf, size_t count, int set) {
  if (!S || !h_buf || count != (size_t)S->n_params) return set_error(FZP_E_INVALID, "bad surrogate or count");
  if (set) {
    FZP_CUDA_TRY(cudaMemcpy(S->params, h_buf, count * sizeof(float), cudaMemcpyHostToDevice));
    fzp_status st = refresh_weights(*S, 0);
    if (st != FZP_OK) return st;
    FZP_CUDA_TRY(cudaDeviceSynchronize());
  } else {
    FZP_CUDA_TRY(cudaMemcpy(h_buf, S->params, count * sizeof(float), cudaMemcpyDeviceToHost));
  }
  return FZP_OK;
}

fzp_status fzp_surrogate_infer(fzp_surrogate_t S, const float* d_x, int batch, float* d_y, void* stream) {
  if (!S || !d_x || !d_y || batch < 1 || batch > S->max_batch) return set_error(FZP_E_INVALID, "bad infer arguments");
  cudaStream_t s = (cudaStream_t)stream;
  return forward(*S, d_x, batch, nullptr, d_y, s);
}

fzp_status fzp_surrogate_grad(fzp_surrogate_t S, const float* d_x, const float* d_y, int batch, float* d_grad,
                              float* d_loss, void* stream) {
  if (!S || !d_x || !d_y || batch < 8 || batch > S->max_batch || (batch % 8) != 0)
    return set_error(FZP_E_INVALID, "bad grad arguments (batch must be a multiple of 8)");
  cudaStream_t s = (cudaStream_t)stream;
  return grad_all(*S, d_x, d_y, batch, d_grad ? d_grad : S->grads, d_loss, s);
}

fzp_status fzp_surrogate_train_step(fzp_surrogate_t S, const float* d_x, const float* d_y, int batch, float lr,
                                    float weight_decay, float* d_loss, void* stream) {
  if (!S || !d_x || !d_y || batch < 8 || batch > S->max_batch || (batch % 8) != 0 || !(lr > 0))
    return set_error(FZP_E_INVALID, "bad train arguments (batch must be a multiple of 8, lr > 0)");
  cudaStream_t s = (cudaStream_t)stream;
  fzp_status st = grad_all(*S, d_x, d_y, batch, S->grads, d_loss, s);
  if (st != FZP_OK) return st;
  S->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)S->step), c2 = 1.f - powf(b2, (float)S->step);
  for (const Layer& ly : S->L)  // off_b follows the layer's weights
    k_adamw<<<blocks((ly.n_in + 1) * ly.n_out), 256, 0, s>>>(ly.n_out, ly.n_in, S->params + ly.off_w, S->grads + ly.off_w,
                                                             S->m + ly.off_w, S->v + ly.off_w, lr, weight_decay, b1, b2,
                                                             1e-8f, c1, c2, ly.Wb, ly.ld_in, ly.WTb, ly.ld_out);
  FZP_CUDA_TRY(cudaGetLastError());
  return FZP_OK;
}

fzp_status fzp_surrogate_destroy(fzp_surrogate_t S) {
  surrogate_release(S);
  return FZP_OK;
}

}  // extern "C"
