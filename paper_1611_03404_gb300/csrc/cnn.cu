// Learned warm start: a small CNN from a source's 5-band 32 x 32 patch to initial variational
// parameters, trained and run by the kernels below (BF16 operands, FP32 accumulation, FP32
// master weights).  Newton remains the solver: the network only supplies its starting point.
//
// Network (NHWC activations, BF16):
//   x [B,32,32,5] -conv3x3 s1-> a1 [B,32,32,32] -conv3x3 s2-> a2 [B,16,16,64]
//     -conv3x3 s2-> a3 [B,8,8,64] -conv3x3 s2-> a4 [B,4,4,64] = [B,1024]
//     -fc-> a5 [B,256] -fc-> y [B,27] (FP32); ReLU after every layer but the last; padding 1.
// Parameters, one FP32 vector (and its BF16 copy), in this order:
//   W1 [32][3][3][5], b1 [32], W2 [64][3][3][32], b2, W3 [64][3][3][64], b3, W4 [64][3][3][64],
//   b4, W5 [256][1024], b5 [256], W6 [27][256], b6 [27].
//
// The forward layers run on tcgen05 (cnn_tc.cu); the mma.sync engine kept beside them is one
// implicit-GEMM kernel (64 x 64 output tiles, k-steps of 32, four warps of 32 x 32 on mma.sync m16n8k16,
// operands gathered element by element).  The backward pass has its own GEMM below.
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cstdint>

#include "celeste_internal.cuh"
#include "cnn_tc.h"
#include "problem.h"

namespace celeste {
namespace cnn {

using bf16 = __nv_bfloat16;

constexpr int IMG = 32, CIN = 5, NOUT = 27;
constexpr int C1 = 32, C2 = 64, C3 = 64, C4 = 64, F5 = 256, FLAT = 4 * 4 * C4;

struct Offsets {
  int64_t w1, b1, w2, b2, w3, b3, w4, b4, w5, b5, w6, b6, total;
};
__host__ __device__ constexpr Offsets offsets() {
  Offsets o{};
  int64_t p = 0;
  o.w1 = p; p += (int64_t)C1 * 9 * CIN;
  o.b1 = p; p += C1;
  o.w2 = p; p += (int64_t)C2 * 9 * C1;
  o.b2 = p; p += C2;
  o.w3 = p; p += (int64_t)C3 * 9 * C2;
  o.b3 = p; p += C3;
  o.w4 = p; p += (int64_t)C4 * 9 * C3;
  o.b4 = p; p += C4;
  o.w5 = p; p += (int64_t)F5 * FLAT;
  o.b5 = p; p += F5;
  o.w6 = p; p += (int64_t)NOUT * F5;
  o.b6 = p; p += NOUT;
  o.total = p;
  return o;
}

// Activation and gradient buffers for a batch of B (BF16 elements, each buffer 256-byte aligned).
struct Ws {
  bf16 *a1, *a2, *a3, *a4, *a5;   // activations after ReLU
  bf16 *d1, *d2, *d3, *d4, *d5;   // gradients w.r.t. those activations' pre-ReLU values
  size_t bytes;
};
inline size_t al256(size_t x) { return (x + 255) & ~size_t(255); }
inline void ws_sizes(int B, size_t (&sz)[5]) {
  sz[0] = (size_t)B * IMG * IMG * C1;
  sz[1] = (size_t)B * 16 * 16 * C2;
  sz[2] = (size_t)B * 8 * 8 * C3;
  sz[3] = (size_t)B * FLAT;
  sz[4] = (size_t)B * F5;
}
inline size_t ws_bytes(int B) {
  size_t sz[5], off = 0;
  ws_sizes(B, sz);
  for (int i = 0; i < 5; ++i) off += 2 * al256(sz[i] * sizeof(bf16));
  return off;
}
inline Ws ws_layout(char* base, int B) {
  size_t sz[5];
  ws_sizes(B, sz);
  Ws w{};
  bf16** act[5] = {&w.a1, &w.a2, &w.a3, &w.a4, &w.a5};
  bf16** grd[5] = {&w.d1, &w.d2, &w.d3, &w.d4, &w.d5};
  size_t off = 0;
  for (int i = 0; i < 5; ++i) {
    *act[i] = reinterpret_cast<bf16*>(base + off);
    off += al256(sz[i] * sizeof(bf16));
    *grd[i] = reinterpret_cast<bf16*>(base + off);
    off += al256(sz[i] * sizeof(bf16));
  }
  w.bytes = off;
  return w;
}

__device__ __forceinline__ bf16 bzero() { return __float2bfloat16(0.f); }

// ------------------------------------------------------------------------------ GEMM core
constexpr int BM = 64, BN = 64, BK = 32, LDS = BK + 8;

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// C[M x N] = sum_k A(m, k) B(k, n) over k in this block's K chunk (blockIdx.z), handed to
// op.store(m, n, value).  op.a / op.b return BF16 operands (zero outside the tensors).
template <class Op>
__global__ void __launch_bounds__(128) gemm_kernel(Op op, int M, int N, int K, int k_chunk) {
  __shared__ __align__(16) bf16 As[BM][LDS];
  __shared__ __align__(16) bf16 Bs[BN][LDS];   // B transposed: Bs[n][k]
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int kb = blockIdx.z * k_chunk, ke = min(K, kb + k_chunk);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32, g = lane >> 2, t = lane & 3;
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
  for (int k0 = kb; k0 < ke; k0 += BK) {
    for (int e = tid; e < BM * BK; e += 128) {
      const int r = e / BK, c = e % BK, k = k0 + c;
      As[r][c] = (m0 + r < M && k < ke) ? op.a(m0 + r, k) : bzero();
      Bs[r][c] = (n0 + r < N && k < ke) ? op.b(k, n0 + r) : bzero();
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; kk += 16) {
      uint32_t a[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = wm + 16 * i + g;
        a[i][0] = *reinterpret_cast<const uint32_t*>(&As[r][kk + 2 * t]);
        a[i][1] = *reinterpret_cast<const uint32_t*>(&As[r + 8][kk + 2 * t]);
        a[i][2] = *reinterpret_cast<const uint32_t*>(&As[r][kk + 2 * t + 8]);
        a[i][3] = *reinterpret_cast<const uint32_t*>(&As[r + 8][kk + 2 * t + 8]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = wn + 8 * j + g;
        const uint32_t b0 = *reinterpret_cast<const uint32_t*>(&Bs[c][kk + 2 * t]);
        const uint32_t b1 = *reinterpret_cast<const uint32_t*>(&Bs[c][kk + 2 * t + 8]);
#pragma unroll
        for (int i = 0; i < 2; ++i) mma16816(acc[i][j], a[i], b0, b1);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int m = m0 + wm + 16 * i + g + (e >> 1) * 8, n = n0 + wn + 8 * j + 2 * t + (e & 1);
        if (m < M && n < N) op.store(m, n, acc[i][j][e]);
      }
}

template <class Op>
cudaError_t gemm(const Op& op, int M, int N, int K, int splits, cudaStream_t st) {
  splits = std::max(1, std::min(splits, (K + BK - 1) / BK));
  int chunk = (K + splits - 1) / splits;
  chunk = (chunk + BK - 1) / BK * BK;
  splits = (K + chunk - 1) / chunk;
  dim3 grid((M + BM - 1) / BM, (N + BN - 1) / BN, splits);
  gemm_kernel<Op><<<grid, 128, 0, st>>>(op, M, N, K, chunk);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ convolution ops
struct ConvGeom {
  int B, H, W, Cin, OH, OW, Cout, stride;
};

// out[b, oh, ow, co] = relu(bias[co] + sum_{kh, kw, ci} in[b, oh s + kh - 1, ow s + kw - 1, ci] W[co, kh, kw, ci])
struct ConvFwd {
  ConvGeom g;
  const bf16* in;
  const bf16* w;
  const float* bias;
  bf16* out;
  __device__ bf16 a(int m, int k) const {
    const int ow = m % g.OW, r = m / g.OW, oh = r % g.OH, b = r / g.OH;
    const int ci = k % g.Cin, kk = k / g.Cin, kh = kk / 3, kw = kk % 3;
    const int ih = oh * g.stride + kh - 1, iw = ow * g.stride + kw - 1;
    if (ih < 0 || ih >= g.H || iw < 0 || iw >= g.W) return bzero();
    return in[(((size_t)b * g.H + ih) * g.W + iw) * g.Cin + ci];
  }
  __device__ bf16 b(int k, int n) const { return w[(size_t)n * 9 * g.Cin + k]; }
  __device__ void store(int m, int n, float v) const {
    out[(size_t)m * g.Cout + n] = __float2bfloat16(fmaxf(v + bias[n], 0.f));
  }
};

// ------------------------------------------------------------------------------ dense ops
// y[b, o] = act(bias[o] + sum_i x[b, i] W[o, i]); the last layer writes FP32, optionally mapped
// to parameter space as y * scale[o] + shift[o].
struct FcFwd {
  int Nin, Nout;
  const bf16* x;
  const bf16* w;
  const float* bias;
  bf16* out_bf;
  float* out_f;
  const float* scale;
  const float* shift;
  __device__ bf16 a(int m, int k) const { return x[(size_t)m * Nin + k]; }
  __device__ bf16 b(int k, int n) const { return w[(size_t)n * Nin + k]; }
  __device__ void store(int m, int n, float v) const {
    v += bias[n];
    if (out_bf) {
      out_bf[(size_t)m * Nout + n] = __float2bfloat16(fmaxf(v, 0.f));
    } else {
      if (scale) v = v * scale[n] + shift[n];
      out_f[(size_t)m * Nout + n] = v;
    }
  }
};

// ------------------------------------------------------------------------------ backward GEMM
// C[M x N] = sum_k A(m, k) B(k, n) on mma.sync m16n8k16 (BF16 in, FP32 accumulate), operands brought in
// 16-byte chunks by cp.async, three stages of 64 x 64 deep, read with ldmatrix.  A lies in memory either
// with k contiguous (rows m: the input gradients) or with m contiguous (rows k: the weight gradients), B
// always with n contiguous (rows k); ldmatrix.trans turns the latter two.  blockIdx.z splits K, or is the
// operation's own index (parity classes of an input gradient).
// What bounds it: reading the operands (a layer's gradients from L2 at the training batch); before, every
// element was gathered and converted on its own, and an input gradient multiplied the three quarters of
// a stride-2 layer's taps that are zero.  A whole training step at batch 512:
// 4.75 ms before, 0.31 now, of which 0.21 is the backward pass.
constexpr int BK2 = 64, LD2 = 72, STAGES2 = 3;     // rows of 64 values, 16 bytes apart from a multiple of 128

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes global -> shared, asynchronously; zeros where !ok (the source is then not read, but has to lie on a
// 16-byte boundary all the same: the operations' any() is an address in the workspace).
__device__ __forceinline__ void copy16(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
// The same from a caller's array, which may start off a 16-byte boundary (then element by element, visible
// after the next barrier).
__device__ __forceinline__ void copy16_any(bf16* dst, const bf16* src, bool ok) {
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    copy16(dst, src, ok);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) dst[i] = ok ? src[i] : __float2bfloat16(0.f);
  }
}
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)) : "memory");
}

// A 16 x 16 operand block at (row, col) of a tile with rows of LD values: as A from [m][k], as A from
// [k][m], and as two adjacent B blocks (n .. n + 15) from [k][n].
template <int LD>
__device__ __forceinline__ void frag_a(uint32_t (&r)[4], const bf16* T, int m, int k, int lane) {
  ldsm4(r, T + (m + (lane & 15)) * LD + k + 8 * (lane >> 4));
}
template <int LD>
__device__ __forceinline__ void frag_at(uint32_t (&r)[4], const bf16* T, int m, int k, int lane) {
  ldsm4t(r, T + (k + (lane & 7) + 8 * (lane >> 4)) * LD + m + 8 * ((lane >> 3) & 1));
}
template <int LD>
__device__ __forceinline__ void frag_b(uint32_t (&r)[4], const bf16* T, int k, int n, int lane) {
  ldsm4t(r, T + (k + (lane & 15)) * LD + n + 8 * (lane >> 4));
}

template <class Op>
__global__ void __launch_bounds__(128) bwd_gemm_kernel(Op op, int M, int N, int K, int k_chunk) {
  constexpr int BN2 = Op::BN;                       // 64, or 32 (then a warp takes 16 rows of C, else 32)
  constexpr int MI = BN2 == 64 ? 2 : 1;             // 16-row blocks per warp; always 32 columns
  extern __shared__ __align__(16) unsigned char dyn[];
  bf16* const As = reinterpret_cast<bf16*>(dyn);
  bf16* const Bs = As + STAGES2 * 64 * LD2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m0 = blockIdx.x * 64, n0 = blockIdx.y * BN2;
  const int wm = MI == 2 ? (warp >> 1) * 32 : warp * 16, wn = MI == 2 ? (warp & 1) * 32 : 0;
  const int c = tid & 7, r0 = tid >> 3;             // this thread's chunk and first row (then every 16th)
  int kb, ke;
  op.range(blockIdx.z, k_chunk, K, kb, ke);
  op.rows(m0, r0, M);                               // what the thread's rows need for all of K
  const int steps = (ke - kb + BK2 - 1) / BK2;
  auto fetch = [&](int s) {
    if (s < steps) {
      const int k0 = kb + s * BK2;
      bf16* A = As + (s % STAGES2) * 64 * LD2;
      bf16* B = Bs + (s % STAGES2) * 64 * LD2;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + 16 * i;
        bool ok;
        const bf16* p = Op::A_K ? op.a(i, k0, k0 + 8 * c, ke, ok) : op.at(k0 + r, m0 + 8 * c, M, ke, ok);
        copy16(A + r * LD2 + 8 * c, ok ? p : op.any(), ok);
        if (8 * c < BN2) {
          const bf16* q = op.b(k0, k0 + r, n0 + 8 * c, N, ke, ok);
          copy16_any(B + r * LD2 + 8 * c, ok ? q : op.any(), ok);
        }
      }
    }
    cp_async_commit();
  };
  float acc[MI][4][4];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
  fetch(0);
  fetch(1);
  for (int s = 0; s < steps; ++s) {
    copy_wait<1>();
    __syncthreads();   // step s is there for every thread; step s - 1 has been read
    fetch(s + 2);
    const bf16* A = As + (s % STAGES2) * 64 * LD2;
    const bf16* B = Bs + (s % STAGES2) * 64 * LD2;
#pragma unroll
    for (int kk = 0; kk < BK2; kk += 16) {
      if (kb + s * BK2 + kk >= ke) break;            // (blocks past K hold zeros)
      uint32_t a[MI][4], b[2][4];
#pragma unroll
      for (int i = 0; i < MI; ++i) {
        if constexpr (Op::A_K) frag_a<LD2>(a[i], A, wm + 16 * i, kk, lane);
        else frag_at<LD2>(a[i], A, wm + 16 * i, kk, lane);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) frag_b<LD2>(b[j], B, kk, wn + 16 * j, lane);
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < MI; ++i) mma16816(acc[i][j], a[i], b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]);
    }
  }
  copy_wait<0>();
  const int g = lane >> 2, t = lane & 3;
  if constexpr (Op::SUM) {
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int m = m0 + wm + 16 * i + g + (e >> 1) * 8, n = n0 + wn + 8 * j + 2 * t + (e & 1);
          if (m < M && n < N) op.add(m, n, acc[i][j][e]);
        }
  } else {
    // BF16 rows of the tile through shared memory, then 16 bytes of a row per thread
    __syncthreads();
    bf16* C = As;
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<__nv_bfloat162*>(C + (wm + 16 * i + g + 8 * h) * LD2 + wn + 8 * j + 2 * t) =
              __floats2bfloat162_rn(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
    __syncthreads();
    for (int e = tid; e < 64 * (BN2 / 8); e += 128) {
      const int r = e / (BN2 / 8), ch = e % (BN2 / 8), m = m0 + r, n = n0 + 8 * ch;
      if (m < M && n < N) op.store(blockIdx.z, m, n, *reinterpret_cast<const uint4*>(C + r * LD2 + 8 * ch));
    }
  }
}

template <class Op>
cudaError_t bwd_gemm(const Op& op, int M, int N, int K, int z, int k_chunk, cudaStream_t st) {
  constexpr int smem = 2 * STAGES2 * 64 * LD2 * (int)sizeof(bf16);
  cudaError_t e = cudaFuncSetAttribute(bwd_gemm_kernel<Op>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  bwd_gemm_kernel<Op><<<dim3((M + 63) / 64, (N + Op::BN - 1) / Op::BN, z), 128, smem, st>>>(op, M, N, K, k_chunk);
  return cudaGetLastError();
}

// The value where the layer's activation was positive, else 0 (the gradient w.r.t. the pre-ReLU value).
__device__ __forceinline__ uint4 relu_mask(uint4 v, const bf16* act) {
  const uint4 x = *reinterpret_cast<const uint4*>(act);
  auto one = [](uint32_t v, uint32_t x) {
    // positive BF16: sign clear, not zero (activations are never NaN after ReLU's maximum)
    const uint32_t lo = (x & 0x8000u) == 0 && (x & 0x7fffu) ? 0xffffu : 0u;
    const uint32_t hi = (x & 0x80000000u) == 0 && (x & 0x7fff0000u) ? 0xffff0000u : 0u;
    return v & (lo | hi);
  };
  return make_uint4(one(v.x, x.x), one(v.y, x.y), one(v.z, x.z), one(v.w, x.w));
}

// Input gradient of a 3x3, stride-2, padding-1 convolution with 64 output channels, one parity class of the
// input pixels (z = 2 (ih & 1) + (iw & 1)) at a time: an even coordinate is reached by tap 1 alone, an odd one by
// taps 0 (from the next output) and 2, so the classes have 1, 2, 2 and 4 taps, taken in ascending order.
// Rows: (b, ih / 2, iw / 2).  din = [in > 0] sum_{taps, co} dout[b, oh, ow, co] W[co, kh, kw, ci].
template <int O, int CIN>
struct ConvDgrad {
  static constexpr bool A_K = true, SUM = false;
  static constexpr int BN = CIN;
  const bf16 *dout, *w, *in;
  bf16* din;
  int pi, pj;
  const bf16* row[4];
  int edge[4];   // 1: no output below, 2: none to the right, 4: no row at all
  __device__ const bf16* any() const { return dout; }
  __device__ void range(int z, int, int, int& kb, int& ke) {
    pi = z >> 1;
    pj = z & 1;
    kb = 0;
    ke = 64 * (1 + pi) * (1 + pj);
  }
  __device__ void rows(int m0, int r0, int M) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + r0 + 16 * i, j = m % O, y = m / O % O;
      row[i] = dout + (int64_t)m * 64;
      edge[i] = (y == O - 1 ? 1 : 0) | (j == O - 1 ? 2 : 0) | (m >= M ? 4 : 0);
    }
  }
  // tap number t of the class: output offsets (dh, dw), kernel position
  __device__ void tap(int t, int& dh, int& dw, int& kk) const {
    const int th = pj ? t >> 1 : t, tw = pj ? t & 1 : 0;
    dh = pi ? 1 - th : 0;
    dw = pj ? 1 - tw : 0;
    kk = 3 * (pi ? 2 * th : 1) + (pj ? 2 * tw : 1);
  }
  __device__ const bf16* a(int i, int k0, int k, int, bool& ok) const {
    int dh, dw, kk;
    tap(k0 >> 6, dh, dw, kk);
    ok = !(edge[i] & (4 | dh | (dw << 1)));
    return row[i] + (dh * O + dw) * 64 + (k & 63);
  }
  __device__ const bf16* at(int, int, int, int, bool&) const { return nullptr; }
  __device__ const bf16* b(int k0, int k, int n, int, int, bool& ok) const {
    int dh, dw, kk;
    tap(k0 >> 6, dh, dw, kk);
    ok = true;
    return w + ((k & 63) * 9 + kk) * CIN + n;
  }
  __device__ void store(int z, int m, int n, uint4 v) const {
    const int j = m % O, y = m / O % O, b = m / (O * O);
    const int64_t at = (((int64_t)b * (2 * O) + 2 * y + (z >> 1)) * (2 * O) + 2 * j + (z & 1)) * CIN + n;
    *reinterpret_cast<uint4*>(din + at) = relu_mask(v, in + at);
  }
  __device__ void add(int, int, float) const {}
};

// K split of the weight gradients.
struct SplitK {
  __device__ static void range(int z, int chunk, int K, int& kb, int& ke) {
    kb = z * chunk;
    ke = min(K, kb + chunk);
  }
};

// Weight gradient of the same convolutions: dW[co, tap, ci] += sum_px dout[px, co] in[px's tap, ci].
template <int O, int CIN>
struct ConvWgrad : SplitK {
  static constexpr bool A_K = false, SUM = true;
  static constexpr int BN = 64;
  const bf16 *dout, *in;
  float* dw;
  __device__ const bf16* any() const { return in; }
  __device__ void rows(int, int, int) {}
  __device__ const bf16* a(int, int, int, int, bool&) const { return nullptr; }
  __device__ const bf16* at(int k, int m, int, int ke, bool& ok) const {
    ok = k < ke;
    return dout + (int64_t)k * 64 + m;
  }
  __device__ const bf16* b(int, int k, int n, int N, int ke, bool& ok) const {
    const int tap = n / CIN, kh = tap / 3, kw = tap % 3, ow = k % O, oh = k / O % O, b = k / (O * O);
    const int y = 2 * oh + kh - 1, x = 2 * ow + kw - 1;   // (never past the lower or right edge)
    ok = k < ke && n < N && y >= 0 && x >= 0;
    return in + (((int64_t)b * (2 * O) + y) * (2 * O) + x) * CIN + n % CIN;
  }
  __device__ void add(int m, int n, float v) const { atomicAdd(dw + m * 9 * CIN + n, v); }
  __device__ void store(int, int, int, uint4) const {}
};

// Dense layers; dy [B][LDY] with NOUT values in use.
// dx[b, i] = [x > 0] sum_o dy[b, o] W[o, i]
template <int NIN, int NOUT, int LDY>
struct FcDgrad : SplitK {
  static constexpr bool A_K = true, SUM = false;
  static constexpr int BN = 64;
  const bf16 *dy, *w, *x;
  bf16* dx;
  const bf16* row[4];
  bool in_range[4];
  __device__ const bf16* any() const { return dy; }
  __device__ void rows(int m0, int r0, int M) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      row[i] = dy + (int64_t)(m0 + r0 + 16 * i) * LDY;
      in_range[i] = m0 + r0 + 16 * i < M;
    }
  }
  __device__ const bf16* a(int i, int, int k, int, bool& ok) const {
    ok = in_range[i] && k < LDY;
    return row[i] + k;
  }
  __device__ const bf16* at(int, int, int, int, bool&) const { return nullptr; }
  __device__ const bf16* b(int, int k, int n, int, int, bool& ok) const {
    ok = k < NOUT;
    return w + (int64_t)k * NIN + n;
  }
  __device__ void store(int, int m, int n, uint4 v) const {
    *reinterpret_cast<uint4*>(dx + (int64_t)m * NIN + n) = relu_mask(v, x + (int64_t)m * NIN + n);
  }
  __device__ void add(int, int, float) const {}
};
// dW[o, i] += sum_b dy[b, o] x[b, i]
template <int NIN, int NOUT, int LDY>
struct FcWgrad : SplitK {
  static constexpr bool A_K = false, SUM = true;
  static constexpr int BN = 64;
  const bf16 *dy, *x;
  float* dw;
  __device__ const bf16* any() const { return x; }
  __device__ void rows(int, int, int) {}
  __device__ const bf16* a(int, int, int, int, bool&) const { return nullptr; }
  __device__ const bf16* at(int k, int m, int, int ke, bool& ok) const {
    ok = k < ke && m < LDY;
    return dy + (int64_t)k * LDY + m;
  }
  __device__ const bf16* b(int, int k, int n, int, int ke, bool& ok) const {
    ok = k < ke;
    return x + (int64_t)k * NIN + n;
  }
  __device__ void add(int m, int n, float v) const { atomicAdd(dw + (int64_t)m * NIN + n, v); }
  __device__ void store(int, int, int, uint4) const {}
};

// The last layer's gradient [B][27] in BF16 rows of 32 (zeros after the 27).
constexpr int LDY6 = 32;
__global__ void last_grad_kernel(const float* __restrict__ dy, int B, bf16* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)B * LDY6; i += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(i % LDY6);
    out[i] = __float2bfloat16(n < NOUT ? dy[i / LDY6 * NOUT + n] : 0.f);
  }
}

// First layer's weight gradient, dW[co, kh, kw, ci] += sum_px d[px, co] x[px's window]: the windows are 45 values
// at a 10-byte stride, so a warp builds them (rows of 48) from the image kept in shared memory, 16 bytes a
// pixel with a border of zeros, one image row of 32 pixels at a time, and multiplies 32 x 48 blocks; a
// CTA's warps take every fourth row of its images and add up in shared memory at the end.
constexpr int W1_IMG_LD = 40, W1_LDB = 56, W1_LDA = 40;
struct W1Smem {
  uint4 img[34 * W1_IMG_LD];
  bf16 Bt[4][32 * W1_LDB], At[4][2][32 * W1_LDA];
  float sum[C1 * 48];
};
__global__ void __launch_bounds__(128) conv1_wgrad_kernel(const bf16* __restrict__ x, const bf16* __restrict__ d, int B,
                                                          float* __restrict__ dw) {
  extern __shared__ __align__(16) unsigned char dyn[];
  W1Smem& S = *reinterpret_cast<W1Smem*>(dyn);
  uint4* const img = S.img;
  auto& Bt = S.Bt;
  auto& At = S.At;
  float* const sum = S.sum;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto at = [](int p) { return p + (p >> 3); };   // a gap after every eighth pixel spreads the writes over the banks
  for (int i = tid; i < 34 * W1_IMG_LD; i += 128) img[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < C1 * 48; i += 128) sum[i] = 0.f;
  float acc[2][6][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
  for (int b = blockIdx.x; b < B; b += gridDim.x) {
    const bf16* dimg = d + (int64_t)b * (IMG * IMG * C1);
    auto fetch = [&](int q) {   // this warp's q-th row of the image: 32 pixels x 32 channels
      if (q < 8) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int e = lane + 32 * i, r = e >> 2, c = e & 3;
          copy16(At[warp][q & 1] + r * W1_LDA + 8 * c, dimg + ((4 * q + warp) * 32 + r) * C1 + 8 * c, true);
        }
      }
      cp_async_commit();
    };
    fetch(0);
    __syncthreads();   // the previous image has been read
    const uint16_t* src = reinterpret_cast<const uint16_t*>(x) + (int64_t)b * (IMG * IMG * CIN);
    for (int p = tid; p < IMG * IMG; p += 128) {
      const uint16_t* s = src + 5 * p;
      img[((p >> 5) + 1) * W1_IMG_LD + at((p & 31) + 1)] =
          make_uint4(s[0] | ((uint32_t)s[1] << 16), s[2] | ((uint32_t)s[3] << 16), s[4], 0u);
    }
    __syncthreads();
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
      fetch(q + 1);
      // windows of output row 4 q + warp, lane = column: three runs of 15 values
      uint32_t r[3][8];
#pragma unroll
      for (int kh = 0; kh < 3; ++kh) {
        const uint4* p = img + (4 * q + warp + kh) * W1_IMG_LD;
        const uint4 p0 = p[at(lane)], p1 = p[at(lane + 1)], p2 = p[at(lane + 2)];
        r[kh][0] = p0.x;
        r[kh][1] = p0.y;
        r[kh][2] = p0.z | (p1.x << 16);
        r[kh][3] = __funnelshift_r(p1.x, p1.y, 16);
        r[kh][4] = __funnelshift_r(p1.y, p1.z, 16);
        r[kh][5] = p2.x;
        r[kh][6] = p2.y;
        r[kh][7] = p2.z;
      }
      uint4* o = reinterpret_cast<uint4*>(Bt[warp] + lane * W1_LDB);
      o[0] = make_uint4(r[0][0], r[0][1], r[0][2], r[0][3]);
      o[1] = make_uint4(r[0][4], r[0][5], r[0][6], r[0][7] | (r[1][0] << 16));
      o[2] = make_uint4(__funnelshift_r(r[1][0], r[1][1], 16), __funnelshift_r(r[1][1], r[1][2], 16),
                        __funnelshift_r(r[1][2], r[1][3], 16), __funnelshift_r(r[1][3], r[1][4], 16));
      o[3] = make_uint4(__funnelshift_r(r[1][4], r[1][5], 16), __funnelshift_r(r[1][5], r[1][6], 16),
                        __funnelshift_r(r[1][6], r[1][7], 16), r[2][0]);
      o[4] = make_uint4(r[2][1], r[2][2], r[2][3], r[2][4]);
      o[5] = make_uint4(r[2][5], r[2][6], r[2][7], 0u);
      copy_wait<1>();
      __syncwarp();
      const bf16* A = At[warp][q & 1];
#pragma unroll
      for (int kk = 0; kk < 32; kk += 16) {
        uint32_t a[2][4], bb[3][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) frag_at<W1_LDA>(a[i], A, 16 * i, kk, lane);
#pragma unroll
        for (int j = 0; j < 3; ++j) frag_b<W1_LDB>(bb[j], Bt[warp], kk, 16 * j, lane);
#pragma unroll
        for (int j = 0; j < 6; ++j)
#pragma unroll
          for (int i = 0; i < 2; ++i) mma16816(acc[i][j], a[i], bb[j >> 1][2 * (j & 1)], bb[j >> 1][2 * (j & 1) + 1]);
      }
      __syncwarp();   // the windows and the row's buffer are rewritten
    }
    copy_wait<0>();
  }
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) atomicAdd(&sum[(16 * i + g + (e >> 1) * 8) * 48 + 8 * j + 2 * t + (e & 1)], acc[i][j][e]);
  __syncthreads();
  for (int i = tid; i < C1 * 9 * CIN; i += 128) atomicAdd(dw + i, sum[i / 45 * 48 + i % 45]);
}

// Bias gradients of all layers, db[c] += sum over rows of g[r, c]: blockIdx.y is the layer; a thread adds up 8
// channels of every so many rows, the block its threads.
struct BiasJob {
  const bf16* g;       // [rows][C] (null: the FP32 one)
  const float* gf;
  int64_t rows;
  int C;
  float* db;
};
struct BiasJobs {
  BiasJob j[6];
};
__global__ void __launch_bounds__(256) bias_grad_kernel(BiasJobs jobs) {
  const BiasJob J = jobs.j[blockIdx.y];
  __shared__ float sum[F5];
  for (int c = threadIdx.x; c < J.C; c += 256) sum[c] = 0.f;
  __syncthreads();
  if (J.g) {
    const int groups = J.C / 8, c = threadIdx.x % groups, lanes = 256 / groups;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int64_t r = (int64_t)blockIdx.x * lanes + threadIdx.x / groups; r < J.rows; r += (int64_t)gridDim.x * lanes) {
      const uint4 v = *reinterpret_cast<const uint4*>(J.g + r * J.C + 8 * c);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        s[2 * i] += __uint_as_float(w[i] << 16);
        s[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) atomicAdd(&sum[8 * c + i], s[i]);
  } else {
    const int lanes = 256 / J.C, c = threadIdx.x % J.C, l = threadIdx.x / J.C;
    float s = 0.f;
    if (l < lanes)
      for (int64_t r = (int64_t)blockIdx.x * lanes + l; r < J.rows; r += (int64_t)gridDim.x * lanes) s += J.gf[r * J.C + c];
    if (l < lanes) atomicAdd(&sum[c], s);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < J.C; c += 256) atomicAdd(J.db + c, sum[c]);
}

// ------------------------------------------------------------------------------ small kernels
// Counter-based standard normal (SplitMix64 of seed and index, Box-Muller).
__device__ inline uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
__device__ inline float normal_at(uint64_t seed, int64_t i) {
  const uint64_t h1 = splitmix64(seed * 0x100000001B3ULL + 2 * (uint64_t)i);
  const uint64_t h2 = splitmix64(seed * 0x100000001B3ULL + 2 * (uint64_t)i + 1);
  const float u1 = ((h1 >> 40) + 0.5f) * (1.0f / 16777216.0f), u2 = (h2 >> 40) * (1.0f / 16777216.0f);
  return sqrtf(-2.f * logf(u1)) * cospif(2.f * u2);
}

// He-normal weights (std sqrt(2 / fan_in)), zero biases; the last layer scaled by 0.1.
__global__ void init_kernel(float* p, bf16* pb, uint64_t seed) {
  constexpr Offsets o = offsets();
  const int64_t n = o.total;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float fan = 0.f, scale = 1.f;
    if (i < o.b1) fan = 9 * CIN;
    else if (i >= o.w2 && i < o.b2) fan = 9 * C1;
    else if (i >= o.w3 && i < o.b3) fan = 9 * C2;
    else if (i >= o.w4 && i < o.b4) fan = 9 * C3;
    else if (i >= o.w5 && i < o.b5) fan = FLAT;
    else if (i >= o.w6 && i < o.b6) { fan = F5; scale = 0.1f; }
    const float v = fan > 0.f ? scale * sqrtf(2.f / fan) * normal_at(seed, i) : 0.f;
    p[i] = v;
    pb[i] = __float2bfloat16(v);
  }
}

// loss += sum_{b, j} w_j (y - t)^2 / (B * 27);  dy = 2 w_j (y - t) / (B * 27)
__global__ void mse_kernel(const float* y, const float* t, const float* w, int n, float* dy, double* loss) {
  __shared__ float red[8];
  const float inv = 1.f / (float)n;
  float s = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float wj = w ? w[i % NOUT] : 1.f, d = y[i] - t[i];
    s += wj * d * d * inv;
    dy[i] = 2.f * wj * d * inv;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.f;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) v += red[i];
    atomicAdd(loss, (double)v);
  }
}

// AdamW with bias correction; the BF16 copy follows the FP32 master weights.
__global__ void adamw_kernel(float* p, bf16* pb, float* m, float* v, const float* g, int64_t n, float lr, float b1,
                             float b2, float eps, float wd, float c1, float c2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] * (1.f - lr * wd) - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    pb[i] = __float2bfloat16(pi);
  }
}

// x[s, i, j, b] = asinh((pixel - sky) / sqrt(sky)) on the 32 x 32 window whose pixel (16, 16) is
// the source's patch centre, taken from the first exposure of band b that holds the source (zero
// where the band is missing or the window leaves the image).
__global__ void extract_patches_kernel(ProblemDev P, bf16* x) {
  const int s = blockIdx.x;
  int img[5] = {-1, -1, -1, -1, -1}, cx[5], cy[5];
  for (int q = P.src_patch[s]; q < P.src_patch[s + 1]; ++q) {
    const PatchDev pt = P.patches[q];
    const ImageDev& im = P.images[pt.image];
    if (img[im.band] >= 0) continue;
    img[im.band] = pt.image;
    const double u = P.u0[2 * s], v = P.u0[2 * s + 1];
    cx[im.band] = (int)floor(im.A[0] * u + im.A[1] * v + im.o[0] + 0.5);
    cy[im.band] = (int)floor(im.A[2] * u + im.A[3] * v + im.o[1] + 0.5);
  }
  for (int e = threadIdx.x; e < IMG * IMG * CIN; e += blockDim.x) {
    const int b = e % CIN, j = (e / CIN) % IMG, i = e / (CIN * IMG);
    float val = 0.f;
    if (img[b] >= 0) {
      const ImageDev& im = P.images[img[b]];
      const int r = cy[b] - 16 + i, c = cx[b] - 16 + j;
      if (r >= 0 && r < im.H && c >= 0 && c < im.W)
        val = asinhf((im.pixels[(size_t)r * im.W + c] - im.sky) * rsqrtf(im.sky));
    }
    x[(size_t)s * IMG * IMG * CIN + e] = __float2bfloat16(val);
  }
}

}  // namespace cnn
}  // namespace celeste

using namespace celeste;
using namespace celeste::cnn;

extern "C" int64_t celeste_cnn_param_count(void) { return offsets().total; }

extern "C" size_t celeste_cnn_workspace_bytes(int batch) {
  if (batch <= 0) return 0;
  return ws_bytes(batch);
}

extern "C" int celeste_cnn_init(float* params, uint16_t* params_bf16, uint64_t seed, celeste_stream_t stream) {
  if (!params || !params_bf16) return fail(CELESTE_ERR_INVALID_ARG, "null parameter buffer");
  init_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(params, reinterpret_cast<bf16*>(params_bf16), seed);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? CELESTE_OK : cuda_fail(e, "cnn init");
}

static int check_ws(int batch, const void* ws, size_t bytes) {
  if (batch <= 0) return fail(CELESTE_ERR_INVALID_ARG, "batch must be > 0");
  if (!ws || reinterpret_cast<uintptr_t>(ws) % 256) return fail(CELESTE_ERR_WORKSPACE, "workspace must be 256-byte aligned");
  if (bytes < ws_bytes(batch)) return fail(CELESTE_ERR_WORKSPACE, "workspace needs %zu bytes", ws_bytes(batch));
  return CELESTE_OK;
}

// Error word of the tensor-core forward path (a bounded wait that ran out).
static __device__ int g_cnn_tc_err;

extern "C" int celeste_cnn_status(void) {
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_cnn_tc_err, sizeof(int));
  if (e != cudaSuccess) return cuda_fail(e, "cnn status");
  if (!v) return CELESTE_OK;
  const int zero = 0;
  cudaMemcpyToSymbol(g_cnn_tc_err, &zero, sizeof(int));
  return fail(CELESTE_ERR_TIMEOUT, "a tensor-core product of the network did not complete in time");
}

extern "C" int celeste_cnn_forward(const float* params, const uint16_t* params_bf16, const uint16_t* x, int batch,
                                   const float* out_scale, const float* out_shift, float* y, void* ws,
                                   size_t ws_bytes, celeste_stream_t stream) {
  return celeste_cnn_forward_ex(params, params_bf16, x, batch, out_scale, out_shift, y, ws, ws_bytes,
                                CELESTE_CNN_TCGEN05, stream);
}

extern "C" int celeste_cnn_forward_ex(const float* params, const uint16_t* params_bf16, const uint16_t* x, int batch,
                                      const float* out_scale, const float* out_shift, float* y, void* ws,
                                      size_t ws_bytes, int engine, celeste_stream_t stream) {
  return celeste_cnn_forward_budget(params, params_bf16, x, batch, out_scale, out_shift, y, ws, ws_bytes, engine, 0,
                                    stream);
}

extern "C" int celeste_cnn_forward_budget(const float* params, const uint16_t* params_bf16, const uint16_t* x,
                                          int batch, const float* out_scale, const float* out_shift, float* y,
                                          void* ws, size_t ws_bytes, int engine, long long wait_budget,
                                          celeste_stream_t stream) {
  if (!params || !params_bf16 || !x || !y) return fail(CELESTE_ERR_INVALID_ARG, "null argument");
  if ((out_scale == nullptr) != (out_shift == nullptr)) return fail(CELESTE_ERR_INVALID_ARG, "scale and shift go together");
  if (engine != CELESTE_CNN_MMA_SYNC && engine != CELESTE_CNN_TCGEN05)
    return fail(CELESTE_ERR_INVALID_ARG, "engine must be CELESTE_CNN_MMA_SYNC or CELESTE_CNN_TCGEN05");
  if (engine == CELESTE_CNN_TCGEN05 && reinterpret_cast<uintptr_t>(params_bf16) % 16)
    return fail(CELESTE_ERR_INVALID_ARG, "params_bf16 must be 16-byte aligned (it is copied 16 bytes at a time)");
  if (batch > INT_MAX / (IMG * IMG))   // (the first layer's rows, one per pixel, are an int)
    return fail(CELESTE_ERR_INVALID_ARG, "batch must be at most %d", INT_MAX / (IMG * IMG));
  int rc = check_ws(batch, ws, ws_bytes);
  if (rc != CELESTE_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  constexpr Offsets o = offsets();
  const bf16* pb = reinterpret_cast<const bf16*>(params_bf16);
  const Ws w = ws_layout(static_cast<char*>(ws), batch);
  const int B = batch;
  const bf16* xin = reinterpret_cast<const bf16*>(x);
  cudaError_t e;
  ConvGeom g1{B, 32, 32, CIN, 32, 32, C1, 1}, g2{B, 32, 32, C1, 16, 16, C2, 2};
  ConvGeom g3{B, 16, 16, C2, 8, 8, C3, 2}, g4{B, 8, 8, C3, 4, 4, C4, 2};
  if (engine == CELESTE_CNN_TCGEN05) {
    int* err = nullptr;
    if ((e = cudaGetSymbolAddress(reinterpret_cast<void**>(&err), g_cnn_tc_err)) != cudaSuccess)
      return cuda_fail(e, "cnn error word");
    int dev = 0, n_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return cuda_fail(e, "SM count");
    auto layer = [&](cnn_tc::LayerId id, int m, int n, const bf16* in, int64_t wo, int64_t bo, bf16* out, float* outf) {
      cnn_tc::Args a{};
      a.M = m, a.N = n, a.B = B;
      a.in = in, a.w = pb + wo, a.bias = params + bo, a.out = out, a.out_f = outf, a.err = err;
      a.wait_budget = wait_budget ? wait_budget : WAIT_BUDGET_DEFAULT;
      if (outf) a.scale = out_scale, a.shift = out_shift;
      return tc_forward(id, a, n_sm, st);
    };
    if ((e = layer(cnn_tc::CONV1, B * 1024, C1, xin, o.w1, o.b1, w.a1, nullptr)) != cudaSuccess ||
        (e = layer(cnn_tc::CONV2, B * 256, C2, w.a1, o.w2, o.b2, w.a2, nullptr)) != cudaSuccess ||
        (e = layer(cnn_tc::CONV3, B * 64, C3, w.a2, o.w3, o.b3, w.a3, nullptr)) != cudaSuccess ||
        (e = layer(cnn_tc::CONV4, B * 16, C4, w.a3, o.w4, o.b4, w.a4, nullptr)) != cudaSuccess ||
        (e = layer(cnn_tc::DENSE1, B, F5, w.a4, o.w5, o.b5, w.a5, nullptr)) != cudaSuccess ||
        (e = layer(cnn_tc::DENSE2, B, NOUT, w.a5, o.w6, o.b6, nullptr, y)) != cudaSuccess)
      return cuda_fail(e, "cnn forward (tensor cores)");
    return CELESTE_OK;
  }
  if ((e = gemm(ConvFwd{g1, xin, pb + o.w1, params + o.b1, w.a1}, B * 1024, C1, 9 * CIN, 1, st)) != cudaSuccess ||
      (e = gemm(ConvFwd{g2, w.a1, pb + o.w2, params + o.b2, w.a2}, B * 256, C2, 9 * C1, 1, st)) != cudaSuccess ||
      (e = gemm(ConvFwd{g3, w.a2, pb + o.w3, params + o.b3, w.a3}, B * 64, C3, 9 * C2, 1, st)) != cudaSuccess ||
      (e = gemm(ConvFwd{g4, w.a3, pb + o.w4, params + o.b4, w.a4}, B * 16, C4, 9 * C3, 1, st)) != cudaSuccess ||
      (e = gemm(FcFwd{FLAT, F5, w.a4, pb + o.w5, params + o.b5, w.a5, nullptr, nullptr, nullptr}, B, F5, FLAT, 1, st)) !=
          cudaSuccess ||
      (e = gemm(FcFwd{F5, NOUT, w.a5, pb + o.w6, params + o.b6, nullptr, y, out_scale, out_shift}, B, NOUT, F5, 1, st)) !=
          cudaSuccess)
    return cuda_fail(e, "cnn forward");
  return CELESTE_OK;
}

extern "C" int celeste_cnn_backward(const float* params, const uint16_t* params_bf16, const uint16_t* x, const float* dy,
                                    int batch, float* grad, void* ws, size_t ws_bytes, celeste_stream_t stream) {
  if (!params || !params_bf16 || !x || !dy || !grad) return fail(CELESTE_ERR_INVALID_ARG, "null argument");
  int rc = check_ws(batch, ws, ws_bytes);
  if (rc != CELESTE_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  constexpr Offsets o = offsets();
  const bf16* pb = reinterpret_cast<const bf16*>(params_bf16);
  const Ws w = ws_layout(static_cast<char*>(ws), batch);
  const int B = batch;
  const bf16* xin = reinterpret_cast<const bf16*>(x);
  cudaError_t e;
  int dev = 0, n_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return cuda_fail(e, "SM count");
  // K split of a weight gradient: about four CTAs per SM, each with at least four K-steps
  auto chunk_for = [n_sm](int tiles, int K) {
    const int want = std::max(1, (4 * n_sm + tiles - 1) / tiles);
    return std::max(4 * BK2, (K / want + BK2 - 1) / BK2 * BK2);
  };
  auto wgrad = [&](const auto& op, int M, int N, int K) {
    const int chunk = chunk_for((M + 63) / 64 * ((N + 63) / 64), K);
    return bwd_gemm(op, M, N, K, (K + chunk - 1) / chunk, chunk, st);
  };
  // The last layer's gradient in BF16 goes to the first layer's gradient buffer, which is written last.
  bf16* dy6 = w.d1;
  last_grad_kernel<<<(int)std::min<int64_t>(((int64_t)B * LDY6 + 255) / 256, 4 * n_sm), 256, 0, st>>>(dy, B, dy6);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "cnn backward output gradient");
  FcWgrad<F5, NOUT, LDY6> w6{};
  w6.dy = dy6, w6.x = w.a5, w6.dw = grad + o.w6;
  FcDgrad<F5, NOUT, LDY6> d6{};
  d6.dy = dy6, d6.w = pb + o.w6, d6.x = w.a5, d6.dx = w.d5;
  FcWgrad<FLAT, F5, F5> w5{};
  w5.dy = w.d5, w5.x = w.a4, w5.dw = grad + o.w5;
  FcDgrad<FLAT, F5, F5> d5{};
  d5.dy = w.d5, d5.w = pb + o.w5, d5.x = w.a4, d5.dx = w.d4;
  if ((e = wgrad(w6, NOUT, F5, B)) != cudaSuccess || (e = bwd_gemm(d6, B, F5, LDY6, 1, LDY6, st)) != cudaSuccess ||
      (e = wgrad(w5, F5, FLAT, B)) != cudaSuccess || (e = bwd_gemm(d5, B, FLAT, F5, 1, F5, st)) != cudaSuccess)
    return cuda_fail(e, "cnn backward dense layers");
  ConvWgrad<4, C3> w4{};
  w4.dout = w.d4, w4.in = w.a3, w4.dw = grad + o.w4;
  ConvDgrad<4, C3> d4{};
  d4.dout = w.d4, d4.w = pb + o.w4, d4.in = w.a3, d4.din = w.d3;
  ConvWgrad<8, C2> w3{};
  w3.dout = w.d3, w3.in = w.a2, w3.dw = grad + o.w3;
  ConvDgrad<8, C2> d3{};
  d3.dout = w.d3, d3.w = pb + o.w3, d3.in = w.a2, d3.din = w.d2;
  ConvWgrad<16, C1> w2{};
  w2.dout = w.d2, w2.in = w.a1, w2.dw = grad + o.w2;
  ConvDgrad<16, C1> d2{};
  d2.dout = w.d2, d2.w = pb + o.w2, d2.in = w.a1, d2.din = w.d1;
  if ((e = wgrad(w4, C4, 9 * C3, B * 16)) != cudaSuccess || (e = bwd_gemm(d4, B * 16, C3, 256, 4, 0, st)) != cudaSuccess ||
      (e = wgrad(w3, C3, 9 * C2, B * 64)) != cudaSuccess || (e = bwd_gemm(d3, B * 64, C2, 256, 4, 0, st)) != cudaSuccess ||
      (e = wgrad(w2, C2, 9 * C1, B * 256)) != cudaSuccess || (e = bwd_gemm(d2, B * 256, C1, 256, 4, 0, st)) != cudaSuccess)
    return cuda_fail(e, "cnn backward convolutions");
  if ((e = cudaFuncSetAttribute(conv1_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(W1Smem))) !=
      cudaSuccess)
    return cuda_fail(e, "cnn backward first layer");
  conv1_wgrad_kernel<<<std::min(B, 2 * n_sm), 128, sizeof(W1Smem), st>>>(xin, w.d1, B, grad + o.w1);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "cnn backward first layer");
  const BiasJobs jobs = {{{w.d1, nullptr, (int64_t)B * 1024, C1, grad + o.b1},
                          {w.d2, nullptr, (int64_t)B * 256, C2, grad + o.b2},
                          {w.d3, nullptr, (int64_t)B * 64, C3, grad + o.b3},
                          {w.d4, nullptr, (int64_t)B * 16, C4, grad + o.b4},
                          {w.d5, nullptr, (int64_t)B, F5, grad + o.b5},
                          {nullptr, dy, (int64_t)B, NOUT, grad + o.b6}}};
  bias_grad_kernel<<<dim3(std::min(n_sm, B), 6), 256, 0, st>>>(jobs);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "cnn backward biases");
  return CELESTE_OK;
}

extern "C" int celeste_cnn_mse(const float* y, const float* target, const float* weight, int batch, float* dy,
                               double* loss, celeste_stream_t stream) {
  if (!y || !target || !dy || !loss || batch <= 0) return fail(CELESTE_ERR_INVALID_ARG, "null argument or empty batch");
  const int n = batch * NOUT;
  mse_kernel<<<std::min(1024, (n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(y, target, weight, n, dy, loss);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? CELESTE_OK : cuda_fail(e, "cnn mse");
}

extern "C" int celeste_cnn_adamw(float* params, uint16_t* params_bf16, float* m, float* v, const float* grad, float lr,
                                 float beta1, float beta2, float eps, float weight_decay, int step,
                                 celeste_stream_t stream) {
  if (!params || !params_bf16 || !m || !v || !grad || step < 1) return fail(CELESTE_ERR_INVALID_ARG, "bad argument");
  const int64_t n = offsets().total;
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  adamw_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(params, reinterpret_cast<bf16*>(params_bf16), m, v, grad, n, lr,
                                                      beta1, beta2, eps, weight_decay, c1, c2);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? CELESTE_OK : cuda_fail(e, "cnn adamw");
}

extern "C" int celeste_extract_patches(celeste_problem* p, uint16_t* x, celeste_stream_t stream) {
  if (!p || !x) return fail(CELESTE_ERR_INVALID_ARG, "null argument");
  if (!p->bound) return fail(CELESTE_ERR_STATE, "bind the problem first");
  extract_patches_kernel<<<p->S, 256, 0, (cudaStream_t)stream>>>(p->dev, reinterpret_cast<bf16*>(x));
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? CELESTE_OK : cuda_fail(e, "extract patches");
}
