// Forward layers of the warm-start network on the fifth-generation tensor cores (tcgen05): the
// convolution and dense products as GEMMs D[M x N] = A[M x K] B[K x N] with BF16 operands and an
// FP32 accumulator in tensor memory.
//
// A row of A is an output pixel's im2col window (k = (kh * 3 + kw) * Cin + ci) or a dense layer's
// input, B the weights [N][K]; both K-major in shared memory, in the 128-byte-swizzled layout (8-row
// atoms of 1024 bytes, 16-byte chunk c of row r at chunk c ^ (r % 8)).
//
// Persistent CTAs of nine warps, one role each, over tiles of 128 rows of D:
//   warps 0-3  bring A in K-steps of 64 into a ring of stages.  The convolutions with 32 or 64
//              input channels copy 16-byte chunks with cp.async, eight lanes to a row so that a warp
//              reads whole 128-byte lines; taps outside the image are zero-filled.  The first layer
//              (5 channels: a window's rows are 30 bytes at a 10-byte stride) keeps whole images in shared
//              memory, 16 bytes a pixel, and builds the windows from there;
//   warp 4     one lane issues tcgen05.mma (K = 16 each, in ascending k) and tcgen05.commit, which frees
//              the stage and, after a tile's last step, hands the accumulator over;
//   warps 5-8  read the accumulator (tcgen05.ld 32x32b; two accumulators, so that the next tile's products
//              run meanwhile), add the bias, apply ReLU (or the last layer's scale and shift) and write
//              full lines through a staging area in shared memory.
// The weights stay in shared memory for all of a CTA's tiles (the 1024-wide dense layer streams them).
//
// What bounds it: a layer reads its input and writes its output once, and both are kept for the backward
// pass; per 4096 patches the four convolutions move 0.9 GB, 0.14 ms at the measured copy rate, and take
// 0.25 ms (107, 78, 47 and 19 us).  The second and third read each input from L2 2.25 times (5.7-7.5 TB/s);
// the first is short of that by the hand-overs of its one-step tiles.  Warps that share a stage paid the
// wait, the fence and the arrival of every K-step one after the other (131 us instead of 78 for the second
// layer); copies through L1 instead of L2 alone were 4 % slower.  20,000 patches, whole forward: 8.58 ms with
// element gathers between every two products, 1.38 ms now; one patch 59 us, 75 before.
//
// Every wait on an mbarrier is bounded (Args::wait_budget); a warp whose wait runs out records it in the
// error word and leaves its loop, all lanes together, the others' waits then run out as well, and the
// CTA waits (bounded) for its products in flight before it frees its tensor memory.  The first layer's
// producers, which also meet at barriers without a bound, go on meeting there until the last image.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "celeste_internal.cuh"
#include "cnn_tc.h"
#include "problem.h"

namespace celeste {
namespace cnn_tc {

using bf16 = __nv_bfloat16;

constexpr int TM = 128;        // rows of D per tile (the MMA's M)
constexpr int TK = 64;         // K per stage: one 128-byte row per operand row
constexpr int MAX_STAGES = 8;
constexpr int A_BYTES = TM * TK * 2;
constexpr int PRODUCERS = 128, EPILOGUE = 128, THREADS = PRODUCERS + 32 + EPILOGUE;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major operand in the 128-byte-swizzled layout, 8-row atoms
// 1024 bytes apart (stride byte offset), start address in 16-byte units, descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);          // start address
  d |= (uint64_t)1u << 16;                          // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024u >> 4) << 32;                // stride byte offset: next 8-row atom
  d |= (uint64_t)1u << 46;                          // descriptor version
  d |= (uint64_t)2u << 61;                          // swizzle: 128 bytes
  return d;
}

// Instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both K-major, M = 128, N.
__device__ __forceinline__ uint32_t instr_desc_bf16(int n) {
  uint32_t d = 0;
  d |= 1u << 4;                      // D format: F32
  d |= 1u << 7;                      // A format: BF16
  d |= 1u << 10;                     // B format: BF16
  d |= (uint32_t)(n >> 3) << 17;     // N / 8
  d |= (uint32_t)(TM >> 4) << 24;    // M / 16
  return d;
}

__device__ __forceinline__ void mma_bf16_tmem(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// A wait of one thread, bounded by the call's budget (negative: gives up without waiting).
__device__ __forceinline__ bool wait_thread(const Args& a, uint64_t* bar, uint32_t parity) {
  return a.wait_budget >= 0 && mbar_wait(bar, parity, a.wait_budget);
}
// The same of a whole warp: every lane gives up if one does (the lanes read the clock on their own, and what
// follows a wait needs the warp together).
__device__ __forceinline__ bool wait_warp(const Args& a, uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, wait_thread(a, bar, parity));
}

// One arrival for the whole warp (32 would be served one after the other).
__device__ __forceinline__ void mbar_arrive_warp(uint64_t* bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// 32 consecutive accumulator columns of this thread's lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,"
      "%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Byte offset of 16-byte chunk c of row r in a 128-byte-swizzled K-major tile.
__device__ __forceinline__ uint32_t sw128(int r, int c) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4));
}

// 16 bytes global -> shared, asynchronously; zeros where !ok (the source is then not read).
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void producers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(PRODUCERS) : "memory"); }

// A layer's shape.  CONV: 3x3, padding 1, stride STRIDE over [IN_W][IN_W][CIN], out [OUT_W][OUT_W][NT] (one tile
// of columns); dense: K inputs, columns in tiles of NT.  RESIDENT: the weights stay in shared memory.
template <bool CONV_, int CIN_, int IN_W_, int STRIDE_, int K_, int NT_, bool RESIDENT_, int STAGES_>
struct Layer {
  static constexpr bool CONV = CONV_, RESIDENT = RESIDENT_, FIRST = CONV_ && CIN_ < 8;
  static constexpr int CIN = CIN_, IN_W = IN_W_, STRIDE = STRIDE_, OUT_W = CONV_ ? IN_W_ / STRIDE_ : 1, K = K_, NT = NT_,
                       STAGES = STAGES_;
  static constexpr int KSTEPS = (K + TK - 1) / TK;
  static constexpr int B_BYTES = NT * TK * 2;                                  // one K-step of the weights
  static constexpr int STAGE = A_BYTES + (RESIDENT ? 0 : B_BYTES);
  static constexpr int OUT_LD = NT * 2 + 16;                                   // staging row (bytes), BF16 output
  static constexpr int STAGING = 32 * (CONV ? OUT_LD : (NT * 4 + 16));         // per epilogue warp
  static constexpr int IMG_LD = 40,                                            // first layer: the image, 16 bytes a pixel
                       IMG_BYTES = FIRST ? 34 * IMG_LD * 16 : 0;
  static constexpr int CTAS = FIRST ? 2 : 1;                                   // per SM
  static constexpr int SMEM = 1024 + (RESIDENT ? KSTEPS * B_BYTES : 0) + STAGES * STAGE + 4 * STAGING + IMG_BYTES;
};
using Conv1 = Layer<true, 5, 32, 1, 45, 32, true, 4>;
using Conv2 = Layer<true, 32, 32, 2, 288, 64, true, 8>;
using Conv3 = Layer<true, 64, 16, 2, 576, 64, true, 8>;
using Conv4 = Layer<true, 64, 8, 2, 576, 64, true, 8>;
using Dense1 = Layer<false, 0, 0, 1, 1024, 64, false, 4>;
using Dense2 = Layer<false, 0, 0, 1, 256, 32, true, 4>;

struct Bars {
  uint64_t full[MAX_STAGES], empty[MAX_STAGES], tfull[2], tempty[2], done;
};

// Ring position after `step` K-steps: stage and the parity of its use.
template <int STAGES>
struct Ring {
  uint32_t step = 0;
  __device__ __forceinline__ int stage() const { return (int)(step % STAGES); }
  __device__ __forceinline__ uint32_t parity() const { return (step / STAGES) & 1u; }
};

// ---------------------------------------------------------------------------------- producers
// Convolutions with 32 or 64 channels, and dense layers.  Each warp brings whole K-steps, every fourth one:
// what a K-step costs besides its copies (the wait for the stage, the fence, the arrival) is then paid by
// four warps at once and once for 32 copies of a lane.  The rows' offsets in the input are compile-time
// multiples of the strides; the stride-2 convolutions leave the image only above (output row 0, kh = 0)
// and on the left (column 0, kw = 0).
template <class L>
__device__ __forceinline__ bool produce(const Args& a, unsigned char* stages, Bars& bar, int n_mine, int n_cols) {
  static_assert(L::STAGES % 4 == 0, "a warp returns to its stages in order");
  constexpr int OWN = L::STAGES / 4;   // stages per warp: K-steps of a warp in flight
  constexpr int CPT = L::CONV ? L::CIN / 8 : 8;   // chunks per tap
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane & 7, r0 = lane >> 3;   // rows r0 + 4 i
  Ring<L::STAGES> issue, land;
  issue.step = land.step = warp;
  auto landed = [&]() {   // this warp's oldest K-step in flight has arrived
    fence_proxy_async_smem();   // before the tensor cores read it
    mbar_arrive_warp(&bar.full[land.stage()]);
    land.step += 4;
  };
  const uint32_t steps = (uint32_t)n_mine * L::KSTEPS;
  for (; issue.step < steps; issue.step += 4) {
    const int q = issue.step / L::KSTEPS, ks = issue.step % L::KSTEPS;
    const int t = (int)blockIdx.x + q * (int)gridDim.x;
    const int m0 = (t / n_cols) * TM, n0 = (t % n_cols) * L::NT;
    const int left = a.M - m0;   // rows of the tile that exist
    const int s = issue.stage();
    if (!wait_warp(a, &bar.empty[s], issue.parity() ^ 1u)) return false;
    const uint32_t As = smem_u32(stages + s * L::STAGE);
    if constexpr (L::CONV) {
      constexpr int OW = L::OUT_W, RPI = OW * OW, ROW = L::IN_W * L::CIN;   // output pixels per image, input row
      const int tap = ks * (8 / CPT) + c / CPT, kh = tap / 3, kw = tap % 3;
      // output pixel (oh, ow) of image b reads input (2 oh + kh - 1, 2 ow + kw - 1)
      const int m = m0 % RPI, b = m0 / RPI, oh0 = m / OW;   // (a tile starts at column 0, or on an image)
      const bf16* src = a.in + (int64_t)b * (L::IN_W * ROW) + (int64_t)(2 * oh0 + kh - 1) * ROW + (2 * r0 + kw - 1) * L::CIN +
                        (c % CPT) * 8;
      const bool real = tap < 9;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        // row r = r0 + 4 i of the tile; 4 i and r0 add without carry into the output row (OW >= 4)
        const int ow = (4 * i) % OW, oh = (4 * i) / OW % OW, im = (4 * i) / RPI;
        const bool top = kh == 0 && oh0 + oh == 0, out_left = kw == 0 && ow + r0 == 0;
        const bool ok = real && !top && !out_left && r0 + 4 * i < left;
        const int64_t off = (int64_t)im * (L::IN_W * ROW) + 2 * oh * ROW + 2 * ow * L::CIN;
        cp_async_zfill(As + sw128(r0 + 4 * i, c), ok ? src + off : a.in, ok);
      }
    } else {
      const bf16* src = a.in + (int64_t)(m0 + r0) * L::K + ks * TK + c * 8;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const bool ok = r0 + 4 * i < left;
        cp_async_zfill(As + sw128(r0 + 4 * i, c), ok ? src + 4 * i * L::K : a.in, ok);
      }
      if constexpr (!L::RESIDENT) {
        const bf16* w = a.w + (int64_t)(n0 + r0) * L::K + ks * TK + c * 8;
#pragma unroll
        for (int i = 0; i < L::NT / 4; ++i) {
          const bool ok = n0 + r0 + 4 * i < a.N;
          cp_async_zfill(As + A_BYTES + sw128(r0 + 4 * i, c), ok ? w + 4 * i * L::K : a.w, ok);
        }
      }
    }
    cp_async_commit();
    if (issue.step - land.step == 4 * (OWN - 1)) {
      cp_async_wait_group<OWN - 1>();
      landed();
    }
  }
  cp_async_wait_group<0>();
  while (land.step < issue.step) landed();
  return true;
}

// First layer: image by image.  The image lies in shared memory with its five channels in 16 bytes per
// pixel and a border of zeros.  Each warp builds whole tiles (four output rows, a lane one column of
// them, its window's input rows moving through registers), every fourth one; the next image's pixels are
// loaded into registers (8 per thread) while the current one's tiles are built.  The four warps meet at two
// barriers per image: one whose wait has run out builds nothing more, but keeps meeting the others.
template <class L>
__device__ __forceinline__ bool produce_first(const Args& a, unsigned char* stages, unsigned char* img, Bars& bar, int images) {
  static_assert(L::STAGES == 4, "a warp's tiles go through one stage");
  const int tid = threadIdx.x, ow = tid & 31, warp = tid >> 5;
  for (int i = tid; i < L::IMG_BYTES / 16; i += PRODUCERS) reinterpret_cast<uint4*>(img)[i] = make_uint4(0u, 0u, 0u, 0u);
  const bool aligned = (reinterpret_cast<uintptr_t>(a.in) & 15) == 0;   // (a caller's slice may start anywhere)
  uint32_t px[20];   // 8 pixels x 5 channels, as in memory
  auto fetch = [&](int b) {
    if (b >= images) return;
    const bf16* src = a.in + (int64_t)b * (32 * 32 * 5) + tid * 40;
    if (aligned) {
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4*>(src) + q);
        px[4 * q] = v.x;
        px[4 * q + 1] = v.y;
        px[4 * q + 2] = v.z;
        px[4 * q + 3] = v.w;
      }
    } else {
      const uint16_t* p = reinterpret_cast<const uint16_t*>(src);
#pragma unroll
      for (int q = 0; q < 20; ++q) px[q] = (uint32_t)p[2 * q] | ((uint32_t)p[2 * q + 1] << 16);
    }
  };
  // a padded row's pixel x (0: the left border) lies after x / 8 gaps, so that the threads' writes of every
  // eighth pixel spread over the banks
  auto at = [](int x) { return x + (x >> 3); };
  // input row y (from -1) around column ow: 15 values, the last word's upper half zero
  auto load_row = [&](int y, uint32_t (&r)[8]) {
    const uint4* p = reinterpret_cast<const uint4*>(img) + (y + 1) * L::IMG_LD;
    const uint4 p0 = p[at(ow)], p1 = p[at(ow + 1)], p2 = p[at(ow + 2)];
    r[0] = p0.x;
    r[1] = p0.y;
    r[2] = p0.z | (p1.x << 16);
    r[3] = __funnelshift_r(p1.x, p1.y, 16);
    r[4] = __funnelshift_r(p1.y, p1.z, 16);
    r[5] = p2.x;
    r[6] = p2.y;
    r[7] = p2.z;
  };
  Ring<L::STAGES> ring;
  ring.step = warp;
  unsigned char* As = stages + warp * L::STAGE;
  bool ok = true;   // the same in every lane of a warp
  fetch(blockIdx.x);
  for (int b = blockIdx.x; b < images; b += gridDim.x) {
    producers_sync();   // the previous image has been read (the border zeroed)
    // pixels 8 tid .. 8 tid + 7: an even pixel starts on a word, an odd one half-way into it
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int p = 8 * tid + i, w = (5 * i) / 2;
      uint4 v;
      if (i % 2 == 0)
        v = make_uint4(px[w], px[w + 1], px[w + 2] & 0xffffu, 0u);
      else
        v = make_uint4(__funnelshift_r(px[w], px[w + 1], 16), __funnelshift_r(px[w + 1], px[w + 2], 16), px[w + 2] >> 16, 0u);
      reinterpret_cast<uint4*>(img)[((p >> 5) + 1) * L::IMG_LD + at((p & 31) + 1)] = v;
    }
    producers_sync();
    fetch(b + gridDim.x);
#pragma unroll 1
    for (int q = warp; q < 8 && ok; q += 4) {
      uint32_t r0[8], r1[8], r2[8];
      load_row(4 * q - 1, r0);
      load_row(4 * q, r1);
      ok = wait_warp(a, &bar.empty[warp], ring.parity() ^ 1u);
      if (!ok) break;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        load_row(4 * q + j + 1, r2);
        // row 32 j + ow of the tile: the three runs of 15 values one after the other, then zeros up to 48
        auto put = [&](int c, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
          *reinterpret_cast<uint4*>(As + sw128(32 * j + ow, c)) = make_uint4(x, y, z, w);
        };
        put(0, r0[0], r0[1], r0[2], r0[3]);
        put(1, r0[4], r0[5], r0[6], r0[7] | (r1[0] << 16));
        put(2, __funnelshift_r(r1[0], r1[1], 16), __funnelshift_r(r1[1], r1[2], 16), __funnelshift_r(r1[2], r1[3], 16),
            __funnelshift_r(r1[3], r1[4], 16));
        put(3, __funnelshift_r(r1[4], r1[5], 16), __funnelshift_r(r1[5], r1[6], 16), __funnelshift_r(r1[6], r1[7], 16), r2[0]);
        put(4, r2[1], r2[2], r2[3], r2[4]);
        put(5, r2[5], r2[6], r2[7], 0u);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          r0[i] = r1[i];
          r1[i] = r2[i];
        }
      }
      fence_proxy_async_smem();
      mbar_arrive_warp(&bar.full[warp]);
      ring.step += 4;
    }
  }
  return ok;
}

// ---------------------------------------------------------------------------------- products
template <class L>
__device__ __forceinline__ bool multiply(const Args& a, unsigned char* weights, unsigned char* stages, Bars& bar, uint32_t tmem,
                                         int n_mine) {
  const uint32_t idesc = instr_desc_bf16(L::NT);
  Ring<L::STAGES> ring;
  for (int q = 0; q < n_mine; ++q) {
    const int acc = q & 1;
    if (!wait_thread(a, &bar.tempty[acc], ((q >> 1) & 1u) ^ 1u)) return false;
    fence_after_sync();
    const uint32_t d = tmem + (uint32_t)(acc * L::NT);
    for (int ks = 0; ks < L::KSTEPS; ++ks) {
      const int s = ring.stage();
      if (!wait_thread(a, &bar.full[s], ring.parity())) return false;
      fence_after_sync();
      const uint32_t ab = smem_u32(stages + s * L::STAGE);
      const uint32_t bb = L::RESIDENT ? smem_u32(weights + ks * L::B_BYTES) : ab + A_BYTES;
      // (blocks past K hold only zeros and are left out)
#pragma unroll
      for (int j = 0; j < TK / 16; ++j)   // K = 16 per product: 32 bytes along the swizzled row
        if (ks * TK + 16 * j < L::K)
          mma_bf16_tmem(d, smem_desc_sw128(ab + 32 * j), smem_desc_sw128(bb + 32 * j), idesc, (ks > 0 || j > 0) ? 1u : 0u);
      mma_commit(&bar.empty[s]);
      ++ring.step;
    }
    mma_commit(&bar.tfull[acc]);
  }
  return true;
}

// ---------------------------------------------------------------------------------- epilogue
template <class L>
__device__ __forceinline__ bool finish(const Args& a, unsigned char* staging, const float* bias, Bars& bar, uint32_t tmem,
                                       int n_tiles, int n_cols) {
  const int lane = threadIdx.x & 31, quad = (threadIdx.x >> 5) & 3;   // the warp's 32 accumulator lanes
  unsigned char* st = staging + quad * L::STAGING;
  for (int q = 0;; ++q) {
    // the CTA's q-th tile, in the producers' order
    const int t = L::FIRST ? 8 * ((int)blockIdx.x + (q >> 3) * (int)gridDim.x) + (q & 7)
                           : (int)blockIdx.x + q * (int)gridDim.x;
    if (t >= n_tiles) break;
    const int acc = q & 1;
    const int row0 = (t / n_cols) * TM + 32 * quad, n0 = (t % n_cols) * L::NT;
    if (!wait_warp(a, &bar.tfull[acc], (q >> 1) & 1u)) return false;
    fence_after_sync();
    float v[L::NT];
    const uint32_t src = tmem + (uint32_t)(acc * L::NT) + ((uint32_t)(32 * quad) << 16);
#pragma unroll
    for (int c = 0; c < L::NT; c += 32) tmem_ld32(src + (uint32_t)c, v + c);
    fence_before_sync();
    mbar_arrive_warp(&bar.tempty[acc]);
    const int rows = min(32, a.M - row0);   // (may be <= 0)
    if (L::CONV || a.out) {
      // BF16 after ReLU: a row of NT values per lane into the staging area, then full lines out
#pragma unroll
      for (int ch = 0; ch < L::NT / 8; ++ch) {
        __align__(16) __nv_bfloat162 o[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int n = 8 * ch + 4 * i;
          const float4 b = *reinterpret_cast<const float4*>(bias + n0 + n);
          o[2 * i] = __floats2bfloat162_rn(fmaxf(v[n] + b.x, 0.f), fmaxf(v[n + 1] + b.y, 0.f));
          o[2 * i + 1] = __floats2bfloat162_rn(fmaxf(v[n + 2] + b.z, 0.f), fmaxf(v[n + 3] + b.w, 0.f));
        }
        *reinterpret_cast<uint4*>(st + lane * L::OUT_LD + 16 * ch) = *reinterpret_cast<const uint4*>(o);
      }
      __syncwarp();
      constexpr int CH = L::NT / 8, RPI = 32 / CH;   // chunks per row, rows per warp store
#pragma unroll
      for (int r = 0; r < 32; r += RPI) {
        const int row = r + lane / CH, ch = lane % CH;
        if (row < rows)
          *reinterpret_cast<uint4*>(a.out + (int64_t)(row0 + row) * a.N + n0 + 8 * ch) =
              *reinterpret_cast<const uint4*>(st + row * L::OUT_LD + 16 * ch);
      }
      __syncwarp();
    } else if constexpr (!L::CONV) {
      // FP32, the tile's rows of a.N values contiguous in memory
      float* sf = reinterpret_cast<float*>(st);
#pragma unroll
      for (int n = 0; n < L::NT; ++n) {
        if (n < a.N) {
          float y = v[n] + bias[n];
          if (a.scale) y = y * a.scale[n] + a.shift[n];
          sf[lane * a.N + n] = y;
        }
      }
      __syncwarp();
      for (int i = lane; i < rows * a.N; i += 32) a.out_f[(int64_t)row0 * a.N + i] = sf[i];
      __syncwarp();
    }
  }
  return true;
}

template <class L>
__global__ void __launch_bounds__(THREADS, L::CTAS) tc_layer_kernel(Args a, int n_tiles, int n_cols) {
  extern __shared__ unsigned char dyn[];
  __shared__ __align__(8) Bars bar;
  __shared__ uint32_t tmem_base;
  __shared__ __align__(16) float bias[256];
  constexpr uint32_t COLS = 2 * L::NT;
  // 1024-byte aligned buffers (the swizzle atom)
  unsigned char* base = dyn + ((1024u - (smem_u32(dyn) & 1023u)) & 1023u);
  unsigned char* weights = base;
  unsigned char* stages = base + (L::RESIDENT ? L::KSTEPS * L::B_BYTES : 0);
  unsigned char* staging = stages + L::STAGES * L::STAGE;
  unsigned char* img = staging + 4 * L::STAGING;
  const int tid = threadIdx.x, warp = tid >> 5;

  if (tid == 0) {
    for (int s = 0; s < L::STAGES; ++s) {
      mbar_init(&bar.full[s], 1);   // (a stage is one producer warp's)
      mbar_init(&bar.empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar.tfull[i], 1);
      mbar_init(&bar.tempty[i], EPILOGUE / 32);
    }
    mbar_init(&bar.done, 1);
  }
  if (warp == 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)), "r"(COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int n = tid; n < min(a.N, 256); n += THREADS) bias[n] = a.bias[n];
  if constexpr (L::RESIDENT) {
    for (int e = tid; e < L::KSTEPS * L::NT * 8; e += THREADS) {
      const int c = e & 7, n = (e >> 3) % L::NT, ks = e / (8 * L::NT), k = ks * TK + 8 * c;
      unsigned char* dst = weights + ks * L::B_BYTES + sw128(n, c);
      if constexpr (L::K % 8 == 0) {
        const bool in = n < a.N && k < L::K;
        cp_async_zfill(smem_u32(dst), in ? a.w + (int64_t)n * L::K + k : a.w, in);
      } else {
        __align__(16) bf16 x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = n < a.N && k + j < L::K ? a.w[(int64_t)n * L::K + k + j] : __float2bfloat16(0.f);
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(x);
      }
    }
    cp_async_wait_all();
    fence_proxy_async_smem();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = tmem_base;

  // tiles of this CTA
  const int n_mine = L::FIRST ? ((a.B - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x) * 8
                              : (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  bool ok = true;
  if (warp < 4) {
    if constexpr (L::FIRST)
      ok = produce_first<L>(a, stages, img, bar, a.B);
    else
      ok = produce<L>(a, stages, bar, n_mine, n_cols);
    cp_async_wait_all();
  } else if (warp == 4) {
    if ((tid & 31) == 0) {
      ok = multiply<L>(a, weights, stages, bar, tmem, n_mine);
      mma_commit(&bar.done);   // every product issued so far
      ok = mbar_wait(&bar.done, 0u, WAIT_BUDGET_DEFAULT) && ok;
    }
    __syncwarp();
  } else {
    ok = finish<L>(a, staging, bias, bar, tmem, n_tiles, n_cols);
  }
  if (!ok) atomicExch(a.err, 1);
  fence_before_sync();
  __syncthreads();
  if (warp == 4) {
    fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
  }
}

template <class L>
static cudaError_t launch(const Args& a, int n_sm, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(tc_layer_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
  if (e != cudaSuccess) return e;
  const int n_cols = (a.N + L::NT - 1) / L::NT, n_tiles = (a.M + TM - 1) / TM * n_cols;
  tc_layer_kernel<L><<<std::min(L::FIRST ? a.B : n_tiles, L::CTAS * n_sm), THREADS, L::SMEM, st>>>(a, n_tiles, n_cols);
  return cudaGetLastError();
}

}  // namespace cnn_tc

cudaError_t tc_forward(cnn_tc::LayerId id, const cnn_tc::Args& a, int n_sm, cudaStream_t st) {
  using namespace cnn_tc;
  if (a.M <= 0) return cudaSuccess;
  switch (id) {
    case CONV1: return launch<Conv1>(a, n_sm, st);
    case CONV2: return launch<Conv2>(a, n_sm, st);
    case CONV3: return launch<Conv3>(a, n_sm, st);
    case CONV4: return launch<Conv4>(a, n_sm, st);
    case DENSE1: return launch<Dense1>(a, n_sm, st);
    default: return launch<Dense2>(a, n_sm, st);
  }
}

}  // namespace celeste
