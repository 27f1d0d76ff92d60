// unet_conv.cuh -- the U-Net's 3x3 convolution (forward and data gradient) on the
// fifth-generation tensor cores, operands copied by TMA, accumulators in tensor memory.
//
// Implicit GEMM, D[m][n] = sum_k A[m][k] B[n][k] with m a pixel, n an output channel and
// k = (tap, input channel). A CTA owns a tile of TH x TW pixels of one image and BN output
// channels. Its input, the tile and a ring of one pixel with all input channels, is copied
// once into shared memory (one TMA box per chunk of 64 or 32 channels: a pixel's chunk is a
// 128- or 64-byte row of the swizzled K-major operand layout). Every tap then reads that
// one copy: the operand of tap (dy, dx) starts dy pitch + dx rows further on (pitch = TW +
// 2 pixels), so a tap costs no copy and shared memory holds each input pixel once instead
// of nine times. 8-row groups of the 128-row operand are eight neighbouring pixels of an
// image row; they lie `sbo` pixels apart:
//   patch   sbo = pitch: 16 image rows x 8 columns, every row of the operand a pixel
//   linear  sbo = 8:     128 consecutive positions of the pitched tile; the two ring
//                        columns of each row are computed and dropped (images with too
//                        few rows, or columns that are no multiple of eight)
// The swizzle is a function of the shared-memory address, so a start anywhere in a
// 1024-byte pattern reads what the copy wrote (matrix base offset 0: the patterns
// themselves are aligned). Rows beyond the first and last image row arrive as the copy's
// zero fill; the periodic columns beyond the first and last image column also arrive as
// zeros and are overwritten with their images by the epilogue warps.
//
// Upsampled input (up = 1, nearest 2x): output pixel (2 y + py, 2 x + px) reads input row
// floor((2 y + py + dy)/2), so each of the four parities (py, px) is a 3x3-tap sum over
// shifts -1, 0, 1 of the low-resolution tile: four accumulators over the same operands,
// nothing upsampled in memory.
//
// The weights stream through a ring of stages, one (tap, chunk) each, in k order; per stage
// one thread issues the K = 16 MMAs of every accumulator. So each accumulator adds the
// same K = 16 products in the same order as conv3x3_kernel's, tap by tap, channels
// ascending, and gives the same bits.
//
// Warps: 0 copies, 1 issues MMAs (and owns the tensor memory), 2..9 patch the periodic
// columns, then drain the accumulators: bias, ReLU, BF16, through shared memory so that
// the mask's loads and the output's stores are whole lines.
//
// What bounds it: the warp that issues the MMAs, whose waits, commits and addresses between two
// stages are not hidden behind the stage's MMAs (40 to 64 cycles each up to N = 128), then the
// copy before and the drain after a tile's MMAs, which only the other CTA of the
// multiprocessor hides, where two fit. Measured on GB300 against the mma.sync kernel
// (conv3x3_kernel), 32 images: 128 -> 128 channels at 16 x 64, 18.4 us (55 us); 256 -> 256 at
// 8 x 32, 24.6 us (75 us). Wide images take conv3x3_rows_kernel below.
//
// Every mbarrier wait is bounded (about a second of %globaltimer); on expiry the kernel
// sets its error word, waits (bounded) for the copies and MMAs in flight, releases its
// tensor memory and writes no further output.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "lb_tma.cuh"
#include "unet_kernels.cuh"

namespace lbu {
namespace tc {

// Shared-memory matrix descriptor of a swizzled operand: start address, leading byte
// offset (unused by the K-major swizzled layouts), stride byte offset between 8-row groups
// (all in 16-byte units), version 1 (bits 46-47), layout type at bits 61-63 (2: 128-byte
// swizzle, 4: 64-byte swizzle).
__host__ __device__ constexpr unsigned long long desc_base(int rowb, unsigned lbo, unsigned sbo) {
  return ((unsigned long long)((lbo >> 4) & 0x3FFFu) << 16) | ((unsigned long long)((sbo >> 4) & 0x3FFFu) << 32) |
         (1ull << 46) | ((rowb == 128 ? 2ull : 4ull) << 61);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A and B (bits
// 7-9 and 10-12 = 1), A and B K-major (bits 15, 16 = 0) or MN-major (= 1), N >> 3 at bits
// 17-22, M >> 4 at 24-28.
__host__ __device__ constexpr unsigned idesc_bf16(int M, int N, bool mn_major = false) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major ? (3u << 15) : 0u) | ((unsigned)(N >> 3) << 17) |
         ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(unsigned* s_addr, unsigned ncols) {  // one whole warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_addr)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned taddr, unsigned ncols) {  // one whole warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D (tensor memory) += A B^T, run by a whole warp and issued by the lane that
// elect.sync picks (always the same one). With the whole warp in the issue loop its
// addresses are warp-uniform values, and the elected predicate needs no per-lane branch.
// Cycles per MMA of M = 128, K = 16, measured: 40, 48, 56, 64, 96 and 127 for N = 32, 64, 96,
// 128, 192 and 256, that is the operands' bytes at 128 a cycle up to N = 128, then the tensor
// cores' rate; a predicate from the lane number gave 50 to 72 up to N = 128, and a branch that
// one lane takes around descriptors built with run-time multiplications 80 to 250.
__device__ __forceinline__ void mma_bf16(unsigned tmem_d, unsigned long long a, unsigned long long b, unsigned idesc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b32 x;\n\tsetp.ne.b32 p, 1, 0;\n\telect.sync x|q, 0xffffffff;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc)
      : "memory");
}
// The same, D = A B^T where acc is 0: a value, as a second copy of a loop costs more than it.
__device__ __forceinline__ void mma_bf16_if(unsigned tmem_d, unsigned long long a, unsigned long long b, unsigned idesc,
                                            int acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b32 x;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync x|q, 0xffffffff;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// The mbarrier receives one arrival when every MMA issued before has completed (whole warp).
__device__ __forceinline__ void mma_commit(unsigned long long* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t.reg .b32 x;\n\telect.sync x|q, 0xffffffff;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar))
      : "memory");
}
// Descriptor from its constant upper half and the lower half at a shared-memory address.
__device__ __forceinline__ unsigned long long desc64(unsigned hi, unsigned lo) {
  return ((unsigned long long)hi << 32) | lo;
}
// The K = 16 MMAs kk = 0 .. KK - 1 of one stage for G accumulators (d + g dstep), whose A
// operands start at the descriptors lo[g]: unrolled, accumulators innermost, so that an MMA
// costs a few instructions of the issuing warp and seldom follows one into its accumulator.
template <int G, int KK>
__device__ __forceinline__ void mma_group(unsigned d, unsigned dstep, const unsigned lo[G], unsigned hiA, unsigned loB,
                                          unsigned hiB, unsigned idesc, int acc) {
#pragma unroll
  for (int kk = 0; kk < KK; ++kk)
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (kk > 0) mma_bf16(d + g * dstep, desc64(hiA, lo[g] + 2 * kk), desc64(hiB, loB + 2 * kk), idesc);
      else mma_bf16_if(d + g * dstep, desc64(hiA, lo[g]), desc64(hiB, loB), idesc, acc);
    }
}
// 16 or 32 consecutive 32-bit columns of this thread's lane (shape 32x32b: lane = warp's base
// + lane id); tmem_wait before the values are used.
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float v[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld32(unsigned taddr, float v[32]) {
  tmem_ld16(taddr, v);
  tmem_ld16(taddr + 16u, v + 16);
  tmem_wait();
}

// Zeros to 16 columns of this thread's lane; tmem_wait_st before they are relied on.
__device__ __forceinline__ void tmem_zero16(unsigned taddr) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
      "%1};" ::"r"(taddr),
      "r"(0u)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Offset of 16-byte piece v of row r in a swizzled operand of ROWB-byte rows whose patterns
// (8 rows of 128 bytes, or of 64) are aligned.
template <int ROWB>
__device__ __forceinline__ unsigned swizzled(int r, int v) {
  const unsigned off = (unsigned)r * ROWB + (unsigned)v * 16u;
  return off ^ (((off >> 7) & (ROWB == 128 ? 7u : 3u)) << 4);
}

}  // namespace tc

// Named barrier of n threads that also says whether `ok` held for all of them.
__device__ __forceinline__ bool bar_all(int id, int n, bool ok) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %3, 0;\n\tbarrier.cta.red.and.pred q, %1, %2, p;\n\t"
      "selp.b32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(id), "r"(n), "r"((int)ok)
      : "memory");
  return r != 0;
}

// A bounded wait of a whole warp: the phase's end, or for every lane the limit. Each lane decides for
// itself whether its wait ran out, so near the limit lanes may differ; what they do on it (leave a
// loop with __syncwarp or barriers in it) has to be the same for all of them. Waits whose outcome
// goes straight into a group's bar_all need no vote before it (in the drains a vote more per row
// cost a batch-8 forward pass 205.1 -> 205.7 us).
__device__ __forceinline__ bool warp_wait(unsigned long long* bar, unsigned parity) {
  return __all_sync(~0u, lbnci::mbar_wait(bar, parity));
}

constexpr int kConvThreads = 320;  // copy warp, MMA warp, eight epilogue warps
constexpr int kConvEpiThreads = 256;

struct ConvTma {
  const bf16* x;      // input, for the periodic columns
  int xs, H, W;       // input pixel stride and image: the grid of positions
  int up;             // 1: the output is 2H x 2W
  int tiles_x, tiles_y, TH, TW, pitch;
  int nm, mstart, sbo;  // M tiles (per parity), positions between their starts, between 8-row groups
  int linear;         // position p of M tile m: (p / pitch, p % pitch), else (l / 8, 8 m + l % 8)
  int nchunk;         // chunks of ROWB/2 input channels
  int a_stride;       // bytes of a chunk's tile in shared memory
  int nstage;         // ring stages of the weights
  int cols;           // tensor-memory columns (a power of two)
  int tail;           // offset of the ConvTail behind the tile, the ring and the output staging
  const float* bias;
  int relu;
  bf16* y;
  int ys;
  const bf16* mask;
  int ms;
};

constexpr int kConvMaxStage = 24;
struct ConvTail {
  unsigned long long bar_a, bar_p, bar_d, bar_full[kConvMaxStage], bar_empty[kConvMaxStage];
  unsigned tmem;
  int fail;
  alignas(16) float bias[128];
};

template <int BN, int ROWB>
__global__ void __launch_bounds__(kConvThreads, 2)
conv3x3_tma_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, ConvTma a,
                   int* err) {
  constexpr int CH = ROWB / 2, KK = CH / 16;  // channels and K = 16 MMAs of a chunk
  constexpr int BBYTES = BN * ROWB;
  constexpr unsigned IDESC = tc::idesc_bf16(128, BN);
  extern __shared__ __align__(1024) unsigned char sm[];  // no static shared memory: it starts the window
  ConvTail& t = *reinterpret_cast<ConvTail*>(sm + a.tail);
  unsigned char* const sA = sm;
  unsigned char* const sB = sm + a.nchunk * a.a_stride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = blockIdx.x % a.tiles_x, ty = (blockIdx.x / a.tiles_x) % a.tiles_y;
  const int b = blockIdx.x / (a.tiles_x * a.tiles_y);
  const int x0 = tx * a.TW, y0 = ty * a.TH, n0 = blockIdx.y * BN;
  const int ni = 9 * a.nchunk, ST = a.nstage;

  if (tid == 0) {
    lbnci::mbar_init(&t.bar_a, 1);
    lbnci::mbar_init(&t.bar_p, kConvEpiThreads / 32);
    lbnci::mbar_init(&t.bar_d, 2);
    for (int s = 0; s < ST; ++s) {
      lbnci::mbar_init(&t.bar_full[s], 1);
      lbnci::mbar_init(&t.bar_empty[s], 1);
    }
    t.fail = (smem_u32(sm) & 1023u) ? 2 : 0;  // the patterns need the alignment: report, do nothing
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tc::tmem_alloc(&t.tmem, (unsigned)a.cols);
  if (tid < BN) t.bias[tid] = a.bias ? a.bias[n0 + tid] : 0.f;
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const unsigned tmem = t.tmem;
  const bool aligned = t.fail == 0;
  auto weights = [&](int i) {
    const int s = i % ST;
    lbnci::mbar_expect_tx(&t.bar_full[s], BBYTES);
    lbnci::tma_load_2d(sB + s * BBYTES, &map_w, i * CH, n0, &t.bar_full[s]);
  };
  if (aligned && tid == 0)  // the first weights, which no kernel of the chain writes, ahead of the wait
    for (int i = 0; i < ST; ++i) weights(i);
  lbnci::pdl_enter();

  if (!aligned) {
    // nothing was started
  } else if (warp == 0) {
    if (lane == 0) {  // copies: the input tile, then the weights through the ring
      lbnci::mbar_expect_tx(&t.bar_a, (unsigned)(a.nchunk * ROWB * (a.TW + 2) * (a.TH + 2)));
      for (int k = 0; k < a.nchunk; ++k)
        lbnci::tma_load_4d(sA + k * a.a_stride, &map_x, k * CH, x0 - 1, y0 - 1, b, &t.bar_a);
      int issued = ST;
      for (int i = ST; i < ni; ++i) {
        const int s = i % ST, u = i / ST;
        if (!lbnci::mbar_wait(&t.bar_empty[s], (unsigned)((u - 1) & 1))) {
          atomicOr(&t.fail, 1);
          break;
        }
        weights(i);
        issued = i + 1;
      }
      // before the CTA may end: every copy has landed (bounded; each was waited for by the
      // MMA warp unless a wait ran out)
      lbnci::mbar_wait(&t.bar_a, 0u);
      for (int i = issued > ST ? issued - ST : 0; i < issued; ++i)
        lbnci::mbar_wait(&t.bar_full[i % ST], (unsigned)((i / ST) & 1));
    }
  } else if (warp == 1) {  // MMAs: the whole warp runs the loop
    bool bad = __any_sync(~0u, !lbnci::mbar_wait(&t.bar_a, 0u) || !lbnci::mbar_wait(&t.bar_p, 0u));
    const unsigned long long dA = tc::desc_base(ROWB, 16u, (unsigned)(a.sbo * ROWB));
    const unsigned long long dB = tc::desc_base(ROWB, 16u, 8u * ROWB);
    const unsigned hiA = (unsigned)(dA >> 32), hiB = (unsigned)(dB >> 32);
    // lower halves in 16-byte units: addresses below 256 KB never carry out of their field
    const unsigned loA0 = (unsigned)dA + (smem_u32(sA) >> 4), loB0 = (unsigned)dB + (smem_u32(sB) >> 4);
    const unsigned mstep = (unsigned)(a.mstart * ROWB) >> 4;
    // A stage's addresses advance by additions and stand before its wait: what the issuing warp
    // does between two stages is time the tensor cores wait for (16 x 64, 256 -> 128 channels,
    // 32 images: 28.6 -> 26.7 us; 8 x 32, 256 -> 256: 26.4 -> 24.6). The loops stay rolled and the
    // first MMAs' "do not accumulate" is a value: in a network each kernel runs once between
    // others, its instructions not cached (batch-8 forward 219 -> 210 us, with the taps of a row
    // unrolled 230).
    const unsigned step = (unsigned)(a.a_stride >> 4), row = (unsigned)(a.pitch * ROWB) >> 4;
    unsigned ph = 0u, lb = loB0;
    int s = 0;
    auto issue = [&](const unsigned at[4], int acc) {  // (a converged warp: __any_sync before it)
      unsigned lo[4];
      if (a.up) {
        for (int m = 0; m < a.nm; ++m) {
#pragma unroll
          for (int q = 0; q < 4; ++q) lo[q] = at[q] + m * mstep;
          tc::mma_group<4, KK>(tmem + m * BN, (unsigned)(a.nm * BN), lo, hiA, lb, hiB, IDESC, acc);
        }
      } else {
#pragma unroll
        for (int g = 0; g < 4; ++g) lo[g] = at[0] + g * mstep;
        int m = 0;
        for (; m + 4 <= a.nm; m += 4) {
          tc::mma_group<4, KK>(tmem + m * BN, BN, lo, hiA, lb, hiB, IDESC, acc);
#pragma unroll
          for (int g = 0; g < 4; ++g) lo[g] += 4 * mstep;
        }
        if (a.nm - m == 3) tc::mma_group<3, KK>(tmem + m * BN, BN, lo, hiA, lb, hiB, IDESC, acc);
        else if (a.nm - m == 2) tc::mma_group<2, KK>(tmem + m * BN, BN, lo, hiA, lb, hiB, IDESC, acc);
        else if (a.nm - m == 1) tc::mma_group<1, KK>(tmem + m * BN, BN, lo, hiA, lb, hiB, IDESC, acc);
      }
    };
#pragma unroll 1
    for (int dy = 0; dy < 3 && !bad; ++dy)
#pragma unroll 1
      for (int dx = 0; dx < 3; ++dx) {
        unsigned at[4];  // up: the parities, at low-resolution row and column floor((parity + tap)/2)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          at[q] = loA0 + (a.up ? (unsigned)((((q >> 1) + dy - 1) >> 1) + 1) * row +
                                     (unsigned)((((((q & 1) + dx - 1) >> 1) + 1) * ROWB) >> 4)
                               : (unsigned)dy * row + (unsigned)((dx * ROWB) >> 4));
        for (int k = 0; k < a.nchunk; ++k) {
          if (!bad) bad = __any_sync(~0u, !lbnci::mbar_wait(&t.bar_full[s], ph));
          if (bad) break;
          tc::fence_after_sync();
          issue(at, dx + dy + k);
          tc::mma_commit(&t.bar_empty[s]);
#pragma unroll
          for (int q = 0; q < 4; ++q) at[q] += step;
          lb += BBYTES >> 4;
          if (++s == ST) {
            s = 0;
            lb = loB0;
            ph ^= 1u;
          }
        }
      }
    if (lane == 0) {
      if (bad) atomicOr(&t.fail, 1);
    }
    tc::mma_commit(&t.bar_d);
    if (lane == 0) lbnci::mbar_arrive(&t.bar_d);
  } else {
    const int et = tid - 64;
    {  // the periodic images of the columns beyond the image: pieces of 16 bytes
      const int vpp = a.nchunk * (ROWB / 16);
      const int left = x0 == 0 ? 1 : 0, right = x0 + a.TW >= a.W ? 1 : 0;
      const int ncol = left + right, count = ncol * (a.TH + 2) * vpp;
      bool ok = true;
      constexpr int U = 4;
      for (int e0 = 0; e0 < count && ok; e0 += U * kConvEpiThreads) {
        uint4 v[U];
        int dst[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const int e = e0 + j * kConvEpiThreads + et;
          dst[j] = -1;
          if (e < count) {
            const int px = e / vpp, p = e - px * vpp;
            const int row = px / ncol, col = px - row * ncol;
            const int yy = y0 - 1 + row;
            if (yy >= 0 && yy < a.H) {
              const bool lft = left && col == 0;
              v[j] = *reinterpret_cast<const uint4*>(a.x + ((size_t)(b * a.H + yy) * a.W + (lft ? a.W - 1 : 0)) * a.xs +
                                                     p * 8);
              const int r = row * a.pitch + (lft ? 0 : a.W - x0 + 1);
              const int k = p / (ROWB / 16);
              dst[j] = k * a.a_stride + (int)tc::swizzled<ROWB>(r, p - k * (ROWB / 16));
            }
          }
        }
        if (e0 == 0) ok = warp_wait(&t.bar_a, 0u);  // the copy's zeros have landed
        if (ok) {
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (dst[j] >= 0) *reinterpret_cast<uint4*>(sA + dst[j]) = v[j];
        }
      }
      if (!ok) atomicOr(&t.fail, 1);
      lbnci::fence_async_smem();  // these writes -> the tensor cores' reads
      __syncwarp();
      if (lane == 0) lbnci::mbar_arrive(&t.bar_p);
    }
    const int Wo = a.W << a.up, Ho = a.H << a.up, nacc = a.nm * (a.up ? 4 : 1);
    auto out_row = [&](int m, int par, int r0) {  // output pixel of operand row r0, -1: none
      int r, c;
      if (a.linear) {
        const int pos = m * a.mstart + r0;
        r = pos / a.pitch;
        c = pos - r * a.pitch;
      } else {
        r = r0 >> 3;
        c = 8 * m + (r0 & 7);
      }
      const int yy = y0 + r, xx = x0 + c;
      if (!(r < a.TH && c < a.TW && yy < a.H && xx < a.W)) return -1;
      return a.up ? (b * Ho + 2 * yy + (par >> 1)) * Wo + 2 * xx + (par & 1) : (b * Ho + yy) * Wo + xx;
    };
    if (a.mask)  // the mask's lines into L2 while the MMAs run
      for (int e = et; e < nacc * 128; e += kConvEpiThreads) {
        const int row = out_row((e >> 7) % a.nm, (e >> 7) / a.nm, e & 127);
        if (row >= 0)
          for (int j = 0; j < BN; j += 64)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.mask + (size_t)row * a.ms + n0 + j));
      }
    // drain: group g of four warps takes accumulators g, g + 2, ...
    const bool done = lbnci::mbar_wait(&t.bar_d, 0u);
    if (!done) atomicOr(&t.fail, 1);
    tc::fence_after_sync();
    if (bar_all(1, kConvEpiThreads, done && *(volatile int*)&t.fail == 0)) {
      const int g = (warp - 2) >> 2, quad = warp & 3, l = quad * 32 + lane, gt = et & 127;
      unsigned char* const stg = sm + g * (128 * BN * 2);
      constexpr int NV = BN / 8;                      // 16-byte pieces of a pixel's output
      auto piece = [](int r, int v) {                 // bank-conflict-free place of piece v of row r
        return r * (BN * 2) + ((v ^ ((BN == 32 ? r >> 1 : r) & (NV < 8 ? NV - 1 : 7))) << 4);
      };
      for (int q = g; q < nacc; q += 2) {
        const int par = a.up ? q / a.nm : 0, m = q - par * a.nm;
        // this thread's pieces k = 0 .. NV - 1 of the tile: row (128 k + gt) / NV, piece gt % NV.
        // The first masks are in flight while the accumulator is drained.
        constexpr int UB = NV < 8 ? 4 : 8;
        int orow[UB];
        uint4 mk[UB];
        auto fetch = [&](int k0) {
#pragma unroll
          for (int k = 0; k < UB; ++k) {
            orow[k] = out_row(m, par, ((k0 + k) * 128 + gt) / NV);
            if (a.mask && orow[k] >= 0)
              mk[k] = *reinterpret_cast<const uint4*>(a.mask + (size_t)orow[k] * a.ms + n0 + (gt % NV) * 8);
          }
        };
        fetch(0);
        const unsigned taddr = tmem + (unsigned)(q * BN) + ((unsigned)(quad * 32) << 16);
#pragma unroll
        for (int c0 = 0; c0 < BN; c0 += 32) {
          float acc[32];
          tc::tmem_ld32(taddr + (unsigned)c0, acc);
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const float4 b0 = *reinterpret_cast<const float4*>(&t.bias[c0 + 8 * v]);
            const float4 b1 = *reinterpret_cast<const float4*>(&t.bias[c0 + 8 * v + 4]);
            float r[8] = {acc[8 * v] + b0.x,     acc[8 * v + 1] + b0.y, acc[8 * v + 2] + b0.z, acc[8 * v + 3] + b0.w,
                          acc[8 * v + 4] + b1.x, acc[8 * v + 5] + b1.y, acc[8 * v + 6] + b1.z, acc[8 * v + 7] + b1.w};
            if (a.relu) {
#pragma unroll
              for (int j = 0; j < 8; ++j) r[j] = fmaxf(r[j], 0.f);
            }
            V8 o;
#pragma unroll
            for (int j = 0; j < 4; ++j) o.h[j] = __floats2bfloat162_rn(r[2 * j], r[2 * j + 1]);
            *reinterpret_cast<uint4*>(stg + piece(l, c0 / 8 + v)) = o.u;
          }
        }
        asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory");
#pragma unroll
        for (int k0 = 0; k0 < NV; k0 += UB) {
          if (k0 > 0) fetch(k0);
#pragma unroll
          for (int k = 0; k < UB; ++k) {
            if (orow[k] < 0) continue;
            V8 o;
            o.u = *reinterpret_cast<const uint4*>(stg + piece(((k0 + k) * 128 + gt) / NV, gt % NV));
            if (a.mask) {
              V8 w;
              w.u = mk[k];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float2 mf = __bfloat1622float2(w.h[j]);
                if (!(mf.x > 0.f)) o.h[j].x = __float2bfloat16_rn(0.f);
                if (!(mf.y > 0.f)) o.h[j].y = __float2bfloat16_rn(0.f);
              }
            }
            *reinterpret_cast<uint4*>(a.y + (size_t)orow[k] * a.ys + n0 + (gt % NV) * 8) = o.u;
          }
        }
        asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory");
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  __syncwarp();
  if (warp == 1) tc::tmem_dealloc(tmem, (unsigned)a.cols);
  if (tid == 0 && t.fail) atomicOr(err, t.fail);
}

// ------------------------------------------------------------------ wide images, few channels
// The same convolution for blocks of 32 or 64 output channels on wide images, row by row. An MMA's
// operand fetch (128 rows of A) costs as much for N = 32 as the products of N = 96, so here
// one MMA multiplies an input row, shifted by dx, with the weights of the three dy at once
// (N = 3 BN, the weights stacked dy = +1, 0, -1) into the accumulators of the three output
// rows h = v - 1, v, v + 1 it contributes to, which lie side by side in tensor memory.
// Input rows go by in order, so every output row still adds dy = -1, 0, +1, dx, channels in
// the order of conv3x3_kernel: the same bits. A CTA takes 128 columns of TH output rows: the
// weights stay in shared memory, input rows pass through a ring (each copied once), output
// rows through a ring of R accumulators; a row is drained while the next ones are computed.
//
// up: virtual input row V of the upsampled image is row V >> 1 of the input, taken twice;
// output columns 2 x + px have accumulators of their own (px = 0, 1), reading the input
// column shifted by floor((px + dx)/2).
//
// An accumulator starts from zeros that the draining warps store (a row's first MMA shares
// its instruction with two rows that accumulate); 0 + a is a.
//
// The issuing warp bounds the kernel: a row is 6 to 24 MMAs of 56 cycles, and each barrier it
// waits on or commits to costs it 100 to 300 cycles. So everything goes by units of two virtual
// rows (up: one input row): a stage of the ring is a unit's input rows, and output rows come
// in pairs q (rows 2q, 2q + 1; up: 2q - 1, 2q), of which unit u begins pair u and completes
// pair u - 1: three waits and two commits per unit instead of per row. Slots are handed out
// by pairs; three pairs at least, so that one drains while the next completes. (One row per
// barrier -> two, 32 images: 64 x 256, 32 -> 32 channels 26.7 -> 22.8 us, 64 -> 32 41.0 -> 28.7,
// 32 -> 64 45.1 -> 37.3; 32 x 128, 64 -> 64 24.6 -> 18.4, 128 -> 64 30.8 -> 24.7.)
//
// Warps: 0 copies, 1 issues MMAs, 2..9 drain (two groups of four, alternate rows), 10 patches
// the periodic columns.
constexpr int kRowsThreads = 352, kRowsMaxStage = 8, kRowsMaxSlot = 16;
struct ConvRows {
  const bf16* x;
  int xs, H, W, up;        // input image
  int tiles_x, tiles_h, TH;  // strips of 128 columns, groups of TH output rows
  int nchunk, cstride;     // chunks of ROWB/2 channels; bytes of a row's chunk in shared memory
  int nrow, R;             // input rows in the ring (even unless up), accumulator slots (output rows, even)
  int w_off, stg_off, tail;
  int cols;
  const float* bias;
  int relu;
  bf16* y;
  int ys;
  const bf16* mask;
  int ms;
};
struct RowsTail {
  unsigned long long bar_w, bar_full[kRowsMaxStage], bar_patched[kRowsMaxStage], bar_empty[kRowsMaxStage];
  unsigned long long bar_row[kRowsMaxSlot / 2], bar_free[kRowsMaxSlot / 2];
  unsigned tmem;
  int fail;
  alignas(16) float bias[64];
};

template <int BN, int ROWB>
__global__ void __launch_bounds__(kRowsThreads, 2)
conv3x3_rows_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, ConvRows a,
                    int* err) {
  constexpr int CH = ROWB / 2, KK = CH / 16, WB = BN * ROWB, XW = 130;
  extern __shared__ __align__(1024) unsigned char sm[];
  RowsTail& t = *reinterpret_cast<RowsTail*>(sm + a.tail);
  unsigned char* const sW = sm + a.w_off;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = blockIdx.x % a.tiles_x, th = (blockIdx.x / a.tiles_x) % a.tiles_h;
  const int b = blockIdx.x / (a.tiles_x * a.tiles_h);
  const int x0 = tx * 128, h0 = th * a.TH, n0 = blockIdx.y * BN;
  const int Ho = a.H << a.up, Wo = a.W << a.up, npx = a.up ? 2 : 1;
  const int nh = min(a.TH, Ho - h0);
  const int first = a.up ? (h0 >> 1) - 1 : h0 - 1, nin = a.up ? (nh >> 1) + 2 : nh + 2;
  const int row_bytes = a.nchunk * a.cstride;
  // units: input rows of a stage, stages, units; output pairs (rows 2q - a.up, + 1) and their slots
  const int rpu = 2 - a.up, ns = a.nrow / rpu, nu = (nin + rpu - 1) / rpu;
  const int nq = a.up ? (nh >> 1) + 1 : (nh + 1) >> 1, RP = a.R >> 1;

  if (tid == 0) {
    lbnci::mbar_init(&t.bar_w, 1);
    for (int s = 0; s < ns; ++s) {
      lbnci::mbar_init(&t.bar_full[s], 1);
      lbnci::mbar_init(&t.bar_patched[s], 1);
      lbnci::mbar_init(&t.bar_empty[s], 1);
    }
    for (int s = 0; s < RP; ++s) {
      lbnci::mbar_init(&t.bar_row[s], 1);
      lbnci::mbar_init(&t.bar_free[s], 8);
    }
    t.fail = (smem_u32(sm) & 1023u) ? 2 : 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tc::tmem_alloc(&t.tmem, (unsigned)a.cols);
  if (tid < BN) t.bias[tid] = a.bias ? a.bias[n0 + tid] : 0.f;
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const unsigned tmem = t.tmem;
  const bool aligned = t.fail == 0;
  if (aligned && tid == 0) {
    // the weights (dx, chunk, dy = +1, 0, -1), which no kernel of the chain writes, ahead of the wait
    lbnci::mbar_expect_tx(&t.bar_w, (unsigned)(9 * a.nchunk * WB));
    for (int dxi = 0; dxi < 3; ++dxi)
      for (int k = 0; k < a.nchunk; ++k)
        for (int j = 0; j < 3; ++j)
          lbnci::tma_load_2d(sW + ((dxi * a.nchunk + k) * 3 + j) * WB, &map_w,
                             (((2 - j) * 3 + dxi) * a.nchunk + k) * CH, n0, &t.bar_w);
  }
  lbnci::pdl_enter();

  if (!aligned) {
    // nothing was started
  } else if (warp == 0) {
    if (lane == 0) {  // copies of the rows
      int issued = 0;
      for (int u = 0; u < nu; ++u) {
        const int s = u % ns, w = u / ns, rows = min(rpu, nin - u * rpu);
        if (w > 0 && !lbnci::mbar_wait(&t.bar_empty[s], (unsigned)((w - 1) & 1))) {
          atomicOr(&t.fail, 1);
          break;
        }
        lbnci::mbar_expect_tx(&t.bar_full[s], (unsigned)(rows * a.nchunk * XW * ROWB));
        for (int r = 0; r < rows; ++r)
          for (int k = 0; k < a.nchunk; ++k)
            lbnci::tma_load_4d(sm + (s * rpu + r) * row_bytes + k * a.cstride, &map_x, k * CH, x0 - 1,
                               first + u * rpu + r, b, &t.bar_full[s]);
        issued = u + 1;
      }
      lbnci::mbar_wait(&t.bar_w, 0u);  // every copy has landed before the CTA may end (bounded)
      for (int u = issued > ns ? issued - ns : 0; u < issued; ++u)
        lbnci::mbar_wait(&t.bar_full[u % ns], (unsigned)((u / ns) & 1));
    }
  } else if (warp == 1) {  // MMAs: the whole warp runs the loop
    const unsigned long long d0 = tc::desc_base(ROWB, 16u, 8u * ROWB);
    const unsigned hi = (unsigned)(d0 >> 32);
    const unsigned loA = (unsigned)d0 + (smem_u32(sm) >> 4), loW = (unsigned)d0 + (smem_u32(sW) >> 4);
    bool bad = __any_sync(~0u, !lbnci::mbar_wait(&t.bar_w, 0u));
    int s = 0, q = 0, last = RP - 1, base = a.R - 2;  // stage, slots of pairs u and u - 1, slot of row v - 1
    unsigned ph = 0u, qph = 0u;
    for (int u = 0; u < nu; ++u) {
      bad = bad || !lbnci::mbar_wait(&t.bar_full[s], ph) || !lbnci::mbar_wait(&t.bar_patched[s], ph) ||
            (u < nq && !lbnci::mbar_wait(&t.bar_free[q], qph));  // the pair's slots are drained and zeroed
      bad = __any_sync(~0u, bad);
      if (bad) break;
      tc::fence_after_sync();
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        const int v = 2 * u - 1 - a.up + pass;  // virtual input row, relative to h0
        if (v >= -1 && v <= nh) {
          const unsigned la = loA + (unsigned)(((s * rpu + (a.up ? 0 : pass)) * row_bytes) >> 4);
          const int lo = max(0, v - 1), n = min(nh - 1, v + 1) - lo + 1, j0 = lo - (v - 1);
          // rows lo .. lo + n - 1 in slots; beyond the last slot they continue at slot 0
          const int at = base + j0, slot = at >= a.R ? at - a.R : at, n1 = min(n, a.R - slot);
          auto rows = [&](int sl, int j, int nn) {
            const unsigned id = tc::idesc_bf16(128, 0) | ((unsigned)(nn * BN / 8) << 17);
            // dx outermost, then channels: the order of the taps
#pragma unroll
            for (int dxi = 0; dxi < 3; ++dxi)
              for (int k = 0; k < a.nchunk; ++k) {
                const unsigned lw = loW + (unsigned)((((dxi * a.nchunk + k) * 3 + j) * WB) >> 4);
                const unsigned lk = la + (unsigned)((k * a.cstride) >> 4);
                for (int px = 0; px < npx; ++px) {
                  const int ox = a.up ? (px + dxi - 1) >> 1 : dxi - 1;
                  const unsigned lr = lk + (unsigned)(((ox + 1) * ROWB) >> 4);
                  const unsigned d = tmem + (unsigned)((px * a.R + sl) * BN);
#pragma unroll
                  for (int kk = 0; kk < KK; ++kk)
                    tc::mma_bf16(d, tc::desc64(hi, lr + 2 * kk), tc::desc64(hi, lw + 2 * kk), id);
                }
              }
          };
          rows(slot, j0, n1);
          if (n1 < n) rows(0, j0 + n1, n - n1);
        }
        if (++base == a.R) base = 0;
      }
      tc::mma_commit(&t.bar_empty[s]);
      if (u > 0) tc::mma_commit(&t.bar_row[last]);  // output pair u - 1 is complete
      last = q;
      if (++q == RP) {
        q = 0;
        qph ^= 1u;
      }
      if (++s == ns) {
        s = 0;
        ph ^= 1u;
      }
    }
    if (lane == 0 && bad) atomicOr(&t.fail, 1);
    // the MMAs issued are done before tensor memory is released: the last pair's barrier below
  } else if (warp == 10) {  // the periodic images of the columns beyond the image
    const int left = x0 == 0 ? 1 : 0, right = x0 + 128 >= a.W ? 1 : 0, ncol = left + right;
    const int vpp = a.nchunk * (ROWB / 16), count = ncol * vpp;
    bool ok = true;
    for (int u = 0; u < nu && ok; ++u) {
      const int s = u % ns;
      for (int e0 = 0; e0 < rpu * count || e0 == 0; e0 += 64) {
        uint4 v[2];
        int dst[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int e = e0 + 32 * j + lane;
          dst[j] = -1;
          const int r = e >= count ? 1 : 0, f = e - r * count, i = u * rpu + r, yy = first + i;
          if (e < rpu * count && i < nin && yy >= 0 && yy < a.H) {
            const int col = f / vpp, p = f - col * vpp, k = p / (ROWB / 16);
            const bool lft = left && col == 0;
            v[j] = *reinterpret_cast<const uint4*>(a.x + ((size_t)(b * a.H + yy) * a.W + (lft ? a.W - 1 : 0)) * a.xs + p * 8);
            dst[j] = (s * rpu + r) * row_bytes + k * a.cstride +
                     (int)tc::swizzled<ROWB>(lft ? 0 : a.W - x0 + 1, p - k * (ROWB / 16));
          }
        }
        if (e0 == 0) ok = warp_wait(&t.bar_full[s], (unsigned)((u / ns) & 1));
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (dst[j] >= 0) *reinterpret_cast<uint4*>(sm + dst[j]) = v[j];
      }
      lbnci::fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        if (!ok) atomicOr(&t.fail, 1);
        lbnci::mbar_arrive(&t.bar_patched[s]);
      }
    }
  } else {  // drain
    const int g = (warp - 2) >> 2, quad = warp & 3, l = quad * 32 + lane, gt = (tid - 64) & 127;
    const unsigned tq = tmem + ((unsigned)(quad * 32) << 16);
    auto zero = [&](int slot) {  // this warp's lanes of a slot's accumulators
      for (int px = 0; px < npx; ++px)
#pragma unroll
        for (int c0 = 0; c0 < BN; c0 += 16) tc::tmem_zero16(tq + (unsigned)((px * a.R + slot) * BN + c0));
      tc::tmem_wait_st();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) lbnci::mbar_arrive(&t.bar_free[slot >> 1]);
    };
    for (int s = g; s < a.R; s += 2) zero(s);
    unsigned char* const stg = sm + a.stg_off + g * (128 * BN * 2);
    constexpr int NV = BN / 8;
    auto piece = [](int r, int v) { return r * (BN * 2) + ((v ^ ((BN == 32 ? r >> 1 : r) & (NV - 1))) << 4); };
    bool ok = true;
    int qs = 0;
    unsigned qph = 0u;
    for (int q = 0; q < nq && ok; ++q) {
      const int h = 2 * q - a.up + g, slot = 2 * qs + g;
      unsigned long long* const done = &t.bar_row[qs];
      const unsigned dph = qph;
      if (++qs == RP) {
        qs = 0;
        qph ^= 1u;
      }
      if (h < 0 || h >= nh) {  // the pair's other row is the image's first or last
        ok = warp_wait(done, dph);
        if (!ok) atomicOr(&t.fail, 1);
        ok = bar_all(1 + g, 128, ok);  // the group leaves the loop together: its barriers count all of it
        if (q + RP < nq) zero(slot);
        continue;
      }
      for (int px = 0; px < npx; ++px) {
        // this thread's pieces: row (128 k + gt) / NV, piece gt % NV; the masks are in flight
        // while the row is awaited
        int orow[NV];
        uint4 mk[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          const int x = x0 + (k * 128 + gt) / NV;
          orow[k] = x < a.W ? (b * Ho + h0 + h) * Wo + (a.up ? 2 * x + px : x) : -1;
          if (a.mask && orow[k] >= 0)
            mk[k] = *reinterpret_cast<const uint4*>(a.mask + (size_t)orow[k] * a.ms + n0 + (gt % NV) * 8);
        }
        if (px == 0) {
          ok = lbnci::mbar_wait(done, dph);
          if (!ok) atomicOr(&t.fail, 1);
          tc::fence_after_sync();
        }
#pragma unroll
        for (int c0 = 0; c0 < BN; c0 += 32) {
          float acc[32];
          tc::tmem_ld32(tq + (unsigned)((px * a.R + slot) * BN + c0), acc);
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const float4 b0 = *reinterpret_cast<const float4*>(&t.bias[c0 + 8 * v]);
            const float4 b1 = *reinterpret_cast<const float4*>(&t.bias[c0 + 8 * v + 4]);
            float r[8] = {acc[8 * v] + b0.x,     acc[8 * v + 1] + b0.y, acc[8 * v + 2] + b0.z, acc[8 * v + 3] + b0.w,
                          acc[8 * v + 4] + b1.x, acc[8 * v + 5] + b1.y, acc[8 * v + 6] + b1.z, acc[8 * v + 7] + b1.w};
            if (a.relu) {
#pragma unroll
              for (int j = 0; j < 8; ++j) r[j] = fmaxf(r[j], 0.f);
            }
            V8 o;
#pragma unroll
            for (int j = 0; j < 4; ++j) o.h[j] = __floats2bfloat162_rn(r[2 * j], r[2 * j + 1]);
            *reinterpret_cast<uint4*>(stg + piece(l, c0 / 8 + v)) = o.u;
          }
        }
        if (px == npx - 1 && q + RP < nq) zero(slot);  // for row h + R
        ok = bar_all(1 + g, 128, ok);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          if (orow[k] < 0 || !ok) continue;
          V8 o;
          o.u = *reinterpret_cast<const uint4*>(stg + piece((k * 128 + gt) / NV, gt % NV));
          if (a.mask) {
            V8 w;
            w.u = mk[k];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float2 mf = __bfloat1622float2(w.h[j]);
              if (!(mf.x > 0.f)) o.h[j].x = __float2bfloat16_rn(0.f);
              if (!(mf.y > 0.f)) o.h[j].y = __float2bfloat16_rn(0.f);
            }
          }
          *reinterpret_cast<uint4*>(a.y + (size_t)orow[k] * a.ys + n0 + (gt % NV) * 8) = o.u;
        }
        asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory");
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  __syncwarp();
  if (warp == 1) tc::tmem_dealloc(tmem, (unsigned)a.cols);
  if (tid == 0 && t.fail) atomicOr(err, t.fail);
}

// ------------------------------------------------------------------ weight gradient
// dw[o][t][c] = sum_p dy[p][o] xpad[p + t][c] as a GEMM with the pixels as K: both operands
// are MN-major (channels contiguous), so the copied tiles are used as they arrive: x as the
// tile and its ring of one pixel (CH = ROWB/2 channels, the chunk blockIdx.y), dy as the
// tile (BN channels, block blockIdx.z). Shifting x by a tap is again only a start address,
// and M = 128 holds several taps: the operand's blocks of CH channels lie `leading byte
// offset` apart, which may be one pixel:
//   CH = 32  3 accumulators, dy = -1, 0, 1; blocks dx = -1, 0, 1 (and 2, dropped)
//   CH = 64  5 accumulators of two taps each, (0, 1), (2, 3), ... (8, dropped)
//   up       the input is low-resolution and dy is copied per parity (py, px) of the output
//            pixels; a parity meets only the shifts (py - 1, py) x (px - 1, px), so 4 x 2
//            accumulators of two neighbouring shifts hold everything, and the reduction
//            adds the parities' parts of each tap.
// CTA (s, k, n) takes the tiles of split s and writes its partial sums; the epilogue warps
// patch the periodic columns of x stage by stage, sum dy for the bias (chunk 0) and drain
// the accumulators. Sums run over the same pixels as in conv3x3_wgrad_kernel with shorter
// chains (more splits).
struct WgradTma {
  const bf16* x;
  int xs, H, W;       // position grid: the image of x
  int up;
  int tiles_x, tiles_y, ntile, nsplit;
  int TH, TW, pitch;
  int x_bytes, d_bytes;  // shared memory of a stage: the x tile, one dy tile (four when up)
  int nstage, cols, tail;
  int Cin, Cout;
  float* part;        // [nsplit][Cout][9 Cin], up: [nsplit][Cout][16 Cin]
  float* bpart;       // [nsplit][Cout] or null
};
struct WgradMaps {
  CUtensorMap x, dy[4];  // dy: all pixels, or the pixels of each parity 2 py + px
};
constexpr int kWgradMaxStage = 4;
struct WgradTail {
  unsigned long long bar_d, bar_full[kWgradMaxStage], bar_patched[kWgradMaxStage], bar_empty[kWgradMaxStage];
  unsigned tmem;
  int fail;
};

template <int BN, int ROWB>
__global__ void __launch_bounds__(kConvThreads, 2)
conv3x3_wgrad_tma_kernel(const __grid_constant__ WgradMaps maps, WgradTma a, int* err) {
  constexpr int CH = ROWB / 2, DROW = BN * 2;
  constexpr unsigned IDESC = tc::idesc_bf16(128, BN, true);
  extern __shared__ __align__(1024) unsigned char sm[];
  WgradTail& t = *reinterpret_cast<WgradTail*>(sm + a.tail);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int split = blockIdx.x, c0 = blockIdx.y * CH, n0 = blockIdx.z * BN;
  const int t0 = (int)((long long)a.ntile * split / a.nsplit), t1 = (int)((long long)a.ntile * (split + 1) / a.nsplit);
  const int nt = t1 - t0, ST = a.nstage, npar = a.up ? 4 : 1;
  const int stage_bytes = a.x_bytes + npar * a.d_bytes;

  if (tid == 0) {
    lbnci::mbar_init(&t.bar_d, 2);
    for (int s = 0; s < ST; ++s) {
      lbnci::mbar_init(&t.bar_full[s], 1);
      lbnci::mbar_init(&t.bar_patched[s], kConvEpiThreads / 32);
      lbnci::mbar_init(&t.bar_empty[s], 1 + kConvEpiThreads / 32);
    }
    t.fail = (smem_u32(sm) & 1023u) ? 2 : 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tc::tmem_alloc(&t.tmem, (unsigned)a.cols);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const unsigned tmem = t.tmem;
  const bool aligned = t.fail == 0;
  lbnci::pdl_enter();
  auto origin = [&](int i, int& b, int& y0, int& x0) {
    const int tt = t0 + i;
    x0 = (tt % a.tiles_x) * a.TW;
    y0 = ((tt / a.tiles_x) % a.tiles_y) * a.TH;
    b = tt / (a.tiles_x * a.tiles_y);
  };

  if (!aligned) {
  } else if (warp == 0) {
    if (lane == 0) {  // copies
      int issued = 0;
      for (int i = 0; i < nt; ++i) {
        const int s = i % ST, u = i / ST;
        if (u > 0 && !lbnci::mbar_wait(&t.bar_empty[s], (unsigned)((u - 1) & 1))) {
          atomicOr(&t.fail, 1);
          break;
        }
        int b, y0, x0;
        origin(i, b, y0, x0);
        unsigned char* sx = sm + s * stage_bytes;
        lbnci::mbar_expect_tx(&t.bar_full[s],
                              (unsigned)(ROWB * (a.TW + 2) * (a.TH + 2) + npar * DROW * a.TW * a.TH));
        lbnci::tma_load_4d(sx, &maps.x, c0, x0 - 1, y0 - 1, b, &t.bar_full[s]);
        for (int q = 0; q < npar; ++q)
          lbnci::tma_load_4d(sx + a.x_bytes + q * a.d_bytes, &maps.dy[q], n0, x0, y0, b, &t.bar_full[s]);
        issued = i + 1;
      }
      for (int i = issued > ST ? issued - ST : 0; i < issued; ++i)
        lbnci::mbar_wait(&t.bar_full[i % ST], (unsigned)((i / ST) & 1));
    }
  } else if (warp == 1) {  // MMAs: the whole warp runs the loop
    bool bad = false;
    const unsigned long long dB = tc::desc_base(DROW, 16u, 8u * DROW);
    const unsigned hiA = (unsigned)(tc::desc_base(ROWB, 16u, 8u * ROWB) >> 32), hiB = (unsigned)(dB >> 32);
    const unsigned base = smem_u32(sm) >> 4;
    const int kx = a.TW / 16;
    // A descriptors of the accumulators relative to the pixel's own position: start (the
    // shift) and leading byte offset (to the next block of channels), lower half
    constexpr int NA = ROWB == 64 ? 3 : 8;
    unsigned rel[NA];
    if constexpr (ROWB == 64) {
#pragma unroll
      for (int j = 0; j < 3; ++j) rel[j] = (unsigned)((j * a.pitch * 64) >> 4) + (4u << 16);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (a.up) {  // parity j >> 1, shift row j & 1
          const int q = j >> 1;
          rel[j] = (unsigned)((((q >> 1) + (j & 1)) * a.pitch + (q & 1)) * 8) + (8u << 16);
        } else {  // taps 2j and 2j + 1
          const int o0 = (2 * j / 3) * a.pitch + (2 * j) % 3, o1 = ((2 * j + 1) / 3) * a.pitch + (2 * j + 1) % 3;
          rel[j] = (unsigned)(o0 * 8) + ((unsigned)((j < 4 ? o1 - o0 : 1) * 8) << 16);
        }
      }
    }
    const unsigned dpar = (unsigned)(a.d_bytes >> 4);
    unsigned ph = 0u;
    int s = 0;
    auto block = [&](unsigned ua, unsigned ub, int acc) {  // the MMAs of K = 16 pixels of a row
      if (ROWB == 128 && a.up) {
#pragma unroll
        for (int j = 0; j < NA; ++j)
          tc::mma_bf16_if(tmem + j * BN, tc::desc64(hiA, ua + rel[j]), tc::desc64(hiB, ub + (unsigned)(j >> 1) * dpar),
                          IDESC, acc);
      } else {
#pragma unroll
        for (int j = 0; j < (ROWB == 64 ? 3 : 5); ++j)
          tc::mma_bf16_if(tmem + j * BN, tc::desc64(hiA, ua + rel[j]), tc::desc64(hiB, ub), IDESC, acc);
      }
    };
    // Only the image's rows of a tile are multiplied: below the last one dy arrives as zeros, which
    // times an infinite x of the row above would be NaN in taps that this x has no part in.
    int tx = t0 % a.tiles_x, ty = (t0 / a.tiles_x) % a.tiles_y;
    for (int i = 0; i < nt; ++i) {
      const int rows = min(a.TH, a.H - ty * a.TH);
      if (++tx == a.tiles_x) {
        tx = 0;
        if (++ty == a.tiles_y) ty = 0;
      }
      bad = __any_sync(~0u, !lbnci::mbar_wait(&t.bar_full[s], ph) || !lbnci::mbar_wait(&t.bar_patched[s], ph));
      if (bad) break;
      tc::fence_after_sync();
      const unsigned ux = base + (unsigned)((s * stage_bytes) >> 4);
      const unsigned ud = ux + (unsigned)(a.x_bytes >> 4) + (unsigned)dB;
      for (int r = 0; r < rows; ++r) {
        unsigned ua = ux + (unsigned)((r * a.pitch * ROWB) >> 4), ub = ud + (unsigned)((r * a.TW * DROW) >> 4);
        for (int c = 0; c < kx; ++c) {
          block(ua, ub, i | r | c);
          ua += ROWB;  // 16 pixels of ROWB bytes, in 16-byte units
          ub += DROW;
        }
      }
      tc::mma_commit(&t.bar_empty[s]);
      if (++s == ST) {
        s = 0;
        ph ^= 1u;
      }
    }
    if (lane == 0 && bad) atomicOr(&t.fail, 1);
    tc::mma_commit(&t.bar_d);
    if (lane == 0) lbnci::mbar_arrive(&t.bar_d);
  } else {
    const int et = tid - 64;
    constexpr int VX = ROWB / 16, VD = DROW / 16, DR = kConvEpiThreads / VD;
    const bool do_bias = a.bpart != nullptr && blockIdx.y == 0;
    float bs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    bool ok = true;
    for (int i = 0; i < nt && ok; ++i) {
      const int s = i % ST;
      const unsigned ph = (unsigned)((i / ST) & 1);
      int b, y0, x0;
      origin(i, b, y0, x0);
      unsigned char* sx = sm + s * stage_bytes;
      const int left = x0 == 0 ? 1 : 0, right = x0 + a.TW >= a.W ? 1 : 0;
      const int ncol = left + right, count = ncol * (a.TH + 2) * VX;
      constexpr int U = 2;
      uint4 v[U];
      int dst[U];
      for (int e0 = 0; e0 < count || e0 == 0; e0 += U * kConvEpiThreads) {
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const int e = e0 + j * kConvEpiThreads + et;
          dst[j] = -1;
          if (e < count) {
            const int px = e / VX, p = e - px * VX;
            const int row = px / ncol, col = px - row * ncol;
            const int yy = y0 - 1 + row;
            if (yy >= 0 && yy < a.H) {
              const bool lft = left && col == 0;
              v[j] = *reinterpret_cast<const uint4*>(a.x + ((size_t)(b * a.H + yy) * a.W + (lft ? a.W - 1 : 0)) * a.xs +
                                                     c0 + p * 8);
              dst[j] = (int)tc::swizzled<ROWB>(row * a.pitch + (lft ? 0 : a.W - x0 + 1), p);
            }
          }
        }
        if (e0 == 0) ok = warp_wait(&t.bar_full[s], ph);
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (dst[j] >= 0) *reinterpret_cast<uint4*>(sx + dst[j]) = v[j];
      }
      lbnci::fence_async_smem();
      __syncwarp();
      if (lane == 0) lbnci::mbar_arrive(&t.bar_patched[s]);
      if (do_bias && ok)
        for (int q = 0; q < npar; ++q)
          for (int r = et / VD; r < a.TH * a.TW; r += DR) {
            V8 d;
            d.u = *reinterpret_cast<const uint4*>(sx + a.x_bytes + q * a.d_bytes + tc::swizzled<DROW>(r, et % VD));
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float2 f = __bfloat1622float2(d.h[j]);
              bs[2 * j] += f.x;
              bs[2 * j + 1] += f.y;
            }
          }
      __syncwarp();
      if (lane == 0) lbnci::mbar_arrive(&t.bar_empty[s]);
    }
    if (!ok) atomicOr(&t.fail, 1);
    if (!warp_wait(&t.bar_d, 0u)) {
      ok = false;
      atomicOr(&t.fail, 1);
    }
    tc::fence_after_sync();
    // every epilogue warp is past the stages
    if (bar_all(1, kConvEpiThreads, ok && *(volatile int*)&t.fail == 0)) {
      if (do_bias) {  // thread sums, added in thread order
        float* red = reinterpret_cast<float*>(sm);
#pragma unroll
        for (int j = 0; j < 8; ++j) red[(et / VD) * BN + (et % VD) * 8 + j] = bs[j];
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (do_bias && et < BN) {
        const float* red = reinterpret_cast<const float*>(sm);
        float v = 0.f;
        for (int r = 0; r < DR; ++r) v += red[r * BN + et];
        a.bpart[(size_t)split * a.Cout + n0 + et] = v;
      }
      const int g = (warp - 2) >> 2, quad = warp & 3, l = quad * 32 + lane;
      const int blk = l / CH, ci = c0 + l % CH;  // block of the operand's M rows, input channel
      const int nacc = a.up ? 8 : (ROWB == 64 ? 3 : 5), nk = a.up ? 16 : 9;
      for (int q = g; q < nacc; q += 2) {
        int k = -1;  // row block of the partial sums: the tap, or (parity, shift)
        if (a.up) k = blk < 2 ? 2 * q + blk : -1;
        else if (ROWB == 64) k = blk < 3 ? 3 * q + blk : -1;
        else k = 2 * q + blk < 9 ? 2 * q + blk : -1;
        float* out = a.part + ((size_t)split * a.Cout + n0) * nk * a.Cin + (size_t)(k < 0 ? 0 : k) * a.Cin + ci;
        const unsigned taddr = tmem + (unsigned)(q * BN) + ((unsigned)(quad * 32) << 16);
#pragma unroll
        for (int j0 = 0; j0 < BN; j0 += 32) {
          float acc[32];
          tc::tmem_ld32(taddr + (unsigned)j0, acc);
          if (k >= 0) {
#pragma unroll
            for (int j = 0; j < 32; ++j) out[(size_t)(j0 + j) * nk * a.Cin] = acc[j];
          }
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  __syncwarp();
  if (warp == 1) tc::tmem_dealloc(tmem, (unsigned)a.cols);
  if (tid == 0 && t.fail) atomicOr(err, t.fail);
}

// Sum the split partials: dw[o][t][c] for c < cin_true (master layout [Cout][3][3][cin_true])
// and db[o] (the last blocks). A block takes 256 / S groups of four consecutive values, S
// threads to each (thread k the splits k, k + S, ...; their sums added in thread order), S
// so large that the grid fills the multiprocessors: whole lines are read, every load of a
// thread is independent. up: a tap's sum also runs over the four parities, each at the
// shift floor((parity + tap)/2) the tap has there, the four loads of a split issued together (32
// images, cold: 12.4, 20.3 and 17.7 us for the three such layers with a parity at a time, all 17
// reductions 174 us, now 158).
__global__ void __launch_bounds__(256) wgrad_reduce_tma_kernel(const float* __restrict__ part,
                                                               const float* __restrict__ bpart, int nsplit, int Cout,
                                                               int Cin, int cin_true, int up, int S, int wblocks,
                                                               float* __restrict__ dw, float* __restrict__ db) {
  __shared__ float4 s[256];
  lbnci::pdl_enter();
  if ((int)blockIdx.x >= wblocks) {  // 32 output channels of the bias, eight threads to each
    float* sb = reinterpret_cast<float*>(s);
    const int o = ((int)blockIdx.x - wblocks) * 32 + (threadIdx.x & 31), share = threadIdx.x >> 5;
    float v = 0.f;
    if (o < Cout) {
#pragma unroll 4
      for (int z = share; z < nsplit; z += 8) v += bpart[(size_t)z * Cout + o];
    }
    sb[threadIdx.x] = v;
    __syncthreads();
    if (share == 0 && o < Cout) {
      float r = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) r += sb[k * 32 + threadIdx.x];
      db[o] = r;
    }
    return;
  }
  const int V = 256 / S, vec = threadIdx.x % V, share = threadIdx.x / V;
  const int nk = up ? 16 : 9, c4 = Cin / 4, n4 = Cout * 9 * c4;
  const int i = blockIdx.x * V + vec;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  int c = 0, tap = 0, o = 0;
  if (i < n4) {
    c = (i % c4) * 4;
    const int r = i / c4;
    tap = r % 9;
    o = r / 9;
    const size_t stride = (size_t)Cout * nk * Cin;
    const int dy = tap / 3 - 1, dx = tap % 3 - 1;
    const float* p[4];  // the parities' parts: shift row py - 1 + sy, column px - 1 + sx
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int py = q >> 1, px = q & 1;
      const int k = up ? 4 * q + 2 * (((py + dy) >> 1) - py + 1) + (((px + dx) >> 1) - px + 1) : tap;
      p[q] = part + ((size_t)o * nk + k) * Cin + c;
    }
    auto add = [&](const float* at) {
      const float4 w = *reinterpret_cast<const float4*>(at);
      v.x += w.x;
      v.y += w.y;
      v.z += w.z;
      v.w += w.w;
    };
    if (up) {
#pragma unroll 2
      for (int z = share; z < nsplit; z += S)
#pragma unroll
        for (int q = 0; q < 4; ++q) add(p[q] + (size_t)z * stride);
    } else {
#pragma unroll 4
      for (int z = share; z < nsplit; z += S) add(p[0] + (size_t)z * stride);
    }
  }
  s[threadIdx.x] = v;
  __syncthreads();
  if (share == 0 && i < n4) {
    for (int k = 1; k < S; ++k) {
      const float4 w = s[k * V + vec];
      v.x += w.x;
      v.y += w.y;
      v.z += w.z;
      v.w += w.w;
    }
    float* out = dw + ((size_t)o * 9 + tap) * cin_true + c;
    if (c < cin_true) out[0] = v.x;
    if (c + 1 < cin_true) out[1] = v.y;
    if (c + 2 < cin_true) out[2] = v.z;
    if (c + 3 < cin_true) out[3] = v.w;
  }
}

}  // namespace lbu
