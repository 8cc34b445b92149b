// Learned post-equaliser (declared in rx_cnn.h): BF16 tensor-core
// convolutions with FP32 accumulation for the forward pass, the input
// gradient and the weight gradient, and an FP32 Adam update.
//
// Layout.  Activations are channels-last BF16 rows [n][c] (c = 16 for the
// 4 input features and for dJ/dy, zero padded; 64 for hidden layers).  A
// convolution out[n][co] = sum_k sum_ci in[n + k - 7][ci] W[k][ci][co] is 15
// accumulated GEMMs over shifted views of the same input rows, so one CTA
// stages a tile of 128 + 14 input rows and all 15 weight matrices in shared
// memory and its 8 warps each produce 16 rows x all output channels with
// mma.m16n8k16 (BF16 in, FP32 accumulate); ldmatrix feeds the fragments
// from rows padded by 16 bytes (conflict-free).  The input gradient is the
// same convolution with the taps reversed and W transposed (packed once per
// update), fused with the ReLU mask of the layer below.  The weight
// gradient dW[k][ci][co] = sum_n in[n + k - 7][ci] dz[n][co] is a GEMM with
// the symbols as the reduction dimension: CTAs own (symbol chunk, 3 taps),
// read both operands transposed by ldmatrix.trans, and add their partial
// sums into the FP32 gradient with atomics.  This mma.sync form runs when tcgen05 is
// switched off (RX_CNN_OPT_TCGEN05 = 0); the default form follows below it.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include "../../include/rx_cnn.h"

namespace {

typedef __nv_bfloat16 bf16;

constexpr int KS = 15, HALF = 7, CH = 64, FEAT = 4, FEATP = 16;
constexpr int TM = 128;          // symbols per tile
constexpr int kThreads = 256;    // 8 warps x 16 rows
constexpr int TG = 5;            // taps per weight-gradient CTA (3 groups)

__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void ldsm_x4(unsigned addr, unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(unsigned addr, unsigned &r0, unsigned &r1, unsigned &r2, unsigned &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(unsigned addr, unsigned &r0, unsigned &r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_t(unsigned addr, unsigned &r0, unsigned &r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(addr));
}
// D = A (16x16, row) * B (16x8, col) + D, BF16 inputs, FP32 accumulate
__device__ __forceinline__ void mma(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                    unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

enum { EPI_RELU = 0, EPI_LAST = 1, EPI_MASK = 2 };

struct ConvArgs {
  const bf16 *in;             // [K][CIN]
  int64_t K;
  const bf16 *w;              // [15][COUT][CIN]
  const float *bias;          // [n_bias] (EPI_RELU, EPI_LAST)
  int n_bias;
  bf16 *out;                  // [K][COUT] (EPI_RELU, EPI_MASK)
  const bf16 *mask;           // [K][COUT] (EPI_MASK): keep where mask > 0
  // EPI_LAST: y = z + conv (4 channels = 2 complex pols); training also
  // forms dJ/dy = 2 (y - t) / (4K) into dout [K][16] and the loss
  const float2 *z; int64_t z_stride;
  float2 *y; int64_t y_stride;
  const float2 *t; int64_t t_stride;
  bf16 *dout;
  double *loss;
  float inv4k;
  // the first kernel of a training pass zeroes what later ones add to
  float *zero;
  int64_t n_zero;
};

template <int CIN, int COUT, int EPI>
__global__ void __launch_bounds__(kThreads, 1) conv_kernel(const ConvArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int CP = CIN + 8;                       // padded shared row (elements)
  bf16 *Ws = reinterpret_cast<bf16 *>(smem_raw);    // [15][COUT][CP]
  bf16 *Xs = Ws + KS * COUT * CP;                   // [TM + 14][CP]
  constexpr int CH8 = CIN / 8;                      // 16-byte pieces per row
  for (int i = threadIdx.x; i < KS * COUT * CH8; i += kThreads) {
    const int row = i / CH8, p = i % CH8;
    *reinterpret_cast<uint4 *>(Ws + row * CP + p * 8) = *reinterpret_cast<const uint4 *>(a.w + (size_t)row * CIN + p * 8);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = lane >> 2, tig = lane & 3;
  const int m0 = warp * 16;
  // ldmatrix row / column of this lane: A (rows 0-7 | 8-15) x (cols 0-7 | 8-15) in
  // fragment order; B (out channels 0-7 | 8-15) x (in channels 0-7 | 8-15)
  const int a_row = (lane & 7) + ((lane >> 3) & 1) * 8, a_col = (lane >> 4) * 8;
  const int b_row = (lane & 7) + (lane >> 4) * 8, b_col = ((lane >> 3) & 1) * 8;
  const int64_t n_tiles = (a.K + TM - 1) / TM;
  double loss_part = 0.0;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t n0 = tile * TM;
    __syncthreads();   // weights staged, previous tile's rows consumed
    for (int i = threadIdx.x; i < (TM + 2 * HALF) * CH8; i += kThreads) {
      const int r = i / CH8, p = i % CH8;
      const int64_t n = n0 - HALF + r;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (n >= 0 && n < a.K) v = *reinterpret_cast<const uint4 *>(a.in + n * CIN + p * 8);
      *reinterpret_cast<uint4 *>(Xs + r * CP + p * 8) = v;
    }
    __syncthreads();
    float acc[COUT / 8][4];
#pragma unroll
    for (int j = 0; j < COUT / 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll 1
    for (int k = 0; k < KS; ++k) {
#pragma unroll
      for (int cc = 0; cc < CIN / 16; ++cc) {
        unsigned a0, a1, a2, a3;
        ldsm_x4(smem_u32(Xs + (m0 + k + a_row) * CP + cc * 16 + a_col), a0, a1, a2, a3);
        if constexpr (COUT >= 16) {
#pragma unroll
          for (int jp = 0; jp < COUT / 16; ++jp) {
            unsigned b0, b1, b2, b3;
            ldsm_x4(smem_u32(Ws + (k * COUT + jp * 16 + b_row) * CP + cc * 16 + b_col), b0, b1, b2, b3);
            mma(acc[2 * jp], a0, a1, a2, a3, b0, b1);
            mma(acc[2 * jp + 1], a0, a1, a2, a3, b2, b3);
          }
        } else {
          unsigned b0, b1;
          ldsm_x2(smem_u32(Ws + (k * COUT + (lane & 7)) * CP + cc * 16 + b_col), b0, b1);
          mma(acc[0], a0, a1, a2, a3, b0, b1);
        }
      }
    }
    // epilogue: rows n0 + m0 + group (+8), channels j*8 + 2 tig (+1)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t n = n0 + m0 + group + 8 * h;
      if (n >= a.K) continue;
      if constexpr (EPI == EPI_LAST) {
        if (tig < 2) {   // channels 2 tig, 2 tig + 1 = (re, im) of pol tig
          const int pol = tig;
          const float2 x = a.z[pol * a.z_stride + n];
          const float b0 = 2 * pol < a.n_bias ? a.bias[2 * pol] : 0.f;
          const float b1 = 2 * pol + 1 < a.n_bias ? a.bias[2 * pol + 1] : 0.f;
          const float2 yv = make_float2(x.x + (acc[0][2 * h] + b0), x.y + (acc[0][2 * h + 1] + b1));
          if (a.y) a.y[pol * a.y_stride + n] = yv;
          if (a.t) {
            const float2 tv = a.t[pol * a.t_stride + n];
            const float dx = yv.x - tv.x, dy = yv.y - tv.y;
            loss_part += (double)dx * dx + (double)dy * dy;
            *reinterpret_cast<__nv_bfloat162 *>(a.dout + n * FEATP + 2 * pol) =
                __floats2bfloat162_rn(2.f * dx * a.inv4k, 2.f * dy * a.inv4k);
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < COUT / 8; ++j) {
          const int co = j * 8 + 2 * tig;
          float v0 = acc[j][2 * h], v1 = acc[j][2 * h + 1];
          if constexpr (EPI == EPI_RELU) {
            v0 = fmaxf(v0 + (co < a.n_bias ? a.bias[co] : 0.f), 0.f);
            v1 = fmaxf(v1 + (co + 1 < a.n_bias ? a.bias[co + 1] : 0.f), 0.f);
          } else {
            const __nv_bfloat162 mk = *reinterpret_cast<const __nv_bfloat162 *>(a.mask + n * COUT + co);
            v0 = __bfloat162float(mk.x) > 0.f ? v0 : 0.f;
            v1 = __bfloat162float(mk.y) > 0.f ? v1 : 0.f;
          }
          *reinterpret_cast<__nv_bfloat162 *>(a.out + n * COUT + co) = __floats2bfloat162_rn(v0, v1);
        }
      }
    }
  }
  if constexpr (EPI == EPI_LAST) {
    if (a.t) {
      for (int o = 16; o >= 1; o >>= 1) loss_part += __shfl_xor_sync(0xffffffffu, loss_part, o);
      if (lane == 0 && loss_part != 0.0) atomicAdd(a.loss, loss_part * (double)a.inv4k);
    }
  }
}

// ---------------------------------------------------------------- tcgen05 path
// All convolutions of the learned form on the 5th-generation tensor cores (BF16 in,
// FP32 accumulate in tensor memory), one tile = 128 symbols (MMA M = 128 rows).
//
// 64 -> 64 layers (conv_tc_kernel): one persistent CTA per SM with all 15 weight
// matrices (120 KB) in shared memory.  Warp 0 loads (TMA), warp 1 issues the MMAs,
// warps 2-5 read the accumulators back and store; no CTA-wide barrier in the loop.
// A tile's 142 input rows (128 + 14 halo, zero-filled beyond the sequence) arrive as one
// box of 142 x 64 channels in the 128-byte-swizzled K-major layout, three stages deep;
// the operand of tap k is the same box 128 k bytes further on.  The swizzle is what
// makes that shift free: a row's 16-byte pieces sit in eight different bank groups
// whatever row the operand starts at, while in the unswizzled layout (8 rows x 16 bytes
// contiguous) a shift by k rows puts every core matrix across two 128-byte lines and
// doubles the operand reads that bound an MMA of N = 64 (4 KB of A per 32 cycles of
// math).  15 taps x 4 groups of 16 channels = 60 MMAs per tile into one of two
// accumulators.  The output goes through swizzled shared memory to one TMA store per
// warp (whole 128-byte rows, clipped at the sequence end).  Bound by shared memory: 48
// cycles of operand reads per MMA, 2880 per tile, and the tile's own traffic through the
// same port; 2^20 symbols 107 us a layer (181 with unswizzled operands, descriptors built
// per MMA and one CTA barrier per tile), 2^14 symbols 7.2 us (8.7).
//
// 4 -> 64 layers (edge_in_kernel: the first layer from the features, and dJ/dh of the
// last one from dJ/dy): a feature row is 16 bytes of shared memory (4 values, 4 zeros), so
// row n of tap k's operand is row n + k and the whole operand is again a shifted start;
// the second half of K = 16 is a block of zeros that every operand shares through its
// leading offset.  15 MMAs per tile, one per tap: the sums of the mma.sync form.
// (Four taps per MMA on overlapping rows would take 4 MMAs, but rounds differently, and a
// flipped BF16 rounding of one hidden value travels through every later layer.)
//
// 64 -> 4 layer (edge_out_kernel): the taps go to the N dimension instead,
// P[m][4 t + c] = sum_ci h[m][ci] W[t][ci][c] (4 MMAs per tile, N = 64), and
// out[n][c] = sum_t P[n + t - 7][4 t + c] is 15 float4 additions per symbol.  A tile of
// 128 rows gives 114 symbols.  Both edge kernels are bound by the 128-byte rows they
// write or read and the latency of their phases; six (five with the mask of the layer below)
// and four CTAs share an SM.  A network of the two alone takes 92 us at 2^20 symbols (mma.sync
// 468; 114 where the 64 -> 4 kernel, with no residency stated, took 72 registers and spilled
// 100 bytes).
constexpr int TC_M = 128;                      // rows per tile (one MMA M)
constexpr int TC_ROWS = TC_M + 2 * HALF;       // 142 rows per TMA box
constexpr int TC_STAGES = 3;
constexpr int TC_A_BYTES = 18432;              // 144 rows x 128 B: stages stay 1024-byte aligned
constexpr int TC_A_TX = TC_ROWS * 128;         // bytes landed per stage
constexpr int TC_WCHUNKS = 3;                  // weights arrive in three pieces of 5 taps
constexpr int TC_W_TAP = CH * CH * 2;          // 8192
constexpr int TC_W_BYTES = KS * TC_W_TAP;      // 122880
constexpr int TC_OUT_BYTES = TC_M * 128;       // 16384 per staging buffer
constexpr int TC_OFF_A = TC_W_BYTES;
constexpr int TC_OFF_OUT = TC_OFF_A + TC_STAGES * TC_A_BYTES;
constexpr int TC_OFF_BIAS = TC_OFF_OUT + 2 * TC_OUT_BYTES;
constexpr int TC_OFF_BAR = TC_OFF_BIAS + CH * 4;
constexpr int TC_SMEM = TC_OFF_BAR + 256 + 1024;   // + slack to align the base to 1024 bytes
constexpr int TC_THREADS = 192;
constexpr unsigned TC_TMEM_COLS = 128;         // two accumulators of 64 FP32 columns
constexpr long long kTcWaitNs = 2000000000ll;  // bounded waits

constexpr int ED_W_BYTES = KS * CH * 16;       // weights of a 4 -> 64 layer: 16 bytes per tap and output
constexpr int ED_TILE = TC_M - 2 * HALF;       // 114 symbols per tile of the 64 -> 4 layer
constexpr unsigned ED_TMEM_COLS = 64;
// CTAs of an edge kernel that one SM holds, by shared memory (37 and 57 KB) and registers (64, 96
// and 100 of each thread): the persistent grids are one wave of them, a CTA more per SM would
// start when the others end and load the weights again.  (The occupancy calculator answers 1
// for kernels with tensor memory.)
constexpr int ED_IN_CTAS = 6, ED_DX_CTAS = 5, ED_OUT_CTAS = 4;

// Instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits
// 7-9 = 1, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22,
// M >> 4 at bits 24-28.
constexpr unsigned TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(CH >> 3) << 17) |
                              ((unsigned)(TC_M >> 4) << 24);

// Shared-memory matrix descriptor: start address, leading byte offset (no swizzle:
// between core matrices adjacent in K) and stride byte offset (between 8-row groups), all
// in 16-byte units; bits 46-47 = 1 (descriptor version); bits 61-63 the swizzle.
__device__ __forceinline__ unsigned long long tc_desc(unsigned saddr, unsigned lbo, unsigned sbo) {
  return (unsigned long long)((saddr >> 4) & 0x3FFFu) | ((unsigned long long)((lbo >> 4) & 0x3FFFu) << 16) |
         ((unsigned long long)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// 128-byte swizzle, rows of 128 bytes, 8-row groups 1024 bytes apart
__device__ __forceinline__ unsigned long long tc_desc_sw(unsigned saddr) {
  return tc_desc(saddr, 16u, 1024u) | (2ull << 61);
}

__device__ __forceinline__ long long tc_now() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait on an mbarrier phase; gives up past the deadline or once another role has.
__device__ __forceinline__ bool tc_wait(unsigned mbar, unsigned parity, long long deadline, volatile int *fail) {
  for (;;) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
    if (*fail) return false;
    if (tc_now() > deadline) {
      *fail = 1;
      return false;
    }
  }
}

// After a failure: a bounded wait (0.1 s) for a copy in flight.
__device__ __forceinline__ void tc_drain(unsigned mbar, unsigned parity) {
  int given_up = 0;
  tc_wait(mbar, parity, tc_now() + 100000000ll, &given_up);
}

__device__ __forceinline__ void tc_bar_init(unsigned mbar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void tc_arrive(unsigned mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void tc_expect(unsigned mbar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" :: "r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tc_commit(unsigned mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void tc_mma(unsigned d, unsigned long long a, unsigned long long b, bool acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      :: "r"(d), "l"(a), "l"(b), "r"(TC_IDESC), "r"(acc ? 1u : 0u)
      : "memory");
}
// 1-D bulk copy global -> shared (both 16-byte aligned)
__device__ __forceinline__ void tc_bulk(unsigned dst, const void *src, unsigned bytes, unsigned mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               :: "r"(dst), "l"(reinterpret_cast<unsigned long long>(src)), "r"(bytes), "r"(mbar)
               : "memory");
}
// Box of 64 channels at row y (negative or past-the-end rows read as zero)
__device__ __forceinline__ void tc_load_box(const CUtensorMap *tmap, unsigned dst, int64_t y, unsigned mbar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
      :: "r"(dst), "l"(reinterpret_cast<unsigned long long>(tmap)), "r"(0), "r"((int)y), "r"(mbar)
      : "memory");
}
// Box of 32 rows x 64 channels to row y >= 0 (rows past the end are not written)
__device__ __forceinline__ void tc_store_box(const CUtensorMap *tmap, unsigned src, int64_t y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];\n"
               :: "l"(reinterpret_cast<unsigned long long>(tmap)), "r"(0), "r"((int)y), "r"(src)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void tc_alloc(unsigned slot, unsigned cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" :: "r"(slot), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tc_dealloc(unsigned tmem, unsigned cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// Results of earlier kernels of the stream are visible after this (a launch with the
// programmatic attribute may start while the one before it drains).
__device__ __forceinline__ void tc_grid_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void tc_grid_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// A load of what the kernel directly in front writes: coherent, and kept behind the wait (__ldg
// would take it for read-only data of the whole kernel, whose life begins while that kernel
// still writes).  What was complete before the kernel in front started may go through __ldg.
__device__ __forceinline__ uint2 tc_load_behind_wait(const uint2 *p) {
  uint2 v;
  asm volatile("ld.global.v2.u32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void tc_ld32(unsigned taddr, float (&v)[32]) {
  unsigned r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// This warp's 32 accumulator rows (one per lane, 64 channels) -> bias + ReLU (EPI_RELU) or
// the mask of the layer below (EPI_MASK) -> BF16 -> the warp's 4 KB of swizzled staging.
template <int EPI>
__device__ __forceinline__ void tc_store_rows(unsigned taddr, const float *bias, const uint4 (&mk)[8], unsigned char *stage,
                                              int lane) {
#pragma unroll
  for (int hv = 0; hv < 2; ++hv) {
    float v[32];
    tc_ld32(taddr + 32 * hv, v);
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int p = 4 * hv + q;
      __nv_bfloat162 o[4];
      if constexpr (EPI == EPI_RELU) {
        const float4 b0 = *reinterpret_cast<const float4 *>(bias + p * 8), b1 = *reinterpret_cast<const float4 *>(bias + p * 8 + 4);
        o[0] = __floats2bfloat162_rn(fmaxf(v[8 * q] + b0.x, 0.f), fmaxf(v[8 * q + 1] + b0.y, 0.f));
        o[1] = __floats2bfloat162_rn(fmaxf(v[8 * q + 2] + b0.z, 0.f), fmaxf(v[8 * q + 3] + b0.w, 0.f));
        o[2] = __floats2bfloat162_rn(fmaxf(v[8 * q + 4] + b1.x, 0.f), fmaxf(v[8 * q + 5] + b1.y, 0.f));
        o[3] = __floats2bfloat162_rn(fmaxf(v[8 * q + 6] + b1.z, 0.f), fmaxf(v[8 * q + 7] + b1.w, 0.f));
      } else {
        const bf16 *m = reinterpret_cast<const bf16 *>(&mk[p]);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          o[e] = __floats2bfloat162_rn(__bfloat162float(m[2 * e]) > 0.f ? v[8 * q + 2 * e] : 0.f,
                                       __bfloat162float(m[2 * e + 1]) > 0.f ? v[8 * q + 2 * e + 1] : 0.f);
      }
      *reinterpret_cast<uint4 *>(stage + lane * 128 + ((p ^ (lane & 7)) << 4)) = *reinterpret_cast<uint4 *>(o);
    }
  }
}

// EPI_RELU: out = relu(acc + bias); EPI_MASK: out = acc * [mask > 0].
template <int EPI>
__global__ void __launch_bounds__(TC_THREADS, 1) conv_tc_kernel(const __grid_constant__ CUtensorMap tin,
                                                                const __grid_constant__ CUtensorMap tout,
                                                                const ConvArgs a, const void *__restrict__ wimg,
                                                                int *__restrict__ err) {
  extern __shared__ unsigned char tc_raw[];
  unsigned char *const sm = tc_raw + ((1024u - (smem_u32(tc_raw) & 1023u)) & 1023u);
  float *const bias = reinterpret_cast<float *>(sm + TC_OFF_BIAS);
  unsigned long long *const bars = reinterpret_cast<unsigned long long *>(sm + TC_OFF_BAR);
  unsigned *const tmem_slot = reinterpret_cast<unsigned *>(bars + 16);
  volatile int *const fail = reinterpret_cast<volatile int *>(bars + 17);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto bar_w = [&](int i) { return smem_u32(&bars[i]); };
  auto bar_full = [&](int s) { return smem_u32(&bars[3 + s]); };     // tile rows landed
  auto bar_free = [&](int s) { return smem_u32(&bars[6 + s]); };     // their MMAs done
  auto bar_acc = [&](int s) { return smem_u32(&bars[9 + s]); };      // accumulator complete
  auto bar_read = [&](int s) { return smem_u32(&bars[11 + s]); };    // accumulator read back
  if (warp == 1) tc_alloc(smem_u32(tmem_slot), TC_TMEM_COLS);
  if (tid == 0) {
    for (int i = 0; i < 11; ++i) tc_bar_init(smem_u32(&bars[i]), 1u);
    for (int s = 0; s < 2; ++s) tc_bar_init(bar_read(s), 4u);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    *fail = 0;
  }
  if (EPI == EPI_RELU && tid < CH) bias[tid] = a.bias[tid];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = *tmem_slot;
  const unsigned w_addr = smem_u32(sm), a_addr = smem_u32(sm + TC_OFF_A);
  const long long deadline = tc_now() + kTcWaitNs;
  const int64_t n_tiles = (a.K + TC_M - 1) / TC_M;
  const int64_t step = gridDim.x;
  if (warp == 0) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];\n" :: "l"(reinterpret_cast<unsigned long long>(&tin)) : "memory");
      // the weights come from before the kernel in front of this one: no wait
      for (int i = 0; i < TC_WCHUNKS; ++i) {
        tc_expect(bar_w(i), (unsigned)(TC_W_BYTES / TC_WCHUNKS));
        tc_bulk(w_addr + i * (TC_W_BYTES / TC_WCHUNKS),
                static_cast<const unsigned char *>(wimg) + i * (TC_W_BYTES / TC_WCHUNKS),
                (unsigned)(TC_W_BYTES / TC_WCHUNKS), bar_w(i));
      }
      tc_grid_wait();
      // the next kernel may start its prologue on SMs that run out of tiles; everything
      // before the kernel in front of this one is complete, so its weights are there
      tc_grid_trigger();
      int it = 0;
      for (int64_t tile = blockIdx.x; tile < n_tiles; tile += step, ++it) {
        const int s = it % TC_STAGES, round = it / TC_STAGES;
        if (round > 0 && !tc_wait(bar_free(s), (unsigned)((round - 1) & 1), deadline, fail)) break;
        tc_expect(bar_full(s), (unsigned)TC_A_TX);
        tc_load_box(&tin, a_addr + s * TC_A_BYTES, tile * TC_M - HALF, bar_full(s));
      }
      if (*fail) {   // no copy left in flight
        for (int i = 0; i < TC_WCHUNKS; ++i) tc_drain(bar_w(i), 0u);
        for (int i = max(0, it - TC_STAGES); i < it; ++i) tc_drain(bar_full(i % TC_STAGES), (unsigned)((i / TC_STAGES) & 1));
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const unsigned long long a0 = tc_desc_sw(a_addr), w0 = tc_desc_sw(w_addr);
      int it = 0;
      bool ok = true;
      for (int64_t tile = blockIdx.x; ok && tile < n_tiles; tile += step, ++it) {
        const int s = it % TC_STAGES, acc = it & 1;
        if (it >= 2) ok = tc_wait(bar_read(acc), (unsigned)(((it >> 1) - 1) & 1), deadline, fail);
        ok = ok && tc_wait(bar_full(s), (unsigned)((it / TC_STAGES) & 1), deadline, fail);
        if (!ok) break;
        tc_fence_after();
        const unsigned d = tmem + (unsigned)(acc * 64);
        // every descriptor is a base plus a constant (the address field counts 16 bytes): with
        // them built per MMA the one issuing thread is the bound (107 cycles per MMA
        // whatever N; 48, the operand reads, as written)
        const unsigned long long ad = a0 + (unsigned)(s * (TC_A_BYTES >> 4));
#pragma unroll
        for (int wc = 0; wc < TC_WCHUNKS; ++wc) {
          if (it == 0 && ok) ok = tc_wait(bar_w(wc), 0u, deadline, fail);
#pragma unroll
          for (int i = 0; i < KS / TC_WCHUNKS * 4; ++i) {
            const int k = wc * (KS / TC_WCHUNKS) + i / 4, kp = i % 4;
            tc_mma(d, ad + (unsigned)(k * 8 + kp * 2), w0 + (unsigned)(k * (TC_W_TAP >> 4) + kp * 2), (k | kp) != 0);
          }
        }
        tc_commit(bar_free(s));
        tc_commit(bar_acc(acc));
      }
    }
  } else {
    const int quad = warp & 3;                  // the TMEM lanes this warp may read
    tc_grid_wait();                             // the mask, and earlier readers of `out`
    int it = 0;
    for (int64_t tile = blockIdx.x; tile < n_tiles; tile += step, ++it) {
      const int acc = it & 1;
      const int64_t n0 = tile * TC_M + quad * 32;
      uint4 mk[8];
      if constexpr (EPI == EPI_MASK) {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.mask + (n0 + lane) * CH);
#pragma unroll
        for (int q = 0; q < 8; ++q) mk[q] = n0 + lane < a.K ? __ldg(&src[q]) : make_uint4(0u, 0u, 0u, 0u);
      }
      if (!tc_wait(bar_acc(acc), (unsigned)((it >> 1) & 1), deadline, fail)) break;
      tc_fence_after();
      unsigned char *stage = sm + TC_OFF_OUT + acc * TC_OUT_BYTES + quad * 4096;
      // the store that last read this staging buffer (two tiles ago) is done with it
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;\n" ::: "memory");
      __syncwarp();
      tc_store_rows<EPI>(tmem + ((unsigned)(quad * 32) << 16) + (unsigned)(acc * 64), bias, mk, stage, lane);
      tc_fence_before();
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        tc_arrive(bar_read(acc));
        if (n0 < a.K) tc_store_box(&tout, smem_u32(stage), n0);
        else asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *fail) atomicExch(err, 1);
  if (warp == 1) {
    tc_fence_after();
    tc_dealloc(tmem, TC_TMEM_COLS);
  }
}

// 4 -> 64: SRC_Z from the received symbols (two pols, FP32), else from BF16 rows of FEATP.
template <bool SRC_Z, int EPI>
__global__ void __launch_bounds__(TC_M) edge_in_kernel(const __grid_constant__ CUtensorMap tout, const ConvArgs a,
                                                       const void *__restrict__ wimg, int *__restrict__ err) {
  __shared__ alignas(1024) unsigned char stage[TC_OUT_BYTES];
  // feature rows, the weights [tap][out][8], and the zeros behind both
  __shared__ struct alignas(128) { uint4 y[TC_ROWS + 2]; unsigned char w[ED_W_BYTES]; uint4 zero[TC_M]; } op;
  __shared__ alignas(16) float bias[CH];
  __shared__ unsigned long long bars[2];
  __shared__ unsigned tmem_slot;
  __shared__ volatile int fail_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned bar_w = smem_u32(&bars[0]), bar_acc = smem_u32(&bars[1]);
  volatile int *const fail = &fail_s;
  if (warp == 0) tc_alloc(smem_u32(&tmem_slot), ED_TMEM_COLS);
  if (tid == 0) {
    tc_bar_init(bar_w, 1u);
    tc_bar_init(bar_acc, 1u);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    fail_s = 0;
    tc_expect(bar_w, (unsigned)ED_W_BYTES);
    tc_bulk(smem_u32(op.w), wimg, (unsigned)ED_W_BYTES, bar_w);
  }
  if (EPI == EPI_RELU && tid < CH) bias[tid] = a.bias[tid];
  op.zero[tid] = make_uint4(0u, 0u, 0u, 0u);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = tmem_slot;
  const long long deadline = tc_now() + kTcWaitNs;
  const int64_t n_tiles = (a.K + TC_M - 1) / TC_M;
  tc_grid_wait();
  if (tid == 0) tc_grid_trigger();
  if (a.zero) {
    for (int64_t i = (int64_t)blockIdx.x * TC_M + tid; i < a.n_zero; i += (int64_t)gridDim.x * TC_M) a.zero[i] = 0.f;
    if (blockIdx.x == 0 && tid == 0) *a.loss = 0.0;
  }
  const unsigned long long y0 = tc_desc(smem_u32(op.y), smem_u32(op.zero) - smem_u32(op.y), 128u);
  const unsigned long long w0 = tc_desc(smem_u32(op.w), smem_u32(op.zero) - smem_u32(op.w), 128u);
  // feature row of symbol n as four BF16 (zero outside the sequence)
  auto feat = [&](int64_t n) -> uint2 {
    if (n < 0 || n >= a.K) return make_uint2(0u, 0u);
    if constexpr (SRC_Z) {
      const float2 p0 = __ldg(&a.z[n]), p1 = __ldg(&a.z[a.z_stride + n]);
      const __nv_bfloat162 v0 = __floats2bfloat162_rn(p0.x, p0.y), v1 = __floats2bfloat162_rn(p1.x, p1.y);
      return make_uint2(*reinterpret_cast<const unsigned *>(&v0), *reinterpret_cast<const unsigned *>(&v1));
    } else {
      return tc_load_behind_wait(reinterpret_cast<const uint2 *>(a.in + n * FEATP));
    }
  };
  int it = 0;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
    const int64_t n0 = tile * TC_M;
    for (int m = tid; m < TC_ROWS; m += TC_M) {
      const uint2 v = feat(n0 - HALF + m);
      op.y[m] = make_uint4(v.x, v.y, 0u, 0u);
    }
    uint4 mk[8];
    const int64_t n = n0 + tid;
    if constexpr (EPI == EPI_MASK) {
      const uint4 *src = reinterpret_cast<const uint4 *>(a.mask + n * CH);
#pragma unroll
      for (int q = 0; q < 8; ++q) mk[q] = n < a.K ? __ldg(&src[q]) : make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    tc_fence_before();
    __syncthreads();   // rows written, the accumulator of the last tile read
    tc_fence_after();
    if (tid == 0 && (it > 0 || tc_wait(bar_w, 0u, deadline, fail))) {
      // one row (or tap) on in the address is 16 bytes less to the zeros
#pragma unroll
      for (int k = 0; k < KS; ++k)
        tc_mma(tmem, y0 + k - ((unsigned long long)k << 16), w0 + k * CH - ((unsigned long long)(k * CH) << 16), k != 0);
      tc_commit(bar_acc);
    }
    const bool ok = tc_wait(bar_acc, (unsigned)(it & 1), deadline, fail);
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
    __syncwarp();
    if (ok) {
      tc_fence_after();
      tc_store_rows<EPI>(tmem + ((unsigned)(warp * 32) << 16), bias, mk, stage + warp * 4096, lane);
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    __syncwarp();
    if (ok && lane == 0 && n0 + warp * 32 < a.K) tc_store_box(&tout, smem_u32(stage + warp * 4096), n0 + warp * 32);
    if (__syncthreads_or(!ok)) break;
  }
  if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
  if (tid == 0 && *fail) tc_drain(bar_w, 0u);
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *fail) atomicExch(err, 1);
  if (warp == 0) {
    tc_fence_after();
    tc_dealloc(tmem, ED_TMEM_COLS);
  }
}

// 64 -> 4 with the residual output and, in training, dJ/dy and the loss (EPI_LAST).
constexpr int ED_OUT_A = 0, ED_OUT_W = TC_OUT_BYTES, ED_OUT_P = ED_OUT_W + CH * CH * 2;
constexpr int ED_OUT_SMEM = ED_OUT_P + KS * TC_M * 16 + 1024;   // + slack to align the base
__global__ void __launch_bounds__(TC_M, ED_OUT_CTAS) edge_out_kernel(const __grid_constant__ CUtensorMap tin, const ConvArgs a,
                                                        const void *__restrict__ wimg, int *__restrict__ err) {
  extern __shared__ unsigned char tc_raw[];
  unsigned char *const sm = tc_raw + ((1024u - (smem_u32(tc_raw) & 1023u)) & 1023u);
  float4 *const P = reinterpret_cast<float4 *>(sm + ED_OUT_P);   // [tap][row]
  __shared__ unsigned long long bars[3];
  __shared__ unsigned tmem_slot;
  __shared__ volatile int fail_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned bar_w = smem_u32(&bars[0]), bar_full = smem_u32(&bars[1]), bar_acc = smem_u32(&bars[2]);
  const unsigned a_addr = smem_u32(sm + ED_OUT_A), w_addr = smem_u32(sm + ED_OUT_W);
  volatile int *const fail = &fail_s;
  if (warp == 0) tc_alloc(smem_u32(&tmem_slot), ED_TMEM_COLS);
  const int64_t n_tiles = (a.K + ED_TILE - 1) / ED_TILE;
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) tc_bar_init(smem_u32(&bars[i]), 1u);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    fail_s = 0;
    tc_expect(bar_w, (unsigned)(CH * CH * 2));
    tc_bulk(w_addr, wimg, (unsigned)(CH * CH * 2), bar_w);
  }
  float4 bias = make_float4(a.bias[0], a.bias[1], a.bias[2], a.bias[3]);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = tmem_slot;
  const long long deadline = tc_now() + kTcWaitNs;
  tc_grid_wait();
  if (tid == 0) tc_grid_trigger();
  if (tid == 0 && blockIdx.x < n_tiles) {
    tc_expect(bar_full, (unsigned)TC_OUT_BYTES);
    tc_load_box(&tin, a_addr, (int64_t)blockIdx.x * ED_TILE - HALF, bar_full);
  }
  double loss_part = 0.0;
  int it = 0;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
    const int64_t n0 = tile * ED_TILE, n = n0 + tid;
    const bool act = tid < ED_TILE && n < a.K;
    float2 z0 = make_float2(0.f, 0.f), z1 = z0, t0 = z0, t1 = z0;
    if (act) {
      z0 = a.z[n];   // y may be z itself
      z1 = a.z[a.z_stride + n];
      if (a.t) {
        t0 = __ldg(&a.t[n]);
        t1 = __ldg(&a.t[a.t_stride + n]);
      }
    }
    // the accumulator of the last tile is read (the barrier at the loop's end)
    if (tid == 0 && (it > 0 || tc_wait(bar_w, 0u, deadline, fail)) &&
        tc_wait(bar_full, (unsigned)(it & 1), deadline, fail)) {
      tc_fence_after();
#pragma unroll
      for (int kp = 0; kp < 4; ++kp) tc_mma(tmem, tc_desc_sw(a_addr + kp * 32), tc_desc_sw(w_addr + kp * 32), kp != 0);
      tc_commit(bar_acc);
    }
    const bool ok = tc_wait(bar_acc, (unsigned)(it & 1), deadline, fail);
    if (ok) {
      tc_fence_after();
      if (tid == 0 && tile + gridDim.x < n_tiles) {      // the rows are consumed: the next tile's
        tc_expect(bar_full, (unsigned)TC_OUT_BYTES);
        tc_load_box(&tin, a_addr, (tile + gridDim.x) * ED_TILE - HALF, bar_full);
      }
      __syncwarp();
#pragma unroll
      for (int hv = 0; hv < 2; ++hv) {
        float v[32];
        tc_ld32(tmem + ((unsigned)(warp * 32) << 16) + 32 * hv, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int t = 0; t < 8; ++t)
          if (8 * hv + t < KS) P[(8 * hv + t) * TC_M + tid] = make_float4(v[4 * t], v[4 * t + 1], v[4 * t + 2], v[4 * t + 3]);
      }
    }
    tc_fence_before();
    if (__syncthreads_or(!ok)) break;
    tc_fence_after();
    if (act) {
      float4 s = P[tid];
#pragma unroll
      for (int t = 1; t < KS; ++t) {
        const float4 v = P[t * TC_M + tid + t];
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
      }
      const float2 y0 = make_float2(z0.x + (s.x + bias.x), z0.y + (s.y + bias.y));
      const float2 y1 = make_float2(z1.x + (s.z + bias.z), z1.y + (s.w + bias.w));
      if (a.y) {
        a.y[n] = y0;
        a.y[a.y_stride + n] = y1;
      }
      if (a.t) {
        const float d0 = y0.x - t0.x, d1 = y0.y - t0.y, d2 = y1.x - t1.x, d3 = y1.y - t1.y;
        loss_part += ((double)d0 * d0 + (double)d1 * d1) + ((double)d2 * d2 + (double)d3 * d3);
        const __nv_bfloat162 o0 = __floats2bfloat162_rn(2.f * d0 * a.inv4k, 2.f * d1 * a.inv4k);
        const __nv_bfloat162 o1 = __floats2bfloat162_rn(2.f * d2 * a.inv4k, 2.f * d3 * a.inv4k);
        *reinterpret_cast<uint2 *>(a.dout + n * FEATP) =
            make_uint2(*reinterpret_cast<const unsigned *>(&o0), *reinterpret_cast<const unsigned *>(&o1));
      }
    }
    __syncthreads();   // P is rewritten by the next tile
  }
  if (tid == 0 && *fail) {
    tc_drain(bar_w, 0u);
    tc_drain(bar_full, (unsigned)(it & 1));
    tc_drain(bar_full, (unsigned)((it + 1) & 1));
  }
  if (a.t) {
    for (int o = 16; o >= 1; o >>= 1) loss_part += __shfl_xor_sync(0xffffffffu, loss_part, o);
    if (lane == 0 && loss_part != 0.0) atomicAdd(a.loss, loss_part * (double)a.inv4k);
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && *fail) atomicExch(err, 1);
  if (warp == 0) {
    tc_fence_after();
    tc_dealloc(tmem, ED_TMEM_COLS);
  }
}

// Where weight W[k][ci][co] of a layer sits in its tcgen05 operand images.
// 64 -> 64: [tap][co][ci] rows of 128 bytes, 16-byte pieces swizzled by row.
__device__ __forceinline__ int img_sw(int row, int col) { return row * CH + (((col >> 3) ^ (row & 7)) << 3) + (col & 7); }
__device__ __forceinline__ int img_tc_f(int k, int ci, int co) { return k * CH * CH + img_sw(co, ci); }
__device__ __forceinline__ int img_tc_b(int k, int ci, int co) { return (KS - 1 - k) * CH * CH + img_sw(ci, co); }
// 4 -> 64 (f: first layer, W[k][f][o]; b: reversed taps of the last layer, W[k][o][f]):
// [tap][o][8], the upper four zero.
__device__ __forceinline__ int img_in(int tap, int f, int o) { return (tap * CH + o) * 8 + f; }
// 64 -> 4: rows 4 tap + c of 64 input channels, swizzled.
__device__ __forceinline__ int img_out(int tap, int ci, int c) { return img_sw(4 * tap + c, ci); }

// tcgen05 images of one layer from the master W[k][ci][co] (padding stays zero).
__global__ void pack_tc_kernel(const float *__restrict__ W, int ci_true, int co_true, bf16 *__restrict__ f, bf16 *__restrict__ b) {
  const int n = KS * ci_true * co_true;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int co = i % co_true, ci = (i / co_true) % ci_true, k = i / (co_true * ci_true);
    const bf16 v = __float2bfloat16_rn(W[i]);
    if (ci_true == FEAT) {
      f[img_in(k, ci, co)] = v;
    } else if (co_true == FEAT) {
      f[img_out(k, ci, co)] = v;
      b[img_in(KS - 1 - k, co, ci)] = v;
    } else {
      f[img_tc_f(k, ci, co)] = v;
      b[img_tc_b(k, ci, co)] = v;
    }
  }
}

// ---------------------------------------------------------------- weight gradients on tcgen05
// All layers' weight and bias gradients in one launch, symbols as the reduction dimension
// (K = 16 symbols per MMA): both operands are read MN-major from the row tiles as they lie
// in memory ([n][64 channels], 128-byte swizzle), no transposition.
//
// Hidden layers: dW[k][ci][co] = sum_n in[n + k - 7][ci] dz[n][co].  An MMA of M = 128 rows
// takes two taps at once: the second 64 rows are the same input rows one symbol on, which
// is a leading offset of one row (128 bytes).  A CTA works through a chunk of tiles for two
// pairs of taps, D in 128 columns of tensor memory; the last pair's second half (tap 15,
// not a tap) reads a block of ones instead: db.
//
// Edge layers: D[4 t + f][o] = sum_n feat[n + t - 7][f] rows[n][o], with feat the input
// features and rows = dz for the first layer (dW[t][f][o] = D), feat = dJ/dy and rows = the
// last hidden layer's output for the last one (dW[14 - t][o][f] = D).  The features lie
// in shared memory as pairs (x[m], x[m+1]) of 16 bytes: a core matrix (8 of M = 2 taps, 8
// symbols) is 8 successive pairs, the next two taps are two pairs on.
//
// A CTA adds its part to the FP32 gradient with 16-byte atomics at the end.  Four layers of
// 2^14 symbols 19 us (four mma.sync launches 43).
constexpr int DW_STAGES = 2;
constexpr int DW_PAIRS = 2;                          // tap pairs per CTA of a hidden layer
constexpr int DW_GROUPS = (KS + 1) / (2 * DW_PAIRS); // CTAs per chunk
constexpr int DW_Z_BYTES = TC_M * 128;
constexpr int DW_STAGE_BYTES = TC_A_BYTES + DW_Z_BYTES;
constexpr int DW_Y_ROWS = TC_M + 32;                 // pairs that an edge tile's operand spans (rows past tap 14: unused)
constexpr int DW_OFF_ONES = DW_STAGES * DW_STAGE_BYTES;
constexpr int DW_ONES_BYTES = 2304;                  // 16 x 128 bytes and one more row group (core matrices 128 apart)
constexpr int DW_OFF_Y = DW_OFF_ONES + DW_ONES_BYTES;
constexpr int DW_OFF_BAR = DW_OFF_Y + DW_Y_ROWS * 16;
constexpr int DW_SMEM = DW_OFF_BAR + 64 + 1024;
constexpr unsigned DW_TMEM_COLS = 128;
// MN-major A and B (bits 15, 16)
constexpr unsigned DW_IDESC = TC_IDESC | (1u << 15) | (1u << 16);
constexpr int DW_MAX_LAYERS = 8;

struct DwTcLayer {
  CUtensorMap x, z;          // hidden: input rows (142-row boxes), dz rows (128); edges: rows in z
  const float2 *sym;         // first layer: the received symbols
  int64_t sym_stride;
  const bf16 *feat;          // last layer: dJ/dy rows of FEATP
  float *dw, *db;
  int first_block;           // of this layer in the grid
  int chunk_tiles;
};
struct DwTcArgs {
  DwTcLayer l[DW_MAX_LAYERS];
  int L;
  int64_t K;
};

__device__ __forceinline__ void dw_mma(unsigned d, unsigned long long a, unsigned long long b, bool acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      :: "r"(d), "l"(a), "l"(b), "r"(DW_IDESC), "r"(acc ? 1u : 0u)
      : "memory");
}

__global__ void __launch_bounds__(TC_M) dw_tc_kernel(const __grid_constant__ DwTcArgs a, int *__restrict__ err) {
  extern __shared__ unsigned char tc_raw[];
  unsigned char *const sm = tc_raw + ((1024u - (smem_u32(tc_raw) & 1023u)) & 1023u);
  unsigned long long *const bars = reinterpret_cast<unsigned long long *>(sm + DW_OFF_BAR);
  unsigned *const tmem_slot = reinterpret_cast<unsigned *>(bars + 5);
  volatile int *const fail = reinterpret_cast<volatile int *>(bars + 6);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto bar_full = [&](int s) { return smem_u32(&bars[s]); };
  auto bar_free = [&](int s) { return smem_u32(&bars[DW_STAGES + s]); };
  const unsigned bar_done = smem_u32(&bars[2 * DW_STAGES]);
  if (warp == 0) tc_alloc(smem_u32(tmem_slot), DW_TMEM_COLS);
  if (tid == 0) {
    for (int i = 0; i < 2 * DW_STAGES + 1; ++i) tc_bar_init(smem_u32(&bars[i]), 1u);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    *fail = 0;
  }
  for (int i = tid; i < DW_ONES_BYTES / 16; i += TC_M)
    *reinterpret_cast<uint4 *>(sm + DW_OFF_ONES + i * 16) = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = *tmem_slot;
  const long long deadline = tc_now() + kTcWaitNs;
  int li = 0;
  while (li + 1 < a.L && (int)blockIdx.x >= a.l[li + 1].first_block) ++li;
  const DwTcLayer &y = a.l[li];
  const bool first = li == 0, last = li == a.L - 1, edge = first || last;
  const int rel = (int)blockIdx.x - y.first_block;
  const int group = edge ? 0 : rel % DW_GROUPS;
  const int64_t n_tiles = (a.K + TC_M - 1) / TC_M;
  const int64_t t0 = (int64_t)(edge ? rel : rel / DW_GROUPS) * y.chunk_tiles;
  const int nt = (int)min((int64_t)y.chunk_tiles, n_tiles - t0);   // >= 1
  tc_grid_wait();
  if (tid == 0) tc_grid_trigger();
  auto load = [&](int i) {                            // tile i of this CTA into its stage
    const int s = i % DW_STAGES;
    const unsigned st = smem_u32(sm + s * DW_STAGE_BYTES);
    const int64_t n0 = (t0 + i) * TC_M;
    tc_expect(bar_full(s), (unsigned)((edge ? 0 : TC_A_TX) + DW_Z_BYTES));
    if (!edge) tc_load_box(&y.x, st, n0 - HALF, bar_full(s));
    tc_load_box(&y.z, st + TC_A_BYTES, n0, bar_full(s));
  };
  if (tid == 0)
    for (int i = 0; i < min(nt, DW_STAGES); ++i) load(i);
  const unsigned ones = smem_u32(sm + DW_OFF_ONES);
  float4 dbp = make_float4(0.f, 0.f, 0.f, 0.f);       // last layer: this thread's part of db
  bool ok = true;
  int it = 0;
  for (; it < nt; ++it) {
    if (!edge && !ok) break;                          // thread 0 alone waits: the others come to the last wait
    const int s = it % DW_STAGES;
    const unsigned st = smem_u32(sm + s * DW_STAGE_BYTES);
    if (edge) {
      // the pairs of this tile (the MMAs of the last one are done: every thread waited below)
      uint2 *const ysm = reinterpret_cast<uint2 *>(sm + DW_OFF_Y);
      const int64_t n0 = (t0 + it) * TC_M;
      for (int m = tid; m <= DW_Y_ROWS; m += TC_M) {
        const int64_t n = n0 - HALF + m;
        uint2 v = make_uint2(0u, 0u);
        if (m < TC_ROWS && n >= 0 && n < a.K) {
          if (first) {
            const float2 p0 = __ldg(&y.sym[n]), p1 = __ldg(&y.sym[y.sym_stride + n]);
            const __nv_bfloat162 v0 = __floats2bfloat162_rn(p0.x, p0.y), v1 = __floats2bfloat162_rn(p1.x, p1.y);
            v = make_uint2(*reinterpret_cast<const unsigned *>(&v0), *reinterpret_cast<const unsigned *>(&v1));
          } else {
            v = __ldg(reinterpret_cast<const uint2 *>(y.feat + n * FEATP));
            if (m >= HALF && m < HALF + TC_M) {       // a symbol of this tile
              const __nv_bfloat162 v0 = *reinterpret_cast<const __nv_bfloat162 *>(&v.x);
              const __nv_bfloat162 v1 = *reinterpret_cast<const __nv_bfloat162 *>(&v.y);
              dbp.x += __bfloat162float(v0.x);
              dbp.y += __bfloat162float(v0.y);
              dbp.z += __bfloat162float(v1.x);
              dbp.w += __bfloat162float(v1.y);
            }
          }
        }
        if (m < DW_Y_ROWS) ysm[2 * m] = v;
        if (m > 0) ysm[2 * m - 1] = v;
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      if (__syncthreads_or(!ok)) break;
    }
    if (tid == 0) {
      ok = tc_wait(bar_full(s), (unsigned)((it / DW_STAGES) & 1), deadline, fail);
      if (ok) {
        tc_fence_after();
        const unsigned long long zd = tc_desc(st + TC_A_BYTES, 16u, 1024u) | (2ull << 61);
        if (edge) {
          // pairs: two taps on = 32 bytes along M, 8 symbols on = 128 bytes along K
          const unsigned long long yd = tc_desc(smem_u32(sm + DW_OFF_Y), 128u, 32u);
          const unsigned long long od = tc_desc(ones, 128u, 128u);
#pragma unroll
          for (int q = 0; q < TC_M / 16; ++q) {
            dw_mma(tmem, yd + q * 16, zd + q * 128, (it | q) != 0);
            if (first) dw_mma(tmem + 64, od, zd + q * 128, (it | q) != 0);
          }
        } else {
#pragma unroll
          for (int pr = 0; pr < DW_PAIRS; ++pr) {
            const unsigned row = st + (unsigned)(2 * (group * DW_PAIRS + pr)) * 128u;
            const bool db = group * DW_PAIRS + pr == (KS - 1) / 2;      // tap 14 and the ones
            const unsigned long long xd = tc_desc(row, db ? ones - row : 128u, 1024u) | (2ull << 61);
            const unsigned long long adv = db ? 128ull - (128ull << 16) : 128ull;   // 16 rows on; the ones stay
#pragma unroll
            for (int q = 0; q < TC_M / 16; ++q) dw_mma(tmem + 64 * pr, xd + q * adv, zd + q * 128, (it | q) != 0);
          }
        }
        tc_commit(bar_free(s));
      }
    }
    // the stage is refilled, and the pairs rewritten, once the MMAs are done
    if (edge || it + DW_STAGES < nt) {
      if (edge || tid == 0) {
        if (ok) ok = tc_wait(bar_free(s), (unsigned)((it / DW_STAGES) & 1), deadline, fail);
        if (ok && tid == 0 && it + DW_STAGES < nt) load(it + DW_STAGES);
      }
    }
  }
  if (tid == 0 && ok) tc_commit(bar_done);            // every MMA
  if (ok) ok = tc_wait(bar_done, 0u, deadline, fail);
  if (*fail && tid == 0) {
    for (int i = max(0, it - 1); i < min(nt, it + DW_STAGES); ++i) tc_drain(bar_full(i % DW_STAGES), (unsigned)((i / DW_STAGES) & 1));
  }
  tc_fence_after();
  if (!__syncthreads_or(!ok)) {
    const unsigned ta = tmem + ((unsigned)(warp * 32) << 16);
    const int r = tid;                                // accumulator row
#pragma unroll 1
    for (int h = 0; h < 4; ++h) {                     // 32 columns at a time
      float v[32];
      tc_ld32(ta + 32 * h, v);
      asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
      const int c0 = (h & 1) * 32;
      float *dst = nullptr;
      if (!edge) {
        const int pr = group * DW_PAIRS + (h >> 1), k = 2 * pr + (r >> 6), ci = r & 63;
        if (k < KS) dst = y.dw + ((size_t)k * CH + ci) * CH + c0;
        else if (ci == 0) dst = y.db + c0;
      } else if (first) {
        if (h < 2 && r < KS * FEAT) dst = y.dw + (size_t)r * CH + c0;
        else if (h >= 2 && r == 0) dst = y.db + c0;
      }
      if (dst) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          atomicAdd(reinterpret_cast<float4 *>(dst) + q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
      }
      if (last && h < 2) {
        // dW[14 - t][o][f] of row 4 t + f: four lanes hold the four f of one t
#pragma unroll
        for (int q = 0; q < 32; ++q) {
          const float v1 = __shfl_down_sync(0xffffffffu, v[q], 1), v2 = __shfl_down_sync(0xffffffffu, v[q], 2),
                      v3 = __shfl_down_sync(0xffffffffu, v[q], 3);
          if (r < KS * FEAT && (lane & 3) == 0)
            atomicAdd(reinterpret_cast<float4 *>(y.dw + ((size_t)(KS - 1 - (r >> 2)) * CH + c0 + q) * FEAT),
                      make_float4(v[q], v1, v2, v3));
        }
      }
    }
    if (last) {
      for (int o = 16; o >= 1; o >>= 1) {
        dbp.x += __shfl_xor_sync(0xffffffffu, dbp.x, o);
        dbp.y += __shfl_xor_sync(0xffffffffu, dbp.y, o);
        dbp.z += __shfl_xor_sync(0xffffffffu, dbp.z, o);
        dbp.w += __shfl_xor_sync(0xffffffffu, dbp.w, o);
      }
      if (lane == 0) atomicAdd(reinterpret_cast<float4 *>(y.db), dbp);
    }
  } else if (tid == 0) {
    atomicExch(err, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tc_dealloc(tmem, DW_TMEM_COLS);
  }
}

struct DwArgs {
  const bf16 *in;     // layer input [K][CIN]
  const bf16 *dz;     // dJ/d(pre-activation) [K][COUT]
  int64_t K, chunk;
  float *dw;          // master layout [15][ci_true][co_true] (accumulated)
  float *db;          // [co_true] (accumulated)
  int ci_true, co_true;
};

// 16-byte asynchronous global -> shared copy; src_bytes 0 zero-fills (nothing is read).
__device__ __forceinline__ void dw_cp16(void *dst, const void *src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes)
               : "memory");
}

template <int CIN, int COUT>
constexpr int dw_smem_bytes() {
  return 2 * ((TM + 2 * HALF) * (CIN + 8) + TM * (COUT + 8)) * (int)sizeof(bf16);
}

// dW[k][ci][co] += sum_n in[n + k - 7][ci] dz[n][co] over this CTA's symbols,
// taps TG blockIdx.y .. + TG - 1; CTAs with blockIdx.y == 0 also add db.  The
// input and gradient tiles of TM symbols are double-buffered in dynamic shared
// memory: the copies of tile i + 1 fly while the MMAs of tile i run.
template <int CIN, int COUT>
__global__ void __launch_bounds__(kThreads) dw_kernel(const DwArgs a) {
  constexpr int CPX = CIN + 8, CPZ = COUT + 8;
  constexpr int XT = (TM + 2 * HALF) * CPX, ZT = TM * CPZ;
  extern __shared__ __align__(16) unsigned char dw_smem[];
  bf16 *const Xb = reinterpret_cast<bf16 *>(dw_smem);     // [2][XT]
  bf16 *const Zb = Xb + 2 * XT;                            // [2][ZT]
  constexpr int CB = CIN / 16, CT = COUT / 8, WPB = 8 / CB, TPW = CT / WPB;
  static_assert(TPW >= 1 && CB * WPB == 8, "warp layout");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = lane >> 2, tig = lane & 3;
  const int cb = warp % CB, tile0 = (warp / CB) * TPW;
  const int tap0 = blockIdx.y * TG;
  const int64_t s0 = (int64_t)blockIdx.x * a.chunk, s1 = min(a.K, s0 + a.chunk);
  float acc[TG][TPW][4];
#pragma unroll
  for (int t = 0; t < TG; ++t)
#pragma unroll
    for (int j = 0; j < TPW; ++j) acc[t][j][0] = acc[t][j][1] = acc[t][j][2] = acc[t][j][3] = 0.f;
  float dbp = 0.f;
  // tile at symbol n0 into buffer `buf`: input rows n0 - 7 .. n0 + TM + 6, gradient rows n0 .. n0 + TM - 1
  auto issue = [&](int buf, int64_t n0) {
    bf16 *Xs = Xb + buf * XT, *Zs = Zb + buf * ZT;
    for (int i = threadIdx.x; i < (TM + 2 * HALF) * (CIN / 8); i += kThreads) {
      const int r = i / (CIN / 8), p = i % (CIN / 8);
      const int64_t n = n0 - HALF + r;
      const bool ok = n >= 0 && n < a.K;
      dw_cp16(Xs + r * CPX + p * 8, ok ? (const void *)(a.in + n * CIN + p * 8) : (const void *)a.in, ok ? 16 : 0);
    }
    for (int i = threadIdx.x; i < TM * (COUT / 8); i += kThreads) {
      const int r = i / (COUT / 8), p = i % (COUT / 8);
      const int64_t n = n0 + r;
      const bool ok = n < s1;
      dw_cp16(Zs + r * CPZ + p * 8, ok ? (const void *)(a.dz + n * COUT + p * 8) : (const void *)a.dz, ok ? 16 : 0);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  // ldmatrix.trans lanes: matrix j = lane / 8
  const int ax_row = (lane & 7) + ((lane >> 4) & 1) * 8, ax_col = cb * 16 + ((lane >> 3) & 1) * 8;
  const int bz_row = (lane & 7) + ((lane >> 3) & 1) * 8;
  if (s0 < s1) issue(0, s0);
  int it = 0;
  for (int64_t n0 = s0; n0 < s1; n0 += TM, ++it) {
    if (n0 + TM < s1) {
      issue((it + 1) & 1, n0 + TM);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    const bf16 *Xs = Xb + (it & 1) * XT, *Zs = Zb + (it & 1) * ZT;
#pragma unroll 1
    for (int s = 0; s < TM / 16; ++s) {
      unsigned b[TPW][2];
#pragma unroll
      for (int j = 0; j < TPW; ++j)
        ldsm_x2_t(smem_u32(Zs + (16 * s + bz_row) * CPZ + (tile0 + j) * 8), b[j][0], b[j][1]);
#pragma unroll
      for (int t = 0; t < TG; ++t) {
        unsigned a0, a1, a2, a3;
        ldsm_x4_t(smem_u32(Xs + (16 * s + tap0 + t + ax_row) * CPX + ax_col), a0, a1, a2, a3);
#pragma unroll
        for (int j = 0; j < TPW; ++j) mma(acc[t][j], a0, a1, a2, a3, b[j][0], b[j][1]);
      }
    }
    if (blockIdx.y == 0 && threadIdx.x < COUT) {
      for (int r = 0; r < TM; ++r) dbp += __bfloat162float(Zs[r * CPZ + threadIdx.x]);
    }
    __syncthreads();  // this buffer is refilled by the copies issued in the next iteration
  }
#pragma unroll
  for (int t = 0; t < TG; ++t) {
    const int k = tap0 + t;
#pragma unroll
    for (int j = 0; j < TPW; ++j) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int ci = cb * 16 + group + 8 * h;
        const int co = (tile0 + j) * 8 + 2 * tig;
        if (ci < a.ci_true) {
          float *d = &a.dw[((size_t)k * a.ci_true + ci) * a.co_true + co];
          if (co + 1 < a.co_true && ((uintptr_t)d & 7) == 0) {
            // both columns in one 8-byte vector atomic
            atomicAdd(reinterpret_cast<float2 *>(d), make_float2(acc[t][j][2 * h], acc[t][j][2 * h + 1]));
          } else {
            if (co < a.co_true) atomicAdd(d, acc[t][j][2 * h]);
            if (co + 1 < a.co_true) atomicAdd(d + 1, acc[t][j][2 * h + 1]);
          }
        }
      }
    }
  }
  if (blockIdx.y == 0 && threadIdx.x < a.co_true && dbp != 0.f) atomicAdd(&a.db[threadIdx.x], dbp);
}

__global__ void features_kernel(const float2 *__restrict__ z, int64_t z_stride, int64_t K, bf16 *__restrict__ x) {
  for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < K; n += (int64_t)gridDim.x * blockDim.x) {
    const float2 p0 = z[n], p1 = z[z_stride + n];
    __nv_bfloat162 v[8];
    v[0] = __floats2bfloat162_rn(p0.x, p0.y);
    v[1] = __floats2bfloat162_rn(p1.x, p1.y);
    for (int i = 2; i < 8; ++i) v[i] = __floats2bfloat162_rn(0.f, 0.f);
    uint4 *dst = reinterpret_cast<uint4 *>(x + n * FEATP);
    dst[0] = *reinterpret_cast<uint4 *>(&v[0]);
    dst[1] = *reinterpret_cast<uint4 *>(&v[4]);
  }
}


// Adam on every parameter with the packed BF16 copies of each updated weight
// written in the same pass (one launch per training step).
struct PackLayer {
  long long off_w, off_b;
  int ci, co, cinp, coutp, copb;
  bf16 *wf, *wb, *wtc_f, *wtc_b;
};
struct PackTable {
  PackLayer l[8];
  int L;
};

__global__ void adam_pack_kernel(const PackTable tab, float *__restrict__ P, const float *__restrict__ G,
                                 float *__restrict__ M, float *__restrict__ V, int64_t n, float lr, float c1, float c2) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float g = G[i];
    const float m = b1 * M[i] + (1.f - b1) * g;
    const float v = b2 * V[i] + (1.f - b2) * g * g;
    M[i] = m;
    V[i] = v;
    const float w = P[i] - lr * (m / c1) / (sqrtf(v / c2) + eps);
    P[i] = w;
    int l = 0;
    while (l + 1 < tab.L && i >= tab.l[l + 1].off_w) ++l;
    const PackLayer &y = tab.l[l];
    if (i >= y.off_b) continue;                  // a bias: read from P directly
    const int r = (int)(i - y.off_w);
    const int co = r % y.co, ci = (r / y.co) % y.ci, k = r / (y.co * y.ci);
    const bf16 wv = __float2bfloat16_rn(w);
    y.wf[((size_t)k * y.coutp + co) * y.cinp + ci] = wv;
    if (y.wb) y.wb[((size_t)(KS - 1 - k) * y.ci + ci) * y.copb + co] = wv;
    if (y.ci == FEAT) {
      y.wtc_f[img_in(k, ci, co)] = wv;
    } else if (y.co == FEAT) {
      y.wtc_f[img_out(k, ci, co)] = wv;
      y.wtc_b[img_in(KS - 1 - k, co, ci)] = wv;
    } else {
      y.wtc_f[img_tc_f(k, ci, co)] = wv;
      y.wtc_b[img_tc_b(k, ci, co)] = wv;
    }
  }
}

// Packed BF16 weights of one layer from the master W[k][ci][co]:
//   wf[k][co][ci]  (forward, COUTP x CINP, zero padded)
//   wb[j][ci][co]  = W[14 - j][ci][co] (input gradient, ci x COPB, zero padded)
__global__ void pack_kernel(const float *__restrict__ W, int ci_true, int co_true, bf16 *__restrict__ wf, int cinp,
                            int coutp, bf16 *__restrict__ wb, int copb) {
  const int nf = KS * coutp * cinp;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nf; i += gridDim.x * blockDim.x) {
    const int k = i / (coutp * cinp), co = (i / cinp) % coutp, ci = i % cinp;
    const float v = (ci < ci_true && co < co_true) ? W[((size_t)k * ci_true + ci) * co_true + co] : 0.f;
    wf[i] = __float2bfloat16_rn(v);
  }
  if (!wb) return;
  const int nb = KS * ci_true * copb;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    const int j = i / (ci_true * copb), ci = (i / copb) % ci_true, co = i % copb;
    const float v = co < co_true ? W[((size_t)(KS - 1 - j) * ci_true + ci) * co_true + co] : 0.f;
    wb[i] = __float2bfloat16_rn(v);
  }
}

__global__ void add_kernel(double *acc, const double *v) { *acc += *v; }

template <int CIN, int COUT, int EPI>
size_t conv_smem() {
  return (size_t)(KS * COUT + TM + 2 * HALF) * (CIN + 8) * sizeof(bf16);
}

template <int CIN, int COUT, int EPI>
cudaError_t conv_prepare() {
  return cudaFuncSetAttribute(conv_kernel<CIN, COUT, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)conv_smem<CIN, COUT, EPI>());
}

}  // namespace

struct rx_cnn {
  int L = 0;
  int64_t Kmax = 0, n_params = 0;
  std::vector<int> ci, co;             // true dims per layer
  std::vector<int64_t> off_w, off_b;   // offsets into the flat parameters
  cudaStream_t stream = nullptr;
  int sms = 0;
  float *P = nullptr, *G = nullptr, *M = nullptr, *V = nullptr;
  std::vector<bf16 *> wf, wb;
  std::vector<bf16 *> wtc_f, wtc_b;    // tcgen05 operand images (wtc_b: none for the first layer)
  bool use_tc = true;
  int *err = nullptr;                  // sticky device error word (bounded waits), in res
  bf16 *x0 = nullptr, *dout = nullptr;
  std::vector<bf16 *> dz;              // dJ/d(pre-activation) of layers 0 .. L-2
  bool dz_shared = false;              // ... two buffers in turn (the device had no room for all)
  std::vector<bf16 *> h;               // hidden outputs h_1 .. h_{L-1}
  struct Result { double loss; int err, pad; };
  Result *res = nullptr, *h_res = nullptr;   // device, and the pinned copy that grads reads back
  double *loss = nullptr;              // in res
  int64_t step = 0;
  std::vector<void *> allocs;
  std::string msg;
  // profiling: event pairs around launches of each kind (RX_CNN_K_*)
  bool profile = false;
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used = 0;
  std::vector<std::pair<int, size_t>> ev_pending;
  double kind_ms[RX_CNN_KINDS] = {0, 0, 0, 0, 0};
  int64_t kind_launches[RX_CNN_KINDS] = {0, 0, 0, 0, 0};
};

namespace {

rx_status cfail(rx_cnn *c, rx_status s, const std::string &m) {
  if (c) c->msg = m;
  return s;
}

#define CX_CUDA(call, where)                                                                   \
  do {                                                                                         \
    cudaError_t e_ = (call);                                                                   \
    if (e_ != cudaSuccess) return cfail(c, RX_ECUDA, std::string(where) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <class Tp>
rx_status calloc_dev(rx_cnn *c, Tp **p, size_t count) {
  void *q = nullptr;
  if (cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(Tp)) != cudaSuccess) {
    cudaGetLastError();
    return cfail(c, RX_ENOMEM, "device allocation failed");
  }
  c->allocs.push_back(q);
  *p = static_cast<Tp *>(q);
  return RX_OK;
}

void release(rx_cnn *c) {
  if (c->h_res) cudaFreeHost(c->h_res);
  c->h_res = nullptr;
  for (void *p : c->allocs) cudaFree(p);
  c->allocs.clear();
}

// Event pair around one launch of a kind, when profiling.
struct KTimer {
  rx_cnn *c;
  int kind;
  size_t idx = (size_t)-1;
  KTimer(rx_cnn *cc, int k) : c(cc), kind(k) {
    c->kind_launches[kind] += 1;
    if (!c->profile) return;
    while (c->ev_pool.size() < c->ev_used + 2) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return;
      c->ev_pool.push_back(e);
    }
    idx = c->ev_used;
    c->ev_used += 2;
    cudaEventRecord(c->ev_pool[idx], c->stream);
  }
  ~KTimer() {
    if (idx == (size_t)-1) return;
    cudaEventRecord(c->ev_pool[idx + 1], c->stream);
    c->ev_pending.push_back({kind, idx});
  }
};

int conv_grid(const rx_cnn *c, int64_t K) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((K + TM - 1) / TM, c->sms));
}

template <int CIN, int COUT, int EPI>
cudaError_t launch_conv(rx_cnn *c, const ConvArgs &a) {
  KTimer tm(c, EPI == EPI_MASK ? RX_CNN_K_DX : (CIN == CH && COUT == CH ? RX_CNN_K_FWD_HIDDEN : RX_CNN_K_FWD_EDGE));
  conv_kernel<CIN, COUT, EPI><<<conv_grid(c, a.K), kThreads, conv_smem<CIN, COUT, EPI>(), c->stream>>>(a);
  return cudaGetLastError();
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime.
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
  // (initialised once whichever threads come first)
  static const EncodeTiledFn fn = []() -> EncodeTiledFn {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(p);
    cudaGetLastError();
    return nullptr;
  }();
  return fn;
}

// Tensor map of [K][64] BF16 rows in boxes of `rows` x 64 channels, 128-byte swizzle.
cudaError_t row_map(CUtensorMap *m, const bf16 *p, int64_t K, unsigned rows) {
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {(cuuint64_t)CH, (cuuint64_t)K};
  const cuuint64_t strides[1] = {(cuuint64_t)CH * sizeof(bf16)};
  const cuuint32_t box[2] = {(cuuint32_t)CH, rows};
  const cuuint32_t estr[2] = {1u, 1u};
  auto encode = [&]() {
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(p), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  };
  CUresult r = encode();
  if (r == CUDA_ERROR_INVALID_CONTEXT || r == CUDA_ERROR_NOT_INITIALIZED) {
    // a host thread whose first CUDA call this is: the driver, unlike the runtime, does not bind
    // the device's context by itself
    const cudaError_t e = cudaFree(nullptr);
    if (e != cudaSuccess) return e;
    r = encode();
  }
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// A launch that may start its prologue while the kernel in front of it drains (pdl).
template <class... KArgs, class... Args>
cudaError_t launch_tc(void (*fn)(KArgs...), int grid, int threads, int smem, cudaStream_t s, bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

int tc_grid(const rx_cnn *c, int64_t K, int tile, int per_sm) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((K + tile - 1) / tile, (int64_t)c->sms * per_sm));
}

template <int EPI>
cudaError_t launch_conv_tc(rx_cnn *c, const ConvArgs &a, const bf16 *img, bool pdl) {
  KTimer tm(c, EPI == EPI_MASK ? RX_CNN_K_DX : RX_CNN_K_FWD_HIDDEN);
  CUtensorMap tin, tout;
  cudaError_t e = row_map(&tin, a.in, a.K, TC_ROWS);
  if (e == cudaSuccess) e = row_map(&tout, a.out, a.K, 32);
  if (e != cudaSuccess) return e;
  return launch_tc(conv_tc_kernel<EPI>, tc_grid(c, a.K, TC_M, 1), TC_THREADS, TC_SMEM, c->stream, pdl, tin, tout, a,
                   (const void *)img, c->err);
}

template <bool SRC_Z, int EPI>
cudaError_t launch_edge_in(rx_cnn *c, const ConvArgs &a, const bf16 *img, bool pdl) {
  KTimer tm(c, EPI == EPI_MASK ? RX_CNN_K_DX : RX_CNN_K_FWD_EDGE);
  CUtensorMap tout;
  const cudaError_t e = row_map(&tout, a.out, a.K, 32);
  if (e != cudaSuccess) return e;
  return launch_tc(edge_in_kernel<SRC_Z, EPI>, tc_grid(c, a.K, TC_M, EPI == EPI_MASK ? ED_DX_CTAS : ED_IN_CTAS), TC_M, 0, c->stream, pdl, tout, a,
                   (const void *)img, c->err);
}

cudaError_t launch_edge_out(rx_cnn *c, const ConvArgs &a, const bf16 *img, bool pdl) {
  KTimer tm(c, RX_CNN_K_FWD_EDGE);
  CUtensorMap tin;
  const cudaError_t e = row_map(&tin, a.in, a.K, TC_M);
  if (e != cudaSuccess) return e;
  return launch_tc(edge_out_kernel, tc_grid(c, a.K, ED_TILE, ED_OUT_CTAS), TC_M, ED_OUT_SMEM, c->stream, pdl, tin, a,
                   (const void *)img, c->err);
}

template <int CIN, int COUT>
cudaError_t launch_dw(rx_cnn *c, const bf16 *in, const bf16 *dz, int64_t K, int l, float *G) {
  KTimer tm(c, RX_CNN_K_DW);
  DwArgs a;
  a.in = in;
  a.dz = dz;
  a.K = K;
  // about one CTA per SM: each partial dW costs 15 x ci x co / TG x ... atomics, so fewer,
  // longer CTAs (their tile copies double-buffered) beat more, shorter ones
  const int64_t want = std::max<int64_t>(1, (int64_t)c->sms / (KS / TG));
  a.chunk = ((K + want - 1) / want + TM - 1) / TM * TM;
  a.dw = G + c->off_w[l];
  a.db = G + c->off_b[l];
  a.ci_true = c->ci[l];
  a.co_true = c->co[l];
  dim3 grid((unsigned)((K + a.chunk - 1) / a.chunk), KS / TG);
  constexpr int smem = dw_smem_bytes<CIN, COUT>();
  cudaFuncSetAttribute(dw_kernel<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  dw_kernel<CIN, COUT><<<grid, kThreads, smem, c->stream>>>(a);
  return cudaGetLastError();
}

// Gradients of the layers [l0, l1) into G (zeroed before the forward pass) from the stored rows.
// A launch of all of them comes behind the input gradients and may overlap the last of those; one of
// a single layer may follow the kernel that wrote dJ/dy, which it reads through __ldg.
cudaError_t launch_dw_tc(rx_cnn *c, const float2 *z, int64_t zs, int64_t K, float *G, int l0, int l1) {
  KTimer tm(c, RX_CNN_K_DW);
  DwTcArgs a;
  memset(&a, 0, sizeof(a));
  a.L = c->L;
  a.K = K;
  const int64_t n_tiles = (K + TC_M - 1) / TC_M;
  // one wave of at most three CTAs per SM: two per SM over the hidden layers, a half over each
  // edge layer
  const int hidden = std::min(l1, c->L - 1) - std::max(l0, 1);
  const int64_t want_h = std::max<int64_t>(1, 2 * c->sms / (DW_GROUPS * std::max(1, hidden)));
  const int64_t want_e = std::max(1, c->sms / 2);
  int blocks = 0;
  for (int l = 0; l < c->L; ++l) {
    DwTcLayer &y = a.l[l];
    const bool edge = l == 0 || l == c->L - 1;
    const int64_t chunk = (n_tiles + (edge ? want_e : want_h) - 1) / (edge ? want_e : want_h);
    y.chunk_tiles = (int)chunk;
    y.first_block = blocks;                            // (a layer outside the range has no blocks)
    if (l < l0 || l >= l1) continue;
    blocks += (int)((n_tiles + chunk - 1) / chunk) * (edge ? 1 : DW_GROUPS);
    y.dw = G + c->off_w[l];
    y.db = G + c->off_b[l];
    y.sym = z;
    y.sym_stride = zs;
    y.feat = c->dout;
    cudaError_t e = row_map(&y.z, l == c->L - 1 ? c->h[l - 1] : c->dz[l], K, TC_M);
    if (e == cudaSuccess && !edge) e = row_map(&y.x, c->h[l - 1], K, TC_ROWS);
    if (e != cudaSuccess) return e;
  }
  return launch_tc(dw_tc_kernel, blocks, TC_M, DW_SMEM, c->stream, l1 - l0 == c->L, a, c->err);
}

rx_status check_sym(rx_cnn *c, const float *p, int64_t stride, int64_t K, const char *what) {
  if (!p) return cfail(c, RX_EINVAL, std::string("null ") + what);
  if ((uintptr_t)p % 8) return cfail(c, RX_EINVAL, std::string(what) + " misaligned");
  if (stride < K) return cfail(c, RX_EINVAL, std::string(what) + " stride too small");
  return RX_OK;
}

// Forward pass; with t, also the loss and dJ/dy, and G and the loss zeroed first.  y may be NULL.
rx_status forward(rx_cnn *c, const float *z, int64_t zs, float *y, int64_t ys, const float *t, int64_t ts, int64_t K,
                  float *G) {
  if (!c->use_tc) {
    if (t) {
      CX_CUDA(cudaMemsetAsync(c->loss, 0, sizeof(double), c->stream), "loss");
      CX_CUDA(cudaMemsetAsync(G, 0, (size_t)c->n_params * sizeof(float), c->stream), "zero grads");
    }
    const int g = (int)std::min<int64_t>((K + 255) / 256, 4 * c->sms);
    features_kernel<<<std::max(1, g), 256, 0, c->stream>>>(reinterpret_cast<const float2 *>(z), zs, K, c->x0);
    CX_CUDA(cudaGetLastError(), "features");
  }
  const int L = c->L;
  for (int l = 0; l < L; ++l) {
    ConvArgs a;
    memset(&a, 0, sizeof(a));
    a.K = K;
    a.w = c->wf[l];
    a.bias = c->P + c->off_b[l];
    a.n_bias = c->co[l];
    a.z = reinterpret_cast<const float2 *>(z);
    a.z_stride = zs;
    if (l < L - 1) {
      a.in = l == 0 ? c->x0 : c->h[l - 1];
      a.out = c->h[l];
      if (l == 0 && c->use_tc) {
        if (t) {
          a.zero = G;
          a.n_zero = c->n_params;
          a.loss = c->loss;
        }
        CX_CUDA((launch_edge_in<true, EPI_RELU>(c, a, c->wtc_f[l], false)), "conv (first)");
      } else if (l == 0) {
        CX_CUDA((launch_conv<FEATP, CH, EPI_RELU>(c, a)), "conv");
      } else if (c->use_tc) {
        CX_CUDA(launch_conv_tc<EPI_RELU>(c, a, c->wtc_f[l], true), "conv (tensor memory)");
      } else {
        CX_CUDA((launch_conv<CH, CH, EPI_RELU>(c, a)), "conv");
      }
    } else {
      a.in = L == 1 ? c->x0 : c->h[L - 2];
      a.y = reinterpret_cast<float2 *>(y);
      a.y_stride = ys;
      a.t = reinterpret_cast<const float2 *>(t);
      a.t_stride = ts;
      a.dout = c->dout;
      a.loss = c->loss;
      a.inv4k = (float)(1.0 / (4.0 * (double)K));
      if (c->use_tc) CX_CUDA(launch_edge_out(c, a, c->wtc_f[l], true), "conv (last)");
      else CX_CUDA((launch_conv<CH, 8, EPI_LAST>(c, a)), "conv (last)");
    }
  }
  return RX_OK;
}

// Backward pass into G (zeroed before the forward pass) from c->dout and the stored
// activations; z: the forward pass's input.
rx_status backward(rx_cnn *c, const float *z, int64_t zs, int64_t K, float *G) {
  const int L = c->L;
  for (int l = L - 1; l >= 0; --l) {
    const bool last = l == L - 1;
    const bf16 *dz = last ? c->dout : c->dz[l];      // [K][16] for the last layer
    if (c->use_tc && c->dz_shared)
      CX_CUDA(launch_dw_tc(c, reinterpret_cast<const float2 *>(z), zs, K, G, l, l + 1), "weight gradient");
    if (!c->use_tc) {
      if (l == 0) {
        CX_CUDA((launch_dw<FEATP, CH>(c, c->x0, dz, K, l, G)), "weight gradient");
      } else if (last) {
        CX_CUDA((launch_dw<CH, FEATP>(c, c->h[l - 1], dz, K, l, G)), "weight gradient");
      } else {
        CX_CUDA((launch_dw<CH, CH>(c, c->h[l - 1], dz, K, l, G)), "weight gradient");
      }
    }
    if (l == 0) break;
    // dJ/d(pre-activation of layer l - 1) = (dz conv W_l^T reversed) * [h_{l-1} > 0]
    ConvArgs a;
    memset(&a, 0, sizeof(a));
    a.in = dz;
    a.K = K;
    a.w = c->wb[l];
    a.mask = c->h[l - 1];
    a.out = c->dz[l - 1];
    if (last && c->use_tc) {
      CX_CUDA((launch_edge_in<false, EPI_MASK>(c, a, c->wtc_b[l], true)), "input gradient");
    } else if (last) {
      CX_CUDA((launch_conv<FEATP, CH, EPI_MASK>(c, a)), "input gradient");
    } else if (c->use_tc) {
      CX_CUDA(launch_conv_tc<EPI_MASK>(c, a, c->wtc_b[l], true), "input gradient (tensor memory)");
    } else {
      CX_CUDA((launch_conv<CH, CH, EPI_MASK>(c, a)), "input gradient");
    }
  }
  if (c->use_tc && !c->dz_shared)
    CX_CUDA(launch_dw_tc(c, reinterpret_cast<const float2 *>(z), zs, K, G, 0, L), "weight gradients");
  return RX_OK;
}

rx_status pack(rx_cnn *c) {
  for (int l = 0; l < c->L; ++l) {
    const int cinp = l == 0 ? FEATP : CH, coutp = l == c->L - 1 ? 8 : CH;
    const int copb = l == c->L - 1 ? FEATP : CH;
    pack_kernel<<<64, 256, 0, c->stream>>>(c->P + c->off_w[l], c->ci[l], c->co[l], c->wf[l], cinp, coutp,
                                             l > 0 ? c->wb[l] : nullptr, copb);
    CX_CUDA(cudaGetLastError(), "pack");
    pack_tc_kernel<<<64, 256, 0, c->stream>>>(c->P + c->off_w[l], c->ci[l], c->co[l], c->wtc_f[l], c->wtc_b[l]);
    CX_CUDA(cudaGetLastError(), "pack (tensor memory)");
  }
  return RX_OK;
}

}  // namespace

extern "C" {

rx_status rx_cnn_create(rx_cnn **out, int layers, int channels, int ksize, int64_t max_symbols) {
  if (!out) return RX_EINVAL;
  *out = nullptr;
  if (layers < 2 || layers > 8 || max_symbols <= 0) return RX_EINVAL;
  if (channels != CH || ksize != KS) return RX_EUNSUPPORTED;
  rx_cnn *c = new (std::nothrow) rx_cnn();
  if (!c) return RX_ENOMEM;
  c->L = layers;
  c->Kmax = max_symbols;
  for (int l = 0; l < layers; ++l) {
    c->ci.push_back(l == 0 ? FEAT : CH);
    c->co.push_back(l == layers - 1 ? FEAT : CH);
    c->off_w.push_back(c->n_params);
    c->n_params += (int64_t)KS * c->ci[l] * c->co[l];
    c->off_b.push_back(c->n_params);
    c->n_params += c->co[l];
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = conv_prepare<FEATP, CH, EPI_RELU>();
  if (e == cudaSuccess) e = conv_prepare<CH, CH, EPI_RELU>();
  if (e == cudaSuccess) e = conv_prepare<CH, 8, EPI_LAST>();
  if (e == cudaSuccess) e = conv_prepare<FEATP, CH, EPI_MASK>();
  if (e == cudaSuccess) e = conv_prepare<CH, CH, EPI_MASK>();
  if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_tc_kernel<EPI_RELU>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_tc_kernel<EPI_MASK>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(dw_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DW_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(edge_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ED_OUT_SMEM);
  if (e != cudaSuccess) {
    delete c;
    return RX_ECUDA;
  }
  *out = c;
#define CX_ALLOC(ptr, count)                      \
  do {                                            \
    rx_status s_ = calloc_dev(c, &(ptr), (count)); \
    if (s_ != RX_OK) { release(c); return s_; }  \
  } while (0)
  CX_ALLOC(c->P, (size_t)c->n_params);
  CX_ALLOC(c->G, (size_t)c->n_params);
  CX_ALLOC(c->M, (size_t)c->n_params);
  CX_ALLOC(c->V, (size_t)c->n_params);
  c->wf.assign(layers, nullptr);
  c->wb.assign(layers, nullptr);
  c->wtc_f.assign(layers, nullptr);
  c->wtc_b.assign(layers, nullptr);
  for (int l = 0; l < layers; ++l) {
    const size_t n = l == 0 || l == layers - 1 ? (size_t)KS * CH * 8 : (size_t)KS * CH * CH;   // edges: at most
    CX_ALLOC(c->wtc_f[l], n);
    if (l > 0) CX_ALLOC(c->wtc_b[l], n);
  }
  for (int l = 0; l < layers; ++l) {
    const int cinp = l == 0 ? FEATP : CH, coutp = l == layers - 1 ? 8 : CH;
    CX_ALLOC(c->wf[l], (size_t)KS * cinp * coutp);
    if (l > 0) CX_ALLOC(c->wb[l], (size_t)KS * CH * (l == layers - 1 ? FEATP : CH));
  }
  const size_t K = (size_t)max_symbols;
  CX_ALLOC(c->x0, K * FEATP);
  CX_ALLOC(c->dout, K * FEATP);
  c->dz.assign(layers - 1, nullptr);
  for (int l = 0; l < std::min(2, layers - 1); ++l) CX_ALLOC(c->dz[l], K * CH);
  c->h.assign(layers - 1, nullptr);
  for (int l = 0; l < layers - 1; ++l) CX_ALLOC(c->h[l], K * CH);
  CX_ALLOC(c->res, 1);
  c->loss = &c->res->loss;
  c->err = &c->res->err;
  if (cudaMallocHost((void **)&c->h_res, sizeof(rx_cnn::Result)) != cudaSuccess) {
    cudaGetLastError();
    release(c);
    return cfail(c, RX_ENOMEM, "pinned result");
  }
#undef CX_ALLOC
  // a buffer per layer lets one launch form every weight gradient from them; without room for
  // that, two serve the layers in turn and each layer's gradient is formed before its turn ends
  const size_t kept = c->allocs.size();
  for (int l = 2; l < layers - 1 && !c->dz_shared; ++l) c->dz_shared = calloc_dev(c, &c->dz[l], K * CH) != RX_OK;
  if (c->dz_shared) {
    for (; c->allocs.size() > kept; c->allocs.pop_back()) cudaFree(c->allocs.back());
    for (int l = 2; l < layers - 1; ++l) c->dz[l] = c->dz[l & 1];
    c->msg.clear();
  }
  CX_CUDA(cudaMemset(c->P, 0, (size_t)c->n_params * sizeof(float)), "init");
  CX_CUDA(cudaMemset(c->M, 0, (size_t)c->n_params * sizeof(float)), "init");
  CX_CUDA(cudaMemset(c->V, 0, (size_t)c->n_params * sizeof(float)), "init");
  CX_CUDA(cudaMemset(c->dout, 0, K * FEATP * sizeof(bf16)), "init");   // channels 4..15 stay zero
  CX_CUDA(cudaMemset(c->res, 0, sizeof(rx_cnn::Result)), "init");
  for (int l : {0, layers - 1}) {        // padding of the edge layers' images
    CX_CUDA(cudaMemset(c->wtc_f[l], 0, (size_t)KS * CH * 8 * sizeof(bf16)), "init");
    if (c->wtc_b[l]) CX_CUDA(cudaMemset(c->wtc_b[l], 0, (size_t)KS * CH * 8 * sizeof(bf16)), "init");
  }
  rx_status s = pack(c);
  if (s != RX_OK) return s;
  CX_CUDA(cudaStreamSynchronize(c->stream), "create");
  return RX_OK;
}

int64_t rx_cnn_param_count(const rx_cnn *c) { return c ? c->n_params : -1; }

rx_status rx_cnn_set_params(rx_cnn *c, const float *params) {
  if (!c || !params) return RX_EINVAL;
  CX_CUDA(cudaMemcpyAsync(c->P, params, (size_t)c->n_params * sizeof(float), cudaMemcpyHostToDevice, c->stream), "set");
  CX_CUDA(cudaMemsetAsync(c->M, 0, (size_t)c->n_params * sizeof(float), c->stream), "set");
  CX_CUDA(cudaMemsetAsync(c->V, 0, (size_t)c->n_params * sizeof(float), c->stream), "set");
  c->step = 0;
  rx_status s = pack(c);
  if (s != RX_OK) return s;
  CX_CUDA(cudaStreamSynchronize(c->stream), "set");
  return RX_OK;
}

namespace {
rx_status timed_out(rx_cnn *c) { return cfail(c, RX_ETIMEOUT, "a bounded device wait gave up (tensor-core convolution)"); }

// Forward and backward pass: the loss in c->res, the gradients in G.
rx_status gradients(rx_cnn *c, const float *z, int64_t zs, const float *t, int64_t ts, int64_t K, float *G) {
  const rx_status s = forward(c, z, zs, nullptr, 0, t, ts, K, G);
  return s == RX_OK ? backward(c, z, zs, K, G) : s;
}

rx_status check_err(rx_cnn *c) {
  int h = 0;
  CX_CUDA(cudaMemcpyAsync(&h, c->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "error word");
  CX_CUDA(cudaStreamSynchronize(c->stream), "error word");
  return h ? timed_out(c) : RX_OK;
}
}  // namespace

rx_status rx_cnn_get_params(rx_cnn *c, float *params) {
  if (!c || !params) return RX_EINVAL;
  CX_CUDA(cudaMemcpyAsync(params, c->P, (size_t)c->n_params * sizeof(float), cudaMemcpyDeviceToHost, c->stream), "get");
  CX_CUDA(cudaStreamSynchronize(c->stream), "get");
  return check_err(c);
}

rx_status rx_cnn_set_option(rx_cnn *c, int key, int value) {
  if (!c) return RX_EINVAL;
  if (key != RX_CNN_OPT_TCGEN05) return cfail(c, RX_EINVAL, "unknown option");
  c->use_tc = value != 0;
  return RX_OK;
}

rx_status rx_cnn_set_cuda_stream(rx_cnn *c, void *s) {
  if (!c) return RX_EINVAL;
  c->stream = (cudaStream_t)s;
  return RX_OK;
}

rx_status rx_cnn_apply(rx_cnn *c, const float *z, int64_t zs, float *y, int64_t ys, int64_t K) {
  if (!c) return RX_EINVAL;
  if (K < 0 || K > c->Kmax) return cfail(c, RX_EINVAL, "K outside 0..max_symbols");
  if (K == 0) return RX_OK;
  rx_status s = check_sym(c, z, zs, K, "input");
  if (s == RX_OK) s = check_sym(c, y, ys, K, "output");
  if (s != RX_OK) return s;
  return forward(c, z, zs, y, ys, nullptr, 0, K, nullptr);
}

rx_status rx_cnn_grads(rx_cnn *c, const float *z, int64_t zs, const float *t, int64_t ts, int64_t K,
                       float *grads_dev, double *loss) {
  if (!c || !grads_dev || !loss) return RX_EINVAL;
  if (K <= 0 || K > c->Kmax) return cfail(c, RX_EINVAL, "K outside 1..max_symbols");
  rx_status s = check_sym(c, z, zs, K, "input");
  if (s == RX_OK) s = check_sym(c, t, ts, K, "target");
  if (s != RX_OK) return s;
  // straight into the caller's buffer where it takes the kernels' 16-byte atomics
  float *G = (uintptr_t)grads_dev % 16 == 0 ? grads_dev : c->G;
  s = gradients(c, z, zs, t, ts, K, G);
  if (s != RX_OK) return s;
  if (G != grads_dev)
    CX_CUDA(cudaMemcpyAsync(grads_dev, G, (size_t)c->n_params * sizeof(float), cudaMemcpyDeviceToDevice, c->stream), "grads");
  CX_CUDA(cudaMemcpyAsync(c->h_res, c->res, sizeof(rx_cnn::Result), cudaMemcpyDeviceToHost, c->stream), "loss");
  CX_CUDA(cudaStreamSynchronize(c->stream), "grads");
  *loss = c->h_res->loss;
  return c->h_res->err ? timed_out(c) : RX_OK;
}

rx_status rx_cnn_train_step(rx_cnn *c, const float *z, int64_t zs, const float *t, int64_t ts, int64_t K, float lr,
                            double *loss_acc) {
  if (!c) return RX_EINVAL;
  if (K <= 0 || K > c->Kmax) return cfail(c, RX_EINVAL, "K outside 1..max_symbols");
  if (!(lr > 0.f)) return cfail(c, RX_EINVAL, "learning rate must be positive");
  rx_status s = check_sym(c, z, zs, K, "input");
  if (s == RX_OK) s = check_sym(c, t, ts, K, "target");
  if (s != RX_OK) return s;
  s = gradients(c, z, zs, t, ts, K, c->G);
  if (s != RX_OK) return s;
  c->step += 1;
  const float c1 = (float)(1.0 - pow(0.9, (double)c->step));
  const float c2 = (float)(1.0 - pow(0.999, (double)c->step));
  {
    KTimer tm(c, RX_CNN_K_UPDATE);
    PackTable tab;
    memset(&tab, 0, sizeof(tab));
    tab.L = c->L;
    for (int l = 0; l < c->L; ++l) {
      PackLayer &y = tab.l[l];
      y.off_w = c->off_w[l];
      y.off_b = c->off_b[l];
      y.ci = c->ci[l];
      y.co = c->co[l];
      y.cinp = l == 0 ? FEATP : CH;
      y.coutp = l == c->L - 1 ? 8 : CH;
      y.copb = l == c->L - 1 ? FEATP : CH;
      y.wf = c->wf[l];
      y.wb = l > 0 ? c->wb[l] : nullptr;
      y.wtc_f = c->wtc_f[l];
      y.wtc_b = c->wtc_b[l];
    }
    adam_pack_kernel<<<std::max(1, std::min(c->sms * 4, (int)((c->n_params + 255) / 256))), 256, 0, c->stream>>>(
        tab, c->P, c->G, c->M, c->V, c->n_params, lr, c1, c2);
    CX_CUDA(cudaGetLastError(), "adam");
  }
  if (loss_acc) {
    add_kernel<<<1, 1, 0, c->stream>>>(loss_acc, c->loss);
    CX_CUDA(cudaGetLastError(), "loss");
  }
  return RX_OK;
}

rx_status rx_cnn_set_profile(rx_cnn *c, int on) {
  if (!c) return RX_EINVAL;
  c->profile = on != 0;
  return RX_OK;
}

rx_status rx_cnn_profile(rx_cnn *c, double *ms, int64_t *launches, int reset) {
  if (!c) return RX_EINVAL;
  CX_CUDA(cudaStreamSynchronize(c->stream), "profile wait");
  for (const auto &pe : c->ev_pending) {
    float t = 0.f;
    CX_CUDA(cudaEventElapsedTime(&t, c->ev_pool[pe.second], c->ev_pool[pe.second + 1]), "profile");
    c->kind_ms[pe.first] += t;
  }
  c->ev_pending.clear();
  c->ev_used = 0;
  for (int i = 0; i < RX_CNN_KINDS; ++i) {
    if (ms) ms[i] = c->kind_ms[i];
    if (launches) launches[i] = c->kind_launches[i];
    if (reset) {
      c->kind_ms[i] = 0;
      c->kind_launches[i] = 0;
    }
  }
  return RX_OK;
}

void rx_cnn_destroy(rx_cnn *c) {
  if (!c) return;
  cudaStreamSynchronize(c->stream);
  for (cudaEvent_t e : c->ev_pool) cudaEventDestroy(e);
  release(c);
  delete c;
}

const char *rx_cnn_last_error(rx_cnn *c) { return c ? c->msg.c_str() : "null handle"; }

}  // extern "C"
