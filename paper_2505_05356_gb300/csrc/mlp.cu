// mlp.cu -- the deformation MLP of Sec. 4 ("MLP") on the 5th-generation
// tensor cores: delta_x = MLP(gamma(x / d_u), gamma(t)), 8 hidden layers of
// 256 with ReLU, a linear head to the 3 offset components, forward and
// backward for B frames x N Gaussians (rows m = b N + g).
//
// Two kinds of kernel, both BF16 operands with FP32 accumulation in TMEM
// (tcgen05.mma issued by one elected thread, operand tiles in shared memory
// in the 128-byte swizzled layout, TMA loads completing on mbarriers):
//  * fused all-layer kernels over pairs of 128-row tiles per CTA (one CTA per
//    SM, the two tiles' accumulators filling TMEM, the epilogue of one tile
//    overlapping the MMAs of the other; a TMA warp streams the weights, an
//    MMA warp, 8 epilogue warps):
//      forward        every layer's output (bias, ReLU, BF16) written back
//                     into the tile as the next layer's operand; training:
//                     each tile also TMA-stored row-major (H_l, the encoding)
//                     and the ReLU masks as bits; inference: nothing kept
//      dZ chain       dZ_7 = (dZ_head W_head) * mask_7, ..., dZ_0, then
//                     d(encoding) = dZ_0 W_0 (FP32), each dZ tile TMA-stored
//                     row-major
//  * a tiled GEMM (TMA pipeline, 4 epilogue warps), for the weight gradients
//    dW_l = dZ_l^T H_{l-1}: the batch rows are the reduction dimension, so
//    both operands are read MN-major straight from the row-major dZ_l and
//    H_{l-1} (transpose bits of the instruction descriptor), the 256 output
//    rows as two M = 128 accumulators sharing each B tile, partial sums per
//    share of rows reduced afterwards; its epilogue warps, idle during the
//    main loop, sum dZ_l's columns (the bias gradient) from each stage.  The
//    same GEMM with other epilogues runs the one-GEMM-per-layer forward and
//    dZ chain, kept as a test mode the fused kernels are checked against.
// Waits on mbarriers are bounded (about 2 s): a wait that runs out records
// GFTORF_ERR_TIMEOUT in the status word and the CTA winds down.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>

#include "gftorf_internal.cuh"

namespace gftorf {
namespace {

constexpr int kW = GFTORF_MLP_WIDTH;    // 256
constexpr int kDepth = GFTORF_MLP_DEPTH;  // 8
constexpr int kIn = GFTORF_MLP_INPUT;   // 128 (84 used)
constexpr int kFreq = 10;
constexpr int kHeadRows = 32;           // head padded to the MMA's N = 32
constexpr int kExt = 16;                // bias column (+ padding) after each dW block
constexpr int BM = 128, BK = 64;

enum Epi { EPI_HIDDEN = 0, EPI_HEAD = 1, EPI_MASK = 2, EPI_F32 = 3, EPI_ATOMIC = 4, EPI_PARTIAL = 5 };
constexpr int kMaxSplits = 192;  // row splits of a weight-gradient GEMM

struct GemmArgs {
  int kb_total;      // k-blocks (of 64) of the reduction
  int kb_per_split;  // k-blocks per CTA along gridDim.z
  int rows_valid;    // output rows that exist (epilogue guard)
  int cols_valid;    // output columns that exist
  const float* bias;
  __nv_bfloat16* out_b;   // row-major bf16 output (ld = ldo)
  int ldo;
  float* out_f;           // FP32 output (ld = ldf)
  int ldf;
  uint32_t* mbits;            // ReLU masks, one bit per unit, [rows][8] words:
                              // written by EPI_HIDDEN, read by EPI_MASK
  float* dbias;               // EPI_PARTIAL with an MN-major A: A's column sums over the
                              // CTA's rows (the bias gradient) added at dbias[n ldb]
  int ldb;
  int inject_no_loads;        // test hook: the producer issues nothing (waits run out)
  unsigned long long wait_ns; // limit of one mbarrier wait
  int* status;
};

// ---- PTX wrappers ----------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait for the phase with the given parity to complete.
__device__ bool mbar_wait(uint32_t bar, uint32_t parity, int* status,
                          unsigned long long limit_ns = 2000000000ull) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try(bar, parity)) return true;
    if (global_ns() - t0 > limit_ns) {
      atomicExch(status, (int)GFTORF_ERR_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
// tile from shared memory to global memory (bulk async-group of this thread)
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0,
                                             int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// this thread's bulk stores have read their shared-memory source
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// ... and have completed
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
// One lane of a converged warp, always the same.  The MMA and load warps run
// their loops with all lanes and let one issue: their control flow and operands
// are then uniform, as the tensor-core and TMA instructions take them.  (With a
// lane-0 branch around the loops every MMA's descriptors were first moved to
// uniform registers one by one: 650 cycles to issue the four MMAs of a weight
// block that run for 512.)
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(ok));
  return ok != 0;
}
// a wait's outcome, the same for the whole warp
__device__ __forceinline__ bool warp_ok(bool ok) { return __all_sync(0xffffffffu, ok); }
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
// K-major operand tile in shared memory, rows of 128 bytes with the 128-byte
// swizzle (8-row groups 1024 bytes apart); the start address may step along K
// inside the 128-byte row.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                             // leading offset (unused here)
  d |= (uint64_t)(1024 >> 4) << 32;                   // stride between 8-row groups
  d |= (uint64_t)1 << 46;                             // descriptor version
  d |= (uint64_t)2 << 61;                             // 128-byte swizzle
  return d;
}
// MN-major operand tile (the M or N index contiguous): 64-element chunks of
// the MN index, each 8192 bytes (64 K-rows of 128 bytes, the 128-byte swizzle
// over 8-row groups 1024 bytes apart), as a TMA box of 64 x 64 lands them;
// the start address steps along K by whole 8-row groups.
__device__ __forceinline__ uint64_t sw128_mn_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)(8192 >> 4) << 16;                   // between 64-element MN chunks
  d |= (uint64_t)(1024 >> 4) << 32;                   // between 8-row K groups
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// kind::f16 instruction descriptor: BF16 x BF16 -> FP32; A and B K-major
// unless mn_a / mn_b (MN-major)
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n, int mn_a = 0, int mn_b = 0) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)mn_a << 15) | ((uint32_t)mn_b << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}
// 32 consecutive FP32 columns of this warp's 32 TMEM lanes (one row per lane)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 64 consecutive FP32 columns of this warp's 32 TMEM lanes, spread as a matrix
// fragment: lane i's value v[32 h + 4 g + 2 s + o] is row 16 h + 8 s + i / 4,
// column 8 g + 2 (i % 4) + o.  A lane then holds only 16 distinct columns, four
// rows each (all 64 columns of one row with the 32x32b shape).
__device__ __forceinline__ void tmem_ld64_frag(uint32_t taddr, float* v) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 {"
        "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr + ((uint32_t)(16 * h) << 16)));
#pragma unroll
    for (int i = 0; i < 32; ++i) v[32 * h + i] = __uint_as_float(r[i]);
  }
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void store_row_bf16(__nv_bfloat16* dst, const float* v) {
  uint4 q[4];
  uint32_t* w = reinterpret_cast<uint32_t*>(q);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<uint32_t*>(&h);
  }
  uint4* d = reinterpret_cast<uint4*>(dst);
#pragma unroll
  for (int i = 0; i < 4; ++i) d[i] = q[i];
}

// ReLU masks, one bit per unit, as the fused epilogues hold a tile: per 128-row
// tile, 32-row quarter, 64-column block and lane two words, whose halves 2 h + s
// are the rows 16 h + 8 s + lane / 4; bit g of a half is column 8 g + 2 (lane %
// 4), bit 8 + g the next column -- the two halves of a packed BF16 pair.  A
// packed comparison (0xFFFF per half) enters them with one logic instruction,
// and one shift and one byte permutation turn a pair of bits back into a mask of
// the packed values (one compare and select per value before: 63 % more
// instructions in the training forward than in inference).
constexpr int kMaskTileWords = BM * kW / 32;  // 1024
__device__ __forceinline__ size_t mask_at(int tile, int q, int cb, int lane) {
  return (size_t)tile * kMaskTileWords + ((q * 4 + cb) * 32 + lane) * 2;
}
// the pair's comparison: bits g (low half) and 24 + g (high half)
__device__ __forceinline__ uint32_t mask_add(uint32_t acc, uint32_t w, int g) {
  const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&w);
  return acc | (__hgt2_mask(h, __nv_bfloat162(__float2bfloat16_rn(0.f), __float2bfloat16_rn(0.f))) &
                (0x01000001u << g));
}
// two rows' comparisons to one word
__device__ __forceinline__ uint32_t mask_word(uint32_t r0, uint32_t r1) {
  r0 |= r0 >> 16;
  r1 |= r1 >> 16;
  return __byte_perm(r0, r1, 0x5410);
}
// 0xFFFF per packed value whose bit is set: pair g of the word's half s
template <int S>
__device__ __forceinline__ uint32_t mask_pair(uint32_t bits, int g) {
  uint32_t m;  // bits g and 8 + g to the bytes' sign bits, each copied over its half
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(m) : "r"(bits << (7 - g)), "n"(S ? 0xBBAA : 0x9988));
  return m;
}
// the byte that holds row m's bits of the block's columns 2 t + odd + 8 g
__device__ __forceinline__ uint8_t* mask_byte(uint32_t* bits, int m, int cb, int t, int odd) {
  const int rr = m & 31;
  uint32_t* w = bits + mask_at(m / BM, (m % BM) >> 5, cb, (rr & 7) * 4 + t) + (rr >> 4);
  return reinterpret_cast<uint8_t*>(w) + 2 * ((rr >> 3) & 1) + odd;
}
// two values to packed BF16, the first in the low half
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t w;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(hi), "f"(lo));
  return w;
}
// the same with the ReLU folded into the conversion: each BF16 value is
// bf16_rn(v) clamped at zero, which equals bf16_rn(max(v, 0))
__device__ __forceinline__ uint32_t pack_bf16_relu(float lo, float hi) {
  uint32_t w;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(hi), "f"(lo));
  return w;
}
// two single-precision additions in one instruction, each rounded on its own
__device__ __forceinline__ void add2(float& a, float& b, float x, float y) {
  unsigned long long u, v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(u) : "f"(a), "f"(b));
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(u) : "l"(v));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(u));
}

// 32 columns [n, n + 32) of output row m
template <int EPI>
__device__ __forceinline__ void epilogue(const GemmArgs& p, int m, int n, float* v) {
  if (EPI == EPI_HIDDEN || EPI == EPI_MASK) {
    if (EPI == EPI_HIDDEN) {
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = fmaxf(v[j] + __ldg(p.bias + n + j), 0.f);
      // columns n..n+31 are half of a block: one nibble of each of its 8 bytes
      const int g0 = (n & 63) / 8;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        uint32_t nib = 0;
#pragma unroll
        for (int g = 0; g < 4; ++g)
          nib |= (__float2bfloat16_rn(v[8 * g + k]) > __float2bfloat16_rn(0.f) ? 1u : 0u) << g;
        uint8_t* d = mask_byte(p.mbits, m, n / 64, k >> 1, k & 1);
        *d = g0 ? (uint8_t)(*d | (nib << 4)) : (uint8_t)nib;
      }
    } else {
      const int g0 = (n & 63) / 8;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint32_t byte = *mask_byte(p.mbits, m, n / 64, k >> 1, k & 1) >> g0;
#pragma unroll
        for (int g = 0; g < 4; ++g)
          if (!((byte >> g) & 1u)) v[8 * g + k] = 0.f;
      }
    }
    store_row_bf16(p.out_b + (size_t)m * p.ldo + n, v);
  } else if (EPI == EPI_HEAD) {
    if (m < p.rows_valid)
      for (int j = 0; j < 3; ++j) p.out_f[(size_t)m * 3 + j] = v[j] + __ldg(p.bias + j);
  } else if (EPI == EPI_F32) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (n + j < p.cols_valid) p.out_f[(size_t)m * p.ldf + n + j] = v[j];
  } else if (EPI == EPI_PARTIAL) {  // this CTA's partial sum over its rows of the batch
    if (m < p.rows_valid && n < p.cols_valid) {
      float4* d = reinterpret_cast<float4*>(
          p.out_f + ((size_t)blockIdx.z * p.rows_valid + m) * p.ldf + n);
#pragma unroll
      for (int q = 0; q < 8; ++q) d[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
  } else {  // EPI_ATOMIC
    if (m < p.rows_valid) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (n + j < p.cols_valid) atomicAdd(p.out_f + (size_t)m * p.ldf + n + j, v[j]);
    }
  }
}

// MT: M = 128 accumulators per CTA sharing each B tile (A tile of 128 MT rows).
// MT = 1: 2 pipeline stages and two CTAs per SM, so that one's epilogue
// overlaps the other's loads and MMAs; MT = 2 fills TMEM (512 columns): one
// CTA per SM with 3 stages.
// MNA / MNB: the operand is read MN-major from a row-major [rows][cols]
// array whose rows are the reduction index (the weight gradients dZ^T H read
// straight from the row-major dZ and H): TMA boxes of 64 columns x 64 rows,
// one per 64 output rows (A) or columns (B), 8 KB each.
template <int BN, int MT>
struct GemmShape {
  static constexpr int kStages = MT == 2 ? 3 : 2;
  static constexpr int A_BYTES = MT * BM * BK * 2, B_BYTES = BN * BK * 2;
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr uint32_t TCOLS = MT * BN < 32 ? 32 : MT * BN;
  static constexpr int SMEM = kStages * STAGE + 1024 + 256;
};

template <int BN, int EPI, int MT, int MNA, int MNB>
__global__ void __launch_bounds__(192, MT == 2 ? 1 : 2)
    umma_gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                     const __grid_constant__ CUtensorMap tmB, const GemmArgs p) {
  grid_begin();
  using S = GemmShape<BN, MT>;
  constexpr int kStages = S::kStages, A_BYTES = S::A_BYTES, STAGE = S::STAGE;
  constexpr uint32_t TCOLS = S::TCOLS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * STAGE);
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 1);
  int* s_ok = reinterpret_cast<int*>(slot + 1);  // the column-sum warps' shared wait outcome
  const uint32_t sbase = smem_u32(smem);
  // the epilogue warps sum A's columns from each stage while the MMAs run
  // (the weight-gradient GEMMs are bound by HBM; their epilogue warps idle)
  constexpr bool COLSUM = EPI == EPI_PARTIAL && MNA && MT == 2;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kStages,
                 done = full0 + 16 * kStages;
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int kb0 = blockIdx.z * p.kb_per_split;
  const int nkb = min(p.kb_per_split, p.kb_total - kb0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, COLSUM ? 2 : 1);  // (+ the column-sum warps)
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(smem_u32(slot), TCOLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = (uint32_t)uniform((int)*slot);

  if (warp == 4) {
    // TMA producer
    if (nkb > 0 && !p.inject_no_loads) {
      int issued = 0;
      for (int i = 0; i < nkb; ++i) {
        const int s = i % kStages;
        const uint32_t ph = (uint32_t)(i / kStages) & 1u;
        if (!warp_ok(mbar_wait(empty0 + 8 * s, ph ^ 1u, p.status, p.wait_ns))) break;
        if (elect_one()) {
          mbar_expect_tx(full0 + 8 * s, STAGE);
          const uint32_t sa = sbase + s * STAGE;
          if (MNA) {
#pragma unroll
            for (int j = 0; j < 2 * MT; ++j)
              tma_load_2d(sa + j * 8192, &tmA, full0 + 8 * s, m0 * MT + 64 * j, (kb0 + i) * BK);
          } else {
            tma_load_2d(sa, &tmA, full0 + 8 * s, (kb0 + i) * BK, m0 * MT);
          }
          if (MNB) {
#pragma unroll
            for (int j = 0; j < BN / 64; ++j)
              tma_load_2d(sa + A_BYTES + j * 8192, &tmB, full0 + 8 * s, n0 + 64 * j,
                          (kb0 + i) * BK);
          } else {
            tma_load_2d(sa + A_BYTES, &tmB, full0 + 8 * s, (kb0 + i) * BK, n0);
          }
        }
        __syncwarp();
        issued = i + 1;
      }
      // every load issued has landed before the CTA may exit
      for (int i = issued - kStages < 0 ? 0 : issued - kStages; i < issued; ++i)
        mbar_wait(full0 + 8 * (i % kStages), (uint32_t)(i / kStages) & 1u, p.status, p.wait_ns);
    }
  } else if (warp == 5) {
    // MMA issuer
    if (nkb > 0) {
      constexpr uint32_t idesc = idesc_bf16(BM, BN, MNA, MNB);
      for (int i = 0; i < nkb; ++i) {
        const int s = i % kStages;
        const uint32_t ph = (uint32_t)(i / kStages) & 1u;
        if (!warp_ok(mbar_wait(full0 + 8 * s, ph, p.status, p.wait_ns))) break;
        tc_fence_after();
        if (elect_one()) {
          const uint32_t sa = sbase + s * STAGE, sb = sa + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
#pragma unroll
            for (int t = 0; t < MT; ++t) {
              // K step of 16: 32 bytes along a K-major row, two 8-row groups MN-major
              const uint64_t da = MNA ? sw128_mn_desc(sa + t * 16384 + 2048 * k)
                                      : sw128_desc(sa + t * BM * 128 + 32 * k);
              const uint64_t db = MNB ? sw128_mn_desc(sb + 2048 * k) : sw128_desc(sb + 32 * k);
              umma_bf16(tmem + (uint32_t)(t * BN), da, db, idesc, (i > 0 || k > 0) ? 1u : 0u);
            }
          umma_commit(empty0 + 8 * s);
        }
        __syncwarp();
      }
      if (elect_one()) umma_commit(done);  // completes once every MMA issued above has
      __syncwarp();
    }
  } else {
    float cs0 = 0.f, cs1 = 0.f;  // COLSUM: columns 2 tid, 2 tid + 1 of A
    bool cs_ok = true;
    if (COLSUM) {
      // A's 64-column chunk tid / 32, 4-byte word (tid % 32) of each 128-byte
      // row (chunk (tid % 32) / 4 of the row, under the swizzle)
      const int tid = threadIdx.x;
      const uint32_t col_off = (uint32_t)(tid >> 5) * 8192u + 4u * (uint32_t)(tid & 3);
      const uint32_t chunk = (uint32_t)((tid & 31) >> 2);
      for (int i = 0; i < nkb; ++i) {
        const int s = i % kStages;
        // one thread waits, the others follow the barrier (all take one branch)
        if (threadIdx.x == 0)
          *s_ok = mbar_wait(full0 + 8 * s, (uint32_t)(i / kStages) & 1u, p.status, p.wait_ns);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (!(cs_ok = *s_ok != 0)) break;
        const uint8_t* st = smem + s * STAGE + col_off;
#pragma unroll 8
        for (int r = 0; r < BK; ++r) {
          const uint32_t w = *reinterpret_cast<const uint32_t*>(
              st + (r >> 3) * 1024 + (r & 7) * 128 + ((chunk ^ (uint32_t)(r & 7)) << 4));
          cs0 += __uint_as_float(w << 16);
          cs1 += __uint_as_float(w & 0xFFFF0000u);
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");  // all four warps have read stage s
        if (threadIdx.x == 0) mbar_arrive(empty0 + 8 * s);
      }
    }
    // epilogue: warp w owns TMEM lanes / output rows 32 w .. 32 w + 31
    if (nkb > 0 && cs_ok && mbar_wait(done, 0, p.status, p.wait_ns)) {
      tc_fence_after();
#pragma unroll 1
      for (int t = 0; t < MT; ++t) {
        const int m = (m0 * MT + t * BM) + warp * 32 + lane;
#pragma unroll 1
        for (int c = 0; c < BN / 32; ++c) {
          float v[32];
          tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(t * BN + c * 32), v);
          epilogue<EPI>(p, m, n0 + c * 32, v);
        }
      }
      if (COLSUM) {
        atomicAdd(p.dbias + (size_t)(2 * threadIdx.x) * p.ldb, cs0);
        atomicAdd(p.dbias + (size_t)(2 * threadIdx.x + 1) * p.ldb, cs1);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, TCOLS);
  }
}

// ---- element-wise kernels ----------------------------------------------------
struct Times {
  float t[kMaxFrames];
};

// offsets in the packed parameter vector, [W_0, b_0, W_1, b_1, ..., W_head, b_head]
__host__ __device__ constexpr size_t bias_off_dev(int l) {
  return l == 0 ? (size_t)kW * kIn
                : (size_t)kW * kIn + kW + (size_t)(l - 1) * ((size_t)kW * kW + kW) + (size_t)kW * kW;
}
__host__ __device__ constexpr size_t head_bias_off_dev() {
  return (size_t)kW * kIn + kW + (size_t)(kDepth - 1) * ((size_t)kW * kW + kW) + 3 * kW;
}

// fp32 packed parameters -> bf16 W and W^T of every layer (head padded to 32 rows)
__global__ void mlp_prep_weights_kernel(const float* __restrict__ theta,
                                        __nv_bfloat16* __restrict__ wb,
                                        __nv_bfloat16* __restrict__ wt) {
  grid_begin_early();
  // packed offsets: layer l (0..7) W at off_w(l), then b; head after
  const int K0 = kIn;
  const size_t total = (size_t)kW * K0 + (size_t)(kDepth - 1) * kW * kW + (size_t)kHeadRows * kW;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    int l, o, i;
    size_t src, dstb, dstt;
    if (e < (size_t)kW * K0) {
      l = 0;
      o = (int)(e / K0), i = (int)(e % K0);
      src = (size_t)o * K0 + i;
      dstb = e;
      dstt = (size_t)i * kW + o;
    } else if (e < (size_t)kW * K0 + (size_t)(kDepth - 1) * kW * kW) {
      const size_t r = e - (size_t)kW * K0;
      l = 1 + (int)(r / ((size_t)kW * kW));
      const size_t q = r % ((size_t)kW * kW);
      o = (int)(q / kW), i = (int)(q % kW);
      const size_t base = (size_t)kW * K0 + kW + (size_t)(l - 1) * ((size_t)kW * kW + kW);
      src = base + q;
      dstb = e;
      dstt = (size_t)kW * K0 + (size_t)(l - 1) * kW * kW + (size_t)i * kW + o;
    } else {
      const size_t r = e - (size_t)kW * K0 - (size_t)(kDepth - 1) * kW * kW;
      l = kDepth;
      o = (int)(r / kW), i = (int)(r % kW);
      const size_t base = (size_t)kW * K0 + kW + (size_t)(kDepth - 1) * ((size_t)kW * kW + kW);
      src = o < 3 ? base + (size_t)o * kW + i : 0;
      dstb = e;
      dstt = (size_t)kW * K0 + (size_t)(kDepth - 1) * kW * kW + (size_t)i * kHeadRows + o;
    }
    const float w = (l == kDepth && o >= 3) ? 0.f : theta[src];
    wb[dstb] = __float2bfloat16_rn(w);
    wt[dstt] = __float2bfloat16_rn(w);
  }
}

// positional encoding of row m = b N + g (zeros for m >= M)
__device__ __forceinline__ void encode_row(const float* __restrict__ means, const Times& tm, int N,
                                           int M, float inv_scale, int m, float* e) {
#pragma unroll
  for (int c = 0; c < kIn; ++c) e[c] = 0.f;
  if (m < M) {
    const int b = m / N, g = m - b * N;
    float x[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = means[(size_t)g * 3 + a] * inv_scale;
    const float t = tm.t[b];
#pragma unroll
    for (int a = 0; a < 3; ++a) e[a] = x[a];
    float f = 1.f;
#pragma unroll
    for (int l = 0; l < kFreq; ++l, f *= 2.f) {
#pragma unroll
      for (int a = 0; a < 3; ++a) sincospif(f * x[a], &e[3 + 6 * l + a], &e[6 + 6 * l + a]);
    }
    e[63] = t;
    f = 1.f;
#pragma unroll
    for (int l = 0; l < kFreq; ++l, f *= 2.f) sincospif(f * t, &e[64 + 2 * l], &e[65 + 2 * l]);
  }
}

// positional encoding of row m = b N + g into enc[m][0..127]
__global__ void mlp_encode_kernel(const float* __restrict__ means, Times tm, int N, int B,
                                  float inv_scale, int M_pad, __nv_bfloat16* __restrict__ enc) {
  grid_begin();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M_pad) return;
  float e[kIn];
  encode_row(means, tm, N, N * B, inv_scale, m, e);
#pragma unroll
  for (int q = 0; q < kIn / 32; ++q) store_row_bf16(enc + (size_t)m * kIn + 32 * q, e + 32 * q);
}

// dL/d(delta) fp32 [M][3] -> BF16, transposed: [3][M_pad] (the head's weight
// gradient reduces over the rows) and, for the one-GEMM-per-layer chain only,
// row-major [M_pad][32] (dz, else null); and the head's bias gradient, the
// column sums of the rounded values.  Rows 3..31 of the transposed array are
// beyond its tensor map and arrive as zeros.  The column sums go through the
// CTA first: with one atomic per warp and column the 28k additions to three
// addresses serialised (19.7 us at 300k rows).
constexpr int kHeadGradThreads = 256;
__global__ void __launch_bounds__(kHeadGradThreads)
    mlp_head_grad_kernel(const float* __restrict__ dd, int M, int M_pad,
                         __nv_bfloat16* __restrict__ dz, __nv_bfloat16* __restrict__ dzt,
                         float* __restrict__ dbias, int ldb) {
  grid_begin_early();
  __shared__ float s_sum[kHeadGradThreads / 32][3];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float sum[3] = {0.f, 0.f, 0.f};
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M_pad; m += gridDim.x * blockDim.x) {
    __nv_bfloat16 q[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      q[j] = __float2bfloat16_rn(m < M ? dd[(size_t)m * 3 + j] : 0.f);
      dzt[(size_t)j * M_pad + m] = q[j];
      sum[j] += __bfloat162float(q[j]);
    }
    if (dz) {
      float v[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = j < 3 ? __bfloat162float(q[j]) : 0.f;
      store_row_bf16(dz + (size_t)m * kHeadRows, v);
    }
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], o);
    if (lane == 0) s_sum[w][j] = sum[j];
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    float b = 0.f;
    for (int k = 0; k < kHeadGradThreads / 32; ++k) b += s_sum[k][threadIdx.x];
    if (b != 0.f) atomicAdd(dbias + (size_t)threadIdx.x * ldb, b);
  }
}

// dL/d(means) from the encoding's gradient (the position part, columns
// 0..62), summed over the frames: two threads per Gaussian, thread h taking the
// bands 5 h .. 5 h + 4 (columns 30 h + 3 .. 30 h + 32) and thread 0 the position
// itself.  The frames' rows are summed first, then the derivative of the
// encoding is applied -- d sin(f pi x)/dx = f pi cos(f pi x), d cos(f pi x)/dx =
// -f pi sin(f pi x).  One warp per Gaussian (a column per lane) evaluated every
// sine-cosine pair twice and spent 15 shuffles per Gaussian: 70 us at 300k
// Gaussians, bound by instruction issue at 1.1 TB/s.
__global__ void __launch_bounds__(128)
    mlp_encode_bwd_kernel(const float* __restrict__ means, const float* __restrict__ denc, int N,
                          int B, float inv_scale, float* __restrict__ dmeans) {
  grid_begin();
  constexpr int kBands = kFreq / 2, kCols = 6 * kBands + 4;  // (even: float2 loads)
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int g = min(i >> 1, N - 1), h = i & 1;  // (a whole warp reaches the shuffles)
  float d[kCols];
#pragma unroll
  for (int c = 0; c < kCols; ++c) d[c] = 0.f;
#pragma unroll 2
  for (int b = 0; b < B; ++b) {
    const float2* row =
        reinterpret_cast<const float2*>(denc + ((size_t)b * N + g) * kIn + 6 * kBands * h);
#pragma unroll
    for (int c = 0; c < kCols / 2; ++c) {
      const float2 v = __ldg(row + c);
      d[2 * c] += v.x;
      d[2 * c + 1] += v.y;
    }
  }
  float acc[3], x[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    acc[a] = h ? 0.f : d[a];
    x[a] = __ldg(means + (size_t)g * 3 + a) * inv_scale;
  }
  float f = h ? (float)(1 << kBands) : 1.f;
#pragma unroll
  for (int l = 0; l < kBands; ++l, f *= 2.f) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float sn, cs;
      sincospif(f * x[a], &sn, &cs);
      acc[a] += f * 3.14159265358979323846f * (cs * d[3 + 6 * l + a] - sn * d[6 + 6 * l + a]);
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], 1);
  if (h == 0 && (i >> 1) < N)
    for (int a = 0; a < 3; ++a) dmeans[(size_t)g * 3 + a] = acc[a] * inv_scale;
}

// extended weight gradients [rows][K + ext] -> packed d_theta (W then b)
__global__ void mlp_unpack_grads_kernel(const float* __restrict__ dwx, float* __restrict__ dth) {
  grid_begin_early();
  const size_t total = (size_t)kW * (kIn + 1) + (size_t)(kDepth - 1) * kW * (kW + 1) + 3 * (kW + 1);
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    // locate layer
    size_t r = e, src_base = 0;
    int K = kIn, rows = kW, l = 0;
    for (;;) {
      const size_t n = (size_t)rows * (K + 1);
      if (r < n) break;
      r -= n;
      src_base += (size_t)(l == kDepth ? kHeadRows : kW) * (K + kExt);
      ++l;
      K = kW;
      rows = l == kDepth ? 3 : kW;
    }
    const int ld = K + kExt;
    float v;
    if (r < (size_t)rows * K) {
      const int o = (int)(r / K), i = (int)(r % K);
      v = dwx[src_base + (size_t)o * ld + i];
    } else {
      const int o = (int)(r - (size_t)rows * K);
      v = dwx[src_base + (size_t)o * ld + K];
    }
    dth[e] = v;
  }
}

// sum of the row-split partials [splits][256][K] -> dW block [256][ld]: a CTA
// takes 32 groups of four consecutive values, its eight warps every eighth
// split each (the partials lie in L2; with one value per thread and all splits
// in a row the loads in flight bounded it: 13.5 us per layer of 152 splits)
constexpr int kReduceWarps = 8;
__global__ void __launch_bounds__(32 * kReduceWarps)
    mlp_reduce_dw_kernel(const float* __restrict__ part, int splits, int K,
                         float* __restrict__ dw, int ld) {
  grid_begin_early();
  __shared__ float4 s_sum[kReduceWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = (blockIdx.x * 32 + lane) * 4;  // 256 K is a multiple of 128
  const size_t stride = (size_t)kW * K;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 5
  for (int z = w; z < splits; z += kReduceWarps) {
    const float4 v = __ldcs(reinterpret_cast<const float4*>(part + (size_t)z * stride + e));
    s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
  }
  s_sum[w][lane] = s;
  __syncthreads();
  if (w != 0) return;
#pragma unroll
  for (int k = 1; k < kReduceWarps; ++k) {
    const float4 v = s_sum[k][lane];
    s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
  }
  const int o = e / K, i = e - o * K;
  *reinterpret_cast<float4*>(dw + (size_t)o * ld + i) = s;
}

// ---- fused forward (inference): all layers of 128-row tiles in one CTA -------
// The activations never leave shared memory: the epilogue warps write each
// layer's output (bias, ReLU, BF16) straight into the 128 x 256 operand tile
// of the next layer, in the swizzled K-major layout of the MMA descriptors,
// while a TMA warp streams the layers' weights through a 3-stage ring.  A CTA
// works on two tiles at once (two activation tiles, two TMEM accumulators),
// alternating (layer, tile) items so that the epilogue of one tile runs while
// the tensor core computes the other.  The arithmetic and its order are those
// of the layer-by-layer forward, so the outputs agree bit for bit; nothing is
// kept for a backward.
constexpr int kFusedStages = 3;
constexpr int kPair = 2;                   // tiles in flight per CTA
constexpr int kActBytes = BM * kW * 2;     // 64 KB per tile
constexpr int kWStageBytes = kW * BK * 2;  // 32 KB (a 256-row k-block of W)
// (the barriers' 256 bytes, one layer's biases, and the alignment)
constexpr int kFusedSmem = kPair * kActBytes + kFusedStages * kWStageBytes + 256 + kW * 4 + 1024;

struct FusedMaps {
  CUtensorMap w[kDepth + 1];  // bf16 W of the hidden layers (256 rows), head (32 rows)
  CUtensorMap enc;            // training forward: the encoding [Mp][128] (stores)
  CUtensorMap act;            // H (forward) or dZ (backward) of all layers [8 Mp][256] (stores)
};

// byte offset of element (r, c) of an activation tile: 64-column blocks of
// 16 KB, rows 128 bytes apart in 1024-byte 8-row atoms, 16-byte chunk j of
// row r at chunk j ^ (r & 7) (the 128-byte swizzle)
__device__ __forceinline__ uint32_t act_off(int r, int c) {
  const int kb = c >> 6, cc = c & 63;
  return (uint32_t)(kb * 16384 + (r >> 3) * 1024 + (r & 7) * 128 +
                    ((((cc >> 3) ^ (r & 7)) << 4) | ((cc & 7) << 1)));
}
__device__ __forceinline__ void store_act8(uint8_t* act, int r, int c, const float* v) {
  *reinterpret_cast<uint4*>(act + act_off(r, c)) =
      make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                 pack_bf16(v[6], v[7]));
}
__device__ __forceinline__ void store_act16(uint8_t* act, int r, int c, const float* v) {
  store_act8(act, r, c, v);
  store_act8(act, r, c + 8, v + 8);
}

// A lane's part of the address of a fragment's store into an activation tile: a
// stmatrix of four 8 x 8 matrices (column groups g, g + 1 of rows 0..7 and 8..15 of
// a 16-row half) takes the matrices' row addresses from the lanes in order.
struct FragStore {
  uint32_t row;  // shared address of the lane's row, first chunk of block 0
  uint32_t x;    // the swizzle and the lane's column group, to be XORed with 16 g
};
__device__ __forceinline__ FragStore frag_store(uint32_t act_s, int q, int lane) {
  const int r = q * 32 + ((lane >> 3) & 1) * 8 + (lane & 7);
  return {act_s + (uint32_t)((r >> 3) * 1024 + (r & 7) * 128),
          (uint32_t)(((lane >> 4) ^ (lane & 7)) << 4)};
}
// packed values of column groups g, g + 1 (g even) of 16-row half h, block cb
__device__ __forceinline__ void store_frag(const FragStore& f, int cb, int h, int g, uint32_t a0,
                                           uint32_t a1, uint32_t b0, uint32_t b1) {
  const uint32_t at = f.row + (uint32_t)(cb * 16384 + h * 2048) + (f.x ^ (uint32_t)(16 * g));
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(at),
               "r"(a0), "r"(a1), "r"(b0), "r"(b1)
               : "memory");
}

// encode_row's values of columns [C0, C0 + 16) from the scaled position (columns
// below 63)
template <int C0>
__device__ __forceinline__ void encode16(const float* x, float* e) {
  float f = 1.f;
#pragma unroll
  for (int l = 0; l < kFreq; ++l, f *= 2.f)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (l == 0 && a >= C0 && a < C0 + 16) e[a - C0] = x[a];
      const int cs = 3 + 6 * l + a, cc = cs + 3;
      const bool is = cs >= C0 && cs < C0 + 16, ic = cc >= C0 && cc < C0 + 16;
      if (is || ic) {
        float sn, co;
        sincospif(f * x[a], &sn, &co);
        if (is) e[cs - C0] = sn;
        if (ic) e[cc - C0] = co;
      }
    }
}

// encode_row's values of one row, straight into the row's place in the tile, by
// four threads: part p takes the position's columns 16 p .. 16 p + 15, part 0
// also the time's (64..83), the others the zeros behind them.  The time's values
// depend on the frame only: where a warp's rows lie in one frame, ten lanes
// evaluate one band each and the warp shares them.  (One thread per row, 40
// sine-cosine pairs: the tensor cores idled through them.)
__device__ __forceinline__ void encode_part(const float* __restrict__ means, const Times& tm,
                                            int N, int M, float inv_scale, int m, int part,
                                            uint8_t* act, int r) {
  const bool in = m < M;
  const int b = in ? m / N : 0, g = in ? m - b * N : 0;
  const float t = tm.t[b];
  float x[3], e[32];
#pragma unroll
  for (int a = 0; a < 3; ++a) x[a] = in ? means[(size_t)g * 3 + a] * inv_scale : 0.f;
  if (part == 0) {
    encode16<0>(x, e);
  } else if (part == 1) {
    encode16<16>(x, e);
  } else if (part == 2) {
    encode16<32>(x, e);
  } else {
    encode16<48>(x, e);
    e[15] = t;
  }
#pragma unroll
  for (int c = 0; c < 16; ++c) e[c] = in ? e[c] : 0.f;
  store_act16(act, r, 16 * part, e);
  if (part != 0) {  // columns 80..127: the last bands' four are part 0's
    uint4* z = reinterpret_cast<uint4*>(act + act_off(r, 80 + 16 * (part - 1)));
    if (part > 1) *z = make_uint4(0, 0, 0, 0);
    *reinterpret_cast<uint4*>(act + act_off(r, 88 + 16 * (part - 1))) = make_uint4(0, 0, 0, 0);
    return;
  }
  float te[24], sn, cs;
  const int lane = threadIdx.x & 31;
  const int b0 = __shfl_sync(0xffffffffu, b, 0);
  if (__all_sync(0xffffffffu, b == b0 || !in)) {
    sincospif((float)(1 << (lane < kFreq ? lane : 0)) * tm.t[b0], &sn, &cs);
#pragma unroll
    for (int l = 0; l < kFreq; ++l) {
      te[2 * l] = __shfl_sync(0xffffffffu, sn, l);
      te[2 * l + 1] = __shfl_sync(0xffffffffu, cs, l);
    }
  } else {
    float f = 1.f;
#pragma unroll
    for (int l = 0; l < kFreq; ++l, f *= 2.f) sincospif(f * t, &te[2 * l], &te[2 * l + 1]);
  }
#pragma unroll
  for (int c = 0; c < 24; ++c) te[c] = c < 2 * kFreq && in ? te[c] : 0.f;
  store_act16(act, r, 64, te);
  store_act8(act, r, 80, te + 16);
}

// warps 0-7: epilogue (warp w: TMEM lanes / rows 32 (w % 4) .. + 31, columns
// 128 (w / 4) .. + 127); warp 8: TMA; warp 9: MMA.
// The epilogue shares with the MMAs the 128 bytes a cycle that shared memory (and
// the L1 data path behind every load) moves: for a tile's layer the MMAs read
// 192 KB of operands (1536 cycles for 2048 of MMA), the weights arrive with 128 KB
// and the epilogue stores 64 KB.  So the epilogue takes the accumulators as matrix
// fragments (a lane: 16 columns of four rows), which needs a quarter of the bias
// values per lane that one row of 64 columns did (those alone took 1024 cycles
// per tile and layer, from global or shared memory alike), and stores them by
// stmatrix.  300k rows of inference: 260 -> 191 us (0.77 of the measured BF16
// peak back to back, 0.73 by single calls), the tensor pipe active 51 -> 72 % of
// the cycles; timelines: 3300 -> 2300 cycles per tile and layer.  Training forward
// 392 -> 319 us, 33 -> 42 %: no unit is above 61 % there (L1 / shared memory 60,
// DRAM 53), what is left is the chain of a tile's layers.  Sixteen epilogue warps
// measured the same.
constexpr int kFusedEpiWarps = 8;
constexpr int kFusedEpiThreads = 32 * kFusedEpiWarps;
constexpr int kFusedThreads = kFusedEpiThreads + 64;
constexpr int kParts = kFusedEpiWarps / 4;       // warps that share a row
constexpr int kBlocks = kW / 64 / kParts;        // 64-column blocks of a thread
__device__ __forceinline__ void epi_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kFusedEpiThreads) : "memory");
}

// What a training forward keeps for the backward (TRAIN): the encoded input
// and every hidden activation (row-major BF16, stored by TMA from the tile in
// shared memory through maps.enc / maps.act), and the ReLU masks as bits (per
// layer Mp kW / 32 words, in the order of mask_at) -- the same values the
// layer-by-layer forward stores.  The stores of tile t are issued (and waited for before the tile is
// written again) by epilogue thread 32 t.
struct FusedKeep {
  uint32_t* bits;
  int Mp;
};

template <bool TRAIN>
__global__ void __launch_bounds__(kFusedThreads, 1)
    mlp_fused_fwd_kernel(const __grid_constant__ FusedMaps maps, const float* __restrict__ theta,
                         const float* __restrict__ means, Times tm, int N, int M, int n_tiles,
                         float inv_scale, float* __restrict__ delta, int* status,
                         unsigned long long wait_ns, int inject_no_loads, FusedKeep keep) {
  grid_begin();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars =
      reinterpret_cast<uint64_t*>(smem + kPair * kActBytes + kFusedStages * kWStageBytes);
  // bars: full[S], empty[S], acc_ready[kPair], act_ready[kPair]
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 2 * kFusedStages + 2 * kPair);
  int* s_ok = reinterpret_cast<int*>(slot + 1);  // the epilogue's shared wait outcome
  float* s_bias = reinterpret_cast<float*>(bars + 32);  // the layer's biases
  const uint32_t act_s = smem_u32(smem), w_s = act_s + kPair * kActBytes;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kFusedStages;
  const uint32_t acc0 = full0 + 16 * kFusedStages, actr0 = acc0 + 8 * kPair;
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int n_pairs = (n_tiles + kPair - 1) / kPair;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kFusedStages; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    for (int t = 0; t < kPair; ++t) {
      mbar_init(acc0 + 8 * t, 1);
      mbar_init(actr0 + 8 * t, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(smem_u32(slot), (uint32_t)(kPair * kW));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = (uint32_t)uniform((int)*slot);

  if (warp == kFusedEpiWarps) {
    // weights of every (layer, tile) item, k-block by k-block
    if (!inject_no_loads) {
      int it = 0;
      bool ok = true;
      for (int pr = blockIdx.x; ok && pr < n_pairs; pr += gridDim.x)
        for (int l = 0; ok && l <= kDepth; ++l)
          for (int t = 0; ok && t < kPair; ++t) {
            const int nkb = (l == 0 ? kIn : kW) / BK;
            const uint32_t bytes = (uint32_t)(l == kDepth ? kHeadRows : kW) * BK * 2;
            for (int kb = 0; kb < nkb; ++kb, ++it) {
              const int s = it % kFusedStages;
              if (!(ok = warp_ok(mbar_wait(empty0 + 8 * s, ((uint32_t)(it / kFusedStages) & 1u) ^ 1u,
                                           status, wait_ns))))
                break;
              if (elect_one()) {
                mbar_expect_tx(full0 + 8 * s, bytes);
                tma_load_2d(w_s + s * kWStageBytes, &maps.w[l], full0 + 8 * s, kb * BK, 0);
              }
            }
          }
      // every load issued has landed before the CTA may exit
      for (int i = it - kFusedStages < 0 ? 0 : it - kFusedStages; i < it; ++i)
        mbar_wait(full0 + 8 * (i % kFusedStages), (uint32_t)(i / kFusedStages) & 1u, status,
                  wait_ns);
    }
  } else if (warp == kFusedEpiWarps + 1) {
    {
      int it = 0;
      uint32_t act_ph[kPair] = {0, 0};
      bool ok = true;
      for (int pr = blockIdx.x; ok && pr < n_pairs; pr += gridDim.x)
        for (int l = 0; ok && l <= kDepth; ++l)
          for (int t = 0; ok && t < kPair; ++t) {
            if (!(ok = warp_ok(mbar_wait(actr0 + 8 * t, act_ph[t], status, wait_ns)))) break;
            act_ph[t] ^= 1u;
            tc_fence_after();
            const int nkb = (l == 0 ? kIn : kW) / BK;
            const uint32_t idesc = l == kDepth ? idesc_bf16(BM, kHeadRows) : idesc_bf16(BM, kW);
            const uint32_t d = tmem + (uint32_t)(t * kW);
            for (int kb = 0; kb < nkb; ++kb, ++it) {
              const int s = it % kFusedStages;
              if (!(ok = warp_ok(mbar_wait(full0 + 8 * s, (uint32_t)(it / kFusedStages) & 1u, status,
                                           wait_ns))))
                break;
              tc_fence_after();
              const uint32_t sa = act_s + t * kActBytes + kb * 16384, sb = w_s + s * kWStageBytes;
              if (elect_one()) {
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                  umma_bf16(d, sw128_desc(sa + 32 * k), sw128_desc(sb + 32 * k), idesc,
                            (kb > 0 || k > 0) ? 1u : 0u);
                umma_commit(empty0 + 8 * s);
              }
              __syncwarp();
            }
            if (elect_one()) umma_commit(acc0 + 8 * t);
            __syncwarp();
          }
    }
  } else {
    // epilogue warps: 32 rows of every tile (the encoding and the head: row r), half of
    // the columns, as fragments
    const int q = warp & 3, part = warp >> 2;
    const int r = q * 32 + lane;
    uint32_t acc_ph[kPair] = {0, 0};
    bool ok = true;
    for (int pr = blockIdx.x; ok && pr < n_pairs; pr += gridDim.x) {
      for (int t = 0; t < kPair; ++t) {
#pragma unroll 1
        for (int k = 0; k < kBlocks; ++k)
          encode_part(means, tm, N, M, inv_scale, (pr * kPair + t) * BM + r, part + k * kParts,
                      smem + t * kActBytes, r);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        epi_sync();
        if (threadIdx.x == 0) mbar_arrive(actr0 + 8 * t);
        if (TRAIN && threadIdx.x == 32 * t && pr * kPair + t < n_tiles) {
          for (int kb = 0; kb < kIn / BK; ++kb)
            tma_store_2d(&maps.enc, act_s + t * kActBytes + kb * 16384, kb * BK,
                         (pr * kPair + t) * BM);
          bulk_commit();
        }
      }
      // (every thread is past the last pair's barrier, so its biases are free)
      if (threadIdx.x < kW) s_bias[threadIdx.x] = __ldg(theta + bias_off_dev(0) + threadIdx.x);
      for (int l = 0; ok && l <= kDepth; ++l)
        for (int t = 0; t < kPair; ++t) {
          // one thread waits, the other epilogue threads follow the barrier, so
          // that all of them take the same branch (no split at the named barriers)
          if (threadIdx.x == 0)
            *s_ok = mbar_wait(acc0 + 8 * t, acc_ph[t], status, wait_ns) ? 1 : 0;
          // the tile's last store has read it before it is written again
          if (TRAIN && threadIdx.x == 32 * t) bulk_wait_read();
          epi_sync();
          // (every step ends at a named barrier that all epilogue threads reach
          // after reading the flag, so thread 0 rewrites it only afterwards)
          if (!(ok = *s_ok != 0)) break;
          acc_ph[t] ^= 1u;
          tc_fence_after();
          const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(t * kW);
          if (l < kDepth) {
            const FragStore fs = frag_store(act_s + t * kActBytes, q, lane);
#pragma unroll 1
            for (int k = 0; k < kBlocks; ++k) {
              const int cb = part * kBlocks + k;
              float v[64];
              tmem_ld64_frag(trow + (uint32_t)(cb * 64), v);
              float2 b[8];
#pragma unroll
              for (int g = 0; g < 8; ++g)
                b[g] = *reinterpret_cast<const float2*>(s_bias + cb * 64 + 8 * g + 2 * (lane & 3));
              tmem_wait_ld();
              uint32_t rows[4] = {0, 0, 0, 0};
#pragma unroll
              for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int g = 0; g < 8; g += 2) {
                  uint32_t w[4];
#pragma unroll
                  for (int i = 0; i < 4; ++i) {  // group g + i / 2, rows 8 (i % 2)
                    float* e = v + 32 * h + 4 * (g + (i >> 1)) + 2 * (i & 1);
                    add2(e[0], e[1], b[g + (i >> 1)].x, b[g + (i >> 1)].y);
                    w[i] = pack_bf16_relu(e[0], e[1]);
                    if (TRAIN)
                      rows[2 * h + (i & 1)] = mask_add(rows[2 * h + (i & 1)], w[i], g + (i >> 1));
                  }
                  store_frag(fs, cb, h, g, w[0], w[1], w[2], w[3]);
                }
              const int tile = pr * kPair + t;
              if (TRAIN && tile < n_tiles)
                *reinterpret_cast<uint2*>(keep.bits + (size_t)l * keep.Mp * (kW / 32) +
                                          mask_at(tile, q, cb, lane)) =
                    make_uint2(mask_word(rows[0], rows[1]), mask_word(rows[2], rows[3]));
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            epi_sync();
            if (threadIdx.x == 0) mbar_arrive(actr0 + 8 * t);
            if (TRAIN && threadIdx.x == 32 * t && pr * kPair + t < n_tiles) {
              for (int kb = 0; kb < kW / BK; ++kb)
                tma_store_2d(&maps.act, act_s + t * kActBytes + kb * 16384, kb * BK,
                             l * keep.Mp + (pr * kPair + t) * BM);
              bulk_commit();
            }
            // both tiles have taken this layer's bias: the next one's
            if (t == kPair - 1 && l + 1 < kDepth && threadIdx.x < kW)
              s_bias[threadIdx.x] = __ldg(theta + bias_off_dev(l + 1) + threadIdx.x);
          } else {
            if (part == 0) {
              float v[32];
              tmem_ld32(trow, v);
              const float* bias = theta + head_bias_off_dev();
              const int m = (pr * kPair + t) * BM + r;
              if (m < M)
                for (int j = 0; j < 3; ++j) delta[(size_t)m * 3 + j] = v[j] + __ldg(bias + j);
            }
            tc_fence_before();
            epi_sync();  // TMEM drained before the next pair
          }
        }
    }
    if (TRAIN && (threadIdx.x & 31) == 0) bulk_wait_all();  // the stores are done
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, (uint32_t)(kPair * kW));
  }
}

// ---- fused backward: the dZ chain of 128-row tiles kept in shared memory ----
// Step s = 0 forms dZ_7 = (dZ_head W_head) * mask_7 from dL/d(delta); steps
// s = 1..7 form dZ_{7-s} = (dZ_{8-s} W_{8-s}) * mask_{7-s}; step 8 forms the
// encoding's gradient dZ_0 W_0 (FP32).  Each dZ tile goes to shared memory as
// the next step's operand and from there by TMA (maps.act, row-major) to
// global memory for the weight gradients (whose GEMMs also form the bias
// gradients, the column sums).  The same operands and order as the
// one-GEMM-per-layer backward: bit-identical dZ.
constexpr int kBwdStages = kFusedStages;
constexpr int kBwdSmem = kFusedSmem;

struct FusedBwdArgs {
  const float* dd;      // dL/d(delta) [M][3]
  const uint32_t* bits; // ReLU masks, per layer Mp kW / 32 words (mask_at)
  float* denc;          // [Mp][128] (out)
  int M, Mp, n_tiles;
};

__global__ void __launch_bounds__(kFusedThreads, 1)
    mlp_fused_bwd_kernel(const __grid_constant__ FusedMaps maps, const FusedBwdArgs a,
                         int* status, unsigned long long wait_ns, int inject_no_loads) {
  grid_begin();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars =
      reinterpret_cast<uint64_t*>(smem + kPair * kActBytes + kBwdStages * kWStageBytes);
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + 2 * kBwdStages + 2 * kPair);
  int* s_ok = reinterpret_cast<int*>(slot + 1);
  const uint32_t act_s = smem_u32(smem), w_s = act_s + kPair * kActBytes;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kBwdStages;
  const uint32_t acc0 = full0 + 16 * kBwdStages, actr0 = acc0 + 8 * kPair;
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int n_pairs = (a.n_tiles + kPair - 1) / kPair;
  constexpr int kSteps = kDepth + 1;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kBwdStages; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    for (int t = 0; t < kPair; ++t) {
      mbar_init(acc0 + 8 * t, 1);
      mbar_init(actr0 + 8 * t, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(smem_u32(slot), (uint32_t)(kPair * kW));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = (uint32_t)uniform((int)*slot);

  if (warp == kFusedEpiWarps) {
    // W^T of the head (step 0) and of layers 7..0 (steps 1..8)
    if (!inject_no_loads) {
      int it = 0;
      bool ok = true;
      for (int pr = blockIdx.x; ok && pr < n_pairs; pr += gridDim.x)
        for (int st = 0; ok && st < kSteps; ++st)
          for (int t = 0; ok && t < kPair; ++t) {
            const int nkb = st == 0 ? 1 : kW / BK;
            for (int kb = 0; kb < nkb; ++kb, ++it) {
              const int s = it % kBwdStages;
              if (!(ok = warp_ok(mbar_wait(empty0 + 8 * s, ((uint32_t)(it / kBwdStages) & 1u) ^ 1u,
                                           status, wait_ns))))
                break;
              if (elect_one()) {
                mbar_expect_tx(full0 + 8 * s, (uint32_t)kWStageBytes);
                tma_load_2d(w_s + s * kWStageBytes, &maps.w[st == 0 ? kDepth : kDepth - st],
                            full0 + 8 * s, kb * BK, 0);
              }
            }
          }
      for (int i = it - kBwdStages < 0 ? 0 : it - kBwdStages; i < it; ++i)
        mbar_wait(full0 + 8 * (i % kBwdStages), (uint32_t)(i / kBwdStages) & 1u, status,
                  wait_ns);
    }
  } else if (warp == kFusedEpiWarps + 1) {
    {
      int it = 0;
      uint32_t act_ph[kPair] = {0, 0};
      bool ok = true;
      constexpr uint32_t idesc = idesc_bf16(BM, kW);
      for (int pr = blockIdx.x; ok && pr < n_pairs; pr += gridDim.x)
        for (int st = 0; ok && st < kSteps; ++st)
          for (int t = 0; ok && t < kPair; ++t) {
            if (!(ok = warp_ok(mbar_wait(actr0 + 8 * t, act_ph[t], status, wait_ns)))) break;
            act_ph[t] ^= 1u;
            tc_fence_after();
            const int nkb = st == 0 ? 1 : kW / BK;
            const uint32_t d = tmem + (uint32_t)(t * kW);
            for (int kb = 0; kb < nkb; ++kb, ++it) {
              const int s = it % kBwdStages;
              if (!(ok = warp_ok(mbar_wait(full0 + 8 * s, (uint32_t)(it / kBwdStages) & 1u, status,
                                           wait_ns))))
                break;
              tc_fence_after();
              const uint32_t sa = act_s + t * kActBytes + kb * 16384, sb = w_s + s * kWStageBytes;
              if (elect_one()) {
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                  umma_bf16(d, sw128_desc(sa + 32 * k), sw128_desc(sb + 32 * k), idesc,
                            (kb > 0 || k > 0) ? 1u : 0u);
                umma_commit(empty0 + 8 * s);
              }
              __syncwarp();
            }
            if (elect_one()) umma_commit(acc0 + 8 * t);
            __syncwarp();
          }
    }
  } else {
    const int q = warp & 3, part = warp >> 2;
    const int r = q * 32 + lane;
    uint32_t acc_ph[kPair] = {0, 0};
    // the ReLU mask words of this thread's row and columns, one step
    // ahead: a tile's next layer is loaded while this one is processed
    struct Bits {
      uint2 k[kBlocks];
    };
    Bits nb[kPair];
    auto load_bits = [&](int layer, int tile) {
      Bits v;
#pragma unroll
      for (int k = 0; k < kBlocks; ++k)
        v.k[k] = tile < a.n_tiles
                     ? __ldg(reinterpret_cast<const uint2*>(a.bits + (size_t)layer * a.Mp * (kW / 32) +
                                                            mask_at(tile, q, part * kBlocks + k, lane)))
                     : make_uint2(0u, 0u);
      return v;
    };
    bool ok = true;
    for (int pr = blockIdx.x; ok && pr < n_pairs; pr += gridDim.x) {
#pragma unroll
      for (int t = 0; t < kPair; ++t) {
        // step 0's operand: BF16 dL/d(delta) in columns 0..2 of k-block 0
        const int m = (pr * kPair + t) * BM + r;
        nb[t] = load_bits(kDepth - 1, pr * kPair + t);
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = 0.f;
        for (int c = 64 - 16; c > 0; c -= 16)  // (free: waited at step 8)
          if ((c >> 4) % kParts == part) store_act16(smem + t * kActBytes, r, c, v);
        if (part == 0) {
          if (m < a.M)
            for (int j = 0; j < 3; ++j) v[j] = a.dd[(size_t)m * 3 + j];
          store_act16(smem + t * kActBytes, r, 0, v);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        epi_sync();
        if (threadIdx.x == 0) mbar_arrive(actr0 + 8 * t);
      }
      for (int st = 0; ok && st < kSteps; ++st)
#pragma unroll
        for (int t = 0; t < kPair; ++t) {
          if (threadIdx.x == 0)
            *s_ok = mbar_wait(acc0 + 8 * t, acc_ph[t], status, wait_ns) ? 1 : 0;
          // the tile's last store has read it before it is written again
          if (threadIdx.x == 32 * t) bulk_wait_read();
          epi_sync();
          if (!(ok = *s_ok != 0)) break;  // (rewritten only after the step's last barrier)
          acc_ph[t] ^= 1u;
          tc_fence_after();
          const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(t * kW);
          if (st < kDepth) {
            const int j = kDepth - 1 - st;  // the layer whose dZ this step forms
            const FragStore fs = frag_store(act_s + t * kActBytes, q, lane);
            const Bits mk = nb[t];
            if (j > 0) nb[t] = load_bits(j - 1, pr * kPair + t);
#pragma unroll
            for (int k = 0; k < kBlocks; ++k) {
              const int cb = part * kBlocks + k;
              float v[64];
              tmem_ld64_frag(trow + (uint32_t)(cb * 64), v);
              tmem_wait_ld();
#pragma unroll
              for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int g = 0; g < 8; g += 2) {
                  const uint32_t bits = h ? mk.k[k].y : mk.k[k].x;
                  const float* e = v + 32 * h + 4 * g;
                  store_frag(fs, cb, h, g, pack_bf16(e[0], e[1]) & mask_pair<0>(bits, g),
                             pack_bf16(e[2], e[3]) & mask_pair<1>(bits, g),
                             pack_bf16(e[4], e[5]) & mask_pair<0>(bits, g + 1),
                             pack_bf16(e[6], e[7]) & mask_pair<1>(bits, g + 1));
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            epi_sync();
            if (threadIdx.x == 0) mbar_arrive(actr0 + 8 * t);
            if (threadIdx.x == 32 * t && pr * kPair + t < a.n_tiles) {
              for (int kb = 0; kb < kW / BK; ++kb)
                tma_store_2d(&maps.act, act_s + t * kActBytes + kb * 16384, kb * BK,
                             j * a.Mp + (pr * kPair + t) * BM);
              bulk_commit();
            }
          } else {
#pragma unroll 1
            for (int cb = part; cb < kIn / 64; cb += kParts) {
              float v[64];
              tmem_ld64_frag(trow + (uint32_t)(cb * 64), v);
              tmem_wait_ld();
              if (pr * kPair + t < a.n_tiles) {
                float* d = a.denc + ((size_t)(pr * kPair + t) * BM + q * 32 + (lane >> 2)) * kIn +
                           cb * 64 + 2 * (lane & 3);
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                  for (int g = 0; g < 8; ++g)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                      *reinterpret_cast<float2*>(d + (16 * h + 8 * i) * kIn + 8 * g) =
                          make_float2(v[32 * h + 4 * g + 2 * i], v[32 * h + 4 * g + 2 * i + 1]);
              }
            }
            tc_fence_before();
            epi_sync();  // TMEM drained before the next pair
          }
        }
    }
    if ((threadIdx.x & 31) == 0) bulk_wait_all();  // the stores are done
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, (uint32_t)(kPair * kW));
  }
}

// ---- host side -----------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// bf16 matrix [rows][cols] with row stride ld elements; boxes of 64 columns x
// box_rows with the 128-byte swizzle
bool make_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint64_t ld,
              uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(base) & 15) != 0 || (ld * 2) % 16 != 0) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
            es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, int EPI, int MT = 1, int MNA = 0, int MNB = 0>
bool gemm(const CUtensorMap& a, const CUtensorMap& b, const GemmArgs& args, int m_tiles,
          int n_tiles, int splits, cudaStream_t st) {
  constexpr int smem = GemmShape<BN, MT>::SMEM;
  static PerDeviceOnce configured;
  if (!configured.run([] {
        return cudaFuncSetAttribute(umma_gemm_kernel<BN, EPI, MT, MNA, MNB>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    smem) == cudaSuccess;
      }))
    return false;
  launch(umma_gemm_kernel<BN, EPI, MT, MNA, MNB>, dim3(m_tiles, n_tiles, splits), 192, smem, st,
         a, b, args);
  count_launches(1);
  return true;
}

struct MlpLayout {
  int N, B, M, M_pad;
  size_t off_status, off_wb, off_wt, off_enc, off_h, off_bits, off_dz, off_dzh, off_dzht,
      off_denc, off_dwx, off_part, total;
};

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

size_t dwx_floats() {
  return (size_t)kW * (kIn + kExt) + (size_t)(kDepth - 1) * kW * (kW + kExt) +
         (size_t)kHeadRows * (kW + kExt);
}
size_t wb_elems() {
  return (size_t)kW * kIn + (size_t)(kDepth - 1) * kW * kW + (size_t)kHeadRows * kW;
}

MlpLayout mlp_layout(int N, int B) {
  MlpLayout L;
  memset(&L, 0, sizeof(L));
  L.N = N, L.B = B, L.M = N * B;
  L.M_pad = (L.M + BM - 1) / BM * BM;
  if (L.M_pad == 0) L.M_pad = BM;
  const size_t Mp = (size_t)L.M_pad;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at_ = o;
    o = align256(o + bytes);
    return at_;
  };
  L.off_status = take(256);
  L.off_wb = take(wb_elems() * 2);
  L.off_wt = take(wb_elems() * 2);
  L.off_enc = take(Mp * kIn * 2);                   // [Mp][128]
  L.off_h = take((size_t)kDepth * Mp * kW * 2);     // [layer][Mp][256]
  L.off_bits = take((size_t)kDepth * Mp * (kW / 32) * 4);
  L.off_dz = take((size_t)kDepth * Mp * kW * 2);    // [layer][Mp][256]
  L.off_dzh = take(Mp * kHeadRows * 2);
  L.off_dzht = take((size_t)kHeadRows * Mp * 2);
  L.off_denc = take(Mp * kIn * 4);
  L.off_dwx = take(dwx_floats() * 4);
  L.off_part = take((size_t)kMaxSplits * kW * kW * 4);
  L.total = o;
  return L;
}

// rows: below 2^27 (the stores address layer l's rows at l Mp + m with
// 32-bit TMA coordinates)
bool mlp_args_ok(int N, int B) {
  return N >= 0 && B >= 1 && B <= kMaxFrames && (int64_t)N * B < (int64_t)1 << 27;
}

// test hooks (gftorf_mlp_debug_inject): 1 = the GEMMs' load warps issue
// nothing, so the MMA and epilogue waits run out; 2 = the training forward
// and the backward's dZ chain run layer by layer (one GEMM per layer)
// instead of fused
std::atomic<int> g_inject{0};

bool fused_configured() {
  static PerDeviceOnce once;
  return once.run([] {
    return cudaFuncSetAttribute(mlp_fused_fwd_kernel<false>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, kFusedSmem) ==
               cudaSuccess &&
           cudaFuncSetAttribute(mlp_fused_fwd_kernel<true>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, kFusedSmem) ==
               cudaSuccess &&
           cudaFuncSetAttribute(mlp_fused_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kBwdSmem) == cudaSuccess;
  });
}

template <typename T>
T* ptr(void* ws, size_t off) {
  return reinterpret_cast<T*>(static_cast<unsigned char*>(ws) + off);
}

// bf16 weights of layer l (l = kDepth: head) and their transposes
size_t wb_off(int l) {
  return l == 0 ? 0 : (size_t)kW * kIn + (size_t)(l - 1) * kW * kW;
}
size_t bias_off(int l) {  // in the packed fp32 vector
  if (l == 0) return (size_t)kW * kIn;
  return (size_t)kW * kIn + kW + (size_t)(l - 1) * ((size_t)kW * kW + kW) + (size_t)kW * kW;
}
size_t head_bias_off() {
  return (size_t)kW * kIn + kW + (size_t)(kDepth - 1) * ((size_t)kW * kW + kW) + 3 * kW;
}
size_t dwx_off(int l) {  // floats
  if (l == 0) return 0;
  return (size_t)kW * (kIn + kExt) + (size_t)(l - 1) * kW * (kW + kExt);
}

}  // namespace
}  // namespace gftorf

using namespace gftorf;

extern "C" size_t gftorf_mlp_infer_workspace_size(void) {
  return 256 + align256(2 * wb_elems() * 2);  // status word, BF16 weights and transposes
}

extern "C" size_t gftorf_mlp_workspace_size(int32_t n_gaussians, int32_t n_frames) {
  if (!mlp_args_ok(n_gaussians, n_frames)) return 0;
  return mlp_layout(n_gaussians, n_frames).total;
}

extern "C" size_t gftorf_mlp_param_count(void) {
  return (size_t)kW * kIn + kW + (size_t)(kDepth - 1) * ((size_t)kW * kW + kW) + 3 * kW + 3;
}

extern "C" gftorf_status gftorf_mlp_forward(int32_t n_gaussians, int32_t n_frames,
                                            const float* theta, const float* means,
                                            const float* times, float inv_scale, float* delta,
                                            void* workspace, size_t workspace_bytes,
                                            void* stream) {
  gftorf::TraceRange trace_("gftorf_mlp_forward");
  if (!mlp_args_ok(n_gaussians, n_frames) || !theta || !times ||
      (n_gaussians > 0 && (!means || !delta)) || !(inv_scale > 0.f))
    return GFTORF_ERR_ARG;
  const MlpLayout L = mlp_layout(n_gaussians, n_frames);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0 ||
      workspace_bytes < L.total)
    return GFTORF_ERR_WORKSPACE;
  for (int b = 0; b < n_frames; ++b)
    if (!std::isfinite(times[b])) return GFTORF_ERR_ARG;
  if (!encode_fn()) return GFTORF_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  void* ws = workspace;
  const int Mp = L.M_pad;
  int* status = ptr<int>(ws, L.off_status);
  cudaMemsetAsync(status, 0, 256, st);  // the status word of this forward and its backward
  if (L.M == 0) return cudaGetLastError() == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
  auto* wb = ptr<__nv_bfloat16>(ws, L.off_wb);
  auto* wt = ptr<__nv_bfloat16>(ws, L.off_wt);
  launch(mlp_prep_weights_kernel, 4 * kSMs, 256, 0, st, theta, wb, wt);
  Times tm;
  memset(&tm, 0, sizeof(tm));
  for (int b = 0; b < n_frames; ++b) tm.t[b] = times[b];
  auto* enc = ptr<__nv_bfloat16>(ws, L.off_enc);
  auto* H = ptr<__nv_bfloat16>(ws, L.off_h);
  const int mt = Mp / BM;
  if (g_inject.load() != 2) {
    // fused: all layers per pair of 128-row tiles, keeping the encoding, the
    // activations and the ReLU masks for the backward
    if (!fused_configured()) return GFTORF_ERR_CUDA;
    FusedMaps maps;
    for (int l = 0; l <= kDepth; ++l) {
      const int K = l == 0 ? kIn : kW, rows = l == kDepth ? kHeadRows : kW;
      if (!make_map(&maps.w[l], wb + wb_off(l), rows, K, K, rows)) return GFTORF_ERR_CUDA;
    }
    if (!make_map(&maps.enc, enc, Mp, kIn, kIn, BM) ||
        !make_map(&maps.act, H, (uint64_t)kDepth * Mp, kW, kW, BM))
      return GFTORF_ERR_CUDA;
    FusedKeep keep;
    keep.bits = ptr<uint32_t>(ws, L.off_bits), keep.Mp = Mp;
    const int sms = sm_count();
    const int n_pairs = (mt + kPair - 1) / kPair;
    const int inj = g_inject.load();
    launch(mlp_fused_fwd_kernel<true>, n_pairs < sms ? n_pairs : sms, kFusedThreads, kFusedSmem, st,
           maps, theta, means, tm, n_gaussians, L.M, mt, inv_scale, delta, status,
           inj == 1 ? 50000000ull : 2000000000ull, inj == 1, keep);
    count_launches(2);
    return cudaGetLastError() == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
  }
  launch(mlp_encode_kernel, (Mp + 127) / 128, 128, 0, st, means, tm, n_gaussians, n_frames,
         inv_scale, Mp, enc);
  count_launches(2);
  for (int l = 0; l < kDepth; ++l) {
    const int K = l == 0 ? kIn : kW;
    const __nv_bfloat16* in = l == 0 ? enc : H + (size_t)(l - 1) * Mp * kW;
    CUtensorMap ma, mb;
    if (!make_map(&ma, in, Mp, K, K, BM) || !make_map(&mb, wb + wb_off(l), kW, K, K, 256))
      return GFTORF_ERR_CUDA;
    GemmArgs a;
    memset(&a, 0, sizeof(a));
    a.kb_total = K / BK, a.kb_per_split = K / BK;
    a.rows_valid = Mp, a.cols_valid = kW;
    a.bias = theta + bias_off(l);
    a.out_b = H + (size_t)l * Mp * kW, a.ldo = kW;
    a.mbits = ptr<uint32_t>(ws, L.off_bits) + (size_t)l * Mp * (kW / 32);
    a.status = status;
    a.inject_no_loads = g_inject.load(std::memory_order_relaxed) == 1;
    a.wait_ns = a.inject_no_loads ? 50000000ull : 2000000000ull;
    if (!gemm<256, EPI_HIDDEN>(ma, mb, a, mt, 1, 1, st)) return GFTORF_ERR_CUDA;
  }
  {
    CUtensorMap ma, mb;
    if (!make_map(&ma, H + (size_t)(kDepth - 1) * Mp * kW, Mp, kW, kW, BM) ||
        !make_map(&mb, wb + wb_off(kDepth), kHeadRows, kW, kW, kHeadRows))
      return GFTORF_ERR_CUDA;
    GemmArgs a;
    memset(&a, 0, sizeof(a));
    a.kb_total = kW / BK, a.kb_per_split = kW / BK;
    a.rows_valid = L.M, a.cols_valid = 3;
    a.bias = theta + head_bias_off();
    a.out_f = delta;
    a.status = status;
    a.inject_no_loads = g_inject.load(std::memory_order_relaxed) == 1;
    a.wait_ns = a.inject_no_loads ? 50000000ull : 2000000000ull;
    if (!gemm<32, EPI_HEAD>(ma, mb, a, mt, 1, 1, st)) return GFTORF_ERR_CUDA;
  }
  return cudaGetLastError() == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
}

extern "C" gftorf_status gftorf_mlp_backward(int32_t n_gaussians, int32_t n_frames,
                                             const float* theta, const float* means,
                                             const float* times, float inv_scale,
                                             const float* d_delta, float* d_theta,
                                             float* d_means, void* workspace,
                                             size_t workspace_bytes, void* stream) {
  gftorf::TraceRange trace_("gftorf_mlp_backward");
  if (!mlp_args_ok(n_gaussians, n_frames) || !theta || !times || !d_theta ||
      (n_gaussians > 0 && (!means || !d_means || !d_delta)) || !(inv_scale > 0.f))
    return GFTORF_ERR_ARG;
  const MlpLayout L = mlp_layout(n_gaussians, n_frames);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0 ||
      workspace_bytes < L.total)
    return GFTORF_ERR_WORKSPACE;
  if (!encode_fn()) return GFTORF_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  void* ws = workspace;
  const int Mp = L.M_pad;
  int* status = ptr<int>(ws, L.off_status);
  float* dwx = ptr<float>(ws, L.off_dwx);
  cudaMemsetAsync(dwx, 0, dwx_floats() * 4, st);
  if (L.M == 0) {
    launch(mlp_unpack_grads_kernel, 4 * kSMs, 256, 0, st, dwx, d_theta);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
  }
  auto* wt = ptr<__nv_bfloat16>(ws, L.off_wt);
  auto* enc = ptr<__nv_bfloat16>(ws, L.off_enc);
  auto H = [&](int l) { return ptr<__nv_bfloat16>(ws, L.off_h) + (size_t)l * Mp * kW; };
  auto* bits = ptr<uint32_t>(ws, L.off_bits);
  auto* dzh = ptr<__nv_bfloat16>(ws, L.off_dzh);
  auto* dzht = ptr<__nv_bfloat16>(ws, L.off_dzht);
  auto dz = [&](int l) { return ptr<__nv_bfloat16>(ws, L.off_dz) + (size_t)l * Mp * kW; };
  float* denc = ptr<float>(ws, L.off_denc);
  const int mt = Mp / BM;
  const int kb_rows = Mp / BK;      // k-blocks of a reduction over the batch rows
  // weight-gradient GEMMs: one CTA per SM (TMEM-bound), the rows split evenly
  const int sms = sm_count();
  const int per_split = max(8, (kb_rows + min(sms, kMaxSplits) - 1) / min(sms, kMaxSplits));
  const int splits = (kb_rows + per_split - 1) / per_split;  // <= kMaxSplits
  float* part = ptr<float>(ws, L.off_part);

  // bias gradient of a layer: column K of its dW block
  auto dbias_of = [&](int l) { return dwx + dwx_off(l) + (l == 0 ? kIn : kW); };
  auto ldb_of = [&](int l) { return (l == 0 ? kIn : kW) + kExt; };
  const bool inj_loads = g_inject.load(std::memory_order_relaxed) == 1;
  const unsigned long long wait_ns = inj_loads ? 50000000ull : 2000000000ull;
  const bool layerwise = g_inject.load(std::memory_order_relaxed) == 2;
  launch(mlp_head_grad_kernel, min((Mp + kHeadGradThreads - 1) / kHeadGradThreads, 4 * sms),
         kHeadGradThreads, 0, st, d_delta, L.M, Mp, layerwise ? dzh : nullptr, dzht,
         dbias_of(kDepth), kW + kExt);
  count_launches(1);
  // head: dW_head += dZh^T H_7 (H_7 read MN-major)
  {
    CUtensorMap ma, mb;
    if (!make_map(&ma, dzht, 3, Mp, Mp, BM) ||
        !make_map(&mb, H(kDepth - 1), Mp, kW, kW, BK))
      return GFTORF_ERR_CUDA;
    GemmArgs a;
    memset(&a, 0, sizeof(a));
    a.kb_total = kb_rows, a.kb_per_split = per_split;
    a.rows_valid = 3, a.cols_valid = kW;
    a.out_f = dwx + dwx_off(kDepth), a.ldf = kW + kExt;
    a.status = status, a.inject_no_loads = inj_loads, a.wait_ns = wait_ns;
    if (!gemm<256, EPI_ATOMIC, 1, 0, 1>(ma, mb, a, 1, 1, splits, st)) return GFTORF_ERR_CUDA;
  }
  if (!layerwise) {
    // fused dZ chain: all layers per pair of 128-row tiles, dZ_l kept in
    // shared memory as the next layer's operand and stored (row-major) for
    // the weight gradients below
    if (!fused_configured()) return GFTORF_ERR_CUDA;
    FusedMaps maps;
    if (!make_map(&maps.w[kDepth], wt + wb_off(kDepth), kW, kHeadRows, kHeadRows, 256))
      return GFTORF_ERR_CUDA;
    for (int l = 0; l < kDepth; ++l)
      if (!make_map(&maps.w[l], wt + wb_off(l), l == 0 ? kIn : kW, kW, kW, 256))
        return GFTORF_ERR_CUDA;
    if (!make_map(&maps.act, dz(0), (uint64_t)kDepth * Mp, kW, kW, BM)) return GFTORF_ERR_CUDA;
    FusedBwdArgs fa;
    memset(&fa, 0, sizeof(fa));
    fa.dd = d_delta, fa.bits = bits, fa.denc = denc;
    fa.M = L.M, fa.Mp = Mp, fa.n_tiles = mt;
    const int n_pairs = (mt + kPair - 1) / kPair;
    launch(mlp_fused_bwd_kernel, n_pairs < sms ? n_pairs : sms, kFusedThreads, kBwdSmem, st,
        maps, fa, status, wait_ns, inj_loads);
    count_launches(1);
  } else {
    // dH_7 = dZh W_head, dZ_7 = dH_7 * (H_7 > 0); then dH_{l-1} = dZ_l W_l
    // (l = 0: the encoding's gradient, FP32), one GEMM per layer
    for (int l = kDepth; l >= 1; --l) {
      const int K = l == kDepth ? kHeadRows : kW;
      CUtensorMap ma, mb;
      if (!make_map(&ma, l == kDepth ? dzh : dz(l), Mp, K, K, BM) ||
          !make_map(&mb, wt + wb_off(l), l == 0 ? kIn : kW, K, K, 256))
        return GFTORF_ERR_CUDA;
      GemmArgs a;
      memset(&a, 0, sizeof(a));
      a.kb_total = l == kDepth ? 1 : kW / BK, a.kb_per_split = a.kb_total;
      a.rows_valid = Mp, a.cols_valid = kW;
      a.out_b = dz(l - 1), a.ldo = kW;
      a.mbits = bits + (size_t)(l - 1) * Mp * (kW / 32);
      a.status = status, a.inject_no_loads = inj_loads, a.wait_ns = wait_ns;
      if (!gemm<256, EPI_MASK>(ma, mb, a, mt, 1, 1, st)) return GFTORF_ERR_CUDA;
    }
    CUtensorMap ma, mb;
    if (!make_map(&ma, dz(0), Mp, kW, kW, BM) || !make_map(&mb, wt, kIn, kW, kW, 256))
      return GFTORF_ERR_CUDA;
    GemmArgs a;
    memset(&a, 0, sizeof(a));
    a.kb_total = kW / BK, a.kb_per_split = kW / BK;
    a.rows_valid = Mp, a.cols_valid = kIn;
    a.out_f = denc, a.ldf = kIn;
    a.status = status, a.inject_no_loads = inj_loads, a.wait_ns = wait_ns;
    if (!gemm<256, EPI_F32>(ma, mb, a, mt, 1, 1, st)) return GFTORF_ERR_CUDA;
  }
  // dW_l += dZ_l^T H_{l-1} (or the encoding): all 256 output rows per CTA,
  // both operands read MN-major from the row-major dZ_l and H_{l-1}
  for (int l = kDepth - 1; l >= 0; --l) {
    const int K = l == 0 ? kIn : kW;
    CUtensorMap ma, mb;
    if (!make_map(&ma, dz(l), Mp, kW, kW, BK) ||
        !make_map(&mb, l == 0 ? enc : H(l - 1), Mp, K, K, BK))
      return GFTORF_ERR_CUDA;
    GemmArgs a;
    memset(&a, 0, sizeof(a));
    a.kb_total = kb_rows, a.kb_per_split = per_split;
    a.rows_valid = kW, a.cols_valid = K;
    a.out_f = part, a.ldf = K;
    a.dbias = dbias_of(l), a.ldb = ldb_of(l);  // the column sums of dZ_l
    a.status = status, a.inject_no_loads = inj_loads, a.wait_ns = wait_ns;
    if (!(l == 0 ? gemm<kIn, EPI_PARTIAL, 2, 1, 1>(ma, mb, a, 1, 1, splits, st)
                 : gemm<kW, EPI_PARTIAL, 2, 1, 1>(ma, mb, a, 1, 1, splits, st)))
      return GFTORF_ERR_CUDA;
    launch(mlp_reduce_dw_kernel, kW * K / 128, 32 * kReduceWarps, 0, st, part, splits, K,
           dwx + dwx_off(l), K + kExt);
    count_launches(1);
  }
  launch(mlp_unpack_grads_kernel, 4 * kSMs, 256, 0, st, dwx, d_theta);
  launch(mlp_encode_bwd_kernel, (n_gaussians + 63) / 64, 128, 0, st, means, denc, n_gaussians,
         n_frames, inv_scale, d_means);
  count_launches(2);
  (void)times;
  return cudaGetLastError() == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
}

extern "C" gftorf_status gftorf_mlp_read_status(void* workspace, size_t workspace_bytes,
                                                void* stream) {
  if (!workspace || workspace_bytes < 256) return GFTORF_ERR_WORKSPACE;
  int s = 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaMemcpyAsync(&s, workspace, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return GFTORF_ERR_CUDA;
  return (gftorf_status)s;
}

extern "C" gftorf_status gftorf_mlp_export(int32_t n_gaussians, int32_t n_frames, int32_t what,
                                           int32_t layer, void* dst, void* workspace,
                                           size_t workspace_bytes, void* stream) {
  if (!mlp_args_ok(n_gaussians, n_frames) || !dst) return GFTORF_ERR_ARG;
  const MlpLayout L = mlp_layout(n_gaussians, n_frames);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0 ||
      workspace_bytes < L.total)
    return GFTORF_ERR_WORKSPACE;
  const size_t Mp = (size_t)L.M_pad, M = (size_t)L.M;
  size_t off, bytes;
  if ((what == 1 || what == 2) && (layer < 0 || layer >= kDepth)) return GFTORF_ERR_ARG;
  switch (what) {
    case 0: off = L.off_enc, bytes = M * kIn * 2; break;
    case 1: off = L.off_h + (size_t)layer * Mp * kW * 2, bytes = M * kW * 2; break;
    case 2: off = L.off_dz + (size_t)layer * Mp * kW * 2, bytes = M * kW * 2; break;
    case 3: off = L.off_denc, bytes = M * kIn * 4; break;
    default: return GFTORF_ERR_ARG;
  }
  if (bytes == 0) return GFTORF_OK;
  const cudaError_t e =
      cudaMemcpyAsync(dst, static_cast<unsigned char*>(workspace) + off, bytes,
                      cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
}

extern "C" void gftorf_mlp_debug_inject(int32_t mode) {
  g_inject.store(mode == 1 || mode == 2 ? mode : 0, std::memory_order_relaxed);
}

extern "C" gftorf_status gftorf_mlp_infer(int32_t n_gaussians, int32_t n_frames,
                                          const float* theta, const float* means,
                                          const float* times, float inv_scale, float* delta,
                                          void* workspace, size_t workspace_bytes, void* stream) {
  gftorf::TraceRange trace_("gftorf_mlp_infer");
  if (!mlp_args_ok(n_gaussians, n_frames) || !theta || !times ||
      (n_gaussians > 0 && (!means || !delta)) || !(inv_scale > 0.f))
    return GFTORF_ERR_ARG;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0 ||
      workspace_bytes < gftorf_mlp_infer_workspace_size())
    return GFTORF_ERR_WORKSPACE;
  for (int b = 0; b < n_frames; ++b)
    if (!std::isfinite(times[b])) return GFTORF_ERR_ARG;
  if (!encode_fn()) return GFTORF_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int* status = ptr<int>(workspace, 0);
  cudaMemsetAsync(status, 0, 256, st);
  const int M = n_gaussians * n_frames;
  if (M == 0) return cudaGetLastError() == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
  auto* wb = ptr<__nv_bfloat16>(workspace, 256);
  auto* wt = wb + wb_elems();
  launch(mlp_prep_weights_kernel, 4 * kSMs, 256, 0, st, theta, wb, wt);
  FusedMaps maps;
  for (int l = 0; l <= kDepth; ++l) {
    const int K = l == 0 ? kIn : kW, rows = l == kDepth ? kHeadRows : kW;
    if (!make_map(&maps.w[l], wb + wb_off(l), rows, K, K, rows)) return GFTORF_ERR_CUDA;
  }
  Times tm;
  memset(&tm, 0, sizeof(tm));
  for (int b = 0; b < n_frames; ++b) tm.t[b] = times[b];
  if (!fused_configured()) return GFTORF_ERR_CUDA;
  const int sms = sm_count();
  const int n_tiles = (M + BM - 1) / BM;
  const int n_pairs = (n_tiles + kPair - 1) / kPair;
  const unsigned long long wait_ns = g_inject.load() == 1 ? 50000000ull : 2000000000ull;
  FusedKeep none;
  memset(&none, 0, sizeof(none));
  launch(mlp_fused_fwd_kernel<false>, n_pairs < sms ? n_pairs : sms, kFusedThreads, kFusedSmem, st,
      maps, theta, means, tm, n_gaussians, M, n_tiles, inv_scale, delta, status, wait_ns,
      g_inject.load() == 1, none);
  count_launches(2);
  return cudaGetLastError() == cudaSuccess ? GFTORF_OK : GFTORF_ERR_CUDA;
}
