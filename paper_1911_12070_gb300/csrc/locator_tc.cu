// locator_tc.cu -- the learned locator's network on the 5th-generation tensor
// cores (tcgen05, accumulators in tensor memory): the whole 128-256-256-3
// network fused per 128-row tile (tc_mlp_kernel, warp-specialised; its design
// is described at its definition) and the training step (train_*_kernel).
//
// W1 and W2 are kept in global memory in the canonical K-major layout without
// swizzle (w1c, w2c; canon_index): 8 x 8 core matrices of 128 contiguous bytes
// (8 rows of 16 bytes), core matrix (r / 8, k / 8) at ((r / 8) (K / 8) + k / 8)
// 128 bytes, so the leading-dimension offset (next core matrix along K) is 128
// bytes and the stride offset (next 8-row group) is 16 K bytes, and a CTA
// takes each by plain bulk copies.  One elected thread
// issues the tcgen05.mma instructions and commits them to mbarriers; warps
// read their 32 TMEM lanes back with tcgen05.ld.  Accumulator columns are
// allocated once per CTA and freed before exit; every mbarrier wait is
// bounded and sets a status flag on timeout.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "qtv_internal.cuh"
#include "sweep_common.cuh"

namespace qtv {
namespace {

using namespace sweep;

constexpr int TM = 128;   // rows per tile (M of one instruction, TMEM lanes)

__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// shared-memory matrix descriptor: no swizzle, K-major
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo & 0x3FFFFu) >> 4) << 16;
  d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of the 5th-generation tensor cores
  return d;                // base offset 0, swizzle none
}

// One contiguous piece (a multiple of 16 bytes) global -> shared, completion
// counted in bytes on bar, in copies of at most 32 KB.
__device__ __forceinline__ void bulk_load(unsigned char* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  for (uint32_t o = 0; o < bytes; o += 32768u)
    bulk_g2s(dst + o, reinterpret_cast<const unsigned char*>(src) + o, min(32768u, bytes - o), bar);
}
// shared -> global; the issuing thread's commit group
__device__ __forceinline__ void bulk_store(void* dst, const unsigned char* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
               "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the shared memory of this thread's committed stores has been read / the
// stores are complete
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ---------------------------------------------------------------------------
// The whole network for 128-row tiles: Y[M][3] = W3 relu(W2 relu(W1 x + b1) +
// b2) + b3, one persistent CTA per SM.  W1 (64 KB) and W2 (128 KB) stay in
// shared memory in the no-swizzle layout above, with b1[0..127] and w3 rows
// 0 and 1; per tile the 128 X rows (32 KB) arrive by two tensor copies
// (cp.async.bulk.tensor, 64 columns each) in the 128-byte-swizzle K-major
// layout.  Tensor memory (512 columns) holds four 128-column quarters:
//   Q0, Q1  layer 1, hidden units 0..127 and 128..255 (FP32); epilogue 1
//           packs relu(. + b1) as BF16 pairs into the first 64 columns of
//           its own quarter (row = lane, two consecutive K values a column)
//   Q2, Q3  layer 2, outputs 0..127 and 128..255 (FP32)
// and every product is M = 128, N = 128, K = 16 so that the epilogues
// overlap the tensor cores.  Per tile t the issuing thread runs
//   L1(Q0) | L1(Q1) | L2(Q2, K 0..127) | L2(Q3, K 0..127) | L2(Q2, K 128..255)
//   L2(Q3, K 128..255)
// where each "|" waits for what the next products read or overwrite: this
// tile's X and layer 2 of t - 1 done with Q0; layer 2 of t - 1 done with Q1;
// epilogue 1 of Q0 and epilogue 2 of t - 1 done with Q2; epilogue 2 of t - 1
// done with Q3; epilogue 1 of Q1.  So epilogue 1 of Q0 runs beside L1(Q1),
// epilogue 1 of Q1 beside the first K half of layer 2, and epilogue 2 of t
// beside layer 1 and the first K half of layer 2 of t + 1; the tensor cores
// wait only for the part of epilogue 1 of Q0 that outlasts L1(Q1).
// Warp roles (14 warps; warp w reaches TMEM lanes 32 (w % 4) ..):
//   0-3    epilogue 1 (bias, ReLU, BF16 pairs) of Q0 and Q1
//   4-7    epilogue 2 of Q2 (hidden units 0..127): Y = partial + b3
//   8-11   epilogue 2 of Q3 (128..255): Y += partial, after warps 4-7
//   12     the issuing thread (tcgen05.mma, tcgen05.commit)
//   13     the X copies, once layer 1 of the previous tile has read X
// Epilogue 2 reads TMEM in the 16x256b shape, where a thread holds two
// adjacent hidden units of four rows, so each weight it loads serves four
// rows.  The epilogues use packed FP32 pair arithmetic (add/fma .f32x2) and
// round with cvt.rn.relu.bf16x2, which clamps at zero as relu followed by
// rounding does.  Every wait is bounded: a thread whose wait runs out stops
// waiting, the kernel finishes on junk in bounds and the status word is set.
// ---------------------------------------------------------------------------
constexpr uint32_t kMlpSmemW1 = 256 * 128 * 2, kMlpSmemW2 = 256 * 256 * 2, kMlpSmemX = 128 * 128 * 2;
constexpr int kMlpThreads = 448;  // 14 warps (roles above)
constexpr uint32_t kMlpBars = 16;  // 8-byte slots: 14 mbarriers, the TMEM base, padding
constexpr uint32_t kMlpSmemBias = (128 + 512) * sizeof(float);  // b1[0 .. 127], w3 rows 0 and 1
constexpr size_t kMlpSmem = (size_t)kMlpSmemW1 + kMlpSmemW2 + kMlpSmemX + 8 * kMlpBars + kMlpSmemBias;
static_assert(kMlpSmem <= 227 * 1024, "fused network shared memory");
// instruction descriptor of kind::f16 for M = 128, N = 128
constexpr uint32_t kIdesc128 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) |
                               ((uint32_t)(TM >> 4) << 24);

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// as tmem_ld32 without the wait (complete with tmem_ld_wait before use)
__device__ __forceinline__ void tmem_ld32_nowait(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
      "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
      "r"(v[15])
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void mma_ss_i(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_ts_i(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// (o0, o1) = (a0 + b0, a1 + b1), one packed FP32 instruction, IEEE rounding per element
__device__ __forceinline__ void add_x2(float& o0, float& o1, float a0, float a1, float b0, float b1) {
  asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
      " add.rn.f32x2 d, a, b;\n mov.b64 {%0, %1}, d;\n}"
      : "=f"(o0), "=f"(o1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// (d0, d1) += (a0 b0, a1 b1), fused per element
__device__ __forceinline__ void fma_x2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
      " mov.b64 c, {%0, %1};\n fma.rn.f32x2 c, a, b, c;\n mov.b64 {%0, %1}, c;\n}"
      : "+f"(d0), "+f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// BF16 pair (lo in the low half) of max(lo, 0), max(hi, 0), round to nearest even
__device__ __forceinline__ uint32_t relu_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// epilogue 1 of one quarter for this warp's 32 rows: columns q .. q + 127 of
// tensor memory (q = the quarter's first column, lane offset included) hold
// layer-1 sums of 128 hidden units; relu(. + b) as BF16 pairs goes to
// columns q .. q + 63, one 32-column block at a time.  b comes from shared
// memory, or (global) from global memory, one coalesced load a block
// broadcast by shuffles.
__device__ __forceinline__ void mlp_epilogue1(uint32_t q, const float* __restrict__ sb, bool global) {
  uint32_t va[32], vb[32];
  tmem_ld32_nowait(q, va);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t* v = (j & 1) ? vb : va;
    tmem_ld_wait();
    // block j + 1 (columns 32 j + 32 ..) is requested before block j is packed
    // into columns 16 j .. 16 j + 15, which blocks 0 .. j have already read
    if (j < 3) tmem_ld32_nowait(q + 32u * (j + 1), (j & 1) ? va : vb);
    uint32_t pk[16];
    // from global memory: lane i loads the bias of column 32 j + i (one
    // coalesced request) and shuffles broadcast it
    const float lb = global ? __ldg(sb + 32 * j + (threadIdx.x & 31)) : 0.f;
#pragma unroll
    for (int c = 0; c < 32; c += 4) {
      float4 b;
      if (global) {
        b.x = __shfl_sync(0xffffffffu, lb, c);
        b.y = __shfl_sync(0xffffffffu, lb, c + 1);
        b.z = __shfl_sync(0xffffffffu, lb, c + 2);
        b.w = __shfl_sync(0xffffffffu, lb, c + 3);
      } else {
        b = *reinterpret_cast<const float4*>(sb + 32 * j + c);
      }
      float a0, a1, a2, a3;
      add_x2(a0, a1, __uint_as_float(v[c]), __uint_as_float(v[c + 1]), b.x, b.y);
      add_x2(a2, a3, __uint_as_float(v[c + 2]), __uint_as_float(v[c + 3]), b.z, b.w);
      pk[c / 2] = relu_bf16x2(a0, a1);
      pk[c / 2 + 1] = relu_bf16x2(a2, a3);
    }
    tmem_st16(q + 16u * j, pk);
  }
}

// tcgen05.ld .16x256b.x4: 16 lanes from the lane of taddr, 32 columns.  For
// column group k (columns 8 k .. 8 k + 7) thread t receives v[4 k], v[4 k + 1]
// = lane t / 4, columns 8 k + 2 (t % 4) and the next one, and v[4 k + 2],
// v[4 k + 3] = lane t / 4 + 8, the same two columns
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// epilogue 2 of one quarter in the 16x256b fragment layout: each thread holds
// two adjacent hidden units of four rows (lanes t/4, t/4 + 8, t/4 + 16,
// t/4 + 24 of the warp's 32), so every weight it loads serves four rows.
// Columns q .. q + 127 hold layer-2 sums of the hidden units h0 .. h0 + 127;
// y[6 i + 2 o], y[6 i + 2 o + 1] are the even and odd partial sums of output
// o for row i.  w3 rows 0 and 1 come from shared memory (sw3), b2 and w3
// row 2 from global memory.
__device__ __forceinline__ void mlp_epilogue2(uint32_t q, const float* __restrict__ sw3,
                                              const float* __restrict__ b2,
                                              const float* __restrict__ w3, int h0, float* y) {
  const int cq = 2 * (threadIdx.x & 3);
  uint32_t va[32], vb[32];
  tmem_ld_16x256b_x4(q, va);
  tmem_ld_16x256b_x4(q + (16u << 16), va + 16);
#pragma unroll
  for (int cc = 0; cc < 4; ++cc) {
    uint32_t* v = (cc & 1) ? vb : va;
    tmem_ld_wait();
    if (cc < 3) {
      uint32_t* n = (cc & 1) ? va : vb;
      tmem_ld_16x256b_x4(q + 32u * (cc + 1), n);
      tmem_ld_16x256b_x4(q + (16u << 16) + 32u * (cc + 1), n + 16);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int h = h0 + 32 * cc + 8 * k + cq;
      const float2 bb = __ldg(reinterpret_cast<const float2*>(b2 + h));
      const float2 u0 = *reinterpret_cast<const float2*>(sw3 + h);
      const float2 u1 = *reinterpret_cast<const float2*>(sw3 + 256 + h);
      const float2 u2 = __ldg(reinterpret_cast<const float2*>(w3 + 512 + h));
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // row i: lanes t/4 (i = 0), t/4 + 8 (1) of the first load, t/4 + 16 (2), t/4 + 24 (3)
        const uint32_t* p = v + (i >> 1) * 16 + 4 * k + 2 * (i & 1);
        float a0, a1;
        add_x2(a0, a1, __uint_as_float(p[0]), __uint_as_float(p[1]), bb.x, bb.y);
        a0 = fmaxf(a0, 0.f);
        a1 = fmaxf(a1, 0.f);
        fma_x2(y[6 * i], y[6 * i + 1], u0.x, u0.y, a0, a1);
        fma_x2(y[6 * i + 2], y[6 * i + 3], u1.x, u1.y, a0, a1);
        fma_x2(y[6 * i + 4], y[6 * i + 5], u2.x, u2.y, a0, a1);
      }
    }
  }
}

// the three outputs of row i of this thread's four (lane t/4 + 8 i of the
// warp's 32): the partial sums of the four threads t & ~3 .. t | 3 added
__device__ __forceinline__ void mlp_outputs(const float* y, float* out) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      float s = y[6 * i + 2 * o] + y[6 * i + 2 * o + 1];
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      out[3 * i + o] = s;
    }
  }
}

// rows y .. y + 127, columns x .. x + 63 of X by one tensor copy in the
// 128-byte swizzle: row r lands at 128 r bytes with its 16-byte pieces
// permuted by r % 8 (the K-major 128-byte-swizzle operand layout); completion
// counted in bytes on bar.  Rows past the matrix read as zero.
__device__ __forceinline__ void tma_load_x(void* dst, const CUtensorMap* map, int x, int y,
                                           uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

__global__ void __launch_bounds__(kMlpThreads, 1) tc_mlp_kernel(
    const __grid_constant__ CUtensorMap xmap, long long M, const uint16_t* __restrict__ W1,
    const uint16_t* __restrict__ W2, const float* __restrict__ b1, const float* __restrict__ b2,
    const float* __restrict__ w3, const float* __restrict__ b3, float* __restrict__ Y,
    unsigned int* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  unsigned char* sW1 = dsm;
  unsigned char* sW2 = dsm + kMlpSmemW1;
  unsigned char* sX = sW2 + kMlpSmemW2;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sX + kMlpSmemX);
  uint64_t* bar_l1a = bars + 0;   // layer 1 of the tile into Q0 done
  uint64_t* bar_l1b = bars + 1;   // layer 1 into Q1 done
  uint64_t* bar_k0 = bars + 2;    // layer 2 has read the first K half (Q0 free)
  uint64_t* bar_l2a = bars + 3;   // layer 2 into Q2 done
  uint64_t* bar_l2b = bars + 4;   // layer 2 into Q3 done (all of layer 2: Q1 free)
  uint64_t* bar_e1a = bars + 5;   // epilogue 1 wrote the BF16 pairs of Q0 (one arrival per warp)
  uint64_t* bar_e1b = bars + 6;   // epilogue 1 wrote those of Q1
  uint64_t* bar_e2a = bars + 7;   // epilogue 2 has read Q2
  uint64_t* bar_e2b = bars + 8;   // epilogue 2 has read Q3
  uint64_t* bar_xr = bars + 9;    // the next tile's X is in shared memory
  uint64_t* bar_ya = bars + 10;   // the first epilogue-2 group wrote its part of Y
  uint64_t* bar_fin = bars + 11;  // every product issued has completed
  uint64_t* bar_w = bars + 12;    // W1 is in shared memory
  uint64_t* bar_w2 = bars + 13;   // W2
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 14);
  float* sb1 = reinterpret_cast<float*>(bars + kMlpBars);  // b1[0 .. 127]
  float* sw3 = sb1 + 128;                                   // w3 rows 0 and 1
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int wq = w & 3;  // TMEM lane quarter (rows 32 wq .. 32 wq + 31)

  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < 5; ++i) mbar_init(bars + i, 1u);
    for (int i = 5; i < 9; ++i) mbar_init(bars + i, 4u);
    mbar_init(bar_xr, 1u);
    mbar_init(bar_ya, 4u);
    mbar_init(bar_fin, 1u);
    mbar_init(bar_w, 1u);
    mbar_init(bar_w2, 1u);
    fence_mbar_init();
    mbar_arrive_expect_tx(bar_w, kMlpSmemW1);
    bulk_load(sW1, W1, kMlpSmemW1, bar_w);
    mbar_arrive_expect_tx(bar_w2, kMlpSmemW2);
    bulk_load(sW2, W2, kMlpSmemW2, bar_w2);
  }
  if (tid < 128) sb1[tid] = __ldg(b1 + tid);
  for (int i = tid; i < 512; i += kMlpThreads) sw3[i] = __ldg(w3 + i);
  const long long ntiles = (M + TM - 1) / TM;
  fence_proxy_async();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const uint32_t lane_off = (uint32_t)(32 * wq) << 16;
  // a thread whose bounded wait has run out stops waiting: the rest of the
  // kernel runs unsynchronised (in bounds, on junk) and the status flags it
  bool tmo = false;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!tmo && !mbar_wait(bar, parity)) tmo = true;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  auto arrive = [&](uint64_t* bar) {  // one arrival per warp, after the warp's tensor-memory accesses
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };

  if (w == 12) {
    // the issuing thread: per tile 16 layer-1 and 32 layer-2 products (M = 128, N = 128, K = 16)
    if (lane == 0) {
      // X in two 128-byte-swizzled halves (K 0..63, 64..127) of 16 KB: 8-row
      // groups 1024 bytes apart; a K step of 16 moves the start by 32 bytes
      const uint64_t xdesc = smem_desc(smem_u32(sX), 16u, 1024u) | ((uint64_t)2 << 61);
      const uint64_t w1d0 = smem_desc(smem_u32(sW1), 128u, 16u * 128u);
      const uint64_t w1d1 = smem_desc(smem_u32(sW1 + 16 * 16 * 128), 128u, 16u * 128u);
      const uint64_t w2d0 = smem_desc(smem_u32(sW2), 128u, 32u * 128u);
      const uint64_t w2d1 = smem_desc(smem_u32(sW2 + 16 * 32 * 128), 128u, 32u * 128u);
      auto layer1 = [&](int n) {  // Q_n = X W1[128 n .. 128 n + 127]^T
        const uint64_t wd = n ? w1d1 : w1d0;
#pragma unroll
        for (int kb = 0; kb < 8; ++kb)
          mma_ss_i(tmem + 128u * n, xdesc + (uint64_t)((kb >> 2) * 1024 + (kb & 3) * 2),
                   wd + (uint64_t)(kb * 16),
                   kIdesc128, kb > 0 ? 1u : 0u);
      };
      auto layer2 = [&](int n, int k) {  // Q_{2+n} += A1 (K half k, in Q_k) W2[128 n .., 128 k ..]^T
        const uint64_t wd = (n ? w2d1 : w2d0) + (uint64_t)(k * 128);
#pragma unroll
        for (int kb = 0; kb < 8; ++kb)
          mma_ts_i(tmem + 256u + 128u * n, tmem + 128u * k + 8u * kb, wd + (uint64_t)(kb * 16),
                   kIdesc128, (k > 0 || kb > 0) ? 1u : 0u);
      };
      uint32_t ph = 0;
      int it = 0;
      for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ph ^= 1u, ++it) {
        wait(bar_xr, ph);                    // this tile's X
        if (it == 0) wait(bar_w, 0u);
        if (it > 0) wait(bar_k0, ph ^ 1u);  // the previous tile's layer 2 done with Q0
        layer1(0);
        mma_commit(bar_l1a);
        if (it > 0) wait(bar_l2b, ph ^ 1u);  // ... and with Q1
        layer1(1);
        mma_commit(bar_l1b);
        wait(bar_e1a, ph);
        if (it == 0) wait(bar_w2, 0u);
        if (it > 0) wait(bar_e2a, ph ^ 1u);  // the previous tile's epilogue 2 has read Q2
        layer2(0, 0);
        if (it > 0) wait(bar_e2b, ph ^ 1u);  // ... and Q3
        layer2(1, 0);
        mma_commit(bar_k0);
        wait(bar_e1b, ph);
        layer2(0, 1);
        mma_commit(bar_l2a);
        layer2(1, 1);
        mma_commit(bar_l2b);
      }
      // every product has completed before the columns are freed
      mma_commit(bar_fin);
      if (!mbar_wait(bar_fin, 0u)) tmo = true;
    }
  } else if (w == 13) {
    // the X copies: two tensor copies of 128 rows x 64 columns per tile,
    // issued once both layer-1 halves of the previous tile have read X
    if (lane == 0) {
      uint32_t ph = 0;
      int it = 0;
      for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ph ^= 1u, ++it) {
        if (it > 0) wait(bar_l1b, ph ^ 1u);
        mbar_arrive_expect_tx(bar_xr, kMlpSmemX);
        tma_load_x(sX, &xmap, 0, (int)(tile * TM), bar_xr);
        tma_load_x(sX + kMlpSmemX / 2, &xmap, 64, (int)(tile * TM), bar_xr);
      }
    }
  } else if (w < 4) {
    // epilogue 1 of both halves
    uint32_t ph = 0;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ph ^= 1u) {
      wait(bar_l1a, ph);
      __syncwarp();
      mlp_epilogue1(tmem + lane_off, sb1, false);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      arrive(bar_e1a);
      wait(bar_l1b, ph);
      __syncwarp();
      mlp_epilogue1(tmem + lane_off + 128u, b1 + 128, true);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      arrive(bar_e1b);
    }
  } else {
    // epilogue 2: warps 4-7 the hidden units 0..127 (Q2), which write
    // Y = their partial sums + b3; warps 8-11 those of 128..255 (Q3), which
    // add theirs once the first group's are in Y
    const bool upper = w >= 8;
    uint32_t ph = 0;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ph ^= 1u) {
      // this thread writes row lane / 4 + 8 (lane % 4) of the warp's 32
      const long long row = tile * TM + 32 * wq + (lane >> 2) + 8 * (lane & 3);
      float y[24];
#pragma unroll
      for (int i = 0; i < 24; ++i) y[i] = 0.f;
      wait(upper ? bar_l2b : bar_l2a, ph);
      __syncwarp();
      mlp_epilogue2(tmem + lane_off + (upper ? 384u : 256u), sw3, b2, w3, upper ? 128 : 0, y);
      float out[12];
      mlp_outputs(y, out);
      const int k = lane & 3;
      float r[3];
#pragma unroll
      for (int o = 0; o < 3; ++o)  // row k of the four (selects, no indexed register array)
        r[o] = k == 0 ? out[o] : k == 1 ? out[3 + o] : k == 2 ? out[6 + o] : out[9 + o];
      if (!upper) {
        arrive(bar_e2a);  // Q2 may be overwritten
        if (row < M) {
          Y[3 * row] = r[0] + __ldg(b3);
          Y[3 * row + 1] = r[1] + __ldg(b3 + 1);
          Y[3 * row + 2] = r[2] + __ldg(b3 + 2);
        }
        __threadfence_block();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_ya);
      } else {
        wait(bar_ya, ph);  // before Q3 is released: keeps the two groups one tile apart at most
        arrive(bar_e2b);
        if (row < M) {
          Y[3 * row] += r[0];
          Y[3 * row + 1] += r[1];
          Y[3 * row + 2] += r[2];
        }
      }
    }
  }
  if (tmo) atomicOr(status, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (w == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
}

// ---------------------------------------------------------------------------
// Training.  One step is three launches: train_rows_kernel (forward, loss and
// the data gradients of 128 rows per CTA), train_grads_kernel (the weight
// gradients as tcgen05 products over the batch, the bias and output-layer
// gradients by chunks of 64 rows) and train_update_kernel (the partial sums
// added in a fixed order, and Adam).  They took about twenty launches (GEMMs
// that each staged their operands anew and stored every activation a second
// time transposed, then transposes and reductions) and 200 us at 4096 rows;
// now 29 us (128 -> 23 at 64 rows, 280 -> 50 at 16384).
// ---------------------------------------------------------------------------
constexpr uint32_t kMajorMnA = 1u << 15, kMajorMnB = 1u << 16;  // operand stored MN-major

// instruction descriptor of kind::f16 for M = 128 and N
constexpr uint32_t idesc_n(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

// Row buffers (A1, A2, D1, D2 and the rows' inputs XB) are kept in the image
// that both the products and the bulk copies take: per tile of 128 rows, blocks
// of 64 columns, in a block 128 bytes a row with the row's eight 16-byte pieces
// permuted by r % 8 (128-byte swizzle).  Read along the columns a block is a
// K-major operand, read along the rows an MN-major one: rows in groups of 8 are
// 1024 bytes apart (stride offset), 64-column blocks a block apart (leading
// offset).  A warp's 16-byte pieces of 32 rows fall on all banks.
constexpr uint32_t kBlock = TM * 128;  // bytes of a block of 64 columns of a tile
constexpr uint64_t kSwizzle128 = (uint64_t)2 << 61;  // descriptor: 128-byte swizzle
__device__ __forceinline__ uint32_t piece(int r, int c8) {  // columns 8 c8 .. of row r
  return (uint32_t)(c8 >> 3) * kBlock + (uint32_t)r * 128u + (uint32_t)((c8 ^ r) & 7) * 16u;
}

__device__ __forceinline__ float bf_lo(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf_hi(uint32_t p) { return __uint_as_float(p & 0xFFFF0000u); }

// 16 words (32 BF16 values, columns c .. c + 31) of row r into a tile image
__device__ __forceinline__ void put_row32(unsigned char* tile, int r, int c, const uint32_t* pk) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    *reinterpret_cast<uint4*>(tile + piece(r, (c >> 3) + q)) =
        make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
}

// relu(v + b) of 32 columns as BF16 pairs
__device__ __forceinline__ void relu_pack32(const uint32_t* v, const float* b, uint32_t* pk) {
#pragma unroll
  for (int c = 0; c < 32; c += 4) {
    const float4 bb = *reinterpret_cast<const float4*>(b + c);
    pk[c / 2] = relu_bf16x2(__uint_as_float(v[c]) + bb.x, __uint_as_float(v[c + 1]) + bb.y);
    pk[c / 2 + 1] = relu_bf16x2(__uint_as_float(v[c + 2]) + bb.z, __uint_as_float(v[c + 3]) + bb.w);
  }
}

constexpr int kTrThreads = 256;
constexpr size_t kTrSmem = (size_t)kMlpSmemW2 + kMlpSmemX + kMlpSmemW1 + 64;

// Forward, loss and data gradients of rows [128 blockIdx.x, ...): X, W1 and W2
// in shared memory; tensor memory columns 0..255 hold the layer-1 sums, then A1
// and later dH2 as BF16 pairs (the A operands of the next products), columns
// 256..511 the layer-2 sums, then those of dH1.  dH1 = dH2 W2 reads W2 from the
// same shared copy as layer 2, as an MN-major operand.  Warp w holds the rows
// 32 (w % 4) .. and the column half w / 4; the output layer runs one row per
// thread of warps 0-3 while warps 4-7 store A2.  Rows leave through a tile
// image in the place of W1 by bulk copies.  With one tile per CTA the chain of
// load, four products and four epilogues bounds it, not their rates: of 28 us
// at first, 7 went to 16-byte cp.async of the operands (bulk copies now) and 12
// to row stores that spread every warp's 16-byte pieces over 32 lines.
__global__ void __launch_bounds__(kTrThreads, 1) train_rows_kernel(
    const uint16_t* __restrict__ X, const float* __restrict__ T, long long n,
    const uint16_t* W1, const uint16_t* W2, const float* b1, const float* b2, const float* w3,
    TrainBuffers B,
    float* __restrict__ wloss, unsigned int* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  unsigned char* sW2 = dsm;
  unsigned char* sX = dsm + kMlpSmemW2;
  unsigned char* sW1 = sX + kMlpSmemX;
  unsigned char* sT = sW1;  // tile image of the rows on their way out, after layer 1
  uint64_t* bars = reinterpret_cast<uint64_t*>(sW1 + kMlpSmemW1);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 5);
  // in the place of X once layer 1 has read it: w3 (3 x 256) and b3, b2, dY
  float* s3 = reinterpret_cast<float*>(sX);
  float* sb2 = s3 + 772;
  float* sdy = sb2 + 256;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int wq = w & 3, half = w >> 2;
  const int rl = 32 * wq + lane;        // this thread's row of the tile
  const long long row = (long long)blockIdx.x * TM + rl;

  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < 5; ++i) mbar_init(bars + i, 1u);
    fence_mbar_init();
  }
  pdl_wait();  // the weights of the previous step
  pdl_trigger();
  if (tid == 0) {
    mbar_arrive_expect_tx(bars + 3, kMlpSmemW1);
    bulk_load(sW1, W1, kMlpSmemW1, bars + 3);
    mbar_arrive_expect_tx(bars + 4, kMlpSmemW2);
    bulk_load(sW2, W2, kMlpSmemW2, bars + 4);
  }
  for (int c = tid; c < TM * 16; c += kTrThreads) {  // 16-byte piece c % 16 of row c / 16
    const int r = c >> 4;
    const long long rr = (long long)blockIdx.x * TM + r;
    const bool in = rr < n;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(sX + piece(r, c & 15))),
                 "l"(X + (in ? rr : 0) * 128 + (c & 15) * 8), "r"(in ? 16 : 0)
                 : "memory");
  }
  cp_async_commit();
  cp_async_wait<0>();
  fence_proxy_async();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const uint32_t lanes = tmem + ((uint32_t)(32 * wq) << 16);
  bool tmo = false;
  auto wait = [&](uint64_t* bar) {
    if (!tmo && !mbar_wait(bar, 0u)) tmo = true;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  // the warps' accesses to shared and tensor memory before the next products
  auto join = [&]() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  // column of K step kb (16 values, 8 columns of pairs) of the packed operand
  auto packed = [&](int kb) { return tmem + (uint32_t)(kb < 8 ? 8 * kb : 128 + 8 * (kb - 8)); };
  // this warp's rows of blocks b0 .. b1 - 1 of the image to their place in M
  auto send = [&](uint16_t* M, int b0, int b1) {
    fence_proxy_async();
    __syncwarp();
    if (lane < b1 - b0) {
      const uint32_t off = (uint32_t)(b0 + lane) * kBlock + (uint32_t)wq * 32u * 128u;
      bulk_store(reinterpret_cast<unsigned char*>(M) + (size_t)blockIdx.x * 4 * kBlock + off, sT + off,
                 32u * 128u);
    }
    bulk_commit();
  };

  if (tid == 0) {  // layer 1: X W1^T
    wait(bars + 3);
    const uint64_t xd = smem_desc(smem_u32(sX), 16u, 1024u) | kSwizzle128;
    const uint64_t wd = smem_desc(smem_u32(sW1), 128u, 16u * 128u);
#pragma unroll
    for (int kb = 0; kb < 8; ++kb)
      mma_ss_i(tmem, xd + (uint64_t)((kb >> 2) * (int)(kBlock >> 4) + (kb & 3) * 2),
               wd + (uint64_t)(kb * 16), idesc_n(256), kb > 0);
    mma_commit(bars);
    bulk_store(reinterpret_cast<unsigned char*>(B.XB) + (size_t)blockIdx.x * 2 * kBlock, sX, 2 * kBlock);
    bulk_commit();
    bulk_wait_read();
  }
  wait(bars);
  __syncthreads();
  float u[4];  // w3 and b3 follow each other; all loads before the stores
#pragma unroll
  for (int q = 0; q < 4; ++q) u[q] = tid + q * kTrThreads < 771 ? w3[tid + q * kTrThreads] : 0.f;
  sb2[tid] = b2[tid];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (tid + q * kTrThreads < 771) s3[tid + q * kTrThreads] = u[q];

  // A1 = relu(. + b1): packed into tensor memory and sent; m1: A1 > 0
  uint32_t m1[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t v[32], pk[16];
    tmem_ld32(lanes + (uint32_t)(128 * half + 32 * j), v);
    relu_pack32(v, b1 + 128 * half + 32 * j, pk);
    tmem_st16(lanes + (uint32_t)(128 * half + 16 * j), pk);
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q)
      m |= ((pk[q] & 0xFFFFu) ? 1u : 0u) << (2 * q) | ((pk[q] >> 16) ? 2u : 0u) << (2 * q);
    m1[j] = m;
    put_row32(sT, rl, 128 * half + 32 * j, pk);
  }
  join();
  if (tid == 0) {  // layer 2: A1 W2^T
    wait(bars + 4);
    const uint64_t wd = smem_desc(smem_u32(sW2), 128u, 32u * 128u);
#pragma unroll
    for (int kb = 0; kb < 16; ++kb)
      mma_ts_i(tmem + 256u, packed(kb), wd + (uint64_t)(kb * 16), idesc_n(256), kb > 0);
    mma_commit(bars + 1);
  }
  __syncwarp();
  send(B.A1, 2 * half, 2 * half + 2);
  wait(bars + 1);
  bulk_wait_read();
  __syncthreads();  // the image is free again

  if (half == 0) {
    // y = A2 w3^T + b3 in ascending order of the hidden units, dY, loss
    float o0 = s3[768], o1 = s3[769], o2 = s3[770];
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
      uint32_t v[32], pk[16];
      tmem_ld32(lanes + 256u + (uint32_t)(32 * j), v);
      relu_pack32(v, sb2 + 32 * j, pk);
#pragma unroll
      for (int c = 0; c < 32; c += 4) {
        const float4 u0 = *reinterpret_cast<const float4*>(s3 + 32 * j + c);
        const float4 u1 = *reinterpret_cast<const float4*>(s3 + 256 + 32 * j + c);
        const float4 u2 = *reinterpret_cast<const float4*>(s3 + 512 + 32 * j + c);
        const float a0 = bf_lo(pk[c / 2]), a1 = bf_hi(pk[c / 2]);
        const float a2 = bf_lo(pk[c / 2 + 1]), a3 = bf_hi(pk[c / 2 + 1]);
        o0 = fmaf(a3, u0.w, fmaf(a2, u0.z, fmaf(a1, u0.y, fmaf(a0, u0.x, o0))));
        o1 = fmaf(a3, u1.w, fmaf(a2, u1.z, fmaf(a1, u1.y, fmaf(a0, u1.x, o1))));
        o2 = fmaf(a3, u2.w, fmaf(a2, u2.z, fmaf(a1, u2.y, fmaf(a0, u2.x, o2))));
      }
    }
    float lsum = 0.f, y0 = 0.f, y1 = 0.f, y2 = 0.f;
    if (row < n) {
      const float d0 = o0 - T[3 * row], d1 = o1 - T[3 * row + 1], d2 = o2 - T[3 * row + 2];
      lsum += d0 * d0 + d1 * d1 + d2 * d2;
      const float sc = 2.f / (float)n;
      y0 = sc * d0;
      y1 = sc * d1;
      y2 = sc * d2;
      B.DY[3 * row] = y0;
      B.DY[3 * row + 1] = y1;
      B.DY[3 * row + 2] = y2;
    }
    sdy[3 * rl] = y0;
    sdy[3 * rl + 1] = y1;
    sdy[3 * rl + 2] = y2;
    for (int d = 16; d; d >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, d);
    if (lane == 0) wloss[4 * blockIdx.x + wq] = lsum;
  } else {
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
      uint32_t v[32], pk[16];
      tmem_ld32(lanes + 256u + (uint32_t)(32 * j), v);
      relu_pack32(v, sb2 + 32 * j, pk);
      put_row32(sT, rl, 32 * j, pk);
    }
    send(B.A2, 0, 4);
    bulk_wait_read();
  }
  __syncthreads();  // dY; the image is free again

  // dH2 = (dY w3) where A2 > 0
  {
    const float y0 = sdy[3 * rl], y1 = sdy[3 * rl + 1], y2 = sdy[3 * rl + 2];
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      const int k0 = 128 * half + 32 * j;
      uint32_t v[32], pk[16];
      tmem_ld32(lanes + 256u + (uint32_t)k0, v);
      relu_pack32(v, sb2 + k0, pk);
#pragma unroll
      for (int q = 0; q < 16; q += 2) {
        const int k = k0 + 2 * q;
        const float4 u0 = *reinterpret_cast<const float4*>(s3 + k);
        const float4 u1 = *reinterpret_cast<const float4*>(s3 + 256 + k);
        const float4 u2 = *reinterpret_cast<const float4*>(s3 + 512 + k);
        float g0 = fmaf(y2, u2.x, fmaf(y0, u0.x, __fmul_rn(y1, u1.x)));
        float g1 = fmaf(y2, u2.y, fmaf(y0, u0.y, __fmul_rn(y1, u1.y)));
        float g2 = fmaf(y2, u2.z, fmaf(y0, u0.z, __fmul_rn(y1, u1.z)));
        float g3 = fmaf(y2, u2.w, fmaf(y0, u0.w, __fmul_rn(y1, u1.w)));
        if (bf_lo(pk[q]) <= 0.f) g0 = 0.f;
        if (bf_hi(pk[q]) <= 0.f) g1 = 0.f;
        if (bf_lo(pk[q + 1]) <= 0.f) g2 = 0.f;
        if (bf_hi(pk[q + 1]) <= 0.f) g3 = 0.f;
        pk[q] = bf16x2_bits(g0, g1);
        pk[q + 1] = bf16x2_bits(g2, g3);
      }
      tmem_st16(lanes + (uint32_t)(128 * half + 16 * j), pk);
      put_row32(sT, rl, k0, pk);
    }
  }
  join();
  if (tid == 0) {  // dH1 = dH2 W2 (K = the outputs of layer 2: rows of W2)
    const uint64_t wd = smem_desc(smem_u32(sW2), 32u * 128u, 128u);
#pragma unroll
    for (int kb = 0; kb < 16; ++kb)
      mma_ts_i(tmem + 256u, packed(kb), wd + (uint64_t)(kb * 512), idesc_n(256) | kMajorMnB, kb > 0);
    mma_commit(bars + 2);
  }
  __syncwarp();
  send(B.D2, 2 * half, 2 * half + 2);
  wait(bars + 2);
  bulk_wait_read();
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint32_t v[32], pk[16];
    tmem_ld32(lanes + 256u + (uint32_t)(128 * half + 32 * j), v);
#pragma unroll
    for (int q = 0; q < 16; ++q)
      pk[q] = bf16x2_bits((m1[j] >> (2 * q)) & 1u ? __uint_as_float(v[2 * q]) : 0.f,
                          (m1[j] >> (2 * q)) & 2u ? __uint_as_float(v[2 * q + 1]) : 0.f);
    put_row32(sT, rl, 128 * half + 32 * j, pk);
  }
  send(B.D1, 2 * half, 2 * half + 2);
  bulk_wait();
  if (tmo) atomicOr(status, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (w == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
}

// Gradients.  The first splits x parts blocks: split s of the batch for
// dW2[o][k] = sum_m dH2[m][o] A1[m][k] and dW1[o][i] = sum_m dH1[m][o] X[m][i];
// both operands are MN-major images, 64 rows a chunk through a ring of four
// stages, FP32 partials per split.  A block takes 128 outputs o and, with at
// least kManySplits splits, all columns (four parts), else 64 of them (twelve):
// a batch whose chunks have no larger divisor is one long sum, which more blocks
// shorten by sharing its columns without touching its order.  The other blocks:
// one chunk of 64 rows each, in ascending row order, of dW3 and db3 (width
// kPart3), db2 and db1.
constexpr int kGrThreads = 256, kGrStages = 4, kGrRows = 64;
constexpr uint32_t kGrBlock = kGrRows * 128;  // bytes of 64 rows of a block
constexpr uint32_t kGrStage = 6 * kGrBlock;   // A: 128 columns, B: up to 256
constexpr size_t kGrSmem = (size_t)kGrStages * kGrStage + 128;
constexpr int kPart3 = 771;
constexpr int kManySplits = 8;

struct GradArgs {
  TrainBuffers B;
  long long n;
  int splits, parts;
  float *part1, *part2;   // [splits][256][128], [splits][256][256]
  float *p3, *pb2, *pb1;  // per 64-row chunk: [kPart3], [256], [256]
  unsigned int* status;
};

__device__ __forceinline__ void grad_chunk(const GradArgs& a, long long chunk, float* sdy) {
  const long long m0 = chunk * kGrRows;
  const int nr = (int)(a.n - m0 < kGrRows ? a.n - m0 : kGrRows);
  for (int i = threadIdx.x; i < 3 * nr; i += kGrThreads) sdy[i] = a.B.DY[3 * m0 + i];
  __syncthreads();
  const int c = threadIdx.x & 127;  // columns 2 c, 2 c + 1
  const size_t first = (size_t)(m0 / TM) * 4 * kBlock + (size_t)(m0 % TM) * 128;
  auto col = [&](const uint16_t* M, int r) {
    return *(reinterpret_cast<const uint32_t*>(reinterpret_cast<const unsigned char*>(M) + first +
                                               piece(r, c >> 2)) + (c & 3));
  };
  if (threadIdx.x < 128) {
    float s0 = 0.f, s1 = 0.f, t0 = 0.f, t1 = 0.f;
#pragma unroll 16
    for (int r = 0; r < nr; ++r) {
      const uint32_t u = col(a.B.D2, r), v = col(a.B.D1, r);
      s0 += bf_lo(u);
      s1 += bf_hi(u);
      t0 += bf_lo(v);
      t1 += bf_hi(v);
    }
    *reinterpret_cast<float2*>(a.pb2 + chunk * 256 + 2 * c) = make_float2(s0, s1);
    *reinterpret_cast<float2*>(a.pb1 + chunk * 256 + 2 * c) = make_float2(t0, t1);
  } else {
    float s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 16
    for (int r = 0; r < nr; ++r) {
      const uint32_t u = col(a.B.A2, r);
#pragma unroll
      for (int o = 0; o < 3; ++o) {
        s[2 * o] = fmaf(sdy[3 * r + o], bf_lo(u), s[2 * o]);
        s[2 * o + 1] = fmaf(sdy[3 * r + o], bf_hi(u), s[2 * o + 1]);
      }
    }
    float* out = a.p3 + chunk * kPart3;
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      out[256 * o + 2 * c] = s[2 * o];
      out[256 * o + 2 * c + 1] = s[2 * o + 1];
    }
    if (c < 3) {
      float b = 0.f;
      for (int r = 0; r < nr; ++r) b += sdy[3 * r + c];
      out[768 + c] = b;
    }
  }
}

__global__ void __launch_bounds__(kGrThreads, 1) train_grads_kernel(const __grid_constant__ GradArgs a) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(dsm + kGrStages * kGrStage);
  uint64_t* empty = full + kGrStages;
  uint64_t* fin = empty + kGrStages;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(fin + 1);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  if ((int)blockIdx.x >= a.parts * a.splits) {
    pdl_wait();
    pdl_trigger();
    grad_chunk(a, (long long)blockIdx.x - a.parts * a.splits, reinterpret_cast<float*>(dsm));
    return;
  }
  // two thirds of a split's blocks for dW2 (256 columns), the others for dW1
  // (128); four parts: two and two
  const int split = blockIdx.x / a.parts, part = blockIdx.x % a.parts;
  const bool whole = a.parts == 4;
  const bool second = part < (whole ? 2 : 8);
  const int o0 = (part & 1) * 128, N = second ? 256 : 128;
  const int cols = whole ? N : 64, n0 = whole ? 0 : ((second ? part : part - 8) >> 1) * 64;
  const int nb = cols / 64;
  const unsigned char* A = reinterpret_cast<const unsigned char*>(second ? a.B.D2 : a.B.D1);
  const unsigned char* Bm = reinterpret_cast<const unsigned char*>(second ? a.B.A1 : a.B.XB);
  const long long nch = (a.n + kGrRows - 1) / kGrRows;
  const long long c0 = nch * split / a.splits, c1 = nch * (split + 1) / a.splits;
  const int nc = (int)(c1 - c0);

  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(256u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < 2 * kGrStages + 1; ++i) mbar_init(full + i, 1u);
    fence_mbar_init();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  pdl_wait();
  pdl_trigger();
  bool tmo = false;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!tmo && !mbar_wait(bar, parity)) tmo = true;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  if (tid == 0) {
    // blocks of the chunk's 64 rows: two of A from column o0, nb of B
    for (int i = 0; i < nc; ++i) {
      const int sl = i % kGrStages;
      if (i >= kGrStages) wait(empty + sl, (uint32_t)(i / kGrStages - 1) & 1u);
      const long long m0 = (c0 + i) * kGrRows;
      const size_t rows = (size_t)(m0 % TM) * 128;
      const unsigned char* as = A + (size_t)(m0 / TM) * 4 * kBlock + (size_t)(o0 / 64) * kBlock + rows;
      const unsigned char* bs = Bm + ((size_t)(m0 / TM) * (N / 64) + n0 / 64) * kBlock + rows;
      unsigned char* d = dsm + (size_t)sl * kGrStage;
      mbar_arrive_expect_tx(full + sl, (uint32_t)(2 + nb) * kGrBlock);
      for (int b = 0; b < 2; ++b) bulk_g2s(d + b * kGrBlock, as + (size_t)b * kBlock, kGrBlock, full + sl);
      for (int b = 0; b < nb; ++b)
        bulk_g2s(d + (2 + b) * kGrBlock, bs + (size_t)b * kBlock, kGrBlock, full + sl);
    }
  } else if (tid == 32) {
    const uint32_t id = idesc_n(cols) | kMajorMnA | kMajorMnB;
    for (int i = 0; i < nc; ++i) {
      const int sl = i % kGrStages;
      wait(full + sl, (uint32_t)(i / kGrStages) & 1u);
      const uint32_t d = smem_u32(dsm + (size_t)sl * kGrStage);
      const uint64_t ad = smem_desc(d, kGrBlock, 1024u) | kSwizzle128;
      const uint64_t bd = smem_desc(d + 2 * kGrBlock, kGrBlock, 1024u) | kSwizzle128;
#pragma unroll
      for (int kb = 0; kb < kGrRows / 16; ++kb)  // 16 rows: two 8-row groups
        mma_ss_i(tmem, ad + (uint64_t)(kb * 128), bd + (uint64_t)(kb * 128), id, (i > 0 || kb > 0) ? 1u : 0u);
      mma_commit(empty + sl);
    }
    mma_commit(fin);
  }
  __syncwarp();
  wait(fin, 0u);
  // rows o0 + 32 (w % 4) + lane, column half w / 4
  const int row = o0 + 32 * (w & 3) + lane;
  float* out = (second ? a.part2 : a.part1) + ((long long)split * 256 + row) * N + n0;
  for (int j = (w >> 2) * (cols / 2); j < ((w >> 2) + 1) * (cols / 2); j += 32) {
    uint32_t v[32];
    tmem_ld32(tmem + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)j, v);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      reinterpret_cast<float4*>(out + j)[q] =
          make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                      __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
  }
  if (tmo) atomicOr(a.status, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (w == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u)
                 : "memory");
}

// part[0], part[pitch], ... summed in that order
__device__ __forceinline__ float sum_in_order(const float* part, long long count, long long pitch) {
  float acc = 0.f;
#pragma unroll 16
  for (long long s = 0; s < count; ++s) acc += part[s * pitch];
  return acc;
}

// Gradient i from its partials in a fixed order and (adam) its Adam step,
// refreshing the BF16 weights; the last block adds the loss: the warps' sums of
// 256 rows in order, divided by n, then those in order.
__global__ void __launch_bounds__(256) train_update_kernel(const __grid_constant__ GradArgs a,
                                                           const __grid_constant__ TrainState t) {
  pdl_wait();
  pdl_trigger();
  const long long chunks = (a.n + kGrRows - 1) / kGrRows;
  const int i = (int)(blockIdx.x * 256u + threadIdx.x);
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x == 0) {
      const long long warps = (a.n + TM - 1) / TM * 4;
      float acc = 0.f;
      for (long long s = 0; s < warps; s += 8) {
        float b = 0.f;
        for (long long q = s; q < s + 8 && q < warps; ++q) b += t.wloss[q];
        acc += b / (float)a.n;
      }
      *t.loss = acc;
    }
    return;
  }
  if (i >= QTV_LOCATOR_PARAMS) return;
  constexpr int oB1 = 256 * 128, oW2 = oB1 + 256, oB2 = oW2 + 256 * 256, oW3 = oB2 + 256;
  float g;
  if (i < oB1) g = sum_in_order(a.part1 + i, a.splits, 256 * 128);
  else if (i < oW2) g = sum_in_order(a.pb1 + (i - oB1), chunks, 256);
  else if (i < oB2) g = sum_in_order(a.part2 + (i - oW2), a.splits, 256 * 256);
  else if (i < oW3) g = sum_in_order(a.pb2 + (i - oB2), chunks, 256);
  else g = sum_in_order(a.p3 + (i - oW3), chunks, kPart3);
  t.G[i] = g;
  if (!t.adam) return;
  const float p = adam_value(t.P[i], g, t.M[i], t.V[i], t.lr, t.beta1, t.beta2, t.eps, t.c1, t.c2);
  t.P[i] = p;
  const __nv_bfloat16 bf = __float2bfloat16_rn(p);
  const uint16_t b = *reinterpret_cast<const uint16_t*>(&bf);
  if (i < oB1) {
    t.w1b[i] = b;
    t.w1c[canon_index(i, 128)] = b;
  } else if (i >= oW2 && i < oB2) {
    t.w2b[i - oW2] = b;
    t.w2c[canon_index(i - oW2, 256)] = b;
  }
}

}  // namespace

// Splits of a batch of k64 chunks of 64 rows for the weight gradients: its
// largest divisor up to kTrainSplits (equal splits, so that the order of a sum
// depends on the batch alone).
int train_splits(long long k64) {
  int s = kTrainSplits;
  while (k64 % s) --s;
  return s;
}

int tc_train(const uint16_t* X, const float* T, long long n, const TrainBuffers& B, const TrainState& t,
             unsigned int* status, cudaStream_t st) {
  if (n <= 0) return QTV_OK;
  if (reinterpret_cast<uintptr_t>(X) & 15u)
    return set_error(QTV_ERR_ARG, "training rows must be 16-byte aligned");
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(train_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kTrSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(train_grads_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kGrSmem);
    if (e != cudaSuccess) return check_cuda(e, "cudaFuncSetAttribute(training)");
    attr = true;
  }
  const long long tiles = (n + TM - 1) / TM, chunks = (n + kGrRows - 1) / kGrRows;
  const float* P = t.P;
  cudaError_t e = launch_dependent(train_rows_kernel, dim3((unsigned)tiles), dim3(kTrThreads), kTrSmem,
                                   st, X, T, n, (const uint16_t*)t.w1c, (const uint16_t*)t.w2c,
                                   P + 256 * 128, P + 256 * 128 + 256 + 256 * 256,
                                   P + 256 * 128 + 512 + 256 * 256, B, t.wloss, status);
  if (e != cudaSuccess) return check_cuda(e, "train_rows_kernel launch");
  GradArgs a;
  a.B = B;
  a.n = n;
  a.splits = train_splits(chunks);
  a.parts = a.splits >= kManySplits ? 4 : 12;
  a.part1 = B.part;
  a.part2 = B.part + (size_t)kTrainSplits * 256 * 128;
  a.p3 = B.chunk;
  a.pb2 = B.chunk + (size_t)chunks * (kPart3 + 1);
  a.pb1 = a.pb2 + (size_t)chunks * 256;
  a.status = status;
  e = launch_dependent(train_grads_kernel, dim3((unsigned)(a.parts * a.splits + chunks)), dim3(kGrThreads),
                       kGrSmem, st, a);
  if (e != cudaSuccess) return check_cuda(e, "train_grads_kernel launch");
  e = launch_dependent(train_update_kernel, dim3((QTV_LOCATOR_PARAMS + 255) / 256 + 1), dim3(256), 0, st,
                       a, t);
  return check_cuda(e, "train_update_kernel launch");
}

// Y[M][3] of the whole network on the tensor cores (see tc_mlp_kernel).
int tc_mlp_forward(const uint16_t* X, long long M, const uint16_t* W1, const uint16_t* W2,
                   const float* b1, const float* b2, const float* w3, const float* b3, float* Y,
                   unsigned int* status, int num_sms, cudaStream_t st) {
  if (M <= 0) return QTV_OK;
  // 16-byte aligned operands (X for the tensor copies, b2 and w3 read as
  // 8-byte pairs); tile rows are 32-bit tensor coordinates
  if (((reinterpret_cast<uintptr_t>(b1) | reinterpret_cast<uintptr_t>(b2) |
        reinterpret_cast<uintptr_t>(w3) | reinterpret_cast<uintptr_t>(X)) & 15u) ||
      M >= (1ll << 31))
    return set_error(QTV_ERR_ARG, "fused network: misaligned operand or too many rows");
  const size_t smem = kMlpSmem;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(tc_mlp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return check_cuda(e, "cudaFuncSetAttribute(tc_mlp)");
    attr = true;
  }
  const long long ntiles = (M + TM - 1) / TM;
  const int grid = (int)(ntiles < num_sms ? ntiles : num_sms);
  // X as a 2-D BF16 tensor (128 columns, M rows, 256-byte rows); boxes of
  // 64 columns x 128 rows, 128-byte swizzle, rows past M read as zero
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
      return check_cuda(e != cudaSuccess ? e : cudaErrorNotSupported, "cuTensorMapEncodeTiled");
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  CUtensorMap xmap;
  const cuuint64_t dims[2] = {128, (cuuint64_t)M};
  const cuuint64_t strides[1] = {256};
  const cuuint32_t box[2] = {64, (cuuint32_t)TM};
  const cuuint32_t estr[2] = {1, 1};
  if (encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(X), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return set_error(QTV_ERR_ARG, "tensor map of the network input");
  tc_mlp_kernel<<<grid, kMlpThreads, smem, st>>>(xmap, M, W1, W2, b1, b2, w3, b3, Y, status);
  return check_cuda(cudaGetLastError(), "tc_mlp_kernel launch");
}

}  // namespace qtv
