// Tensor-core products on operands held as 16-bit slices (tcgen05 kind::f16).
//
// Three kernels share the layout: K-major slices [slice][row][k] in global
// memory, TMA into swizzled shared memory, one thread issuing the MMAs, FP32
// accumulators in tensor memory, and warps that only fold those.
//
// k_gemm_int8x7: FP64 products in exact integer arithmetic.  The FP64 units
// of this GPU give about two FMAs per SM and clock (1.2 TFLOP/s on the whole
// chip), the 16-bit tensor cores 4096.  Every row of A and every column of B
// gets one power-of-two scale, under which an entry is an integer of 55 bits
// and a sign, written as seven balanced base-256 digits d_0 .. d_6 (|d| <=
// 128, exact in FP16).  A product of two digits is at most 2^14, so the FP32
// accumulators add up to 7 x 128 of them (2^23.8) without rounding.  The
// digit products of equal weight, i + j = c, share one accumulator; classes
// c = 0 .. 7 are formed (34 of 49 products).  What is left out lies below 2^-59
// of the row's and the column's largest entries, under the 2^-54 of the two
// operands' rounding.  (Without class 7 it reaches 2^-51.4, and rows whose
// entries spread over 2^40 came out up to seven times as far off as on the FP64
// units.)  After every 128 columns of K the eight accumulators, all of tensor
// memory, are folded into two 64-bit integers per entry, and the sum is rounded
// to FP64 once, at the end.  Bound by shared memory: an MMA of 128 x 64 x 16
// reads 6 KB (48 clocks against 32 of tensor work), 68 of them and the copies of
// a stage come to 2.1 us, measured 3.2 us a stage of 32 of K (tensor pipe 35 %).
// 131072 x 2048 x 256: 6.8 ms with the digits' preparation (FP64 units: 110 ms).
//
// k_gemm_a16: FP32-accurate products of 16-bit data.  A (BF16 or FP16) is
// exact as it is stored and comes in by TMA straight into the MMA operand;
// B (FP32 values) is split once into three slices of A's type (24 bits in
// BF16, 33 in FP16), for FP16 scaled per column to its range.  Three 16-bit MMAs
// per product; each K block of 64 starts a fresh accumulator, smallest slice
// first, which the fold adds to FP32 registers, rounding to nearest (the
// tensor core's own accumulation truncates).  Bound by two stages of 112 KB:
// the copies of a block of K (94 KB at N = 400) and its MMAs mostly take turns
// (tensor pipe 47 %, L2 22 %).  C leaves in whole sectors (262144 x 2000 x 400:
// 1.57 -> 1.20 ms).
//
// k_gemm_f32x2: FP32 products of FP32 data at twice the TF32 rate.  An FP16
// pair holds as much of an FP32 value as a TF32 pair (11 + 11 bits) once it is
// scaled into FP16's range, and the 16-bit MMA is twice as fast and reads
// half the shared memory.  B is split once in global memory (two slices,
// scaled per column); four warps split each staged tile of A in place, one
// power-of-two scale per row and 64 of K, which the 16 fold warps undo when
// they add the 64 to their FP32 sums: hi lo + lo hi + hi hi, smallest first;
// what is dropped (lo lo and the rounding of both lo) lies below 2^-21 of each
// product, or 2^-38 of the row's largest entry in the 64 where that is more.
// 2^18 x 4096 x 512: 2.93 ms (TF32 form 4.48), 704 threads of 80 registers, 136
// to 144 bytes of spilled stores a thread.
// Without the split and the fold it takes 2.2 ms, without two of the three MMAs
// as well 1.9 ms: no single part bounds it (tensor pipe 48 %, L1 and shared
// memory 47 %, L2 35 %), but their use of shared memory, 152 KB per 32 of K against
// 768 clocks of MMA, and what a CTA alone on its SM does not overlap.  Measured on the
// way: the fold warps splitting too, 3.9 ms; folding every 32 of K, 3.3 ms; two
// CTAs loading half of B each for both, 2.98 ms (and 1.20 as above for
// k_gemm_a16): every CTA loads its own.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "common.cuh"
#include "tma.cuh"
#include "tmem.cuh"

namespace bsrht {
namespace sl {

constexpr int kDig = 7;               // digits of an FP64 operand
constexpr int kCls = 8;               // classes of digit products that are formed
constexpr int BM = 128;
constexpr uint32_t kWaitSl = 1u << 24;  // bounded mbarrier waits
constexpr int kErrSl = 8;             // status bit of a failed wait (kStatusTcWait)
constexpr int kThreads = 64 + 256;    // warps 0: TMA, 1: MMA, 2..9: fold
constexpr int kNonFiniteExp = 0x7FF;  // biased exponent of Inf / NaN

// 3-D tiled TMA load of box {x, y, z} (x innermost).
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int32_t x, int32_t y,
                                            int32_t z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
      "[%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// K-major operand descriptors: rows of 128 bytes (128-byte swizzle, 8-row
// atoms 1024 bytes apart) or 64 bytes (64-byte swizzle, 512 bytes apart).
template <int ROW_BYTES>
__device__ __forceinline__ uint64_t desc_k(uint32_t saddr) {
  static_assert(ROW_BYTES == 128 || ROW_BYTES == 64, "swizzle span");
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)((8u * ROW_BYTES) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)(ROW_BYTES == 128 ? 2 : 4) << 61;
  return d;
}

// Instruction descriptor: D FP32, A and B FP16 (bf16: BF16), both K-major.
__device__ __forceinline__ uint32_t idesc_f16(bool bf16, int n) {
  const uint32_t t = bf16 ? 1u : 0u;
  return (1u << 4) | (t << 7) | (t << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// ------------------------------------------------------------ digit split
// The 55-bit fixed-point value of the FP64 bits `raw` under the scale
// exponent E (>= the biased exponent of every entry that shares it, E >= 1):
// t = round(x 2^(55 - (E - 1022))), |t| < 2^55.  With u = t +
// 0x0080808080808080 (0 <= u < 2^57) the balanced base-256 digits of t are
// the bytes 0 .. 5 of u and its bits 48 .. 56, each less 128.
__device__ __forceinline__ int64_t fixed55(uint64_t raw, int E) {
  const uint32_t hi = (uint32_t)(raw >> 32);
  const int e = (int)((hi >> 20) & 0x7FFu);
  const uint64_t mant = (raw & 0x000FFFFFFFFFFFFFull) | ((uint64_t)(e != 0) << 52);
  const int sh = (e ? e : 1) - E + 2;  // <= 2
  uint64_t q;
  if (sh >= 0) {
    q = mant << sh;
  } else {
    const int r = min(-sh, 63);
    q = (mant + (1ull << (r - 1))) >> r;  // half up: r <= 63, mant < 2^53
  }
  return (int64_t)raw < 0 ? -(int64_t)q : (int64_t)q;
}
__device__ __forceinline__ uint64_t digit_bytes(int64_t t) { return (uint64_t)t + 0x0080808080808080ull; }

// Digit s (0 the highest) of the two values u0, u1 as an FP16 pair: a value b
// <= 256 in the low mantissa bits under the exponent of 1024 is 1024 + b
// exactly, and 1152 off it is the digit.
__device__ __forceinline__ uint32_t digit_pair(uint64_t u0, uint64_t u1, int s) {
  const uint32_t mask = s == 0 ? 0x1FFu : 0xFFu;
  const uint32_t x0 = (uint32_t)(u0 >> (8 * (6 - s))) & mask, x1 = (uint32_t)(u1 >> (8 * (6 - s))) & mask;
  const uint32_t v = x0 | (x1 << 16) | 0x64006400u;
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&v), __floats2half2_rn(1152.f, 1152.f));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// FP64 nearest to (h 2^32 + l) 2^x.
__device__ __forceinline__ double scale_int(int64_t h, int64_t l, int x) {
  uint64_t lo = ((uint64_t)h << 32) + (uint64_t)l;
  int64_t hi = (h >> 32) + (l >> 63) + (lo < (uint64_t)l ? 1 : 0);
  const bool neg = hi < 0;
  uint64_t uh = (uint64_t)hi, ul = lo;
  if (neg) {
    ul = 0ull - ul;
    uh = ~uh + (ul == 0 ? 1 : 0);
  }
  if ((uh | ul) == 0) return 0.0;
  const int lz = uh ? __clzll((long long)uh) : 64 + __clzll((long long)ul);
  uint64_t top;
  bool sticky;
  if (lz >= 64) {
    top = ul << (lz - 64);
    sticky = false;
  } else {
    top = lz ? (uh << lz) | (ul >> (64 - lz)) : uh;
    sticky = lz < 64 && (ul << lz) != 0;
  }
  uint64_t m = top >> 11;
  const uint32_t rem = (uint32_t)top & 0x7FFu;
  m += (rem > 0x400u || (rem == 0x400u && (sticky || (m & 1)))) ? 1 : 0;
  int e = x + (127 - lz) + 1023;  // biased exponent of the leading bit
  if (m >> 53) {
    m >>= 1;
    ++e;
  }
  double v;
  if (e >= 1 && e <= 2046)
    v = __longlong_as_double((long long)((m & 0x000FFFFFFFFFFFFFull) | ((uint64_t)e << 52)));
  else
    v = ldexp((double)m, e - 1023 - 52);
  return neg ? -v : v;
}

// ------------------------------------------------------- FP64 (7 digits)
struct Int8x7 {
  static constexpr int BN = 64, BK = 32, STAGES = 2;
  static constexpr int KG = 4;  // stages (128 columns of K) between folds
  static constexpr uint32_t A_SLICE = BM * BK * 2, B_SLICE = BN * BK * 2;
  static constexpr uint32_t A_BYTES = kDig * A_SLICE, B_BYTES = kDig * B_SLICE;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr size_t smem_bytes() { return 1024 + (size_t)STAGES * STAGE_BYTES + 256; }
  static constexpr uint32_t TMEM_COLS = kCls * BN;
  // Exact sums: 2^14 per product, at most 7 products a class, KG BK columns.
  static_assert(kDig * KG * BK * (1 << 14) <= (1 << 24), "exact FP32 accumulation");
  static_assert(A_SLICE % 1024 == 0 && B_SLICE % 1024 == 0, "swizzle atoms");
};

struct Int8x7Args {
  int64_t M, N, K;
  double* C;       // output, or partials [z][M][N] when `part`
  int64_t ldc;
  const int* ea;   // scale exponents of the rows of A and the columns of B
  const int* eb;
  int part, gram, b_upper;
  int* err;
};

__host__ __device__ __forceinline__ bool int8x7_skipped(int64_t bm, int64_t bn) {
  return bm * BM >= (bn + 1) * Int8x7::BN;
}

__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_int8x7(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, Int8x7Args g) {
  using S = Int8x7;
  constexpr int BN = S::BN, BK = S::BK, STAGES = S::STAGES, KG = S::KG;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (reinterpret_cast<uintptr_t>(smem_raw) & 1023)) & 1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + STAGES * S::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;     // [kCls] class finished
  uint64_t* accfree = accf + kCls;     // [kCls] class folded
  uint64_t* drain = accfree + kCls;    // every MMA issued has finished
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tn = (g.N + BN - 1) / BN;
  const int64_t bm = (int64_t)blockIdx.x / tn, bn = (int64_t)blockIdx.x - bm * tn;
  const int64_t m0 = bm * BM, n0 = bn * BN;
  if (g.gram && int8x7_skipped(bm, bn)) return;  // uniform: before any barrier
  const int64_t kmax = g.b_upper ? (g.K < n0 + BN ? g.K : n0 + BN) : g.K;
  // Split K in groups of KG stages, so that every fold but the last is full.
  const int64_t ngr = (kmax + KG * BK - 1) / (KG * BK);
  const int64_t g0 = ngr * blockIdx.z / gridDim.z, g1 = ngr * (blockIdx.z + 1) / gridDim.z;
  const int64_t kb0 = g0 * KG;
  const int64_t kb_end = (kmax + BK - 1) / BK < g1 * KG ? (kmax + BK - 1) / BK : g1 * KG;
  const int nst = (int)(kb_end > kb0 ? kb_end - kb0 : 0);
  const int ngroups = (nst + KG - 1) / KG;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int c = 0; c < kCls; ++c) {
      mbar_init(&accf[c], 1);
      mbar_init(&accfree[c], 8);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(tmem_slot, S::TMEM_COLS);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool failed = false;

  if (warp == 0) {
    if (lane == 0) {  // TMA producer
      int issued = 0;
      for (int st = 0; st < nst; ++st) {
        const int s = st % STAGES, u = st / STAGES;
        if (u > 0 && !mbar_wait_bounded(&empty[s], (uint32_t)((u - 1) & 1), kWaitSl)) {
          failed = true;
          break;
        }
        unsigned char* p = base + (size_t)s * S::STAGE_BYTES;
        mbar_arrive_expect_tx(&full[s], S::STAGE_BYTES);
        const int32_t kx = (int32_t)((kb0 + st) * BK);
        tma_load_3d(p, &mapA, &full[s], kx, (int32_t)m0, 0);
        tma_load_3d(p + S::A_BYTES, &mapB, &full[s], kx, (int32_t)n0, 0);
        issued = st + 1;
      }
      if (failed)  // shared memory must not be released under copies still landing
        for (int st = (issued > STAGES ? issued - STAGES : 0); st < issued; ++st)
          if (!mbar_wait_bounded(&full[st % STAGES], (uint32_t)((st / STAGES) & 1), kWaitSl)) atomicOr(g.err, kErrSl);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      const uint32_t idesc = idesc_f16(false, BN);
      for (int st = 0; st < nst && !failed; ++st) {
        const int s = st % STAGES, u = st / STAGES, grp = st / KG;
        const bool first = st % KG == 0, last = st % KG == KG - 1 || st == nst - 1;
        if (!mbar_wait_bounded(&full[s], (uint32_t)(u & 1), kWaitSl)) {
          failed = true;
          break;
        }
        tc::tc_fence_after();
        const uint32_t a0 = smem_u32(base + (size_t)s * S::STAGE_BYTES), b0 = a0 + S::A_BYTES;
        // Fully unrolled, operand addresses as constants on the stage's two
        // descriptors: one thread issues 56 MMAs a stage, and forming each
        // one's descriptors anew took longer than the MMA (3.8 us a stage).
        // Class by class: a class starts as soon as its last sums are folded,
        // and is folded as soon as it is complete.
        const uint64_t da = desc_k<64>(a0), db = desc_k<64>(b0);
#pragma unroll
        for (int c = 0; c < kCls; ++c) {
          if (first && grp > 0 && !failed) {
            failed = !mbar_wait_bounded(&accfree[c], (uint32_t)((grp - 1) & 1), kWaitSl);
            tc::tc_fence_after();
          }
          if (!failed) {
#pragma unroll
            for (int i = c < kDig ? 0 : c - kDig + 1; i <= c && i < kDig; ++i) {
#pragma unroll
              for (int kk = 0; kk < BK / 16; ++kk)
                mma_f16(tmem + (uint32_t)(c * BN), da + ((i * S::A_SLICE + 32 * kk) >> 4),
                        db + (((c - i) * S::B_SLICE + 32 * kk) >> 4), idesc,
                        (first && (i == 0 || c - i == kDig - 1) && kk == 0) ? 0u : 1u);
            }
            if (last) mma_commit(&accf[c]);
          }
        }
        if (failed) break;
        mma_commit(&empty[s]);
      }
      // Never free TMEM under MMAs that may still run.
      mma_commit(drain);
      if (!mbar_wait_bounded(drain, 0, kWaitSl)) atomicOr(g.err, kErrSl);
    }
  } else {
    const int wq = warp & 3;              // TMEM lane quarter of this warp
    const int ch = (warp - 2) >> 2;       // column half: 32 columns
    const uint32_t lane_base = tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)(32 * ch);
    int64_t H[32], L[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) H[q] = L[q] = 0;
    auto fold = [&](int c, int grp, int64_t(&T)[32], int w) -> bool {
      const bool ok = mbar_wait_bounded(&accf[c], (uint32_t)(grp & 1), kWaitSl);
      if (!__all_sync(0xffffffffu, ok)) return false;
      tc::tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[16];
        tc::tmem_ld16(lane_base + (uint32_t)(c * BN + 16 * h), v);
#pragma unroll
        for (int q = 0; q < 16; ++q) T[16 * h + q] += (int64_t)__float2int_rn(v[q]) * w;
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accfree[c]);
      return true;
    };
    for (int grp = 0; grp < ngroups && !failed; ++grp) {
      failed = !(fold(0, grp, H, 1 << 24) && fold(1, grp, H, 1 << 16) && fold(2, grp, H, 1 << 8) &&
                 fold(3, grp, H, 1) && fold(4, grp, L, 1 << 24) && fold(5, grp, L, 1 << 16) &&
                 fold(6, grp, L, 1 << 8) && fold(7, grp, L, 1));
    }
    const int64_t row = m0 + 32 * wq + lane;
    const int64_t c0 = n0 + 32 * ch;
    if (row < g.M && c0 < g.N) {
      const int ea = g.ea[row];
      double* dst = g.part ? g.C + ((int64_t)blockIdx.z * g.M + row) * g.N + c0 : g.C + row * g.ldc + c0;
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        if (c0 + q >= g.N) break;
        const int eb = g.eb[c0 + q];
        // Entry scales 2^(E - 1022 - 55) each; weights 2^40 and up.
        double v = scale_int(H[q], L[q], 40 + (ea - 1077) + (eb - 1077));
        if (failed || ea >= kNonFiniteExp || eb >= kNonFiniteExp) v = __longlong_as_double(0x7ff8000000000000ll);
        dst[q] = v;
      }
    }
  }
  if (failed) atomicOr(g.err, kErrSl);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, S::TMEM_COLS);
}

// Stores a warp's 32 x NC piece of C (row0 + lane in v, columns scaled by
// bscale; NaN if failed): through shared memory
// (buf, 32 rows of NC + 4 words), so that every store covers whole sectors
// whatever ldc and C's alignment are; straight from the registers each
// instruction would touch 32 rows.  ct: the transposed copy, 128 bytes a store
// as it stands.
template <int NC>
constexpr uint32_t store_buf_bytes() {
  return 32 * (NC + 4) * 4;
}
template <typename TC, int NC>
__device__ __forceinline__ void store_warp_tile(const float (&v)[NC], float* buf, TC* C, int64_t ldc, float* Ct,
                                                int64_t ldct, int64_t row0, int64_t M, int64_t c0, int ncol,
                                                const float* bscale, bool failed) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < NC; q += 4)
    *reinterpret_cast<float4*>(buf + lane * (NC + 4) + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  __syncwarp();
  const int rows = (int)(M - row0 < 32 ? M - row0 : 32);
  const float nan = __int_as_float(0x7fc00000);
  float sc[NC / 32];
#pragma unroll
  for (int c = 0; c < NC / 32; ++c) sc[c] = failed ? nan : 32 * c + lane < ncol ? __ldg(bscale + c0 + 32 * c + lane) : 0.f;
  TC* dst = C + row0 * ldc + c0;
#pragma unroll 4
  for (int r = 0; r < rows; ++r) {
#pragma unroll
    for (int c = 0; c < NC / 32; ++c)
      if (32 * c + lane < ncol) dst[r * ldc + 32 * c + lane] = (TC)(buf[r * (NC + 4) + 32 * c + lane] * sc[c]);
  }
  if (Ct && lane < rows) {
    float* ct = Ct + c0 * ldct + row0 + lane;
#pragma unroll
    for (int q = 0; q < NC; ++q)
      if (q < ncol) ct[(int64_t)q * ldct] = failed ? nan : v[q] * __ldg(bscale + c0 + q);
  }
}

// --------------------------------------------- 16-bit A, B in three slices
struct A16 {
  static constexpr int BNMAX = 256, BK = 64, STAGES = 2, NB = 3;
  static constexpr uint32_t A_BYTES = BM * BK * 2;
  static constexpr uint32_t B_SLICE_MAX = BNMAX * BK * 2;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + NB * B_SLICE_MAX;
  static constexpr size_t smem_bytes() { return 1024 + (size_t)STAGES * STAGE_BYTES + 256; }
  static constexpr uint32_t TMEM_COLS = 2 * BNMAX;
  static_assert(STAGES * STAGE_BYTES + 1280 <= 227 * 1024, "shared memory");
  static_assert(8 * store_buf_bytes<128>() <= STAGES * STAGE_BYTES, "the stages hold the stored tile");
};

struct A16Args {
  int64_t M, N, K;
  float* C;
  int64_t ldc;
  const float* bscale;  // undoes the column scale of B's slices
  float* Ct;            // optional FP32 copy of C transposed (N x M)
  int64_t ldct;
  int bn;               // tile width: a multiple of 16, at most 256
  int bf16;
  int* err;
};

__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_a16(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, A16Args g) {
  using S = A16;
  constexpr int BK = S::BK, STAGES = S::STAGES;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (reinterpret_cast<uintptr_t>(smem_raw) & 1023)) & 1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + STAGES * S::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;  // [2]
  uint64_t* accfree = accf + 2;     // [2]
  uint64_t* drain = accfree + 2;    // every MMA issued has finished
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bnw = g.bn;
  const int64_t tn = (g.N + bnw - 1) / bnw;
  const int64_t bm = (int64_t)blockIdx.x / tn, bn = (int64_t)blockIdx.x - bm * tn;
  const int64_t m0 = bm * BM, n0 = bn * bnw;
  const int nkb = (int)((g.K + BK - 1) / BK);
  const uint32_t bslice = (uint32_t)bnw * BK * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&accfree[b], 8);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(tmem_slot, S::TMEM_COLS);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool failed = false;

  if (warp == 0) {
    if (lane == 0) {  // TMA producer
      int issued = 0;
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES;
        if (u > 0 && !mbar_wait_bounded(&empty[s], (uint32_t)((u - 1) & 1), kWaitSl)) {
          failed = true;
          break;
        }
        unsigned char* p = base + (size_t)s * S::STAGE_BYTES;
        mbar_arrive_expect_tx(&full[s], S::A_BYTES + S::NB * bslice);
        tma_load_2d(p, &mapA, &full[s], kb * BK, (int32_t)m0);
#pragma unroll
        for (int q = 0; q < S::NB; ++q)
          tma_load_3d(p + S::A_BYTES + q * bslice, &mapB, &full[s], kb * BK, (int32_t)n0, q);
        issued = kb + 1;
      }
      if (failed)
        for (int kb = (issued > STAGES ? issued - STAGES : 0); kb < issued; ++kb)
          if (!mbar_wait_bounded(&full[kb % STAGES], (uint32_t)((kb / STAGES) & 1), kWaitSl)) atomicOr(g.err, kErrSl);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      const uint32_t idesc = idesc_f16(g.bf16 != 0, bnw);
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES, b = kb & 1;
        if (!mbar_wait_bounded(&full[s], (uint32_t)(u & 1), kWaitSl) ||
            (kb >= 2 && !mbar_wait_bounded(&accfree[b], (uint32_t)(((kb >> 1) - 1) & 1), kWaitSl))) {
          failed = true;
          break;
        }
        tc::tc_fence_after();
        const uint32_t a0 = smem_u32(base + (size_t)s * S::STAGE_BYTES);
        const uint64_t da = desc_k<128>(a0), db = desc_k<128>(a0 + S::A_BYTES);
        const uint32_t d = tmem + (uint32_t)(b * S::BNMAX);
        // Smallest slice first: the truncating additions then happen while
        // the accumulator is small.
#pragma unroll
        for (int q = S::NB - 1; q >= 0; --q) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_f16(d, da + 2 * kk, db + (q * bslice >> 4) + 2 * kk, idesc,
                    (q == S::NB - 1 && kk == 0) ? 0u : 1u);
        }
        mma_commit(&empty[s]);
        mma_commit(&accf[b]);
      }
      // Never free TMEM under MMAs that may still run.
      mma_commit(drain);
      if (!mbar_wait_bounded(drain, 0, kWaitSl)) atomicOr(g.err, kErrSl);
    }
  } else {
    const int wq = warp & 3;
    const int ch = (warp - 2) >> 2;  // column half: 128 columns of the tile
    const uint32_t lane_base = tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)(128 * ch);
    const int nc = min(128, max(0, bnw - 128 * ch));  // columns of this warp (uniform)
    float run[128];
#pragma unroll
    for (int i = 0; i < 128; ++i) run[i] = 0.f;
    for (int kb = 0; kb < nkb; ++kb) {
      const bool ok = mbar_wait_bounded(&accf[kb & 1], (uint32_t)((kb >> 1) & 1), kWaitSl);
      if (!__all_sync(0xffffffffu, ok)) {
        failed = true;
        break;
      }
      tc::tc_fence_after();
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (16 * c < nc) {
          float v[16];
          tc::tmem_ld16(lane_base + (uint32_t)((kb & 1) * S::BNMAX + 16 * c), v);
#pragma unroll
          for (int q = 0; q < 16; ++q) run[16 * c + q] += v[q];
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accfree[kb & 1]);
    }
    const int64_t row0 = m0 + 32 * wq, c0 = n0 + 128 * ch, left = g.N - c0;
    const int ncol = (int)(left < nc ? left : nc);
    // The last accumulator is full: no copy or MMA uses the stages any more
    // (after a failure they may, so each warp waits for that).
    if (failed) mbar_wait_bounded(drain, 0, kWaitSl);
    if (row0 < g.M && ncol > 0) {
      float* buf = reinterpret_cast<float*>(base + (warp - 2) * store_buf_bytes<128>());
      store_warp_tile<float, 128>(run, buf, g.C, g.ldc, g.Ct, g.ldct, row0, g.M, c0, ncol, g.bscale, failed);
    }
  }
  if (failed) atomicOr(g.err, kErrSl);
  __syncwarp();
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, S::TMEM_COLS);
}

// ------------------------------------------------ FP32 A, two slices each
struct F32x2 {
  static constexpr int BNMAX = 256, BK = 32, STAGES = 4, NB = 2;
  static constexpr uint32_t A_BYTES = BM * BK * 4;  // rows of 128 bytes: FP32, then hi | lo
  static constexpr uint32_t B_SLICE_MAX = BNMAX * BK * 2;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + NB * B_SLICE_MAX;
  static constexpr int RING = 8;  // K blocks whose split is remembered; half as many row scales
  static constexpr int SPLIT_WARPS = 4, FOLD_WARPS = 16, NC = 64;
  // The sums are kept at LOWER times B's scale over the product: divided by the
  // column's largest entry, 2^-11 to 1 in an orthonormal one.  (At B's own scale,
  // 2^13 more, they overflowed where the product was above 2^111.)
  static constexpr float LOWER = 0x1.0p-13f;
  static constexpr int THREADS = 32 * (2 + SPLIT_WARPS + FOLD_WARPS);
  static constexpr size_t smem_bytes() { return 1024 + (size_t)STAGES * STAGE_BYTES + RING / 2 * BM * 4 + 256; }
  static constexpr uint32_t TMEM_COLS = 2 * BNMAX;
  static_assert(STAGES * STAGE_BYTES + RING / 2 * BM * 4 + 1280 <= 227 * 1024, "shared memory");
  static_assert(FOLD_WARPS * store_buf_bytes<NC>() <= STAGES * STAGE_BYTES, "the stages hold the stored tile");
};

struct F32x2Args {
  int64_t M, N, K;
  void* C;
  int64_t ldc;
  const float* bscale;  // undoes the column scale of B's slices and LOWER
  float* Ct;            // optional FP32 copy of C transposed (N x M)
  int64_t ldct;
  int bn;               // tile width: a multiple of 16, at most 256
  int b_upper;          // B[k][n] = 0 for k > n
  int* err;
};

template <typename TC>
__global__ void __launch_bounds__(F32x2::THREADS, 1)
    k_gemm_f32x2(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, F32x2Args g) {
  using S = F32x2;
  constexpr int BK = S::BK, STAGES = S::STAGES, RING = S::RING;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (reinterpret_cast<uintptr_t>(smem_raw) & 1023)) & 1023);
  float* rscale = reinterpret_cast<float*>(base + STAGES * S::STAGE_BYTES);  // [RING / 2][BM]
  uint64_t* full = reinterpret_cast<uint64_t*>(rscale + RING / 2 * BM);
  uint64_t* ready = full + STAGES;  // [RING]: A split, row scales written
  uint64_t* empty = ready + RING;
  uint64_t* accf = empty + STAGES;  // [2]
  uint64_t* accfree = accf + 2;     // [2]
  uint64_t* drain = accfree + 2;    // every MMA issued has finished
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bnw = g.bn;
  const int64_t tn = (g.N + bnw - 1) / bnw;
  const int64_t bm = (int64_t)blockIdx.x / tn, bn = (int64_t)blockIdx.x - bm * tn;
  const int64_t m0 = bm * BM, n0 = bn * bnw;
  const int64_t kmax = g.b_upper ? (g.K < n0 + bnw ? g.K : n0 + bnw) : g.K;
  const int nkb = (int)((kmax + BK - 1) / BK);
  const uint32_t bslice = (uint32_t)bnw * BK * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < RING; ++s) mbar_init(&ready[s], S::SPLIT_WARPS);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&accfree[b], S::FOLD_WARPS);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) tc::tmem_alloc(tmem_slot, S::TMEM_COLS);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool failed = false;

  if (warp == 0) {
    if (lane == 0) {  // TMA producer
      int issued = 0;
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES;
        if (u > 0 && !mbar_wait_bounded(&empty[s], (uint32_t)((u - 1) & 1), kWaitSl)) {
          failed = true;
          break;
        }
        unsigned char* p = base + (size_t)s * S::STAGE_BYTES;
        mbar_arrive_expect_tx(&full[s], S::A_BYTES + S::NB * bslice);
        tma_load_2d(p, &mapA, &full[s], kb * BK, (int32_t)m0);
#pragma unroll
        for (int q = 0; q < S::NB; ++q)
          tma_load_3d(p + S::A_BYTES + q * bslice, &mapB, &full[s], kb * BK, (int32_t)n0, q);
        issued = kb + 1;
      }
      if (failed)
        for (int kb = (issued > STAGES ? issued - STAGES : 0); kb < issued; ++kb)
          if (!mbar_wait_bounded(&full[kb % STAGES], (uint32_t)((kb / STAGES) & 1), kWaitSl)) atomicOr(g.err, kErrSl);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      const uint32_t idesc = idesc_f16(false, bnw);
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES, p = kb >> 1, b = p & 1;
        const bool first = (kb & 1) == 0;
        if (!mbar_wait_bounded(&ready[kb % RING], (uint32_t)((kb / RING) & 1), kWaitSl) ||
            !mbar_wait_bounded(&full[s], (uint32_t)(u & 1), kWaitSl) ||
            (first && p >= 2 && !mbar_wait_bounded(&accfree[b], (uint32_t)(((p >> 1) - 1) & 1), kWaitSl))) {
          failed = true;
          break;
        }
        tc::tc_fence_after();
        const uint32_t a0 = smem_u32(base + (size_t)s * S::STAGE_BYTES);
        const uint64_t a_hi = desc_k<128>(a0), a_lo = a_hi + (2 * BK >> 4);
        const uint64_t b_hi = desc_k<64>(a0 + S::A_BYTES), b_lo = b_hi + (bslice >> 4);
        const uint32_t d = tmem + (uint32_t)(b * S::BNMAX);
        // The small terms first: the truncating additions then happen while
        // the accumulator is small.
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) mma_f16(d, a_hi + 2 * kk, b_lo + 2 * kk, idesc, (first && kk == 0) ? 0u : 1u);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) mma_f16(d, a_lo + 2 * kk, b_hi + 2 * kk, idesc, 1u);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) mma_f16(d, a_hi + 2 * kk, b_hi + 2 * kk, idesc, 1u);
        mma_commit(&empty[s]);
        if (!first || kb == nkb - 1) mma_commit(&accf[b]);
      }
      // Never free TMEM under MMAs that may still run.
      mma_commit(drain);
      if (!mbar_wait_bounded(drain, 0, kWaitSl)) atomicOr(g.err, kErrSl);
    }
  } else if (warp < 2 + S::SPLIT_WARPS) {
    // Split: one thread per row, in place.  A row's 32 values (128 bytes,
    // 16-byte chunk q at q ^ (row & 7)) become 32 hi and 32 lo halves, the
    // same row of a K-major FP16 tile; 8 lanes cover the 8 chunk positions, so
    // neither loads nor stores meet bank conflicts.  Two K blocks share an
    // accumulator and therefore the row's scale.
    const int r = threadIdx.x - 64;
    auto row_of = [&](int kb) { return base + (size_t)(kb % STAGES) * S::STAGE_BYTES + 128 * r; };
    auto load = [&](int kb, uint4 (&x)[8], uint32_t mx) {
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = *reinterpret_cast<const uint4*>(row_of(kb) + 16 * (q ^ (r & 7)));
#pragma unroll
      for (int q = 0; q < 8; ++q)
        mx = max(max(mx, max(x[q].x & 0x7FFFFFFFu, x[q].y & 0x7FFFFFFFu)),
                 max(x[q].z & 0x7FFFFFFFu, x[q].w & 0x7FFFFFFFu));
      return mx;
    };
    auto split = [&](int kb, const uint4 (&x)[8], float sc) {
      unsigned char* row = row_of(kb);
      auto two = [&](uint32_t v0, uint32_t v1, uint32_t& hi, uint32_t& lo) {
        const float a0 = __uint_as_float(v0) * sc, a1 = __uint_as_float(v1) * sc;
        const __half2 hh = __floats2half2_rn(a0, a1);
        const float2 f = __half22float2(hh);
        const __half2 ll = __floats2half2_rn(a0 - f.x, a1 - f.y);
        hi = *reinterpret_cast<const uint32_t*>(&hh);
        lo = *reinterpret_cast<const uint32_t*>(&ll);
      };
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint4 hi, lo;
        two(x[2 * q].x, x[2 * q].y, hi.x, lo.x);
        two(x[2 * q].z, x[2 * q].w, hi.y, lo.y);
        two(x[2 * q + 1].x, x[2 * q + 1].y, hi.z, lo.z);
        two(x[2 * q + 1].z, x[2 * q + 1].w, hi.w, lo.w);
        *reinterpret_cast<uint4*>(row + 16 * (q ^ (r & 7))) = hi;
        *reinterpret_cast<uint4*>(row + 16 * ((4 + q) ^ (r & 7))) = lo;
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ready[kb % RING]);
    };
    for (int kb = 0; kb < nkb; kb += 2) {
      const bool two = kb + 1 < nkb;
      const bool ok = mbar_wait_bounded(&full[kb % STAGES], (uint32_t)((kb / STAGES) & 1), kWaitSl) &&
                      (!two || mbar_wait_bounded(&full[(kb + 1) % STAGES], (uint32_t)(((kb + 1) / STAGES) & 1), kWaitSl));
      if (!__all_sync(0xffffffffu, ok)) {
        failed = true;
        break;
      }
      uint4 x[8];
      uint32_t mx = two ? load(kb + 1, x, 0u) : 0u;  // its size only, loaded again below
      mx = load(kb, x, mx);
      // Largest entry into [2^13, 2^14).
      const int sh = min(max(140 - (int)(mx >> 23), -126), 126);
      const float sc = __uint_as_float((uint32_t)(127 + sh) << 23);
      rscale[(kb / 2) % (RING / 2) * BM + r] = __uint_as_float((uint32_t)(127 - sh) << 23) * S::LOWER;
      split(kb, x, sc);
      if (two) {
        load(kb + 1, x, 0u);
        split(kb + 1, x, sc);
      }
    }
  } else {
    const int wq = warp & 3, fw = warp - 2 - S::SPLIT_WARPS;
    const int c = S::NC * (fw >> 2);  // this warp's columns of the tile
    const int nc = min(S::NC, max(0, bnw - c));
    const uint32_t lane_base = tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)c;
    float run[S::NC];
#pragma unroll
    for (int i = 0; i < S::NC; ++i) run[i] = 0.f;
    for (int p = 0; 2 * p < nkb; ++p) {
      // The ring is long enough for these parities: the split of pair p + 4
      // needs the MMAs of pair p + 2, which need the fold of pair p.
      const bool ok = mbar_wait_bounded(&accf[p & 1], (uint32_t)((p >> 1) & 1), kWaitSl) &&
                      mbar_wait_bounded(&ready[2 * p % RING], (uint32_t)((2 * p / RING) & 1), kWaitSl);
      if (!__all_sync(0xffffffffu, ok)) {
        failed = true;
        break;
      }
      tc::tc_fence_after();
      const float rs = rscale[p % (RING / 2) * BM + 32 * wq + lane];
#pragma unroll
      for (int q = 0; q < S::NC / 8; ++q) {
        if (8 * q < nc) {
          float v[8];
          tc::tmem_ld8(lane_base + (uint32_t)((p & 1) * S::BNMAX + 8 * q), v);
#pragma unroll
          for (int i = 0; i < 8; ++i) run[8 * q + i] = fmaf(v[i], rs, run[8 * q + i]);
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accfree[p & 1]);
    }
    const int64_t c0 = n0 + c, left = g.N - c0;
    const int ncol = (int)(left < nc ? left : nc);
    const int64_t row0 = m0 + 32 * wq;
    // The last accumulator is full: no copy or MMA uses the stages any more
    // (after a failure they may, so each warp waits for that).
    if (failed) mbar_wait_bounded(drain, 0, kWaitSl);
    if (row0 < g.M && ncol > 0) {
      float* buf = reinterpret_cast<float*>(base + fw * store_buf_bytes<S::NC>());
      store_warp_tile<TC, S::NC>(run, buf, static_cast<TC*>(g.C), g.ldc, g.Ct, g.ldct, row0, g.M, c0, ncol,
                                 g.bscale, failed);
    }
  }
  if (failed) atomicOr(g.err, kErrSl);
  __syncwarp();
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, S::TMEM_COLS);
}

}  // namespace sl
}  // namespace bsrht
