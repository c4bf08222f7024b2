// Host side and operand preparation of the sliced tensor-core products
// (gemm_slices.cuh).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "dla.cuh"
#include "gemm_slices.cuh"
#include "sketch.cuh"

namespace bsrht {

#define TRY_SL(expr)                 \
  do {                               \
    const int st_ = (expr);          \
    if (st_ != BSRHT_OK) return st_; \
  } while (0)

namespace {

using sl::kDig;

__device__ __forceinline__ int exp_of(double x) {
  return (int)((uint32_t)((uint64_t)__double_as_longlong(x) >> 52) & 0x7FFu);
}

// Digits of the rows of A (rows x K, row-major): out[s][i][k] (row length
// ldk, even; k in [K, ldk) zero) and the rows' scale exponents.  One warp per
// row; the second read of the row comes from the caches.
__global__ void __launch_bounds__(256) k_digits_rows(const double* __restrict__ A, int64_t rows, int64_t K,
                                                     int64_t lda, uint32_t* __restrict__ out, int64_t ldk,
                                                     int* __restrict__ exps) {
  const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= rows) return;
  const double* a = A + i * lda;
  int E = 1;
  for (int64_t k = lane; k < K; k += 32) E = max(E, exp_of(a[k]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  if (lane == 0) exps[i] = E;
  const int64_t plane = rows * (ldk / 2);
  uint32_t* o = out + i * (ldk / 2);
  for (int64_t k = 2 * lane; k < ldk; k += 64) {
    const double x0 = k < K ? a[k] : 0.0, x1 = k + 1 < K ? a[k + 1] : 0.0;
    const uint64_t u0 = sl::digit_bytes(sl::fixed55((uint64_t)__double_as_longlong(x0), E));
    const uint64_t u1 = sl::digit_bytes(sl::fixed55((uint64_t)__double_as_longlong(x1), E));
#pragma unroll
    for (int s = 0; s < kDig; ++s) o[(int64_t)s * plane + k / 2] = sl::digit_pair(u0, u1, s);
  }
}

// exps[c] = max(1, biased exponents of column c) of B (K x N, row-major),
// exps zeroed before.  blockIdx.y: a range of `per` rows.
__global__ void k_col_exps(const double* __restrict__ B, int64_t K, int64_t N, int64_t ldb, int64_t per,
                           int* __restrict__ exps) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= N) return;
  const int64_t k0 = (int64_t)blockIdx.y * per, k1 = min(K, k0 + per);
  int E = 1;
#pragma unroll 8
  for (int64_t k = k0; k < k1; ++k) E = max(E, exp_of(B[k * ldb + c]));
  atomicMax(&exps[c], E);
}

// Digits of the columns of B (K x N, row-major), K-major: out[s][c][k] (row
// length ldk, even; k in [K, ldk) zero).  64 (k) x 32 (c) tiles through
// shared memory.
__global__ void __launch_bounds__(256) k_digits_cols(const double* __restrict__ B, int64_t K, int64_t N, int64_t ldb,
                                                     uint32_t* __restrict__ out, int64_t ldk,
                                                     const int* __restrict__ exps, int64_t tiles_n) {
  __shared__ double t[64][33];
  const int64_t tk = (int64_t)blockIdx.x / tiles_n, tb = (int64_t)blockIdx.x - tk * tiles_n;
  const int64_t k0 = tk * 64, c0 = tb * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int r = ty; r < 64; r += 8) {
    const int64_t k = k0 + r, c = c0 + tx;
    t[r][tx] = (k < K && c < N) ? B[k * ldb + c] : 0.0;
  }
  __syncthreads();
  const int64_t plane = N * (ldk / 2);
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int64_t c = c0 + r, k = k0 + 2 * tx;
    if (c >= N || k >= ldk) continue;
    const int E = exps[c];
    const uint64_t u0 = sl::digit_bytes(sl::fixed55((uint64_t)__double_as_longlong(t[2 * tx][r]), E));
    const uint64_t u1 = sl::digit_bytes(sl::fixed55((uint64_t)__double_as_longlong(t[2 * tx + 1][r]), E));
    uint32_t* o = out + c * (ldk / 2) + k / 2;
#pragma unroll
    for (int s = 0; s < kDig; ++s) o[(int64_t)s * plane] = sl::digit_pair(u0, u1, s);
  }
}

// Fixed-order sum of the split-K partials; for a Gram product the tiles
// skipped below the diagonal are read from their mirror images.
__global__ void k_int8x7_reduce(const double* __restrict__ P, double* __restrict__ C, int64_t M, int64_t N,
                                int64_t ldc, int parts, int gram) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= M * N) return;
  const int64_t i = idx / N, j = idx - i * N;
  int64_t si = i, sj = j;
  if (gram && sl::int8x7_skipped(i / sl::BM, j / sl::Int8x7::BN)) {
    si = j;
    sj = i;
  }
  double s = 0.0;
  for (int z = 0; z < parts; ++z) s += P[((int64_t)z * M + si) * N + sj];
  C[i * ldc + j] = s;
}

// NS 16-bit slices of the columns of B (K x N, row-major, read as FP32),
// K-major: out[s][c][k], row length ldk; scale[c] undoes the column's power of
// two.  FP16: with 2^(E - 127) <= max |column| < 2^(E - 126) the column is scaled
// by 2^(140 - E), so its largest entry lies in [2^13, 2^14) (FP16's range with
// 2^-24 as the smallest step).  BF16 has FP32's range and A is not scaled: only
// columns above 1, or so small that the last slice would be subnormal, are, so
// that no sum overflows that the product itself does not.
template <typename TB, typename T16, int NS>
__global__ void __launch_bounds__(256) k_slices16_cols(const TB* __restrict__ B, int64_t K, int64_t N, int64_t ldb,
                                                       T16* __restrict__ out, int64_t ldk,
                                                       const int* __restrict__ exps, int64_t tiles_n,
                                                       float* __restrict__ scale, float undo) {
  __shared__ float t[64][65];
  const int64_t tk = (int64_t)blockIdx.x / tiles_n, tb = (int64_t)blockIdx.x - tk * tiles_n;
  const int64_t k0 = tk * 64, c0 = tb * 64;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int r = ty; r < 64; r += 8) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t k = k0 + r, c = c0 + tx + 32 * h;
      t[r][tx + 32 * h] = (k < K && c < N) ? (float)B[k * ldb + c] : 0.f;
    }
  }
  __syncthreads();
  const int64_t plane = N * ldk;
#pragma unroll
  for (int r = ty; r < 64; r += 8) {
    const int64_t c = c0 + r;
    if (c >= N) continue;
    // exps: FP32 biased exponents.  Columns at the ends of the range are
    // scaled as far as one FP32 factor and its inverse reach.
    const int E = exps[c];
    const int sh = std::is_same<T16, __half>::value ? min(max(140 - E, -126), 126)
                                                    : (E > 127 ? 127 - E : E < 63 ? 63 - E : 0);
    const float f = __uint_as_float((uint32_t)(127 + sh) << 23);
    if (tk == 0 && tx == 0) scale[c] = __uint_as_float((uint32_t)(127 - sh) << 23) * undo;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t k = k0 + tx + 32 * h;
      if (k >= ldk) continue;
      float x = t[tx + 32 * h][r] * f;
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const T16 d = (T16)x;
        out[(int64_t)s * plane + c * ldk + k] = d;
        x -= (float)d;
      }
    }
  }
}

// exps[c] = FP32 biased exponent of the largest entry of column c (exps
// zeroed before).
template <typename TB>
__global__ void k_col_exps32(const TB* __restrict__ B, int64_t K, int64_t N, int64_t ldb, int64_t per,
                             int* __restrict__ exps) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= N) return;
  const int64_t k0 = (int64_t)blockIdx.y * per, k1 = min(K, k0 + per);
  uint32_t E = 0;
#pragma unroll 8
  for (int64_t k = k0; k < k1; ++k) E = max(E, __float_as_uint((float)B[k * ldb + c]) & 0x7F800000u);
  atomicMax(&exps[c], (int)(E >> 23));
}

// 3-D map [planes][rows][k] of 16-bit K-major slices, rows of ldk elements.
bool make_slice_map(CUtensorMap* map, const void* base, CUtensorMapDataType dt, int64_t k, int64_t rows, int planes,
                    int64_t ldk, uint32_t box_k, uint32_t box_rows, CUtensorMapSwizzle swz, int box_planes) {
  return make_tensor_map_3d(map, base, dt, 2, (uint64_t)k, (uint64_t)rows, (uint64_t)planes, (uint64_t)ldk,
                            (uint64_t)(ldk * rows), box_k, box_rows, (uint32_t)box_planes, swz);
}

int64_t round_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

unsigned row_parts(int64_t K, int64_t col_blocks) {
  // Enough CTAs to fill the GPU, at least 16 rows each (a thread's loads
  // follow one another).
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((4 * (int64_t)num_sms() + col_blocks - 1) / col_blocks,
                                                          (K + 15) / 16));
}

int digits_rows(const Dla& d, const double* A, int64_t rows, int64_t K, int64_t lda, uint32_t* out, int64_t ldk,
                int* exps) {
  k_digits_rows<<<(unsigned)((rows + 7) / 8), 256, 0, d.s>>>(A, rows, K, lda, out, ldk, exps);
  BSRHT_CUDA_TRY(cudaGetLastError());
  note_launches(1);
  return BSRHT_OK;
}

int digits_cols(const Dla& d, const double* B, int64_t K, int64_t N, int64_t ldb, uint32_t* out, int64_t ldk,
                int* exps) {
  BSRHT_CUDA_TRY(cudaMemsetAsync(exps, 0, sizeof(int) * (size_t)N, d.s));
  const unsigned cb = (unsigned)((N + 63) / 64), ry = row_parts(K, cb);
  k_col_exps<<<dim3(cb, ry), 64, 0, d.s>>>(B, K, N, ldb, (K + ry - 1) / ry, exps);
  BSRHT_CUDA_TRY(cudaGetLastError());
  const int64_t tn = (N + 31) / 32, tiles = tn * ((ldk + 63) / 64);
  if (tiles > 0x7FFFFFFF) return BSRHT_EUNSUP;
  k_digits_cols<<<(unsigned)tiles, 256, 0, d.s>>>(B, K, N, ldb, out, ldk, exps, tn);
  BSRHT_CUDA_TRY(cudaGetLastError());
  note_launches(2);
  return BSRHT_OK;
}

size_t digit_bytes_of(int64_t rows, int64_t ldk) { return (size_t)kDig * 2 * (size_t)rows * (size_t)ldk; }

}  // namespace

// Scratch the digits of one launch may take, 14 bytes an entry: a bound on the
// workspace rather than a rule of speed.  A pass with fewer tiles than SMs splits
// K instead, as far as half a wave is gained (N = 256: a whole wave of 128 x 64
// tiles up to K = 2800, at K = 4096 a pass has 108 tiles).
constexpr size_t kDigitScratch = (size_t)192 << 20;

// Measured on GB300 (int8x7 against the CUDA-core GEMM, FP64): below about 20
// million FMAs the preparation's launches cost more than they save (256^3
// 0.051 / 0.050 ms, 300^3 0.050 / 0.083, 400^3 0.053 / 0.197).
bool gemm_int8x7_wants(int64_t M, int64_t N, int64_t K) {
  return M >= 32 && N >= 16 && K >= 32 && (double)M * (double)N * (double)K >= 2e7;
}

// See dla.cuh.
int gemm_int8x7(const Dla& d, Arena& ar, int64_t M, int64_t N, int64_t K, const double* A, int64_t lda, bool a_trans,
                const double* B, int64_t ldb, double* C, int64_t ldc, bool b_upper, bool gram) {
  using S = sl::Int8x7;
  if (gram && !a_trans) return BSRHT_EUNSUP;
  if (gram || a_trans) b_upper = false;
  const int64_t tn = (N + S::BN - 1) / S::BN;
  // What take() below uses, to the byte: a product that is the peak of a call
  // runs as it was measured in a workspace of the measured size.
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t avail = ar.measure ? (size_t)-1 : (ar.cap > up(ar.used) ? ar.cap - up(ar.used) : 0);
  const int64_t sms = num_sms();
  // Rows of A (A^T: columns of K) whose digits are made and used at a time.
  // Both dimensions of a pass stay small enough that the digits of one pass
  // fit the scratch; the split of K fills the SMs when the tiles do not.
  int64_t mc = M, kc = K;
  const int64_t ldk_full = round_up(K, 8);
  int splits = 1, passes = 1;
  auto tiles_of = [&](int64_t m) {
    int64_t t = 0;
    const int64_t tm = (m + sl::BM - 1) / sl::BM;
    for (int64_t bm = 0; bm < tm; ++bm)
      for (int64_t bn = 0; bn < tn; ++bn) t += (gram && sl::int8x7_skipped(bm, bn)) ? 0 : 1;
    return t;
  };
  auto splits_of = [&](int64_t tiles, int64_t k) {
    const int64_t groups = (k + S::KG * S::BK - 1) / (S::KG * S::BK);
    if (tiles >= sms) return (int64_t)1;
    return std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>((sms + tiles / 2) / tiles, groups), 64));
  };
  auto need = [&]() {
    const int64_t rows = a_trans ? M : mc, ld = a_trans ? round_up(kc, 8) : ldk_full;
    const bool part = splits > 1 || gram || (a_trans && passes > 1);
    return up(digit_bytes_of(N, ld)) + up(sizeof(int) * (size_t)N) +
           (gram ? 0 : up(digit_bytes_of(rows, ld)) + up(sizeof(int) * (size_t)rows)) +
           (part ? sizeof(double) * (size_t)(a_trans ? splits * passes : splits) * (size_t)M * (size_t)N : 0);
  };
  if (!a_trans) {
    const size_t of_b = up(digit_bytes_of(N, ldk_full)) + up(sizeof(int) * (size_t)N);
    const size_t budget = std::min(kDigitScratch, avail > of_b ? avail - of_b : 0);
    const int64_t fit = (int64_t)(budget / digit_bytes_of(1, ldk_full));
    if (fit < std::min<int64_t>(M, sl::BM)) return BSRHT_EUNSUP;
    if (mc > fit) {
      mc = fit / sl::BM * sl::BM;
      // Whole waves of tiles when a pass holds at least one.
      const int64_t wave = std::max<int64_t>(1, sms / tn) * sl::BM;
      if (mc > wave) mc = mc / wave * wave;
    }
    splits = (int)splits_of(tiles_of(mc), K);
    if (need() > avail) splits = 1;
    while (need() > avail && mc > sl::BM) mc = (mc - 1) / sl::BM * sl::BM;
    passes = (int)((M + mc - 1) / mc);
  } else {
    const size_t per_k = digit_bytes_of(gram ? N : M + N, 8) / 8;
    const int64_t groups_min = S::KG * S::BK;
    const int64_t tiles = tiles_of(M);
    auto plan = [&](size_t budget) {
      kc = std::min<int64_t>(K, (int64_t)(budget / per_k) / groups_min * groups_min);
      if (kc < groups_min && kc < K) return false;
      passes = (int)((K + kc - 1) / kc);
      kc = std::min<int64_t>(K, round_up((K + passes - 1) / passes, groups_min));
      passes = (int)((K + kc - 1) / kc);
      splits = (int)splits_of(tiles, kc);
      return true;
    };
    if (!plan(kDigitScratch)) return BSRHT_EUNSUP;
    if (need() > avail && !plan(std::min(kDigitScratch, avail / 2))) return BSRHT_EUNSUP;
  }
  if (need() > avail) return BSRHT_EUNSUP;
  const int64_t ldk = round_up(a_trans ? kc : K, 8);
  uint32_t* bd = static_cast<uint32_t*>(ar.take(digit_bytes_of(N, ldk)));
  uint32_t* ad = gram ? bd : static_cast<uint32_t*>(ar.take(digit_bytes_of(a_trans ? M : mc, ldk)));
  int* eb = static_cast<int*>(ar.take(sizeof(int) * (size_t)N));
  int* ea = gram ? eb : static_cast<int*>(ar.take(sizeof(int) * (size_t)(a_trans ? M : mc)));
  // Partials: split K, several passes over K, or the mirror of a Gram.
  const bool part = splits > 1 || gram || (a_trans && passes > 1);
  const int parts = a_trans ? splits * passes : splits;
  double* P = part ? static_cast<double*>(ar.take(sizeof(double) * (size_t)parts * M * N)) : nullptr;
  if (!ar.ok()) return BSRHT_ENOMEM;
  if (ar.measure) return BSRHT_OK;

  BSRHT_CUDA_TRY(cudaFuncSetAttribute(sl::k_gemm_int8x7, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)S::smem_bytes()));
  const CUtensorMapDataType f16 = CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  const CUtensorMapSwizzle swz = CU_TENSOR_MAP_SWIZZLE_64B;
  auto launch = [&](int64_t m, int64_t k, double* out, int64_t ldo, int z) -> int {
    CUtensorMap ma, mb;
    if (!make_slice_map(&ma, ad, f16, k, m, kDig, ldk, S::BK, sl::BM, swz, kDig) ||
        !make_slice_map(&mb, bd, f16, k, N, kDig, ldk, S::BK, S::BN, swz, kDig))
      return BSRHT_EUNSUP;
    const int64_t tiles = (m + sl::BM - 1) / sl::BM * tn;
    if (tiles > 0x7FFFFFFF) return BSRHT_EUNSUP;
    sl::Int8x7Args g{m, N, k, out, ldo, ea, eb, part ? 1 : 0, gram ? 1 : 0, b_upper ? 1 : 0, d.status};
    sl::k_gemm_int8x7<<<dim3((unsigned)tiles, 1u, (unsigned)z), sl::kThreads, S::smem_bytes(), d.s>>>(ma, mb, g);
    BSRHT_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return BSRHT_OK;
  };
  auto reduce = [&](int64_t m, double* c) -> int {
    k_int8x7_reduce<<<(unsigned)((m * N + 255) / 256), 256, 0, d.s>>>(P, c, m, N, ldc, parts, gram ? 1 : 0);
    BSRHT_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return BSRHT_OK;
  };
  if (!a_trans) {
    TRY_SL(digits_cols(d, B, K, N, ldb, bd, ldk, eb));
    for (int64_t i0 = 0; i0 < M; i0 += mc) {
      const int64_t m = std::min(mc, M - i0);
      TRY_SL(digits_rows(d, A + i0 * lda, m, K, lda, ad, ldk, ea));
      TRY_SL(launch(m, K, part ? P : C + i0 * ldc, ldc, splits));
      if (part) TRY_SL(reduce(m, C + i0 * ldc));
    }
    return BSRHT_OK;
  }
  for (int q = 0; q < passes; ++q) {
    const int64_t k0 = (int64_t)q * kc, k = std::min(kc, K - k0);
    TRY_SL(digits_cols(d, B + k0 * ldb, k, N, ldb, bd, ldk, eb));
    if (!gram) TRY_SL(digits_cols(d, A + k0 * lda, k, M, lda, ad, ldk, ea));
    TRY_SL(launch(M, k, part ? P + (size_t)q * splits * M * N : C, ldc, splits));
  }
  return part ? reduce(M, C) : BSRHT_OK;
}

namespace {

// Scratch and preparation of the NS slices of B (K x N) shared by the two
// kernels that split it once: slices (16-bit, K-major), column scales.
struct SlicedB {
  void* slices;
  float* scale;
  int64_t ldk;
  int bn;  // column tiles of equal width (a multiple of 16, at most 256)
};

size_t sliced_b_bytes(int64_t K, int64_t N, int ns) {
  return 2 * (size_t)ns * (size_t)N * (size_t)round_up(K, 8) + 8 * (size_t)N + 4096;
}

template <typename T16, int NS>
int slice_b(const Dla& d, Arena& ar, int64_t K, int64_t N, DT tb, const void* B, int64_t ldb, SlicedB* out,
            float undo = 1.f) {
  out->ldk = round_up(K, 8);
  out->slices = ar.take(2 * (size_t)NS * (size_t)N * out->ldk);
  int* exps = static_cast<int*>(ar.take(sizeof(int) * (size_t)N));
  out->scale = static_cast<float*>(ar.take(sizeof(float) * (size_t)N));
  const int64_t tn = (N + 255) / 256;
  out->bn = (int)round_up((N + tn - 1) / tn, 16);
  if (!ar.ok()) return BSRHT_ENOMEM;
  if (ar.measure) return BSRHT_OK;
  BSRHT_CUDA_TRY(cudaMemsetAsync(exps, 0, sizeof(int) * (size_t)N, d.s));
  const unsigned cb = (unsigned)((N + 63) / 64), ry = row_parts(K, cb);
  const int64_t t64 = (N + 63) / 64, tk = t64 * ((out->ldk + 63) / 64);
  if (tk > 0x7FFFFFFF) return BSRHT_EUNSUP;
  auto prep = [&](auto* b) {
    using TB = std::remove_pointer_t<decltype(b)>;
    k_col_exps32<TB><<<dim3(cb, ry), 64, 0, d.s>>>(b, K, N, ldb, (K + ry - 1) / ry, exps);
    k_slices16_cols<TB, T16, NS><<<(unsigned)tk, 256, 0, d.s>>>(b, K, N, ldb, static_cast<T16*>(out->slices), out->ldk,
                                                                 exps, t64, out->scale, undo);
  };
  if (tb == DT::F64)
    prep(static_cast<const double*>(B));
  else
    prep(static_cast<const float*>(B));
  BSRHT_CUDA_TRY(cudaGetLastError());
  note_launches(2);
  return BSRHT_OK;
}

}  // namespace

bool gemm_a16_eligible(DT ta, int64_t M, int64_t N, int64_t K, const void* A, int64_t lda) {
  return (ta == DT::BF16 || ta == DT::F16) && M >= 256 && N >= 1 && K >= 64 && (lda % 8) == 0 &&
         (reinterpret_cast<uintptr_t>(A) % 16) == 0;
}

int gemm_a16(const Dla& d, Arena& ar, DT ta, int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, DT tb,
             const void* B, int64_t ldb, float* C, int64_t ldc, float* Ct) {
  using S = sl::A16;
  if (tb != DT::F32 && tb != DT::F64) return BSRHT_EUNSUP;
  if (!ar.measure && ar.used + sliced_b_bytes(K, N, S::NB) > ar.cap) return BSRHT_EUNSUP;
  const bool bf = ta == DT::BF16;
  SlicedB b;
  TRY_SL(bf ? (slice_b<__nv_bfloat16, S::NB>(d, ar, K, N, tb, B, ldb, &b))
            : (slice_b<__half, S::NB>(d, ar, K, N, tb, B, ldb, &b)));
  if (ar.measure) return BSRHT_OK;
  const int64_t tiles = (M + sl::BM - 1) / sl::BM * ((N + b.bn - 1) / b.bn);
  if (tiles > 0x7FFFFFFF) return BSRHT_EUNSUP;
  const CUtensorMapDataType dt = bf ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  CUtensorMap ma, mb;
  if (!make_tensor_map_2d(&ma, A, dt, 2, (uint64_t)M, (uint64_t)K, (uint64_t)lda, S::BK, sl::BM,
                          CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_slice_map(&mb, b.slices, dt, K, N, S::NB, b.ldk, S::BK, (uint32_t)b.bn, CU_TENSOR_MAP_SWIZZLE_128B,
                      1))
    return BSRHT_EUNSUP;
  BSRHT_CUDA_TRY(
      cudaFuncSetAttribute(sl::k_gemm_a16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem_bytes()));
  sl::A16Args g{M, N, K, C, ldc, b.scale, Ct, M, b.bn, bf ? 1 : 0, d.status};
  sl::k_gemm_a16<<<(unsigned)tiles, sl::kThreads, S::smem_bytes(), d.s>>>(ma, mb, g);
  BSRHT_CUDA_TRY(cudaGetLastError());
  note_launches(1);
  return BSRHT_OK;
}

// Tiles enough for most SMs (the other kernel splits K instead) and not a wave
// with little more than it (12290 x 1536 x 257, 1.3 waves: 0.111 ms against 0.102
// in TF32; 16000 x 1536 x 512, 1.6 waves: 0.126 against 0.151), K short enough for
// a chain of at most 256 folds, and K and the tile long and wide against a
// tile's start and stores, which nothing overlaps: 65536 x 2000 x 400 0.44 ms
// against 0.70 in TF32, 262144 x 1024 x 256 0.58 against 0.69, but 2^20 x 512 x 512
// (upper triangular) 2.7 ms against 2.8, 2^20 x 512 x 100 1.32 against 1.24 and
// 262144 x 2048 x 128, one 128-wide tile, 0.81 against 0.73.
bool gemm_f32x2_eligible(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda) {
  const int64_t tiles = (M + sl::BM - 1) / sl::BM * ((N + 255) / 256), sms = num_sms();
  return M >= 128 * 96 && N > 128 && (tiles <= sms || 2 * tiles >= 3 * sms) && K >= 1024 && K <= 256 * 64 &&
         (lda % 4) == 0 && (reinterpret_cast<uintptr_t>(A) % 16) == 0;
}

int gemm_f32x2(const Dla& d, Arena& ar, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, DT tb,
               const void* B, int64_t ldb, DT tc_out, void* C, int64_t ldc, bool b_upper, float* Ct) {
  using S = sl::F32x2;
  if ((tb != DT::F32 && tb != DT::F64) || (tc_out != DT::F32 && tc_out != DT::F64)) return BSRHT_EUNSUP;
  if (!ar.measure && ar.used + sliced_b_bytes(K, N, S::NB) > ar.cap) return BSRHT_EUNSUP;
  SlicedB b;
  TRY_SL((slice_b<__half, S::NB>(d, ar, K, N, tb, B, ldb, &b, 1.f / S::LOWER)));
  if (ar.measure) return BSRHT_OK;
  const int64_t tiles = (M + sl::BM - 1) / sl::BM * ((N + b.bn - 1) / b.bn);
  if (tiles > 0x7FFFFFFF) return BSRHT_EUNSUP;
  CUtensorMap ma, mb;
  if (!make_tensor_map_2d(&ma, A, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (uint64_t)M, (uint64_t)K, (uint64_t)lda, S::BK,
                          sl::BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_slice_map(&mb, b.slices, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, K, N, S::NB, b.ldk, S::BK,
                      (uint32_t)b.bn, CU_TENSOR_MAP_SWIZZLE_64B, 1))
    return BSRHT_EUNSUP;
  sl::F32x2Args g{M, N, K, C, ldc, b.scale, Ct, M, b.bn, b_upper ? 1 : 0, d.status};
  auto launch = [&](auto kern) -> int {
    BSRHT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem_bytes()));
    kern<<<(unsigned)tiles, S::THREADS, S::smem_bytes(), d.s>>>(ma, mb, g);
    BSRHT_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return BSRHT_OK;
  };
  return tc_out == DT::F32 ? launch(sl::k_gemm_f32x2<float>) : launch(sl::k_gemm_f32x2<double>);
}

}  // namespace bsrht
