// FP32 one-sided Jacobi of l <= 768 columns in one thread-block cluster.
//
// The columns live in the shared memory of the cluster's NC CTAs for the
// whole iteration (no global memory, no grid barrier between rounds): 2 NC
// blocks of B columns on a line, CTA c holding positions 2c and 2c + 1.
// Odd-even ordering: in an even step each CTA treats the cross pairs of its
// two blocks, in an odd step those of positions 2c + 1 and 2c + 2; the two
// blocks of a step change places afterwards, so 2 NC steps bring every pair of
// blocks together once, and one block per CTA moves to a neighbour's shared
// memory between steps (even -> odd to the left, odd -> even to the right).
// The pairs inside the blocks are treated in the first step of a sweep.
//
// A step: warp w keeps columns 2w and 2w + 1 of the first block in registers
// over B / 2 rounds and meets columns 2q and 2q + 1, q = (w + r) mod (B / 2),
// of the second one: two times two independent pairs per round, so that one
// pair's latency (dot product, warp sum, rotation scalars) hides the other's
// and a column moves through shared memory once for two rotations.  What
// bounds it: that latency chain and one barrier a round (l = 512: 256 rounds
// of 1.5 us a sweep).
//
// No rotations are accumulated: the columns rotated are those of M^T, and
// when they are orthogonal their directions are M's right singular vectors.
#pragma once

#include <cooperative_groups.h>

#include "f32x2.cuh"

namespace bsrht {
namespace jc {

namespace cg = cooperative_groups;

constexpr int kMaxB = 24;
constexpr int kMaxRows = 768;

struct Args {
  float* X;          // l columns of `rows` entries, contiguous
  int l, rows, ld;   // ld: column stride in shared memory (rows rounded up to 4)
  int B;             // columns per block (even)
  float tol2, tstop2;   // squared cosine thresholds: rotate / significant
  float tiny2;          // columns both at or below this squared norm are left alone
  int lead;          // a rotation counts when one of its columns is among the `lead` largest (0: always)
  int need;          // columns above the zero threshold without which there is nothing to do
  int max_sweeps;
  int* rot_counts;   // [max_sweeps + 1], zeroed; the last one counts the columns above the threshold
  float* nrm;        // [2 NC B]: squared column norms between sweeps
};

inline size_t smem_bytes(int B, int ld, int nc) {
  return sizeof(float) * (3 * (size_t)B * ld + 3 * (size_t)B + 2 * (size_t)nc * B) + 64;
}

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// tan(theta) of the rotation that makes a pair with squared norms alpha,
// beta and product gamma orthogonal (the smaller root), h / (|d| + sqrt(d^2 +
// h^2)) with d = beta - alpha, h = 2 gamma: norms are at most 4 and one of
// the two is above the zero threshold, so the squares stay in range.
// Approximate root and division: the rotation is orthogonal for any t, and a
// relative error of t leaves that fraction of the cosine.
__device__ __forceinline__ float tangent(float alpha, float beta, float gamma) {
  const float d = beta - alpha, h = 2.f * gamma;
  const float t = __fdividef(h, fabsf(d) + sqrt_approx(fmaf(d, d, h * h)));
  return d >= 0.f ? t : -t;
}

// JQ: 16-byte chunks of a column per lane (rows <= 128 JQ).
template <int JQ, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_jacobi_cluster(Args a) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) float js[];
  const int NC = (int)cluster.num_blocks(), c = (int)cluster.block_rank();
  const int B = a.B, ld = a.ld, bl = B * ld;
  float* nrm = js + 3 * (size_t)bl;                      // [3][B]
  float* all_nrm = nrm + 3 * B;                          // [2 NC B]
  int* ids = reinterpret_cast<int*>(all_nrm + 2 * NC * B);  // block held by each buffer
  float* s_th = reinterpret_cast<float*>(ids + 3);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, NT = blockDim.x;
  const int n4 = ld / 4;                                  // 16-byte chunks of a column
  const ulonglong2 z2 = make_ulonglong2(0ull, 0ull);

  // Buffers: lo, hi hold positions 2c and 2c + 1, fr is free.  Every CTA but
  // the last has the same assignment; the last one's (L*) differs because
  // its upper block stays where it is in odd steps.
  int lo = 0, hi = 1, fr = 2, Llo = 0, Lhi = 1;
  const bool is_last = c == NC - 1;
  auto my = [&](int u, int v) { return is_last ? v : u; };
  for (int e = threadIdx.x; e < 2 * B * ld; e += NT) {
    const int h = e / bl, r = e - h * bl, j = r / ld, i = r - j * ld;
    const int64_t col = (int64_t)(2 * c + h) * B + j;
    js[e] = (col < a.l && i < a.rows) ? a.X[col * a.rows + i] : 0.f;
  }
  if (threadIdx.x < 3) ids[threadIdx.x] = 2 * c + (int)threadIdx.x;
  if (threadIdx.x == 0) *s_th = 0.f;
  __syncthreads();

  int mycount = 0;
  float th = 0.f;  // squared norm that makes a rotation count
  auto chunk = [&](int e) { return 32 * e + lane; };
  auto sq = [&](const ulonglong2* p) {
    f2 g0 = 0ull, g1 = 0ull;
#pragma unroll
    for (int e = 0; e < JQ; ++e) {
      const ulonglong2 v = chunk(e) < n4 ? p[chunk(e)] : z2;
      g0 = f2_fma(v.x, v.x, g0);
      g1 = f2_fma(v.y, v.y, g1);
    }
    const float2 g = f2_to_float2(f2_add(g0, g1));
    return wsum(g.x + g.y);
  };
  auto load = [&](ulonglong2(&x)[JQ], const ulonglong2* p) {
#pragma unroll
    for (int e = 0; e < JQ; ++e) x[e] = chunk(e) < n4 ? p[chunk(e)] : z2;
  };
  auto store = [&](const ulonglong2(&x)[JQ], ulonglong2* p) {
#pragma unroll
    for (int e = 0; e < JQ; ++e)
      if (chunk(e) < n4) p[chunk(e)] = x[e];
  };
  auto dot = [&](const ulonglong2(&x)[JQ], const ulonglong2(&y)[JQ]) {
    f2 g0 = 0ull, g1 = 0ull;
#pragma unroll
    for (int e = 0; e < JQ; ++e) {
      g0 = f2_fma(x[e].x, y[e].x, g0);
      g1 = f2_fma(x[e].y, y[e].y, g1);
    }
    const float2 g = f2_to_float2(f2_add(g0, g1));
    return g.x + g.y;
  };
  // Tangent of the pair's rotation, 0 for none; squared norms updated.
  auto scalars = [&](float gamma, float& alpha, float& beta) {
    const float g2 = gamma * gamma, ab = alpha * beta;
    if (!(g2 > a.tol2 * ab) || (alpha <= a.tiny2 && beta <= a.tiny2)) return 0.f;
    const float t = tangent(alpha, beta, gamma);
    if (g2 > a.tstop2 * ab && fmaxf(alpha, beta) >= th) ++mycount;
    alpha = fmaf(-t, gamma, alpha);
    beta = fmaf(t, gamma, beta);
    return t;
  };
  auto rotate = [&](ulonglong2(&x)[JQ], ulonglong2(&y)[JQ], float t) {
    const float cs = rsqrtf(fmaf(t, t, 1.f)), sn = cs * t;
    const f2 C2 = f2_splat(cs), S2 = f2_splat(sn), N2 = f2_splat(-sn);
#pragma unroll
    for (int e = 0; e < JQ; ++e) {
      const ulonglong2 u = x[e], v = y[e];
      x[e].x = f2_fma(v.x, N2, f2_mul(u.x, C2));
      x[e].y = f2_fma(v.y, N2, f2_mul(u.y, C2));
      y[e].x = f2_fma(v.x, C2, f2_mul(u.x, S2));
      y[e].y = f2_fma(v.y, C2, f2_mul(u.y, S2));
    }
  };
  // Two independent pairs (x1, y1) and (x2, y2), side by side.
  auto pair2 = [&](ulonglong2(&x1)[JQ], float& a1, ulonglong2(&y1)[JQ], float& b1, ulonglong2(&x2)[JQ], float& a2,
                   ulonglong2(&y2)[JQ], float& b2) {
    float g1 = dot(x1, y1), g2 = dot(x2, y2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      g1 += __shfl_xor_sync(0xffffffffu, g1, o);
      g2 += __shfl_xor_sync(0xffffffffu, g2, o);
    }
    const float t1 = scalars(g1, a1, b1), t2 = scalars(g2, a2, b2);
    if (t1 != 0.f || t2 != 0.f) {  // warp-uniform
      rotate(x1, y1, t1);
      rotate(x2, y2, t2);
    }
  };
  auto colp = [&](int buf, int j) { return reinterpret_cast<ulonglong2*>(js + (size_t)buf * bl + (size_t)j * ld); };

  // Cross pairs of the blocks in buffers P and Q.
  const int H = B / 2;
  auto cross = [&](int P, int Q) {
    ulonglong2 x1[JQ], x2[JQ];
    load(x1, colp(P, 2 * w));
    load(x2, colp(P, 2 * w + 1));
    float a1 = wsum(dot(x1, x1)), a2 = wsum(dot(x2, x2));
    {
      const float q1 = sq(colp(Q, 2 * w)), q2 = sq(colp(Q, 2 * w + 1));
      if (lane == 0) {
        nrm[Q * B + 2 * w] = q1;
        nrm[Q * B + 2 * w + 1] = q2;
      }
    }
    __syncthreads();
    int q = w;
    for (int r = 0; r < H; ++r) {
      ulonglong2 y1[JQ], y2[JQ];
      ulonglong2 *p1 = colp(Q, 2 * q), *p2 = colp(Q, 2 * q + 1);
      load(y1, p1);
      load(y2, p2);
      float2* bn = reinterpret_cast<float2*>(&nrm[Q * B + 2 * q]);
      float2 b = *bn;
      pair2(x1, a1, y1, b.x, x2, a2, y2, b.y);
      pair2(x1, a1, y2, b.y, x2, a2, y1, b.x);
      store(y1, p1);
      store(y2, p2);
      if (lane == 0) *bn = b;
      if (++q == H) q = 0;
      __syncthreads();
    }
    store(x1, colp(P, 2 * w));
    store(x2, colp(P, 2 * w + 1));
  };
  // Pairs inside both blocks (round robin; each warp one pair of each).
  auto inside = [&](int P, int Q) {
    for (int h = 0; h < 2; ++h) {
      const float pn = sq(colp(P, 2 * w + h)), qn = sq(colp(Q, 2 * w + h));
      if (lane == 0) {
        nrm[P * B + 2 * w + h] = pn;
        nrm[Q * B + 2 * w + h] = qn;
      }
    }
    __syncthreads();
    for (int r = 0; r < B - 1; ++r) {
      const int i = w == 0 ? 0 : 1 + (w - 1 + r) % (B - 1);
      const int j = 1 + (B - 2 - w + r) % (B - 1);
      ulonglong2 x1[JQ], y1[JQ], x2[JQ], y2[JQ];
      load(x1, colp(P, i));
      load(y1, colp(P, j));
      load(x2, colp(Q, i));
      load(y2, colp(Q, j));
      float a1 = nrm[P * B + i], b1 = nrm[P * B + j], a2 = nrm[Q * B + i], b2 = nrm[Q * B + j];
      pair2(x1, a1, y1, b1, x2, a2, y2, b2);
      store(x1, colp(P, i));
      store(y1, colp(P, j));
      store(x2, colp(Q, i));
      store(y2, colp(Q, j));
      __syncwarp();
      if (lane == 0) {
        nrm[P * B + i] = a1;
        nrm[P * B + j] = b1;
        nrm[Q * B + i] = a2;
        nrm[Q * B + j] = b2;
      }
      __syncthreads();
    }
  };
  // Copies this CTA's buffer `from` into buffer `to` of CTA `rank`.
  auto send = [&](int from, int to, int rank) {
    float4* dst = reinterpret_cast<float4*>(cluster.map_shared_rank(js, rank)) + (size_t)to * bl / 4;
    const float4* src = reinterpret_cast<const float4*>(js) + (size_t)from * bl / 4;
#pragma unroll 4
    for (int e = threadIdx.x; e < bl / 4; e += NT) dst[e] = src[e];
    if (threadIdx.x == 0) cluster.map_shared_rank(ids, rank)[to] = ids[from];
  };

  // A matrix whose `need` largest triplets FP32 does not resolve (rows of a
  // triangular factor at the rounding of the largest) is left as it is: the
  // caller finds its columns far from orthogonal and takes another path, which
  // it would after the sweeps as well (rSVD of 16384 x 800, l = 400, sigma_i =
  // exp(-i / 40): 29.4 -> 25.5 ms; the count costs 1 us).
  {
    int live = 0;
    for (int h = 0; h < 2; ++h)
      live += (sq(colp(lo, 2 * w + h)) > a.tiny2) + (sq(colp(hi, 2 * w + h)) > a.tiny2);
    if (lane == 0) atomicAdd(&a.rot_counts[a.max_sweeps], live);
    __threadfence();
  }
  cluster.sync();
  if (__ldcg(&a.rot_counts[a.max_sweeps]) < a.need) return;  // the same in every CTA
  for (int sweep = 0; sweep < a.max_sweeps; ++sweep) {
    mycount = 0;
    for (int step = 0; step < NC; ++step) {
      {  // even step: positions 2c, 2c + 1
        const int P = my(lo, Llo), Q = my(hi, Lhi);
        if (step == 0) inside(P, Q);
        cross(P, Q);
        __syncthreads();
        // The block of Q is now the lower one: it goes left.
        if (c > 0) send(Q, fr, c - 1);
        cluster.sync();
      }
      {  // odd step: positions 2c + 1 (buffer lo) and 2c + 2 (buffer fr)
        if (!is_last) {
          cross(lo, fr);
          __syncthreads();
          // The block of lo is now the upper one: it goes right, where the
          // buffer of the block sent left is free.
          send(lo, c + 1 == NC - 1 ? Lhi : hi, c + 1);
        }
        cluster.sync();
        // Lower block in hi (CTA 0 kept it there), upper one in fr, lo free;
        // the last CTA's upper block stayed in its lo.
        int t = lo;
        lo = hi;
        hi = fr;
        fr = t;
        t = Llo;
        Llo = Lhi;
        Lhi = t;
      }
    }
    // Norms of the columns by position, the sweep's count, and the norm a
    // counting rotation needs in the next sweep.
    {
      const int b0 = my(lo, Llo), b1 = my(hi, Lhi);
      for (int h = 0; h < 2; ++h) {
        const float n0 = sq(colp(b0, 2 * w + h)), n1 = sq(colp(b1, 2 * w + h));
        if (lane == 0) {
          a.nrm[(2 * c) * B + 2 * w + h] = n0;
          a.nrm[(2 * c + 1) * B + 2 * w + h] = n1;
        }
      }
      if (lane == 0 && mycount) atomicAdd(&a.rot_counts[sweep], mycount);
      __threadfence();
      cluster.sync();
      if (__ldcg(&a.rot_counts[sweep]) == 0) break;
      if (a.lead > 0) {
        const int tot = 2 * NC * B;
        for (int j = threadIdx.x; j < tot; j += NT) all_nrm[j] = __ldcg(&a.nrm[j]);
        __syncthreads();
        for (int j = threadIdx.x; j < tot; j += NT) {
          const float v = all_nrm[j];
          int rank = 0;
          for (int e = 0; e < tot; ++e) {
            const float u = all_nrm[e];
            rank += (u > v) || (u == v && e < j);
          }
          if (rank == a.lead - 1) *s_th = 0.999f * v;
        }
        __syncthreads();
        th = *s_th;
      }
    }
  }
  __syncthreads();
  for (int h = 0; h < 2; ++h) {
    const int buf = h ? my(hi, Lhi) : my(lo, Llo);
    const int64_t c0 = (int64_t)ids[buf] * B;
    const float* src = js + (size_t)buf * bl;
    for (int e = threadIdx.x; e < bl; e += NT) {
      const int j = e / ld, i = e - j * ld;
      if (c0 + j < a.l && i < a.rows) a.X[(c0 + j) * a.rows + i] = src[e];
    }
  }
  cluster.sync();  // no CTA leaves while a neighbour may still write to it
}

}  // namespace jc
}  // namespace bsrht
