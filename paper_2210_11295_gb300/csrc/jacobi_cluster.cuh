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
// A step: one warp per pair.  Warp w keeps column w of the first block in
// registers over the B rounds and meets column (w + r) mod B of the second
// one in shared memory, so a round moves one column in and out instead of
// two.  What bounds it: the latency of a round (dot product, warp sum,
// rotation scalars, barrier) and, from l = 512 on, shared-memory bandwidth.
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
  int max_sweeps;
  int* rot_counts;   // [max_sweeps], zeroed
  float* nrm;        // [2 NC B]: squared column norms between sweeps
};

inline size_t smem_bytes(int B, int ld) { return sizeof(float) * (3 * (size_t)B * ld + 3 * (size_t)B) + 64; }

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
// beta and product gamma orthogonal (the smaller root).  Approximate division
// and square root: the rotation is orthogonal for any t, and a relative
// error of t leaves that fraction of the cosine.
__device__ __forceinline__ float tangent(float alpha, float beta, float gamma) {
  const float z = __fdividef(beta - alpha, 2.f * gamma);
  const float az = fabsf(z);
  const float t = az > 1e9f ? __fdividef(0.5f, az) : __fdividef(1.f, az + sqrt_approx(fmaf(az, az, 1.f)));
  return copysignf(t, z);
}

// JQ: 16-byte chunks of a column per lane (rows <= 128 JQ).
template <int JQ, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_jacobi_cluster(Args a) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) float js[];
  const int NC = (int)cluster.num_blocks(), c = (int)cluster.block_rank();
  const int B = a.B, ld = a.ld, bl = B * ld;
  float* nrm = js + 3 * (size_t)bl;                      // [3][B]
  int* ids = reinterpret_cast<int*>(nrm + 3 * B);        // block held by each buffer
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
  // Rotates x (registers) against the column yp (shared memory).
  auto pair = [&](ulonglong2(&x)[JQ], float& alpha, ulonglong2* yp, float* ynrm) {
    constexpr bool kKeep = JQ <= 4;  // y in registers between dot and rotation
    ulonglong2 y[kKeep ? JQ : 1];
    f2 g0 = 0ull, g1 = 0ull;
#pragma unroll
    for (int e = 0; e < JQ; ++e) {
      const ulonglong2 v = chunk(e) < n4 ? yp[chunk(e)] : z2;
      if constexpr (kKeep) y[e] = v;
      g0 = f2_fma(x[e].x, v.x, g0);
      g1 = f2_fma(x[e].y, v.y, g1);
    }
    const float beta = *ynrm;
    const float2 g = f2_to_float2(f2_add(g0, g1));
    const float gamma = wsum(g.x + g.y);
    const float g2 = gamma * gamma, ab = alpha * beta;
    if (!(g2 > a.tol2 * ab) || (alpha <= a.tiny2 && beta <= a.tiny2)) return;
    const float t = tangent(alpha, beta, gamma);
    const float cs = rsqrtf(fmaf(t, t, 1.f)), sn = cs * t;
    const f2 C2 = f2_splat(cs), S2 = f2_splat(sn), N2 = f2_splat(-sn);
#pragma unroll
    for (int e = 0; e < JQ; ++e) {
      if (chunk(e) < n4) {
        ulonglong2 v;
        if constexpr (kKeep)
          v = y[e];
        else
          v = yp[chunk(e)];
        ulonglong2 nx, ny;
        nx.x = f2_fma(v.x, N2, f2_mul(x[e].x, C2));
        nx.y = f2_fma(v.y, N2, f2_mul(x[e].y, C2));
        ny.x = f2_fma(v.x, C2, f2_mul(x[e].x, S2));
        ny.y = f2_fma(v.y, C2, f2_mul(x[e].y, S2));
        x[e] = nx;
        yp[chunk(e)] = ny;
      }
    }
    if (g2 > a.tstop2 * ab && fmaxf(alpha, beta) >= th) ++mycount;
    alpha = fmaf(-t, gamma, alpha);
    __syncwarp();  // every lane has read *ynrm
    if (lane == 0) *ynrm = fmaf(t, gamma, beta);
  };
  auto load_x = [&](ulonglong2(&x)[JQ], const ulonglong2* p) {
#pragma unroll
    for (int e = 0; e < JQ; ++e) x[e] = chunk(e) < n4 ? p[chunk(e)] : z2;
  };
  auto store_x = [&](const ulonglong2(&x)[JQ], ulonglong2* p) {
#pragma unroll
    for (int e = 0; e < JQ; ++e)
      if (chunk(e) < n4) p[chunk(e)] = x[e];
  };
  auto colp = [&](int buf, int j) { return reinterpret_cast<ulonglong2*>(js + (size_t)buf * bl + (size_t)j * ld); };

  // Cross pairs of the blocks in buffers P and Q.
  auto cross = [&](int P, int Q) {
    ulonglong2 x[JQ];
    load_x(x, colp(P, w));
    float alpha = 0.f;
    {
      f2 g0 = 0ull, g1 = 0ull;
#pragma unroll
      for (int e = 0; e < JQ; ++e) {
        g0 = f2_fma(x[e].x, x[e].x, g0);
        g1 = f2_fma(x[e].y, x[e].y, g1);
      }
      const float2 g = f2_to_float2(f2_add(g0, g1));
      alpha = wsum(g.x + g.y);
    }
    const float qn = sq(colp(Q, w));
    if (lane == 0) nrm[Q * B + w] = qn;
    __syncthreads();
    int q = w;
    for (int r = 0; r < B; ++r) {
      pair(x, alpha, colp(Q, q), &nrm[Q * B + q]);
      if (++q == B) q = 0;
      __syncthreads();
    }
    store_x(x, colp(P, w));
    if (lane == 0) nrm[P * B + w] = alpha;
  };
  // Pairs inside both blocks (round robin; warps 0 .. B/2-1 the first block).
  auto inside = [&](int P, int Q) {
    {
      const float pn = sq(colp(P, w)), qn = sq(colp(Q, w));
      if (lane == 0) {
        nrm[P * B + w] = pn;
        nrm[Q * B + w] = qn;
      }
    }
    __syncthreads();
    const int buf = w < B / 2 ? P : Q, k = w < B / 2 ? w : w - B / 2;
    for (int r = 0; r < B - 1; ++r) {
      const int i = k == 0 ? 0 : 1 + (k - 1 + r) % (B - 1);
      const int j = 1 + (B - 2 - k + r) % (B - 1);
      ulonglong2 x[JQ];
      load_x(x, colp(buf, i));
      float alpha = nrm[buf * B + i];
      pair(x, alpha, colp(buf, j), &nrm[buf * B + j]);
      store_x(x, colp(buf, i));
      __syncwarp();
      if (lane == 0) nrm[buf * B + i] = alpha;
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

  cluster.sync();
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
      const float n0 = sq(colp(b0, w)), n1 = sq(colp(b1, w));
      if (lane == 0) {
        a.nrm[(2 * c) * B + w] = n0;
        a.nrm[(2 * c + 1) * B + w] = n1;
        if (mycount) atomicAdd(&a.rot_counts[sweep], mycount);
      }
      __threadfence();
      cluster.sync();
      if (__ldcg(&a.rot_counts[sweep]) == 0) break;
      if (a.lead > 0) {
        const int tot = 2 * NC * B;
        for (int j = threadIdx.x; j < tot; j += NT) {
          const float v = __ldcg(&a.nrm[j]);
          int rank = 0;
          for (int e = 0; e < tot; ++e) {
            const float u = __ldcg(&a.nrm[e]);
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
