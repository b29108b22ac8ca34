// Pivoted Cholesky of a Hermitian PSD matrix with the rows in registers,
// by one CTA or by one thread-block cluster (FP32 and FP64).
//
// The factorisation is a chain of m dependent pivot steps, so it is bound by
// the latency of one step.  The CTA's last warp keeps the remaining diagonal
// and the pivot order; the other warps own whole rows (a lane holds every 32nd
// column).  Per step every row's owner stores its scaled entry of the pivot
// column into shared memory (of every CTA of the cluster), one barrier, then
// the row warps update their rows while the last warp updates the diagonal,
// finds the next pivot and takes its root and reciprocal, and a second barrier
// of the CTA alone.  Rows are never exchanged: a pivot only relabels them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tnbp {
namespace chol {

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// Address of this CTA's shared variable p in CTA `rank` of the cluster.
template <class T>
__device__ __forceinline__ T* in_cta(T* p, unsigned rank) {
  uint64_t q;
  asm("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(rank));
  return reinterpret_cast<T*>(q);
}

// a b + c d with the second product rounded first.
__device__ __forceinline__ float sum2(float a, float b, float c, float d) {
  return __fmaf_rn(a, b, __fmul_rn(c, d));
}

// a -= l_i conj(l_j)
__device__ __forceinline__ void update(float2& a, float2 li, float2 lj) {
  a.x = __fsub_rn(a.x, sum2(li.x, lj.x, li.y, lj.y));
  a.y = __fsub_rn(a.y, sum2(li.y, lj.x, -li.x, lj.y));
}
__device__ __forceinline__ void update(double2& a, double2 li, double2 lj) {
  a.x = fma(-li.x, lj.x, a.x);
  a.x = fma(-li.y, lj.y, a.x);
  a.y = fma(-li.y, lj.x, a.y);
  a.y = fma(li.x, lj.y, a.y);
}
// the same for a diagonal entry's real part
__device__ __forceinline__ void update_diag(float& d, float2 l) {
  d = __fsub_rn(d, sum2(l.x, l.x, l.y, l.y));
}
__device__ __forceinline__ void update_diag(double& d, double2 l) {
  d = fma(-l.x, l.x, d);
  d = fma(-l.y, l.y, d);
}

// Largest value over the warp and the lowest position that holds it.  Only
// values above zero matter (a non-positive pivot ends the factorisation), and
// for those the bit patterns order like the values.
__device__ __forceinline__ float warp_argmax(float v, unsigned pos, unsigned* at) {
  const int key = __float_as_int(v);
  const int top = __reduce_max_sync(0xffffffffu, key);
  *at = __reduce_min_sync(0xffffffffu, key == top ? pos : 0xffffffffu);
  return __int_as_float(top);
}
__device__ __forceinline__ double warp_argmax(double v, unsigned pos, unsigned* at) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int th = __reduce_max_sync(0xffffffffu, hi);
  const unsigned tl = __reduce_max_sync(0xffffffffu, hi == th ? lo : 0u);
  *at = __reduce_min_sync(0xffffffffu, hi == th && lo == tl ? pos : 0xffffffffu);
  return __hiloint2double(th, (int)tl);
}

__device__ __forceinline__ float root(float v) { return sqrtf(v); }
__device__ __forceinline__ double root(double v) { return sqrt(v); }
__device__ __forceinline__ float shfl(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ double shfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// v[u] for a warp-uniform u.
template <int N, class T>
__device__ __forceinline__ T pick(const T (&v)[N], int u) {
  T r = v[0];
#pragma unroll
  for (int i = 1; i < N; ++i)
    if (u == i) r = v[i];
  return r;
}

// P^T A P = L L^H of the m x m matrix load(i, j), called by every thread of the
// cluster (`ctas` CTAs, this one `rank`; 1: the CTA alone).  CV = ceil(m / 32)
// columns per lane and RW rows per row warp at least; column: shared [2][m].
// emit(i, k, l) receives L's entry of original row i in pivot column k from one
// lane (only entries that are not zero by construction); perm (shared, may be
// null) the original row at every pivot position.  A pivot at or below rel_tol
// times the largest initial diagonal ends it; returns the rank.  The caller
// synchronises before it reads what emit and perm wrote.
template <int CV, int RW, class T, class C, class Load, class Emit>
__device__ __forceinline__ int pivoted_cholesky(int m, int ctas, int rank, C* column, T rel_tol,
                                                Load load, Emit emit, int* perm) {
  __shared__ T next_root, next_inv;
  __shared__ int next_row;  // original row of the next pivot; -1 ends
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row_warps = (blockDim.x >> 5) - 1;
  if (warp == row_warps) {
    int order[CV];
    T d[CV];
#pragma unroll
    for (int u = 0; u < CV; ++u) {
      const int p = u * 32 + lane;
      order[u] = p;
      d[u] = p < m ? load(p, p).x : T(0);
    }
    T d0 = T(0);
    int k = 0;
    for (;; ++k) {
      // the pivot of step k, the lowest position among equal ones
      T best = T(-1);
      unsigned bp = 0xffffffffu, piv;
#pragma unroll
      for (int u = 0; u < CV; ++u) {
        const int p = u * 32 + lane;
        if (p >= k && p < m && d[u] > best) { best = d[u]; bp = p; }
      }
      const T pv = warp_argmax(best, bp, &piv);
      if (k == 0) d0 = pv > T(0) ? pv : T(0);
      const bool go = k < m && d0 > T(0) && pv > rel_tol * d0;
      if (go) {
        // relabel: positions k and piv change places
        const int ip = __shfl_sync(0xffffffffu, pick(order, piv >> 5), piv & 31);
        const int ik = __shfl_sync(0xffffffffu, pick(order, k >> 5), k & 31);
        const T dk = shfl(pick(d, k >> 5), k & 31);
#pragma unroll
        for (int u = 0; u < CV; ++u) {
          const int p = u * 32 + lane;
          if (p == (int)piv) { order[u] = ik; d[u] = dk; }
          if (p == k) order[u] = ip;
        }
        if (lane == 0) {
          const T dg = root(pv);
          next_root = dg;
          next_inv = T(1) / dg;
          next_row = ip;
        }
      } else if (lane == 0) {
        next_row = -1;
      }
      __syncthreads();
      if (!go) break;
      if (ctas == 1) __syncthreads();
      else cluster_sync();
      const C* col = column + (k & 1) * m;
#pragma unroll
      for (int u = 0; u < CV; ++u) {
        const int p = u * 32 + lane;
        if (p > k && p < m) update_diag(d[u], col[order[u]]);
      }
    }
    if (perm)
#pragma unroll
      for (int u = 0; u < CV; ++u)
        if (u * 32 + lane < m) perm[u * 32 + lane] = order[u];
    return k;
  }
  const int first = rank * row_warps + warp, stride = ctas * row_warps;
  C a[RW][CV];
  bool live[RW];
#pragma unroll
  for (int s = 0; s < RW; ++s) {
    const int i = first + s * stride;
    live[s] = i < m;
#pragma unroll
    for (int u = 0; u < CV; ++u) {
      const int c = u * 32 + lane;
      a[s][u].x = a[s][u].y = T(0);
      if (live[s] && c < m) a[s][u] = load(i, c);
    }
  }
  int k = 0;
  for (;; ++k) {
    __syncthreads();
    const int ip = next_row;
    if (ip < 0) break;
    const T inv = next_inv;
    C* col = column + (k & 1) * m;
#pragma unroll
    for (int s = 0; s < RW; ++s) {
      if (!live[s]) continue;
      const int i = first + s * stride;
      C l = pick(a[s], ip >> 5);
      l.x = shfl(l.x, ip & 31) * inv;
      l.y = shfl(l.y, ip & 31) * inv;
      if (i == ip) {
        live[s] = false;
        l.x = next_root;
        l.y = T(0);
      } else if (ctas == 1) {
        if (lane == 0) col[i] = l;
      } else if (lane < ctas) {
        *in_cta(col + i, lane) = l;
      }
      if (lane == 0) emit(i, k, l);
    }
    if (ctas == 1) __syncthreads();
    else cluster_sync();
    C lj[CV];
#pragma unroll
    for (int u = 0; u < CV; ++u)
      if (u * 32 + lane < m) lj[u] = col[u * 32 + lane];
#pragma unroll
    for (int s = 0; s < RW; ++s) {
      if (!live[s]) continue;
      const C li = col[first + s * stride];
#pragma unroll
      for (int u = 0; u < CV; ++u)
        if (u * 32 + lane < m) update(a[s][u], li, lj[u]);
    }
  }
  return k;
}

}  // namespace chol
}  // namespace tnbp
