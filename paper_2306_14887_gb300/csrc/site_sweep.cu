// One BP sweep's message contractions for small bond dimensions (chi <= 16) in
// one launch, FP32: every CTA carries one site's chain to one open leg (two mode
// products and the close) through shared memory.
//
// At these sizes the contractions of a sweep are a dozen dependent launches of a
// few microseconds of work each; the site tensor (64 KB at chi = 16) and the
// chain's intermediate fit an SM, so nothing but T is read and nothing but the
// message is written.  Bound by the shared-memory reads of the products.
// Measured, a whole sweep with normalisation and stop rule: 127 qubits at chi =
// 16 46 us (147 us as separate GEMM launches), 338 sites at chi = 16 79 us (201),
// 65 sites at chi = 9 24 us (173 with the GEMM before its rewrite).
//
// Every sum is taken exactly as the CUDA-core GEMM takes it (16-deep slices of
// the contraction in the same order, slice sums added by compensated two-sums,
// split-K parts added in FP64), so the messages are the same bit for bit.
//
// Degree 3, open leg o, first contracted leg f, second g (the chains of the
// sweep plan): a warp owns a slab (p, o), a chi x chi matrix over (g, f):
//   Y1[g][f'] = sum_f T[p, o, g, f] Mf[f][f'],  Y2[g'][f'] = sum_g Y1[g][f'] Mg[g][g']
// in place in shared memory; then all warps close over k = (p, g', f'),
//   out[o][o'] = sum_k Y2[o; k] conj(T[o'; k]),
// each warp taking every eighth slice for all outputs.
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "tnbp.h"

namespace tnbp {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxChi = 16;
constexpr int kOpen = 8;      // open-leg values per degree-3 CTA: two CTAs per site and leg at
                              // chi = 16, two of them on an SM
constexpr int kSlice = 16;    // slice depth of the CUDA-core GEMM

// s + c += b with s the rounded sum and c the accumulated rounding errors.
__device__ __forceinline__ void two_sum_acc(float& s, float& c, float b) {
  const float t = __fadd_rn(s, b);
  const float bb = __fsub_rn(t, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(b, bb));
  s = t;
  c = __fadd_rn(c, e);
}
// acc += a b
__device__ __forceinline__ void cmac(float& pr, float& pi, float ar, float ai, float br, float bi) {
  pr = fmaf(ar, br, pr);
  pi = fmaf(ar, bi, pi);
  pr = fmaf(-ai, bi, pr);
  pi = fmaf(ai, br, pi);
}

// rows x chi values of a planar global matrix into padded shared rows.
__device__ __forceinline__ void load_rows(float* dst, int ld, int64_t dst_plane, const float* src,
                                          int64_t plane, int rows, int chi) {
  const int per = kThreads / chi, r0 = threadIdx.x / chi, c = threadIdx.x - r0 * chi;
  if (r0 >= per) return;
#pragma unroll 8
  for (int r = r0; r < rows; r += per) {
    dst[r * ld + c] = src[(int64_t)r * chi + c];
    dst[dst_plane + r * ld + c] = src[plane + (int64_t)r * chi + c];
  }
}

__global__ void __launch_bounds__(kThreads, 2)
    site_sweep_kernel(const SiteJob* jobs, int chi, int3 splits3, const double* comp_state) {
  extern __shared__ __align__(16) float sm[];
  const SiteJob job = jobs[blockIdx.x];
  // a converged component of a union keeps its messages
  if (comp_state && comp_state[4 * job.comp + 3] != 0.0) return;
  const int ld = chi | 1, c2 = chi * chi;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (job.deg == 3) {
    const int trows = 2 * c2, tplane = trows * ld;
    const int yplane = 2 * kOpen * chi * ld;
    float* sT = sm;
    float* sMf = sT + 2 * tplane;
    float* sMg = sMf + 2 * c2;
    float* sY = sMg + 2 * c2;
    load_rows(sT, ld, tplane, job.T, 2 * (int64_t)c2 * chi, trows, chi);
    for (int i = tid; i < 2 * c2; i += kThreads) {
      sMf[i] = job.mf[i];
      sMg[i] = job.mg[i];
    }
    __syncthreads();
    // strides of the legs in the padded T: leg 0, 1, 2
    const int so = job.open == 0 ? chi * ld : job.open == 1 ? ld : 1;
    const int sf = job.open == 2 ? chi * ld : 1;       // f: leg 2, or leg 0 when leg 2 is open
    const int sg = job.open == 1 ? chi * ld : ld;      // g: leg 1, or leg 0 when leg 1 is open
    const int sp = c2 * ld;
    const int rg = lane >> 3, cg = lane & 7;
    for (int s = warp; s < 2 * job.on; s += kWarps) {
      const int p = s & 1, ol = s >> 1;
      const float* a0 = sT + p * sp + (job.o0 + ol) * so;
      float* y = sY + s * chi * ld;
      float pr[4][2], pi[4][2];
      int row[4], col[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) row[i] = min(rg + 4 * i, chi - 1);
#pragma unroll
      for (int j = 0; j < 2; ++j) col[j] = min(cg + 8 * j, chi - 1);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) pr[i][j] = pi[i][j] = 0.f;
      for (int k = 0; k < chi; ++k) {
        float ar[4], ai[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float* q = a0 + row[i] * sg + k * sf;
          ar[i] = q[0];
          ai[i] = q[tplane];
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float br = sMf[k * chi + col[j]], bi = sMf[c2 + k * chi + col[j]];
#pragma unroll
          for (int i = 0; i < 4; ++i) cmac(pr[i][j], pi[i][j], ar[i], ai[i], br, bi);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (rg + 4 * i < chi && cg + 8 * j < chi) {
            y[(rg + 4 * i) * ld + cg + 8 * j] = pr[i][j];
            y[yplane + (rg + 4 * i) * ld + cg + 8 * j] = pi[i][j];
          }
      __syncwarp();
      // rows f', columns g', contracting g down the slab's rows
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) pr[i][j] = pi[i][j] = 0.f;
      for (int k = 0; k < chi; ++k) {
        float ar[4], ai[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          ar[i] = y[k * ld + row[i]];
          ai[i] = y[yplane + k * ld + row[i]];
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float br = sMg[k * chi + col[j]], bi = sMg[c2 + k * chi + col[j]];
#pragma unroll
          for (int i = 0; i < 4; ++i) cmac(pr[i][j], pi[i][j], ar[i], ai[i], br, bi);
        }
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (rg + 4 * i < chi && cg + 8 * j < chi) {
            y[(cg + 8 * j) * ld + rg + 4 * i] = pr[i][j];
            y[yplane + (cg + 8 * j) * ld + rg + 4 * i] = pi[i][j];
          }
    }
    __syncthreads();
    // close: slice t covers k = 16 t .. 16 t + 15 of (p, g', f')
    constexpr int kPer = 2 * kMaxChi * kMaxChi / kSlice / kWarps;  // slices per warp at most
    const int K = 2 * c2, ns = (K + kSlice - 1) / kSlice;
    float psr[kPer][2][2], psi[kPer][2][2];
    {
      int ro[2], co[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        ro[i] = min((lane & 3) + 4 * i, job.on - 1) * 2 * chi * ld;
        co[i] = min((lane >> 2) + 8 * i, chi - 1) * so;
      }
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int t = warp + u * kWarps;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) psr[u][i][j] = psi[u][i][j] = 0.f;
        if (t >= ns) continue;
        const int k0 = t * kSlice;
        int p = k0 / c2, g = (k0 - p * c2) / chi, f = k0 - p * c2 - g * chi;
        const int kend = min(K, k0 + kSlice);
        for (int k = k0; k < kend; ++k) {
          const float* yb = sY + (p * chi + g) * ld + f;
          const float* tb = sT + p * sp + g * sg + f * sf;
          float yr[2], yi[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            yr[i] = yb[ro[i]];
            yi[i] = yb[yplane + ro[i]];
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float tr = tb[co[j]], ti = tb[tplane + co[j]];
#pragma unroll
            for (int i = 0; i < 2; ++i) cmac(psr[u][i][j], psi[u][i][j], yr[i], yi[i], tr, -ti);
          }
          if (++f == chi) {
            f = 0;
            if (++g == chi) { g = 0; ++p; }
          }
        }
      }
    }
    __syncthreads();  // Y2 is done with: its space takes the slice sums [slice][plane][o][o']
    const int nout = job.on * chi;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int t = warp + u * kWarps;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int o = (lane & 3) + 4 * i, c = (lane >> 2) + 8 * j;
          if (t < ns && o < job.on && c < chi) {
            sY[(t * 2) * nout + o * chi + c] = psr[u][i][j];
            sY[(t * 2 + 1) * nout + o * chi + c] = psi[u][i][j];
          }
        }
    }
    __syncthreads();
    const int splits = job.open == 0 ? splits3.x : job.open == 1 ? splits3.y : splits3.z;
    // slices per split-K part, as the GEMM cuts K
    const int per = splits > 1 ? ((K + splits - 1) / splits + kSlice - 1) / kSlice : ns;
    if (tid < 2 * nout) {
      const int pl = tid >= nout, o = tid - pl * nout;
      double sum = 0.0;
      float val = 0.f;
      for (int q = 0; q < splits; ++q) {
        float s = 0.f, c = 0.f;
        for (int t = q * per; t < min(ns, (q + 1) * per); ++t)
          two_sum_acc(s, c, sY[(t * 2 + pl) * nout + o]);
        val = __fadd_rn(s, c);
        sum += (double)val;
      }
      job.out[pl * c2 + job.o0 * chi + o] = splits > 1 ? (float)sum : val;
    }
    return;
  }
  // degree 2: Y[p, o][f'] = sum_f T[p, o, f] Mf[f][f'], closed over k = (p, f');
  // degree 1: Y = T, closed over p
  const int trows = job.deg == 2 ? 2 * chi : 2, tplane = 2 * chi * ld;
  float* sT = sm;
  float* sMf = sT + 2 * tplane;
  float* sY = sMf + 2 * c2;
  load_rows(sT, ld, tplane, job.T, (int64_t)trows * chi, trows, chi);
  if (job.deg == 2)
    for (int i = tid; i < 2 * c2; i += kThreads) sMf[i] = job.mf[i];
  __syncthreads();
  const int so = job.deg == 1 || job.open == 1 ? 1 : ld;
  const int sf = job.deg == 1 ? 0 : job.open == 1 ? ld : 1;
  const int sp = job.deg == 1 ? ld : chi * ld;
  const int nf = job.deg == 2 ? chi : 1;  // values of f
  if (job.deg == 2) {
    for (int i = tid; i < 2 * c2; i += kThreads) {
      const int p = i / c2, o = (i - p * c2) / chi, n = i - p * c2 - o * chi;
      const float* a0 = sT + p * sp + o * so;
      float pr = 0.f, pi = 0.f;
      for (int k = 0; k < chi; ++k)
        cmac(pr, pi, a0[k * sf], a0[tplane + k * sf], sMf[k * chi + n], sMf[c2 + k * chi + n]);
      sY[(p * chi + o) * ld + n] = pr;
      sY[tplane + (p * chi + o) * ld + n] = pi;
    }
    __syncthreads();
  }
  const float* Y = job.deg == 2 ? sY : sT;
  const int yo = job.deg == 2 ? ld : so, yf = job.deg == 2 ? 1 : 0;
  for (int i = tid; i < c2; i += kThreads) {
    const int o = i / chi, n = i - o * chi;
    float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f, pr = 0.f, pi = 0.f;
    int left = kSlice;
    for (int p = 0; p < 2; ++p)
      for (int f = 0; f < nf; ++f) {
        const float* y = Y + p * sp + o * yo + f * yf;
        const float* t = sT + p * sp + n * so + f * sf;
        cmac(pr, pi, y[0], y[tplane], t[0], -t[tplane]);
        if (--left == 0) {
          two_sum_acc(sr, cr, pr);
          two_sum_acc(si, ci, pi);
          pr = pi = 0.f;
          left = kSlice;
        }
      }
    if (left < kSlice) {
      two_sum_acc(sr, cr, pr);
      two_sum_acc(si, ci, pi);
    }
    job.out[i] = __fadd_rn(sr, cr);
    job.out[c2 + i] = __fadd_rn(si, ci);
  }
}

size_t smem_floats(int chi) {
  const size_t ld = chi | 1;
  return 2 * 2 * (size_t)chi * chi * ld + 4 * (size_t)chi * chi + 2 * 2 * (size_t)kOpen * chi * ld;
}

}  // namespace

bool site_sweep_supported(int chi) { return chi >= 1 && chi <= kMaxChi; }
int site_sweep_open(int chi) { return std::min(chi, kOpen); }

cudaError_t site_sweep_prepare() {
  static std::once_flag once;
  static cudaError_t result = cudaSuccess;
  std::call_once(once, [] {
    result = cudaFuncSetAttribute(site_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(sizeof(float) * smem_floats(kMaxChi)));
  });
  return result;
}

cudaError_t launch_site_sweep(const SiteJob* jobs, int n_jobs, int chi, const int splits[3],
                              const double* comp_state, cudaStream_t s) {
  if (n_jobs <= 0) return cudaSuccess;
  if (!site_sweep_supported(chi)) return cudaErrorInvalidValue;
  site_sweep_kernel<<<n_jobs, kThreads, sizeof(float) * smem_floats(chi), s>>>(
      jobs, chi, make_int3(splits[0], splits[1], splits[2]), comp_state);
  return cudaGetLastError();
}

}  // namespace tnbp
