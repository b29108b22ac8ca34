// One BP sweep's message contractions for small bond dimensions (chi <= 32) in
// one launch, FP32: every CTA carries one site's chain to one open leg (two mode
// products and the close) through shared memory.
//
// At these sizes the contractions of a sweep are a dozen dependent launches of a
// few microseconds of work each.  Up to chi = 16 the site tensor (64 KB) and the
// chain's intermediate fit an SM, so nothing but T is read and nothing but the
// message is written; larger chi below.  Bound by the latency of a CTA's phases and
// the shared-memory reads of the products.  Measured, a whole sweep with normalisation and stop rule: 127 qubits at chi =
// 16 46 us (147 us as separate GEMM launches), 338 sites at chi = 16 79 us (201),
// 65 sites at chi = 9 24 us (173 with the GEMM before its rewrite).
//
// Up to chi = 16 every sum is taken exactly as the CUDA-core GEMM takes it (16-deep
// slices of the contraction in the same order, slice sums added by compensated
// two-sums, split-K parts added in FP64), so the messages are the same bit for bit.
//
// Degree 3, open leg o, first contracted leg f, second g (the chains of the
// sweep plan): a warp owns a slab (p, o), a chi x chi matrix over (g, f):
//   Y1[g][f'] = sum_f T[p, o, g, f] Mf[f][f'],  Y2[g'][f'] = sum_g Y1[g][f'] Mg[g][g']
// in place in shared memory; then all warps close over k = (p, g', f'),
//   out[o][o'] = sum_k Y2[o; k] conj(T[o'; k]),
// each warp taking every eighth slice for all outputs.
//
// A gate layer's environments are the same chains with p left open: two parts, one
// per p, each closed over (g', f') into out[p][o][o'].  A step's three layers, as
// GEMM launches and as one launch each: 127 qubits at chi = 16 0.465 and 0.071 ms, 24
// 0.56 and 0.14, 32 0.62 and 0.24; 65 sites at chi = 9 0.407 and 0.044, 23 0.55 and
// 0.13, 31 0.69 and 0.25; 433 sites at chi = 32 1.30 and 0.92.  Up to chi = 16 their
// K = chi^2 is never split and the sums are the GEMM's.  The streamed kernels take
// the parts as a template argument: as a runtime value they cost the sweep 6 percent.
#include <algorithm>

#include "common.cuh"
#include "tnbp.h"

namespace tnbp {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxChi = 16;        // the site tensor fits twice into an SM
constexpr int kSms = 152;
constexpr int kNarrowMaxChi = 24;  // three column groups of eight to a slab
constexpr int kStreamMaxChi = 32;  // rows of a slab a warp holds
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
    site_sweep_kernel(const SiteJob* jobs, int chi, int parts, int3 splits3,
                      const double* comp_state) {
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
    const int K = 2 * c2 / parts, nsp = (K + kSlice - 1) / kSlice, ns = parts * nsp;
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
        const int q = t >= nsp, k0 = q * K + (t - q * nsp) * kSlice;
        int p = k0 / c2, g = (k0 - p * c2) / chi, f = k0 - p * c2 - g * chi;
        const int kend = min((q + 1) * K, k0 + kSlice);
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
    const int per = splits > 1 ? ((K + splits - 1) / splits + kSlice - 1) / kSlice : nsp;
    for (int i = tid; i < parts * 2 * nout; i += kThreads) {
      const int r = i / nout, pl = r & 1, o = i - r * nout, t0 = (r >> 1) * nsp;
      double sum = 0.0;
      float val = 0.f;
      for (int q = 0; q < splits; ++q) {
        float s = 0.f, c = 0.f;
        for (int t = q * per; t < min(nsp, (q + 1) * per); ++t)
          two_sum_acc(s, c, sY[((t0 + t) * 2 + pl) * nout + o]);
        val = __fadd_rn(s, c);
        sum += (double)val;
      }
      job.out[r * c2 + job.o0 * chi + o] = splits > 1 ? (float)sum : val;
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
  for (int i = tid; i < parts * c2; i += kThreads) {
    const int q = i / c2, o = (i - q * c2) / chi, n = i - q * c2 - o * chi;
    float sr = 0.f, cr = 0.f, si = 0.f, ci = 0.f, pr = 0.f, pi = 0.f;
    int left = kSlice;
    for (int p = q; p < (parts == 2 ? q + 1 : 2); ++p)
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
    job.out[2 * q * c2 + o * chi + n] = __fadd_rn(sr, cr);
    job.out[(2 * q + 1) * c2 + o * chi + n] = __fadd_rn(si, ci);
  }
}

size_t smem_floats(int chi) {
  const size_t ld = chi | 1;
  return 2 * 2 * (size_t)chi * chi * ld + 4 * (size_t)chi * chi + 2 * 2 * (size_t)kOpen * chi * ld;
}

// --- chi = 17 .. 24 ---------------------------------------------------------
// T and the messages no longer fit an SM beside a block of slabs: a CTA of 16 warps
// holds its slabs (one per warp, interleaved complex, 77 KB at chi = 24), and the
// close streams T through two stages of 256 contraction indices, one 16-deep slice
// per warp and stage.  Bound by the issue of the products' operand reads and of the
// transposing 4-byte copies.  A whole sweep with normalisation and stop rule, before
// (eight GEMM launches) and now: 65 sites at chi = 17 181 and 63 us, 22 224 and 74,
// 23 184 and 83; 127 qubits at chi = 23 255 and 134; 433 sites at chi = 24 490 and
// 391.  Two CTAs of eight warps per SM took 71, 96, 97, 133 and 454.
// Every product is summed as above.  The close is one chain of compensated sums:
// split-K parts, each rounded to FP32 and added in FP64, kept the FP64 units busy
// for as long as the products took.
constexpr int kStreamThreads = 512, kStreamWarps = kStreamThreads / 32;
constexpr int kStageK = kStreamWarps * kSlice;
constexpr int kStageLd = kStageK + 1;  // float2 per o' row of a stage

// kRI x kCJ values of a slab per lane (4 x 8 lanes), kOI x kPJ of a close (kOL lanes
// along the open leg, 8 along o').
constexpr int kRI = 6, kCJ = 3, kOL = 4, kOI = 2, kPJ = 3;

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() {
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// y <- (y M)^T of one slab (rows x contracted, interleaved complex, in place):
// two 16-deep slices at most, whose compensated sum is their rounded sum.
// M's entries are (re, im, -im, re).
__device__ __forceinline__ void slab_product(float2* y, const float4* M, int chi, int ld) {
  const int lane = threadIdx.x & 31, rg = lane >> 3, cg = lane & 7;
  int row[kRI], col[kCJ];
#pragma unroll
  for (int i = 0; i < kRI; ++i) row[i] = min(rg + 4 * i, chi - 1) * ld;
#pragma unroll
  for (int j = 0; j < kCJ; ++j) col[j] = min(cg + 8 * j, chi - 1);
  float2 acc[kRI][kCJ], head[kRI][kCJ];
#pragma unroll
  for (int i = 0; i < kRI; ++i)
#pragma unroll
    for (int j = 0; j < kCJ; ++j) acc[i][j] = make_float2(0.f, 0.f);
  for (int k0 = 0; k0 < chi; k0 += kSlice) {
    if (k0 == kSlice)
#pragma unroll
      for (int i = 0; i < kRI; ++i)
#pragma unroll
        for (int j = 0; j < kCJ; ++j) {
          head[i][j] = acc[i][j];
          acc[i][j] = make_float2(0.f, 0.f);
        }
    const int kend = min(chi, k0 + kSlice);
    for (int k = k0; k < kend; ++k) {
      float2 a[kRI];
#pragma unroll
      for (int i = 0; i < kRI; ++i) a[i] = y[row[i] + k];
#pragma unroll
      for (int j = 0; j < kCJ; ++j) {
        const float4 b = M[k * chi + col[j]];
#pragma unroll
        for (int i = 0; i < kRI; ++i)
          acc[i][j] = __ffma2_rn(make_float2(a[i].x, a[i].x), make_float2(b.x, b.y), acc[i][j]);
#pragma unroll
        for (int i = 0; i < kRI; ++i)
          acc[i][j] = __ffma2_rn(make_float2(a[i].y, a[i].y), make_float2(b.z, b.w), acc[i][j]);
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < kRI; ++i)
#pragma unroll
    for (int j = 0; j < kCJ; ++j) {
      const int r = rg + 4 * i, c = cg + 8 * j;
      if (r < chi && c < chi)
        y[c * ld + r] = make_float2(__fadd_rn(head[i][j].x, acc[i][j].x),
                                    __fadd_rn(head[i][j].y, acc[i][j].y));
    }
  __syncwarp();
}

// One site of degree 1 or 2 (T[p, o, f]), the chains of site_sweep_kernel with a
// 2 x 4 tile of the product and a 2 x 2 tile of the close per thread.
__device__ void stream_low_degree(const SiteJob& job, float* sm, int chi, int parts) {
  const int ld = chi | 1, c2 = chi * chi, tid = threadIdx.x;
  float2* sT = (float2*)sm;
  float2* sY = sT + 2 * chi * ld;
  float2* sM = sY + 2 * chi * ld;
  const int trows = job.deg == 2 ? 2 * chi : 2;
  for (int i = tid; i < trows * chi; i += kStreamThreads) {
    const int r = i / chi;
    sT[r * ld + i - r * chi] = make_float2(job.T[i], job.T[trows * chi + i]);
  }
  if (job.deg == 2)
    for (int i = tid; i < c2; i += kStreamThreads) sM[i] = make_float2(job.mf[i], job.mf[c2 + i]);
  __syncthreads();
  const int so = job.deg == 1 || job.open == 1 ? 1 : ld;
  const int sf = job.deg == 1 ? 0 : job.open == 1 ? ld : 1;
  const int sp = job.deg == 1 ? ld : chi * ld;
  const int nf = job.deg == 2 ? chi : 1;
  if (job.deg == 2) {
    const int tr = chi, tc = (chi + 3) / 4;  // rows (p, o) in pairs o, o + half; columns by fours
    for (int i = tid; i < tr * tc; i += kStreamThreads) {
      const int r = i / tc, n0 = 4 * (i - r * tc);
      // rows r and r + chi of the 2 chi rows (p, o): the two spins
      const float2* a0 = sT + r * so;
      float2 acc[2][4], head[2][4];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[u][j] = head[u][j] = make_float2(0.f, 0.f);
      for (int k = 0; k < chi; ++k) {
        if (k == kSlice)
#pragma unroll
          for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              head[u][j] = acc[u][j];
              acc[u][j] = make_float2(0.f, 0.f);
            }
        const float2 a[2] = {a0[k * sf], a0[sp + k * sf]};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 b = sM[k * chi + min(n0 + j, chi - 1)];
#pragma unroll
          for (int u = 0; u < 2; ++u)
            cmac(acc[u][j].x, acc[u][j].y, a[u].x, a[u].y, b.x, b.y);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (n0 + j < chi)
            sY[(u * chi + r) * ld + n0 + j] = make_float2(__fadd_rn(head[u][j].x, acc[u][j].x),
                                                          __fadd_rn(head[u][j].y, acc[u][j].y));
    }
    __syncthreads();
  }
  const float2* Y = job.deg == 2 ? sY : sT;
  const int yo = job.deg == 2 ? ld : so, yf = job.deg == 2 ? 1 : 0;
  const int half = (chi + 1) / 2;
  for (int i = tid; i < parts * half * half; i += kStreamThreads) {
    const int q = i >= half * half, i0 = i - q * half * half;
    const int o0 = i0 / half, n0 = i0 - o0 * half;
    const int o[2] = {o0, min(o0 + half, chi - 1)}, n[2] = {n0, min(n0 + half, chi - 1)};
    float2 acc[2][2], sum[2][2], err[2][2];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int w = 0; w < 2; ++w) acc[u][w] = sum[u][w] = err[u][w] = make_float2(0.f, 0.f);
    const int K = 2 * nf / parts;
    int p = q, f = 0;
    for (int k0 = 0; k0 < K; k0 += kSlice) {
      for (int k = k0; k < min(K, k0 + kSlice); ++k) {
        float2 y[2], t[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          y[u] = Y[p * sp + o[u] * yo + f * yf];
          t[u] = sT[p * sp + n[u] * so + f * sf];
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int w = 0; w < 2; ++w)
            cmac(acc[u][w].x, acc[u][w].y, y[u].x, y[u].y, t[w].x, -t[w].y);
        if (++f == nf) { f = 0; ++p; }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          two_sum_acc(sum[u][w].x, err[u][w].x, acc[u][w].x);
          two_sum_acc(sum[u][w].y, err[u][w].y, acc[u][w].y);
          acc[u][w] = make_float2(0.f, 0.f);
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int w = 0; w < 2; ++w) {  // a repeated edge value is written twice, the same
        job.out[2 * q * c2 + o[u] * chi + n[w]] = __fadd_rn(sum[u][w].x, err[u][w].x);
        job.out[(2 * q + 1) * c2 + o[u] * chi + n[w]] = __fadd_rn(sum[u][w].y, err[u][w].y);
      }
  }
}

template <int PARTS>
__global__ void __launch_bounds__(kStreamThreads, 1)
    site_stream_kernel(const SiteJob* jobs, int chi, int open_max, uint32_t inv_chi,
                       const double* comp_state) {
  extern __shared__ __align__(16) float sm[];
  const SiteJob job = jobs[blockIdx.x];
  if (comp_state && comp_state[4 * job.comp + 3] != 0.0) return;
  if (job.deg < 3) {
    stream_low_degree(job, sm, chi, PARTS);
    return;
  }
  const int ld = chi | 1, c2 = chi * chi, K = 2 * c2 / PARTS;
  const int nsp = (K + kSlice - 1) / kSlice, ns = PARTS * nsp;  // slices per part, of all
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // both stages first (16-byte aligned), the slice sums, the slabs
  const int stage_len = (chi * kStageLd + 1) / 2 * 2;
  float2* sStage = (float2*)sm;
  float* sums = (float*)(sStage + 2 * stage_len);
  float2* sY = (float2*)(sums + kStreamWarps * 2 * open_max * chi);
  float4* sMf = (float4*)(sStage + stage_len);  // the messages lie there until the second stage is needed
  float4* sMg = sMf + c2;
  // strides of the legs in T
  const int so = job.open == 0 ? c2 : job.open == 1 ? chi : 1;
  const int sf = job.open == 2 ? c2 : 1;
  const int sg = job.open == 1 ? c2 : chi;
  const int sp = c2 * chi;
  const float* T = job.T;
  const int plane = 2 * sp;
  // first k of slice t; the k of position kk of stage st, or -1
  auto second = [&](int t) { return PARTS == 2 && t >= nsp; };
  auto slice_k = [&](int t) { return second(t) ? K + (t - nsp) * kSlice : t * kSlice; };
  auto stage_k = [&](int st, int kk) {
    if (PARTS == 1) return st * kStageK + kk < K ? st * kStageK + kk : -1;
    const int t = st * kStreamWarps + kk / kSlice, k = slice_k(t) + kk % kSlice;
    return t < ns && k < (second(t) ? 2 * K : K) ? k : -1;
  };
  // stage st: k = kStageK st .. + kStageK - 1 of (p, g, f), as [o'][k]
  auto load_stage = [&](int st) {
    float2* dst = sStage + (st & 1) * stage_len;
    if (job.open < 2) {  // contiguous along f
      const int kk = tid & (kStageK - 1), k = stage_k(st, kk);
      if (k >= 0) {
        const int r = (int)((uint32_t)k * inv_chi >> 20), p = r >= chi;
        const float* src = T + p * sp + (r - p * chi) * sg + (k - r * chi) * sf;
        for (int o = tid / kStageK; o < chi; o += kStreamThreads / kStageK) {
          cp_async4(&dst[o * kStageLd + kk].x, src + o * so);
          cp_async4(&dst[o * kStageLd + kk].y, src + o * so + plane);
        }
      }
    } else if (lane < chi) {  // contiguous along o'
      for (int kk = warp; kk < kStageK; kk += kStreamWarps) {
        const int k = stage_k(st, kk);
        if (k < 0) continue;
        const int r = (int)((uint32_t)k * inv_chi >> 20), p = r >= chi;
        const float* src = T + p * sp + (r - p * chi) * sg + (k - r * chi) * sf + lane;
        cp_async4(&dst[lane * kStageLd + kk].x, src);
        cp_async4(&dst[lane * kStageLd + kk].y, src + plane);
      }
    }
    cp_commit();
  };
  // the slabs [2 o + p][g][f]
  if (job.open < 2) {
    if (lane < chi)
      for (int r = warp; r < 2 * job.on * chi; r += kStreamWarps) {
        const int s = (int)((uint32_t)r * inv_chi >> 20), g = r - s * chi;
        const float* src = T + (s & 1) * sp + (job.o0 + (s >> 1)) * so + g * sg + lane;
        cp_async4(&sY[r * ld + lane].x, src);
        cp_async4(&sY[r * ld + lane].y, src + plane);
      }
  } else if ((lane & 7) < job.on) {
    const int ol = lane & 7;
    for (int r = tid >> 3; r < 2 * c2; r += kStreamThreads / 8) {  // (p, f, g)
      const int q = (int)((uint32_t)r * inv_chi >> 20), p = q >= chi;
      float2* dst = sY + ((2 * ol + p) * chi + r - q * chi) * ld + q - p * chi;
      const float* src = T + r * chi + job.o0 + ol;
      cp_async4(&dst->x, src);
      cp_async4(&dst->y, src + plane);
    }
  }
  load_stage(0);
  for (int i = tid; i < c2; i += kStreamThreads) {
    float re = job.mf[i], im = job.mf[c2 + i];
    sMf[i] = make_float4(re, im, -im, re);
    re = job.mg[i];
    im = job.mg[c2 + i];
    sMg[i] = make_float4(re, im, -im, re);
  }
  cp_wait_all();
  __syncthreads();
  for (int s = warp; s < 2 * job.on; s += kStreamWarps) {
    slab_product(sY + s * chi * ld, sMf, chi, ld);  // [f'][g]
    slab_product(sY + s * chi * ld, sMg, chi, ld);  // [g'][f']
  }
  const int nst = (ns + kStreamWarps - 1) / kStreamWarps;
  const int nout = job.on * chi;
  const int ol = lane % kOL, cl = lane / kOL;
  int yo[kOI], to[kPJ];
#pragma unroll
  for (int i = 0; i < kOI; ++i) yo[i] = min(ol + kOL * i, job.on - 1) * 2 * chi * ld;
#pragma unroll
  for (int j = 0; j < kPJ; ++j) to[j] = min(cl + 32 / kOL * j, chi - 1) * kStageLd;
  // thread tid < 2 nout sums the slices of output part tid
  float total = 0.f, lost = 0.f;
  auto store = [&](int q) {
    const int pl = tid >= nout;
    job.out[(2 * q + pl) * c2 + job.o0 * chi + tid - pl * nout] = __fadd_rn(total, lost);
    total = lost = 0.f;
  };
  for (int st = 0; st < nst; ++st) {
    cp_wait_all();
    __syncthreads();  // stage st is there; the other stage and the sums are done with
    if (st + 1 < nst) load_stage(st + 1);
    const int t = st * kStreamWarps + warp;
    if (t < ns) {
      float2 acc[kOI][kPJ];
#pragma unroll
      for (int i = 0; i < kOI; ++i)
#pragma unroll
        for (int j = 0; j < kPJ; ++j) acc[i][j] = make_float2(0.f, 0.f);
      const int k0 = slice_k(t), kend = min(second(t) ? 2 * K : K, k0 + kSlice);
      int r = (int)((uint32_t)k0 * inv_chi >> 20), f = k0 - r * chi;
      const float2* yb = sY + r * ld + f;
      const float2* tb = sStage + (st & 1) * stage_len + warp * kSlice;
#pragma unroll 4
      for (int k = k0; k < kend; ++k) {
        float2 y[kOI];
#pragma unroll
        for (int i = 0; i < kOI; ++i) y[i] = yb[yo[i]];
#pragma unroll
        for (int j = 0; j < kPJ; ++j) {
          const float2 b = tb[to[j]];
#pragma unroll
          for (int i = 0; i < kOI; ++i) {
            acc[i][j] = __ffma2_rn(make_float2(y[i].x, y[i].x), make_float2(b.x, -b.y), acc[i][j]);
            acc[i][j] = __ffma2_rn(make_float2(y[i].y, y[i].y), make_float2(b.y, b.x), acc[i][j]);
          }
        }
        ++tb;
        ++yb;
        if (++f == chi) {
          f = 0;
          yb += ld - chi;
        }
      }
      float* d = sums + warp * 2 * nout;
#pragma unroll
      for (int i = 0; i < kOI; ++i)
#pragma unroll
        for (int j = 0; j < kPJ; ++j) {
          const int o = ol + kOL * i, c = cl + 32 / kOL * j;
          if (o < job.on && c < chi) {
            d[o * chi + c] = acc[i][j].x;
            d[nout + o * chi + c] = acc[i][j].y;
          }
        }
    }
    __syncthreads();
    if (tid < 2 * nout)
#pragma unroll
      for (int w = 0; w < kStreamWarps; ++w)
        if (st * kStreamWarps + w < ns) {
          if (PARTS == 2 && st * kStreamWarps + w == nsp) store(0);  // the second part begins
          two_sum_acc(total, lost, sums[w * 2 * nout + tid]);
        }
  }
  if (tid < 2 * nout) store(PARTS - 1);
}

size_t stream_bytes(int chi, int open) {
  const size_t ld = chi | 1;
  return 2 * sizeof(float2) * (((size_t)chi * kStageLd + 1) / 2 * 2) +
         sizeof(float) * kStreamWarps * 2 * open * chi + sizeof(float2) * 2 * open * chi * ld;
}
// --- chi = 25 .. 32 ---------------------------------------------------------
// As above with 144 KB of slabs: two warps share a slab and a slice, and with fewer
// registers to a warp the slabs lie planar, their contracted leg slow, so that every
// operand of the packed products (two rows; two values o') is one aligned read.
// Bound by the operand reads, the transposing copies and the last wave of one CTA
// per SM (31 percent of the FP32 rate at chi = 32).  A whole sweep, before (GEMM
// launches) and now: 65 sites at chi = 25 220 and 136 us, 31 257 and 185, 32 181 and
// 171; 127 qubits at chi = 26 280 and 201, 28 255 and 206, 32 267 and 246; 433 sites
// at chi = 31 1028 and 933, but 28 656 and 677, 32 795 and 860: with rows of whole
// 16-byte pieces and enough sites the GEMM launches stay (site_sweep_preferred).
constexpr int kWideSlices = kStreamWarps / 2, kWideK = kWideSlices * kSlice;
constexpr int kWideFloats = 2 * kWideK * 32;  // planes of [k][o'], o' rotated by 2 k
constexpr int kLd = 36;  // slab rows: conflict-free transposed copies and stores
__host__ __device__ inline int slab_plane(int chi) { return chi * kLd; }
// o -> o + 1: two spins of two planes; 4 mod 32 banks apart
__host__ __device__ inline int slab_open(int chi) { return 4 * slab_plane(chi) + 4; }

// Meets the other warp of the pair (both run the same slabs).
__device__ __forceinline__ void pair_sync(int pair) {
  asm volatile("bar.sync %0, 64;" ::"r"(pair + 1) : "memory");
}

// One slab's product in place.  y is planar [k][row] (k the contracted leg); the
// result goes to [row][col], or with FLIP to [col][row].  M's entries are (re, re,
// im, im).  Two warps share a slab, sixteen columns each; a lane holds the row pairs
// 2 rg + 8 h and the columns cg + 8 j.  The sum is taken in two 16-deep slices,
// whose compensated sum is their rounded sum.
template <bool FLIP>
__device__ __forceinline__ void pair_product(float* y, const float4* M, int chi) {
  constexpr int RP = 4, CJ = 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rg = lane >> 3, cg = (lane & 7) + 16 * (warp & 1), plane = slab_plane(chi);
  float2 pr[RP][CJ], pi[RP][CJ], hr[RP][CJ], hi[RP][CJ];
#pragma unroll
  for (int h = 0; h < RP; ++h)
#pragma unroll
    for (int j = 0; j < CJ; ++j) pr[h][j] = pi[h][j] = make_float2(0.f, 0.f);
  int col[CJ];
#pragma unroll
  for (int j = 0; j < CJ; ++j) col[j] = min(cg + 8 * j, chi - 1);
  const float* a = y + 2 * rg;
  for (int k0 = 0; k0 < chi; k0 += kSlice) {
    if (k0 == kSlice)
#pragma unroll
      for (int h = 0; h < RP; ++h)
#pragma unroll
        for (int j = 0; j < CJ; ++j) {
          hr[h][j] = pr[h][j];
          hi[h][j] = pi[h][j];
          pr[h][j] = pi[h][j] = make_float2(0.f, 0.f);
        }
    const int kend = min(chi, k0 + kSlice);
    for (int k = k0; k < kend; ++k) {
      float2 ar[RP], ai[RP];
#pragma unroll
      for (int h = 0; h < RP; ++h) {
        ar[h] = *(const float2*)(a + k * kLd + 8 * h);
        ai[h] = *(const float2*)(a + plane + k * kLd + 8 * h);
      }
#pragma unroll
      for (int j = 0; j < CJ; ++j) {
        const float4 b = M[k * chi + col[j]];
        const float2 br = make_float2(b.x, b.y), bi = make_float2(b.z, b.w);
        const float2 bm = make_float2(-b.z, -b.w);
#pragma unroll
        for (int h = 0; h < RP; ++h) {
          pr[h][j] = __ffma2_rn(ar[h], br, pr[h][j]);
          pi[h][j] = __ffma2_rn(ar[h], bi, pi[h][j]);
        }
#pragma unroll
        for (int h = 0; h < RP; ++h) {
          pr[h][j] = __ffma2_rn(ai[h], bm, pr[h][j]);
          pi[h][j] = __ffma2_rn(ai[h], br, pi[h][j]);
        }
      }
    }
  }
  pair_sync(warp >> 1);
#pragma unroll
  for (int h = 0; h < RP; ++h)
#pragma unroll
    for (int j = 0; j < CJ; ++j) {
      const int r = 2 * rg + 8 * h, c = cg + 8 * j;
      const float2 re = make_float2(__fadd_rn(hr[h][j].x, pr[h][j].x),
                                    __fadd_rn(hr[h][j].y, pr[h][j].y));
      const float2 im = make_float2(__fadd_rn(hi[h][j].x, pi[h][j].x),
                                    __fadd_rn(hi[h][j].y, pi[h][j].y));
      if (c < chi && r < chi) {
        if (FLIP) {  // a row beyond the last one falls into the padding
          *(float2*)(y + c * kLd + r) = re;
          *(float2*)(y + plane + c * kLd + r) = im;
        } else {
          y[r * kLd + c] = re.x;
          y[plane + r * kLd + c] = im.x;
          if (r + 1 < chi) {
            y[(r + 1) * kLd + c] = re.y;
            y[plane + (r + 1) * kLd + c] = im.y;
          }
        }
      }
    }
  pair_sync(warp >> 1);
}

// VEC: chi is a multiple of four, and the close reads four contraction indices of a
// slab at a time.
template <bool VEC, int PARTS>
__global__ void __launch_bounds__(kStreamThreads, 1)
    site_wide_kernel(const SiteJob* jobs, int chi, int open_max, uint32_t inv_chi,
                     const double* comp_state) {
  extern __shared__ __align__(16) float sm[];
  const SiteJob job = jobs[blockIdx.x];
  if (comp_state && comp_state[4 * job.comp + 3] != 0.0) return;
  if (job.deg < 3) {
    stream_low_degree(job, sm, chi, PARTS);
    return;
  }
  const int c2 = chi * chi, K = 2 * c2 / PARTS, splane = slab_plane(chi), sopen = slab_open(chi);
  const int nsp = (K + kSlice - 1) / kSlice, ns = PARTS * nsp;  // slices per part, of all
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* sStage = sm;                     // two stages
  float* sY = sStage + 2 * kWideFloats;   // the slabs [o][p][plane]
  float* sums = sY + open_max * sopen;    // a stage's slice sums [slice][plane][o][o']
  float4* sMf = (float4*)(sStage + kWideFloats);  // until the second stage is needed
  float4* sMg = sMf + c2;
  // strides of the legs in T
  const int so = job.open == 0 ? c2 : job.open == 1 ? chi : 1;
  const int sf = job.open == 2 ? c2 : 1;
  const int sg = job.open == 1 ? c2 : chi;
  const int sp = c2 * chi;
  const float* T = job.T;
  const int tplane = 2 * sp;
  // first k of slice t; the k of position kk of stage st, or -1
  auto second = [&](int t) { return PARTS == 2 && t >= nsp; };
  auto slice_k = [&](int t) { return second(t) ? K + (t - nsp) * kSlice : t * kSlice; };
  auto stage_k = [&](int st, int kk) {
    if (PARTS == 1) return st * kWideK + kk < K ? st * kWideK + kk : -1;
    const int t = st * kWideSlices + kk / kSlice, k = slice_k(t) + kk % kSlice;
    return t < ns && k < (second(t) ? 2 * K : K) ? k : -1;
  };
  // stage st: k = 128 st .. + 127 of (p, g, f)
  auto load_stage = [&](int st) {
    float* dst = sStage + (st & 1) * kWideFloats;
    if (job.open < 2) {  // contiguous along f
      const int kk = tid & (kWideK - 1), k = stage_k(st, kk);
      if (k >= 0) {
        const int r = (int)((uint32_t)k * inv_chi >> 20), p = r >= chi;
        const float* src = T + p * sp + (r - p * chi) * sg + (k - r * chi) * sf;
        for (int o = tid / kWideK; o < chi; o += kStreamThreads / kWideK) {
          float* d = dst + kk * 32 + ((o + 2 * kk) & 31);
          cp_async4(d, src + o * so);
          cp_async4(d + kWideK * 32, src + o * so + tplane);
        }
      }
    } else if (lane < chi) {  // contiguous along o'
      for (int kk = warp; kk < kWideK; kk += kStreamWarps) {
        const int k = stage_k(st, kk);
        if (k < 0) continue;
        const int r = (int)((uint32_t)k * inv_chi >> 20), p = r >= chi;
        const float* src = T + p * sp + (r - p * chi) * sg + (k - r * chi) * sf + lane;
        float* d = dst + kk * 32 + ((lane + 2 * kk) & 31);
        cp_async4(d, src);
        cp_async4(d + kWideK * 32, src + tplane);
      }
    }
    cp_commit();
  };
  // the slabs as [o][p][plane][f][g]
  if (job.open < 2) {  // eight f by four g per warp
    const int fb = (chi + 7) / 8, gb = (chi + 3) / 4, nb = fb * gb;
    for (int i = warp; i < 2 * job.on * nb; i += kStreamWarps) {
      const int s = i / nb, bl = i - s * nb, f = 8 * (bl % fb) + (lane & 7);
      const int g = 4 * (bl / fb) + (lane >> 3);
      if (f < chi && g < chi) {
        const float* src = T + (s & 1) * sp + (job.o0 + (s >> 1)) * so + g * sg + f;
        float* d = sY + (s >> 1) * sopen + (s & 1) * 2 * splane + f * kLd + g;
        cp_async4(d, src);
        cp_async4(d + splane, src + tplane);
      }
    }
  } else if ((lane & 7) < job.on) {  // eight o by four g
    const int ol = lane & 7;
    for (int r = tid >> 3; r < 2 * c2; r += kStreamThreads / 8) {  // (p, f, g)
      const int q = (int)((uint32_t)r * inv_chi >> 20), p = q >= chi;
      float* d = sY + ol * sopen + p * 2 * splane + (q - p * chi) * kLd + r - q * chi;
      const float* src = T + r * chi + job.o0 + ol;
      cp_async4(d, src);
      cp_async4(d + splane, src + tplane);
    }
  }
  load_stage(0);
  for (int i = tid; i < c2; i += kStreamThreads) {
    float re = job.mf[i], im = job.mf[c2 + i];
    sMf[i] = make_float4(re, re, im, im);
    re = job.mg[i];
    im = job.mg[c2 + i];
    sMg[i] = make_float4(re, re, im, im);
  }
  cp_wait_all();
  __syncthreads();
  for (int s = warp >> 1; s < 2 * job.on; s += kStreamWarps / 2) {
    float* y = sY + (s >> 1) * sopen + (s & 1) * 2 * splane;
    pair_product<false>(y, sMf, chi);  // [f][g] -> [g][f']
    pair_product<true>(y, sMg, chi);   // [g][f'] -> [g'][f']
  }
  const int nst = (ns + kWideSlices - 1) / kWideSlices;
  const int nout = job.on * chi;
  // two warps share a slice, four open values each: a lane closes o = ol, ol + 2 with
  // the pair o' = 2 cl, 2 cl + 1
  const int slice = warp >> 1, ol = (lane >> 4) + 4 * (warp & 1), cl = lane & 15;
  int yo[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) yo[i] = min(ol + 2 * i, job.on - 1) * sopen;
  // thread tid < 2 nout sums the slices of output part tid
  float total = 0.f, lost = 0.f;
  auto store = [&](int q) {
    const int pl = tid >= nout;
    job.out[(2 * q + pl) * c2 + job.o0 * chi + tid - pl * nout] = __fadd_rn(total, lost);
    total = lost = 0.f;
  };
  for (int st = 0; st < nst; ++st) {
    cp_wait_all();
    __syncthreads();  // stage st is there; the other stage and the sums are done with
    if (st + 1 < nst) load_stage(st + 1);
    const int t = st * kWideSlices + slice;
    if (t < ns) {
      float2 pr[2], pi[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) pr[i] = pi[i] = make_float2(0.f, 0.f);
      const int k0 = slice_k(t), n = min((second(t) ? 2 * K : K) - k0, kSlice);
      int r = (int)((uint32_t)k0 * inv_chi >> 20), f = k0 - r * chi;
      // row r = (p, g') of a slab: spin 1 starts two planes after spin 0
      const float* yb = sY + (r + (r >= chi ? chi : 0)) * kLd + f;
      const float* tb = sStage + (st & 1) * kWideFloats + slice * kSlice * 32;
      auto step = [&](int kk, const float (&yr)[2], const float (&yi)[2]) {
        const float* q = tb + kk * 32 + ((2 * cl + 2 * kk) & 31);  // 32 | 2 kSlice
        const float2 tr = *(const float2*)q, ti = *(const float2*)(q + kWideK * 32);
        const float2 tm = make_float2(-ti.x, -ti.y);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float2 y2 = make_float2(yr[i], yr[i]);
          pr[i] = __ffma2_rn(y2, tr, pr[i]);
          pi[i] = __ffma2_rn(y2, tm, pi[i]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float2 y2 = make_float2(yi[i], yi[i]);
          pr[i] = __ffma2_rn(y2, ti, pr[i]);
          pi[i] = __ffma2_rn(y2, tr, pi[i]);
        }
      };
      auto advance = [&](int by) {
        yb += by;
        f += by;
        if (f == chi) {
          f = 0;
          yb += kLd - chi;
          if (++r == chi) yb += splane;
        }
      };
      if (VEC) {  // K is a multiple of 16, f of 4
#pragma unroll
        for (int kk = 0; kk < kSlice; kk += 4) {
          float4 vr[2], vi[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            vr[i] = *(const float4*)(yb + yo[i]);
            vi[i] = *(const float4*)(yb + splane + yo[i]);
          }
          step(kk, {vr[0].x, vr[1].x}, {vi[0].x, vi[1].x});
          step(kk + 1, {vr[0].y, vr[1].y}, {vi[0].y, vi[1].y});
          step(kk + 2, {vr[0].z, vr[1].z}, {vi[0].z, vi[1].z});
          step(kk + 3, {vr[0].w, vr[1].w}, {vi[0].w, vi[1].w});
          advance(4);
        }
      } else {
#pragma unroll 2
        for (int kk = 0; kk < n; ++kk) {
          step(kk, {yb[yo[0]], yb[yo[1]]}, {yb[splane + yo[0]], yb[splane + yo[1]]});
          advance(1);
        }
      }
      float* d = sums + slice * 2 * nout;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int o = ol + 2 * i, c = 2 * cl;
        if (o < job.on && c < chi) {
          d[o * chi + c] = pr[i].x;
          d[nout + o * chi + c] = pi[i].x;
          if (c + 1 < chi) {
            d[o * chi + c + 1] = pr[i].y;
            d[nout + o * chi + c + 1] = pi[i].y;
          }
        }
      }
    }
    __syncthreads();
    if (tid < 2 * nout)
#pragma unroll
      for (int w = 0; w < kWideSlices; ++w)
        if (st * kWideSlices + w < ns) {
          if (PARTS == 2 && st * kWideSlices + w == nsp) store(0);  // the second part begins
          two_sum_acc(total, lost, sums[w * 2 * nout + tid]);
        }
  }
  if (tid < 2 * nout) store(PARTS - 1);
}

size_t wide_bytes(int chi, int open) {
  return sizeof(float) *
         (2 * kWideFloats + (size_t)open * slab_open(chi) + kWideSlices * 2 * open * chi);
}

// Open-leg values per degree-3 CTA, in even blocks of at most kOpen.
int stream_open(int chi) {
  const int blocks = (chi + kOpen - 1) / kOpen;
  return (chi + blocks - 1) / blocks;
}

}  // namespace

bool site_sweep_supported(int chi) { return chi >= 1 && chi <= kStreamMaxChi; }
bool site_sweep_preferred(int chi, int n_deg3_jobs) {
  return chi <= kNarrowMaxChi || chi % 4 != 0 || n_deg3_jobs <= 4 * kSms;
}
int site_sweep_open(int chi) { return chi <= kMaxChi ? std::min(chi, kOpen) : stream_open(chi); }

cudaError_t site_sweep_prepare() {
  static DeviceOnce once;
  return once([] {
    cudaError_t result = cudaSuccess;
    auto raise = [&](auto kernel, size_t bytes) {
      if (result == cudaSuccess)
        result = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)bytes);
    };
    const size_t narrow = stream_bytes(kNarrowMaxChi, stream_open(kNarrowMaxChi));
    raise(site_sweep_kernel, sizeof(float) * smem_floats(kMaxChi));
    raise(site_stream_kernel<1>, narrow);
    raise(site_stream_kernel<2>, narrow);
    raise(site_wide_kernel<true, 1>, wide_bytes(32, kOpen));
    raise(site_wide_kernel<true, 2>, wide_bytes(32, kOpen));
    raise(site_wide_kernel<false, 1>, wide_bytes(31, kOpen));
    raise(site_wide_kernel<false, 2>, wide_bytes(31, kOpen));
    return result;
  });
}

namespace {
cudaError_t launch_parts(const SiteJob* jobs, int n_jobs, int chi, int parts, int3 splits,
                         const double* comp_state, cudaStream_t s) {
  if (n_jobs <= 0) return cudaSuccess;
  if (!site_sweep_supported(chi)) return cudaErrorInvalidValue;
  if (chi <= kMaxChi) {
    site_sweep_kernel<<<n_jobs, kThreads, sizeof(float) * smem_floats(chi), s>>>(
        jobs, chi, parts, splits, comp_state);
    return cudaGetLastError();
  }
  const uint32_t inv = ((1u << 20) + chi - 1) / chi;  // x / chi = x inv >> 20 for x <= 2 chi^2
  const int open = stream_open(chi);
  if (chi <= kNarrowMaxChi)
    (parts == 2 ? site_stream_kernel<2> : site_stream_kernel<1>)<<<
        n_jobs, kStreamThreads, stream_bytes(chi, open), s>>>(jobs, chi, open, inv, comp_state);
  else {
    auto kernel = chi % 4 ? (parts == 2 ? site_wide_kernel<false, 2> : site_wide_kernel<false, 1>)
                          : (parts == 2 ? site_wide_kernel<true, 2> : site_wide_kernel<true, 1>);
    kernel<<<n_jobs, kStreamThreads, wide_bytes(chi, open), s>>>(jobs, chi, open, inv, comp_state);
  }
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_site_sweep(const SiteJob* jobs, int n_jobs, int chi, const int splits[3],
                              const double* comp_state, cudaStream_t s) {
  return launch_parts(jobs, n_jobs, chi, 1, make_int3(splits[0], splits[1], splits[2]), comp_state,
                      s);
}

cudaError_t launch_site_env(const SiteJob* jobs, int n_jobs, int chi, cudaStream_t s) {
  return launch_parts(jobs, n_jobs, chi, 2, make_int3(1, 1, 1), nullptr, s);
}

}  // namespace tnbp
