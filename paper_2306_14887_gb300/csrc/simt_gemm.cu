// Plain FP32 batched complex GEMM on the CUDA cores (GemmDesc, planar data).
//
// Summation: every 16-deep slice of K is summed into fresh registers and the
// slice sums are added to the running total with an error-free two-sum whose
// rounding errors are carried in a compensation term (Knuth's TwoSum).  The
// contractions run over K up to 2 chi^2 (8192 at chi = 64); a single running
// FP32 sum would carry an error growing with K, while this keeps it at the
// 32-term slice plus a few roundings of the total.
//
// Bound by the FP32 pipe (4 FMAs per complex multiply-add, 128 lanes a clock):
// a thread holds 4 x 4 complex outputs, so one slice step costs four
// 16-byte shared reads per 64 FMAs, issued as packed pairs (the pair rate per
// lane is the scalar one, but it leaves issue slots for the reads and copies:
// 2.61 against 2.81 ms a sweep).  The two-sums take another 18 % of the pipe.
// Slices reach shared memory through a 3-stage ring of asynchronous copies laid
// out [k][row]: 16-byte copies where four rows are one block of memory, else
// 4-byte ones, which serve every stride and alignment a descriptor may have (odd
// chi, K-contiguous operands) without staging registers; the copies of slice
// s + 2 are in flight while slice s is multiplied.  The copies are the second
// cost: an operand held twice in shared memory (to spare the register copies of
// packed pairs) lost 15 %, 16-byte copies gained 10 %.
// Measured on the 127-qubit sweep at chi = 64: 2.10 ms a sweep (78.8 GFLOP, 37
// of the pipe's 77 TFLOP/s; a probe with this inner loop alone reaches 56).  With
// scalar global loads into a single shared buffer and 16 scalar shared reads per
// step it took 8.08 ms.  A persistent form, its copies running ahead across
// tiles, spilled registers and took 2.95 against 2.61 ms.
#include <algorithm>

#include "common.cuh"
#include "tnbp.h"

namespace tnbp {
namespace {

constexpr int BK = 16;       // slice depth: fixes the rounding of every sum
constexpr int kStages = 3;
constexpr int kPlanTile = 64;  // output tile the split-K heuristic counts with

// s + c += b with s the rounded sum and c the accumulated rounding errors.
__device__ __forceinline__ void two_sum_acc(float& s, float& c, float b) {
  const float t = __fadd_rn(s, b);
  const float bb = __fsub_rn(t, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(b, bb));
  s = t;
  c = __fadd_rn(c, e);
}

// 4-byte asynchronous copy global -> shared, zero fill when !ok.
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src),
               "r"(ok ? 4 : 0)
               : "memory");
}

// 16-byte asynchronous copy global -> shared, zero fill when !ok.
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}

// Quotients by n as products: x / n = x inv >> 40 with inv = ceil(2^40 / n), exact
// for x n < 2^40 (here x <= 2^17, n <= 2^16).
inline uint64_t inverse40(int n) { return n > 0 ? ((1ull << 40) + n - 1) / n : 0; }
__device__ __forceinline__ int quotient(int x, uint64_t inv) {
  return (int)(((uint64_t)(uint32_t)x * inv) >> 40);
}

// How an operand's contraction index runs: k = (k1, k2), with K0 > 0
// k1 = (i, j), j < K0, at i s0 + j s1.
struct KIndex {
  int K1, K2, K0, s0, s1, s2;
  uint64_t inv2, inv0;  // inverse40 of K2 and K0
  __device__ __forceinline__ int off(int k) const {
    if (K1 == 1) return k * s2;
    const int k1 = quotient(k, inv2);
    const int k2 = k - k1 * K2;
    if (K0 == 0) return k1 * s1 + k2 * s2;
    const int i = quotient(k1, inv0);
    return i * s0 + (k1 - i * K0) * s1 + k2 * s2;
  }
};

// BM x BN outputs, TM x TM of them per thread.
template <int BM, int BN, int TM>
struct Tile {
  static constexpr int kThreads = BM * BN / (TM * TM);
  static constexpr int kLda = BM + 4, kLdb = BN + 4;  // rows stay 16-byte aligned
  static constexpr int kStageFloats = 2 * BK * (kLda + kLdb);
  static constexpr int kBytes = kStages * kStageFloats * 4;
};

// TM floats as one shared-memory or global access.
template <int TM> struct Vec;
template <> struct Vec<4> { using type = float4; };
template <> struct Vec<2> { using type = float2; };

// How a slice of an operand is copied: by single values along K or along the
// rows, whichever is contiguous, or by 16-byte pieces of four rows.
enum CopyMode { kAlongK = 0, kAlongRows = 1, kFourRows = 2 };

// What one thread copies of one operand per slice.  kAlongK: the K offset
// tid % 16 of every THREADS / 16-th row; kAlongRows: row tid % ROWS at every
// THREADS / ROWS-th K offset; kFourRows: rows 4 (tid % (ROWS / 4)) .. + 3 at
// every 4 THREADS / ROWS-th K offset.
template <int ROWS, int LD, int THREADS>
struct Loader {
  static constexpr int kCount = ROWS * BK / THREADS;
  static_assert(kCount * THREADS == ROWS * BK && THREADS % ROWS == 0, "whole copies per thread");
  static constexpr int kStep4 = THREADS / (ROWS / 4);  // K offsets one pass of 16-byte copies has
  const float* base;
  int off[kCount];   // row offsets (kAlongK) or off[0]
  unsigned ok;       // valid rows, one bit per copy
  int mode, plane;
  KIndex ki;

  template <class RowOff>
  __device__ void init(const float* p, int mode_, int row0, int rows, const KIndex& ki_,
                       int64_t plane_, RowOff row_off) {
    base = p;
    mode = mode_;
    ki = ki_;
    plane = (int)plane_;
    ok = 0;
    const int tid = threadIdx.x;
    if (mode == kAlongK) {
#pragma unroll
      for (int i = 0; i < kCount; ++i) {
        const int r = row0 + (tid >> 4) + i * (THREADS / BK);
        off[i] = r < rows ? (int)row_off(r) : 0;
        ok |= (r < rows ? 1u : 0u) << i;
      }
    } else {
      const int r = row0 + (mode == kFourRows ? 4 * (tid % (ROWS / 4)) : tid % ROWS);
      off[0] = r < rows ? (int)row_off(r) : 0;
      ok = r < rows ? 1u : 0u;
    }
  }
  __device__ __forceinline__ void load(uint32_t dst, int k0, int kend) const {
    const int tid = threadIdx.x;
    if (mode == kFourRows) {
      const int r = 4 * (tid % (ROWS / 4));
#pragma unroll
      for (int i = 0; i < (BK + kStep4 - 1) / kStep4; ++i) {
        const int kk = tid / (ROWS / 4) + i * kStep4, k = k0 + kk;
        if (kStep4 > BK && kk >= BK) break;
        const bool v = k < kend && ok;
        const float* q = base + off[0] + (v ? ki.off(k) : 0);
        const uint32_t d0 = dst + 4 * (kk * LD + r);
        cp_async16(d0, q, v);
        cp_async16(d0 + 4 * BK * LD, q + plane, v);
      }
    } else if (mode == kAlongK) {
      const int kk = tid & (BK - 1), k = k0 + kk;
      const bool kok = k < kend;
      const int ko = kok ? ki.off(k) : 0;
      const uint32_t d0 = dst + 4 * (kk * LD + (tid >> 4));
#pragma unroll
      for (int i = 0; i < kCount; ++i) {
        const float* q = base + off[i] + ko;
        const bool v = kok && ((ok >> i) & 1);
        cp_async4(d0 + 4 * i * (THREADS / BK), q, v);
        cp_async4(d0 + 4 * (i * (THREADS / BK) + BK * LD), q + plane, v);
      }
    } else {
      const int r = tid % ROWS;
#pragma unroll
      for (int i = 0; i < kCount; ++i) {
        const int kk = tid / ROWS + i * (THREADS / ROWS), k = k0 + kk;
        const bool v = k < kend && ok;
        const float* q = base + off[0] + (v ? ki.off(k) : 0);
        const uint32_t d0 = dst + 4 * (kk * LD + r);
        cp_async4(d0, q, v);
        cp_async4(d0 + 4 * BK * LD, q + plane, v);
      }
    }
  }
};

// The copies of a slice follow the operand's contiguous index; rows in pieces of
// four when every piece is a whole 16-byte block of memory.
__device__ __forceinline__ int copy_mode_a(const GemmDesc& d, const float* A) {
  const bool three = d.M3 > 1, two = !three && d.M2 > 1;
  const int64_t row = three ? d.a_m3 : two ? d.a_m2 : d.a_m;  // stride of the innermost level
  if (row != 1 || (d.a_k2 == 1 && !three && !two)) return d.a_k2 == 1 ? kAlongK : kAlongRows;
  const int level = three ? d.M3 : two ? d.M2 : d.M;
  const int64_t strides = (three || two ? d.a_m : 0) | (three ? d.a_m2 : 0) | d.a_k1 | d.a_k2 |
                          d.plane_a;
  const bool whole = level % 4 == 0 && strides % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  return whole ? kFourRows : kAlongRows;
}
__device__ __forceinline__ int copy_mode_b(const GemmDesc& d, const float* B) {
  if (d.b_n != 1) return kAlongK;
  const int64_t strides = d.b_k0 | d.b_k1 | d.b_k2 | d.plane_b;
  const bool whole = d.N % 4 == 0 && strides % 4 == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  return whole ? kFourRows : kAlongRows;
}

template <int BM, int BN, int TM, bool CONJ_B>
__global__ void __launch_bounds__(Tile<BM, BN, TM>::kThreads, 512 / Tile<BM, BN, TM>::kThreads)
    cgemm_simt_kernel(GemmDesc d, float* part, int splits, int k_per_split, uint64_t inv2,
                      uint64_t inv0) {
  using T = Tile<BM, BN, TM>;
  using V = typename Vec<TM>::type;
  constexpr int NT = T::kThreads, LDA = T::kLda, LDB = T::kLdb;
  extern __shared__ __align__(16) float sm[];
  int z = blockIdx.z;
  const int split = z % splits;
  z /= splits;
  const int outer = z / d.n_inner;
  const int inner = z - outer * d.n_inner;
  if (outer_frozen(d, outer)) return;  // a converged component of a union
  const float* A = d.A[outer] + inner * d.a_in;
  const float* B = d.B[outer] + inner * d.b_in;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int tid = threadIdx.x;
  const int tx = tid % (BN / TM), ty = tid / (BN / TM);
  // this CTA's K range (all of K without split-K)
  const int kb = split * k_per_split;
  const int K = min(d.K1 * d.K2, kb + k_per_split);
  const int ns = K > kb ? (K - kb + BK - 1) / BK : 0;

  Loader<BM, LDA, NT> la;
  Loader<BN, LDB, NT> lb;
  la.init(A, copy_mode_a(d, A), m0, d.M,
          KIndex{d.K1, d.K2, 0, 0, (int)d.a_k1, (int)d.a_k2, inv2, 0}, d.plane_a,
          [&](int m) { return ROW_A(d, m); });
  lb.init(B, copy_mode_b(d, B), n0, d.N,
          KIndex{d.K1, d.K2, d.K0, (int)d.b_k0, (int)d.b_k1, (int)d.b_k2, inv2, inv0}, d.plane_b,
          [&](int n) { return (int64_t)n * d.b_n; });
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(sm);
  auto issue = [&](int s) {
    if (s < ns) {
      const uint32_t st = s0 + 4 * (s % kStages) * T::kStageFloats;
      la.load(st, kb + s * BK, K);
      lb.load(st + 4 * 2 * BK * LDA, kb + s * BK, K);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  issue(0);
  issue(1);

  float accr[TM][TM], acci[TM][TM], cmpr[TM][TM], cmpi[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) accr[i][j] = acci[i][j] = cmpr[i][j] = cmpi[i][j] = 0.f;

  for (int s = 0; s < ns; ++s) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();  // slice s has landed; everybody is done with slice s - 1
    issue(s + 2);
    const float* As = sm + (s % kStages) * T::kStageFloats + ty * TM;
    const float* Bs = sm + (s % kStages) * T::kStageFloats + 2 * BK * LDA + tx * TM;
    // two outputs of a row per packed FMA (half the issue slots of scalar FMAs)
    float2 pr[TM][TM / 2], pi[TM][TM / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM / 2; ++j) pr[i][j] = pi[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int kk = 0; kk < BK; ++kk) {
      float ar[TM], ai[TM], br[TM], bi[TM];
      *reinterpret_cast<V*>(ar) = *reinterpret_cast<const V*>(As + kk * LDA);
      *reinterpret_cast<V*>(ai) = *reinterpret_cast<const V*>(As + (BK + kk) * LDA);
      *reinterpret_cast<V*>(br) = *reinterpret_cast<const V*>(Bs + kk * LDB);
      *reinterpret_cast<V*>(bi) = *reinterpret_cast<const V*>(Bs + (BK + kk) * LDB);
      // C_re += a_re b_re - a_im b_im, C_im += a_re b_im + a_im b_re (b_im negated under CONJ_B)
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float2 a2 = make_float2(ar[i], ar[i]);
#pragma unroll
        for (int j = 0; j < TM / 2; ++j) {
          const float2 bp = make_float2(bi[2 * j], bi[2 * j + 1]);
          const float2 bm = make_float2(-bi[2 * j], -bi[2 * j + 1]);
          pr[i][j] = __ffma2_rn(a2, make_float2(br[2 * j], br[2 * j + 1]), pr[i][j]);
          pi[i][j] = __ffma2_rn(a2, CONJ_B ? bm : bp, pi[i][j]);
        }
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float2 a2 = make_float2(ai[i], ai[i]);
#pragma unroll
        for (int j = 0; j < TM / 2; ++j) {
          const float2 bp = make_float2(bi[2 * j], bi[2 * j + 1]);
          const float2 bm = make_float2(-bi[2 * j], -bi[2 * j + 1]);
          pr[i][j] = __ffma2_rn(a2, CONJ_B ? bp : bm, pr[i][j]);
          pi[i][j] = __ffma2_rn(a2, make_float2(br[2 * j], br[2 * j + 1]), pi[i][j]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM / 2; ++j) {
        two_sum_acc(accr[i][2 * j], cmpr[i][2 * j], pr[i][j].x);
        two_sum_acc(accr[i][2 * j + 1], cmpr[i][2 * j + 1], pr[i][j].y);
        two_sum_acc(acci[i][2 * j], cmpi[i][2 * j], pi[i][j].x);
        two_sum_acc(acci[i][2 * j + 1], cmpi[i][2 * j + 1], pi[i][j].y);
      }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) {
      accr[i][j] = __fadd_rn(accr[i][j], cmpr[i][j]);
      acci[i][j] = __fadd_rn(acci[i][j], cmpi[i][j]);
    }

  // Output: row-major partials or C.
  float* C;
  int64_t cn, plane;
  const bool to_part = splits > 1;
  if (to_part) {
    // split-K partial [split][outer][inner][re|im][M][N], summed by the reduce
    C = part + ((((int64_t)split * d.n_outer + outer) * d.n_inner + inner) * 2) * (int64_t)d.M * d.N;
    cn = 1;
    plane = (int64_t)d.M * d.N;
  } else {
    C = d.C[outer] + inner * d.c_in;
    cn = d.c_n;
    plane = d.plane_c;
  }
  auto row_c = [&](int m) { return to_part ? (int64_t)m * d.N : (int64_t)ROW_C(d, m); };
  const bool base16 = (reinterpret_cast<uintptr_t>(C) & 15) == 0 && plane % 4 == 0;
  // size of the innermost row level and whether its rows are adjacent in C
  const int lev = d.M3 > 1 ? d.M3 : d.M2 > 1 ? d.M2 : d.M;
  const int64_t lev_stride = d.M3 > 1 ? d.c_m3 : d.M2 > 1 ? d.c_m2 : d.c_m;
  if (cn != 1 && !to_part && lev_stride == 1) {
    // rows contiguous: one plane at a time through shared memory, so that
    // consecutive lanes store consecutive rows.  Column n holds BM / 4 chunks
    // of four rows, chunk c at c ^ (n / 4) % 8: conflict-free both ways.
    const bool vec = base16 && lev % 4 == 0 && cn % 4 == 0 &&
                     (d.M2 <= 1 || d.c_m % 4 == 0) && (d.M3 <= 1 || d.c_m2 % 4 == 0);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int pl = 0; pl < 2; ++pl) {
      __syncthreads();
#pragma unroll
      for (int j = 0; j < TM; ++j) {
        float v[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) v[i] = pl ? acci[i][j] : accr[i][j];
        const int n = tx * TM + j, m = ty * TM;
        *reinterpret_cast<V*>(sm + n * BM + 4 * ((m >> 2) ^ ((n >> 2) & 7)) + (m & 3)) =
            *reinterpret_cast<const V*>(v);
      }
      __syncthreads();
      for (int idx = tid; idx < BN * BM / 4; idx += NT) {
        const int n = idx / (BM / 4), c = idx % (BM / 4), m = m0 + 4 * c;
        if (n0 + n >= d.N || m >= d.M) continue;
        const float4 v = *reinterpret_cast<const float4*>(sm + n * BM + 4 * (c ^ ((n >> 2) & 7)));
        float* q = C + (pl ? plane : 0) + (int64_t)(n0 + n) * cn;
        if (vec) {
          *reinterpret_cast<float4*>(q + ROW_C(d, m)) = v;
        } else {
          const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (m + i < d.M) q[ROW_C(d, m + i)] = e[i];
        }
      }
    }
    return;
  }
  const bool vec = cn == 1 && base16 && d.N % 4 == 0 &&
                   (to_part || (d.c_m % 4 == 0 && (d.M2 <= 1 || d.c_m2 % 4 == 0) &&
                                (d.M3 <= 1 || d.c_m3 % 4 == 0)));
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty * TM + i, n = n0 + tx * TM;
    if (m >= d.M || n >= d.N) continue;
    float* q = C + row_c(m) + (int64_t)n * cn;
    if (vec) {
      *reinterpret_cast<V*>(q) = *reinterpret_cast<const V*>(accr[i]);
      *reinterpret_cast<V*>(q + plane) = *reinterpret_cast<const V*>(acci[i]);
    } else {
#pragma unroll
      for (int j = 0; j < TM; ++j) {
        if (n + j >= d.N) continue;
        q[j * cn] = accr[i][j];
        q[j * cn + plane] = acci[i][j];
      }
    }
  }
}

template <int BM, int BN, int TM>
cudaError_t prepare_tile() {
  const cudaError_t e = cudaFuncSetAttribute(cgemm_simt_kernel<BM, BN, TM, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Tile<BM, BN, TM>::kBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(cgemm_simt_kernel<BM, BN, TM, true>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              Tile<BM, BN, TM>::kBytes);
}

template <int BM, int BN, int TM>
void launch_tile(const GemmDesc& d, float* part, int splits, int kps, cudaStream_t s) {
  using T = Tile<BM, BN, TM>;
  const dim3 grid((d.M + BM - 1) / BM, (d.N + BN - 1) / BN, d.n_outer * d.n_inner * splits);
  const uint64_t inv2 = inverse40(d.K2), inv0 = inverse40(d.K0);
  if (d.conj_b)
    cgemm_simt_kernel<BM, BN, TM, true><<<grid, T::kThreads, T::kBytes, s>>>(d, part, splits, kps, inv2,
                                                                            inv0);
  else
    cgemm_simt_kernel<BM, BN, TM, false><<<grid, T::kThreads, T::kBytes, s>>>(d, part, splits, kps, inv2,
                                                                            inv0);
}

}  // namespace

// Split-K for the CUDA-core GEMM: a launch whose grid of 64 x 64 tiles is under
// one wave (152 CTAs: a few sites with a long contraction, e.g. the closes) is
// split into at most 64 pieces of at least 256 K values, each summed with the
// compensated slices, the pieces then summed in FP64 in a fixed order by the
// reduce.
int cgemm_plan(const GemmDesc& d, size_t* part_floats, int force_splits) {
  const int64_t K = (int64_t)d.K1 * d.K2;
  const int64_t ctas = (int64_t)((d.N + kPlanTile - 1) / kPlanTile) *
                       ((d.M + kPlanTile - 1) / kPlanTile) * d.n_outer * d.n_inner;
  int s = 1;
  if (force_splits > 0)
    s = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)force_splits, 64, (K + BK - 1) / BK}));
  else if (ctas < 152)
    while (s < 64 && ctas * s * 2 <= 2 * 152 && K / (2 * s) >= 256) s *= 2;
  *part_floats = s > 1 ? (size_t)s * d.n_outer * d.n_inner * 2 * d.M * d.N : 0;
  return s;
}

// Kernel attributes, set on each device before any launch (and before any stream capture).
cudaError_t simt_prepare() {
  static DeviceOnce once;
  return once([] {
    cudaError_t e = prepare_tile<64, 64, 4>();
    if (e == cudaSuccess) e = prepare_tile<128, 32, 4>();
    if (e == cudaSuccess) e = prepare_tile<256, 16, 4>();
    if (e == cudaSuccess) e = prepare_tile<32, 32, 2>();
    return e;
  });
}

// Element offsets inside one operand are 32-bit (a site plane holds at most
// 2 chi^3 = 2^25 floats at the largest chi).  No caller conjugates A or
// accumulates into C.
cudaError_t launch_cgemm(const GemmDesc& d, cudaStream_t s, float* part, size_t part_cap,
                         int* n_kernels, int force_splits) {
  if (n_kernels) *n_kernels = 0;
  if (d.M <= 0 || d.N <= 0 || d.n_outer <= 0 || d.n_inner <= 0) return cudaSuccess;
  if (d.conj_a || d.accumulate) return cudaErrorInvalidValue;
  const cudaError_t pe = simt_prepare();
  if (pe != cudaSuccess) return pe;
  size_t pf = 0;
  int splits = part ? cgemm_plan(d, &pf, force_splits) : 1;
  if (splits > 1 && pf > part_cap) splits = 1;  // the caller's partial buffer is too small
  const int K = d.K1 * d.K2;
  const int kps = splits > 1 ? ((K + splits - 1) / splits + BK - 1) / BK * BK : K;
  // the tile's width follows N (a 64-wide tile would spend 3/4 of its FMAs on
  // padding at chi = 16); outputs of few rows, the closes, take a small square
  // tile with 2 x 2 outputs a thread, so that a CTA still has eight warps
  if (d.N > 32) launch_tile<64, 64, 4>(d, part, splits, kps, s);
  else if (d.M <= 64) launch_tile<32, 32, 2>(d, part, splits, kps, s);
  else if (d.N > 16) launch_tile<128, 32, 4>(d, part, splits, kps, s);
  else launch_tile<256, 16, 4>(d, part, splits, kps, s);
  if (n_kernels) *n_kernels = splits > 1 ? 2 : 1;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || splits == 1) return e;
  return launch_tc_reduce(d, part, splits, s);
}

}  // namespace tnbp
