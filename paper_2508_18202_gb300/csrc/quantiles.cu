// quantiles.cu -- confidence bounds from the gPC surrogate (Sec. 2.4 step 7:
// confidence intervals from the expansion coefficients; Sec. 4 profile
// bands).  For each requested cell the surrogate y_m = sum_a c_a(x) Phi_a(s_m)
// is defined at the M input samples and its k-th smallest values are written.
//
// An order statistic needs few of the M values exactly.  A block evaluates
// the surrogate of several cells in FP32 (each basis value loaded once for all
// of them), with a bound E on the difference to the FP64 value.  The k-th
// smallest of the FP32 values lies in one bucket of a histogram, and since
// order statistics move by no more than the values do, the k-th smallest y
// lies within E of that bucket: samples whose FP32 value is more than 2E
// below it are below the answer, those more than 2E above are above, and only
// the handful between are evaluated in FP64, with the same operations as a
// full evaluation, and ranked.  The result is the value a full FP64 sort
// gives, bit for bit.  A cell the bound or the bucket does not separate
// (repeated samples, a surrogate flat to FP32, coefficients outside the FP32
// range) is evaluated and sorted whole in FP64.
//
// Bound: latency of a block's passes over its values (16 warps an SM, the
// shared memory holds 8 cells' values).  4096 cells, 4096 samples, 21 terms: a
// bitonic sort of the FP64 values of each cell took 4848 us (FP64 compares,
// pipe 82% busy), this form takes 152 us.  Where every cell is sorted whole the
// call takes 2.17 ms (5.10 with that sort alone; 1000 samples: 0.64 and 1.04).
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "sclbm_internal.h"

namespace sclbm {
namespace {

constexpr int kThreads = 512;
constexpr int kSMs = 152;
constexpr int kBuckets = 1024;
constexpr int kCandidates = 192;  // exact evaluations held per (cell, quantile)

// Largest |Phi_a| over the samples, rounded up.
struct BasisBound {
  float m[kMaxGpcP];
};

// phi [M][P] (FP64) -> phif [P][Mf] (FP32, Mf the row length, pad 0).
__global__ void __launch_bounds__(256) basis_float_kernel(const double* __restrict__ phi, int M, int P, int Mf,
                                                          float* __restrict__ phif) {
  const int k = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (k >= P * Mf) return;
  const int a = k / Mf, m = k - a * Mf;
  phif[k] = m < M ? (float)phi[(long long)m * P + a] : 0.0f;
}

// The surrogate at one sample in FP64, terms in order.
__device__ __forceinline__ double surrogate(const double* __restrict__ row, const double* cs, int P) {
  double v = 0.0;
#pragma unroll 4
  for (int a = 0; a < P; ++a) v = fma(cs[a], row[a], v);
  return v;
}

// A double as a signed integer of the same order, and back (compared on the
// integer pipe); every NaN is the largest.
__device__ __forceinline__ long long ordered(double v) {
  const long long b = __double_as_longlong(v);
  if ((b & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL) return 0x7fffffffffffffffLL;
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double from_ordered(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}

__device__ __forceinline__ void bar_group(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// G cells a block; threads [g T, (g + 1) T), T = kThreads / G, select in cell g.
// Dynamic shared memory: max(G Mf floats, Mp doubles) of surrogate values.
template <int G>
__global__ void __launch_bounds__(kThreads) gpc_quantile_kernel(
    const double* __restrict__ coef, long long ncell, int P, const int32_t* __restrict__ cells, int n_cells,
    const double* __restrict__ phi, const float* __restrict__ phif, int M, int Mf, int Mp,
    const __grid_constant__ BasisBound bound, const int32_t* __restrict__ kidx, int nq, double* __restrict__ out) {
  extern __shared__ double values[];
  float* const val = reinterpret_cast<float*>(values);
  constexpr int T = kThreads / G, kWarps = T / 32;
  __shared__ double cs[G][kMaxGpcP];
  __shared__ float4 cf[kMaxGpcP][(G + 3) / 4];
  __shared__ int hist[G][kBuckets];
  __shared__ float lims[G][2 * kWarps], err[G], mid[G], spread[G];
  __shared__ short cand[G][kCandidates];
  __shared__ long long exact[G][kCandidates];  // FP64 values as integers of the same order
  __shared__ int n_cand[G], n_below[G], bucket[G], whole[G];
  const int cell0 = blockIdx.x * G;
  for (int k = threadIdx.x; k < G * P; k += kThreads) {
    const int g = k / P, a = k - g * P;
    const double c = cell0 + g < n_cells ? coef[(long long)a * ncell + cells[cell0 + g]] : 0.0;
    cs[g][a] = c;
    reinterpret_cast<float*>(cf[a])[g] = (float)c;
  }
  // E[g] >= |FP32 value - FP64 value| for every sample: with S = sum_a |c_a|
  // max |Phi_a| a rounding of the coefficient, one of the basis value and P of
  // the sum make at most (P + 2) 2^-24 S (1 + O(2^-24)); twice that is taken.
  // 0 for a cell without coefficients, +inf where a float does not carry a
  // factor or S (a coefficient or its basis bound outside 1e-30 .. 1e30, S
  // outside 1e-20 .. 1e25), or one is not a number.  A basis bound from 1e30 on
  // counts without a coefficient as well: the basis value may be infinite as a
  // float, and zero times it is no number.  In FP32, one warp a cell: in FP64
  // by every thread it was half of the kernel.
  for (int g = threadIdx.x / 32; g < G; g += kThreads / 32) {
    const int a = threadIdx.x % 32;
    const double c = a < P && cell0 + g < n_cells ? coef[(long long)a * ncell + cells[cell0 + g]] : 0.0;
    const bool some = (__double_as_longlong(c) << 1) != 0;
    const float f = fabsf((float)c), m = a < P ? bound.m[a] : 1.0f;
    float S = some ? f * m : 0.0f, v2 = a > 0 ? f * f : 0.0f;
    const bool off = !(m < 1e30f) || (some && !(f > 1e-30f && f < 1e30f && m > 1e-30f));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      S += __shfl_xor_sync(0xffffffffu, S, o);
      v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    }
    const bool any = __any_sync(0xffffffffu, some), bad = __any_sync(0xffffffffu, off);
    if (a == 0) {
      err[g] = bad ? INFINITY : !any ? 0.0f : S > 1e-20f && S < 1e25f ? S * (float)(P + 4) * 1.1920929e-7f : INFINITY;
      mid[g] = (float)c;
      spread[g] = 5.0f * sqrtf(v2);
    }
  }
  for (int k = threadIdx.x; k < G * kBuckets; k += kThreads) hist[k / kBuckets][k % kBuckets] = 0;
  __syncthreads();
  // FP32 values of the G cells, four samples a thread
  for (int m = 4 * threadIdx.x; m < Mf; m += 4 * kThreads) {
    float4 v[G];
#pragma unroll
    for (int g = 0; g < G; ++g) v[g] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int a = 0; a < P; ++a) {
      const float4 b = __ldg(reinterpret_cast<const float4*>(phif + (long long)a * Mf + m));
#pragma unroll
      for (int h = 0; h < (G + 3) / 4; ++h) {
        const float4 c4 = cf[a][h];
        const float c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (4 * h + j < G) {
            float4& w = v[4 * h + j];
            w.x = fmaf(c[j], b.x, w.x);
            w.y = fmaf(c[j], b.y, w.y);
            w.z = fmaf(c[j], b.z, w.z);
            w.w = fmaf(c[j], b.w, w.w);
          }
      }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) *reinterpret_cast<float4*>(val + g * Mf + m) = v[g];
  }
  __syncthreads();
  const int g = threadIdx.x / T, t = threadIdx.x - g * T, lane = t & 31, wid = t >> 5;
  const bool mine = cell0 + g < n_cells;
  const float* const y32 = val + g * Mf;
  // range of the FP32 values
  float mn = INFINITY, mx = -INFINITY;
  for (int m = t; m < M; m += T) {
    mn = fminf(mn, y32[m]);
    mx = fmaxf(mx, y32[m]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if (lane == 0) lims[g][2 * wid] = mn, lims[g][2 * wid + 1] = mx;
  bar_group(1 + g, T);
#pragma unroll
  for (int w = 0; w < kWarps; ++w) mn = fminf(mn, lims[g][2 * w]), mx = fmaxf(mx, lims[g][2 * w + 1]);
  const float E = err[g];
  const bool zero = E == 0.0f;  // a solid cell: every value is 0
  // the buckets cover five standard deviations about the mean (those of the
  // surrogate for its own input law: c_0 and the root of the other c_a^2), so
  // that a few far samples do not widen them; the first and the last one are
  // open and take what lies outside
  const float b0 = fmaxf(mn, mid[g] - spread[g]), b1 = fminf(mx, mid[g] + spread[g]);
  const float scale = (float)kBuckets / (b1 - b0);
  bool sort = !zero && !(E < 1e25f && b1 > b0 && scale < 1e30f);
  if (mine && !zero && !sort) {
    for (int m = t; m < M; m += T) atomicAdd(&hist[g][max(0, min((int)((y32[m] - b0) * scale), kBuckets - 1))], 1);
  }
  bar_group(1 + g, T);
  // running counts, in place: hist[b] = values in buckets 0 .. b (one warp a cell)
  if (wid == 0) {
    int carry = 0;
    for (int b = lane; b < kBuckets; b += 32) {
      int s = hist[g][b];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += up;
      }
      s += carry;
      hist[g][b] = s;
      carry = __shfl_sync(0xffffffffu, s, 31);
    }
  }
  // slack of the bucket limits as computed in floats
  const float slack = 4.0f * 1.1920929e-7f * fmaxf(fabsf(mn), fabsf(mx));
  for (int j = 0; j < nq; ++j) {
    const int k = kidx[j];
    if (t == 0) n_cand[g] = 0, n_below[g] = 0;
    bar_group(1 + g, T);
    if (!zero && !sort)
      for (int b = t; b < kBuckets; b += T)
        if (hist[g][b] >= k && (b == 0 || hist[g][b - 1] < k)) bucket[g] = b;
    bar_group(1 + g, T);
    if (zero || sort || !mine) {
      if (mine && zero && t == 0) out[(long long)j * n_cells + cell0 + g] = 0.0;
      continue;
    }
    const int b = bucket[g];
    const float lo = b == 0 ? -INFINITY : b0 + (float)b / scale - slack - 2.0f * E;
    const float hi = b == kBuckets - 1 ? INFINITY : b0 + (float)(b + 1) / scale + slack + 2.0f * E;
    int below = 0;
    for (int m = t; m < M; m += T) {
      const float v = y32[m];
      below += v < lo;
      if (v >= lo && v <= hi) {
        const int n = atomicAdd(&n_cand[g], 1);
        if (n < kCandidates) cand[g][n] = (short)m;
      }
    }
    below = __reduce_add_sync(0xffffffffu, below);
    if (lane == 0) atomicAdd(&n_below[g], below);
    bar_group(1 + g, T);
    const int n = n_cand[g], r = k - 1 - n_below[g];  // the answer's rank among the candidates
    bar_group(1 + g, T);  // the counts are cleared for the next quantile
    if (n > kCandidates) {
      sort = true;
      continue;
    }
    for (int i = t; i < n; i += T) exact[g][i] = ordered(surrogate(phi + (long long)cand[g][i] * P, cs[g], P));
    bar_group(1 + g, T);
    for (int i = t; i < n; i += T) {
      const long long y = exact[g][i];
      int less = 0, same = 0;
      for (int l = 0; l < n; ++l) {
        less += exact[g][l] < y;
        same += exact[g][l] == y && l < i;
      }
      if (less + same == r) out[(long long)j * n_cells + cell0 + g] = from_ordered(y);
    }
    bar_group(1 + g, T);
  }
  if (t == 0) whole[g] = mine && sort;
  __syncthreads();
  // cells left whole: all M values in FP64, as integers of their order sorted
  // ascending with a bitonic network over Mp >= M (a power of two) of them, the
  // tail padded with the largest one
  long long* const keys = reinterpret_cast<long long*>(values);
  for (int h = 0; h < G; ++h) {
    if (!whole[h]) continue;
    for (int m = threadIdx.x; m < Mp; m += kThreads)
      keys[m] = m < M ? ordered(surrogate(phi + (long long)m * P, cs[h], P)) : 0x7fffffffffffffffLL;
    __syncthreads();
    for (int k = 2; k <= Mp; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int p = threadIdx.x; p < Mp / 2; p += kThreads) {  // the pairs (i, i + j)
          const int i = 2 * p - (p & (j - 1)), l = i + j;
          const long long a = keys[i], b = keys[l];
          if ((a > b) == ((i & k) == 0)) {
            keys[i] = b;
            keys[l] = a;
          }
        }
        __syncthreads();
      }
    for (int j = threadIdx.x; j < nq; j += kThreads)
      out[(long long)j * n_cells + cell0 + h] = from_ordered(keys[kidx[j] - 1]);
    __syncthreads();
  }
}

template <int G>
int launch_group(const double* coef, long long ncell, int P, const int32_t* cells, int n_cells, const double* phi,
                 const float* phif, int M, int Mf, int Mp, const BasisBound& bound, const int32_t* kidx, int nq,
                 double* out, cudaStream_t s) {
  const size_t smem = std::max(sizeof(float) * (size_t)G * Mf, sizeof(double) * (size_t)Mp);
  // the same limit from every call, so that calls from several threads do not
  // lower one another's
  constexpr int kMostValues = 4 * 8 * 4096;
  static_assert(4 * 4 * SC_QUANTILE_MAX_SAMPLES <= kMostValues && 8 * SC_QUANTILE_MAX_SAMPLES <= kMostValues,
                "four cells' FP32 values and one cell's FP64 values fit");
  cudaError_t e = cudaFuncSetAttribute(gpc_quantile_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostValues);
  if (e != cudaSuccess) return (int)e;
  gpc_quantile_kernel<G><<<(n_cells + G - 1) / G, kThreads, smem, s>>>(coef, ncell, P, cells, n_cells, phi, phif, M,
                                                                       Mf, Mp, bound, kidx, nq, out);
  return (int)cudaGetLastError();
}

}  // namespace

int launch_gpc_quantiles(const double* coef, long long ncell, int P, const int32_t* cells, int n_cells,
                         const double* phi, const double* phi_max, float* phif, int M, const int32_t* kidx, int nq,
                         double* out, void* stream) {
  if (n_cells <= 0) return (int)cudaSuccess;
  cudaStream_t s = (cudaStream_t)stream;
  int Mp = 1;
  while (Mp < M) Mp <<= 1;
  const int Mf = (M + 3) / 4 * 4;
  BasisBound bound;
  for (int a = 0; a < kMaxGpcP; ++a)  // rounded up; one that is not finite sends the cells to the sort
    bound.m[a] = a < P ? nextafterf((float)phi_max[a], INFINITY) : 0.0f;
  basis_float_kernel<<<(P * Mf + 255) / 256, 256, 0, s>>>(phi, M, P, Mf, phif);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return (int)e;
  // eight cells share a basis value while their FP32 values fit the shared
  // memory of one block an SM (and the cells fill the chip); four above 4096
  // samples; one when there are few cells
  if (n_cells < 2 * kSMs)
    return launch_group<1>(coef, ncell, P, cells, n_cells, phi, phif, M, Mf, Mp, bound, kidx, nq, out, s);
  if (M > 4096 || n_cells < 8 * kSMs)
    return launch_group<4>(coef, ncell, P, cells, n_cells, phi, phif, M, Mf, Mp, bound, kidx, nq, out, s);
  return launch_group<8>(coef, ncell, P, cells, n_cells, phi, phif, M, Mf, Mp, bound, kidx, nq, out, s);
}

}  // namespace sclbm
