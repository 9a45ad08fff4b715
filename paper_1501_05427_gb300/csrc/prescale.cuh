// a1: parameter unpack and input prescale (shared by the context path and the
// allocation-free K V entry point).
//
// What bounds it: latency and the FP64 pipe (1.7 lanes per clock per SM).  The 1 / l_k are
// formed once per CTA, one exponential per thread; x^ = x / l in float comes from the product with
// 1 / l_k held as a pair of floats (48 bits) where that decides the rounding of the FP64 product,
// so that hardly any element takes an FP64 multiply and two conversions.  With every thread
// forming all 1 / l_k and FP64 products the launch took 10.7 us at n = 9,937, d = 4 and 27.5 us at
// n = 50,000, d = 8 (mixed precision: then two more launches of 5 us for the row norms and the
// TF32 images, now the same launch).  A whole product call, which also loses the copies of psi, V
// and U, went from 45 to 25 us at n = 1,030, d = 8, 5 columns (FP32) and from 840 to 795 us at
// n = 50,000 (mixed).
#pragma once

#include <algorithm>

#include "pack_v.cuh"
#include "tc_common.cuh"
#include "ulisse_internal.cuh"

namespace ulisse {

// Parameters by value (a host call's psi needs no copy of its own), else from psi_dev.
struct PsiArg {
  double v[kMaxP];
  int by_value;
};

// A product's operand V (R columns, leading dimension n) packed by the prescale launch (V null: no).
struct PackV {
  const float* V;
  int R, N;        // columns, MMA columns
  void* Vp;
  int first_cta;   // the CTAs from here on pack (set by the launcher)
};

inline int pack_v_ctas(long long n, int N, int threads, int num_sms) {
  const long long total = (n + 31) / 32 * 32 * N;
  return (int)std::max<long long>(1, std::min<long long>((total + 4 * threads - 1) / (4 * threads),
                                                         8LL * num_sms * 256 / threads));
}

// 1 / l_k as a double and as the pair hi + lo of floats.
struct InvLength {
  double inv[kMaxD];
  float hi[kMaxD], lo[kMaxD];
};

// Every CTA: 1 / l_k into s; CTA 0 also writes the derived parameters (and psi when given by
// value).  Ends with a barrier; needs at least kMaxP threads.
__device__ inline void unpack_params(const PsiArg& pa, double* __restrict__ psi_dev, int d,
                                     DevParams* __restrict__ P, InvLength& s) {
  const int k = threadIdx.x;
  if (k < d + 2) {
    const double p = pa.by_value ? pa.v[k] : psi_dev[k];
    const double e = exp(k < d ? -p : p);
    if (k < d) {
      s.inv[k] = e;
      s.hi[k] = (float)e;
      s.lo[k] = (float)(e - (double)s.hi[k]);
    }
    if (blockIdx.x == 0) {
      P->psi[k] = p;
      if (pa.by_value) psi_dev[k] = p;
      if (k < d) P->inv_l[k] = e;
      if (k == d) {
        P->sigma2 = e;
        P->c0f = (float)log2(e);
        P->c1f = (float)(0.5 * 1.4426950408889634);  // log2(e) / 2
      }
      if (k == d + 1) {
        P->lambda = e;
        P->lambdaf = (float)e;
      }
    }
  }
  __syncthreads();
}

// (float)(x / l), rounded as the FP64 product is: x (hi + lo) from the pair, whose error (the pair's
// 48 bits, the rounding of c) is below 2^-46 of it, where the ends of p + c (1 -+ 2^-44 p) round to
// one float and neither part nor the product's error term can leave the normal range; else the
// FP64 product (about one element in 2^19).
__device__ __forceinline__ float scale_by_pair(float x, const InvLength& s, int k) {
  const float hi = s.hi[k];
  const float p = x * hi;
  if (fabsf(p) < 1e30f && fabsf(p) > 1e-28f && hi > 1e-28f && hi < 1e30f) {
    const float c = fmaf(x, s.lo[k], fmaf(x, hi, -p)), w = fabsf(p) * 0x1p-44f;
    const float y = p + (c - w);
    if (y == p + (c + w)) return y;
  }
  return x == 0.f ? x : (float)((double)x * s.inv[k]);
}

template <typename T>
__device__ __forceinline__ T scaled(float x, const InvLength& s, int k) {
  if constexpr (sizeof(T) == 4) return scale_by_pair(x, s, k);
  else return (double)x * s.inv[k];
}

// x^ = x / l for rows [0, n) (rows >= n stay zero; dims >= d zero), one element per thread; the
// CTAs from row_blocks on copy (and convert) R columns of V, leading dimension n, to D, leading
// dimension ldn, or pack pv.
template <typename T, typename TV>
__global__ void __launch_bounds__(256) prescale_kernel(
    const PsiArg pa, double* __restrict__ psi_dev, const float* __restrict__ X,
    T* __restrict__ xhat, long long n, int d, int log2_dp, DevParams* __restrict__ P,
    int row_blocks, const TV* __restrict__ V, T* __restrict__ D, long long ldn, int R,
    const PackV pv) {
  __shared__ InvLength s;
  if ((int)blockIdx.x < row_blocks) {
    unpack_params(pa, psi_dev, d, P, s);
    const long long total = n << log2_dp;
    for (long long idx = blockIdx.x * 256LL + threadIdx.x; idx < total; idx += row_blocks * 256LL) {
      const int k = (int)(idx & ((1 << log2_dp) - 1));
      const long long i = idx >> log2_dp;
      xhat[idx] = k < d ? scaled<T>(X[i * d + k], s, k) : T(0);
    }
    return;
  }
  if (pv.V) {   // FP32 tensor-core products
    pack_v3(pv.V, n, nullptr, pv.R, pv.N, n, (n + 31) / 32, static_cast<__nv_bfloat16*>(pv.Vp),
            blockIdx.x - row_blocks, gridDim.x - row_blocks);
    return;
  }
  const long long total = n * R, step = (gridDim.x - row_blocks) * 256LL;
  for (long long idx = (blockIdx.x - row_blocks) * 256LL + threadIdx.x; idx < total; idx += step) {
    const long long c = idx / n;
    D[c * ldn + (idx - c * n)] = (T)V[idx];
  }
}

inline int log2_of(int dp) { return dp == 2 ? 1 : dp == 4 ? 2 : dp == 8 ? 3 : 4; }

// Launch of prescale_kernel; V and pv.V null: no columns to copy or pack.
template <typename T, typename TV>
cudaError_t launch_prescale(const PsiArg& pa, double* psi_dev, const float* X, T* xhat, long long n,
                            int d, int DP, DevParams* P, const TV* V, T* D, long long ldn, int R,
                            PackV pv, int num_sms, cudaStream_t s) {
  // four elements per thread, at most eight CTAs per SM for each of the two parts
  auto blocks = [&](long long total) {
    return (int)std::max<long long>(1, std::min<long long>((total + 1023) / 1024, 8LL * num_sms));
  };
  const int rb = blocks(n * DP);
  const int more = pv.V ? pack_v_ctas(n, pv.N, 256, num_sms) : V ? blocks(n * R) : 0;
  prescale_kernel<T, TV><<<rb + more, 256, 0, s>>>(pa, psi_dev, X, xhat, n, d, log2_of(DP), P, rb, V,
                                                   D, ldn, R, pv);
  return cudaGetLastError();
}

}  // namespace ulisse
