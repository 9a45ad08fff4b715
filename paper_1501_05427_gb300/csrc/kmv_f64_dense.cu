// FP64 K V from kernel values that a solve has formed (launch_form_kmat) and all its rounds read.
//
// What bounds it: the FP64 pipe, about 1.7 lanes per clock per SM, now with R operations per entry
// (the pair form, which makes the values anew for each product, (2d + 7) / 2 + R).  K lies in L2
// at the usual sizes; even from HBM a value's 8 bytes take a tenth of the time its making does.
//
// A cluster of eight CTAs takes 32 rows and up to eight columns of V: each CTA an eighth of the
// points j, each warp every eighth of those, a row per lane (K is symmetric, so the lanes read
// row j of K, 256 contiguous bytes).  The eight warps' sums are added in shared memory and the
// eight CTAs' over distributed shared memory, both in a fixed order: one launch, no scratch.
// Eight columns per CTA, because a load of K per eight FMAs is no burden at this rate and the
// columns then divide evenly; CTAs of eight warps hide the 64-clock FP64 latency.  Against the pair
// form in every round: 100 predictions with variance (n = 1,030, 101 columns) 19.0 -> 13.4 ms; a
// round of 101 columns takes 215 us or so, the pipe's time is 200.  The second form below, with
// the row-block kernel's additions, serves the truncated solves: ten SGLD steps (n = 1,000, d = 2,
// 5 columns) 13.0 ms with that kernel, 6.3 ms here (5.0 ms with the first form's additions).
#include <cooperative_groups.h>

#include <algorithm>

#include "ulisse_internal.cuh"

namespace ulisse {
namespace {

namespace cg = cooperative_groups;

constexpr int kDnNT = 256;
constexpr int kDnWarps = kDnNT / 32;
constexpr int kDnC = 8;         // CTAs per cluster
constexpr int kDnW = 8;         // columns per CTA, at most
constexpr int kDnUnroll = 8;

struct Dense64Args {
  const double* K;
  long long ldk;
  long long n;
  const double* V;
  long long ldv;
  const int* vmap;
  int R;
  double* U;
  long long ldu;
  const int* umap;
  const DevParams* params;
  int per;                      // points j per CTA
};

// Doubles of shared memory: the CTA's part of V, then (same place) its warps' sums; and the CTA's
// sums, which the cluster reads.
constexpr size_t dense_smem(int per) {
  return sizeof(double) * kDnW * ((size_t)(per > kDnNT ? per : kDnNT) + 32);
}

template <int W>
__device__ __forceinline__ void dense_body(const Dense64Args& a, const int c0, double* sm) {
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cl.block_rank();
  const long long i0 = (long long)blockIdx.y * 32, j0 = (long long)rank * a.per;
  const long long left = a.n - j0;
  const int jn = left <= 0 ? 0 : left < a.per ? (int)left : a.per;
  double* sum = sm + kDnW * (a.per > kDnNT ? a.per : kDnNT);

  for (int e = tid; e < jn * W; e += kDnNT) {
    const int r = e / jn, j = e - r * jn;
    sm[j * W + r] = a.V[(long long)a.vmap[c0 + r] * a.ldv + j0 + j];
  }
  __syncthreads();
  double acc[W];
#pragma unroll
  for (int r = 0; r < W; ++r) acc[r] = 0.0;
  const double* K = a.K + j0 * a.ldk + i0 + lane;
  for (int j = warp; j < jn; j += kDnWarps * kDnUnroll) {
    double k[kDnUnroll];
#pragma unroll
    for (int q = 0; q < kDnUnroll; ++q) {
      const int jq = j + q * kDnWarps;
      k[q] = jq < jn ? K[jq * a.ldk] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kDnUnroll; ++q) {
      const int jq = j + q * kDnWarps;
      if (jq < jn) {
#pragma unroll
        for (int r = 0; r < W; ++r) acc[r] = fma(k[q], sm[jq * W + r], acc[r]);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < W; ++r) sm[(warp * W + r) * 32 + lane] = acc[r];
  __syncthreads();
  if (tid < 32 * W) {
    const double* p = sm + tid;
    const int st = W * 32;
    sum[tid] = ((p[0] + p[st]) + (p[2 * st] + p[3 * st])) + ((p[4 * st] + p[5 * st]) + (p[6 * st] + p[7 * st]));
  }
  cl.sync();
  // output o = column x row: each CTA of the cluster finishes 4 W of the 32 W
  if (tid < 4 * W) {
    const int o = rank * 4 * W + tid, r = o >> 5;
    const long long i = i0 + (o & 31);
    double v[kDnC];
#pragma unroll
    for (int c = 0; c < kDnC; ++c) v[c] = *cl.map_shared_rank(sum + o, c);
    double u = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    if (i < a.n) {
      u *= a.params->sigma2;
      u = fma(a.params->lambda, a.V[(long long)a.vmap[c0 + r] * a.ldv + i], u);
      a.U[(long long)a.umap[c0 + r] * a.ldu + i] = u;
    }
  }
  cl.sync();   // the others may still be reading this CTA's sums
}

// Grid (cluster, row block, column chunk); the columns are spread evenly over the chunks.
__global__ void __launch_bounds__(kDnNT) kmv_f64_dense_kernel(const Dense64Args a) {
  extern __shared__ __align__(16) double sm[];
  const int chunks = gridDim.z, z = blockIdx.z;
  const int base = a.R / chunks, more = a.R - base * chunks;
  const int c0 = z * base + min(z, more);
  switch (base + (z < more)) {
    case 1: dense_body<1>(a, c0, sm); break;
    case 2: dense_body<2>(a, c0, sm); break;
    case 3: dense_body<3>(a, c0, sm); break;
    case 4: dense_body<4>(a, c0, sm); break;
    case 5: dense_body<5>(a, c0, sm); break;
    case 6: dense_body<6>(a, c0, sm); break;
    case 7: dense_body<7>(a, c0, sm); break;
    default: dense_body<8>(a, c0, sm); break;
  }
}

// The same products with the row-block kernel's additions (kmv_kernel.cuh): a row's sum over each
// split's points one after the other, then the splits' sums.  A truncated solve's estimates follow
// the rounding of its products (the trajectory amplifies 2^-53 to 1e-3 within ten steps of a
// chain), so a solve's products keep theirs.  A warp takes 32 rows, up to eight columns and one
// split at a time; the cluster's CTAs share the splits.  The chains of dependent additions are as
// long as a split, but a warp has a chain per column and every SM quarter has a warp or two, which
// the FP64 pipe's 64 clocks per instruction and quarter keep busy.
constexpr int kOrWarps = 4;
constexpr int kOrNT = 32 * kOrWarps;
constexpr int kOrTile = 64;
constexpr int kOrMaxSplits = 64;   // of a plan
constexpr int kOrStage = kOrTile * kDnW;

template <int W>
__device__ __forceinline__ void ordered_body(const Dense64Args& a, const int c0, const int nsplit,
                                             const int tps, double* sm) {
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
  const int spc = (nsplit + C - 1) / C;   // splits per CTA
  const long long i0 = (long long)blockIdx.y * 32;
  double* sv = sm + warp * kOrStage;
  double* part = sm + kOrWarps * kOrStage;

  const int s1 = min(nsplit, (rank + 1) * spc);
  for (int sp = rank * spc + warp; sp < s1; sp += kOrWarps) {
    double acc[W];
#pragma unroll
    for (int r = 0; r < W; ++r) acc[r] = 0.0;
    for (int t = 0; t < tps; ++t) {
      const long long j0 = ((long long)sp * tps + t) * kOrTile;
      const long long left = a.n - j0;
      if (left <= 0) break;
      const int jn = left < kOrTile ? (int)left : kOrTile;
      __syncwarp();
      for (int e = lane; e < kOrTile * W; e += 32) {
        const int r = e / kOrTile, j = e - r * kOrTile;
        sv[j * W + r] = j < jn ? a.V[(long long)a.vmap[c0 + r] * a.ldv + j0 + j] : 0.0;
      }
      const double* K = a.K + j0 * a.ldk + i0 + lane;
      double k[kDnUnroll];
#pragma unroll
      for (int q = 0; q < kDnUnroll; ++q) k[q] = q < jn ? K[q * a.ldk] : 0.0;
      __syncwarp();
#pragma unroll 1
      for (int j = 0; j < jn; j += kDnUnroll) {
        double next[kDnUnroll];
#pragma unroll
        for (int q = 0; q < kDnUnroll; ++q) {
          const int jq = j + kDnUnroll + q;
          next[q] = jq < jn ? K[jq * a.ldk] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < kDnUnroll; ++q)
#pragma unroll
          for (int r = 0; r < W; ++r) acc[r] = fma(k[q], sv[(j + q) * W + r], acc[r]);
#pragma unroll
        for (int q = 0; q < kDnUnroll; ++q) k[q] = next[q];
      }
    }
#pragma unroll
    for (int r = 0; r < W; ++r) part[((sp - rank * spc) * W + r) * 32 + lane] = acc[r];
  }
  cl.sync();
  for (int o = rank * kOrNT + tid; o < 32 * W; o += C * kOrNT) {
    const int r = o >> 5;
    const long long i = i0 + (o & 31);
    double u = 0.0;
    for (int s0 = 0; s0 < nsplit; s0 += 8) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int c = (s0 + q) / spc, l = s0 + q - c * spc;
        v[q] = s0 + q < nsplit ? *cl.map_shared_rank(part + l * W * 32 + o, c) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (s0 + q < nsplit) u += v[q];
    }
    if (i < a.n) {
      u = fma(a.params->lambda, a.V[(long long)a.vmap[c0 + r] * a.ldv + i], u);
      a.U[(long long)a.umap[c0 + r] * a.ldu + i] = u;
    }
  }
  cl.sync();   // the others may still be reading this CTA's sums
}

__global__ void __launch_bounds__(kOrNT) kmv_f64_ordered_kernel(const Dense64Args a, const int nsplit,
                                                                const int tps) {
  extern __shared__ __align__(16) double sm[];
  const int chunks = gridDim.z, z = blockIdx.z;
  const int base = a.R / chunks, more = a.R - base * chunks;
  const int c0 = z * base + min(z, more);
  switch (base + (z < more)) {
    case 1: ordered_body<1>(a, c0, nsplit, tps, sm); break;
    case 2: ordered_body<2>(a, c0, nsplit, tps, sm); break;
    case 3: ordered_body<3>(a, c0, nsplit, tps, sm); break;
    case 4: ordered_body<4>(a, c0, nsplit, tps, sm); break;
    case 5: ordered_body<5>(a, c0, nsplit, tps, sm); break;
    case 6: ordered_body<6>(a, c0, nsplit, tps, sm); break;
    case 7: ordered_body<7>(a, c0, nsplit, tps, sm); break;
    default: ordered_body<8>(a, c0, nsplit, tps, sm); break;
  }
}

template <typename... Params, typename... Args>
cudaError_t launch_cluster(void (*kernel)(Params...), dim3 grid, int threads, size_t smem,
                           cudaStream_t s, Args... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = grid.x;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

Dense64Args dense_args(const KmvLaunch& L) {
  Dense64Args a;
  a.K = L.kmat;
  a.ldk = kmat_ld(L.n);
  a.n = L.n;
  a.V = static_cast<const double*>(L.V);
  a.ldv = L.ldv;
  a.vmap = L.vmap;
  a.R = L.R;
  a.U = static_cast<double*>(L.U);
  a.ldu = L.ldu;
  a.umap = L.umap;
  a.params = L.params;
  a.per = (int)((L.n + kDnC - 1) / kDnC);
  return a;
}

bool dense_plan(KmvLaunch& L) {
  L.planned_nsplit = 1;
  L.launches = 1;
  if (!L.plan_only) return false;
  L.need_partials_bytes = 0;
  L.need_counters = 0;
  return true;
}

}  // namespace

cudaError_t launch_kmv_f64_dense(KmvLaunch& L, cudaStream_t s) {
  if (dense_plan(L)) return cudaSuccess;
  const Dense64Args a = dense_args(L);
  static_assert(dense_smem((kKmatMaxN + kDnC - 1) / kDnC) <= 48 * 1024, "shared memory");
  const dim3 grid(kDnC, (unsigned)((L.n + 31) / 32), (unsigned)((L.R + kDnW - 1) / kDnW));
  return launch_cluster(kmv_f64_dense_kernel, grid, kDnNT, dense_smem(a.per), s, a);
}

cudaError_t launch_kmv_f64_ordered(KmvLaunch& L, int nsplit, cudaStream_t s) {
  if (dense_plan(L)) return cudaSuccess;
  const int ntiles = (int)((L.n + kOrTile - 1) / kOrTile);
  if (nsplit < 1 || nsplit > kOrMaxSplits) return cudaErrorInvalidValue;
  const int tps = (ntiles + nsplit - 1) / nsplit;
  const int C = std::min(8, (nsplit + kOrWarps - 1) / kOrWarps), spc = (nsplit + C - 1) / C;
  const size_t smem = sizeof(double) * (kOrWarps * kOrStage + spc * kDnW * 32);
  static_assert(sizeof(double) * (kOrWarps * kOrStage + kOrMaxSplits / 8 * kDnW * 32) <= 48 * 1024,
                "shared memory");
  const dim3 grid(C, (unsigned)((L.n + 31) / 32), (unsigned)((L.R + kDnW - 1) / kDnW));
  return launch_cluster(kmv_f64_ordered_kernel, grid, kOrNT, smem, s, dense_args(L), nsplit, tps);
}

}  // namespace ulisse
