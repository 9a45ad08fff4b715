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
// form in every round: ten SGLD steps (n = 1,000, d = 2, 5 columns) 6.47 -> 5.00 ms, 100
// predictions with variance (n = 1,030, 101 columns) 19.0 -> 15.6 ms.
#include <cooperative_groups.h>

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

}  // namespace

cudaError_t launch_kmv_f64_dense(KmvLaunch& L, cudaStream_t s) {
  L.planned_nsplit = 1;
  if (L.plan_only) {
    L.need_partials_bytes = 0;
    L.need_counters = 0;
    return cudaSuccess;
  }
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
  static_assert(dense_smem((kKmatMaxN + kDnC - 1) / kDnC) <= 48 * 1024, "shared memory");
  L.launches = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(kDnC, (unsigned)((L.n + 31) / 32), (unsigned)((L.R + kDnW - 1) / kDnW));
  c.blockDim = dim3(kDnNT);
  c.dynamicSmemBytes = dense_smem(a.per);
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kDnC;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kmv_f64_dense_kernel, a);
}

}  // namespace ulisse
