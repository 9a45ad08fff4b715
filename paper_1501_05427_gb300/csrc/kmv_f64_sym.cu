// FP64 K V over unordered block pairs: k_ij = k_ji is formed once and applied to both rows.
//
// One CTA takes a pair (I, J), I <= J, of T-point blocks: it forms the T x T kernel values into
// shared memory, then adds K_IJ V_J to the rows of I and K_IJ^T V_I to the rows of J.  Both
// partial products go to scratch; a second launch sums each block's partials in partner order,
// multiplies by sigma^2 and adds the lambda V diagonal term (deterministic).  The sums are a
// launch of their own because a chain of FP64 adds takes 64 clocks each: spread over the SMs it
// is 3 us, on the last-arriving CTAs of the pair launch it took 25 us at n = 1,000.
//
// What bounds it: the FP64 pipe, about 1.7 lanes per clock per SM.  An ordered pair costs
// (2d + 7) / 2 + R operations here (exp64.cuh's exponential, sigma^2 taken out of the sums)
// against 2d + 17 + R one row block at a time with the library's exponential.  Shared-memory
// reads (two per FMA, no register tile) and the partials' traffic (nb x n x R doubles for nb
// blocks) stay far below the pipe, so the tile loops are plain.  T = 32 up to 2,048 points, so
// that the pairs (528 at n = 1,000) fill the SMs; 64 above, where a quarter as many partials
// matter more.  n = 1,000, d = 2, 5 columns: 70 us (row-block kernel, library exponential) ->
// 29 us + 4 us for the sums, 48% more than the pipe's 22 us (three or four pairs per SM, and
// 320 outputs over 128 threads); n = 1,030, 32 columns: 83 us.
#include <algorithm>
#include <mutex>

#include "exp64.cuh"
#include "ulisse_internal.cuh"

namespace ulisse {

__global__ void fill_exp_tab_kernel(double* __restrict__ tab) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < kExpTabN) tab[j] = exp2((double)j / (double)kExpTabN);
}

cudaError_t launch_fill_exp_tab(double* tab, cudaStream_t s) {
  fill_exp_tab_kernel<<<kExpTabN / 256, 256, 0, s>>>(tab);
  return cudaGetLastError();
}

namespace {

struct Sym64Args {
  const double* xhat;
  long long n;
  const double* V;
  long long ldv;
  const int* vmap;
  int R;
  double* U;
  long long ldu;
  const int* umap;
  const DevParams* params;
  const double* exp_tab;
  int which;
  int nb;                // blocks of T points
  double* partials;      // [block][partner][R][T]
};

constexpr long long kSymMaxPartialBytes = 256LL << 20;
constexpr int kSymRedNT = 128;
constexpr int kFillNT = 128;
constexpr int sym_tile(long long n) { return n <= 2048 ? 32 : 64; }

// U = sigma^2 (the block's nb partials in partner order) + lambda V.  Four lanes per element,
// each a quarter of the partners with eight loads in flight, then added pairwise: the chain of
// FP64 adds and of L2 round trips is a quarter as long.
template <int T, int MODE>
__global__ void __launch_bounds__(kSymRedNT) kmv_f64_sym_reduce_kernel(const Sym64Args a) {
  const int b = blockIdx.y;
  const int outs = a.R * T;
  const int t = blockIdx.x * kSymRedNT + threadIdx.x;
  const int o = min(t >> 2, outs - 1), q = t & 3;   // every lane takes part in the shuffles
  const int r = o / T;
  const long long i = (long long)b * T + (o - r * T);
  const int per = (a.nb + 3) / 4, c1 = min(a.nb, (q + 1) * per);
  const double* base = a.partials + (long long)b * a.nb * outs + o;
  double u = 0.0;
  for (int c = q * per; c < c1; c += 8) {
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = c + k < c1 ? base[(long long)(c + k) * outs] : 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (c + k < c1) u += v[k];
  }
  u += __shfl_xor_sync(0xffffffffu, u, 1);
  u += __shfl_xor_sync(0xffffffffu, u, 2);
  if (q != 0 || (t >> 2) >= outs || i >= a.n) return;
  u *= a.params->sigma2;
  if constexpr (MODE == kModeK)
    u = fma(a.params->lambda, a.V[(long long)a.vmap[r] * a.ldv + i], u);
  a.U[(long long)a.umap[r] * a.ldu + i] = u;
}

// pair p -> (bi, bj), bi <= bj: p = bj (bj + 1) / 2 + bi
__device__ __forceinline__ void pair_blocks(long long p, int& bi, long long& bj) {
  bj = (long long)((sqrtf(8.f * (float)p + 1.f) - 1.f) * 0.5f);
  while (bj * (bj + 1) / 2 > p) --bj;
  while ((bj + 1) * (bj + 2) / 2 <= p) ++bj;
  bi = (int)(p - bj * (bj + 1) / 2);
}

// The pair's T x T kernel values (sigma^2 left out; LIB: with it, by the library's exponential) into sK, rows of T + 1; sXI holds DP x T.
// Barriers before (the caller's own shared stores are then visible too) and after.
template <int DP, int T, int NT, int MODE, bool LIB = false>
__device__ __forceinline__ void form_pair(const double* __restrict__ xhat, long long n,
                                          const double* __restrict__ exp_tab, int which,
                                          long long i0, long long j0, double* sXI, double* sK,
                                          double sigma2 = 0.0) {
  constexpr int LD = T + 1;   // padded row: the transposed pass reads columns
  const int tid = threadIdx.x;
  for (int e = tid; e < DP * T; e += NT) {
    const int i = e / DP, k = e - i * DP;
    sXI[k * T + i] = i0 + i < n ? xhat[(i0 + i) * DP + k] : 0.0;
  }
  // thread's column j is fixed (NT is a multiple of T)
  const int j = tid % T;
  double xj[DP];
#pragma unroll
  for (int k = 0; k < DP; ++k) xj[k] = j0 + j < n ? xhat[(j0 + j) * DP + k] : 0.0;
  double xjw = 0.0;
  if constexpr (MODE == kModeDLen) xjw = j0 + j < n ? xhat[(j0 + j) * DP + which] : 0.0;
  __syncthreads();
#pragma unroll 4
  for (int i = tid / T; i < T; i += NT / T) {
    const double d0 = sXI[i] - xj[0];
    double dist = d0 * d0;
#pragma unroll
    for (int k = 1; k < DP; ++k) {
      const double df = sXI[k * T + i] - xj[k];
      dist = fma(df, df, dist);
    }
    double kv;
    if constexpr (LIB) kv = sigma2 * exp(-0.5 * dist);
    else kv = exp_neg_half(dist, exp_tab);
    if constexpr (MODE == kModeDLen) {
      const double dw = sXI[which * T + i] - xjw;
      kv *= dw * dw;
    }
    sK[i * LD + j] = kv;
  }
  __syncthreads();
}

template <int DP, int T, int NT, int MODE>
__global__ void __launch_bounds__(NT) kmv_f64_sym_kernel(const Sym64Args a) {
  constexpr int LD = T + 1;   // padded row: the transposed pass reads columns
  extern __shared__ __align__(16) double sm[];
  double* sK = sm;                       // T x LD
  double* sXI = sK + T * LD;             // DP x T
  double* sVI = sXI + DP * T;            // R x T
  double* sVJ = sVI + a.R * T;           // R x T
  const int tid = threadIdx.x;
  int bi;
  long long bj;
  pair_blocks(blockIdx.x, bi, bj);
  const long long i0 = (long long)bi * T, j0 = bj * T;
  const bool diag = bi == bj;

  for (int e = tid; e < a.R * T; e += NT) {
    const int r = e / T, i = e - r * T;
    const double* v = a.V + (long long)a.vmap[r] * a.ldv;
    sVI[e] = i0 + i < a.n ? v[i0 + i] : 0.0;
    sVJ[e] = j0 + i < a.n ? v[j0 + i] : 0.0;
  }
  form_pair<DP, T, NT, MODE>(a.xhat, a.n, a.exp_tab, a.which, i0, j0, sXI, sK);
  // rows of I: K V_J; rows of J: K^T V_I (a diagonal pair holds both orders itself)
  const int outs = a.R * T;
  double* partI = a.partials + ((long long)bi * a.nb + bj) * outs;
  double* partJ = a.partials + (bj * a.nb + bi) * outs;
  for (int o = tid; o < (diag ? outs : 2 * outs); o += NT) {
    const bool side_j = o >= outs;
    const int q = side_j ? o - outs : o;
    const int r = q / T, x = q - r * T;
    const double* kp = side_j ? sK + x : sK + x * LD;
    const int step = side_j ? LD : 1;
    const double* v = (side_j ? sVI : sVJ) + r * T;
    double u0 = 0.0, u1 = 0.0;
#pragma unroll 8
    for (int y = 0; y < T; y += 2) {
      u0 = fma(kp[y * step], v[y], u0);
      u1 = fma(kp[(y + 1) * step], v[y + 1], u1);
    }
    (side_j ? partJ : partI)[q] = u0 + u1;
  }
}

// The kernel values themselves, as form_pair, both orders of every pair: K is ldk x ldk, ldk a
// multiple of T.  Values of rows and columns past n are finite where x is, and unused.
template <int DP, bool LIB>
__global__ void __launch_bounds__(kFillNT) form_kmat_kernel(const double* __restrict__ xhat,
                                                            long long n,
                                                            const double* __restrict__ exp_tab,
                                                            const DevParams* __restrict__ params,
                                                            double* __restrict__ K, long long ldk) {
  constexpr int T = 32, LD = T + 1;
  __shared__ double sK[T * LD], sXI[DP * T];
  int bi;
  long long bj;
  pair_blocks(blockIdx.x, bi, bj);
  const long long i0 = (long long)bi * T, j0 = bj * T;
  form_pair<DP, T, kFillNT, kModeK, LIB>(xhat, n, exp_tab, 0, i0, j0, sXI, sK, params->sigma2);
  const int j = threadIdx.x % T;
  for (int i = threadIdx.x / T; i < T; i += kFillNT / T) {
    K[(i0 + i) * ldk + j0 + j] = sK[i * LD + j];
    if (bi != bj) K[(j0 + i) * ldk + i0 + j] = sK[j * LD + i];
  }
}

template <int DP, int T, int MODE>
cudaError_t sym_launch(KmvLaunch& L, cudaStream_t s) {
  constexpr int NT = T == 32 ? 128 : 256;
  auto fn = kmv_f64_sym_kernel<DP, T, NT, MODE>;
  static std::once_flag once;
  std::call_once(once, [&] {
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(double) * (T * (T + 1) + DP * T + 2 * kMaxRChunk * T));
  });
  Sym64Args a;
  a.xhat = static_cast<const double*>(L.xhat);
  a.n = L.n;
  a.V = static_cast<const double*>(L.V);
  a.ldv = L.ldv;
  a.vmap = L.vmap;
  a.R = L.R;
  a.U = static_cast<double*>(L.U);
  a.ldu = L.ldu;
  a.umap = L.umap;
  a.params = L.params;
  a.exp_tab = L.exp_tab;
  a.which = L.which;
  a.nb = (int)((L.n + T - 1) / T);
  a.partials = static_cast<double*>(L.partials);
  const long long pairs = (long long)a.nb * (a.nb + 1) / 2;
  const size_t smem = sizeof(double) * (size_t)(T * (T + 1) + DP * T + 2 * L.R * T);
  L.launches = 2;
  fn<<<(unsigned)pairs, NT, smem, s>>>(a);
  kmv_f64_sym_reduce_kernel<T, MODE>
      <<<dim3((unsigned)((4 * L.R * T + kSymRedNT - 1) / kSymRedNT), (unsigned)a.nb), kSymRedNT, 0, s>>>(a);
  return cudaGetLastError();
}

template <int DP, int T>
cudaError_t sym_mode(KmvLaunch& L, cudaStream_t s) {
  switch (L.mode) {
    case kModeK: return sym_launch<DP, T, kModeK>(L, s);
    case kModeDLen: return sym_launch<DP, T, kModeDLen>(L, s);
    case kModeDSig: return sym_launch<DP, T, kModeDSig>(L, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int DP>
cudaError_t sym_dp(KmvLaunch& L, cudaStream_t s) {
  return sym_tile(L.n) == 32 ? sym_mode<DP, 32>(L, s) : sym_mode<DP, 64>(L, s);
}

}  // namespace

template <bool LIB>
static cudaError_t form_kmat(const double* xhat, long long n, int DP, const double* exp_tab,
                             const DevParams* P, double* K, long long ldk, cudaStream_t s) {
  const long long nb = (n + 31) / 32;
  const unsigned pairs = (unsigned)(nb * (nb + 1) / 2);
  switch (DP) {
    case 2: form_kmat_kernel<2, LIB><<<pairs, kFillNT, 0, s>>>(xhat, n, exp_tab, P, K, ldk); break;
    case 4: form_kmat_kernel<4, LIB><<<pairs, kFillNT, 0, s>>>(xhat, n, exp_tab, P, K, ldk); break;
    case 8: form_kmat_kernel<8, LIB><<<pairs, kFillNT, 0, s>>>(xhat, n, exp_tab, P, K, ldk); break;
    case 16: form_kmat_kernel<16, LIB><<<pairs, kFillNT, 0, s>>>(xhat, n, exp_tab, P, K, ldk); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_form_kmat(const double* xhat, long long n, int DP, const double* exp_tab,
                             const DevParams* P, double* K, long long ldk, cudaStream_t s) {
  return exp_tab ? form_kmat<false>(xhat, n, DP, exp_tab, P, K, ldk, s)
                 : form_kmat<true>(xhat, n, DP, exp_tab, P, K, ldk, s);
}

size_t kmv_f64_sym_bytes(long long n, int R) {
  const size_t T = (size_t)sym_tile(n), nb = ((size_t)n + T - 1) / T;
  return nb * nb * T * R * 8;
}

// The pair form's scratch grows as n^2 R / T doubles; it is used while that is at most 256 MiB
// (n = 11,584 with 16 columns, 8,192 with 32) and can be had, else the row-block kernel runs, which
// the caller asks for by r_min; dK/dlog lambda has no pairs.
bool kmv_f64_sym_applies(const KmvLaunch& L) {
  if (L.mode == kModeDLam || L.r_min > 0 || !L.exp_tab) return false;
  return kmv_f64_sym_bytes(L.n, L.R) <= (size_t)kSymMaxPartialBytes;
}

cudaError_t launch_kmv_f64_sym(KmvLaunch& L, cudaStream_t s) {
  const size_t need = kmv_f64_sym_bytes(L.n, L.R);
  L.planned_nsplit = 1;
  if (L.plan_only || need > L.partials_bytes) {
    L.need_partials_bytes = need;
    L.need_counters = 0;
    return L.plan_only ? cudaSuccess : cudaErrorMemoryAllocation;
  }
  switch (L.DP) {
    case 2: return sym_dp<2>(L, s);
    case 4: return sym_dp<4>(L, s);
    case 8: return sym_dp<8>(L, s);
    case 16: return sym_dp<16>(L, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ulisse
