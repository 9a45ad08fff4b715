// FP32 tile-generating K V with the contraction on the tensor cores, from BF16 parts of each float.
//
// The kernel values are formed as the SIMT kernel forms them (distance from the differences of
// the prescaled inputs, one FMA, one ex2, FP32 throughout).  The contraction U_I += K_IJ V_J runs
// as BF16 products of an exact split: a float is the sum of three BF16 values (24 bits = 3 x 8),
// and of the nine products of (h + m + l)_K (h + m + l)_V the six above 2^-24 are taken,
//     l h + m m + h l,  m h + h m,  h h   (small terms first),
// accumulated by the tensor cores in FP32.  Tensor memory truncates each accumulation, which adds
// up over a long range; here a 32-point tile's product (12 MMAs) starts from zero and is added to
// running FP32 sums in registers (round to nearest) by four draining warps, so that the rounding
// is that of n / 32 FP32 additions instead of the SIMT kernel's n FMAs in sequence.
//
// Rounding, against 64 bits: the three products left out are below 2^-26 of a term; of the 12
// truncations the last two, of the halves of h h, are of the tile's own size, so a tile's product
// is off by 2.1 2^-23 at most and low by 1.1 2^-24 on average: sums come out low by 6e-8 of
// themselves (the SIMT kernel's by 2e-8).  Errors of products are 0.3 to 0.8 of the SIMT
// kernel's over n = 500 to 22,784, d = 1 to 16 at the lengthscales in use, where its chain of n
// roundings counts; with K close to sigma^2 I (lengthscales 0.1 to 0.3 of those, n = 1,030, d = 4
// to 16) one term makes a row and they are up to 1.09 of it (5.5e-8 / 6.1e-8).
//
// What bounds it: the FP32 pipe, 2 DP + 4 lanes per entry (distance, exponent, the split's
// subtractions), whatever the column count, against 2 DP + 1 + R in the SIMT kernel; the BF16
// conversions (three per two entries at 32 lanes per clock per SM) come next.  n = 22,784, d = 8:
// 0.47 ms at any count up to 32 columns (ncu: issue 73%, FMA pipe 68%); the SIMT kernel takes 0.74
// ms at 17 columns and 1.12 ms at 32.
//
// Roles (544 threads, two CTAs per SM): warp 0 copies x^_J and V_J into a ring of stages and
// issues the MMAs (warp-uniform, one lane elected); warps 1-12 make the kernel values in three
// sets of four (one warp per tensor-memory lane quadrant, a row per thread): set h takes the
// tiles h, h + 3, ... and owns the K buffer h (48 columns: per 16 points high | middle | low);
// warps 13-16 drain the two accumulator buffers.  Every wait is bounded.  The split j range and
// the fixed-order fix-up of the partial sums are those of the other K V kernels.
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "batch.cuh"
#include "kmv_kernel.cuh"
#include "pack_v.cuh"
#include "tc_common.cuh"

namespace ulisse {

// The split of a problem's j range: by its size alone, so that a problem gives the same bits on
// its own and in a batch (the tiles' sums are added in the same order).  The other kernels' plan
// stops at four waves of CTAs; from about 32,000 points on (several hundred row blocks on 304 places)
// that leaves up to a quarter of the places empty in the last wave, and a product of 7 to 9 columns
// took up to 19% longer than the SIMT kernel's (d = 2, n = 64,000: 2.70 against 2.28 ms).  There a
// larger split is taken when it saves 5% of the waves' tiles (a CTA's start and end count as 8 tiles)
// with partial sums of at most 64 MiB, which a context comes with.
int f3_nsplit(long long n, int num_sms) {
  const long long ntiles = (n + 31) / 32, nrb = (n + 127) / 128, slots = 2 * num_sms;
  auto whole = [&](long long s) {   // without empty ranges
    const long long tps = (ntiles + s - 1) / s;
    return (ntiles + tps - 1) / tps;
  };
  auto cost = [&](long long s) {
    return (nrb * s + slots - 1) / slots * ((ntiles + s - 1) / s + 8);
  };
  const long long plan = whole(plan_split(n, 128, 32, 4, (int)slots).nsplit);
  if (2 * nrb <= slots) return (int)plan;
  long long best = plan;
  for (long long s = plan + 1; s <= 64 && nrb * s * (32 * 128 * 4) <= (64LL << 20); ++s)
    if (cost(s) < cost(best)) best = s;
  best = whole(best);
  return (int)(100 * cost(best) < 95 * cost(plan) ? best : plan);
}

// Consecutive ranges that a CTA of a batch takes one after the other, `tiles` tiles or more: the sums
// are those of the product on its own, which has a CTA per range to fill the SMs by itself.  Many
// problems fill them anyway, and with one or two tiles per CTA (n = 1,000) their starts and ends,
// about 8 tiles' time each, were most of a launch: a round of 64 problems of 300 to 2,000 points,
// 9 columns, 357 -> 295 us (the SIMT kernel 338); few problems keep a CTA per range.
int f3_ranges_per_cta(long long n, int nsplit, long long tiles) {
  const long long ntiles = (n + 31) / 32, tps = (ntiles + nsplit - 1) / nsplit;
  return (int)std::max(1LL, std::min<long long>(nsplit, (tiles + tps - 1) / tps));
}

size_t kmv_tile_partial_bytes(long long n, int num_sms, bool mixed) {
  const size_t nrb = ((size_t)n + 127) / 128;
  size_t ns = f3_nsplit(n, num_sms);
  if (mixed) ns = tc_bound_split(plan_split(n, 128, 32, 4, 4 * num_sms), n, 128, 32, 32).nsplit;
  return ns > 1 ? nrb * ns * 32 * 128 * 4 : 0;
}

namespace {

constexpr int kF3BN = 32;
constexpr int kF3BM = 128;
constexpr int kF3Sets = 3;
constexpr int kF3Drain = 1 + 4 * kF3Sets;            // first draining warp
constexpr int kF3Threads = 32 * (kF3Drain + 4);
constexpr uint32_t kF3Cols = 256;                    // tensor-memory columns per CTA

struct F3Args {
  const float* xhat;
  const __nv_bfloat16* Vp;   // tiles of V: high | middle | low part; then pack_v3's words
  const float* V;
  long long ldv;
  const int* vmap;
  int R;
  const int* R_dev;          // batched launches: the live column count on the device (else null)
  float* U;
  long long ldu;
  const int* umap;
  long long n;
  int DP;
  const DevParams* params;
  int which;                 // kModeDLen: the dimension
  int add_diag;              // lambda V (K), not for the derivatives
  int nsplit, tiles_per_split, ntiles;
  float* partials;
  int* counters;
  int* status;
};

template <int DP, int N>
struct F3Shape {
  static constexpr uint32_t X_BYTES = kF3BN * DP * 4;
  static constexpr uint32_t V_PART = N * kF3BN * 2;
  static constexpr uint32_t STAGE_BYTES = X_BYTES + 3 * V_PART;
  static constexpr int ST = 8;
  static constexpr uint32_t OFF_BARS = ST * STAGE_BYTES;
  static constexpr int NBARS = ST + 2 * kF3Sets + 4 + 1;   // full, k_full, b_free, u_full/free, done
  static constexpr uint32_t SMEM = OFF_BARS + NBARS * 8 + 64;
  static constexpr uint32_t COL_U = 48 * kF3Sets;
  static_assert(COL_U + 2 * 32 <= kF3Cols, "tensor memory layout exceeds the allocation");
  static_assert(2 * (SMEM + 2048) <= 228 * 1024, "two CTAs per SM");
};

__global__ void pack_v3_kernel(const float* __restrict__ V, long long ldv,
                               const int* __restrict__ vmap, int R, int N, long long n,
                               long long ntiles, __nv_bfloat16* __restrict__ Vp) {
  pack_v3(V, ldv, vmap, R, N, n, ntiles, Vp, blockIdx.x, gridDim.x);
}

// One problem per grid row; problems below the line are the SIMT launch's.
__global__ void pack_v3_batch_kernel(const F3Args* __restrict__ args, int N) {
  const F3Args& a = args[blockIdx.y];
  const int R = a.R_dev ? *a.R_dev : a.R;
  if (!batch_tc_columns(a.n, R)) return;
  pack_v3(a.V, a.ldv, a.vmap, R, N, a.n, a.ntiles, const_cast<__nv_bfloat16*>(a.Vp), blockIdx.x,
          gridDim.x);
}

// Kernel values (j, j + 1) of a row against two points of the tile: xj points at point j.
template <int DP>
__device__ __forceinline__ float f3_dist(const float2 (&nx)[DP / 2], const float* xj) {
  float2 acc = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k < DP; k += 4) {
    float2 a, b;
    if constexpr (DP >= 4) {
      const float4 x = *reinterpret_cast<const float4*>(xj + k);
      a = make_float2(x.x, x.y);
      b = make_float2(x.z, x.w);
    } else {
      a = *reinterpret_cast<const float2*>(xj);
    }
    const float2 da = __fadd2_rn(a, nx[k / 2]);
    acc = k == 0 ? __fmul2_rn(da, da) : __ffma2_rn(da, da, acc);
    if constexpr (DP >= 4) {
      const float2 db = __fadd2_rn(b, nx[k / 2 + 1]);
      acc = __ffma2_rn(db, db, acc);
    }
  }
  return acc.x + acc.y;
}

__device__ __forceinline__ uint32_t f3_bits(const __nv_bfloat162& v) {
  return *reinterpret_cast<const uint32_t*>(&v);
}

// Rows whose sum came out as NaN, once more: a column of V that holds an infinity meets zeros and
// both signs among the parts of K, where k_ij > 0 itself gives that infinity.  The terms that are
// not finite decide such a sum, so only they are formed, from the words that the packing wrote;
// a column without any stays as it is (its sum overflowed, or the inputs are not finite).
// From sigma^2 = 2^127 on, the kernel values' high parts can be infinite too: then all terms are.
// Not reached by finite results.  n = 22,784, d = 8, 17 columns, 0.51 ms per call: with a NaN among the
// inputs (every result a NaN) 0.52 ms, 9.6 with a scan of V per entry; with an infinity in one
// column 0.72, then 2.2.
template <int N, int MODE>
__device__ __noinline__ void f3_not_finite(const F3Args& a, const long long row0, const int R,
                                           unsigned* s_cols) {
  const uint32_t* bad =
      reinterpret_cast<const uint32_t*>(a.Vp + (long long)a.ntiles * 3 * N * kF3BN);
  if (threadIdx.x == 0) *s_cols = 0;   // the columns with a value that is not finite
  __syncthreads();
  for (int e = threadIdx.x; e < a.ntiles * N; e += kF3Threads)
    if (bad[e]) atomicOr(s_cols, 1u << (e % N));
  __syncthreads();
  const float c0 = a.params->c0f, c1 = a.params->c1f;
  const bool all = !(c0 < 127.f);
  const unsigned cols = all ? ~0u : *s_cols;
  for (int idx = threadIdx.x; idx < R * kF3BM; idx += kF3Threads) {
    const int r = idx / kF3BM;
    const long long i = row0 + (idx - r * kF3BM);
    if (i >= a.n || !(cols >> r & 1u)) continue;
    float* out = a.U + (long long)a.umap[r] * a.ldu + i;
    if (!isnan(*out)) continue;
    const float* v = a.V + (long long)a.vmap[r] * a.ldv;
    const float* xi = a.xhat + i * a.DP;
    float u = 0.f;
    for (int t = 0; t < a.ntiles && !isnan(u); ++t) {
      uint32_t m = all ? ~0u : bad[t * N + r];
      for (; m; m &= m - 1) {
        const long long j = (long long)t * kF3BN + __ffs(m) - 1;
        if (j >= a.n) break;
        const float* xj = a.xhat + j * a.DP;
        float dist = 0.f;
        for (int k = 0; k < a.DP; ++k) dist = fmaf(xi[k] - xj[k], xi[k] - xj[k], dist);
        float kv = ex2_approx(fmaf(-c1, dist, c0));
        if constexpr (MODE == kModeDLen) {
          const float dw = xi[a.which] - xj[a.which];
          kv *= dw * dw;
        }
        u = fmaf(kv, v[j], u);
      }
    }
    if (a.add_diag) u = fmaf((float)a.params->lambda, v[i], u);
    *out = u;
  }
}

// One CTA's work: row block rb, the j ranges sp .. sp + nsp - 1 (one unless MULTI), R columns.  Shared by
// the single-problem kernel and the batched one.
template <int DP, int N, int MODE, bool MULTI>
__device__ __forceinline__ void f3_body(const F3Args& a, const int rb, const int sp, const int nsp,
                                        const int R) {
  using S = F3Shape<DP, N>;
  constexpr int ST = S::ST;
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t smem0 = smem_u32(smem);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::OFF_BARS);
  uint64_t* k_full = full + ST;
  uint64_t* b_free = k_full + kF3Sets;
  uint64_t* u_full = b_free + kF3Sets;
  uint64_t* u_free = u_full + 2;
  uint64_t* done = u_free + 2;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* s_fail = reinterpret_cast<volatile int*>(s_tmem + 1);
  int* s_last = reinterpret_cast<int*>(s_tmem + 2);
  volatile int* s_nan = reinterpret_cast<volatile int*>(s_tmem + 3);   // a sum came out as NaN
  const uint32_t full0 = smem_u32(full), k_full0 = smem_u32(k_full), b_free0 = smem_u32(b_free),
                 u_full0 = smem_u32(u_full), u_free0 = smem_u32(u_free);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const long long slot = (long long)rb * a.nsplit + sp;   // the first range's partial-sum slot
  const long long row0 = (long long)rb * kF3BM;
  const int tile_begin = sp * a.tiles_per_split;
  const int nt = max(0, min(tile_begin + nsp * a.tiles_per_split, a.ntiles) - tile_begin);

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) mbar_init(&full[s], 1);
    for (int h = 0; h < kF3Sets; ++h) {
      mbar_init(&k_full[h], 4);
      mbar_init(&b_free[h], 1);
    }
    for (int u = 0; u < 2; ++u) {
      mbar_init(&u_full[u], 1);
      mbar_init(&u_free[u], 4);
    }
    mbar_init(done, 1);
    fence_barrier_init();
    *s_fail = 0;
    *s_nan = 0;
  }
  if (warp == 0) tc::tmem_alloc(s_tmem, kF3Cols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = __shfl_sync(0xffffffffu, *s_tmem, 0);
  int issued = 0;

  if (warp == 0) {
    // ------ copies and MMAs ------
    constexpr uint32_t idesc = tc::instr_desc(1, kF3BM, N);
    const uint64_t dV0 = tc::smem_desc(smem0 + S::X_BYTES, 128, 512);
    auto copy_tile = [&](int p, int s) {
      const long long t = tile_begin + p;
      unsigned char* st = smem + s * S::STAGE_BYTES;
      mbar_arrive_expect_tx(&full[s], S::STAGE_BYTES);
      bulk_g2s(st, a.xhat + t * kF3BN * DP, S::X_BYTES, &full[s]);
      bulk_g2s(st + S::X_BYTES, a.Vp + t * 3 * N * kF3BN, 3 * S::V_PART, &full[s]);
    };
    const int pre = min(ST, nt);
    if (tc::elect_one())
      for (int p = 0; p < pre; ++p) copy_tile(p, p);
    __syncwarp();
    issued = pre;
    bool ok = true;
    int s = 0, ph_s = 0, h = 0, ph_h = 0;
#pragma unroll 1
    for (int p = 0; p < nt; ++p) {
      const uint32_t ub = (uint32_t)(p & 1);
      ok = tc::warp_wait_uniform(full0 + 8u * s, ph_s) &&
           tc::warp_wait_uniform(k_full0 + 8u * h, ph_h) &&
           (p < 2 || tc::warp_wait_uniform(u_free0 + 8u * ub, (uint32_t)(((p >> 1) - 1) & 1)));
      if (!ok) break;
      tc::fence_after();
      if (tc::elect_one()) {
        const uint64_t dV = dV0 + (uint64_t)s * (S::STAGE_BYTES >> 4);
        const uint32_t kcol = tbase + (uint32_t)(48 * h), ucol = tbase + S::COL_U + 32u * ub;
        // (K part, V part), parts 0 high, 1 middle, 2 low
        constexpr int ka[6] = {2, 1, 0, 1, 0, 0}, vb[6] = {0, 1, 2, 0, 1, 0};
#pragma unroll
        for (int term = 0; term < 6; ++term)
#pragma unroll
          for (int ks = 0; ks < 2; ++ks)
            tc::mma_bf16_ts(ucol, kcol + 24u * ks + 8u * ka[term],
                            dV + (uint64_t)(vb[term] * (S::V_PART >> 4)) + 16u * ks, idesc,
                            (term | ks) != 0);
        tc::commit(&u_full[ub]);
        tc::commit(&b_free[h]);
      }
      __syncwarp();
      // the stage of the tile before takes tile p - 1 + ST once its MMAs are complete
      if (p >= 1 && p - 1 + ST < nt) {
        const int hp = h == 0 ? kF3Sets - 1 : h - 1, sp1 = s == 0 ? ST - 1 : s - 1;
        ok = tc::warp_wait_uniform(b_free0 + 8u * hp, (uint32_t)(((p - 1) / kF3Sets) & 1));
        if (!ok) break;
        if (tc::elect_one()) copy_tile(p - 1 + ST, sp1);
        __syncwarp();
        issued = p + ST;
      }
      if (++s == ST) { s = 0; ph_s ^= 1; }
      if (++h == kF3Sets) { h = 0; ph_h ^= 1; }
    }
    if (!ok) *s_fail = 1;
    if (tc::elect_one()) tc::commit(done);
    __syncwarp();
  } else if (warp < kF3Drain) {
    // ------ kernel values: a row per thread, the set's tiles whole, eight columns at a time ------
    const int eq = warp & 3;
    const int set = (warp - 1) >> 2;
    const long long i = row0 + eq * 32 + lane;
    const uint32_t kbase = tbase + ((uint32_t)(eq * 32) << 16) + (uint32_t)(48 * set);
    const float2 c0 = make_float2(a.params->c0f, a.params->c0f);
    const float2 nc1 = make_float2(-a.params->c1f, -a.params->c1f);
    const float2 minus1 = make_float2(-1.f, -1.f);
    float2 nx[DP / 2];   // -x^_i
#pragma unroll
    for (int k = 0; k < DP / 2; ++k) {
      const float2 x = i < a.n ? *reinterpret_cast<const float2*>(a.xhat + i * DP + 2 * k)
                               : make_float2(0.f, 0.f);
      nx[k] = make_float2(-x.x, -x.y);
    }
    const float xw = (MODE == kModeDLen && i < a.n) ? a.xhat[i * DP + a.which] : 0.f;
    bool ok = true;
    int s = set, ph_s = 0, ph = 1;   // ph: parity of the buffer's previous release
#pragma unroll 1
    for (int lt = set; lt < nt; lt += kF3Sets) {
      ok = tc::warp_wait_uniform(full0 + 8u * s, ph_s) &&
           (lt < kF3Sets || tc::warp_wait_uniform(b_free0 + 8u * set, ph));
      if (!ok) break;
      tc::fence_after();
      const float* tx = reinterpret_cast<const float*>(smem + s * S::STAGE_BYTES);
#pragma unroll 1
      for (int g = 0; g < 4; ++g) {
        uint32_t hi[4], mi[4], lo[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float* xj = tx + (8 * g + 2 * q) * DP;
          const float2 dist = make_float2(f3_dist<DP>(nx, xj), f3_dist<DP>(nx, xj + DP));
          const float2 e = __ffma2_rn(nc1, dist, c0);
          float2 k = make_float2(ex2_approx(e.x), ex2_approx(e.y));
          if constexpr (MODE == kModeDLen) {
            const float d0 = xw - xj[a.which], d1 = xw - xj[DP + a.which];
            k = __fmul2_rn(k, make_float2(d0 * d0, d1 * d1));
          }
          const __nv_bfloat162 h = __floats2bfloat162_rn(k.x, k.y);
          const float2 r1 = __ffma2_rn(__bfloat1622float2(h), minus1, k);
          const __nv_bfloat162 m = __floats2bfloat162_rn(r1.x, r1.y);
          const float2 r2 = __ffma2_rn(__bfloat1622float2(m), minus1, r1);
          const __nv_bfloat162 l = __floats2bfloat162_rn(r2.x, r2.y);
          hi[q] = f3_bits(h);
          mi[q] = f3_bits(m);
          lo[q] = f3_bits(l);
        }
        const uint32_t col = kbase + (uint32_t)((g >> 1) * 24 + (g & 1) * 4);
        tc::tmem_st4(col, hi);
        tc::tmem_st4(col + 8, mi);
        tc::tmem_st4(col + 16, lo);
      }
      tc::tmem_wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&k_full[set]);
      ph ^= 1;
      s += kF3Sets;
      if (s >= ST) { s -= ST; ph_s ^= 1; }
    }
    if (!ok) *s_fail = 1;
  } else {
    // ------ running sums: each tile's product, round to nearest ------
    const int eq = warp & 3;
    const int il = eq * 32 + lane;
    const long long i = row0 + il;
    const uint32_t ubase = tbase + ((uint32_t)(eq * 32) << 16) + S::COL_U;
    float2 acc[N / 2];
#pragma unroll
    for (int q = 0; q < N / 2; ++q) acc[q] = make_float2(0.f, 0.f);
    bool ok = true;
    auto put = [&](int range) {   // the CTA's range-th partial sums
      float* part = a.partials + (slot + range) * N * kF3BM + il;
#pragma unroll
      for (int r = 0; r < N; ++r) part[r * kF3BM] = r & 1 ? acc[r / 2].y : acc[r / 2].x;
    };
    int end = MULTI ? a.tiles_per_split : nt;   // of the current range
#pragma unroll 1
    for (int p = 0; p < nt; ++p) {
      const uint32_t ub = (uint32_t)(p & 1);
      ok = tc::warp_wait_uniform(u_full0 + 8u * ub, (uint32_t)((p >> 1) & 1));
      if (!ok) break;
      tc::fence_after();
#pragma unroll
      for (int c = 0; c < N / 16; ++c) {
        float v[16];
        tc::tmem_ld16(ubase + 32u * ub + 16u * c, v);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          acc[8 * c + q] = __fadd2_rn(acc[8 * c + q], make_float2(v[2 * q], v[2 * q + 1]));
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&u_free[ub]);
      if (MULTI && p + 1 == end && p + 1 < nt) {   // on to the next range
        put(p / a.tiles_per_split);
#pragma unroll
        for (int q = 0; q < N / 2; ++q) acc[q] = make_float2(0.f, 0.f);
        end += a.tiles_per_split;
      }
    }
    if (!ok) {
      *s_fail = 1;
    } else if (a.nsplit == 1) {
      if (i < a.n) {
        const float lam = a.add_diag ? (float)a.params->lambda : 0.f;
#pragma unroll
        for (int r = 0; r < N; ++r)
          if (r < R) {
            float u = r & 1 ? acc[r / 2].y : acc[r / 2].x;
            if (a.add_diag) u = fmaf(lam, a.V[(long long)a.vmap[r] * a.ldv + i], u);
            a.U[(long long)a.umap[r] * a.ldu + i] = u;
            if (isnan(u)) *s_nan = 1;
          }
      }
    } else {
      put(MULTI ? (nt - 1) / a.tiles_per_split : 0);
    }
  }

  // -------- all roles: release tensor memory; last CTA of the row block reduces --------
  if (warp == 0) (void)tc::warp_wait_uniform(smem_u32(done), 0);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, kF3Cols);
  if (*s_fail) {
    if (tid == 0) {
      atomicOr(a.status, kStatusTimeout);
      // let the copies still in flight land before the CTA's shared memory goes away
      for (int lt2 = max(0, issued - ST); lt2 < issued; ++lt2)
        (void)mbar_wait_bounded(&full[lt2 % ST], (uint32_t)((lt2 / ST) & 1));
    }
    return;
  }
  if (a.nsplit == 1) {
    if (*s_nan) f3_not_finite<N, MODE>(a, row0, R, s_tmem + 4);
    return;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) *s_last = (atomicAdd(&a.counters[rb], nsp) == a.nsplit - nsp);
  __syncthreads();
  if (!*s_last) return;
  __threadfence();
  const float* base = a.partials + (long long)rb * a.nsplit * N * kF3BM;
  const float lam = (float)a.params->lambda;
  for (int idx = tid; idx < R * kF3BM; idx += kF3Threads) {
    const int r = idx / kF3BM, il = idx - r * kF3BM;
    const long long i = row0 + il;
    if (i >= a.n) continue;
    float u = 0.f;
    for (int s2 = 0; s2 < a.nsplit; ++s2) u += __ldcg(base + ((long long)s2 * N + r) * kF3BM + il);
    if (a.add_diag) u = fmaf(lam, a.V[(long long)a.vmap[r] * a.ldv + i], u);
    a.U[(long long)a.umap[r] * a.ldu + i] = u;
    if (isnan(u)) *s_nan = 1;
  }
  if (tid == 0) a.counters[rb] = 0;
  __syncthreads();
  if (*s_nan) f3_not_finite<N, MODE>(a, row0, R, s_tmem + 4);
}

template <int DP, int N, int MODE>
__global__ void __launch_bounds__(kF3Threads, 2) kmv_f32_tc_kernel(const F3Args a) {
  const int rb = blockIdx.x / a.nsplit;
  f3_body<DP, N, MODE, false>(a, rb, blockIdx.x - rb * a.nsplit, 1, a.R);
}

// Many problems in one launch (mode K, padded d <= 8): CTA b takes work item items[b] = (problem,
// row block, first range, ranges) with that problem's arguments.
template <int N>
__global__ void __launch_bounds__(kF3Threads, 2) kmv_f32_tc_batch_kernel(
    const F3Args* __restrict__ args, const int4* __restrict__ items) {
  __shared__ F3Args s_a;
  const int4 it = items[blockIdx.x];
  if (threadIdx.x == 0) s_a = args[it.x];
  __syncthreads();
  const int R = s_a.R_dev ? *s_a.R_dev : s_a.R;
  if (!batch_tc_columns(s_a.n, R)) return;
  switch (s_a.DP) {
    case 2: f3_body<2, N, kModeK, true>(s_a, it.y, it.z, it.w, R); break;
    case 4: f3_body<4, N, kModeK, true>(s_a, it.y, it.z, it.w, R); break;
    default: f3_body<8, N, kModeK, true>(s_a, it.y, it.z, it.w, R); break;
  }
}

template <int DP, int N, int MODE>
cudaError_t f3_launch(KmvLaunch& L, cudaStream_t s) {
  using S = F3Shape<DP, N>;
  KmvPlan p{};
  p.n_rb = (int)((L.n + kF3BM - 1) / kF3BM);
  p.nsplit = f3_nsplit(L.n, L.num_sms);
  const long long ntiles = (L.n + kF3BN - 1) / kF3BN;
  const size_t pbytes = p.nsplit > 1 ? (size_t)p.n_rb * p.nsplit * N * kF3BM * 4 : 0;
  L.planned_nsplit = p.nsplit;
  if (L.plan_only) {
    L.need_partials_bytes = pbytes;
    L.need_counters = p.nsplit > 1 ? p.n_rb : 0;
    return cudaSuccess;
  }
  if (pbytes > L.partials_bytes || (p.nsplit > 1 && p.n_rb > L.counters_len)) {
    L.need_partials_bytes = pbytes;
    L.need_counters = p.n_rb;
    return cudaErrorMemoryAllocation;
  }
  auto fn = kmv_f32_tc_kernel<DP, N, MODE>;
  static std::once_flag once;
  std::call_once(once, [&] {
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  });
  __nv_bfloat16* Vp = static_cast<__nv_bfloat16*>(L.v3);
  if (!L.v_packed) {
    const long long total = ntiles * N * kF3BN;
    const int blocks = (int)std::min<long long>((total + 255) / 256, 8LL * L.num_sms);
    pack_v3_kernel<<<blocks, 256, 0, s>>>(static_cast<const float*>(L.V), L.ldv, L.vmap, L.R, N,
                                          L.n, ntiles, Vp);
  }
  F3Args a;
  a.xhat = static_cast<const float*>(L.xhat);
  a.Vp = Vp;
  a.V = static_cast<const float*>(L.V);
  a.ldv = L.ldv;
  a.vmap = L.vmap;
  a.R = L.R;
  a.R_dev = nullptr;
  a.U = static_cast<float*>(L.U);
  a.ldu = L.ldu;
  a.umap = L.umap;
  a.n = L.n;
  a.DP = DP;
  a.params = L.params;
  a.which = L.which;
  a.add_diag = L.mode == kModeK;
  a.tiles_per_split = (int)((ntiles + p.nsplit - 1) / p.nsplit);
  a.nsplit = p.nsplit;
  a.ntiles = (int)ntiles;
  a.partials = static_cast<float*>(L.partials);
  a.counters = L.counters;
  a.status = L.status;
  L.launches = L.v_packed ? 1 : 2;
  fn<<<p.n_rb * a.nsplit, kF3Threads, S::SMEM, s>>>(a);
  return cudaGetLastError();
}

template <int DP>
cudaError_t f3_dp(KmvLaunch& L, cudaStream_t s) {
  if (L.mode == kModeDLen)
    return L.R <= 16 ? f3_launch<DP, 16, kModeDLen>(L, s) : f3_launch<DP, 32, kModeDLen>(L, s);
  return L.R <= 16 ? f3_launch<DP, 16, kModeK>(L, s) : f3_launch<DP, 32, kModeK>(L, s);
}

}  // namespace

// The time here does not depend on the column count up to 32; the SIMT kernel's grows with it.
// Calls, SIMT / here, us (SIMT with two rows per thread, its default):
//   d = 8, n = 1,030: 1 column 18 / 19, 5 columns 26 / 21, 17 columns 51 / 23; n = 9,937: 3 columns
//   101 / 114, 5 columns 113 / 115, 17 columns 208 / 121, 32 columns 325 / 128; n = 50,000: 6 columns
//   2,200 / 2,295, 7 columns 2,494 / 2,296, 32 columns 5,223 / 2,275.
// By padded width, 5 columns at n = 8,000: d = 2 68 / 60, 4 78 / 65, 8 87 / 81, 16 125 / 116; 7 columns at
// n = 10,100: 100 / 83, 118 / 92, 151 / 120, 199 / 175; at 31,000: 609 / 536, 712 / 630, 1,016 / 880,
// 1,508 / 1,329; at 64,000: 2,285 / 2,210, 2,836 / 2,620, 3,989 / 3,701, 6,117 / 5,606; at 120,000: 7,680 /
// 7,611, 10,137 / 9,085, 14,011 / 12,911, 22,269 / 19,606.  So one line for all widths; what it loses
// most is 7 and 8 columns at d <= 2, n = 35,000, 725 / 773 (one wave of CTAs, nine tenths full; 3% at
// most for the other widths there), and 4% at d <= 2, n = 75,000.
// (Error against 64 bits, relative: 1.7e-7 / 1.3e-7 at n = 1,030, 8.5e-7 / 2.8e-7 at n = 22,784, 17
// columns.)
bool kmv_f32_tc_applies(const KmvLaunch& L) {
  return L.v3 && L.mode != kModeDLam && !L.simt && f32_tc_columns(L.n, L.R);
}

cudaError_t launch_kmv_f32_tc(KmvLaunch& L, cudaStream_t s) {
  switch (L.DP) {
    case 2: return f3_dp<2>(L, s);
    case 4: return f3_dp<4>(L, s);
    case 8: return f3_dp<8>(L, s);
    case 16: return f3_dp<16>(L, s);
    default: return cudaErrorInvalidValue;
  }
}

// ---------------------------------------------------------------------------------------
// Batched launches.
// ---------------------------------------------------------------------------------------
size_t f3_batch_args_bytes(int B) { return sizeof(F3Args) * (size_t)B; }

cudaError_t f3_batch_upload_args(const F3Problem* P, int B, void* args_dev, cudaStream_t s) {
  std::vector<F3Args> h((size_t)B);
  for (int b = 0; b < B; ++b) {
    const F3Problem& q = P[b];
    F3Args& a = h[b];
    const BatchKmvDesc& k = q.k;
    a.xhat = k.xhat;
    a.Vp = static_cast<const __nv_bfloat16*>(q.v3);
    a.V = k.V;
    a.ldv = k.ldv;
    a.vmap = k.vmap;
    a.R = 0;
    a.R_dev = k.nlive;
    a.U = k.U;
    a.ldu = k.ldu;
    a.umap = k.umap;
    a.n = k.n;
    a.DP = k.DP;
    a.params = k.params;
    a.which = -1;
    a.add_diag = 1;
    a.ntiles = (int)((k.n + kF3BN - 1) / kF3BN);
    a.tiles_per_split = (a.ntiles + q.nsplit - 1) / q.nsplit;
    a.nsplit = (a.ntiles + a.tiles_per_split - 1) / a.tiles_per_split;
    if (a.nsplit != q.nsplit || k.DP > 8) return cudaErrorInvalidValue;
    a.partials = q.partials;
    a.counters = q.counters;
    a.status = q.status;
  }
  return cudaMemcpyAsync(args_dev, h.data(), sizeof(F3Args) * (size_t)B, cudaMemcpyHostToDevice, s);
}

template <int N>
static cudaError_t f3_batch_launch(const F3Args* args, int B, const int4* items, int n_items,
                                   bool prime_only, cudaStream_t s) {
  static std::once_flag once;
  std::call_once(once, [] {
    auto fn = kmv_f32_tc_batch_kernel<N>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F3Shape<8, N>::SMEM);
    cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  });
  if (prime_only) return cudaSuccess;
  pack_v3_batch_kernel<<<dim3(64, (unsigned)B), 256, 0, s>>>(args, N);
  if (n_items > 0)
    kmv_f32_tc_batch_kernel<N><<<n_items, kF3Threads, F3Shape<8, N>::SMEM, s>>>(args, items);
  return cudaGetLastError();
}

cudaError_t launch_kmv_f32_tc_batch(const void* args_dev, int B, const int4* items, int n_items,
                                    int R_max, cudaStream_t s, bool prime_only) {
  const F3Args* args = static_cast<const F3Args*>(args_dev);
  if (prime_only) {
    f3_batch_launch<16>(args, B, items, n_items, true, s);
    return f3_batch_launch<32>(args, B, items, n_items, true, s);
  }
  if (R_max > 32) return cudaErrorInvalidValue;
  return R_max <= 16 ? f3_batch_launch<16>(args, B, items, n_items, false, s)
                     : f3_batch_launch<32>(args, B, items, n_items, false, s);
}

}  // namespace ulisse
