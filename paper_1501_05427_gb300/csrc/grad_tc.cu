// Mixed-precision fused gradient pass on the 5th-generation tensor cores (Eq. gradient:unbiased,
// Sec. 4.1): the components of
//     g~_i = sum_m a_m^T dK_i b_m
// for all parameters at once, through W_ij = sum_m a_m[i] b_m[j] and P_ij = k_s(i,j) W_ij:
//     g~_{log l_k}     = sum_ij P_ij (x^_ik - x^_jk)^2
//     g~_{log sigma^2} = sum_ij P_ij
//     g~_{log lambda}  = lambda sum_i W_ii.
// Both double sums weigh the pair (i, j) by a symmetric function (k_s and the squared
// difference), so they take each unordered pair once with the symmetric weight
//     W'_ij = W_ij + W_ji = [A^_i | b_i] . [b_j | A^_j]     (A^ = the scaled a-columns),
// a product over 2M factors: the pass visits, for the block of 128 rows I, only the 32-point
// tiles J at or after the block's own points (J >= I), with weight 1/2 on the four tiles of
// I itself (there both (i, j) and (j, i) are visited).  With P'_ij = k_s(i,j) W'_ij on the
// visited pairs,
//     g~_{log l_k}     = sum_i [ x^_ik^2 S_i - 2 x^_ik G_ik + H_ik ],
//                        S_i = sum_j P'_ij,  G_ik = sum_j P'_ij x^_jk,  H_ik = sum_j P'_ij x^_jk^2
//     g~_{log sigma^2} = sum_i S_i,
// so half the kernel values of the full square are formed.  Nothing is written per point j,
// which is why the symmetry is free here (a K V product would have to add K_IJ^T V_I to the
// rows of J).  For a block of 128 rows I and each visited 32-point tile J:
//   1. W'_IJ = [A^ | B]_I [B | A^]_J^T on the tensor cores (K = 2M factors, both operands
//      split into BF16 high + low parts: three products), into tensor memory;
//   2. for padded d <= 8, C_IJ = A_I B_J^T on the tensor cores as in the K V pass (the TF32
//      row images A_j = x^_j, B_j = 2 c1 x^_j, three TF32 products) into its own tensor-memory
//      buffer; the epilogue warps read W and C back (tcgen05.ld), form the kernel values as the
//      K V kernel does (exponent (a_i + b_j) + C_ij from the row norms, one ex2; for d = 16
//      the cross term on the FP32 pipe), multiply, split P into BF16 high + low parts and
//      store them over W's own tensor-memory columns;
//   3. [S | G | H]_I += P_IJ Z_J on the tensor cores, Z_j = [x^_j, x^_j^2, 1] split the same
//      way, accumulated in tensor memory across all tiles of the CTA's j range.
// The per-row combination and the diagonal sum run in FP64 at the end; CTA partials are summed
// in a fixed order by the last CTA to arrive (as in the SIMT gradient kernel).  The left operands
// [A^ | B]_I and A_I lie in tensor memory (in shared memory where 128 factor slots leave no room).
// Roles: three issuing warps, one per stream of MMAs (warp 0: C; warp 1: W; warp 2: P Z and the
// copies of B_J's TF32 image with b_J, or x^_J and b_J for d = 16, then B^_J and Z_J as one block,
// into a ring of 4 to 8 stages), their loops warp-uniform with a lane elected for the issuing
// instructions; twelve epilogue warps (eight for d = 16) make P in sets of four (one warp per
// tensor-memory lane quadrant): set h takes the tiles h, h + 3, ... whole and owns the W/P buffer
// h, so that each wait and hand-off covers 32 entries per thread; C has two buffers (one with 64
// factor slots), given back as soon as they are read.  A W/P buffer is refilled, and the tile's
// stage, only after the MMAs that read P have completed.  Every wait is bounded.
//
// What bounds it: the epilogue's issue slots and the chain W, C -> epilogue -> P Z -> refill of
// each set.  n = 50,000, d = 8, M = 17 (kernel alone): 1.224 ms with eight epilogue warps that
// shared every tile by column halves behind one C buffer and one divergent issuing lane (three
// CTAs per SM); 0.976 ms with the sets and one uniform issuing warp (two CTAs of 256
// tensor-memory columns); 0.64 ms with the left operands in tensor memory (an MMA with A in shared
// memory takes 40 clocks, 16 otherwise) and an issuing warp per stream.
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "kmv_kernel.cuh"
#include "tc_common.cuh"

namespace ulisse {

constexpr int kGtBN = 32;
constexpr int kGtBM = 128;
constexpr int kGtIssuers = 3;      // warps 0-2: C; W; P Z and the copies
constexpr uint32_t kGtCols = 256;  // tensor-memory columns per CTA (two CTAs per SM)
static_assert(16 * 8 + 48 <= kGtScratchRows, "operand images exceed the gradient scratch");

__device__ inline void split_bf16(float v, __nv_bfloat16& h, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(v);
  l = __float2bfloat16_rn(v - __bfloat162float(h));
}

// One element of a tile's operand block: [b_j | A^_j] as a K-major canonical image of 32 points
// (rows) x K1 factor slots (slot m < M holding b_m[j], slot M + m holding sa[m] a_m[j], slots
// >= 2M zero), then Z_j = [x^_j (DP), x^_j^2 (DP), 1, 0...] as an image of N2 rows (accumulator
// columns) x 32 points; each as BF16 high part and low part, the four parts back to back, so
// that a tile is one bulk copy.  Points j >= n are zero.
__device__ inline void gt_pack_element(long long idx, int K1, int N2, int DP, int M, long long n,
                                       const float* __restrict__ xhat, const float* __restrict__ A,
                                       const int* __restrict__ amap, const float* __restrict__ sa,
                                       const float* __restrict__ B, const int* __restrict__ bmap,
                                       long long ld, __nv_bfloat16* __restrict__ tiles) {
  const int per_b = kGtBN * K1, per_z = N2 * kGtBN, per = per_b + per_z;
  const long long t = idx / per;
  const int rem = (int)(idx - t * per);
  const int j = rem % kGtBN;
  const long long jj = t * kGtBN + j;
  float v = 0.f;
  uint32_t off, part;
  if (rem < per_b) {
    const int m = rem / kGtBN;
    if (jj < n) {
      if (m < M) v = B[(long long)bmap[m] * ld + jj];
      else if (m < 2 * M) v = sa[m - M] * A[(long long)amap[m - M] * ld + jj];
    }
    off = tc::canon_offset(j, m, 2, K1 / 8) / 2;
    part = (uint32_t)per_b;
  } else {
    const int c = (rem - per_b) / kGtBN;
    if (jj < n) {
      if (c < DP) {
        v = xhat[jj * DP + c];
      } else if (c < 2 * DP) {
        const float x = xhat[jj * DP + (c - DP)];
        v = x * x;
      } else if (c == 2 * DP) {
        v = 1.f;
      }
    }
    off = 2u * per_b + tc::canon_offset(c, j, 2, kGtBN / 8) / 2;
    part = (uint32_t)per_z;
  }
  __nv_bfloat16 h, l;
  split_bf16(v, h, l);
  __nv_bfloat16* o = tiles + t * (2LL * per) + off;
  o[0] = h;
  o[part] = l;
}

__global__ void pack_gt_kernel(int K1, int N2, int DP, int M, long long n, long long ntiles,
                               const float* __restrict__ xhat, const float* __restrict__ A,
                               const int* __restrict__ amap, const float* __restrict__ sa,
                               const float* __restrict__ B, const int* __restrict__ bmap,
                               long long ld, __nv_bfloat16* __restrict__ tiles) {
  const long long total = ntiles * kGtBN * (K1 + N2);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x)
    gt_pack_element(idx, K1, N2, DP, M, n, xhat, A, amap, sa, B, bmap, ld, tiles);
}

struct GtDevArgs {
  const float* xhat;   // x^ rows (ld x DP, row-major)
  const float* bneg;   // -c1 |x^|^2
  const __nv_bfloat16* tiles;   // per tile B^ high | low, Z high | low (gt_pack_element)
  const float* A;      // left factors: column amap[m], scaled by sa[m]
  const int* amap;
  const float* sa;
  const float* B;      // right factors (the diagonal term reads them unsplit)
  const int* bmap;
  long long ld;
  int M;
  long long n;
  int d;
  const DevParams* params;
  int nsplit, ntiles;
  int n_cta;           // CTAs of this problem (row blocks x nsplit): the last one reduces
  // padded d <= 8: the TF32 row images of the tensor-core K V pass (8 columns, 32-row
  // K-major canonical tiles; high part and remainder), A_j = [x^_j, 1?] and
  // B_j = [2 c1 x^_j, b_j?]; c_has_bj when the augmented column carries b_j
  const float* XA_hi;
  const float* XA_lo;
  const float* XB;     // tiles of B_J: high part | remainder | b_J (tc2_b_stride floats)
  int c_has_bj;
  double* partials;
  int* counter;
  double* g_out;
  int* status;
};

// XC (padded d <= 8): the exponent's cross term C = A_I B_J^T on the tensor cores from the
// TF32 row images (three TF32 products, as the K V pass); the stage carries B_J's image instead
// of x^_J.  Padded d = 16 keeps the FP32 cross term.
template <int DP, int KS>
struct GtShape {
  static constexpr bool XC = DP <= 8;
  // epilogue sets of four warps: three; two for padded d = 16, whose cross term needs registers
  static constexpr int SETS = XC ? 3 : 2;
  static constexpr int THREADS = 32 * (kGtIssuers + 4 * SETS);
  // the left operands [A^ | B]_I and A_I in tensor memory (128 factor slots leave no room: then
  // they stay in shared memory)
  static constexpr bool TS = KS <= 4;
  static constexpr int K1 = 16 * KS;                   // factor slots (2M), padded
  static constexpr int N2 = (2 * DP + 1 + 15) / 16 * 16;
  static constexpr int K8 = 8;                         // columns of the TF32 row images
  static constexpr uint32_t A_BYTES = TS ? 0 : kGtBM * K1 * 2;           // one part of A^_I
  static constexpr uint32_t XA_BYTES = XC && !TS ? kGtBM * K8 * 4 : 0;   // one part of A_I (TF32)
  static constexpr uint32_t X_BYTES = XC ? 2 * kGtBN * K8 * 4 : kGtBN * DP * 4;
  static constexpr uint32_t XB_BYTES = kGtBN * K8 * 4;  // one part of B_J (TF32)
  static constexpr uint32_t BN_BYTES = kGtBN * 4;
  static constexpr uint32_t BT_BYTES = kGtBN * K1 * 2;
  static constexpr uint32_t Z_BYTES = N2 * kGtBN * 2;
  static constexpr uint32_t TILE_BYTES = 2 * BT_BYTES + 2 * Z_BYTES;   // the packed block
  // stage: x^_J (FP32) or B_J (TF32 high | remainder), b_J, B^_J high | low, Z_J high | low
  static constexpr uint32_t OFF_BN = X_BYTES;
  static constexpr uint32_t OFF_BT = OFF_BN + BN_BYTES;
  static constexpr uint32_t OFF_Z = OFF_BT + 2 * BT_BYTES;
  static constexpr uint32_t STAGE_BYTES = OFF_Z + 2 * Z_BYTES;
  // C buffers: two while they fit beside the left operands, else one
  static constexpr int NC = !XC ? 0 : KS == 4 ? 1 : 2;
  // c_full per tile mod 6: each barrier then serves one set, whose waits visit its phases in
  // order whatever the number of buffers
  static constexpr int NCF = 2 * SETS;
  // w_full, p_full, b_free per set; c_full; c_free per buffer; done
  static constexpr int NBARS_FIXED = 3 * SETS + NCF + 2 + 1;
  static constexpr uint32_t FIXED = 2 * A_BYTES + 2 * XA_BYTES + (8 + NBARS_FIXED) * 8 + 64;
  // as many stages (3 to 8) as let two CTAs share the SM's 228 KB, else as fit one
  static constexpr int fit(uint32_t budget) { return (int)((budget - FIXED) / STAGE_BYTES); }
  static constexpr uint32_t kHalfSm = 108u * 1024u, kWholeSm = 220u * 1024u;
  static constexpr int ST_HALF = FIXED < kHalfSm ? fit(kHalfSm) : 0;
  static constexpr int OCC = ST_HALF > SETS ? 2 : 1;   // CTAs per SM
  static constexpr int ST_ANY = OCC == 2 ? ST_HALF : fit(kWholeSm);
  static constexpr int ST = ST_ANY > 8 ? 8 : ST_ANY;
  static_assert(ST > SETS, "a stage beyond those in flight");
  static constexpr uint32_t OFF_XA = 2 * A_BYTES;
  static constexpr uint32_t OFF_STAGES = OFF_XA + 2 * XA_BYTES;
  static constexpr uint32_t OFF_BARS = OFF_STAGES + ST * STAGE_BYTES;
  static constexpr int NBARS = ST + NBARS_FIXED;    // full per stage, then the fixed ones
  static constexpr uint32_t SMEM = OFF_BARS + NBARS * 8 + 64;
  // tensor-memory columns: the sets' W/P buffers of 32, the C buffers of 32, the [G | H | S]
  // accumulator, then the left operands' high and low parts
  static constexpr uint32_t COL_C = 32 * SETS;
  static constexpr uint32_t COL_D2 = COL_C + 32 * NC;
  static constexpr uint32_t COL_A = COL_D2 + N2;             // two BF16 per column
  static constexpr uint32_t COL_XA = COL_A + (TS ? K1 : 0);
  static_assert(COL_XA + (TS && XC ? 2 * K8 : 0) <= kGtCols, "tensor memory layout exceeds the allocation");
  static_assert(X_BYTES % 16 == 0 && STAGE_BYTES % 16 == 0 && A_BYTES % 16 == 0 &&
                    OFF_BT % 16 == 0 && OFF_Z % 16 == 0 && OFF_STAGES % 16 == 0,
                "bulk copies and descriptors need 16-byte alignment");
};

// Two 16-column tensor-memory loads at independent addresses and one wait.
__device__ inline void gt_tmem_ld16_two(uint32_t ta, uint32_t tb, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,"
      "%27,%28,%29,%30,%31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(ta), "r"(tb)
      : "memory");
}

// One CTA's work: row block rb, split sp of its tile range.  Shared by the single-problem
// kernel and the batched one.
template <int DP, int KS>
__device__ __forceinline__ void gt_body(const GtDevArgs& a, const int rb, const int sp) {
  using S = GtShape<DP, KS>;
  constexpr int ST = S::ST, K1 = S::K1, N2 = S::N2, SETS = S::SETS;
  constexpr int NACC = DP + 2;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ double s_red[4][NACC];
  unsigned char* sAh = smem;
  unsigned char* sAl = smem + S::A_BYTES;
  const uint32_t smem0 = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::OFF_BARS);
  uint64_t* full = bars;
  uint64_t* w_full = bars + ST;            // W of the set's tile formed (MMA commit)
  uint64_t* p_full = w_full + SETS;     // P written by the set's four warps
  uint64_t* b_free = p_full + SETS;     // P Z of the set's tile done (MMA commit)
  uint64_t* c_full = b_free + SETS;     // C of the tile formed (MMA commit), tile mod NCF
  uint64_t* c_free = c_full + S::NCF;      // C read by the set's four warps, per buffer
  uint64_t* done = c_free + 2;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + S::OFF_BARS + S::NBARS * 8);
  volatile int* s_fail = reinterpret_cast<volatile int*>(s_tmem + 1);
  int* s_last = reinterpret_cast<int*>(s_tmem + 2);
  const uint32_t full0 = smem_u32(full), w_full0 = smem_u32(w_full), p_full0 = smem_u32(p_full),
                 b_free0 = smem_u32(b_free), c_full0 = smem_u32(c_full), c_free0 = smem_u32(c_free);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler
  // Row block rb visits the tiles [4 rb, ntiles) (its own four tiles, then every later
  // one), cut into nsplit equal ranges; CTAs start in row-block order, longest ranges first.
  constexpr int kTilesPerBlock = kGtBM / kGtBN;
  const long long slot = (long long)rb * a.nsplit + sp;   // this CTA's partial-sum slot
  const long long row0 = (long long)rb * kGtBM;
  const int diag_end = min(kTilesPerBlock * (rb + 1), a.ntiles);   // tiles of I itself
  const int span = a.ntiles - kTilesPerBlock * rb;
  const int per = (span + a.nsplit - 1) / a.nsplit;
  const int tile_begin = kTilesPerBlock * rb + sp * per;
  const int nt = max(0, min(tile_begin + per, a.ntiles) - tile_begin);

  // [A^_I | B_I]: slot m < M holds sa[m] a_m[i], slot M + m holds b_m[i]; split into BF16
  // high and low parts
  auto left = [&](int m, long long i) -> float {
    if (i >= a.n) return 0.f;
    if (m < a.M) return a.sa[m] * a.A[(long long)a.amap[m] * a.ld + i];
    return m < 2 * a.M ? a.B[(long long)a.bmap[m - a.M] * a.ld + i] : 0.f;
  };
  if constexpr (!S::TS) {   // K-major canonical images in shared memory
    for (int idx = tid; idx < kGtBM * K1; idx += S::THREADS) {
      const int m = idx / kGtBM, il = idx - m * kGtBM;
      __nv_bfloat16 h, l;
      split_bf16(left(m, row0 + il), h, l);
      const uint32_t off = tc::canon_offset(il, m, 2, K1 / 8);
      *reinterpret_cast<__nv_bfloat16*>(sAh + off) = h;
      *reinterpret_cast<__nv_bfloat16*>(sAl + off) = l;
    }
    if constexpr (S::XC) {
      // A_I's TF32 image (high part, then remainder): 128 rows of the packed images, which
      // are zero beyond n
      constexpr int kQ = kGtBM * S::K8 / 4;   // float4 per part
      float4* sx = reinterpret_cast<float4*>(smem + S::OFF_XA);
      const float4* gh = reinterpret_cast<const float4*>(a.XA_hi + row0 * S::K8);
      const float4* gl = reinterpret_cast<const float4*>(a.XA_lo + row0 * S::K8);
      for (int idx = tid; idx < 2 * kQ; idx += S::THREADS)
        sx[idx] = idx < kQ ? gh[idx] : gl[idx - kQ];
    }
    tc::fence_async_smem();
  }
  if (tid == 0) {
    for (int s = 0; s < ST; ++s) mbar_init(&full[s], 1);
    for (int h = 0; h < SETS; ++h) {
      mbar_init(&w_full[h], 1);
      mbar_init(&p_full[h], 4);
      mbar_init(&b_free[h], 1);
    }
    for (int c = 0; c < S::NCF; ++c) mbar_init(&c_full[c], 1);
    for (int c = 0; c < 2; ++c) mbar_init(&c_free[c], 4);
    mbar_init(done, 1);
    fence_barrier_init();
    *s_fail = 0;
  }
  if (warp == 0) tc::tmem_alloc(s_tmem, kGtCols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = __shfl_sync(0xffffffffu, *s_tmem, 0);
  if (S::TS && warp >= kGtIssuers && warp < kGtIssuers + 4) {
    // the left operands into tensor memory, a row per thread (an MMA whose A comes from shared
    // memory takes 40 clocks for its 4 KB, from tensor memory 16)
    const int eq = warp & 3;
    const long long i = row0 + eq * 32 + lane;
    const uint32_t dst = tbase + ((uint32_t)(eq * 32) << 16);
#pragma unroll 1
    for (int ks = 0; ks < KS; ++ks) {
      uint32_t hi[8], lo[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float v0 = left(16 * ks + 2 * q, i), v1 = left(16 * ks + 2 * q + 1, i);
        const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
        const float2 hf = __bfloat1622float2(h);
        const __nv_bfloat162 l = __floats2bfloat162_rn(v0 - hf.x, v1 - hf.y);
        hi[q] = *reinterpret_cast<const uint32_t*>(&h);
        lo[q] = *reinterpret_cast<const uint32_t*>(&l);
      }
      tc::tmem_st8(dst + S::COL_A + 8u * ks, hi);
      tc::tmem_st8(dst + S::COL_A + (uint32_t)(K1 / 2) + 8u * ks, lo);
    }
    if constexpr (S::XC) {
      const long long off =
          (i / 32) * 32 * S::K8 + tc::canon_offset((int)(i % 32), 0, 4, S::K8 / 4) / 4;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        const float* src = (part == 0 ? a.XA_hi : a.XA_lo) + off;
        const uint4 x = *reinterpret_cast<const uint4*>(src);
        const uint4 y = *reinterpret_cast<const uint4*>(src + 32);
        const uint32_t v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        tc::tmem_st8(dst + S::COL_XA + (uint32_t)(part * S::K8), v);
      }
    }
    tc::tmem_wait_st();
  }
  if constexpr (S::TS) {
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
  }
  int issued = 0;   // tiles whose copies were started (warp 2)

  double acc[NACC];
#pragma unroll
  for (int k = 0; k < NACC; ++k) acc[k] = 0.0;

  // Three issuing warps, so that no stream of MMAs and waits holds up another: the loops run
  // warp-uniformly, one elected lane issues.
  if (warp == 0) {
    // ------ C_J = A_I B_J^T (three TF32 products, K = 8) ------
    if constexpr (S::XC) {
      constexpr uint32_t idesc_c = tc::instr_desc(2, kGtBM, kGtBN);   // TF32
      constexpr uint32_t sbo_x = (S::K8 / 4) * 128;
      const uint64_t dXA0 = tc::smem_desc(smem0 + S::OFF_XA, 128, sbo_x);
      const uint64_t dXB0 = tc::smem_desc(smem0 + S::OFF_STAGES, 128, sbo_x);
      bool ok = true;
      int s = 0, ph_s = 0, c = 0, ph_c = 1, cf = 0;   // ph_c: parity of the buffer's last release
#pragma unroll 1
      for (int p = 0; p < nt; ++p) {
        ok = tc::warp_wait_uniform(full0 + 8u * s, ph_s) &&
             (p < S::NC || tc::warp_wait_uniform(c_free0 + 8u * c, ph_c));
        if (!ok) break;
        tc::fence_after();
        if (tc::elect_one()) {
          const uint64_t so = (uint64_t)s * (S::STAGE_BYTES >> 4);
          const uint32_t dC = tbase + S::COL_C + (uint32_t)(c * 32);
#pragma unroll
          for (int term = 0; term < 3; ++term) {
            const uint64_t B = dXB0 + so + (term == 1 ? (S::XB_BYTES >> 4) : 0u);
            if constexpr (S::TS)
              tc::mma_tf32_ts(dC, tbase + S::COL_XA + (term == 2 ? (uint32_t)S::K8 : 0u), B, idesc_c,
                              term != 0);
            else
              tc::mma_tf32(dC, dXA0 + (term == 2 ? (S::XA_BYTES >> 4) : 0u), B, idesc_c, term != 0);
          }
          tc::commit(&c_full[cf]);
        }
        __syncwarp();
        if (++s == ST) { s = 0; ph_s ^= 1; }
        if (++c == S::NC) { c = 0; ph_c ^= 1; }
        if (++cf == S::NCF) cf = 0;
      }
      if (!ok) *s_fail = 1;
    }
  } else if (warp == 1) {
    // ------ W = A^ B^T ------
    constexpr uint32_t idesc_w = tc::instr_desc(1, kGtBM, kGtBN);
    constexpr uint32_t sbo_k1 = (K1 / 8) * 128;
    const uint64_t dA0 = tc::smem_desc(smem0, 128, sbo_k1);
    const uint64_t dBT0 = tc::smem_desc(smem0 + S::OFF_STAGES + S::OFF_BT, 128, sbo_k1);
    bool ok = true;
    int s = 0, ph_s = 0, h = 0, ph_h = 1;   // ph_h: parity of the buffer's last release
#pragma unroll 1
    for (int p = 0; p < nt; ++p) {
      ok = tc::warp_wait_uniform(full0 + 8u * s, ph_s) &&
           (p < SETS || tc::warp_wait_uniform(b_free0 + 8u * h, ph_h));
      if (!ok) break;
      tc::fence_after();
      if (tc::elect_one()) {
        const uint64_t dBT = dBT0 + (uint64_t)s * (S::STAGE_BYTES >> 4);
        const uint32_t dW = tbase + (uint32_t)(h * 32);
#pragma unroll
        for (int term = 0; term < 3; ++term) {
          const uint64_t B = dBT + (term == 1 ? (S::BT_BYTES >> 4) : 0u);
#pragma unroll
          for (int ks = 0; ks < KS; ++ks) {
            if constexpr (S::TS)
              tc::mma_bf16_ts(dW, tbase + S::COL_A + (term == 2 ? (uint32_t)(K1 / 2) : 0u) + 8u * ks,
                              B + 16u * ks, idesc_w, (term | ks) != 0);
            else
              tc::mma_bf16(dW, dA0 + (term == 2 ? (S::A_BYTES >> 4) : 0u) + 16u * ks, B + 16u * ks,
                           idesc_w, (term | ks) != 0);
          }
        }
        tc::commit(&w_full[h]);
      }
      __syncwarp();
      if (++s == ST) { s = 0; ph_s ^= 1; }
      if (++h == SETS) { h = 0; ph_h ^= 1; }
    }
    if (!ok) *s_fail = 1;
  } else if (warp == 2) {
    // ------ [G | H | S] += P Z, and the copies: a stage is refilled once its tile's P Z, the
    //        last to read it, is complete (looked at one tile late, when it is) ------
    constexpr uint32_t idesc_g = tc::instr_desc(1, kGtBM, N2);
    const uint64_t dZ0 = tc::smem_desc(smem0 + S::OFF_STAGES + S::OFF_Z, 128, 512);
    auto copy_tile = [&](int p, int s) {   // elected lane
      const long long t = tile_begin + p;
      unsigned char* st = smem + S::OFF_STAGES + s * S::STAGE_BYTES;
      mbar_arrive_expect_tx(&full[s], S::STAGE_BYTES);
      if constexpr (S::XC) {
        bulk_g2s(st, a.XB + t * tc2_b_stride(S::K8), S::X_BYTES + S::BN_BYTES, &full[s]);
      } else {
        bulk_g2s(st, a.xhat + t * kGtBN * DP, S::X_BYTES, &full[s]);
        bulk_g2s(st + S::OFF_BN, a.bneg + t * kGtBN, S::BN_BYTES, &full[s]);
      }
      bulk_g2s(st + S::OFF_BT, a.tiles + t * (S::TILE_BYTES / 2), S::TILE_BYTES, &full[s]);
    };
    const int pre = min(ST, nt);
    if (tc::elect_one())
      for (int p = 0; p < pre; ++p) copy_tile(p, p);
    __syncwarp();
    issued = pre;
    bool ok = true;
    int s = 0, h = 0, ph_h = 0;
#pragma unroll 1
    for (int p = 0; p < nt; ++p) {
      ok = tc::warp_wait_uniform(p_full0 + 8u * h, ph_h);
      if (!ok) break;
      tc::fence_after();
      if (tc::elect_one()) {
        const uint64_t dZ = dZ0 + (uint64_t)s * (S::STAGE_BYTES >> 4);
        const uint32_t pcol = tbase + (uint32_t)(h * 32);
#pragma unroll
        for (int term = 0; term < 3; ++term) {
          const uint32_t A = pcol + (term == 2 ? 8u : 0u);   // P high | P low per 16 points
          const uint64_t B = dZ + (term == 1 ? (S::Z_BYTES >> 4) : 0u);
#pragma unroll
          for (int ks = 0; ks < kGtBN / 16; ++ks)
            tc::mma_bf16_ts(tbase + S::COL_D2, A + ks * 16, B + 16u * ks, idesc_g,
                            (p | term | ks) != 0);
        }
        tc::commit(&b_free[h]);
      }
      __syncwarp();
      if (p >= 1 && p - 1 + ST < nt) {
        const int hp = h == 0 ? SETS - 1 : h - 1, s1 = s == 0 ? ST - 1 : s - 1;
        ok = tc::warp_wait_uniform(b_free0 + 8u * hp, (uint32_t)(((p - 1) / SETS) & 1));
        if (!ok) break;
        if (tc::elect_one()) copy_tile(p - 1 + ST, s1);
        __syncwarp();
        issued = p + ST;
      }
      if (++s == ST) s = 0;
      if (++h == SETS) { h = 0; ph_h ^= 1; }
    }
    if (!ok) *s_fail = 1;
    // a CTA with an empty range issues nothing and waits on nothing
    if (nt > 0 && tc::elect_one()) tc::commit(done);
    __syncwarp();
  } else {
    // ------ epilogue: warp (lane quadrant eq, set h) takes the tiles h, h + 3, ... whole ------
    const int eq = warp & 3;
    const int set = (warp - kGtIssuers) >> 2;
    const int il = eq * 32 + lane;
    const long long i = row0 + il;
    const uint32_t lane_base = (uint32_t)(eq * 32) << 16;
    const float c0 = a.params->c0f, c1 = a.params->c1f;
    const float two_c1 = 2.f * c1;
    float xi[S::XC ? 1 : DP];
    if constexpr (!S::XC) {
#pragma unroll
      for (int k = 0; k < DP; ++k) xi[k] = (i < a.n) ? two_c1 * a.xhat[i * DP + k] : 0.f;
    }
    const float ai = c0 + ((i < a.n) ? a.bneg[i] : 0.f);
    const bool add_bj = !S::XC || !a.c_has_bj;   // else the augmented C carries b_j
    const float2 minus1 = make_float2(-1.f, -1.f);
    const float2 ai2 = make_float2(ai, ai);
    bool ok = true;
    int s = set, ph_s = 0, ph = 0;   // set < ST
    int c = S::NC > 0 ? set % S::NC : 0, cf = set, ph_cf = 0;
#pragma unroll 1
    for (int lt = set; lt < nt; lt += SETS) {
      // b_J (and x^_J) are read from the stage: wait for its copy too (the stage is refilled
      // only after this tile's P Z, which waits for this warp's P)
      ok = tc::warp_wait_uniform(w_full0 + 8u * set, ph) &&
           tc::warp_wait_uniform(full0 + 8u * s, ph_s);
      if constexpr (S::XC) ok = ok && tc::warp_wait_uniform(c_full0 + 8u * cf, ph_cf);
      if (!ok) break;
      tc::fence_after();
      const bool own = tile_begin + lt < diag_end;   // a tile of I itself: weight 1/2
      const float* tx = reinterpret_cast<const float*>(smem + S::OFF_STAGES + s * S::STAGE_BYTES);
      const float* tb = reinterpret_cast<const float*>(smem + S::OFF_STAGES + s * S::STAGE_BYTES +
                                                       S::OFF_BN);
#pragma unroll
      for (int half = 0; half < 2; ++half) {   // 16 columns at a time
        const uint32_t wcol = tbase + lane_base + (uint32_t)(set * 32 + half * 16);
        float w[16], cx[S::XC ? 16 : 1];
        if constexpr (S::XC) {
          uint32_t r[32];
          gt_tmem_ld16_two(wcol, tbase + lane_base + S::COL_C + (uint32_t)(c * 32 + half * 16), r);
          if (half == 1) {   // the C buffer may take its next tile
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&c_free[c]);
          }
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            w[q] = __uint_as_float(r[q]);
            cx[q] = __uint_as_float(r[16 + q]);
          }
        } else {
          tc::tmem_ld16(wcol, w);
        }
        if (own) {   // (i, j) and (j, i) are both visited
#pragma unroll
          for (int q = 0; q < 16; ++q) w[q] *= 0.5f;
        }
        uint32_t hi[8], lo[8];
        // packed FP32x2 instructions: the cross term two coordinates at a time (FP32 pipe) or
        // the exponent two entries at a time (tensor-core C), the weight and the high/low split
        // two entries at a time
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          const float4 b4 = *reinterpret_cast<const float4*>(tb + half * 16 + 4 * q4);
#pragma unroll
          for (int q2 = 0; q2 < 2; ++q2) {
            const int q = 2 * q4 + q2;
            const float2 bj = q2 == 0 ? make_float2(b4.x, b4.y) : make_float2(b4.z, b4.w);
            float ex[2];
            if constexpr (S::XC) {
              // (a_i + b_j) + C_ij, the order of the K V pass
              const float2 base = add_bj ? __fadd2_rn(ai2, bj) : ai2;
              const float2 e2 = __fadd2_rn(base, make_float2(cx[2 * q], cx[2 * q + 1]));
              ex[0] = e2.x;
              ex[1] = e2.y;
            } else {
#pragma unroll
              for (int h2 = 0; h2 < 2; ++h2) {
                const int j = half * 16 + 2 * q + h2;
                float xj[DP];
                load_row<float, DP>(tx + j * DP, xj);
                float2 acc2 = make_float2(ai + (h2 == 0 ? bj.x : bj.y), 0.f);
#pragma unroll
                for (int k = 0; k < DP; k += 2)
                  acc2 = __ffma2_rn(make_float2(xi[k], xi[k + 1]), make_float2(xj[k], xj[k + 1]), acc2);
                ex[h2] = acc2.x + acc2.y;
              }
            }
            const float2 pk = __fmul2_rn(make_float2(ex2_approx(fminf(ex[0], c0)),
                                                     ex2_approx(fminf(ex[1], c0))),
                                         make_float2(w[2 * q], w[2 * q + 1]));
            const __nv_bfloat162 h = __floats2bfloat162_rn(pk.x, pk.y);
            const float2 r = __ffma2_rn(__bfloat1622float2(h), minus1, pk);   // pk - high part
            const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
            hi[q] = *reinterpret_cast<const uint32_t*>(&h);
            lo[q] = *reinterpret_cast<const uint32_t*>(&l);
          }
        }
        // P over this warp's own W columns: high parts first, then low parts
        tc::tmem_st8(wcol, hi);
        tc::tmem_st8(wcol + 8, lo);
      }
      tc::tmem_wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&p_full[set]);
      ph ^= 1;
      s += SETS;
      if (s >= ST) { s -= ST; ph_s ^= 1; }
      if constexpr (S::XC) {
        c = (c + SETS) % S::NC;
        cf += SETS;
        if (cf >= S::NCF) { cf -= S::NCF; ph_cf ^= 1; }
      }
    }
    if (!ok) *s_fail = 1;
    const bool fin = ok && (nt == 0 || tc::warp_wait_uniform(smem_u32(done), 0));
    ok = __all_sync(0xffffffffu, fin && !*s_fail);
    if (ok && nt > 0) {
      tc::fence_after();
      if (set == 0) {
        float g[N2];
#pragma unroll
        for (int c = 0; c < N2 / 16; ++c) {
          float v[16];
          tc::tmem_ld16(tbase + lane_base + S::COL_D2 + (uint32_t)(c * 16), v);
#pragma unroll
          for (int q = 0; q < 16; ++q) g[c * 16 + q] = v[q];
        }
        if (i < a.n) {
          const double Ssum = g[2 * DP];
#pragma unroll
          for (int k = 0; k < DP; ++k) {
            const double x = a.xhat[i * DP + k];
            acc[k] = x * x * Ssum - 2.0 * x * (double)g[k] + (double)g[DP + k];
          }
          acc[DP] = Ssum;
        }
      } else if (set == 1 && sp == 0 && i < a.n) {
        // diagonal W_ii for the lambda component, once per row
        float wii = 0.f;
        for (int m = 0; m < a.M; ++m)
          wii = fmaf(a.sa[m] * a.A[(long long)a.amap[m] * a.ld + i],
                     a.B[(long long)a.bmap[m] * a.ld + i], wii);
        acc[DP + 1] = wii;
      }
    }
  }

  // -------- all roles: release tensor memory; CTA reduction; last CTA sums the partials -------
  if (warp == 0 && nt > 0) (void)tc::warp_wait_uniform(smem_u32(done), 0);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, kGtCols);
  if (*s_fail) {
    if (tid == 0) {
      atomicOr(a.status, kStatusTimeout);
      // let the copies still in flight land before the CTA's shared memory goes away
      for (int lt2 = max(0, issued - S::ST); lt2 < issued; ++lt2)
        (void)mbar_wait_bounded(&full[lt2 % S::ST], (uint32_t)((lt2 / S::ST) & 1));
    }
    return;
  }
  // set 0 holds the lengthscale and sigma^2 sums, set 1 the diagonal's
  const int ew = warp - kGtIssuers;
  if (ew >= 0 && ew < 4) {
#pragma unroll
    for (int k = 0; k <= DP; ++k) {
      const double v = warp_sum(acc[k]);
      if (lane == 0) s_red[ew][k] = v;
    }
  } else if (ew >= 4 && ew < 8) {
    const double v = sp == 0 ? warp_sum(acc[DP + 1]) : 0.0;
    if (lane == 0) s_red[ew - 4][DP + 1] = v;
  }
  __syncthreads();
  double* part = a.partials + slot * kMaxP;
  if (tid < NACC) {
    double v = 0.0;
    for (int ww = 0; ww < 4; ++ww) v += s_red[ww][tid];
    // slots: lengthscales 0..d-1, then sigma^2 at d, lambda at d+1
    if (tid < a.d) part[tid] = v;
    else if (tid == DP) part[a.d] = v;
    else if (tid == DP + 1) part[a.d + 1] = v;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) *s_last = (atomicAdd(a.counter, 1) == a.n_cta - 1);
  __syncthreads();
  if (!*s_last) return;
  __threadfence();
  __shared__ double s_sum[S::THREADS];
  const double v = sum_partial_rows<S::THREADS>(a.partials, a.n_cta, a.d + 2, s_sum);
  if (tid < a.d + 2) a.g_out[tid] = tid == a.d + 1 ? v * a.params->lambda : v;
  if (tid == 0) *a.counter = 0;
}

template <int DP, int KS>
__global__ void __launch_bounds__(GtShape<DP, KS>::THREADS, GtShape<DP, KS>::OCC) grad_tc_kernel(const GtDevArgs a) {
  const int rb = blockIdx.x / a.nsplit;
  gt_body<DP, KS>(a, rb, blockIdx.x - rb * a.nsplit);
}

// Many problems of one input width in one launch: CTA b takes work item items[b] =
// (problem, row block, split) with that problem's arguments.
template <int DP, int KS>
__global__ void __launch_bounds__(GtShape<DP, KS>::THREADS, GtShape<DP, KS>::OCC) grad_tc_batch_kernel(
    const GtDevArgs* __restrict__ args, const int4* __restrict__ items) {
  __shared__ GtDevArgs s_a;
  const int4 it = items[blockIdx.x];
  if (threadIdx.x == 0) s_a = args[it.x];
  __syncthreads();
  gt_body<DP, KS>(s_a, it.y, it.z);
}

// The operand blocks of every problem of a batched launch (one problem per grid row), as
// pack_gt_kernel.
template <int DP, int KS>
__global__ void pack_gt_batch_kernel(const GtDevArgs* __restrict__ args) {
  using S = GtShape<DP, KS>;
  const GtDevArgs& a = args[blockIdx.y];
  const long long total = (long long)a.ntiles * kGtBN * (S::K1 + S::N2);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x)
    gt_pack_element(idx, S::K1, S::N2, DP, a.M, a.n, a.xhat, a.A, a.amap, a.sa, a.B, a.bmap, a.ld,
                    const_cast<__nv_bfloat16*>(a.tiles));
}

// Split of each row block's tile range into s CTAs.  The SMs share the visited tiles plus a
// fixed cost per CTA (the operand image, the pipeline fill and the reduction, about six
// tiles' worth); a CTA shares its SM with others, so the longest range (row block 0, ntiles / s
// tiles) takes about occ x its length and must not end the pass.  The ranges also bound the
// rounding of the sums, which tensor memory accumulates in FP32 with truncation: occ is taken
// as 3 (2 for four or more factor steps or padded d = 16, 1 for eight), not the two CTAs that
// share an SM, because ranges 1.5 times as long would raise the error of the gradient 1.4 times.
static int plan_gt_split(long long n_rb, long long ntiles, int num_sms, int occ) {
  const long long per_block = kGtBM / kGtBN;
  const long long visited = n_rb * ntiles - per_block * n_rb * (n_rb - 1) / 2;
  // no more than kTcMaxSplitTiles tiles per CTA: the sums accumulate in FP32 in tensor memory
  const int s_min = (int)((ntiles + kTcMaxSplitTiles - 1) / kTcMaxSplitTiles);
  long long best = -1;
  int best_s = s_min;
  for (int s = s_min; s <= std::max(64, s_min) && s <= ntiles; ++s) {
    const long long shared = (visited + 6 * n_rb * s + num_sms - 1) / num_sms;
    const long long longest = ((ntiles + s - 1) / s + 6) * occ;
    const long long cost = std::max(shared, longest);
    if (best < 0 || cost < best) {
      best = cost;
      best_s = s;
    }
  }
  return best_s;
}

// The TF32 row images of the K V pass (A rows at X_hi / X_lo, B tiles at X_b).
static void gt_set_images(GtDevArgs& a, const GradLaunch& L) {
  a.XA_hi = L.X_hi;
  a.XA_lo = L.X_lo;
  a.XB = L.X_b;
  a.c_has_bj = L.c_has_bj ? 1 : 0;
}

template <int DP, int KS>
struct GtInst {
  using S = GtShape<DP, KS>;
  static constexpr int kPlanOcc = KS >= 8 ? 1 : (KS >= 4 || DP >= 16) ? 2 : 3;
  static void prime() {
    static std::once_flag once;
    std::call_once(once, [] {
      auto fn = grad_tc_kernel<DP, KS>;
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
      cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    });
  }
  static cudaError_t launch(GradLaunch& L, cudaStream_t s) {
    prime();
    const long long ntiles = (L.n + kGtBN - 1) / kGtBN;
    const int n_rb = (int)((L.n + kGtBM - 1) / kGtBM);
    const int nsplit = plan_gt_split(n_rb, ntiles, L.num_sms, kPlanOcc);
    const size_t need = (size_t)n_rb * nsplit * kMaxP;
    if (L.plan_only) {
      L.need_partials_len = need;
      return cudaSuccess;
    }
    if (need > L.partials_len) {
      L.need_partials_len = need;
      return cudaErrorMemoryAllocation;
    }
    __nv_bfloat16* tiles = static_cast<__nv_bfloat16*>(L.tc_tiles);
    {
      const long long total = ntiles * kGtBN * (S::K1 + S::N2);
      const int blocks = (int)std::min<long long>((total + 255) / 256, 8LL * L.num_sms);
      pack_gt_kernel<<<blocks, 256, 0, s>>>(
          S::K1, S::N2, DP, L.M, L.n, ntiles, static_cast<const float*>(L.xhat),
          static_cast<const float*>(L.A), L.amap, static_cast<const float*>(L.sa),
          static_cast<const float*>(L.B), L.bmap, L.ld, tiles);
    }
    GtDevArgs a;
    a.xhat = static_cast<const float*>(L.xhat);
    a.bneg = L.bneg;
    a.tiles = tiles;
    a.A = static_cast<const float*>(L.A);
    a.amap = L.amap;
    a.sa = static_cast<const float*>(L.sa);
    a.B = static_cast<const float*>(L.B);
    a.bmap = L.bmap;
    a.ld = L.ld;
    a.M = L.M;
    a.n = L.n;
    a.d = L.d;
    a.params = L.params;
    a.nsplit = nsplit;
    a.n_cta = n_rb * nsplit;
    a.ntiles = (int)ntiles;
    gt_set_images(a, L);
    a.partials = L.partials;
    a.counter = L.counter;
    a.g_out = L.g_out;
    a.status = L.status;
    grad_tc_kernel<DP, KS><<<n_rb * nsplit, S::THREADS, S::SMEM, s>>>(a);
    return cudaGetLastError();
  }
};

// KS = 16-wide steps of the 2M factor slots.
template <int DP>
static cudaError_t grad_tc_dispatch_m(GradLaunch& L, cudaStream_t s) {
  if (L.M <= 8) return GtInst<DP, 1>::launch(L, s);
  if (L.M <= 16) return GtInst<DP, 2>::launch(L, s);
  if (L.M <= 24) return GtInst<DP, 3>::launch(L, s);
  if (L.M <= 32) return GtInst<DP, 4>::launch(L, s);
  if (L.M <= 64) return GtInst<DP, 8>::launch(L, s);
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------------------
// Batched launches: many problems of one padded width in one launch.
// ---------------------------------------------------------------------------------------
size_t gt_batch_args_bytes(int B) { return sizeof(GtDevArgs) * (size_t)B; }

cudaError_t gt_batch_upload_args(const GradLaunch* L, const int* nsplit, int B, void* args_dev,
                                 cudaStream_t s) {
  std::vector<GtDevArgs> h((size_t)B);
  for (int b = 0; b < B; ++b) {
    const GradLaunch& l = L[b];
    const long long ntiles = (l.n + kGtBN - 1) / kGtBN;
    const long long n_rb = (l.n + kGtBM - 1) / kGtBM;
    if (l.M < 1 || l.M > kMaxM || nsplit[b] < 1 || l.DP != L[0].DP || !l.tc_tiles ||
        !l.X_hi || !l.X_lo || !l.X_b ||
        (ntiles + nsplit[b] - 1) / nsplit[b] > kTcMaxSplitTiles)
      return cudaErrorInvalidValue;
    GtDevArgs& a = h[b];
    a.xhat = static_cast<const float*>(l.xhat);
    a.bneg = l.bneg;
    a.tiles = static_cast<const __nv_bfloat16*>(l.tc_tiles);
    a.A = static_cast<const float*>(l.A);
    a.amap = l.amap;
    a.sa = static_cast<const float*>(l.sa);
    a.B = static_cast<const float*>(l.B);
    a.bmap = l.bmap;
    a.ld = l.ld;
    a.M = l.M;
    a.n = l.n;
    a.d = l.d;
    a.params = l.params;
    a.nsplit = nsplit[b];
    a.ntiles = (int)ntiles;
    a.n_cta = (int)(n_rb * nsplit[b]);
    gt_set_images(a, l);
    a.partials = l.partials;
    a.counter = l.counter;
    a.g_out = l.g_out;
    a.status = l.status;
  }
  return cudaMemcpyAsync(args_dev, h.data(), sizeof(GtDevArgs) * (size_t)B,
                         cudaMemcpyHostToDevice, s);
}

template <int DP, int KS>
static void gt_batch_prime() {
  static std::once_flag once;
  std::call_once(once, [] {
    auto fn = grad_tc_batch_kernel<DP, KS>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)GtShape<DP, KS>::SMEM);
    cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  });
}

template <int DP, int KS>
static cudaError_t gt_batch_launch(const GtDevArgs* args, int B, const int4* items, int n_items,
                                   bool prime_only, cudaStream_t s) {
  gt_batch_prime<DP, KS>();
  if (prime_only) return cudaSuccess;
  pack_gt_batch_kernel<DP, KS><<<dim3(64, (unsigned)B), 256, 0, s>>>(args);
  if (n_items > 0)
    grad_tc_batch_kernel<DP, KS><<<n_items, GtShape<DP, KS>::THREADS, GtShape<DP, KS>::SMEM, s>>>(args, items);
  return cudaGetLastError();
}

template <int DP>
static cudaError_t gt_batch_dispatch_m(const GtDevArgs* args, int B, const int4* items,
                                       int n_items, int M, bool prime_only, cudaStream_t s) {
  if (M <= 8) return gt_batch_launch<DP, 1>(args, B, items, n_items, prime_only, s);
  if (M <= 16) return gt_batch_launch<DP, 2>(args, B, items, n_items, prime_only, s);
  if (M <= 24) return gt_batch_launch<DP, 3>(args, B, items, n_items, prime_only, s);
  if (M <= 32) return gt_batch_launch<DP, 4>(args, B, items, n_items, prime_only, s);
  if (M <= 64) return gt_batch_launch<DP, 8>(args, B, items, n_items, prime_only, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_grad_tc_batch(const void* args_dev, int B, const int4* items, int n_items,
                                 int DP, int M, cudaStream_t s, bool prime_only) {
  const GtDevArgs* args = static_cast<const GtDevArgs*>(args_dev);
  if (B < 1 && !prime_only) return cudaErrorInvalidValue;
  switch (DP) {
    case 2: return gt_batch_dispatch_m<2>(args, B, items, n_items, M, prime_only, s);
    case 4: return gt_batch_dispatch_m<4>(args, B, items, n_items, M, prime_only, s);
    case 8: return gt_batch_dispatch_m<8>(args, B, items, n_items, M, prime_only, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_grad_tc(GradLaunch& L, cudaStream_t s) {
  if (L.M < 1 || L.M > kMaxM || !L.tc_tiles || !L.bneg) return cudaErrorInvalidValue;
  if (L.DP <= 8 && (!L.X_hi || !L.X_lo || !L.X_b)) return cudaErrorInvalidValue;
  switch (L.DP) {
    case 2: return grad_tc_dispatch_m<2>(L, s);
    case 4: return grad_tc_dispatch_m<4>(L, s);
    case 8: return grad_tc_dispatch_m<8>(L, s);
    case 16: return grad_tc_dispatch_m<16>(L, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ulisse
