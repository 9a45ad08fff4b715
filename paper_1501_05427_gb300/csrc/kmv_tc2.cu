// Mixed-precision tile-generating K V with the cross term on the tensor cores too.
//
// For a block of 128 output rows I and a 32-point tile J:
//   1. C_IJ = A_I B_J^T on the tensor cores (kind::tf32).  With padded d = 2 or 4 the rows
//      carry the column term too,
//          A_i = [x^_i, 1],  B_j = [2 c1 x^_j, b_j],   b_j = -c1 |x^_j|^2, c1 = log2(e)/2,
//      so that C_ij = 2 c1 x^_i . x^_j + b_j in one 8-wide K step; with padded d = 8 or 16
//      the rows are A_i = x^_i, B_j = 2 c1 x^_j (K = d: the augmented column would cost a
//      whole further K step, three MMAs per tile that warp 0 would issue and the tensor pipe
//      run) and the epilogue adds b_j.  Both sides split into a TF32 high part and the
//      remainder, three products (Ah Bh + Ah Bl + Al Bh), FP32 accumulation into a 32-column
//      tensor-memory buffer;
//   2. the epilogue warps read C back (tcgen05.ld) and form
//          k_ij = exp2(a_i + C_ij)  or  exp2((a_i + b_j) + C_ij),
//          a_i = log2(sigma^2) - c1 |x^_i|^2
//      (one or two FADDs and one ex2 per entry), split k into BF16 high and low parts and
//      store them over C's own columns (tcgen05.st);
//   3. U_I += K_IJ V_J on the tensor cores with V split into BF16 high + low parts (three
//      products), FP32 accumulation in tensor memory, as in the FP32-pipe variant.
// The TF32 images of A and B (high and low parts, K-major canonical, 32-point tiles) are written
// once per parameter value by the prescale launch; B's tiles and V's tiles each lie contiguously
// with all their parts, so that a unit of tiles is two bulk copies.  A_I goes into tensor memory
// once per CTA, and every MMA reads its A operand there (from shared memory the 4 KB take 40 clocks
// per MMA, against 16 for the product itself at N = 32).  Roles: warp 0 copies (B_J, b_J and V_J
// into a ring of stages) and issues the exponent's MMAs; warp 1 issues the contraction's; the
// epilogue warps make the kernel values in sets of four (one per tensor-memory lane quadrant).  A
// set takes a unit of G consecutive tiles whole, so that each wait and hand-off covers 32 G
// entries per thread: three sets and units of two tiles up to N = 32, four sets and units of one
// where the accumulator takes 64 columns.  A buffer is refilled only after the MMAs that read it
// have completed, and the stage of that unit is refilled at the same moment.  Every wait is
// bounded.  The split j range, the fixed-order fix-up of the partial sums and the FP32 diagonal
// term lambda V are those of the FP32-pipe variant.
//
// What bounds it: the epilogue's issue slots (ncu at n = 50,000, d = 8, N = 32: 7.6 thread
// instructions per entry, schedulers 77% busy), at N = 64 the tensor pipe (77% busy).  The issuing
// warps come next: a tile takes about a hundred of their instructions, which wait their turn
// among the epilogue's.  Times of the kernel at n = 50,000, d = 8, 17 columns: 1.046 ms with a
// copying warp and one divergent lane issuing for four CTAs of eight epilogue warps per SM; 0.777
// ms with one warp-uniform warp doing both (a lane elected for the issuing instructions keeps the
// descriptors in uniform registers; 56 registers instead of 48); 0.677 ms with A in tensor memory,
// two CTAs of twelve epilogue warps per SM, units of two tiles and the two issuing warps (with
// one: 0.75 ms; units of one tile and four sets: 0.77 ms).  n = 200,000, d = 16, 64 columns: 19.2,
// 15.6 and 14.6 ms per call.
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "kmv_kernel.cuh"
#include "pack_v.cuh"
#include "prescale.cuh"
#include "tc_common.cuh"

namespace ulisse {

constexpr int kT2BN = 32;
constexpr int kT2BM = 128;
constexpr uint32_t kT2Cols = 256;  // tensor-memory columns per CTA (two CTAs per SM)

// The prescale of the mixed path, one row per thread: x^_j, the row norm b_j = -c1 |x^_j|^2
// (summed in FP64), and the rows A_j = [x^_j, 1, 0...] and B_j = [2 c1 x^_j, b_j, 0...] as TF32
// high part and remainder, K8 columns, in 32-row K-major canonical tiles.  Rows j in [n, rows)
// are zero (x^ itself is written for j < n only).  When K8 == DP there is no slot for the
// augmented column (A_j = x^_j, B_j = 2 c1 x^_j); the batched launches leave it out for every d
// (aug = 0) and add b_j in the epilogue.  A's parts are two arrays; B's tiles hold high part,
// remainder and the tile's 32 b_j back to back (tc2_b_stride floats each), so that a tile is one
// bulk copy.
template <int DP>
__global__ void __launch_bounds__(128) prescale_mixed_kernel(
    const PsiArg pa, double* __restrict__ psi_dev, const float* __restrict__ X,
    float* __restrict__ xhat, long long n, long long rows, int d, int aug,
    DevParams* __restrict__ P, float* __restrict__ bneg, float* __restrict__ Ahi,
    float* __restrict__ Alo, float* __restrict__ Bt, const PackV pv) {
  constexpr int K8 = DP >= 8 ? DP : 8;
  __shared__ InvLength s;
  if ((int)blockIdx.x >= pv.first_cta) {   // a product's operand rides along
    pack_v2(pv.V, n, nullptr, pv.R, pv.N, n, (n + kT2BN - 1) / kT2BN,
            static_cast<__nv_bfloat16*>(pv.Vp), blockIdx.x - pv.first_cta, gridDim.x - pv.first_cta);
    return;
  }
  unpack_params(pa, psi_dev, d, P, s);
  const float two_c1 = 2.f * (float)(0.5 * 1.4426950408889634);   // 2 c1f
  for (long long j = blockIdx.x * 128LL + threadIdx.x; j < rows; j += pv.first_cta * 128LL) {
    float x[K8];
    double s2 = 0.0;
#pragma unroll
    for (int k = 0; k < K8; ++k) {
      x[k] = (k < d && j < n) ? scale_by_pair(X[j * d + k], s, k) : 0.f;
      if (k < d) s2 += (double)x[k] * (double)x[k];
    }
    if (j < n) {
      if constexpr (DP >= 4) {
#pragma unroll
        for (int k = 0; k < DP; k += 4)
          *reinterpret_cast<float4*>(xhat + j * DP + k) = make_float4(x[k], x[k + 1], x[k + 2], x[k + 3]);
      } else {
        *reinterpret_cast<float2*>(xhat + j * DP) = make_float2(x[0], x[1]);
      }
    }
    const float b = (float)(-0.5 * 1.4426950408889634 * s2);
    bneg[j] = b;
    const long long t = j / kT2BN;
    const int jj = (int)(j - t * kT2BN);
    float* bt = Bt + t * tc2_b_stride(K8);
    bt[2 * kT2BN * K8 + jj] = b;
#pragma unroll
    for (int k0 = 0; k0 < K8; k0 += 4) {
      float ah[4], al[4], bh[4], bl[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = k0 + q;
        float va = x[k], vb = two_c1 * x[k];
        if (DP < K8 && k == DP && aug && j < n) {
          va = 1.f;
          vb = b;
        }
        ah[q] = tc::tf32_round(va);
        al[q] = va - ah[q];
        bh[q] = tc::tf32_round(vb);
        bl[q] = vb - bh[q];
      }
      const uint32_t in_tile = tc::canon_offset(jj, k0, 4, K8 / 4) / 4;
      const long long off = t * kT2BN * K8 + in_tile;
      *reinterpret_cast<float4*>(Ahi + off) = make_float4(ah[0], ah[1], ah[2], ah[3]);
      *reinterpret_cast<float4*>(Alo + off) = make_float4(al[0], al[1], al[2], al[3]);
      *reinterpret_cast<float4*>(bt + in_tile) = make_float4(bh[0], bh[1], bh[2], bh[3]);
      *reinterpret_cast<float4*>(bt + kT2BN * K8 + in_tile) = make_float4(bl[0], bl[1], bl[2], bl[3]);
    }
  }
}

struct Tc2DevArgs {
  const float* A_hi;     // TF32 image of the augmented A rows (high part)
  const float* A_lo;     // remainder
  const float* B;        // TF32 tiles of the augmented B rows: high part | remainder | b_j
  const float* bneg;     // -c1 |x^|^2
  const __nv_bfloat16* Vp;   // BF16 tiles of V: high | low part
  const float* V;        // FP32 operand columns (diagonal term)
  long long ldv;
  const int* vmap;
  int R;
  const int* R_dev;      // batched launches: the live column count on the device (else null)
  float* U;
  long long ldu;
  const int* umap;
  long long n;
  const DevParams* params;
  int nsplit, tiles_per_split, ntiles;
  float* partials;
  int* counters;
  int* status;
};

// BJ: the epilogue adds b_j (the rows are not augmented); the stage then carries b_J.
template <int K8, int N, bool BJ>
struct Tc2Shape {
  // A unit is G consecutive tiles handed over together: one wait, fence and arrival per unit.
  // The accumulator and the A rows (high part and remainder, K8 columns each) leave room for
  // three units of two tiles up to N = 32 (three sets of epilogue warps); with N = 64 for five
  // units of one tile (four sets).
  static constexpr int G = N <= 32 ? 2 : 1;
  static constexpr int NBUF = N <= 32 ? 3 : 5;
  static constexpr int SETS = N <= 32 ? 3 : 4;
  static constexpr int THREADS = 32 * (2 + 4 * SETS);   // copies and C, contraction, the sets
  static constexpr uint32_t XB_BYTES = kT2BN * K8 * 4;  // one part of a B tile
  static constexpr uint32_t V_BYTES = N * kT2BN * 2;    // one part of a BF16 V tile
  static constexpr uint32_t BN_BYTES = kT2BN * 4;       // a tile's b_j
  static constexpr uint32_t X_COPY = 2 * XB_BYTES + BN_BYTES;   // B high | remainder | b
  static constexpr uint32_t OFF_BN = 2 * XB_BYTES;              // within a tile
  static constexpr uint32_t OFF_V = G * X_COPY;                 // within a stage
  static constexpr uint32_t STAGE_BYTES = OFF_V + G * 2 * V_BYTES;
  // as many stages (units) as let two CTAs fit in shared memory, at most 8
  static constexpr int ST_FIT = (int)((108u * 1024u) / STAGE_BYTES);
  static constexpr int ST = ST_FIT > 8 ? 8 : ST_FIT;
  static_assert(ST > NBUF, "a stage beyond those in flight");
  static constexpr uint32_t OFF_BARS = ST * STAGE_BYTES;
  // full per stage; c_full, k_full, b_free per buffer; done
  static constexpr int NBARS = ST + 3 * NBUF + 1;
  static constexpr uint32_t SMEM = OFF_BARS + NBARS * 8 + 64;
  // tensor-memory columns: the C/K buffers, the accumulator, A's two parts
  static constexpr uint32_t COL_U = NBUF * G * 32;
  static constexpr uint32_t COL_A = COL_U + N;
  static_assert(COL_A + 2 * K8 <= kT2Cols, "tensor memory layout exceeds the allocation");
  static_assert(STAGE_BYTES % 16 == 0 && XB_BYTES % 16 == 0 && X_COPY % 16 == 0 && OFF_V % 16 == 0,
                "bulk copies and descriptors need 16-byte alignment");
};

template <int NH>
__device__ inline void t2_ld_cols(uint32_t taddr, float (&v)[NH]) {
  if constexpr (NH == 8) {
    tc::tmem_ld8(taddr, v);
  } else if constexpr (NH == 16) {
    tc::tmem_ld16(taddr, v);
  } else {
    // two 16-column loads: the registers of one are free again before the other's arrive
    float v0[16], v1[16];
    tc::tmem_ld16(taddr, v0);
    tc::tmem_ld16(taddr + 16, v1);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      v[q] = v0[q];
      v[16 + q] = v1[q];
    }
  }
}

// One CTA's work: row block rb, j-range split sp, R live columns.  Shared by the
// single-problem kernel (rb, sp from the block index) and the batched one (from its work list).
template <int K8, int N, bool BJ>
__device__ __forceinline__ void tc2_body(const Tc2DevArgs& a, const int rb, const int sp,
                                         const int R) {
  using S = Tc2Shape<K8, N, BJ>;
  constexpr int ST = S::ST, G = S::G, NBUF = S::NBUF, SETS = S::SETS;
  constexpr int NH = N / 2;
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t smem0 = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::OFF_BARS);
  uint64_t* full = bars;
  uint64_t* c_full = bars + ST;
  uint64_t* k_full = c_full + NBUF;
  uint64_t* b_free = k_full + NBUF;
  uint64_t* done = b_free + NBUF;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + S::OFF_BARS + S::NBARS * 8);
  volatile int* s_fail = reinterpret_cast<volatile int*>(s_tmem + 1);
  int* s_last = reinterpret_cast<int*>(s_tmem + 2);
  const uint32_t full0 = smem_u32(full), c_full0 = smem_u32(c_full), k_full0 = smem_u32(k_full),
                 b_free0 = smem_u32(b_free);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler
  const long long slot = (long long)rb * a.nsplit + sp;   // this CTA's partial-sum slot
  const long long row0 = (long long)rb * kT2BM;
  const int tile_begin = sp * a.tiles_per_split;
  const int nt = max(0, min(tile_begin + a.tiles_per_split, a.ntiles) - tile_begin);
  const int nu = (nt + G - 1) / G;   // units; the last may hold fewer tiles

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) mbar_init(&full[s], 1);
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(&c_full[b], 1);
      mbar_init(&k_full[b], 4);   // the four epilogue warps of the unit's set
      mbar_init(&b_free[b], 1);
    }
    mbar_init(done, 1);
    fence_barrier_init();
    *s_fail = 0;
  }
  if (warp == 0) tc::tmem_alloc(s_tmem, kT2Cols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = __shfl_sync(0xffffffffu, *s_tmem, 0);
  if (warp >= 2 && warp <= 5) {
    // A_I into tensor memory, a row per thread: the cross term's A operand is then read there
    // (an MMA whose A comes from shared memory takes 40 clocks for its 4 KB, from tensor memory 16)
    const int eq = warp & 3;
    const long long i = row0 + eq * 32 + lane;
    const long long off = (i / 32) * 32 * K8 + tc::canon_offset((int)(i % 32), 0, 4, K8 / 4) / 4;
    const uint32_t dst = tbase + ((uint32_t)(eq * 32) << 16) + S::COL_A;
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      const float* src = (part == 0 ? a.A_hi : a.A_lo) + off;
#pragma unroll
      for (int k = 0; k < K8; k += 8) {
        const uint4 x = *reinterpret_cast<const uint4*>(src + k / 4 * 32);
        const uint4 y = *reinterpret_cast<const uint4*>(src + (k / 4 + 1) * 32);
        const uint32_t v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        tc::tmem_st8(dst + (uint32_t)(part * K8 + k), v);
      }
    }
    tc::tmem_wait_st();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  int issued = 0;   // units whose copies were started (warp 0)

  if (warp == 0) {
    // ------ copies and MMAs of the cross term, C = x^_I x^_J^T; one elected lane issues, the
    //        whole warp runs the loop, so that descriptors and addresses stay warp-uniform ------
    constexpr uint32_t idesc_c = tc::instr_desc(2, kT2BM, kT2BN);   // TF32
    constexpr uint32_t sbo_x = (K8 / 4) * 128;
    const uint64_t dB0 = tc::smem_desc(smem0, 128, sbo_x);
    const float* srcX = a.B + (long long)tile_begin * tc2_b_stride(K8);
    const __nv_bfloat16* srcV = a.Vp + (long long)tile_begin * 2 * N * kT2BN;
    auto copy_unit = [&](int u, int s) {   // elected lane: the unit's B (with b) and V tiles
      const uint32_t m = (uint32_t)min(G, nt - u * G);
      unsigned char* st = smem + s * S::STAGE_BYTES;
      mbar_arrive_expect_tx(&full[s], m * (S::X_COPY + 2 * S::V_BYTES));
      bulk_g2s(st, srcX + (long long)u * G * tc2_b_stride(K8), m * S::X_COPY, &full[s]);
      bulk_g2s(st + S::OFF_V, srcV + (long long)u * G * 2 * N * kT2BN, m * 2 * S::V_BYTES, &full[s]);
    };
    auto mma_c = [&](int u, int s, int b) {   // elected lane: the unit's C into buffer b
#pragma unroll
      for (int g = 0; g < G; ++g) {
        if (g > 0 && u * G + g >= nt) break;
        const uint64_t dBh = dB0 + (uint64_t)((s * S::STAGE_BYTES + g * S::X_COPY) >> 4);
        const uint32_t dC = tbase + (uint32_t)(b * G * 32 + g * 32);
#pragma unroll
        for (int term = 0; term < 3; ++term) {
          const uint32_t A = tbase + S::COL_A + (term == 2 ? (uint32_t)K8 : 0u);
          const uint64_t B = term == 1 ? dBh + (S::XB_BYTES >> 4) : dBh;
#pragma unroll
          for (int ks = 0; ks < K8 / 8; ++ks)
            tc::mma_tf32_ts(dC, A + 8u * ks, B + 16u * ks, idesc_c, (term | ks) != 0);
        }
      }
      tc::commit(&c_full[b]);
    };
    const int pre = min(ST, nu);
    if (tc::elect_one())
      for (int u = 0; u < pre; ++u) copy_unit(u, u);
    __syncwarp();
    issued = pre;
    bool ok = true;
    int s_c = 0, ph_c = 0;   // stage of the next unit whose C is issued
    for (int u = 0; u < NBUF && u < nu && ok; ++u) {
      ok = tc::warp_wait_uniform(full0 + 8u * s_c, ph_c);
      tc::fence_after();
      if (ok && tc::elect_one()) mma_c(u, s_c, u);
      __syncwarp();
      if (++s_c == ST) { s_c = 0; ph_c ^= 1; }
    }
    // the buffer and the stage of unit v are refilled once its contraction has read them
    int s = 0, b = 0, ph_b = 0;
#pragma unroll 1
    for (int v = 0; ok && v + min(NBUF, ST) < nu; ++v) {
      ok = tc::warp_wait_uniform(b_free0 + 8u * b, ph_b);
      if (ok && v + NBUF < nu) {
        ok = tc::warp_wait_uniform(full0 + 8u * s_c, ph_c);
        tc::fence_after();
        if (ok && tc::elect_one()) mma_c(v + NBUF, s_c, b);
        __syncwarp();
        if (++s_c == ST) { s_c = 0; ph_c ^= 1; }
      }
      if (ok && v + ST < nu) {
        if (tc::elect_one()) copy_unit(v + ST, s);
        __syncwarp();
        issued = v + ST + 1;
      }
      if (++s == ST) s = 0;
      if (++b == NBUF) { b = 0; ph_b ^= 1; }
    }
    if (!ok) *s_fail = 1;
  } else if (warp == 1) {
    // ------ MMAs of the contraction: U += K V; a warp of their own, so that neither stream of
    //        issuing instructions (about a hundred per tile, in turn with the epilogue's) and
    //        waits holds up the other ------
    constexpr uint32_t idesc_u = tc::instr_desc(1, kT2BM, N);       // BF16
    const uint64_t dV0 = tc::smem_desc(smem0 + S::OFF_V, 128, 512);
    bool ok = true;
    int s = 0, b = 0, ph_b = 0;
#pragma unroll 1
    for (int u = 0; u < nu; ++u) {
      ok = tc::warp_wait_uniform(k_full0 + 8u * b, ph_b);
      if (!ok) break;
      tc::fence_after();
      if (tc::elect_one()) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
          if (g > 0 && u * G + g >= nt) break;
          const uint64_t dVh = dV0 + (uint64_t)((s * S::STAGE_BYTES + g * 2 * S::V_BYTES) >> 4);
          const uint32_t kcol = tbase + (uint32_t)(b * G * 32 + g * 32);
#pragma unroll
          for (int term = 0; term < 3; ++term) {
            const uint32_t A = kcol + (term == 2 ? 8u : 0u);   // K high | K low per 16 points
            const uint64_t B = term == 1 ? dVh + (S::V_BYTES >> 4) : dVh;
#pragma unroll
            for (int ks = 0; ks < kT2BN / 16; ++ks)
              tc::mma_bf16_ts(tbase + S::COL_U, A + ks * 16, B + 16u * ks, idesc_u,
                              (u | g | term | ks) != 0);
          }
        }
        // buffer b takes unit u + NBUF's C, and stage s unit u + ST's operands, only after
        // these MMAs have read its K and V
        tc::commit(&b_free[b]);
      }
      __syncwarp();
      if (++s == ST) s = 0;
      if (++b == NBUF) { b = 0; ph_b ^= 1; }
    }
    if (!ok) *s_fail = 1;
    if (tc::elect_one()) tc::commit(done);
    __syncwarp();
  } else {
    // ------ epilogue: warp (lane quadrant eq, set h) takes the units h, h + SETS, ... whole ------
    const int eq = warp & 3;
    const int set = (warp - 2) >> 2;
    const int half = set;   // sets 0 and 1 read back the two halves of U
    const int il = eq * 32 + lane;
    const long long i = row0 + il;
    const uint32_t lane_base = (uint32_t)(eq * 32) << 16;
    const float ai = a.params->c0f + a.bneg[i];   // bneg covers the padded rows (zero there)
    // two entries per packed FP32x2 instruction (FADD2 / FFMA2, the same rounding as the
    // scalar forms)
    const float2 ai2 = make_float2(ai, ai);
    const float2 minus1 = make_float2(-1.f, -1.f);
    bool ok = true;
    int s = set, ph_s = 0, b = set, ph_b = 0;   // set < NBUF < ST
#pragma unroll 1
    for (int u = set; u < nu; u += SETS) {
      // A wait for the unit's use of its buffer cannot see the use before last: that one's C was
      // committed before the C of unit u - SETS, which this set has finished.
      ok = tc::warp_wait_uniform(c_full0 + 8u * b, ph_b);
      // b_J is read from the stage: wait for its copy too (the stage is refilled only after
      // this unit's contraction, which waits for this warp's K)
      if constexpr (BJ) ok = ok && tc::warp_wait_uniform(full0 + 8u * s, ph_s);
      if (!ok) break;
      tc::fence_after();
      const int m = G == 1 ? 1 : min(G, nt - u * G);
#pragma unroll 1
      for (int g = 0; g < m; ++g) {
        const float4* bj = reinterpret_cast<const float4*>(smem + s * S::STAGE_BYTES +
                                                           g * S::X_COPY + S::OFF_BN);
        // all 32 columns of a tile's C in one tensor-memory round trip
        const uint32_t ccol = tbase + lane_base + (uint32_t)(b * G * 32 + g * 32);
        uint32_t c[32];
        tc::tmem_ld16x2(ccol, c);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          uint32_t hi[8], lo[8];
#pragma unroll
          for (int g4 = 0; g4 < 4; ++g4) {
            float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (BJ) b4 = bj[4 * hh + g4];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const int e0 = 16 * hh + 4 * g4 + 2 * q;
              // the exponent is <= log2 sigma^2 up to rounding (about 1e-6 relative in k)
              float2 e = ai2;
              if constexpr (BJ) e = __fadd2_rn(e, q == 0 ? make_float2(b4.x, b4.y) : make_float2(b4.z, b4.w));
              e = __fadd2_rn(e, make_float2(__uint_as_float(c[e0]), __uint_as_float(c[e0 + 1])));
              const float2 k = make_float2(ex2_approx(e.x), ex2_approx(e.y));
              const __nv_bfloat162 h = __floats2bfloat162_rn(k.x, k.y);
              const float2 r = __ffma2_rn(__bfloat1622float2(h), minus1, k);   // k - high part
              const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
              hi[2 * g4 + q] = *reinterpret_cast<const uint32_t*>(&h);
              lo[2 * g4 + q] = *reinterpret_cast<const uint32_t*>(&l);
            }
          }
          // columns [16 hh, 16 hh + 16): high parts, then low parts (the A operand of the
          // contraction's k-step hh)
          tc::tmem_st8(ccol + 16 * hh, hi);
          tc::tmem_st8(ccol + 16 * hh + 8, lo);
        }
      }
      tc::tmem_wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&k_full[b]);
      s += SETS;
      if (s >= ST) { s -= ST; ph_s ^= 1; }
      b += SETS;
      if (b >= NBUF) { b -= NBUF; ph_b ^= 1; }
    }
    if (!ok) *s_fail = 1;
    const bool fin = ok && tc::warp_wait_uniform(smem_u32(done), 0);
    ok = __all_sync(0xffffffffu, fin && !*s_fail);
    if (half > 1) {
      // the other sets have nothing to read back
    } else if (ok && nt > 0) {
      tc::fence_after();
      float u[NH];
      t2_ld_cols<NH>(tbase + lane_base + S::COL_U + (uint32_t)(half * NH), u);
      if (a.nsplit == 1) {
        if (i < a.n) {
          const float lam = (float)a.params->lambda;
#pragma unroll
          for (int q = 0; q < NH; ++q) {
            const int r = half * NH + q;
            if (r < R)
              a.U[(long long)a.umap[r] * a.ldu + i] =
                  fmaf(lam, a.V[(long long)a.vmap[r] * a.ldv + i], u[q]);
          }
        }
      } else {
        float* part = a.partials + slot * N * kT2BM;
#pragma unroll
        for (int q = 0; q < NH; ++q) part[(half * NH + q) * kT2BM + il] = u[q];
      }
    } else if (ok && a.nsplit > 1) {
      float* part = a.partials + slot * N * kT2BM;
#pragma unroll
      for (int q = 0; q < NH; ++q) part[(half * NH + q) * kT2BM + il] = 0.f;
    }
  }

  // -------- all roles: release tensor memory; last CTA of the row block reduces --------
  if (warp == 0) (void)tc::warp_wait_uniform(smem_u32(done), 0);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, kT2Cols);
  if (*s_fail) {
    if (tid == 0) {
      atomicOr(a.status, kStatusTimeout);
      // let the copies still in flight land before the CTA's shared memory goes away
      for (int lt2 = max(0, issued - ST); lt2 < issued; ++lt2)
        (void)mbar_wait_bounded(&full[lt2 % ST], (uint32_t)((lt2 / ST) & 1));
    }
    return;
  }
  if (a.nsplit == 1) return;
  __threadfence();
  __syncthreads();
  if (tid == 0) *s_last = (atomicAdd(&a.counters[rb], 1) == a.nsplit - 1);
  __syncthreads();
  if (!*s_last) return;
  __threadfence();
  const float* base = a.partials + (long long)rb * a.nsplit * N * kT2BM;
  const float lam = (float)a.params->lambda;
  for (int idx = tid; idx < R * kT2BM; idx += S::THREADS) {
    const int r = idx / kT2BM, il = idx - r * kT2BM;
    const long long i = row0 + il;
    if (i >= a.n) continue;
    float u = 0.f;
    for (int s2 = 0; s2 < a.nsplit; ++s2) u += __ldcg(base + ((long long)s2 * N + r) * kT2BM + il);
    a.U[(long long)a.umap[r] * a.ldu + i] = fmaf(lam, a.V[(long long)a.vmap[r] * a.ldv + i], u);
  }
  if (tid == 0) a.counters[rb] = 0;
}

template <int K8, int N, bool BJ>
__global__ void __launch_bounds__(Tc2Shape<K8, N, BJ>::THREADS, 2) kmv_tc2_kernel(const Tc2DevArgs a) {
  const int rb = blockIdx.x / a.nsplit;
  tc2_body<K8, N, BJ>(a, rb, blockIdx.x - rb * a.nsplit, a.R);
}

// Many problems in one launch: CTA b takes work item items[b] = (problem, row block, split)
// with that problem's arguments; a problem with no live columns is skipped.
template <int K8, int N, bool BJ>
__global__ void __launch_bounds__(Tc2Shape<K8, N, BJ>::THREADS, 2) kmv_tc2_batch_kernel(
    const Tc2DevArgs* __restrict__ args, const int4* __restrict__ items) {
  __shared__ Tc2DevArgs s_a;
  const int4 it = items[blockIdx.x];
  if (threadIdx.x == 0) s_a = args[it.x];
  __syncthreads();
  const int R = s_a.R_dev ? *s_a.R_dev : s_a.R;
  if (R <= 0) return;
  tc2_body<K8, N, BJ>(s_a, it.y, it.z, R);
}

// The BF16 high and low parts of every problem's live V columns (as pack_v_kernel, one
// problem per grid row): K-major canonical images of N rows (columns of V) x 32 points.
__global__ void pack_v_batch_kernel(const Tc2DevArgs* __restrict__ args, int N) {
  const Tc2DevArgs& a = args[blockIdx.y];
  const int R = a.R_dev ? *a.R_dev : a.R;
  if (R <= 0) return;
  pack_v2(a.V, a.ldv, a.vmap, R, N, a.n, a.ntiles, const_cast<__nv_bfloat16*>(a.Vp), blockIdx.x,
          gridDim.x);
}

template <int K8, int N, bool BJ>
struct Tc2Inst {
  using S = Tc2Shape<K8, N, BJ>;
  // The split plan counts four CTAs' worth of work per SM.  The ranges it gives also set the
  // rounding of the sums, which tensor memory accumulates with truncation (kTcMaxSplitTiles).
  static constexpr int kPlanOcc = 4;
  static void prime() {
    static std::once_flag once;
    std::call_once(once, [] {
      auto fn = kmv_tc2_kernel<K8, N, BJ>;
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
      cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    });
  }
  static cudaError_t launch(TcLaunch& L, cudaStream_t s) {
    KmvPlan p = L.nsplit > 0 ? plan_split_forced(L.n, kT2BM, N, 4, L.nsplit)
                             : plan_split(L.n, kT2BM, N, 4, L.num_sms * kPlanOcc);
    p = tc_bound_split(p, L.n, kT2BM, N, kT2BN);
    const size_t pbytes = p.nsplit > 1 ? (size_t)p.n_rb * p.nsplit * N * kT2BM * 4 : 0;
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
    const long long ntiles = (L.n + kT2BN - 1) / kT2BN;
    if (!L.v_packed) launch_pack_v(L, N, ntiles, s);
    Tc2DevArgs a;
    a.A_hi = L.X_hi;
    a.A_lo = L.X_lo;
    a.B = L.X_b;
    a.bneg = L.bneg;
    a.Vp = static_cast<const __nv_bfloat16*>(L.Vp);
    a.V = static_cast<const float*>(L.V);
    a.ldv = L.ldv;
    a.vmap = L.vmap;
    a.R = L.R;
    a.R_dev = nullptr;
    a.U = static_cast<float*>(L.U);
    a.ldu = L.ldu;
    a.umap = L.umap;
    a.n = L.n;
    a.params = L.params;
    a.tiles_per_split = (int)((ntiles + p.nsplit - 1) / p.nsplit);
    a.nsplit = (int)((ntiles + a.tiles_per_split - 1) / a.tiles_per_split);
    a.ntiles = (int)ntiles;
    a.partials = static_cast<float*>(L.partials);
    a.counters = L.counters;
    a.status = L.status;
    prime();
    const int nrb = (int)((L.n + kT2BM - 1) / kT2BM);
    kmv_tc2_kernel<K8, N, BJ><<<nrb * a.nsplit, S::THREADS, S::SMEM, s>>>(a);
    return cudaGetLastError();
  }
};

template <int K8, bool BJ>
static cudaError_t tc2_dispatch_n(TcLaunch& L, cudaStream_t s) {
  const int r = std::max(L.R, L.n_min);
  if (r <= 16) return Tc2Inst<K8, 16, BJ>::launch(L, s);
  if (r <= 32) return Tc2Inst<K8, 32, BJ>::launch(L, s);
  if (r <= 64) return Tc2Inst<K8, 64, BJ>::launch(L, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_kmv_tc2(TcLaunch& L, cudaStream_t s) {
  if (L.R < 1 || L.R > 64 || !L.X_hi || !L.X_lo || !L.X_b) return cudaErrorInvalidValue;
  switch (L.DP) {
    case 2:
    case 4: return tc2_dispatch_n<8, false>(L, s);
    case 8: return tc2_dispatch_n<8, true>(L, s);
    case 16: return tc2_dispatch_n<16, true>(L, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_prescale_mixed(const PsiArg& pa, double* psi_dev, const float* X, float* xhat,
                                  long long n, long long ld128, int d, int DP, bool aug,
                                  DevParams* P, float* bneg, float* X_hi, float* X_lo, float* X_b,
                                  PackV pv, int num_sms, cudaStream_t s) {
  const int blocks = (int)std::min<long long>(ld128 / 128, 8LL * num_sms);
  pv.first_cta = blocks;
  const int more = pv.V ? pack_v_ctas(n, pv.N, 128, num_sms) : 0;
  auto go = [&](auto kernel) {
    kernel<<<blocks + more, 128, 0, s>>>(pa, psi_dev, X, xhat, n, ld128, d, aug ? 1 : 0, P, bneg,
                                         X_hi, X_lo, X_b, pv);
  };
  switch (DP) {
    case 2: go(prescale_mixed_kernel<2>); break;
    case 4: go(prescale_mixed_kernel<4>); break;
    case 8: go(prescale_mixed_kernel<8>); break;
    case 16: go(prescale_mixed_kernel<16>); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Batched launches: many problems' K V in one launch (padded d <= 8, K8 = 8, b_j in the
// epilogue, the rows packed without the augmented column).
// ---------------------------------------------------------------------------------------
size_t tc2_batch_args_bytes(int B) { return sizeof(Tc2DevArgs) * (size_t)B; }

cudaError_t tc2_batch_upload_args(const TcLaunch* L, int B, void* args_dev, cudaStream_t s) {
  std::vector<Tc2DevArgs> h((size_t)B);
  for (int b = 0; b < B; ++b) {
    const TcLaunch& l = L[b];
    if (l.DP > 8 || l.nsplit < 1) return cudaErrorInvalidValue;
    Tc2DevArgs& a = h[b];
    const long long ntiles = (l.n + kT2BN - 1) / kT2BN;
    a.A_hi = l.X_hi;
    a.A_lo = l.X_lo;
    a.B = l.X_b;
    a.bneg = l.bneg;
    a.Vp = static_cast<const __nv_bfloat16*>(l.Vp);
    a.V = static_cast<const float*>(l.V);
    a.ldv = l.ldv;
    a.vmap = l.vmap;
    a.R = l.R;
    a.R_dev = l.R_dev;
    a.U = static_cast<float*>(l.U);
    a.ldu = l.ldu;
    a.umap = l.umap;
    a.n = l.n;
    a.params = l.params;
    a.tiles_per_split = (int)((ntiles + l.nsplit - 1) / l.nsplit);
    a.nsplit = (int)((ntiles + a.tiles_per_split - 1) / a.tiles_per_split);
    if (a.nsplit != l.nsplit || a.tiles_per_split > kTcMaxSplitTiles) return cudaErrorInvalidValue;
    a.ntiles = (int)ntiles;
    a.partials = static_cast<float*>(l.partials);
    a.counters = l.counters;
    a.status = l.status;
  }
  return cudaMemcpyAsync(args_dev, h.data(), sizeof(Tc2DevArgs) * (size_t)B,
                         cudaMemcpyHostToDevice, s);
}

template <int N>
static void tc2_batch_prime() {
  static std::once_flag once;
  std::call_once(once, [] {
    auto fn = kmv_tc2_batch_kernel<8, N, true>;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)Tc2Shape<8, N, true>::SMEM);
    cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  });
}

void prime_kmv_tc2_batch() {
  tc2_batch_prime<16>();
  tc2_batch_prime<32>();
}

template <int N>
static cudaError_t tc2_batch_launch(const Tc2DevArgs* args, int B, const int4* items,
                                    int n_items, cudaStream_t s) {
  tc2_batch_prime<N>();
  pack_v_batch_kernel<<<dim3(64, (unsigned)B), 256, 0, s>>>(args, N);
  if (n_items > 0)
    kmv_tc2_batch_kernel<8, N, true><<<n_items, Tc2Shape<8, N, true>::THREADS,
                                       Tc2Shape<8, N, true>::SMEM, s>>>(
        args, items);
  return cudaGetLastError();
}

cudaError_t launch_kmv_tc2_batch(const void* args_dev, int B, const int4* items, int n_items,
                                 int R_max, cudaStream_t s) {
  const Tc2DevArgs* args = static_cast<const Tc2DevArgs*>(args_dev);
  if (B < 1 || R_max < 1 || R_max > 32) return cudaErrorInvalidValue;
  return R_max <= 16 ? tc2_batch_launch<16>(args, B, items, n_items, s)
                     : tc2_batch_launch<32>(args, B, items, n_items, s);
}

}  // namespace ulisse
