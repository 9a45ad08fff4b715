// Mixed-precision tile-generating K V with the cross term on the tensor cores too.
//
// For a block of 128 output rows I and a 32-point tile J:
//   1. C_IJ = A_I B_J^T on the tensor cores (kind::tf32).  With padded d = 2 or 4 the rows
//      carry the column term too,
//          A_i = [x^_i, 1],  B_j = [2 c1 x^_j, b_j],   b_j = -c1 |x^_j|^2, c1 = log2(e)/2,
//      so that C_ij = 2 c1 x^_i . x^_j + b_j in one 8-wide K step; with padded d = 8 or 16
//      the rows are A_i = x^_i, B_j = 2 c1 x^_j (K = d: the augmented column would cost a
//      whole further K step, three MMAs per tile on the one issuing thread that paces the
//      kernel) and the epilogue adds b_j.  Both sides split into a TF32 high part and the
//      remainder, three products (Ah Bh + Ah Bl + Al Bh), FP32 accumulation into a 32-column
//      tensor-memory buffer;
//   2. the epilogue warps read C back (tcgen05.ld) and form
//          k_ij = exp2(a_i + C_ij)  or  exp2((a_i + b_j) + C_ij),
//          a_i = log2(sigma^2) - c1 |x^_i|^2
//      (one or two FADDs and one ex2 per entry), split k into BF16 high and low parts and
//      store them over C's own columns (tcgen05.st);
//   3. U_I += K_IJ V_J on the tensor cores with V split into BF16 high + low parts (three
//      products), FP32 accumulation in tensor memory, as in the FP32-pipe variant.
// The TF32 images of A and B (high and low parts, K-major canonical, 32-point tiles back to
// back so that four tiles form the 128-row A operand) are written once per parameter value by
// pack_x_tf32_kernel; B's tiles and V's tiles each lie contiguously with all their parts, so
// that a tile is two bulk copies.  Roles: warp 0 copies (the A image once, then B_J, b_J and
// V_J into a ring of 3 to 8 stages) and issues the MMAs; eight epilogue warps make the kernel
// values, in two sets of four (one per tensor-memory lane quadrant) that take alternate tiles
// whole, so that each wait and hand-off covers 32 entries per thread.  Three C/K buffers (two
// when the accumulator takes 64 columns); a buffer is refilled only after the MMAs that read it
// have completed, and the stage of that tile is refilled at the same moment, so the copies need
// no barrier and no warp of their own.  Every wait is bounded.  The split j range, the
// fixed-order fix-up of the partial sums and the FP32 diagonal term lambda V are those of the
// FP32-pipe variant.
//
// What bounds it: the issue slots of the epilogue's instruction stream and, next to them, the
// chain C -> epilogue -> contraction -> refill, whose middle is one warp's instructions.  That
// warp runs its loop warp-uniformly and elects a lane only for the issuing instructions: the
// descriptors then live in uniform registers.  With a separate copying warp and one divergent
// lane issuing (moving every descriptor to uniform registers per MMA) a product at n = 50,000,
// d = 8, 17 columns took 1.046 ms; nine warps instead of ten also raise the register budget from
// 48 to 56, so that the high and low parts get registers of their own.  Now 0.78 ms.
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "kmv_kernel.cuh"
#include "prescale.cuh"
#include "tc_common.cuh"

namespace ulisse {

constexpr int kT2BN = 32;
constexpr int kT2BM = 128;
constexpr int kT2Threads = 288;    // warp 0 copies and MMAs, warps 1-8 epilogue
constexpr uint32_t kT2Cols = 128;  // tensor-memory columns per CTA

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
    float* __restrict__ Alo, float* __restrict__ Bt) {
  constexpr int K8 = DP >= 8 ? DP : 8;
  __shared__ InvLength s;
  unpack_params(pa, psi_dev, d, P, s);
  const float two_c1 = 2.f * (float)(0.5 * 1.4426950408889634);   // 2 c1f
  for (long long j = blockIdx.x * 128LL + threadIdx.x; j < rows; j += gridDim.x * 128LL) {
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
  static constexpr uint32_t A_BYTES = kT2BM * K8 * 4;   // one part of the A_I image
  static constexpr uint32_t XB_BYTES = kT2BN * K8 * 4;  // one part of the B_J image
  static constexpr uint32_t V_BYTES = N * kT2BN * 2;    // one part of the BF16 V_J tile
  static constexpr uint32_t BN_BYTES = BJ ? kT2BN * 4 : 0;   // b_J
  static constexpr uint32_t X_COPY = 2 * XB_BYTES + BN_BYTES;   // B_J high | remainder | b_J
  static constexpr uint32_t OFF_BN = 2 * XB_BYTES;              // within a stage
  static constexpr uint32_t OFF_V = X_COPY;
  static constexpr uint32_t STAGE_BYTES = X_COPY + 2 * V_BYTES;
  // as many stages (at most 8) as let four CTAs fit in shared memory (~54 KB each), at least 3
  static constexpr int ST_FIT = (int)((54u * 1024u - 2 * A_BYTES) / STAGE_BYTES);
  static constexpr int ST = ST_FIT > 8 ? 8 : ST_FIT < 3 ? 3 : ST_FIT;
  static constexpr uint32_t OFF_STAGES = 2 * A_BYTES;
  static constexpr uint32_t OFF_BARS = OFF_STAGES + ST * STAGE_BYTES;
  // C/K buffers of 32 columns: three while they fit beside the accumulator, else two
  static constexpr int NB = (3 * 32 + N <= (int)kT2Cols) ? 3 : 2;
  // full per stage; a_full; c_full per tile mod 6 (so that each barrier serves one
  // epilogue set and its phases are waited in order); k_full, b_free per buffer; done
  static constexpr int NCF = 6;
  static constexpr int NBARS = ST + 1 + NCF + 2 * NB + 1;
  static constexpr uint32_t SMEM = OFF_BARS + NBARS * 8 + 64;
  static constexpr uint32_t COL_U = NB * 32;   // after the C/K buffers
  static_assert(COL_U + N <= kT2Cols, "tensor memory layout exceeds the allocation");
  static_assert(STAGE_BYTES % 16 == 0 && A_BYTES % 16 == 0 && XB_BYTES % 16 == 0 &&
                    X_COPY % 16 == 0,
                "bulk copies and descriptors need 16-byte alignment");
  static_assert(NCF % NB == 0, "a c_full barrier belongs to one buffer");
};

template <int NH>
__device__ inline void t2_ld_cols(uint32_t taddr, float (&v)[NH]) {
  if constexpr (NH == 8) {
    tc::tmem_ld8(taddr, v);
  } else if constexpr (NH == 16) {
    tc::tmem_ld16(taddr, v);
  } else {
    // two 16-column loads: a 32-register load does not fit the 48-register budget
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
  constexpr int ST = S::ST;
  constexpr int NB = S::NB;
  constexpr int NH = N / 2;
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t smem0 = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::OFF_BARS);
  uint64_t* full = bars;
  uint64_t* a_full = bars + ST;
  uint64_t* c_full = a_full + 1;
  uint64_t* k_full = c_full + S::NCF;
  uint64_t* b_free = k_full + NB;
  uint64_t* done = b_free + NB;
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

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) mbar_init(&full[s], 1);
    mbar_init(a_full, 1);
    for (int c = 0; c < S::NCF; ++c) mbar_init(&c_full[c], 1);
    for (int b = 0; b < NB; ++b) {
      mbar_init(&k_full[b], 4);   // the four epilogue warps of the tile's set
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
  int issued = 0;   // tiles whose copies were started (warp 0)

  if (warp == 0) {
    // ------ copies and MMAs: C = x^_I x^_J^T, then U += K V; one elected lane issues, the
    //        whole warp runs the loop, so that descriptors and addresses stay warp-uniform ------
    constexpr uint32_t idesc_c = tc::instr_desc(2, kT2BM, kT2BN);   // TF32
    constexpr uint32_t idesc_u = tc::instr_desc(1, kT2BM, N);       // BF16
    constexpr uint32_t sbo_x = (K8 / 4) * 128;
    const uint64_t dAh = tc::smem_desc(smem0, 128, sbo_x);
    const uint64_t dAl = tc::smem_desc(smem0 + S::A_BYTES, 128, sbo_x);
    const uint64_t dB0 = tc::smem_desc(smem0 + S::OFF_STAGES, 128, sbo_x);
    const uint64_t dV0 = tc::smem_desc(smem0 + S::OFF_STAGES + S::OFF_V, 128, 512);
    const float* srcX = a.B + (long long)tile_begin * tc2_b_stride(K8);
    const __nv_bfloat16* srcV = a.Vp + (long long)tile_begin * 2 * N * kT2BN;
    auto copy_tile = [&](int p, int s) {   // elected lane: tile p's B_J (with b_J) and V_J
      unsigned char* st = smem + S::OFF_STAGES + s * S::STAGE_BYTES;
      mbar_arrive_expect_tx(&full[s], S::STAGE_BYTES);
      bulk_g2s(st, srcX + (long long)p * tc2_b_stride(K8), S::X_COPY, &full[s]);
      bulk_g2s(st + S::OFF_V, srcV + (long long)p * 2 * N * kT2BN, 2 * S::V_BYTES, &full[s]);
    };
    auto mma_c = [&](int s, int b, int cf) {   // elected lane: C into buffer b
      const uint64_t dBh = dB0 + (uint64_t)s * (S::STAGE_BYTES >> 4), dBl = dBh + (S::XB_BYTES >> 4);
      const uint32_t dC = tbase + (uint32_t)(b * 32);
#pragma unroll
      for (int term = 0; term < 3; ++term) {
        const uint64_t A = term == 2 ? dAl : dAh;
        const uint64_t B = term == 1 ? dBl : dBh;
#pragma unroll
        for (int ks = 0; ks < K8 / 8; ++ks)
          tc::mma_tf32(dC, A + 16u * ks, B + 16u * ks, idesc_c, (term | ks) != 0);
      }
      tc::commit(&c_full[cf]);
    };
    const int pre = min(ST, nt);
    if (tc::elect_one()) {
      mbar_arrive_expect_tx(a_full, 2 * S::A_BYTES);
      bulk_g2s(smem, a.A_hi + row0 * K8, S::A_BYTES, a_full);
      bulk_g2s(smem + S::A_BYTES, a.A_lo + row0 * K8, S::A_BYTES, a_full);
      for (int p = 0; p < pre; ++p) copy_tile(p, p);
    }
    issued = pre;
    bool ok = tc::warp_wait_uniform(smem_u32(a_full), 0);
    // s_c, cf: stage and c_full barrier of the next tile whose C is issued; s, b: stage and
    // buffer of tile p
    int s_c = 0, ph_c = 0, cf = 0;
    for (int p = 0; p < NB && p < nt && ok; ++p) {
      ok = tc::warp_wait_uniform(full0 + 8u * s_c, ph_c);
      tc::fence_after();
      if (ok && tc::elect_one()) mma_c(s_c, p, cf);
      __syncwarp();
      if (++s_c == ST) { s_c = 0; ph_c ^= 1; }
      if (++cf == S::NCF) cf = 0;
    }
    int s = 0, b = 0, ph_b = 0;
#pragma unroll 1
    for (int p = 0; p < nt && ok; ++p) {
      ok = tc::warp_wait_uniform(k_full0 + 8u * b, ph_b);
      if (!ok) break;
      tc::fence_after();
      const bool more_c = p + NB < nt, more_v = p + ST < nt;
      if (tc::elect_one()) {
        const uint64_t dVh = dV0 + (uint64_t)s * (S::STAGE_BYTES >> 4), dVl = dVh + (S::V_BYTES >> 4);
        const uint32_t kcol = tbase + (uint32_t)(b * 32);
#pragma unroll
        for (int term = 0; term < 3; ++term) {
          const uint32_t A = kcol + (term == 2 ? 8u : 0u);   // K high | K low per 16 points
          const uint64_t B = term == 1 ? dVl : dVh;
#pragma unroll
          for (int ks = 0; ks < kT2BN / 16; ++ks)
            tc::mma_bf16_ts(tbase + S::COL_U, A + ks * 16, B + 16u * ks, idesc_u, (p | term | ks) != 0);
        }
        // buffer b takes tile p + NB's C, and stage s tile p + ST's operands, only after these
        // MMAs have read its K and V
        if (more_c || more_v) tc::commit(&b_free[b]);
      }
      __syncwarp();
      if (more_c || more_v) {
        ok = tc::warp_wait_uniform(b_free0 + 8u * b, ph_b);
        if (ok && more_c) {
          ok = tc::warp_wait_uniform(full0 + 8u * s_c, ph_c);
          tc::fence_after();
          if (ok && tc::elect_one()) mma_c(s_c, b, cf);
          __syncwarp();
          if (++s_c == ST) { s_c = 0; ph_c ^= 1; }
          if (++cf == S::NCF) cf = 0;
        }
        if (ok && more_v) {
          if (tc::elect_one()) copy_tile(p + ST, s);
          __syncwarp();
          issued = p + ST + 1;
        }
      }
      if (++s == ST) s = 0;
      if (++b == NB) { b = 0; ph_b ^= 1; }
    }
    if (!ok) *s_fail = 1;
    if (tc::elect_one()) tc::commit(done);
    __syncwarp();
  } else {
    // ------ epilogue: 8 warps; warp (lane quadrant eq, set h) takes the tiles h, h + 2, ...
    //        with all 32 of their columns ------
    const int eq = warp & 3;
    const int half = (warp - 1) >> 2;   // tile set; also the half of U it reads back
    const int il = eq * 32 + lane;
    const long long i = row0 + il;
    const uint32_t lane_base = (uint32_t)(eq * 32) << 16;
    const float ai = a.params->c0f + a.bneg[i];   // bneg covers the padded rows (zero there)
    bool ok = true;
    int s = half % ST, ph_s = 0, b = half % NB, cf = half, ph_cf = 0;
#pragma unroll 1
    for (int lt = half; lt < nt; lt += 2) {
      ok = tc::warp_wait_uniform(c_full0 + 8u * cf, ph_cf);
      // b_J is read from the stage: wait for its copy too (the stage is refilled only after
      // this tile's contraction, which waits for this warp's K)
      if constexpr (BJ) ok = ok && tc::warp_wait_uniform(full0 + 8u * s, ph_s);
      if (!ok) break;
      tc::fence_after();
      const float4* bj = reinterpret_cast<const float4*>(smem + S::OFF_STAGES + s * S::STAGE_BYTES +
                                                         S::OFF_BN);
      // all 32 columns of C in one tensor-memory round trip; each pair's K high and low parts
      // are written back into the pair's own registers (no extra registers live)
      const uint32_t ccol = tbase + lane_base + (uint32_t)(b * 32);
      uint32_t c[32];
      tc::tmem_ld16x2(ccol, c);
      // two entries per packed FP32x2 instruction (FADD2 / FFMA2, the same rounding as the
      // scalar forms)
      const float2 ai2 = make_float2(ai, ai);
      const float2 minus1 = make_float2(-1.f, -1.f);
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        uint32_t hi[8], lo[8];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
          if constexpr (BJ) b4 = bj[4 * hh + g];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int e0 = 16 * hh + 4 * g + 2 * q;
            // the exponent is <= log2 sigma^2 up to rounding (about 1e-6 relative in k)
            float2 e = ai2;
            if constexpr (BJ) e = __fadd2_rn(e, q == 0 ? make_float2(b4.x, b4.y) : make_float2(b4.z, b4.w));
            e = __fadd2_rn(e, make_float2(__uint_as_float(c[e0]), __uint_as_float(c[e0 + 1])));
            const float2 k = make_float2(ex2_approx(e.x), ex2_approx(e.y));
            const __nv_bfloat162 h = __floats2bfloat162_rn(k.x, k.y);
            const float2 r = __ffma2_rn(__bfloat1622float2(h), minus1, k);   // k - high part
            const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
            hi[2 * g + q] = *reinterpret_cast<const uint32_t*>(&h);
            lo[2 * g + q] = *reinterpret_cast<const uint32_t*>(&l);
          }
        }
        // columns [16 hh, 16 hh + 16): high parts, then low parts (the A operand of the
        // contraction's k-step hh)
        tc::tmem_st8(ccol + 16 * hh, hi);
        tc::tmem_st8(ccol + 16 * hh + 8, lo);
      }
      tc::tmem_wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&k_full[b]);
      s += 2;
      if (s >= ST) { s -= ST; ph_s ^= 1; }
      b += 2;
      if (b >= NB) b -= NB;
      cf += 2;
      if (cf >= S::NCF) { cf -= S::NCF; ph_cf ^= 1; }
    }
    if (!ok) *s_fail = 1;
    const bool fin = ok && tc::warp_wait_uniform(smem_u32(done), 0);
    ok = __all_sync(0xffffffffu, fin && !*s_fail);
    if (ok && nt > 0) {
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
      (void)mbar_wait_bounded(a_full, 0);
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
  for (int idx = tid; idx < R * kT2BM; idx += kT2Threads) {
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
__global__ void __launch_bounds__(kT2Threads, 4) kmv_tc2_kernel(const Tc2DevArgs a) {
  const int rb = blockIdx.x / a.nsplit;
  tc2_body<K8, N, BJ>(a, rb, blockIdx.x - rb * a.nsplit, a.R);
}

// Many problems in one launch: CTA b takes work item items[b] = (problem, row block, split)
// with that problem's arguments; a problem with no live columns is skipped.
template <int K8, int N, bool BJ>
__global__ void __launch_bounds__(kT2Threads, 4) kmv_tc2_batch_kernel(
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
  const long long ntiles = a.ntiles;
  const long long per_tile = (long long)N * kT2BN;
  __nv_bfloat16* Vp = const_cast<__nv_bfloat16*>(a.Vp);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < ntiles * per_tile;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long t = idx / per_tile;
    const int rem = (int)(idx - t * per_tile);
    const int r = rem / kT2BN, jj = rem - r * kT2BN;
    const long long j = t * kT2BN + jj;
    const float v = (r < R && j < a.n) ? a.V[(long long)a.vmap[r] * a.ldv + j] : 0.f;
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    const __nv_bfloat16 l = __float2bfloat16_rn(v - __bfloat162float(h));
    const long long off = t * 2 * per_tile + tc::canon_offset(r, jj, 2, kT2BN / 8) / 2;
    Vp[off] = h;
    Vp[off + per_tile] = l;
  }
}

template <int K8, int N, bool BJ>
struct Tc2Inst {
  using S = Tc2Shape<K8, N, BJ>;
  // CTAs per SM: shared memory, tensor memory (512 columns) and the launch bound.
  static int occupancy() {
    static int occ = -1;
    static std::once_flag once;
    std::call_once(once, [] {
      auto fn = kmv_tc2_kernel<K8, N, BJ>;
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
      cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
      int dev = 0, smem_sm = 0;
      cudaGetDevice(&dev);
      if (cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
          cudaSuccess)
        smem_sm = 228 * 1024;
      const int by_smem = smem_sm / (int)(S::SMEM + 1024);
      occ = std::max(1, std::min({by_smem, (int)(512 / kT2Cols), 4}));
    });
    return occ;
  }
  static cudaError_t launch(TcLaunch& L, cudaStream_t s) {
    KmvPlan p = L.nsplit > 0 ? plan_split_forced(L.n, kT2BM, N, 4, L.nsplit)
                             : plan_split(L.n, kT2BM, N, 4, L.num_sms * occupancy());
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
    launch_pack_v(L, N, ntiles, s);
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
    (void)occupancy();
    const int nrb = (int)((L.n + kT2BM - 1) / kT2BM);
    kmv_tc2_kernel<K8, N, BJ><<<nrb * a.nsplit, kT2Threads, S::SMEM, s>>>(a);
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
                                  int num_sms, cudaStream_t s) {
  const int blocks = (int)std::min<long long>(ld128 / 128, 8LL * num_sms);
  auto go = [&](auto kernel) {
    kernel<<<blocks, 128, 0, s>>>(pa, psi_dev, X, xhat, n, ld128, d, aug ? 1 : 0, P, bneg, X_hi,
                                  X_lo, X_b);
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
    kmv_tc2_batch_kernel<8, N, true><<<n_items, kT2Threads, Tc2Shape<8, N, true>::SMEM, s>>>(
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
