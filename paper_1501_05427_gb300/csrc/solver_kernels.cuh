// Vector kernels of the solver path: parameter unpack + prescale, Hutchinson probes,
// batched CG (Algorithm 1) with the ULISSE truncation and reweighting (Sec. 4), and the
// SGLD update (Sec. 2.1).  Vectors are T (float or double); every scalar recurrence --
// e^T e, d^T K d, alpha, beta, the early-stop test and the ULISSE weights -- is FP64.
#pragma once

#include <cooperative_groups.h>

#include "prescale.cuh"
#include "ulisse_internal.cuh"

namespace ulisse {

constexpr int kCgChunkNT = 256;   // threads of the CG start
constexpr int kMaxCgChunks = 64;  // row ranges with a partial sum each, per column

// ------------------------------------------------------------------------------------
// a2: probes r_j (column j = 1..nr of B): +-1 from the top bit, or N(0,1) by Box-Muller,
// element i of probe j from Philox counter (i, j, epoch, 1) keyed by (seed, 0).
// ------------------------------------------------------------------------------------
// Step of a chain run from a CUDA graph: the kernels of the graph read the step number,
// the step size and the trace slot from here (one graph serves every step of the chain);
// the SGLD update, the graph's last kernel, advances k.
struct ChainSlot {
  long long k;                  // index of the step within the chain call
  unsigned long long step0;     // step number of k = 0
  const double* eps;            // step sizes, one per k
  double* trace;                // NULL or p doubles per k
};

template <typename T>
__global__ void probes_kernel(T* __restrict__ B, long long ld, long long n, int nr, int kind,
                              unsigned long long seed, unsigned long long epoch,
                              const ChainSlot* __restrict__ cs = nullptr, int refresh = 1) {
  if (cs) epoch = (cs->step0 + (unsigned long long)cs->k) / (unsigned long long)refresh;
  const int j = blockIdx.y + 1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    uint64_t w[4];
    philox4x64_10((uint64_t)i, (uint64_t)j, epoch, kPurposeProbe, seed, 0, w);
    T v;
    if (kind == 0) v = (w[0] >> 63) ? T(-1) : T(1);
    else v = (T)box_muller(w[0], w[1]);
    B[(long long)j * ld + i] = v;
  }
}

template <typename T>
struct CgArgs {
  T* S;          // iterates s_m
  T* E;          // residuals e_m
  T* D;          // directions d_m
  const T* KD;   // K d_m (or K s_0 before the first iteration)
  const T* B;    // right-hand sides
  T* SE;         // ULISSE estimates
  long long n, ld;
  ColState* st;
  ColState* st_next;     // state written by an iteration, committed by compact_kernel
  const int* live;
  double* part1;         // the CG start's partial sums per (column, chunk): residual
  double* part2;         // ... and right-hand side
  int nchunk;            // CTAs per column of the CG start
  long long chunk;       // rows per CTA
  int ordered;           // FP64: rows per chunk of cg_ordered_dot's sums, 0: sums in any order
  int o_chunks, o_per;   // ... the column's chunks, and those of a CTA (chunk rows)
  double alpha_thr, eps, beta;
  int max_iter;
  int has_s0;
  unsigned long long seed, step;
  const ChainSlot* cs;   // when set, the step number comes from the chain slot
  const int* n_live;     // batched launches: this problem's live column count
  // Warm-started solves (Sec. 5.1's probe reuse): when warm_refresh > 0, S holds the final
  // CG iterates of the previous step's solve of every column (valid while *warm_valid is
  // nonzero).  Column 0 (y, never changes) starts from its iterate -- or from the learned
  // warm start when y_learned -- and probe columns start from theirs while the probes are
  // unchanged (step % warm_refresh != 0).  The keep-if-better rule still applies.
  int warm_refresh;
  const int* warm_valid;
  int y_learned;
  T* Sbest;              // warm-started solves: per column, the iterate of smallest residual
                         // seen (the start of the next step's solve)
  int* status;
};

// Accepted steps after the early stop: j = 1, 2, ... while u_j < 1/w_j = exp(-beta j).
__device__ inline int draw_J(unsigned long long seed, unsigned long long step, int colid,
                             int est, double beta, int jcap) {
  int J = 0;
  for (int j = 1; j <= jcap; ++j) {
    uint64_t w[4];
    philox4x64_10((uint64_t)j, (uint64_t)colid, step, kPurposeUlisse | ((uint64_t)est << 8),
                  seed, 0, w);
    if (u01_53(w[0]) < exp(-beta * (double)j)) J = j;
    else break;
  }
  return J;
}

// prod_{r=0}^{j} w_r, w_r = exp(beta r).
__device__ inline double weight_product(int j, double beta) {
  double W = 1.0;
  for (int r = 0; r <= j; ++r) W *= exp(beta * (double)r);
  return W;
}

template <typename T>
__device__ inline void chunk_range(const CgArgs<T>& a, int ch, long long* i0, long long* i1) {
  *i0 = (long long)ch * a.chunk;
  *i1 = min(a.n, *i0 + a.chunk);
}

// Whether column c starts from its initial iterate (else from s_0 = 0): every column with
// has_s0; with warm-started solves, column 0 (y) when its start is valid or learned, and the
// probe columns while the probes are unchanged.
template <typename T>
__device__ inline bool init_use_s0(const CgArgs<T>& a, int c) {
  if (a.warm_refresh <= 0) return a.has_s0 != 0;
  const unsigned long long step = a.cs ? a.cs->step0 + (unsigned long long)a.cs->k : a.step;
  const bool valid = *a.warm_valid != 0;
  return (c == 0) ? (a.y_learned || valid)
                  : (valid && step % (unsigned long long)a.warm_refresh != 0);
}

// b^T b and, when use_s0, (b - K s_0)^T (b - K s_0) over rows [i0, i1) of column c (FP64),
// summed over the block; rr = bb otherwise.
template <typename T>
__device__ inline void init_sums(const CgArgs<T>& a, int c, bool use_s0, long long i0,
                                 long long i1, double* red, double* bb, double* rr) {
  const T* b = a.B + c * a.ld;
  const T* ks0 = a.KD + c * a.ld;
  double pb = 0.0, pr = 0.0;
  for (long long i = i0 + threadIdx.x; i < i1; i += kCgChunkNT) {
    const double bi = (double)b[i];
    pb += bi * bi;
    if (use_s0) {
      const double ri = (double)(T)(b[i] - ks0[i]);
      pr += ri * ri;
    }
  }
  *bb = block_sum<kCgChunkNT>(pb, red);
  *rr = use_s0 ? block_sum<kCgChunkNT>(pr, red) : *bb;
}

// The CG start's sums per (chunk, column) when a column spans several chunks (part2: b^T b,
// part1: the residual's); cg_init_kernel adds them in chunk order.
template <typename T>
__global__ void __launch_bounds__(kCgChunkNT) cg_init_dot_kernel(const CgArgs<T> a) {
  __shared__ double red[kCgChunkNT / 32];
  const int c = blockIdx.y, ch = blockIdx.x;
  long long i0, i1;
  chunk_range(a, ch, &i0, &i1);
  double bb, rr;
  init_sums(a, c, init_use_s0(a, c), i0, i1, red, &bb, &rr);
  if (threadIdx.x == 0) {
    a.part2[(long long)c * a.nchunk + ch] = bb;
    a.part1[(long long)c * a.nchunk + ch] = rr;
  }
}

// e_0 = b - K s_0, d_0 = e_0, draws of J; grid (chunk, column).  With one chunk per column
// the CTA forms the sums itself; with several, every CTA of the column adds the partial sums
// of cg_init_dot_kernel in chunk order, so all of them take the same decision.
template <typename T>
__global__ void __launch_bounds__(kCgChunkNT) cg_init_kernel(const CgArgs<T> a) {
  __shared__ double red[kCgChunkNT / 32];
  const int c = blockIdx.y, ch = blockIdx.x;
  ColState& st = a.st[c];
  T* s = a.S + c * a.ld;
  T* e = a.E + c * a.ld;
  T* d = a.D + c * a.ld;
  const T* b = a.B + c * a.ld;
  const T* ks0 = a.KD + c * a.ld;
  const bool warm = a.warm_refresh > 0;
  T* sb = warm ? a.Sbest + c * a.ld : nullptr;
  // with warm-started solves the start comes from Sbest (y_learned: column 0 from S)
  const T* s0 = (warm && !(c == 0 && a.y_learned)) ? sb : s;
  const bool use_s0 = init_use_s0(a, c);
  long long i0, i1;
  chunk_range(a, ch, &i0, &i1);
  // An initial iterate is kept only when it lowers the residual norm below that of s_0 = 0.
  // The choice depends on the parameters, the data and the iterate alone (no random draw),
  // so every estimator built on it stays unbiased.
  double bb, rr;
  if (a.nchunk == 1) {
    init_sums(a, c, use_s0, i0, i1, red, &bb, &rr);
  } else {
    bb = 0.0;
    rr = 0.0;
    for (int k = 0; k < a.nchunk; ++k) {
      bb += a.part2[(long long)c * a.nchunk + k];
      rr += a.part1[(long long)c * a.nchunk + k];
    }
    if (!use_s0) rr = bb;
  }
  const bool keep = use_s0 && rr < bb;
  for (long long i = i0 + threadIdx.x; i < i1; i += kCgChunkNT) {
    const T si = keep ? s0[i] : T(0);
    s[i] = si;
    if (warm) sb[i] = si;
    const T ei = keep ? b[i] - ks0[i] : b[i];
    e[i] = ei;
    d[i] = ei;
  }
  const double ee = keep ? rr : bb;
  const int n_est = st.n_est;
  const bool done = sqrt(ee) < a.eps;
  if (done) {
    for (int t = 0; t < n_est; ++t) {
      T* se = a.SE + (long long)(st.est_off + t) * a.ld;
      for (long long i = i0 + threadIdx.x; i < i1; i += kCgChunkNT) se[i] = s[i];
    }
  }
  if (ch == 0 && threadIdx.x == 0) {
    st.ee = ee;
    st.best_ee = ee;
    st.l = 0;
    st.m = 0;
    st.outcome = 0;
    const unsigned long long step = a.cs ? a.cs->step0 + (unsigned long long)a.cs->k : a.step;
    st.J[0] = draw_J(a.seed, step, st.colid, 0, a.beta, a.max_iter);
    st.J[1] = n_est > 1 ? draw_J(a.seed, step, st.colid, 1, a.beta, a.max_iter) : -1;
    st.phase = done ? kDone : kPre;
  }
}

// One CG iteration (Algorithm 1) on every live column, with the ULISSE bookkeeping, in one
// launch: a cluster of CTAs per column (grid (CTAs of the column, live column)), each on its
// range of rows, with two sums over the cluster:
//   d^T K d         -> alpha = e^T e / d^T K d
//   s += alpha d, e -= alpha K d, the ULISSE tail term; e'^T e'
//   the early-stop / convergence / max_iter decisions (every CTA of a column reaches the same
//   ones), the copy of s_l into the estimators at the early stop, d = e' + beta d, and the new
//   column state (into st_next; the compaction commits it).
// The increment delta_{m+1} = alpha_m d_m is added with weight prod_{r<=j} w_r to every
// estimator whose J >= j (j = m+1-l) once the early stop at l has been reached.
//
// What bounds it: latency (cluster barriers, L2 round trips) and, per scalar, the FP64 pipe (64
// clocks per warp instruction and SM quarter): the scalars are formed by one warp of each CTA
// and read from shared memory, not by every thread.  As three launches that exchanged their
// sums through global memory, with every thread forming the scalars, an iteration took 49 us at
// n = 50,000, 17 columns, and 26 us at n = 1,030, 101 columns in FP64.
constexpr int kCgNT = 512;
constexpr int kCgMaxCluster = 8;

// 16 bytes of a vector.
template <typename T>
struct alignas(16) CgVec {
  static constexpr int N = 16 / (int)sizeof(T);
  T v[N];
};

// The padding rows [n, ld) of every column hold zeros (the products read whole tiles) and stay
// zero whatever the scalars: an infinite step would make 0 * inf of them.
template <typename T>
__device__ __forceinline__ void cg_keep_padding(CgVec<T>& x, long long i, long long n) {
  if ((i + 1) * CgVec<T>::N > n) {
#pragma unroll
    for (int q = 0; q < CgVec<T>::N; ++q)
      if (i * CgVec<T>::N + q >= n) x.v[q] = T(0);
  }
}

// Sum of v over the cluster's CTAs, in a fixed order, valid in warp 0.  slot: this use's shared
// double (the peers read it: one slot per use within a launch).
__device__ inline double cluster_sum_warp0(double v, double* red, double* slot) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  v = warp_sum(v);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = warp_sum(lane < kCgNT / 32 ? red[lane] : 0.0);
    if (lane == 0) *slot = v;
  }
  cl.sync();
  if (warp == 0) {
    const int nc = (int)cl.num_blocks();
    v = lane < nc ? *cl.map_shared_rank(slot, lane) : 0.0;
#pragma unroll
    for (int o = kCgMaxCluster / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    v = __shfl_sync(0xffffffffu, v, 0);
  }
  return v;
}

// FP64 iterations whose sums keep one order, whatever the cluster: kCgChunkNT threads take every
// kCgChunkNT'th row of a chunk of a.ordered rows, then the warps' and the chunks' sums are added one
// by one.  A CTA takes as many chunks as its rows hold, two at a time.  A truncated solve's estimates
// follow the rounding of these sums, so it is part of the result.  parts: a shared double per chunk
// of the CTA (the peers read them).  The sum is valid in warp 0.
template <typename T>
__device__ inline double cg_ordered_dot(const CgArgs<T>& a, const T* x, const T* y, int ch,
                                        double* red, double* parts) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  constexpr int kWarps = kCgChunkNT / 32, kGroups = kCgNT / kCgChunkNT;
  const int tid = threadIdx.x, g = tid / kCgChunkNT, lane = tid & 31;
  const int rows = a.ordered, per = a.o_per;
  const long long at = (long long)ch * a.chunk;
  x += at;
  y += at;
  const int left = (int)min(a.chunk, max(a.n - at, 0LL));   // the CTA's rows
#pragma unroll 1
  for (int q0 = 0; q0 < per; q0 += kGroups) {
    const int q = q0 + g, end = min(left, (q + 1) * rows);
    double p = 0.0;
#pragma unroll 4
    for (int i = q * rows + tid % kCgChunkNT; i < end; i += kCgChunkNT)
      p += (double)x[i] * (double)y[i];
    p = warp_sum(p);
    if (lane == 0) red[tid >> 5] = p;
    __syncthreads();
    if (tid % kCgChunkNT == 0 && q < per) {
      double t = 0.0;
      for (int w = 0; w < kWarps; ++w) t += red[g * kWarps + w];
      parts[q] = t;
    }
    if (q0 + kGroups < per) __syncthreads();
  }
  cl.sync();
  double t = 0.0;
  if (tid < 32) {
    if (per == 1) {
      for (int k = 0; k < a.o_chunks; ++k) t += *cl.map_shared_rank(parts, k);
    } else {
      for (int k0 = 0; k0 < a.o_chunks; k0 += 32) {
        const int k = k0 + lane;
        const double v = k < a.o_chunks ? *cl.map_shared_rank(parts + k % per, k / per) : 0.0;
        for (int l = 0; l < min(32, a.o_chunks - k0); ++l) t += __shfl_sync(0xffffffffu, v, l);
      }
    }
  }
  return t;
}

// The scalars warp 0 hands to the CTA.
template <typename T>
struct CgShared {
  double red[kCgNT / 32];
  double slot[2];
  double parts[2][kMaxCgChunks / kCgMaxCluster];   // ordered sums
  T al, w0, w1, bt;
  int breakdown, copy_s, better, done;
};

// One column's iteration; ch: this CTA's rank in the column's cluster, li: its live-list index.
template <typename T>
__device__ inline void cg_round_body(const CgArgs<T>& a, int ch, int li, CgShared<T>& sh) {
  using V = CgVec<T>;
  constexpr int VN = V::N;
  const int tid = threadIdx.x, lane = tid & 31;
  const bool warp0 = tid < 32;
  const int c = a.live[li];
  const ColState st = a.st[c];
  const long long col = c * a.ld;
  // rows in vectors of 16 bytes, the last one padded
  const long long nv = (a.n + VN - 1) / VN, per = a.chunk / VN;
  const long long v0 = min(nv, ch * per), v1 = min(nv, v0 + per);
  V* s = reinterpret_cast<V*>(a.S + col);
  V* e = reinterpret_cast<V*>(a.E + col);
  V* d = reinterpret_cast<V*>(a.D + col);
  const V* kd = reinterpret_cast<const V*>(a.KD + col);
  V* se0 = reinterpret_cast<V*>(a.SE + (long long)st.est_off * a.ld);
  V* se1 = se0 + a.ld / VN;

  const bool ordered = sizeof(T) == 8 && a.ordered > 0;
  double dKd;
  if (ordered) {
    dKd = cg_ordered_dot(a, a.D + col, a.KD + col, ch, sh.red, sh.parts[0]);
  } else {
    double p = 0.0;
#pragma unroll 4
    for (long long i = v0 + tid; i < v1; i += kCgNT) {
      const V di = d[i], ki = kd[i];
#pragma unroll
      for (int q = 0; q < VN; ++q) p += (double)di.v[q] * (double)ki.v[q];
    }
    dKd = cluster_sum_warp0(p, sh.red, &sh.slot[0]);
  }
  if (warp0) {
    const bool bad = !(dKd > 0.0) || !isfinite(dKd);
    const double al = bad ? 0.0 : st.ee / dKd;
    T w0 = T(0), w1 = T(0);
    const int j = st.m + 1 - st.l;
    if (!bad && st.phase == kTail && (st.J[0] >= j || (st.n_est > 1 && st.J[1] >= j))) {
      // prod_{r <= j} exp(beta r) in the order of weight_product, the exponentials one per lane
      double W = 1.0;
      if (j < 32) {
        const double w = exp(a.beta * (double)lane);
        for (int r = 0; r <= j; ++r) W *= __shfl_sync(0xffffffffu, w, r);
      } else {
        W = weight_product(j, a.beta);
      }
      const double Wa = W * al;
      if (st.J[0] >= j) w0 = (T)Wa;
      if (st.n_est > 1 && st.J[1] >= j) w1 = (T)Wa;
    }
    if (lane == 0) {
      sh.breakdown = bad;
      sh.al = (T)al;
      sh.w0 = w0;
      sh.w1 = w1;
    }
  }
  __syncthreads();
  if (sh.breakdown) {
    // K is not positive definite along d, or a value is not finite
    if (st.phase == kPre)
      for (int t = 0; t < st.n_est; ++t)
        for (long long i = v0 + tid; i < v1; i += kCgNT) (t == 0 ? se0 : se1)[i] = s[i];
    if (ch == 0 && tid == 0) {
      ColState nx = st;
      nx.outcome = 3;
      nx.phase = kDone;
      a.st_next[c] = nx;
      atomicOr(a.status, kStatusBreakdown);
    }
    return;
  }

  const T al = sh.al, w0 = sh.w0, w1 = sh.w1;
  double p2 = 0.0;
#pragma unroll 2
  for (long long i = v0 + tid; i < v1; i += kCgNT) {
    const V di = d[i], ki = kd[i];
    V si = s[i], ei = e[i];
#pragma unroll
    for (int q = 0; q < VN; ++q) {
      si.v[q] = fma(al, di.v[q], si.v[q]);
      ei.v[q] = fma(-al, ki.v[q], ei.v[q]);
    }
    cg_keep_padding(si, i, a.n);
    cg_keep_padding(ei, i, a.n);
    s[i] = si;
    e[i] = ei;
#pragma unroll
    for (int q = 0; q < VN; ++q) p2 += (double)ei.v[q] * (double)ei.v[q];
    if (w0 != T(0)) {
      V x = se0[i];
#pragma unroll
      for (int q = 0; q < VN; ++q) x.v[q] = fma(w0, di.v[q], x.v[q]);
      cg_keep_padding(x, i, a.n);
      se0[i] = x;
    }
    if (w1 != T(0)) {
      V x = se1[i];
#pragma unroll
      for (int q = 0; q < VN; ++q) x.v[q] = fma(w1, di.v[q], x.v[q]);
      cg_keep_padding(x, i, a.n);
      se1[i] = x;
    }
  }
  double ee1;
  if (ordered) {
    __syncthreads();
    ee1 = cg_ordered_dot(a, a.E + col, a.E + col, ch, sh.red, sh.parts[1]);
  } else {
    ee1 = cluster_sum_warp0(p2, sh.red, &sh.slot[1]);
  }
  if (warp0) {
    const int m1 = st.m + 1;
    int ph = st.phase, l1 = st.l, outcome = st.outcome;
    bool copy_s = false, done = false;
    const int jmax = (st.n_est > 1 && st.J[1] > st.J[0]) ? st.J[1] : st.J[0];
    const double norm = sqrt(ee1);
    if (ph == kPre && norm < a.alpha_thr) {
      l1 = m1;
      ph = kTail;
      copy_s = true;
    }
    const bool conv = norm < a.eps;
    if (ph == kPre && conv) {
      copy_s = true;
      done = true;
    } else if (ph == kTail && (m1 - l1 >= jmax || conv)) {
      done = true;
    } else if (m1 >= a.max_iter) {
      if (ph == kPre) copy_s = true;
      outcome = 4;
      done = true;
    }
    // warm-started solves: remember the iterate of smallest residual
    const bool better = a.warm_refresh > 0 && ee1 < st.best_ee;
    if (lane == 0) {
      sh.copy_s = copy_s;
      sh.better = better;
      sh.done = done;
      sh.bt = done ? T(0) : (T)(ee1 / st.ee);
      if (ch == 0) {
        ColState nx = st;
        nx.ee = ee1;
        if (better) nx.best_ee = ee1;
        nx.m = m1;
        nx.l = l1;
        nx.outcome = outcome;
        nx.phase = done ? kDone : ph;
        a.st_next[c] = nx;
        if (outcome == 4) atomicOr(a.status, kStatusMaxIter);
      }
    }
  }
  __syncthreads();
  if (sh.copy_s || sh.better) {
    V* sb = sh.better ? reinterpret_cast<V*>(a.Sbest + col) : nullptr;
    for (long long i = v0 + tid; i < v1; i += kCgNT) {
      const V si = s[i];
      if (sh.copy_s) {
        se0[i] = si;
        if (st.n_est > 1) se1[i] = si;
      }
      if (sb) sb[i] = si;
    }
  }
  if (!sh.done) {
    const T bt = sh.bt;
#pragma unroll 4
    for (long long i = v0 + tid; i < v1; i += kCgNT) {
      V di = d[i];
      const V ei = e[i];
#pragma unroll
      for (int q = 0; q < VN; ++q) di.v[q] = fma(bt, di.v[q], ei.v[q]);
      cg_keep_padding(di, i, a.n);
      d[i] = di;
    }
  }
}

// The peers read this CTA's shared slots: nobody leaves before all have.
template <typename T>
__global__ void __launch_bounds__(kCgNT) cg_round_kernel(const CgArgs<T> a) {
  __shared__ CgShared<T> sh;
  cg_round_body(a, blockIdx.x, blockIdx.y, sh);
  cooperative_groups::this_cluster().sync();
}

// Batched form: grid (CTAs of a column, live-list index, problem); a cluster past its problem's
// live count returns at once.
template <typename T>
__global__ void __launch_bounds__(kCgNT) cg_round_batch_kernel(const CgArgs<T>* __restrict__ args) {
  __shared__ CgShared<T> sh;
  const CgArgs<T>& a = args[blockIdx.z];
  if ((int)blockIdx.y >= *a.n_live) return;
  cg_round_body(a, blockIdx.x, blockIdx.y, sh);
  cooperative_groups::this_cluster().sync();
}

// CTAs per column: about 1,024 rows each, a power of two up to kCgMaxCluster.
inline int cg_cluster_size(long long n) {
  int c = 1;
  while (c < kCgMaxCluster && n > 1024LL * c) c *= 2;
  return c;
}

// Rows per CTA of a column of leading dimension ld (a multiple of 64) over c CTAs.
inline long long cg_cluster_rows(long long ld, int c) {
  return ((ld + c - 1) / c + 63) / 64 * 64;
}

template <typename... Params, typename... Args>
cudaError_t launch_clustered(void (*kernel)(Params...), dim3 grid, int cluster, cudaStream_t s,
                             Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kCgNT);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One CG iteration of nl live columns.  Ordered sums: chunks of at least 2,048 rows, about two
// CTAs' worth per SM over all columns and at most kMaxCgChunks, shared by up to kCgMaxCluster CTAs.
template <typename T>
cudaError_t launch_cg_round(CgArgs<T> a, int nl, int num_sms, cudaStream_t s) {
  int c = cg_cluster_size(a.n);
  a.chunk = cg_cluster_rows(a.ld, c);
  if (a.ordered) {
    const long long target = std::max(1, (2 * num_sms + nl - 1) / nl);
    long long ch = std::max<long long>((a.n + target - 1) / target, 2048);
    ch = std::max<long long>(ch, (a.n + kMaxCgChunks - 1) / kMaxCgChunks);
    ch = (ch + 255) / 256 * 256;
    const int nc = (int)((a.n + ch - 1) / ch), per = (nc + kCgMaxCluster - 1) / kCgMaxCluster;
    c = (nc + per - 1) / per;
    a.chunk = per * ch;
    a.ordered = (int)ch;
    a.o_chunks = nc;
    a.o_per = per;
  }
  return launch_clustered(cg_round_kernel<T>, dim3((unsigned)c, (unsigned)nl), c, s, a);
}

// Commit the state of the first n_prev columns of the live list, then rebuild the list in column
// order; returns the live count.  One warp, a lane per column: as one thread it took 39 us for
// 101 columns (each column's state a dependent chain of global loads), now 3 us.
__device__ inline int commit_and_compact(ColState* __restrict__ st,
                                         const ColState* __restrict__ st_next, int R, int n_prev,
                                         int* __restrict__ live) {
  const int lane = threadIdx.x & 31;
  for (int k = lane; k < n_prev; k += 32) {
    const int c = live[k];
    st[c] = st_next[c];
  }
  __syncwarp();
  int n = 0;
  for (int c0 = 0; c0 < R; c0 += 32) {
    const int c = c0 + lane;
    const bool alive = c < R && st[c].phase != kDone;
    const unsigned mask = __ballot_sync(0xffffffffu, alive);
    if (alive) live[n + __popc(mask & ((1u << lane) - 1u))] = c;
    n += __popc(mask);
  }
  __syncwarp();
  return n;
}

// The compaction of one solve (one warp); count to *n_live.
__global__ void compact_kernel(ColState* __restrict__ st, const ColState* __restrict__ st_next,
                               int R, int n_prev, int* __restrict__ live,
                               int* __restrict__ n_live) {
  const int k = commit_and_compact(st, st_next, R, n_prev, live);
  if (threadIdx.x == 0) *n_live = k;
}

constexpr int kCompactBatchNT = 1024;

// Column bookkeeping of one problem of a batch (compact_batch_kernel).
struct BatchCgProb {
  ColState* st;
  const ColState* st_next;
  int* live;
  int* n_live;
  int R;
  long long n;
};

// K V width bucket of the batched product for a largest live count r: 0..4 for r <= 2, 4,
// 9, 17, 32 (the compiled widths of the batched kernel).
__host__ __device__ inline int batch_width_bucket(int r) {
  return r <= 2 ? 0 : r <= 4 ? 1 : r <= 9 ? 2 : r <= 17 ? 3 : 4;
}

// compact_kernel for every problem of a batch in one launch (a warp per problem; the
// live lists and counts are those of the previous round, the counts 0 before the first):
// commit, rebuild, and the largest live count to *rmax.  Inside a step graph it also sets
// the loop condition (another round while any column is live) and the branch (the width
// bucket of rmax; none when 0).  A round cap stops a loop that would not end.
// stat (may be null): [rounds, sum of n_b^2 x live columns, launches, rounds this call].
__global__ void __launch_bounds__(kCompactBatchNT) compact_batch_kernel(
    const BatchCgProb* __restrict__ probs, int B, int* __restrict__ rmax, int in_graph,
    cudaGraphConditionalHandle h_loop, cudaGraphConditionalHandle h_branch, int max_rounds,
    int tc_from, int tc_launches, long long* __restrict__ stat, int* __restrict__ status) {
  constexpr int NW = kCompactBatchNT / 32;
  __shared__ int s_max[NW];
  __shared__ long long s_ent[NW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int mx = 0;
  long long ent = 0;
  for (int b = warp; b < B; b += NW) {
    const BatchCgProb P = probs[b];
    const int k = commit_and_compact(P.st, P.st_next, P.R, *P.n_live, P.live);
    if (lane == 0) *P.n_live = k;
    mx = max(mx, k);
    ent += P.n * P.n * (long long)k;
  }
  if (lane == 0) {
    s_max[warp] = mx;
    s_ent[warp] = ent;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int t = 1; t < NW; ++t) {
    mx = max(mx, s_max[t]);
    ent += s_ent[t];
  }
  if (stat) {
    const long long it = stat[3]++;
    if (mx > 0 && it >= max_rounds) {
      atomicOr(status, kStatusMaxIter);
      for (int b = 0; b < B; ++b) *probs[b].n_live = 0;
      mx = 0;
      ent = 0;
    }
    stat[2] += 1;
    if (mx > 0) {
      stat[0] += 1;
      stat[1] += ent;
      // the batched K V, its tensor-core launches from tc_from columns on, the CG iteration
      stat[2] += 2 + (mx >= tc_from ? tc_launches : 0);
    }
  }
  *rmax = mx;
  if (in_graph) {
    cudaGraphSetConditional(h_loop, mx > 0 ? 1u : 0u);
    cudaGraphSetConditional(h_branch, mx > 0 ? (unsigned)batch_width_bucket(mx) : 5u);
  }
}

// ------------------------------------------------------------------------------------
// a7: SGLD proposal psi' = psi + eps/2 M (g + grad log p) + sqrt(eps) L xi, L L^T = M,
// xi_k standard normal from Philox counter (k, 0, step, 3).  One warp: lane i owns row i of
// L and component i (p <= kMaxP <= 32); each element's sums run in the serial order.
// ------------------------------------------------------------------------------------
__device__ inline void sgld_body(double* __restrict__ psi, const double* __restrict__ g,
                                 const double* __restrict__ M, const double* __restrict__ prior,
                                 double eps, int p, unsigned long long seed,
                                 unsigned long long step, double* __restrict__ trace,
                                 int* __restrict__ status) {
  __shared__ double L[kMaxP * kMaxP];
  __shared__ double xi[kMaxP], v[kMaxP];
  const int lane = threadIdx.x & 31;
  auto Mij = [&](int i, int j) -> double {
    return M ? M[i * p + j] : (i == j ? 1.0 : 0.0);
  };
  if (lane < p) {
    uint64_t w[4];
    philox4x64_10((uint64_t)lane, 0, step, kPurposeSgld, seed, 0, w);
    xi[lane] = box_muller(w[0], w[1]);
    v[lane] = g[lane] + (prior ? prior[lane] : 0.0);
    for (int j = 0; j < p; ++j) L[lane * p + j] = 0.0;
  }
  __syncwarp();
  // Cholesky M = L L^T, column by column: the diagonal on lane 0, then the column below it
  for (int j = 0; j < p; ++j) {
    int bad = 0;
    if (lane == 0) {
      double sj = Mij(j, j);
      for (int k = 0; k < j; ++k) sj -= L[j * p + k] * L[j * p + k];
      bad = !(sj > 0.0);
      if (!bad) L[j * p + j] = sqrt(sj);
    }
    if (__shfl_sync(0xffffffffu, bad, 0)) {
      if (lane == 0) atomicOr(status, kStatusBadM);
      return;
    }
    __syncwarp();
    if (lane > j && lane < p) {
      double t = Mij(lane, j);
      for (int k = 0; k < j; ++k) t -= L[lane * p + k] * L[j * p + k];
      L[lane * p + j] = t / L[j * p + j];
    }
    __syncwarp();
  }
  if (lane < p) {
    double drift = 0.0, noise = 0.0;
    for (int j = 0; j < p; ++j) drift += Mij(lane, j) * v[j];
    for (int j = 0; j <= lane; ++j) noise += L[lane * p + j] * xi[j];
    const double out = psi[lane] + 0.5 * eps * drift + sqrt(eps) * noise;
    psi[lane] = out;
    if (trace) trace[lane] = out;
  }
}

// Launched with one warp.
__global__ void sgld_kernel(double* __restrict__ psi, const double* __restrict__ g,
                            const double* __restrict__ M, const double* __restrict__ prior,
                            const double* __restrict__ eps_arr, double eps_scalar, int p,
                            unsigned long long seed, unsigned long long step,
                            double* __restrict__ trace, int* __restrict__ status) {
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  sgld_body(psi, g, M, prior, eps_arr ? *eps_arr : eps_scalar, p, seed, step, trace, status);
}

// The same update inside a chain graph: step, step size and trace slot from the chain
// slot, which then moves on to the next step.  Launched with one warp.
__global__ void sgld_chain_kernel(double* __restrict__ psi, const double* __restrict__ g,
                                  const double* __restrict__ M, const double* __restrict__ prior,
                                  int p, unsigned long long seed, ChainSlot* __restrict__ cs,
                                  int* __restrict__ status, int advance = 1,
                                  int trace_stride = 0, int trace_off = 0) {
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  const long long k = cs->k;
  const long long stride = trace_stride > 0 ? trace_stride : p;
  sgld_body(psi, g, M, prior, cs->eps[k], p, seed, cs->step0 + (unsigned long long)k,
            cs->trace ? cs->trace + k * stride + trace_off : nullptr, status);
  __syncwarp();   // every lane has read the slot
  if (advance && threadIdx.x == 0) cs->k = k + 1;
}

// The chain slot moves on to the next step (batched step graphs: after every problem's
// update).
__global__ void chain_advance_kernel(ChainSlot* __restrict__ cs) {
  if (threadIdx.x == 0 && blockIdx.x == 0) cs->k += 1;
}

// Graph form of compact_kernel: commits the previous iteration's column states (the live
// list and count are still those of the previous iteration; the count is 0 before the
// first), rebuilds the list, and sets the graph's loop conditions -- the WHILE body runs
// again while columns are live, and the SWITCH picks the branch compiled for that many
// live columns (none when 0).  A round cap (max_iter + 2) stops a loop that would not end.
// stat: [rounds, sum of live columns over rounds, kernel launches, iterations this call].
__global__ void compact_graph_kernel(ColState* __restrict__ st, const ColState* __restrict__ st_next,
                                     int R, int* __restrict__ live, int* __restrict__ n_live,
                                     cudaGraphConditionalHandle h_loop,
                                     cudaGraphConditionalHandle h_branch,
                                     const int* __restrict__ kv_launches, int max_rounds,
                                     long long* __restrict__ stat, int* __restrict__ status) {
  int k = commit_and_compact(st, st_next, R, *n_live, live);
  if (threadIdx.x != 0) return;
  const long long it = stat[3]++;
  if (k > 0 && it >= max_rounds) {
    atomicOr(status, kStatusMaxIter);
    k = 0;
  }
  *n_live = k;
  stat[2] += 1;
  if (k > 0) {
    stat[0] += 1;
    stat[1] += k;
    stat[2] += 1 + kv_launches[k - 1];   // the CG iteration, and the K V of k columns
  }
  cudaGraphSetConditional(h_loop, k > 0 ? 1u : 0u);
  cudaGraphSetConditional(h_branch, k > 0 ? (unsigned)(k - 1) : (unsigned)R);
}

// ulisse_dk_bilinear's scales by value.
struct BilinearScales {
  double v[kMaxM];
};

// Scales to sa, the status word to 0, and (A not null) columns 0..M-1 of A and B, leading
// dimension n, to the context's buffers, leading dimension ld: column c of A, then of B, per grid
// row.
template <typename T>
__global__ void __launch_bounds__(256) bilinear_prepare_kernel(
    const BilinearScales sc, int M, T* __restrict__ sa, int* __restrict__ status,
    const float* __restrict__ A, T* __restrict__ Ad, const float* __restrict__ B,
    T* __restrict__ Bd, long long n, long long ld) {
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    if ((int)threadIdx.x < M) sa[threadIdx.x] = (T)sc.v[threadIdx.x];
    if (threadIdx.x == 0) *status = 0;
  }
  if (!A) return;
  const int c = (int)blockIdx.y < M ? blockIdx.y : blockIdx.y - M;
  const float* src = ((int)blockIdx.y < M ? A : B) + c * n;
  T* dst = ((int)blockIdx.y < M ? Ad : Bd) + c * ld;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL)
    dst[i] = (T)src[i];
}

// Element-type conversion between caller buffers and the context's (FP64 contexts).
template <typename S, typename D>
__global__ void convert_cols_kernel(const S* __restrict__ src, long long lds, D* __restrict__ dst,
                                    long long ldd, long long n) {
  const int c = blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[c * ldd + i] = (D)src[c * lds + i];
}

}  // namespace ulisse
