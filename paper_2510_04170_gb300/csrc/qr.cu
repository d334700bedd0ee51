// Householder QR of the sketch B = S_k J (Sec. 4.1, "thin QR B = Q R") giving
// the right preconditioner R.  Blocked right-looking Householder with the
// compact-WY trailing update (Schreiber & Van Loan):
//
//   k_panel     (cooperative) factors 32 columns, one exchange between the CTAs
//               per column.  Reflector H = I - tau v v^T, v_0 = 1,
//               beta = -sign(alpha) ||x||.
//   k_gram, k_panel_t: the panel's V^T V by chunks of rows and its compact-WY
//               factor T
//   k_vta       W_z = V^T A_trail over a K-slice z (split K, deterministic)
//   k_wt        W2 = T^T sum_z W_z
//   k_update    A_trail -= V W2
//   k_diag, k_flip, k_floor: rows of R flipped to a positive diagonal, pivots
//               below 1e-14 max_j R_jj floored (rank guard; flag raised).
//
// All sums are reduced in a fixed order, so repeated runs give identical bits.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "rfm_internal.cuh"

namespace {

constexpr int NB = 32;

// ---------------------------------------------------------------------------
// Cooperative panel factorisation k_panel (up to 32 columns).
//
// GB300's FP64 unit takes 64 cycles (31 ns) for a warp instruction, the same
// for a dependent chain as for independent ones and for one lane as for 32
// (measured).  What bounds a column of the factorisation is therefore the
// number of FP64 warp instructions on one SM partition, plus one exchange
// between the CTAs; the kernel is laid out to issue few of them: the lanes of a
// warp are the 32 columns of the panel, so a row of the panel is one instruction
// for the products and one for the update, and no reduction over lanes is needed.
// Two warps per SM partition keep its FP64 unit busy through each other's loads.
//
// The order of every sum is fixed by the row count (and a cap on the chunks), not
// by how the rows are spread over CTAs, so that R has the same bits on any split:
// a last bit of R can change the step counts of a solve at cond(R) = 1e9.  The
// panel's rows are P chunks of `chunk` rows.  A chunk's sum has 32 chains, rows of
// equal remainder modulo 32, added pairwise at distances 16, 8, 4, 2, 1; chunks q,
// q + 32, .. are added in turn, and the 32 sums that leaves pairwise at distances
// 16 .. 1 again.  Spread over the chip:
//  - a cluster of CL CTAs owns the chunks of one remainder modulo 32 (or, CL =
//    1, a CTA owns one chunk), and a warp in it 4 / CL chains of each.
//  - the chains' sums meet in the cluster through distributed shared memory and
//    one cluster barrier (0.2 us); each rank finishes 32 / CL columns and publishes
//    them as 16-byte records {low, tag, high, tag} whose tag is the column's
//    number.  A reader polls the records themselves, so there is no fence, no
//    counter and no second trip to L2.  Two slots alternate; a CTA can only be one
//    exchange ahead of another.  (With a record per chunk every CTA reads 78 KB per
//    column, which is L2 bound.)
// After the exchange a warp of every CTA forms beta, tau, 1 / (alpha - beta) and
//     w_k = v^T A_k = A_jk + p_k / (alpha - beta)     (v_j = 1, v_r = x_r / (alpha - beta))
// with p_k = sum x_r A_rk; the column is scaled, the next column updated with
// the lanes as rows, and then one pass over the rows updates the other columns
// and takes the next column's products.
//
// Per column at 12,288 rows: 16.5 us with one grid barrier and a butterfly
// reduction in every warp (the former kernel), now 6.0 (2.5 the pass over the
// rows, 0.25 cluster barrier, 0.8 trees, 0.8 poll, 1.4 scalars, 0.3 scaling); at
// 3,072 rows 4.4.  One warp per partition took 3.5 us for the pass.
constexpr int KP_THREADS = 256;
constexpr int KP_SMEM = 227 * 1024;  // dynamic shared memory of a CTA
constexpr int KP_CHUNK = 800;        // most rows of a chunk
constexpr int KP_MAXP = 256;         // most chunks
constexpr int KP_SLOT = (KP_MAXP + 1) * NB * 2;  // 8-byte words of an exchange slot (last record: the pivot row)

struct PanelArgs {
  double* A;
  long long lda;
  long long s;
  long long j0;
  int nbw;             // columns in this panel (<= NB)
  int P;               // chunks
  int chunk;           // rows of a chunk
  int kpc;             // rows of a chain in a chunk, at most
  int U;               // chunks per cluster, at most
  int NG;              // clusters (and records of an exchange)
  unsigned long long* xch;  // [2][KP_SLOT] exchange records
  double* tau;         // [n]
  unsigned int* err;
};

// Slab element (local row r, column c): rows of 33, so that both a row (lanes =
// columns) and a column (lanes = rows) are free of bank conflicts.
constexpr int KP_LD = NB + 1;
__device__ __forceinline__ int kp_at(int r, int c) { return r * KP_LD + c; }

// x != 0 (true for NaN) without an FP64 instruction.
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }

__device__ __forceinline__ void kp_copy8(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Doubles of shared memory beside the slab: the chains' sums of this rank's columns
// [U][32][32 / CL], their sums over a chunk [U][32 / CL], the warps' shares [8][32],
// the columns' factors and three scalars [36], the chains' lengths [32 / CL][U].
constexpr long long kp_fixed(int CL, int U) {
  return (long long)U * (NB + 1) * (NB / CL) + 8 * NB + 36 + (NB / CL * U + 1) / 2;
}
// Rows of the slab.
constexpr long long kp_slab_rows(int CL, int U, int kpc) { return (long long)U * (NB / CL) * kpc; }

template <int N>
struct Int {
  static constexpr int value = N;
};

template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(KP_THREADS, 1) k_panel(PanelArgs a) {
  if (!in_cluster(CL, a.err)) return;
  constexpr int NC = NB / CL, NS = NC / 8, OC = NB / CL;  // chains per CTA and per warp, columns per rank
  extern __shared__ __align__(16) double kp_sm[];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int rank = blockIdx.x % CL, g = blockIdx.x / CL, U = a.U, kpc = a.kpc, NG = a.NG;
  double* wp = kp_sm;               // [U][32][OC]
  double* gs = wp + U * NB * OC;    // [U][OC]
  double* rs = gs + U * OC;         // [8][NB]
  double* fs = rs + 8 * NB;         // [NB] factors, then tau, 1 / (alpha - beta), beta
  int* kns = reinterpret_cast<int*>(fs + 36);      // [NC][U]
  double* sl = fs + 36 + (NC * U + 1) / 2;         // slab
  // rows of this cluster's chunk u
  auto rows_of = [&](int u) {
    const int q = g + 32 * u;
    const long long beg = a.j0 + (long long)q * a.chunk;
    return q < a.P && beg < a.s ? (int)min((long long)a.chunk, a.s - beg) : 0;
  };
  // Row c + 32 k of chunk u with c = rank NC + cin: warp cin & 7, slab row (cin U + u) kpc + k
  for (int idx = lane; idx < U * NC * kpc; idx += 32) {
    const int cin = idx % NC, rest = idx / NC, k = rest % kpc, u = rest / kpc;
    const int r = rank * NC + cin + 32 * k, row = (cin * U + u) * kpc + k;
    const bool in = r < rows_of(u);
    const double* src = a.A + a.j0 + (long long)(g + 32 * u) * a.chunk + r;
    for (int cc = w; cc < NB; cc += 8) {
      if (in && cc < a.nbw) kp_copy8(sl + kp_at(row, cc), src + (size_t)(a.j0 + cc) * a.lda);
      else sl[kp_at(row, cc)] = 0.0;
    }
  }
  for (int i = tid; i < NC * U; i += KP_THREADS) kns[i] = max(0, rows_of(i % U) - rank * NC - i / U + 31) >> 5;
  asm volatile("cp.async.wait_all;" ::: "memory");
  RecWait kw(a.err, tid);
  __syncthreads();
  if (CL > 1) {
    cluster_arrive();
    cluster_wait();  // all ranks run: their shared memory may be written
  }
  // slab row of the panel's row j (a pivot: first of its chain in chunk 0) if this warp owns it, else -1
  auto pivot_row = [&](int j) {
    const int cin = j - rank * NC;
    return g == 0 && cin >= 0 && cin < NC && (cin & 7) == w ? cin * U * kpc : -1;
  };
  // Rows below the pivot jj - 1: with `upd`, A_rk -= f_k v_r for the columns past
  // jj, v the column jj - 1; then this warp's chains of x^T A_k over the rows below
  // jj, x the column jj, to the rank that adds them up.
  auto pass = [&](int jj, bool upd, double f) {
#pragma unroll
    for (int sub = 0; sub < NS; ++sub)
      for (int u = 0; u < U; ++u) {
        const int cin = w + 8 * sub, c = rank * NC + cin, row0 = (cin * U + u) * kpc;
        const int kn = kns[cin * U + u];
        double acc = 0.0;
        int k = 0;
        if (g == 0 && u == 0 && c <= jj && kn > 0) {  // rows up to the pivots lead the chains of chunk 0
          if (c == jj && upd) {
            const double v = sl[kp_at(row0, jj - 1)], e = sl[kp_at(row0, lane)];
            if (lane > jj) sl[kp_at(row0, lane)] = fma(-v, f, e);
          }
          k = 1;
        }
        // batches of rows: their loads first, as no load moves above a store to the slab
        auto batch = [&](auto count) {
          constexpr int N = decltype(count)::value;
          double x[N], e[N], v[N];
#pragma unroll
          for (int i = 0; i < N; ++i) {
            if (upd) v[i] = sl[kp_at(row0 + k + i, jj - 1)];
            x[i] = sl[kp_at(row0 + k + i, jj)];
            e[i] = sl[kp_at(row0 + k + i, lane)];
          }
          if (upd) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
              const double t = fma(-v[i], f, e[i]);
              e[i] = lane > jj ? t : e[i];
            }
          }
#pragma unroll
          for (int i = 0; i < N; ++i) acc = fma(x[i], e[i], acc);
          if (upd) {
#pragma unroll
            for (int i = 0; i < N; ++i) sl[kp_at(row0 + k + i, lane)] = e[i];
          }
          k += N;
        };
        while (k + 4 <= kn) batch(Int<4>{});
        const int left = kn - k;
        if (left == 3) batch(Int<3>{});
        else if (left == 2) batch(Int<2>{});
        else if (left == 1) batch(Int<1>{});
        double* dst = wp + (u * NB + c) * OC + lane % OC;
        if (CL > 1) st_cluster(dst, lane / OC, acc);
        else *dst = acc;
      }
  };
  pass(0, false, 0.0);
  for (int jj = 0; jj < a.nbw; ++jj) {
    const unsigned int tag = (unsigned int)(a.j0 + jj + 1);
    unsigned long long* slot = a.xch + (size_t)(jj & 1) * KP_SLOT;
    const int prow = pivot_row(jj);
    if (prow >= 0) {
      __syncwarp();
      rec_publish(slot + ((size_t)NG * NB + lane) * 2, sl[kp_at(prow, lane)], tag);
    }
    if (CL > 1) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
    // a chunk's tree over its 32 chains, eight columns a warp (lane = 4 column +
    // part), then the sum over the cluster's chunks
    for (int task = w; task < U * (OC / 8); task += 8) {
      const int u = task / (OC / 8), col = task % (OC / 8) * 8 + (lane >> 2);
      const double* x = wp + (u * NB + (lane & 3)) * OC + col;
      double t = ((x[0] + x[16 * OC]) + (x[8 * OC] + x[24 * OC])) +
                 ((x[4 * OC] + x[20 * OC]) + (x[12 * OC] + x[28 * OC]));
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      if ((lane & 3) == 0) {
        if (U == 1) rec_publish(slot + ((size_t)g * NB + rank * OC + col) * 2, t, tag);
        else gs[u * OC + col] = t;
      }
    }
    if (U > 1) {
      __syncthreads();
      if (tid < OC) {
        double t = gs[tid];
        for (int u = 1; u < U; ++u) t += gs[u * OC + tid];
        rec_publish(slot + ((size_t)g * NB + rank * OC + tid) * 2, t, tag);
      }
      __syncwarp();
    }
    // Sum over the clusters, warp w the remainders w, w + 8, .. modulo 32; warp 0
    // also reads the pivot row (record NG).  A complete record of this cluster
    // says that all its ranks have read wp.
    double s[4] = {0.0, 0.0, 0.0, 0.0}, piv = 0.0;
    for (int q0 = w; q0 < NG; q0 += 32) {
      unsigned long long lo[5], hi[5];
      unsigned int spins = 0;
      for (;;) {
        bool all = true;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (q0 + 8 * i < NG) rec_load(slot + ((size_t)(q0 + 8 * i) * NB + lane) * 2, lo[i], hi[i]);
        if (w == 0) rec_load(slot + ((size_t)NG * NB + lane) * 2, lo[4], hi[4]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (q0 + 8 * i < NG) all = all && rec_ready(lo[i], hi[i], tag);
        if (w == 0) all = all && rec_ready(lo[4], hi[4], tag);
        if (__all_sync(0xffffffffu, all) || !__all_sync(0xffffffffu, kw.spin(spins))) break;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (q0 + 8 * i < NG) s[i] += rec_value(lo[i], hi[i]);
      if (w == 0) piv = rec_value(lo[4], hi[4]);
    }
    rs[w * NB + lane] = (s[0] + s[2]) + (s[1] + s[3]);
    __syncthreads();
    if (w == 0) {
      const double* x = rs + lane;
      const double tot = ((x[0] + x[4 * NB]) + (x[2 * NB] + x[6 * NB])) + ((x[NB] + x[5 * NB]) + (x[3 * NB] + x[7 * NB]));
      const double alpha = __shfl_sync(0xffffffffu, piv, jj), sigma = __shfl_sync(0xffffffffu, tot, jj);
      double tau = 0.0, beta = alpha, scale = 0.0;
      if (nonzero(sigma)) {
        const double nrm = sqrt(alpha * alpha + sigma);
        beta = __double2hiint(alpha) < 0 && nonzero(alpha) ? nrm : -nrm;
        // lane 0 (beta - alpha) / beta, the others 1 / (alpha - beta), in one division
        const double d = alpha - beta;
        const double t = (lane == 0 ? -d : 1.0) / (lane == 0 ? beta : d);
        tau = __shfl_sync(0xffffffffu, t, 0);
        scale = __shfl_sync(0xffffffffu, t, 1);
      }
      fs[lane] = tau * (piv + scale * tot);  // tau w_k
      if (lane < 3) fs[NB + lane] = lane == 0 ? tau : lane == 1 ? scale : beta;
      if (blockIdx.x == 0 && lane == 0) a.tau[a.j0 + jj] = tau;
    }
    __syncthreads();
    const double f = fs[lane], scale = fs[NB + 1];
    const bool upd = nonzero(fs[NB]);
    if (upd) {
      // v_r = x_r / (alpha - beta) below the pivot, and the next column (lanes are rows)
      const double f1 = fs[(jj + 1) & 31];
#pragma unroll
      for (int sub = 0; sub < NS; ++sub) {
        const int cin = w + 8 * sub;
        for (int i = lane; i < U * kpc; i += 32) {
          const int row = cin * U * kpc + i;
          if (g == 0 && i == 0 && rank * NC + cin <= jj) continue;
          const double v = sl[kp_at(row, jj)] * scale;
          sl[kp_at(row, jj)] = v;
          if (jj + 1 < NB) sl[kp_at(row, jj + 1)] = fma(-v, f1, sl[kp_at(row, jj + 1)]);
        }
      }
    }
    if (prow >= 0) {
      double* e = sl + kp_at(prow, lane);
      if (lane > jj && upd) *e -= f;
      if (lane == jj) *e = fs[NB + 2];
    }
    __syncwarp();
    if (jj + 1 < a.nbw) pass(jj + 1, upd, f);
  }
  __syncthreads();
  // R on and above the diagonal and v below back to global memory (the last
  // cluster barrier came after the last remote store)
  for (int idx = lane; idx < U * NC * kpc; idx += 32) {
    const int cin = idx % NC, rest = idx / NC, k = rest % kpc, u = rest / kpc;
    const int r = rank * NC + cin + 32 * k, row = (cin * U + u) * kpc + k;
    if (r >= rows_of(u)) continue;
    double* dst = a.A + a.j0 + (long long)(g + 32 * u) * a.chunk + r;
    for (int cc = w; cc < a.nbw; cc += 8) dst[(size_t)(a.j0 + cc) * a.lda] = sl[kp_at(row, cc)];
  }
}

// Vector of panel column p at global row gr (unit pivot, zero above).
__device__ __forceinline__ double vval(const double* A, long long lda, long long j0, int p, long long gr) {
  const long long piv = j0 + p;
  if (gr < piv) return 0.0;
  if (gr == piv) return 1.0;
  return A[(size_t)(j0 + p) * lda + gr];
}

// Strict upper part of the panel's V^T V over the rows of each chunk, one
// thread per two entries, the rows in turn: gram[chunk][KG_LD], entry (p, q) at
// kg_at(p, q).
constexpr int KG_LD = 512;
__host__ __device__ constexpr int kg_at(int p, int q) { return q * (q - 1) / 2 + p; }  // p < q
constexpr int KG_ROWS = 64;  // rows staged at a time

__global__ void __launch_bounds__(256) k_gram(const double* __restrict__ A, long long lda, long long s, long long j0,
                                              int nbw, int chunk, double* __restrict__ gram) {
  __shared__ double Vs[KG_ROWS][NB + 1];
  const int tid = threadIdx.x;
  const long long beg = j0 + (long long)blockIdx.x * chunk, end = min(s, beg + chunk);
  int p[2], q[2];
  double acc[2] = {0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int e = tid + 256 * i;
    q[i] = 1;
    while (q[i] < NB - 1 && kg_at(0, q[i] + 1) <= e) ++q[i];
    p[i] = min(e - kg_at(0, q[i]), NB - 1);
  }
  for (long long r0 = beg; r0 < end; r0 += KG_ROWS) {
    for (int idx = tid; idx < KG_ROWS * NB; idx += 256) {
      const int rr = idx & (KG_ROWS - 1), c = idx / KG_ROWS;
      const long long gr = r0 + rr;
      Vs[rr][c] = gr < end && c < nbw ? vval(A, lda, j0, c, gr) : 0.0;
    }
    __syncthreads();
    const int nr = (int)min((long long)KG_ROWS, end - r0);
#pragma unroll 4
    for (int r = 0; r < nr; ++r)
#pragma unroll
      for (int i = 0; i < 2; ++i) acc[i] = fma(Vs[r][p[i]], Vs[r][q[i]], acc[i]);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (tid + 256 * i < NB * (NB - 1) / 2) gram[(size_t)blockIdx.x * KG_LD + tid + 256 * i] = acc[i];
}

// The panel's compact-WY factor T (row-major [NB][NB]) from the chunks' sums and
// tau: T_jj = tau_j, T_ij = -tau_j sum_{i <= l < j} T_il G_lj.  Eight CTAs of a
// cluster add the chunks (a thread per entry, 64 to a CTA, the chunks in turn);
// then a warp takes the rows i and 31 - i of T, lanes = columns, each step one
// product and one multiply-add for all columns to the right.  On one CTA the
// sums alone would take 20 us at 152 chunks.
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(64) k_panel_t(const double* __restrict__ gram, int P,
                                                                           const double* __restrict__ tau, int nbw,
                                                                           double* __restrict__ G,
                                                                           double* __restrict__ T) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int e = blockIdx.x * 64 + tid;
  double sum = 0.0;
  for (int q0 = 0; q0 < P; q0 += 32) {
    double t[32];
#pragma unroll
    for (int u = 0; u < 32; ++u) t[u] = q0 + u < P ? __ldcg(gram + (size_t)(q0 + u) * KG_LD + e) : 0.0;
#pragma unroll
    for (int u = 0; u < 32; ++u)
      if (q0 + u < P) sum += t[u];
  }
  __stcg(G + e, sum);
  __threadfence();
  cluster_arrive();
  cluster_wait();
  double g[NB];  // column `lane` of G above the diagonal
#pragma unroll
  for (int l = 0; l < NB; ++l) g[l] = l < lane ? __ldcg(G + kg_at(l, lane)) : 0.0;
  const double tj = lane < nbw ? tau[lane] : 0.0;
  const int wi = blockIdx.x * 2 + (tid >> 5);
  for (int half = 0; half < 2; ++half) {
    const int i = half == 0 ? wi : NB - 1 - wi;
    double v = 0.0, row = 0.0;  // row: T_i,lane
#pragma unroll
    for (int l = 0; l < NB; ++l) {
      if (l < i) continue;  // warp-uniform
      if (lane == l) row = l == i ? tj : -tj * v;
      const double til = __shfl_sync(0xffffffffu, row, l);
      if (lane > l) v = fma(til, g[l], v);
    }
    T[i * NB + lane] = i < nbw && lane < nbw ? row : 0.0;
  }
}

// Wp[z][col][p] = sum_{r in K-slice z} v_p(r) A[r, j1 + col], in tiles of TC
// columns.  Every output is one chain over the slice's rows whatever the tile;
// narrow tiles spread the work over the SMs (n = 1,024, 3,072 rows: 31 launches
// 5.5 -> 3.2 ms; at most 96 columns of 12,288 rows: 148 -> 71 us each).
template <int TC>
__host__ __device__ constexpr int vta_threads() { return TC >= 32 ? 256 : 128; }

template <int TC>
__global__ void __launch_bounds__(vta_threads<TC>()) k_vta(const double* __restrict__ A, long long lda, long long s,
                                                           long long j0, int nbw, long long j1, long long nt,
                                                           long long kchunk, double* __restrict__ Wp) {
  // threads over columns (CX) and reflectors (AY), NQ columns and NA reflectors each
  constexpr int NT = vta_threads<TC>(), NQ = TC >= 16 ? 4 : 2, CX = TC / NQ, AY = NT / CX, NA = NB / AY;
  __shared__ double Vs[32][NB + 1];
  __shared__ double As[32][TC + 1];
  const int tid = threadIdx.x;
  const long long col0 = (long long)blockIdx.x * TC;
  const int z = blockIdx.y;
  const long long kb = j0 + (long long)z * kchunk;
  const long long ke = min(s, kb + kchunk);
  const int ay = tid / CX, cx = tid % CX;
  double acc[NA][NQ];
#pragma unroll
  for (int h = 0; h < NA; ++h)
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[h][q] = 0.0;
  for (long long r0 = kb; r0 < ke; r0 += 32) {
    for (int idx = tid; idx < 32 * NB; idx += NT) {
      const int rr = idx & 31, p = idx >> 5;
      const long long gr = r0 + rr;
      Vs[rr][p] = (gr < ke && p < nbw) ? vval(A, lda, j0, p, gr) : 0.0;
    }
    for (int idx = tid; idx < 32 * TC; idx += NT) {
      const int rr = idx & 31, cc = idx >> 5;
      const long long gr = r0 + rr, gc = col0 + cc;
      As[rr][cc] = (gr < ke && gc < nt) ? A[(size_t)(j1 + gc) * lda + gr] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int rr = 0; rr < 32; ++rr) {
      double v[NA];
#pragma unroll
      for (int h = 0; h < NA; ++h) v[h] = Vs[rr][ay + AY * h];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const double av = As[rr][cx + CX * q];
#pragma unroll
        for (int h = 0; h < NA; ++h) acc[h][q] += v[h] * av;
      }
    }
    __syncthreads();
  }
  for (int h = 0; h < NA; ++h)
    for (int q = 0; q < NQ; ++q) {
      const long long gc = col0 + cx + CX * q;
      const int p = ay + AY * h;
      if (gc < nt) Wp[((size_t)z * nt + gc) * NB + p] = acc[h][q];
    }
}

// W2 = T^T sum_z Wp[z], one warp per column, lanes = p: both the sum over z and
// the row of T^T are chains of FP64 instructions of 31 ns; one column per warp
// keeps all columns independent.  (One thread per column took 120 us at 12,288
// rows.)
__global__ void __launch_bounds__(128) k_wt(const double* __restrict__ Wp, int nz, const double* __restrict__ T,
                                            int nbw, long long nt, double* __restrict__ W2) {
  const int lane = threadIdx.x & 31;
  const long long col = blockIdx.x * 4LL + (threadIdx.x >> 5);
  if (col >= nt) return;
  double x = 0.0;
  for (int z0 = 0; z0 < nz; z0 += 8) {
    double t[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = z0 + u < nz ? Wp[((size_t)(z0 + u) * nt + col) * NB + lane] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (z0 + u < nz) x += t[u];
  }
  double tq[NB], y = 0.0;
#pragma unroll
  for (int q = 0; q < NB; ++q) tq[q] = T[q * NB + lane];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const double xq = __shfl_sync(0xffffffffu, x, q);
    if (q <= lane && q < nbw) y = fma(tq[q], xq, y);
  }
  W2[(size_t)lane * nt + col] = lane < nbw ? y : 0.0;
}

// A[r, j1 + col] -= sum_p v_p(r) W2[p][col] for r in [j0, s), in tiles of 64 rows
// x 16 columns: lanes are rows, a warp takes four columns.  FP64 bound, so a
// tile needs no reuse beyond its own; what counts is that the tiles spread
// evenly over the SMs' FP64 units (128 x 64 tiles, 16 times the work each, left
// 1,200 x 400 on 30 SMs: 77 us a launch, now 23 us; 3,072 x 1,024: 124 ->
// 85 us against 77 us of FMAs).  The 32 products are summed by themselves and
// subtracted once: subtracted one by one from A they left R 1.4 times as far
// from a 64-bit reference (6.7e-14 against 4.7e-14 at n = 1,024).
constexpr int UR = 64, UC = 16;

__global__ void __launch_bounds__(128) k_update(double* __restrict__ A, long long lda, long long s, long long j0,
                                                int nbw, long long j1, long long nt, const double* __restrict__ W2) {
  __shared__ double Vs[NB][UR];
  __shared__ double Ws[NB][UC];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const long long r0 = j0 + (long long)blockIdx.x * UR;
  const long long c0 = (long long)blockIdx.y * UC;
  for (int idx = tid; idx < NB * UR; idx += 128) {
    const int rr = idx & (UR - 1), p = idx / UR;
    const long long gr = r0 + rr;
    Vs[p][rr] = (gr < s && p < nbw) ? vval(A, lda, j0, p, gr) : 0.0;
  }
  for (int idx = tid; idx < NB * UC; idx += 128) {
    const int cc = idx & (UC - 1), p = idx / UC;
    const long long gc = c0 + cc;
    Ws[p][cc] = gc < nt ? W2[(size_t)p * nt + gc] : 0.0;
  }
  double a[2][4], d[2][4];  // A's entries, and the sums to be subtracted once
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long gr = r0 + lane + 32 * i, gc = c0 + 4 * w + q;
      d[i][q] = 0.0;
      a[i][q] = gr < s && gc < nt ? A[(size_t)(j1 + gc) * lda + gr] : 0.0;
    }
  __syncthreads();
#pragma unroll 4
  for (int p = 0; p < NB; ++p) {
    const double v0 = Vs[p][lane], v1 = Vs[p][lane + 32];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double y = Ws[p][4 * w + q];
      d[0][q] = fma(v0, y, d[0][q]);
      d[1][q] = fma(v1, y, d[1][q]);
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long gr = r0 + lane + 32 * i, gc = c0 + 4 * w + q;
      if (gr < s && gc < nt) A[(size_t)(j1 + gc) * lda + gr] = a[i][q] - d[i][q];
    }
}

__global__ void k_diag(const double* __restrict__ A, long long lda, long long n, double* __restrict__ dg) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) dg[i] = A[(size_t)i * lda + i];
}

// Flip row i of R when R_ii < 0 (upper triangle only).
__global__ void k_flip(double* __restrict__ A, long long lda, long long n, const double* __restrict__ dg) {
  const long long col = blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i <= col; i += (long long)gridDim.x * blockDim.x)
    if (dg[i] < 0.0) A[(size_t)col * lda + i] = -A[(size_t)col * lda + i];
}

__global__ void k_floor(double* __restrict__ A, long long lda, long long n, unsigned int* flag) {
  __shared__ double sh[40];
  double mx = 0.0;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) mx = fmax(mx, A[(size_t)i * lda + i]);
  mx = warp_max(mx);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    v = warp_max(v);
    if (threadIdx.x == 0) sh[32] = v;
  }
  __syncthreads();
  const double fl = 1e-14 * sh[32];
  for (long long i = threadIdx.x; i < n; i += blockDim.x)
    if (A[(size_t)i * lda + i] < fl) {
      A[(size_t)i * lda + i] = fl;
      atomicExch(flag, 1u);
    }
}

struct QrScratch {
  unsigned long long* xch;  // exchange records of k_panel
  double* gram;             // [chunks][KG_LD] of a panel
  double* G;                // their sum
  double* tau;
  double* T;
  double* Wp;
  double* W2;
  double* dg;
};

}  // namespace

// Doubles of the panel scratch: exchange records, Gram, T, tau, and the split-K
// partials, W2 and diagonal of the trailing update.
__host__ __device__ constexpr long long qr_scratch_len(long long n) {
  return 2LL * KP_SLOT + (KP_MAXP + 1LL) * KG_LD + NB * NB + 64LL * NB * n + NB * n + n + n + 64;
}

long long rfm_householder_scratch(long long s, long long n) {
  (void)s;
  return qr_scratch_len(n);
}

namespace {

QrScratch carve(double* scratch, long long n) {
  QrScratch q;
  double* w = scratch;
  q.xch = reinterpret_cast<unsigned long long*>(w); w += 2LL * KP_SLOT;
  q.gram = w; w += (long long)KP_MAXP * KG_LD;
  q.G = w; w += KG_LD;
  q.T = w; w += NB * NB;
  q.Wp = w; w += 64LL * NB * n;
  q.W2 = w; w += (long long)NB * n;
  q.tau = w; w += n;
  q.dg = w;
  return q;
}

rfm_status qr_init_device() {
  for (const void* fn : {(const void*)k_panel<1>, (const void*)k_panel<2>, (const void*)k_panel<4>})
    if (rfm_smem_attr(fn, KP_SMEM) != cudaSuccess) {  // once per device
      rfm_set_error("householder: device set-up failed");
      return RFM_ECUDA;
    }
  if (rfm_num_sms() == 0) {
    rfm_set_error("householder: device set-up failed");
    return RFM_ECUDA;
  }
  return RFM_OK;
}

// CTAs of k_panel in clusters of cl that can be resident together with the
// largest slab (depends on how the device's SMs are grouped), per device; 0 on failure.
template <int CL>
int kp_max_ctas() {
  static std::mutex mu;
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lk(mu);
  if (cached[dev] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL);
    cfg.blockDim = dim3(KP_THREADS);
    cfg.dynamicSmemBytes = KP_SMEM;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_panel<CL>, &cfg) != cudaSuccess) {
      cudaGetLastError();  // the caller takes a form without clusters; no later check may find this error
      return 0;
    }
    cached[dev] = n * CL;
  }
  return cached[dev];
}

// tags of an earlier factorisation must not be mistaken for this one's
rfm_status qr_begin(const QrScratch& q, cudaStream_t st) {
  RFM_CUDA(cudaMemsetAsync(q.xch, 0, 2LL * KP_SLOT * sizeof(unsigned long long), st));
  return RFM_OK;
}

// Factors the panel of nbw columns at j0 (rows j0..s) in place; *chunks and
// *chunk the row split of its sums.
rfm_status factor_panel(double* A, long long s, long long lda, long long j0, int nbw, cudaStream_t st,
                        const QrScratch& q, unsigned int* sync, int panel_cap, int* chunks, int* chunk_rows) {
  const int nsm = rfm_num_sms();
  const long long rows = s - j0;
  // chunks of at least 64 rows, one per SM (or per CTA of the cap) at most
  const long long cap = panel_cap > 0 ? std::min(panel_cap, nsm) : nsm;
  long long P = std::min<long long>(std::min<long long>((rows + 63) / 64, cap), KP_MAXP);
  if (P < 1) P = 1;
  long long chunk = (rows + P - 1) / P;
  if (chunk > KP_CHUNK && cap < nsm) {  // the cap's chunks would overflow shared memory: take the fewest that fit
    P = std::min<long long>((rows + KP_CHUNK - 1) / KP_CHUNK, nsm);
    chunk = (rows + P - 1) / P;
  }
  if (chunk > KP_CHUNK) {
    rfm_set_error("householder: sketch too tall for the panel kernel");
    return RFM_EINVAL;
  }
  PanelArgs a;
  a.A = A; a.lda = lda; a.s = s; a.j0 = j0; a.nbw = nbw; a.P = (int)P; a.chunk = (int)chunk;
  a.kpc = (int)((chunk + 31) / 32);
  a.xch = q.xch; a.tau = q.tau; a.err = sync + SYNC_ERR;
  // Clusters over the chunks of one remainder modulo 32, the largest size that
  // the cap allows and whose slab fits; else a CTA per chunk.
  const int ng = (int)std::min<long long>(P, 32), u = (int)((P + 31) / 32);
  auto fits = [&](int cl) {
    return (kp_fixed(cl, u) + kp_slab_rows(cl, u, a.kpc) * KP_LD) * (long long)sizeof(double) <= KP_SMEM;
  };
  int cl = 1;
  a.U = 1;
  a.NG = (int)P;
  if (ng * 4 <= std::min<long long>(panel_cap > 0 ? cap : 1 << 20, kp_max_ctas<4>()) && fits(4)) cl = 4;
  else if (ng * 2 <= std::min<long long>(panel_cap > 0 ? cap : 1 << 20, kp_max_ctas<2>()) && fits(2)) cl = 2;
  if (cl > 1) {
    a.U = u;
    a.NG = ng;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // all CTAs co-resident: they wait on each other's records
  at[0].val.cooperative = 1;
  cfg.gridDim = dim3((unsigned)(a.NG * cl));
  cfg.blockDim = dim3(KP_THREADS);
  cfg.dynamicSmemBytes = (size_t)((kp_fixed(cl, a.U) + kp_slab_rows(cl, a.U, a.kpc) * KP_LD) * sizeof(double));
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  ProfScope ps(PF_QR_PANEL, st);
  RFM_CUDA(cudaLaunchKernelEx(&cfg, cl == 4 ? k_panel<4> : cl == 2 ? k_panel<2> : k_panel<1>, a));
  RFM_CHECK_LAUNCH();
  *chunks = (int)P;
  *chunk_rows = (int)chunk;
  return RFM_OK;
}

// Householder factorisation of columns [c0, c1) (rows c0..s) in NB-wide
// panels; the FP64 compact-WY update of each panel is applied to the columns
// up to cend (cend >= c1).
rfm_status factor_range(double* A, long long s, long long lda, long long c0, long long c1, long long cend,
                        cudaStream_t st, const QrScratch& q, unsigned int* sync, int panel_cap) {
  const int nsm = rfm_num_sms();
  for (long long j0 = c0; j0 < c1; j0 += NB) {
    const int nbw = (int)std::min<long long>(NB, c1 - j0);
    const long long rows = s - j0;
    int chunks = 0, chunk = 0;
    RFM_TRY(factor_panel(A, s, lda, j0, nbw, st, q, sync, panel_cap, &chunks, &chunk));
    const long long j1 = j0 + nbw;
    const long long nt = cend - j1;
    if (nt <= 0) continue;
    // K slices: two per SM and 64-column tile, of 256 rows at least
    const long long ctiles = (nt + 63) / 64;
    long long nz = (2LL * nsm + ctiles - 1) / ctiles;
    nz = std::max<long long>(1, std::min<long long>(nz, std::min<long long>(64, (rows + 255) / 256)));
    const long long kchunk = (rows + nz - 1) / nz;
    nz = (rows + kchunk - 1) / kchunk;
    {
      ProfScope ps(PF_QR_VTA, st);
      rfm_prof_work(PF_QR_VTA, 2.0 * nbw * (double)nt * (double)rows);  // FP64 flops
      k_gram<<<(unsigned)chunks, 256, 0, st>>>(A, lda, s, j0, nbw, chunk, q.gram);
      RFM_CHECK_LAUNCH();
      k_panel_t<<<8, 64, 0, st>>>(q.gram, chunks, q.tau + j0, nbw, q.G, q.T);
      RFM_CHECK_LAUNCH();
      // the tile with the least FP64 work on the busiest SM, the widest of equals
      int tc = 64;
      long long cost = 0;
      for (int c : {64, 32, 16, 8}) {
        const long long v = ((nt + c - 1) / c * nz + nsm - 1) / nsm * c;
        if (c == 64 || v < cost) {
          cost = v;
          tc = c;
        }
      }
      const dim3 grid((unsigned)((nt + tc - 1) / tc), (unsigned)nz);
      if (tc == 64) k_vta<64><<<grid, vta_threads<64>(), 0, st>>>(A, lda, s, j0, nbw, j1, nt, kchunk, q.Wp);
      else if (tc == 32) k_vta<32><<<grid, vta_threads<32>(), 0, st>>>(A, lda, s, j0, nbw, j1, nt, kchunk, q.Wp);
      else if (tc == 16) k_vta<16><<<grid, vta_threads<16>(), 0, st>>>(A, lda, s, j0, nbw, j1, nt, kchunk, q.Wp);
      else k_vta<8><<<grid, vta_threads<8>(), 0, st>>>(A, lda, s, j0, nbw, j1, nt, kchunk, q.Wp);
      RFM_CHECK_LAUNCH();
      k_wt<<<(unsigned)((nt + 3) / 4), 128, 0, st>>>(q.Wp, (int)nz, q.T, nbw, nt, q.W2);
      RFM_CHECK_LAUNCH();
    }
    ProfScope psu(PF_QR_UPDATE, st);
    rfm_prof_work(PF_QR_UPDATE, 2.0 * nbw * (double)nt * (double)rows);  // FP64 flops
    k_update<<<dim3((unsigned)((rows + UR - 1) / UR), (unsigned)((nt + UC - 1) / UC)), 128, 0, st>>>(A, lda, s, j0, nbw, j1,
                                                                                                     nt, q.W2);
    RFM_CHECK_LAUNCH();
  }
  return RFM_OK;
}

// Positive diagonal and pivot floor; reads back the rank flag and the error word.
rfm_status finish_r(double* A, long long n, long long lda, cudaStream_t st, const QrScratch& q, unsigned int* sync,
                    int* rank_flag_host) {
  k_diag<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(A, lda, n, q.dg);
  RFM_CHECK_LAUNCH();
  k_flip<<<dim3((unsigned)std::min<long long>(64, (n + 255) / 256), (unsigned)n), 256, 0, st>>>(A, lda, n, q.dg);
  RFM_CHECK_LAUNCH();
  RFM_CUDA(cudaMemsetAsync(sync + SYNC_BAR + 2, 0, sizeof(unsigned int), st));
  k_floor<<<1, 1024, 0, st>>>(A, lda, n, sync + SYNC_BAR + 2);
  RFM_CHECK_LAUNCH();
  if (rank_flag_host) {
    unsigned int hv[2] = {0, 0};
    RFM_CUDA(cudaMemcpyAsync(hv, sync + SYNC_BAR + 2, sizeof(unsigned int), cudaMemcpyDeviceToHost, st));
    RFM_CUDA(cudaMemcpyAsync(hv + 1, sync + SYNC_ERR, sizeof(unsigned int), cudaMemcpyDeviceToHost, st));
    RFM_CUDA(cudaStreamSynchronize(st));
    *rank_flag_host = (int)hv[0];
    if (hv[1]) {
      rfm_set_error("householder: a bounded device wait timed out (code " + std::to_string(hv[1]) + ")");
      return RFM_ETIMEOUT;
    }
  }
  return RFM_OK;
}

}  // namespace

rfm_status rfm_householder_inplace(double* A, long long s, long long n, long long lda, cudaStream_t st,
                                   double* scratch, long long scratch_len, unsigned int* sync, int* rank_flag_host,
                                   int panel_cap, long long ncols) {
  if (s < n || n <= 0) {
    rfm_set_error("householder: need s >= n > 0");
    return RFM_EINVAL;
  }
  if (scratch_len < rfm_householder_scratch(s, n)) {
    rfm_set_error("householder: scratch too small");
    return RFM_EINVAL;
  }
  RFM_TRY(qr_init_device());
  const QrScratch q = carve(scratch, n);
  RFM_TRY(qr_begin(q, st));
  const long long c1 = ncols < 0 ? n : std::min<long long>(n, ((ncols + NB - 1) / NB) * NB);
  RFM_TRY(factor_range(A, s, lda, 0, c1, n, st, q, sync, panel_cap));
  return finish_r(A, n, lda, st, q, sync, rank_flag_host);
}

// ---------------------------------------------------------------------------
// Allocation-free Householder R.
//
// Same computation as rfm_householder_r, for callers that must not allocate
// device memory while they run: services that reserve all device memory up
// front through their own pool (where a cudaMalloc fails or implicitly
// synchronises the device and stalls other streams), or loops with fixed
// latency budgets.  The QR scratch lives in file-scope device arrays of fixed
// size (9.9 MB of scratch + 16 KB of barrier words per GPU that loads the
// library, held until the process exits), sized for n <= 512 columns.
// Every call shares these arrays and they keep the last call's contents;
// calls that overlap on the GPU (two streams, or two host threads) race on
// them and must be serialised by the caller.
#define RFM_NOALLOC_MAX_N 512
#define RFM_NOALLOC_MAX_DEVICES 64

namespace {
constexpr long long kNoallocScratch = qr_scratch_len(RFM_NOALLOC_MAX_N);
static_assert(kNoallocScratch * 8 == 9852416, "the size stated above and in rfm.h");
}  // namespace

static __device__ __align__(256) double g_noalloc_scratch[kNoallocScratch];
static __device__ __align__(256) unsigned int g_noalloc_sync[RFM_SYNC_WORDS];

namespace {

struct NoallocDev {
  double* scratch = nullptr;
  unsigned int* sync = nullptr;
};
NoallocDev g_noalloc_dev[RFM_NOALLOC_MAX_DEVICES];
std::mutex g_noalloc_mu;

__global__ void k_noalloc_copy_r(const double* __restrict__ A, long long lda, long long n, double* __restrict__ R) {
  const long long col = blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    R[(size_t)col * n + i] = i <= col ? A[(size_t)col * lda + i] : 0.0;
}

// Device addresses of the fixed arrays for the current device, resolved once
// per device (host code must not pass the arrays' host-side names to kernels).
rfm_status noalloc_setup(NoallocDev* out) {
  int dev = 0;
  RFM_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= RFM_NOALLOC_MAX_DEVICES) {
    rfm_set_error("rfm_householder_r_noalloc: device ordinal out of range");
    return RFM_EINVAL;
  }
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  NoallocDev& d = g_noalloc_dev[dev];
  if (!d.scratch) {
    void* ps = nullptr;
    void* py = nullptr;
    cudaError_t e1 = cudaGetSymbolAddress(&ps, g_noalloc_scratch);
    if (e1 != cudaSuccess) {
      rfm_set_error(std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e1));
      return RFM_ECUDA;
    }
    cudaError_t e2 = cudaGetSymbolAddress(&py, g_noalloc_sync);
    if (e2 != cudaSuccess) {
      rfm_set_error(std::string("cudaGetSymbolAddress(sync): ") + cudaGetErrorString(e2));
      return RFM_ECUDA;
    }
    d.scratch = static_cast<double*>(ps);
    d.sync = static_cast<unsigned int*>(py);
  }
  *out = d;
  return RFM_OK;
}

}  // namespace

extern "C" rfm_status rfm_householder_r_noalloc(double* A_dev, int64_t s, int64_t n, void* cuda_stream,
                                                double* R_dev, int* rank_flag_host) {
  if (!A_dev || !R_dev || n <= 0 || s < n) {
    rfm_set_error("rfm_householder_r_noalloc: need A, R and s >= n > 0");
    return RFM_EINVAL;
  }
  if (n > RFM_NOALLOC_MAX_N) {
    rfm_set_error("rfm_householder_r_noalloc: n = " + std::to_string(n) + " exceeds the fixed scratch limit of " +
                  std::to_string(RFM_NOALLOC_MAX_N) + " columns; use rfm_householder_r");
    return RFM_EINVAL;
  }
  NoallocDev d;
  RFM_TRY(noalloc_setup(&d));
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // barrier counters, flags and the error word must start at zero
  RFM_CUDA(cudaMemsetAsync(d.sync, 0, RFM_SYNC_WORDS * sizeof(unsigned int), st));
  int flag = 0;
  RFM_TRY(rfm_householder_inplace(A_dev, s, n, s, st, d.scratch, kNoallocScratch, d.sync, &flag));
  dim3 grid((unsigned)std::min<long long>(64, (n + 255) / 256), (unsigned)n);
  k_noalloc_copy_r<<<grid, 256, 0, st>>>(A_dev, s, n, R_dev);
  RFM_CHECK_LAUNCH();
  RFM_CUDA(cudaStreamSynchronize(st));
  if (rank_flag_host) *rank_flag_host = flag;
  return RFM_OK;
}

// ---------------------------------------------------------------------------
// Householder QR with the trailing update on the tensor cores.
//
// Blocks of QB = 128 columns are factored by factor_range (FP64 inside the
// block); the block's reflectors V (rows x 128, unit diagonal) update the columns
// to its right in compact-WY form
//     W = V^T A_t,  W2 = T^T W,  A_t -= V W2
// with all products on the emulated-FP64 tensor-core GEMM (digit splitting,
// exact level accumulation).  T (128 x 128) comes from the Gram V^T V, which the
// first product returns next to W, and the reflector coefficients,
// T_jj = tau_j, T_{:j,j} = -tau_j T_{:j,:j} G_{:j,j}.
//
// 128 columns are a quarter of the GEMM's exact chunk, so an update of depth 128
// drains its accumulators four times as often as it need.  Blocks of 512 columns,
// with V sliced without its unit diagonal, took 48 instead of 65 ms at n = 4,096
// and 613 instead of 980 ms at n = 16,384, and R was nearer to the exact one; but
// it was another R (by 1e-10), and one in three solves of n = 4,096 took another
// number of LSQR steps.

rfm_status rfm_oz_slice_house_v(const double* A, long long lda, long long j0, long long rows, long long nb, int ndig,
                                int* e, uint16_t* out, cudaStream_t st);
// Digit slices written into row tiles rt0 .. of planes holding plane_rtiles row
// tiles each, so that several slices form one GEMM operand.
rfm_status rfm_oz_slice_strided_at(const double* base, long long si, long long sk, long long R, long long K, int ndig,
                                   int tile_rows, int* e, uint16_t* out, long long plane_rtiles, long long rt0,
                                   cudaStream_t st);
rfm_status rfm_oz_slice_house_vt_at(const double* A, long long lda, long long j0, long long nb, long long K, int ndig,
                                    int tile_rows, int* e, uint16_t* out, long long plane_rtiles, long long rt0,
                                    cudaStream_t st);

namespace {

constexpr int QB = 128;
constexpr int QDIG = 8;

// T from G (symmetric) and tau: T_ij = -tau_j sum_{i <= l < j} T_il G_lj, l in
// turn.  One warp per row i of T, lanes = columns (four each): the rows are
// independent, and a step is one product and at most four multiply-adds.  (Column
// after column on one CTA took 447 us, this 34.)  T is row-major.
__global__ void __launch_bounds__(128) k_block_t(const double* __restrict__ G, const double* __restrict__ tau,
                                                 double* __restrict__ T) {
  constexpr int U = QB / 32;
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5);
  double v[U], row[U], tj[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    v[u] = row[u] = 0.0;
    tj[u] = tau[lane + 32 * u];
  }
#pragma unroll
  for (int h = 0; h < U; ++h)  // column l = 32 h + ll of the row is held in row[h]
    for (int ll = max(0, i - 32 * h); ll < 32; ++ll) {
      const int l = 32 * h + ll;
      double g[U];
#pragma unroll
      for (int u = h; u < U; ++u) g[u] = G[(size_t)l * QB + lane + 32 * u];
      if (lane == ll) row[h] = l == i ? tj[h] : -tj[h] * v[h];
      const double t = __shfl_sync(0xffffffffu, row[h], ll);
#pragma unroll
      for (int u = h; u < U; ++u)
        if (u > h || lane > ll) v[u] = fma(t, g[u], v[u]);
    }
#pragma unroll
  for (int u = 0; u < U; ++u) T[(size_t)i * QB + lane + 32 * u] = row[u];
}

}  // namespace

long long rfm_householder_emulated_bytes(long long s, long long n) {
  long long b = 0;
  b += rfm_oz_digit_bytes(n + QB, s, QDIG, 64);  // [V, A_t]: the Gram and V^T A_t in one product
  b += rfm_oz_digit_bytes(QB, QB, QDIG, 128);    // T^T
  b += rfm_oz_digit_bytes(s, QB, QDIG, 128);     // V
  b += rfm_oz_digit_bytes(n, QB, QDIG, 64);      // W2
  b += 8LL * (2LL * QB * (n + QB) + QB * QB);    // [G, W], W2, T
  b += 8LL * 8 * QB * (n + QB);                  // split-K partials of V^T [V, A_t]
  b += 4LL * (QB + n + QB + s + n) + 4096;
  return b;
}

rfm_status rfm_householder_emulated(double* A, long long s, long long n, long long lda, cudaStream_t st,
                                    double* scratch, long long scratch_len, unsigned int* sync, void* emu,
                                    long long emu_bytes, int* rank_flag_host, int panel_cap, long long ncols) {
  if (s < n || n <= 0) {
    rfm_set_error("householder: need s >= n > 0");
    return RFM_EINVAL;
  }
  if (scratch_len < rfm_householder_scratch(s, n) || emu_bytes < rfm_householder_emulated_bytes(s, n)) {
    rfm_set_error("householder: scratch too small");
    return RFM_EINVAL;
  }
  RFM_TRY(qr_init_device());
  const QrScratch q = carve(scratch, n);
  char* w = static_cast<char*>(emu);
  auto take = [&](long long bytes) {
    char* r = w;
    w += (bytes + 255) & ~255LL;
    return r;
  };
  uint16_t* d_at = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(n + QB, s, QDIG, 64)));
  uint16_t* d_t = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(QB, QB, QDIG, 128)));
  uint16_t* d_v = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(s, QB, QDIG, 128)));
  uint16_t* d_w2 = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(n, QB, QDIG, 64)));
  double* Wm = reinterpret_cast<double*>(take(8LL * QB * (n + QB)));  // [G, W] = V^T [V, A_t]
  double* W2 = reinterpret_cast<double*>(take(8LL * QB * n));
  double* T = reinterpret_cast<double*>(take(8LL * QB * QB));
  const long long part_elems = 8LL * QB * (n + QB);
  double* part = reinterpret_cast<double*>(take(8LL * part_elems));
  int* e_at = reinterpret_cast<int*>(take(4LL * (n + QB)));
  int* e_t = reinterpret_cast<int*>(take(4LL * QB));
  int* e_v = reinterpret_cast<int*>(take(4LL * s));
  int* e_w2 = reinterpret_cast<int*>(take(4LL * n));
  unsigned int* err = sync + SYNC_ERR;
  RFM_TRY(qr_begin(q, st));
  const long long cstop = ncols < 0 ? n : std::min<long long>(n, ncols);
  for (long long J0 = 0; J0 < cstop; J0 += QB) {
    const long long c1 = std::min<long long>(n, J0 + QB);
    const long long rows = s - J0, nt = n - c1;
    RFM_TRY(factor_range(A, s, lda, J0, c1, c1, st, q, sync, panel_cap));
    if (nt <= 0) break;
    {
      // One emulated product gives the block's Gram and V^T A_t: its B operand
      // is [V, A_t] (V^T as the first two 64-row tiles, then the trailing
      // columns), its A operand the same V^T tiles, so C = [G, W] with G = V^T V
      // (exactly symmetric: the digit pairs (p, q) and (q, p) give the same
      // integer level sums).
      ProfScope ps(PF_QR_VTA, st);
      const long long prt = QB / 64 + (nt + 63) / 64;  // row tiles of the B operand
      RFM_TRY(rfm_oz_slice_house_vt_at(A, lda, J0, QB, rows, QDIG, 64, e_at, d_at, prt, 0, st));
      RFM_TRY(rfm_oz_slice_strided_at(A + (size_t)c1 * lda + J0, lda, 1, nt, rows, QDIG, 64, e_at + QB, d_at, prt,
                                      QB / 64, st));
      RFM_TRY(rfm_oz_gemm_part(d_at, QDIG, e_at, d_at, QDIG, e_at, QB, QB + nt, rows, QDIG + 1, Wm, QB, 0, err, st,
                               part, part_elems, prt));
      k_block_t<<<QB / 4, 128, 0, st>>>(Wm, q.tau + J0, T);
      RFM_CHECK_LAUNCH();
      // W2 = T^T W on the emulated GEMM as well (M = K = 128, N = nt).
      // T is stored row-major, T(q, p) = T[q QB + p], so T^T(p, q) = T[p + q QB].
      RFM_TRY(rfm_oz_slice_strided(T, 1, QB, QB, QB, QDIG, 128, e_t, d_t, st));
      RFM_TRY(rfm_oz_slice_strided(Wm + (size_t)QB * QB, QB, 1, nt, QB, QDIG, 64, e_w2, d_w2, st));
      RFM_TRY(rfm_oz_gemm(d_t, QDIG, e_t, d_w2, QDIG, e_w2, QB, nt, QB, QDIG + 1, W2, QB, 0, err, st));
    }
    ProfScope ps(PF_QR_UPDATE, st);
    RFM_TRY(rfm_oz_slice_house_v(A, lda, J0, rows, QB, QDIG, e_v, d_v, st));
    RFM_TRY(rfm_oz_slice_strided(W2, QB, 1, nt, QB, QDIG, 64, e_w2, d_w2, st));
    RFM_TRY(rfm_oz_gemm(d_v, QDIG, e_v, d_w2, QDIG, e_w2, rows, nt, QB, QDIG + 1, A + (size_t)c1 * lda + J0, lda, 1,
                        err, st));
  }
  return finish_r(A, n, lda, st, q, sync, rank_flag_host);
}
