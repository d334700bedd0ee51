// Householder QR of the sketch B = S_k J (Sec. 4.1, "thin QR B = Q R") giving
// the right preconditioner R.  Blocked right-looking Householder with the
// compact-WY trailing update (Schreiber & Van Loan):
//
//   k_block     (cooperative) factors a block of up to 128 columns (32 when the
//               trailing update is in FP64), one exchange between the CTAs per
//               column.  Reflector H = I - tau v v^T, v_0 = 1,
//               beta = -sign(alpha) ||x||.
//   k_vta       W_z = V^T A_trail over a K-slice z (split K, deterministic)
//   k_wt        W2 = T^T sum_z W_z, T the panel's compact-WY factor
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
// Cooperative block factorisation k_block.
//
// GB300's FP64 unit takes 64 cycles (31 ns) for a warp instruction, the same
// for a dependent chain as for independent ones and for one lane as for 32
// (measured).  What bounds a column of the factorisation is therefore the
// number of FP64 warp instructions on one SM partition, plus one exchange
// between the CTAs; the kernel is laid out to issue few of them:
//  - 4 warps per CTA, one per SM partition; the lanes of a warp are the 32
//    columns of the panel, so a row of the panel is one instruction and no
//    reduction over lanes is needed.  A warp owns every fourth row.
//  - the columns k < j already hold their reflectors u_k, so the same
//    instruction that gives x^T a_k for the columns to the right (and
//    sigma = x^T x in lane j) gives u_k^T x for the columns to the left: the
//    panel's Gram comes with the reduction and needs no pass of its own.
//  - H = I - gamma u u^T with the unscaled u = (alpha - beta, x) and
//    gamma = 1 / (beta (beta - alpha)): the column is scaled once, at the end
//    of the panel.  sqrt and the reciprocal are one third-order step
//    (Householder's iteration) from an FP32 seed, 18 instructions where the
//    library's sqrt and two divisions take 28 (0.86 us).
//  - a column's reflector is applied to the next column at once and to the others
//    while the next column's exchange is on its way.  The next column's products
//    are then taken with a_k still lacking that reflector f_k u, and
//    x^T (a_k - f_k u) = x^T a_k - f_k x^T u is formed after the sum, x^T u being
//    the Gram entry in its lane.  The error against ||x|| ||a_k|| is that of the
//    step before, so the sum of all steps' errors is the same.
//  - the 32 sums are first combined in clusters of four CTAs (each rank sums
//    eight columns of the 16 warps, through distributed shared memory and one
//    cluster barrier, 0.2 us), then between the clusters as 16-byte records
//    {low, tag, high, tag} whose tag is the column's number: a reader polls the
//    records themselves, so there is no fence, no counter and no second trip to
//    L2.  Two slots alternate; a CTA can only be one exchange ahead of another.
//    (With a record per CTA every CTA read 78 KB per column, which is L2 bound,
//    and added 38 records per warp.)  Four is the largest cluster that still
//    puts a CTA on 144 of the 152 SMs (eight: 120).
// Between the panels of a block, the block's remaining columns (in the same
// shared-memory slab) are updated with W = V^T A, W2 = T^T W, A -= V W2: CTA c
// sums column c of W over the CTAs and solves for its column of W2.
//
// Per column at 12,288 rows: 16.5 us with one grid barrier and a redundant
// butterfly reduction per column (the former panel kernel), then 5.2 us (0.95
// products, 0.4 cluster barrier, 0.25 publish, 1.7 poll and sums, 1.05 scalars,
// 0.8 update).  The poll leaves the FP64 pipes idle, so only the next column is
// updated at once; a reflector's other columns follow while the next column's
// records are on their way.  A 128-column block with its in-block updates: 3.7
// -> 0.94 ms, with the deferred updates 0.87 ms.
constexpr int KB_THREADS = 128;
constexpr int KB_SMEM = 227 * 1024;              // dynamic shared memory of a CTA
constexpr long long KB_WIDE_ROWS = 16384;
constexpr int KB_CL = 4;                         // CTAs of a cluster
constexpr int KB_MAXP = 256;                     // CTAs of one factorisation
constexpr int KB_POLL = 10;                      // records in flight per lane and poll round
constexpr int KB_SLOT = (KB_MAXP / KB_CL + 1) * NB * 2;  // 8-byte words of an exchange slot (last record: the pivot row)

struct BlockArgs {
  double* A;
  long long lda;
  long long s;
  long long j0;
  int nb;              // columns of the block (<= 128)
  int P;               // CTAs (a multiple of KB_CL)
  int chunk;           // rows per CTA
  unsigned long long* xch;  // [2][KB_SLOT] exchange records
  double* part;        // [P][3 NB][NB] partial W of the in-block update
  double* w2;          // [NB][3 NB]
  double* tau;         // [n]
  double* G;           // [NB][NB] of the last panel: G[p * NB + q] = tau_p v_q^T v_p for q < p, else 0
  unsigned int* bar;   // arrival counter of the grid barriers
  unsigned int bar0;   // its value before this launch
  unsigned int* err;
};

constexpr int KB_TRI = NB * (NB - 1) / 2;  // entries q < p of the panel's Gram
__host__ __device__ constexpr int kb_tri(int p, int q) { return p * (p - 1) / 2 + q; }
__host__ __device__ constexpr size_t kb_fixed_smem() { return (size_t)(KB_TRI + 13 * NB) * sizeof(double); }

// Slab element (local row r, column c): 32-column groups with the column index
// XORed by the row, so that both a row (lanes = columns) and a column (lanes =
// rows) are free of bank conflicts.
__device__ __forceinline__ int kb_at(int r, int c, int ld) { return r * ld + (c & ~31) + ((c ^ r) & 31); }

// Arrivals of all CTAs up to the count `want` (the counter only grows).
__device__ __forceinline__ void kb_barrier(unsigned int* bar, unsigned int want, RecWait& kw) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned int n = 0;
    while ((int)(ld_acquire(bar) - want) < 0)
      if (!kw.spin(n)) break;
  }
  __syncthreads();
}

// x != 0 (true for NaN) without an FP64 compare.
__device__ __forceinline__ bool kb_nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }

// norm = sqrt(alpha^2 + sigma) and gamma = 1 / (norm^2 + |alpha| norm) for
// sigma > 0.  In the scaled variables m = t 2^-e in [1, 4) (e even), the
// seeds are FP32 (2^-21) and one step of third order leaves ~2^-63; sqrt gets
// one Newton correction.  Exponents near the ends of the range (and Inf, NaN)
// take the library functions.
__device__ __forceinline__ void kb_norm_gamma(double alpha, double sigma, double& nrm, double& gam) {
  const double t = fma(alpha, alpha, sigma);
  const int hi = __double2hiint(t), lo = __double2loint(t);
  const int ex = ((hi >> 20) & 0x7FF) - 1023;
  if (ex < -900 || ex > 900 || hi < 0) {
    nrm = sqrt(t);
    gam = 1.0 / fma(fabs(alpha), nrm, t);
    return;
  }
  const int e = ex & ~1;
  const int mh = hi - (e << 20);  // m = t 2^-e
  const double m = __hiloint2double(mh, lo);
  // FP32 value of m with its low bits cut off (integer operations only)
  const float mf = __int_as_float(((mh >> 20) - 1023 + 127) << 23 | (mh & 0xFFFFF) << 3 | (int)((unsigned)lo >> 29));
  const int yb = __float_as_int(rsqrtf(mf));
  const double y0 = __hiloint2double((((yb >> 23) - 127 + 1023) << 20) | ((yb & 0x7FFFFF) >> 3), (int)((unsigned)(yb & 7) << 29));
  const double h = m * y0;
  const double r = fma(-h, y0, 1.0);
  const double y = fma(y0, fma(r, 0.375, 0.5) * r, y0);  // 1 / sqrt(m)
  double q = m * y;                                        // sqrt(m)
  const double half_y = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));
  q = fma(fma(-q, q, m), half_y, q);
  const double back = __hiloint2double((1023 - (e >> 1)) << 20, 0);  // 2^(-e/2)
  const double d = fma(fabs(alpha) * back, q, m);                    // in [1, 8)
  const int dh = __double2hiint(d), dl = __double2loint(d);
  const float df = __int_as_float(((dh >> 20) - 1023 + 127) << 23 | (dh & 0xFFFFF) << 3 | (int)((unsigned)dl >> 29));
  const int gb = __float_as_int(__frcp_rn(df));
  const double g0 = __hiloint2double((((gb >> 23) - 127 + 1023) << 20) | ((gb & 0x7FFFFF) >> 3), (int)((unsigned)(gb & 7) << 29));
  const double w = fma(-d, g0, 1.0);
  const double g = fma(g0, fma(w, w, w), g0);  // 1 / d
  nrm = __hiloint2double(__double2hiint(q) + ((e >> 1) << 20), __double2loint(q));
  gam = __hiloint2double(__double2hiint(g) - (e << 20), __double2loint(g));
}

__device__ __forceinline__ void kb_copy8(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// In-block W = V^T A of a CTA's rows: lanes are the columns of a group, warp w
// takes p = 8 w .. 8 w + 7, NG groups of columns follow the panel at p0.
template <int NG>
__device__ __forceinline__ void kb_wpart(const double* sl, int ld, int p0, int r0, int nr, int w, int lane,
                                         double* out) {
  double acc[NG][8];
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int p = 0; p < 8; ++p) acc[g][p] = 0.0;
#pragma unroll 2
  for (int r = r0; r < nr; ++r) {
    double av[NG], v[8];
#pragma unroll
    for (int g = 0; g < NG; ++g) av[g] = sl[kb_at(r, p0 + NB * (g + 1) + lane, ld)];
#pragma unroll
    for (int p = 0; p < 8; ++p) v[p] = sl[kb_at(r, p0 + 8 * w + p, ld)];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
      for (int g = 0; g < NG; ++g) acc[g][p] = fma(v[p], av[g], acc[g][p]);
  }
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int p = 0; p < 8; p += 2)
      __stcg(reinterpret_cast<double2*>(out + (g * NB + lane) * NB + 8 * w + p),
             make_double2(acc[g][p], acc[g][p + 1]));
}

// In-block A -= V W2 of a CTA's rows for the column group at pc: a lane keeps
// its column of W2.
__device__ __forceinline__ void kb_wupdate(double* sl, int ld, int p0, int pc, int r0, int nr, int w, int lane,
                                           const double* w2) {
  double y[NB];
#pragma unroll
  for (int p = 0; p < NB; ++p) y[p] = __ldcg(w2 + p * (3 * NB) + lane);
  for (int r = r0 + ((w - r0) & 3); r < nr; r += 4) {
    double* e = sl + kb_at(r, pc + lane, ld);
    const double* v = sl + r * ld + p0;
    // summed by itself and subtracted once: 32 roundings at the size of the sum, not of A
    double x = 0.0;
#pragma unroll
    for (int p = 0; p < NB; ++p) x = fma(v[(p ^ r) & 31], y[p], x);
    *e -= x;
  }
}

// A_rk -= f_k u_r for this warp's rows r >= r0 of the panel at p0, u its column jj,
// f the lanes' factors (0 up to column jj + 1, which is up to date).
__device__ __forceinline__ void kb_apply(double* sl, int ld, int p0, int jj, double f, int r0, int nr, int w,
                                         int lane) {
  const int rw = r0 + ((w - r0) & 3);
  if (jj < 15) {
    if (rw < nr) {
      const int last = nr - 1 - ((nr - 1 - rw) & 3);
      double x = sl[kb_at(rw, p0 + jj, ld)], e = sl[kb_at(rw, p0 + lane, ld)];
#pragma unroll 4
      for (int r = rw; r < last; r += 4) {
        const double xn = sl[kb_at(r + 4, p0 + jj, ld)], en = sl[kb_at(r + 4, p0 + lane, ld)];
        sl[kb_at(r, p0 + lane, ld)] = fma(-f, x, e);
        x = xn;
        e = en;
      }
      sl[kb_at(last, p0 + lane, ld)] = fma(-f, x, e);
    }
  } else {
    // only columns 17 .. 31 are left: two rows per instruction
    const int ch = 16 + (lane & 15);
    const double fh = __shfl_sync(0xffffffffu, f, ch);
    int r = rw + 4 * (lane >> 4);
    for (; r + 24 < nr; r += 32) {
      double x[4], e[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x[u] = sl[kb_at(r + 8 * u, p0 + jj, ld)];
        e[u] = sl[kb_at(r + 8 * u, p0 + ch, ld)];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        e[u] = fma(-fh, x[u], e[u]);
        if (ch > jj + 1) sl[kb_at(r + 8 * u, p0 + ch, ld)] = e[u];
      }
    }
    for (; r < nr; r += 8) {
      double* e = sl + kb_at(r, p0 + ch, ld);
      const double x = fma(-fh, sl[kb_at(r, p0 + jj, ld)], *e);
      if (ch > jj + 1) *e = x;
    }
  }
  __syncwarp();
}

__global__ void __cluster_dims__(KB_CL, 1, 1) __launch_bounds__(KB_THREADS, 1) k_block(BlockArgs a) {
  if (!in_cluster(KB_CL, a.err)) return;
  extern __shared__ __align__(16) double kb_sm[];
  double* Gs = kb_sm;              // tau_p v_q^T v_p of the panel at kb_tri(p, q), q < p
  double* wp = Gs + KB_TRI;        // [4][4][8] partial sums of this rank's 8 columns, by CTA and warp of the cluster
  double* rs = wp + 4 * NB;        // [4][NB] the warps' shares of the sums over CTAs
  double* pv = rs + 4 * NB;        // [NB] pivot row
  double* dab = pv + NB;           // [NB] alpha - beta
  double* gam = dab + NB;          // [NB] gamma
  double* scl = gam + NB;          // [NB] 1 / (alpha - beta)
  double* taus = scl + NB;         // [NB]
  double* sl = kb_sm + (kb_fixed_smem() / sizeof(double));  // slab [rows][ld]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int c = blockIdx.x, P = a.P;
  const int rank = c % KB_CL, cl = c / KB_CL, ncl = P / KB_CL;
  const long long rbeg = a.j0 + (long long)c * a.chunk;
  const long long rend = min(a.s, rbeg + a.chunk);
  const int nr = rbeg < rend ? (int)(rend - rbeg) : 0;
  const int np = (a.nb + NB - 1) / NB, ld = np * NB;
  RecWait kw(a.err, tid);
  unsigned int barrier = a.bar0;
  for (int cc = w; cc < ld; cc += 4) {
    const double* col = a.A + (size_t)(a.j0 + cc) * a.lda + rbeg;
    for (int r = lane; r < nr; r += 32) {
      if (cc < a.nb) kb_copy8(sl + kb_at(r, cc, ld), col + r);
      else sl[kb_at(r, cc, ld)] = 0.0;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  cluster_arrive();
  cluster_wait();  // all ranks run: their shared memory may be written
  for (int pi = 0; pi < np; ++pi) {
    const int p0 = pi * NB, nbw = min(NB, a.nb - p0);
    double fprev = 0.0;  // factors of the previous column's reflector that columns past jj still lack
    for (int jj = 0; jj < nbw; ++jj) {
      const long long j = a.j0 + p0 + jj;  // pivot row and column
      const unsigned int tag = (unsigned int)(j + 1);
      unsigned long long* slot = a.xch + (size_t)(jj & 1) * KB_SLOT;
      const int lr = j + 1 > rbeg ? (int)min((long long)nr, j + 1 - rbeg) : 0;  // rows below the pivot
      const int rw = lr + ((w - lr) & 3);                                       // this warp's first one
      double acc = 0.0;
      if (rw < nr) {  // the next row's loads go ahead of a row's instruction
        const int last = nr - 1 - ((nr - 1 - rw) & 3);
        double x = sl[kb_at(rw, p0 + jj, ld)], e = sl[kb_at(rw, p0 + lane, ld)];
#pragma unroll 4
        for (int r = rw; r < last; r += 4) {
          const double xn = sl[kb_at(r + 4, p0 + jj, ld)], en = sl[kb_at(r + 4, p0 + lane, ld)];
          acc = fma(x, e, acc);
          x = xn;
          e = en;
        }
        acc = fma(x, e, acc);
      }
      st_cluster(wp + (rank * 4 + w) * 8 + (lane & 7), lane >> 3, acc);
      cluster_arrive();
      cluster_wait();
      if (w == 0) {
        const double* x = wp + (lane >> 3) * 32 + (lane & 7);
        double sm = (x[0] + x[8]) + (x[16] + x[24]);
        sm += __shfl_xor_sync(0xffffffffu, sm, 8);
        sm += __shfl_xor_sync(0xffffffffu, sm, 16);
        if (lane < 8) rec_publish(slot + ((size_t)cl * NB + rank * 8 + lane) * 2, sm, tag);
      } else if (w == 1 && j >= rbeg && j < rend) {
        const int r = (int)(j - rbeg);
        double v = sl[kb_at(r, p0 + lane, ld)];
        if (jj > 0) v = fma(-fprev, sl[kb_at(r, p0 + jj - 1, ld)], v);
        rec_publish(slot + ((size_t)ncl * NB + lane) * 2, v, tag);
      }
      // meanwhile the previous column's reflector on the columns past jj
      if (jj > 0) {
        if (j >= rbeg && j < rend) __syncthreads();  // warp 1 has read the pivot row
        kb_apply(sl, ld, p0, jj - 1, fprev, j > rbeg ? (int)min((long long)nr, j - rbeg) : 0, nr, w, lane);
      }
      // sum over the clusters, warp w the clusters w, w + 4, ... in increasing
      // order; record ncl is the pivot row.  A complete record of this cluster
      // also says that all its ranks have read wp.
      double sum = 0.0;
      for (int q0 = w; q0 <= ncl; q0 += 4 * KB_POLL) {
        unsigned long long lo[KB_POLL], hi[KB_POLL];
        unsigned int spins = 0;
        for (;;) {
          bool all = true;
#pragma unroll
          for (int i = 0; i < KB_POLL; ++i)
            if (q0 + 4 * i <= ncl) rec_load(slot + ((size_t)(q0 + 4 * i) * NB + lane) * 2, lo[i], hi[i]);
#pragma unroll
          for (int i = 0; i < KB_POLL; ++i)
            if (q0 + 4 * i <= ncl) all = all && rec_ready(lo[i], hi[i], tag);
          if (__all_sync(0xffffffffu, all) || !__all_sync(0xffffffffu, kw.spin(spins))) break;
        }
#pragma unroll
        for (int i = 0; i < KB_POLL; ++i) {
          const int q = q0 + 4 * i;
          if (q < ncl) sum += rec_value(lo[i], hi[i]);
          else if (q == ncl) pv[lane] = rec_value(lo[i], hi[i]);
        }
      }
      rs[w * NB + lane] = sum;
      __syncthreads();
      double tot = (rs[lane] + rs[NB + lane]) + (rs[2 * NB + lane] + rs[3 * NB + lane]);
      if (jj > 0) tot = fma(-fprev, __shfl_sync(0xffffffffu, tot, jj - 1), tot);
      const double piv = pv[lane];
      const double alpha = pv[jj];
      const double sigma = __shfl_sync(0xffffffffu, tot, jj);
      double dj = 0.0, gj = 0.0, beta = alpha;
      if (kb_nonzero(sigma)) {
        double nrm;
        kb_norm_gamma(alpha, sigma, nrm, gj);
        beta = __double2hiint(alpha) < 0 && kb_nonzero(alpha) ? nrm : -nrm;
        dj = alpha - beta;
      }
      // u^T a_k for the columns to the right, u_k^T u for those to the left
      const double wk = fma(dj, piv, tot);
      const double f = lane > jj ? gj * wk : 0.0;
      if (w == 0) {
        if (lane < jj) Gs[kb_tri(jj, lane)] = wk;
        if (lane == jj) {
          dab[jj] = dj;
          gam[jj] = gj;
        }
      }
      // the next column only (lanes are rows); the others wait for the next exchange
      if (jj + 1 < NB) {
        const double f1 = __shfl_sync(0xffffffffu, f, jj + 1);
        for (int r = rw + 4 * lane; r < nr; r += 128) {
          double* e = sl + kb_at(r, p0 + jj + 1, ld);
          *e = fma(-f1, sl[kb_at(r, p0 + jj, ld)], *e);
        }
      }
      fprev = lane > jj + 1 ? f : 0.0;
      if (j >= rbeg && j < rend && w == ((int)(j - rbeg) & 3)) {  // the pivot row itself
        double* e = sl + kb_at((int)(j - rbeg), p0 + lane, ld);
        if (lane > jj) *e = fma(-f, dj, *e);
        if (lane == jj) *e = beta;
      }
      __syncwarp();
    }
    __syncthreads();
    if (w == 0) {
      const double d = lane < nbw ? dab[lane] : 0.0;
      const bool on = d != 0.0;
      scl[lane] = on ? 1.0 / d : 0.0;
      taus[lane] = on ? gam[lane] * (d * d) : 0.0;
      if (c == 0 && lane < nbw) a.tau[a.j0 + p0 + lane] = taus[lane];
    }
    __syncthreads();
    for (int idx = tid; idx < NB * NB; idx += KB_THREADS) {
      const int p = idx / NB, q = idx % NB;
      double g = 0.0;
      if (q < p && p < nbw) {
        g = Gs[kb_tri(p, q)] * scl[q] * scl[p] * taus[p];
        Gs[kb_tri(p, q)] = g;
      }
      if (c == 0) a.G[idx] = g;
    }
    // R on and above the diagonal and v below to global memory; the slab keeps
    // v with its unit diagonal and zeros above
    for (int cc = w; cc < nbw; cc += 4) {
      const long long pr = a.j0 + p0 + cc;  // this column's pivot row
      double* col = a.A + (size_t)pr * a.lda + rbeg;
      const double sc = scl[cc];
      for (int r = lane; r < nr; r += 32) {
        double* e = sl + kb_at(r, p0 + cc, ld);
        const long long gr = rbeg + r;
        const double v = gr > pr ? *e * sc : *e;
        col[r] = v;
        *e = gr > pr ? v : (gr == pr ? 1.0 : 0.0);
      }
    }
    __syncthreads();
    const int ng = np - 1 - pi;  // column groups to the right in the block
    if (ng == 0) break;  // the last cluster barrier came after the last remote store
    const long long first = a.j0 + p0;
    const int lv = first > rbeg ? (int)min((long long)nr, first - rbeg) : 0;  // rows before are zero in V
    if (ng == 3) kb_wpart<3>(sl, ld, p0, lv, nr, w, lane, a.part + (size_t)c * 3 * NB * NB);
    else if (ng == 2) kb_wpart<2>(sl, ld, p0, lv, nr, w, lane, a.part + (size_t)c * 3 * NB * NB);
    else kb_wpart<1>(sl, ld, p0, lv, nr, w, lane, a.part + (size_t)c * 3 * NB * NB);
    barrier += P;
    kb_barrier(a.bar, barrier, kw);
    for (int col = c; col < ng * NB; col += P) {
      double sum = 0.0;
      for (int q0 = w; q0 < P; q0 += 4 * KB_POLL) {
        double t[KB_POLL];
#pragma unroll
        for (int i = 0; i < KB_POLL; ++i) {
          const int q = q0 + 4 * i;
          t[i] = q < P ? __ldcg(a.part + ((size_t)q * 3 * NB + col) * NB + lane) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < KB_POLL; ++i)
          if (q0 + 4 * i < P) sum += t[i];
      }
      rs[w * NB + lane] = sum;
      __syncthreads();
      if (w == 0) {
        // W2 = T^T W from T^-1 = diag(1 / tau) + strict upper part of V^T V:
        // y_p = tau_p w_p - sum_{q<p} (tau_p v_q^T v_p) y_q
        double x = ((rs[lane] + rs[NB + lane]) + (rs[2 * NB + lane] + rs[3 * NB + lane])) * taus[lane];
        for (int q = 0; q < nbw; ++q) {
          const double y = __shfl_sync(0xffffffffu, x, q);
          if (lane > q && lane < nbw) x = fma(-Gs[kb_tri(lane, q)], y, x);
        }
        __stcg(a.w2 + lane * (3 * NB) + col, x);
      }
      __syncthreads();
    }
    barrier += P;
    kb_barrier(a.bar, barrier, kw);
    for (int g = 0; g < ng; ++g) kb_wupdate(sl, ld, p0, p0 + NB * (g + 1), lv, nr, w, lane, a.w2 + g * NB);
    __syncthreads();
  }
}

// Vector of panel column p at global row gr (unit pivot, zero above).
__device__ __forceinline__ double vval(const double* A, long long lda, long long j0, int p, long long gr) {
  const long long piv = j0 + p;
  if (gr < piv) return 0.0;
  if (gr == piv) return 1.0;
  return A[(size_t)(j0 + p) * lda + gr];
}

// Wp[z][col][p] = sum_{r in K-slice z} v_p(r) A[r, j1 + col]
__global__ void __launch_bounds__(256) k_vta(const double* __restrict__ A, long long lda, long long s, long long j0,
                                             int nbw, long long j1, long long nt, long long kchunk,
                                             double* __restrict__ Wp) {
  __shared__ double Vs[32][NB + 1];
  __shared__ double As[32][64 + 1];
  const int tid = threadIdx.x;
  const long long col0 = (long long)blockIdx.x * 64;
  const int z = blockIdx.y;
  const long long kb = j0 + (long long)z * kchunk;
  const long long ke = min(s, kb + kchunk);
  const int ay = tid >> 4, cx = tid & 15;
  double acc[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
  for (long long r0 = kb; r0 < ke; r0 += 32) {
    for (int idx = tid; idx < 32 * NB; idx += 256) {
      const int rr = idx & 31, p = idx >> 5;
      const long long gr = r0 + rr;
      Vs[rr][p] = (gr < ke && p < nbw) ? vval(A, lda, j0, p, gr) : 0.0;
    }
    for (int idx = tid; idx < 32 * 64; idx += 256) {
      const int rr = idx & 31, cc = idx >> 5;
      const long long gr = r0 + rr, gc = col0 + cc;
      As[rr][cc] = (gr < ke && gc < nt) ? A[(size_t)(j1 + gc) * lda + gr] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int rr = 0; rr < 32; ++rr) {
      const double v0 = Vs[rr][ay], v1 = Vs[rr][ay + 16];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double av = As[rr][cx + 16 * q];
        acc[0][q] += v0 * av;
        acc[1][q] += v1 * av;
      }
    }
    __syncthreads();
  }
  for (int h = 0; h < 2; ++h)
    for (int q = 0; q < 4; ++q) {
      const long long gc = col0 + cx + 16 * q;
      const int p = ay + 16 * h;
      if (gc < nt) Wp[((size_t)z * nt + gc) * NB + p] = acc[h][q];
    }
}

// W2 = T^T sum_z Wp[z], one warp per column, lanes = p.  T is not formed: with
// T^-1 = diag(1 / tau) + strict upper part of V^T V the column is a forward
// substitution, y_p = tau_p w_p - sum_{q<p} G_pq y_q with G_pq = tau_p v_q^T v_p.
// Both the sum over z and the substitution are chains of FP64 instructions of
// 31 ns; one column per warp leaves them short and all columns independent.
// (The form with one thread per column and T^T W took 120 us at 12,288 rows.)
__global__ void __launch_bounds__(128) k_wt(const double* __restrict__ Wp, int nz, const double* __restrict__ G,
                                            const double* __restrict__ tau, int nbw, long long nt,
                                            double* __restrict__ W2) {
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
  x = lane < nbw ? x * tau[lane] : 0.0;
  double g[NB];
#pragma unroll
  for (int q = 0; q < NB; ++q) g[q] = G[lane * NB + q];  // 0 for q >= lane
#pragma unroll
  for (int q = 0; q < NB; ++q) x = fma(-g[q], __shfl_sync(0xffffffffu, x, q), x);
  W2[(size_t)lane * nt + col] = x;
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
  unsigned long long* xch;  // exchange records of k_block
  double* part;             // its partial products of the in-block update
  double* bw2;              // and their W2
  double* tau;
  double* G;
  double* Wp;
  double* W2;
  double* dg;
};

}  // namespace

// Doubles of the panel scratch: exchange records, in-block partials and W2 of
// k_block, tau, G, and the split-K partials, W2 and diagonal of the trailing update.
__host__ __device__ constexpr long long qr_scratch_len(long long n) {
  return 2LL * KB_SLOT + (long long)KB_MAXP * 3 * NB * NB + 3LL * NB * NB + n + NB * NB + 64LL * NB * n + NB * n + n +
         64;
}

long long rfm_householder_scratch(long long s, long long n) {
  (void)s;
  return qr_scratch_len(n);
}

namespace {

QrScratch carve(double* scratch, long long n) {
  QrScratch q;
  double* w = scratch;
  q.xch = reinterpret_cast<unsigned long long*>(w); w += 2LL * KB_SLOT;
  q.part = w; w += (long long)KB_MAXP * 3 * NB * NB;
  q.bw2 = w; w += 3LL * NB * NB;
  q.G = w; w += NB * NB;
  q.Wp = w; w += 64LL * NB * n;
  q.W2 = w; w += (long long)NB * n;
  q.tau = w; w += n;
  q.dg = w;
  return q;
}

rfm_status qr_init_device() {
  const cudaError_t attr = rfm_smem_attr((const void*)k_block, KB_SMEM);  // once per device
  if (attr != cudaSuccess || rfm_num_sms() == 0) {
    rfm_set_error("householder: device set-up failed");
    return RFM_ECUDA;
  }
  return RFM_OK;
}

// CTAs of k_block that can be resident together with the largest slab (whole
// clusters; depends on how the device's SMs are grouped), per device; 0 on failure.
int kb_max_ctas() {
  static std::mutex mu;
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lk(mu);
  if (cached[dev] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(KB_CL);
    cfg.blockDim = dim3(KB_THREADS);
    cfg.dynamicSmemBytes = KB_SMEM;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_block, &cfg) != cudaSuccess) return 0;
    cached[dev] = std::min(n * KB_CL, KB_MAXP);
  }
  return cached[dev];
}

// Rows of k_block's slab for np 32-column groups.
long long kb_max_rows(int np) { return (long long)((KB_SMEM - kb_fixed_smem()) / (NB * np * sizeof(double))); }

// Widest block (32 .. 128 columns) that k_block can hold in shared memory for
// `rows` rows on all SMs.
int kb_width(long long rows) {
  const long long ctas = std::max(1, kb_max_ctas());
  const long long per = (rows + ctas - 1) / ctas;
  for (int np = 4; np > 1; --np)
    if (per <= kb_max_rows(np)) return np * NB;
  return NB;
}

// State of one factorisation's exchange: barrier arrivals so far.
struct KbState {
  unsigned int arrived = 0;
};

rfm_status kb_begin(const QrScratch& q, unsigned int* sync, cudaStream_t st) {
  // tags and barrier count of an earlier factorisation must not be mistaken for this one's
  RFM_CUDA(cudaMemsetAsync(q.xch, 0, 2LL * KB_SLOT * sizeof(unsigned long long), st));
  RFM_CUDA(cudaMemsetAsync(sync + SYNC_BAR, 0, sizeof(unsigned int), st));
  return RFM_OK;
}

// Factors columns [c0, c0 + nb) (rows c0..s) in place, nb <= kb_width.
rfm_status factor_block(double* A, long long s, long long lda, long long c0, int nb, cudaStream_t st,
                        const QrScratch& q, unsigned int* sync, int panel_cap, KbState* ks) {
  const long long rows = s - c0;
  const int np = (nb + NB - 1) / NB;
  const int ctas = kb_max_ctas();
  if (ctas < KB_CL) {
    rfm_set_error("householder: no cluster of the panel kernel fits on the device");
    return RFM_ECUDA;
  }
  // In 31 ns instructions a 32-column panel costs rows / (2 P) a column for its
  // products and updates, P / 16 for the sum over the clusters of P CTAs and,
  // with columns to the right in the block, rows / P a column for their update:
  // least at P^2 = 8 rows (one panel) or 24 rows (a block of four).
  const double opt = sqrt((np > 1 ? 24.0 : 8.0) * (double)rows);
  const long long cap = panel_cap > 0 ? std::min(panel_cap, ctas) : ctas;
  auto whole = [](long long v) { return std::max<long long>(KB_CL, v / KB_CL * KB_CL); };
  long long P = whole(std::min<long long>((long long)opt, cap));
  const long long most = kb_max_rows(np);
  if ((rows + P - 1) / P > most)  // a cap would overflow shared memory: take the fewest clusters that fit
    P = ((rows + most - 1) / most + KB_CL - 1) / KB_CL * KB_CL;
  const long long chunk = (rows + P - 1) / P;
  if (P > ctas || chunk > most) {
    rfm_set_error("householder: sketch too tall for the panel kernel");
    return RFM_EINVAL;
  }
  BlockArgs a;
  a.A = A; a.lda = lda; a.s = s; a.j0 = c0; a.nb = nb; a.P = (int)P; a.chunk = (int)chunk;
  a.xch = q.xch; a.part = q.part; a.w2 = q.bw2; a.tau = q.tau; a.G = q.G;
  a.bar = sync + SYNC_BAR; a.bar0 = ks->arrived; a.err = sync + SYNC_ERR;
  ks->arrived += 2u * (unsigned)(np - 1) * (unsigned)P;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // all CTAs co-resident: they wait on each other's records
  at[0].val.cooperative = 1;
  cfg.gridDim = dim3((unsigned)P);
  cfg.blockDim = dim3(KB_THREADS);
  cfg.dynamicSmemBytes = kb_fixed_smem() + (size_t)NB * np * chunk * sizeof(double);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  ProfScope ps(PF_QR_PANEL, st);
  RFM_CUDA(cudaLaunchKernelEx(&cfg, k_block, a));
  RFM_CHECK_LAUNCH();
  return RFM_OK;
}

// Householder factorisation of columns [c0, c1) (rows c0..s); the reflectors
// are applied in FP64 to the columns up to cend (cend >= c1).  Without columns
// past c1 the blocks are as wide as shared memory allows (k_block updates
// inside them); with them, 32 columns at a time.
rfm_status factor_range(double* A, long long s, long long lda, long long c0, long long c1, long long cend,
                        cudaStream_t st, const QrScratch& q, unsigned int* sync, int panel_cap, KbState* ks) {
  const int nsm = rfm_num_sms();
  if (cend == c1 && kb_width(s - c0) >= c1 - c0)
    return factor_block(A, s, lda, c0, (int)(c1 - c0), st, q, sync, panel_cap, ks);
  for (long long j0 = c0; j0 < c1; j0 += NB) {
    const int nbw = (int)std::min<long long>(NB, c1 - j0);
    const long long rows = s - j0;
    RFM_TRY(factor_block(A, s, lda, j0, nbw, st, q, sync, panel_cap, ks));
    const long long j1 = j0 + nbw;
    const long long nt = cend - j1;
    if (nt <= 0) continue;
    const long long ctiles = (nt + 63) / 64;
    // K slices of whole 32-row steps: the count that leaves the fewest steps on
    // the busiest SM (FP64 bound, so co-resident CTAs only share the unit)
    const long long steps = (rows + 31) / 32;
    long long nz = 1, best = -1;
    for (long long z = 1; z <= std::min<long long>(64, steps); ++z) {
      const long long per = (steps + z - 1) / z, zz = (steps + per - 1) / per;
      const long long cost = ((ctiles * zz + nsm - 1) / nsm) * per * 64 + zz;  // + k_wt's sum over slices
      if (best < 0 || cost < best) {
        best = cost;
        nz = zz;
      }
    }
    const long long kchunk = (steps + nz - 1) / nz * 32;
    nz = (rows + kchunk - 1) / kchunk;
    {
      ProfScope ps(PF_QR_VTA, st);
      rfm_prof_work(PF_QR_VTA, 2.0 * nbw * (double)nt * (double)rows);  // FP64 flops
      k_vta<<<dim3((unsigned)ctiles, (unsigned)nz), 256, 0, st>>>(A, lda, s, j0, nbw, j1, nt, kchunk, q.Wp);
      RFM_CHECK_LAUNCH();
      k_wt<<<(unsigned)((nt + 3) / 4), 128, 0, st>>>(q.Wp, (int)nz, q.G, q.tau + j0, nbw, nt, q.W2);
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
  KbState ks;
  RFM_TRY(kb_begin(q, sync, st));
  const long long c1 = ncols < 0 ? n : std::min<long long>(n, ((ncols + NB - 1) / NB) * NB);
  RFM_TRY(factor_range(A, s, lda, 0, c1, n, st, q, sync, panel_cap, &ks));
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
// size (15.1 MB of scratch + 16 KB of barrier words per GPU that loads the
// library, held until the process exits), sized for n <= 512 columns.
// Every call shares these arrays and they keep the last call's contents;
// calls that overlap on the GPU (two streams, or two host threads) race on
// them and must be serialised by the caller.
#define RFM_NOALLOC_MAX_N 512
#define RFM_NOALLOC_MAX_DEVICES 64

namespace {
constexpr long long kNoallocScratch = qr_scratch_len(RFM_NOALLOC_MAX_N);
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
// A block of w columns is factored recursively: its left half, the block
// reflector of that half applied to the right half, then the right half; blocks
// of kb_base columns go to k_block.  A factored block's reflectors V (rows x w,
// unit diagonal) update the columns to its right in compact-WY form
//     W = V^T A_t,  W2 = T^T W,  A_t -= V W2
// with all products on the emulated-FP64 tensor-core GEMM (digit splitting,
// exact level accumulation).  T (w x w) comes from the Gram V^T V, which the
// first product returns next to W, and the reflector coefficients,
// T_jj = tau_j, T_{:j,j} = -tau_j T_{:j,:j} G_{:j,j}.
//
// The trailing matrix is updated once per QB columns: its digits are formed and
// C is read and written once per pass, and the update's depth K = w is the MMA
// work of an output tile for one drain of its accumulators.  With w = 128 the
// update ran at 35 % of the tensor rate and the digits of the trailing matrix
// took 20 % of the time; w = 512 is one exact chunk of the GEMM, the largest
// depth that one drain covers.

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

constexpr int QB = 512;   // columns of an outer block (n >= 2 QB)
constexpr int QDIG = 8;

// T from G and tau: T^-1 = diag(1 / tau) + strict upper part of G, so column j
// of T is a back substitution, t_j = tau_j, t_i = -tau_i sum_{l>i} G_il t_l (no
// division; tau_i = 0 gives a zero row).  One warp per column, lane L holding
// rows L, L + 32, ..: the columns are independent, and a step is one shuffle
// and at most U FP64 instructions.  (Column after column on one CTA, whose
// FP64 unit had to do all of it, took 447 us for 128 columns; now 35 us.)
// G is column-major, T row-major, both w x w with w = 32 U.
template <int U>
__global__ void __launch_bounds__(128) k_block_t(const double* __restrict__ G, const double* __restrict__ tau,
                                                 double* __restrict__ T) {
  constexpr int w = 32 * U;
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * 4 + (threadIdx.x >> 5);
  double t[U], tu[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    t[u] = lane + 32 * u == j ? 1.0 : 0.0;  // e_j, then the right-hand side less the solved part
    tu[u] = tau[lane + 32 * u];
  }
#pragma unroll
  for (int h = U - 1; h >= 0; --h)  // row l = 32 h + ll is held in t[h]
    for (int l = min(j, 32 * h + 31); l >= 32 * h; --l) {
      double g[U];
#pragma unroll
      for (int u = 0; u <= h; ++u) g[u] = G[(size_t)l * w + lane + 32 * u];
      if (lane == (l & 31)) t[h] *= tu[h];
      const double y = __shfl_sync(0xffffffffu, t[h], l & 31);
#pragma unroll
      for (int u = 0; u <= h; ++u)
        if (u < h || lane < (l & 31)) t[u] = fma(-g[u], y, t[u]);
    }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = lane + 32 * u;
    T[(size_t)i * w + j] = i <= j ? t[u] : 0.0;
  }
}

// [G, W] (w x N, ld w) += E^T [V, A_t] + V'^T E [I, 0] of the block at c0: the
// rows c0 .. c0 + w of the trailing columns; in the Gram's upper part (all that
// T needs), V'^T E, entry (p, j) = v_p(j) for p < j.
__global__ void __launch_bounds__(64) k_add_top(const double* __restrict__ A, long long lda, long long c0, int w,
                                                long long N, double* __restrict__ C) {
  const int p = blockIdx.x * 64 + threadIdx.x;
  for (long long j = blockIdx.y; j < N; j += gridDim.y) {
    double add = 0.0;
    if (j >= w) add = A[(size_t)(c0 + j) * lda + c0 + p];
    else if (p < j) add = A[(size_t)(c0 + p) * lda + c0 + j];
    C[(size_t)j * w + p] += add;
  }
}

// Workspace of the block reflectors' application.
struct EmuWs {
  uint16_t *at, *t, *v, *w2;  // digits of [V, A_t], T^T, V, W2 (and of W before it)
  double *Wm, *W2, *T, *part;
  long long part_elems;
  int *e_at, *e_t, *e_v, *e_w2;
};

long long emu_part_elems(long long n) { return 16LL * 128 * (n + QB); }

rfm_status apply_block(double* A, long long s, long long lda, long long c0, int w, long long cend, cudaStream_t st,
                       const double* tau, const EmuWs& e, unsigned int* err) {
  const long long rows = s - c0, c1 = c0 + w, nt = cend - c1;
  {
    // One emulated product gives the block's Gram and V^T A_t.  V is sliced
    // without its unit diagonal, V = E + V': the digits of a row are scaled by
    // its largest entry, and beside the 1 the others (about 1 / sqrt(2 rows))
    // would keep 5 to 7 bits less.  The B operand is [V', A_t] (V'^T as the
    // first w / 64 row tiles, then the trailing columns), the A operand the
    // same V'^T tiles, and k_add_top adds E^T [V, A_t] and V'^T E in FP64.
    // (With the unit diagonal in the digits R of a 12,288 x 4,096 sketch was
    // four times as far from the exact one as the FP64 path's.)
    ProfScope ps(PF_QR_VTA, st);
    const long long prt = w / 64 + (nt + 63) / 64;  // row tiles of the B operand
    RFM_TRY(rfm_oz_slice_house_vt_at(A, lda, c0, w, rows, QDIG, 64, e.e_at, e.at, prt, 0, st));
    RFM_TRY(rfm_oz_slice_strided_at(A + (size_t)c1 * lda + c0, lda, 1, nt, rows, QDIG, 64, e.e_at + w, e.at, prt,
                                    w / 64, st));
    RFM_TRY(rfm_oz_gemm_part(e.at, QDIG, e.e_at, e.at, QDIG, e.e_at, w, w + nt, rows, QDIG + 1, e.Wm, w, 0, err, st,
                             e.part, e.part_elems, prt));
    k_add_top<<<dim3((unsigned)(w / 64), (unsigned)std::min<long long>(w + nt, 32768)), 64, 0, st>>>(
        A, lda, c0, w, w + nt, e.Wm);
    RFM_CHECK_LAUNCH();
    if (w == 64) k_block_t<2><<<w / 4, 128, 0, st>>>(e.Wm, tau + c0, e.T);
    else if (w == 128) k_block_t<4><<<w / 4, 128, 0, st>>>(e.Wm, tau + c0, e.T);
    else if (w == 256) k_block_t<8><<<w / 4, 128, 0, st>>>(e.Wm, tau + c0, e.T);
    else k_block_t<16><<<w / 4, 128, 0, st>>>(e.Wm, tau + c0, e.T);
    RFM_CHECK_LAUNCH();
    // W2 = T^T W on the emulated GEMM as well (M = K = w, N = nt).
    // T is stored row-major, T(q, p) = T[q w + p], so T^T(p, q) = T[p + q w].
    RFM_TRY(rfm_oz_slice_strided(e.T, 1, w, w, w, QDIG, 128, e.e_t, e.t, st));
    RFM_TRY(rfm_oz_slice_strided(e.Wm + (size_t)w * w, w, 1, nt, w, QDIG, 64, e.e_w2, e.w2, st));
    RFM_TRY(rfm_oz_gemm(e.t, QDIG, e.e_t, e.w2, QDIG, e.e_w2, w, nt, w, QDIG + 1, e.W2, w, 0, err, st));
  }
  ProfScope ps(PF_QR_UPDATE, st);
  RFM_TRY(rfm_oz_slice_house_v(A, lda, c0, rows, w, QDIG, e.e_v, e.v, st));
  RFM_TRY(rfm_oz_slice_strided(e.W2, w, 1, nt, w, QDIG, 64, e.e_w2, e.w2, st));
  return rfm_oz_gemm(e.v, QDIG, e.e_v, e.w2, QDIG, e.e_w2, rows, nt, w, QDIG + 1, A + (size_t)c1 * lda + c0, lda, 1,
                     err, st);
}

// Columns of one k_block: 128 while its slab holds them and the FP64 update
// inside the block (rows x 128 columns on the FP64 units) costs less than the
// dozen small launches of an emulated one, else 64.
int kb_base(long long rows) { return rows <= KB_WIDE_ROWS && kb_width(rows) >= 128 ? 128 : 64; }

rfm_status factor_recursive(double* A, long long s, long long lda, long long c0, int w, cudaStream_t st,
                            const QrScratch& q, const EmuWs& e, unsigned int* sync, int panel_cap, KbState* ks) {
  const int base = kb_base(s - c0);
  if (w <= base) return factor_range(A, s, lda, c0, c0 + w, c0 + w, st, q, sync, panel_cap, ks);
  int h = base;
  while (2 * h < w) h *= 2;
  RFM_TRY(factor_recursive(A, s, lda, c0, h, st, q, e, sync, panel_cap, ks));
  RFM_TRY(apply_block(A, s, lda, c0, h, c0 + w, st, q.tau, e, sync + SYNC_ERR));
  return factor_recursive(A, s, lda, c0 + h, w - h, st, q, e, sync, panel_cap, ks);
}

}  // namespace

long long rfm_householder_emulated_bytes(long long s, long long n) {
  long long b = 0;
  b += rfm_oz_digit_bytes(n + QB, s, QDIG, 64);  // [V, A_t]: the Gram and V^T A_t in one product
  b += rfm_oz_digit_bytes(QB, QB, QDIG, 128);    // T^T
  b += rfm_oz_digit_bytes(s, QB, QDIG, 128);     // V
  b += rfm_oz_digit_bytes(n, QB, QDIG, 64);      // W2
  b += 8LL * (2LL * QB * (n + QB) + QB * QB);    // [G, W], W2, T
  b += 8LL * emu_part_elems(n);                  // split-K partials of V^T [V, A_t]
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
  char* p = static_cast<char*>(emu);
  auto take = [&](long long bytes) {
    char* r = p;
    p += (bytes + 255) & ~255LL;
    return r;
  };
  EmuWs e;
  e.at = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(n + QB, s, QDIG, 64)));
  e.t = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(QB, QB, QDIG, 128)));
  e.v = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(s, QB, QDIG, 128)));
  e.w2 = reinterpret_cast<uint16_t*>(take(rfm_oz_digit_bytes(n, QB, QDIG, 64)));
  e.Wm = reinterpret_cast<double*>(take(8LL * QB * (n + QB)));  // [G, W] = V^T [V, A_t]
  e.W2 = reinterpret_cast<double*>(take(8LL * QB * n));
  e.T = reinterpret_cast<double*>(take(8LL * QB * QB));
  e.part_elems = emu_part_elems(n);
  e.part = reinterpret_cast<double*>(take(8LL * e.part_elems));
  e.e_at = reinterpret_cast<int*>(take(4LL * (n + QB)));
  e.e_t = reinterpret_cast<int*>(take(4LL * QB));
  e.e_v = reinterpret_cast<int*>(take(4LL * s));
  e.e_w2 = reinterpret_cast<int*>(take(4LL * n));
  KbState ks;
  RFM_TRY(kb_begin(q, sync, st));
  // Outer blocks of 512 columns; narrower ones where n holds only a few, and
  // for a timing probe of the first ncols columns.
  int wb = QB;
  while (wb > 128 && (wb * 2 > n || (ncols >= 0 && wb > ncols))) wb /= 2;
  const long long cstop = ncols < 0 ? n : std::min<long long>(n, ncols);
  for (long long J0 = 0; J0 < cstop; J0 += wb) {
    const int w = (int)std::min<long long>(wb, n - J0);
    RFM_TRY(factor_recursive(A, s, lda, J0, w, st, q, e, sync, panel_cap, &ks));
    if (J0 + w < n) RFM_TRY(apply_block(A, s, lda, J0, w, n, st, q.tau, e, sync + SYNC_ERR));
  }
  return finish_r(A, n, lda, st, q, sync, rank_flag_host);
}
