// Matrix-vector kernels of the LSQR inner solve on J R^{-1} (Alg. 1 steps 3-4).
//
//  * k_jmv:   y = s1 * J x + s2 * y.  One warp per four rows; a row is W
//             contiguous doubles of its primary block (and W more of the
//             secondary block for interface rows), read once, coalesced.
//  * k_jtmv:  y = J^T x.  One warp per (column block, 32-column chunk, eighth of
//             the block's rows); the rows are walked in a fixed order and the
//             eight partial sums are added in a fixed order (k_jtmv_sum), so the
//             result is deterministic.
//  * k_trsv_chain: x = R^{-1} b or x = R^{-T} b for the upper-triangular
//             preconditioner R (column-major, leading dimension ldr), in one
//             cooperative launch: a cluster of four CTAs solves the 64-row
//             blocks in dependency order, and helper CTAs stream the rest of R
//             once, each adding the contributions of published blocks to the
//             blocks it owns (details at the kernel).
//  * k_trsv:  the same solve for sizes with more blocks than the helpers can
//             own: 64-row blocks are claimed through a ticket counter in
//             dependency order, each block waits (bounded) on the per-block
//             flags of the blocks it needs, accumulates their contribution
//             with coalesced column reads of R, solves its diagonal block in
//             one warp and publishes its part of x with a release flag.
//  * k_partial_norm2, k_finish: deterministic two-stage norms.
#include <algorithm>
#include <mutex>
#include <string>

#include "rfm_internal.cuh"

namespace {

constexpr int TB = 64;  // triangular block

// Four rows per warp: an FP64 warp instruction takes 31 ns on GB300 whatever it
// does, so the reduction over the lanes (five additions a row) counts beside the
// W / 32 products; reducing four rows together takes six additions for all.
// FP64 bound: 124,416 rows of 512 take 110 us at two FMAs per clock and SM
// (one row per warp: 178 us, four: 147).
constexpr int JMV_ROWS = 4;

__global__ void __launch_bounds__(256) k_jmv(const double* __restrict__ Jp, const double* __restrict__ Js,
                                             const int4* __restrict__ meta, long long m, long long m_int, int W,
                                             const double* __restrict__ x, double s1, double s2,
                                             const double* __restrict__ s2dev, const int* __restrict__ skip,
                                             double* __restrict__ y) {
  if (skip && *skip) return;
  if (s2dev) s2 *= s2dev[0];
  const int lane = threadIdx.x & 31;
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long i0 = (blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5)) * JMV_ROWS; i0 < m;
       i0 += nwarps * JMV_ROWS) {
    const double *row[JMV_ROWS], *xb[JMV_ROWS];
    double acc[JMV_ROWS];
#pragma unroll
    for (int r = 0; r < JMV_ROWS; ++r) {
      const long long i = min(i0 + r, m - 1);
      row[r] = Jp + (size_t)i * W;
      xb[r] = x + (size_t)meta[i].y * W;
      acc[r] = 0.0;
    }
#pragma unroll 2
    for (int j = lane; j < W; j += 32) {
      double v[JMV_ROWS], xv[JMV_ROWS];
#pragma unroll
      for (int r = 0; r < JMV_ROWS; ++r) {
        v[r] = __ldcs(row[r] + j);
        xv[r] = xb[r][j];
      }
#pragma unroll
      for (int r = 0; r < JMV_ROWS; ++r) acc[r] += v[r] * xv[r];
    }
    if (i0 + JMV_ROWS > m_int) {
#pragma unroll
      for (int r = 0; r < JMV_ROWS; ++r) {
        const long long i = min(i0 + r, m - 1);
        const int4 mt = meta[i];
        if ((mt.x & 0xF) == 1) {
          const double* row2 = Js + (size_t)(i - m_int) * W;
          const double* xb2 = x + (size_t)mt.z * W;
          for (int j = lane; j < W; j += 32) acc[r] += row2[j] * xb2[j];
        }
      }
    }
    // lanes with bit 4 set keep rows 2, 3, bit 3 picks the odd row of the pair
    {
      const bool hi = lane & 16, odd = lane & 8;
      const double a0 = (hi ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, hi ? acc[0] : acc[2], 16);
      const double a1 = (hi ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, hi ? acc[1] : acc[3], 16);
      double a = (odd ? a1 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      const long long i = i0 + (hi ? 2 : 0) + (odd ? 1 : 0);
      if ((lane & 7) == 0 && i < m) y[i] = s2 == 0.0 ? s1 * a : __fma_rn(s1, a, __dmul_rn(s2, y[i]));
    }
  }
}

// Slice z of column block b: its rows z, z + JT_SLICES, z + 2 JT_SLICES, .., one
// chain of products per column (lane).  Which rows form a chain and the order of
// the sums over slices do not depend on how the work is spread, so the result
// keeps its bits, and the chains of a column may run on different SMs: with all
// eight in one CTA, 15,552 rows of 8 blocks of 128 were 16 CTAs and took 60 us
// (now 20; 124,416 rows of 64 blocks of 512: 148 -> 136 us, 110 of them FP64
// instructions).  A warp keeps 8 to 16 rows' loads in flight, the
// indices and factors of 32 rows a batch ahead.
__global__ void __launch_bounds__(128) k_jtmv(const double* __restrict__ Jp, const double* __restrict__ Js,
                                              const int* __restrict__ colptr, const int* __restrict__ colrows,
                                              long long m_int, int W, const double* __restrict__ x,
                                              const int* __restrict__ skip, double* __restrict__ part, long long n) {
  if (skip && *skip) return;
  const int b = blockIdx.x, lane = threadIdx.x & 31;
  const int c0 = (blockIdx.y * 4 + (threadIdx.x >> 5)) * 32;
  if (c0 >= W) return;
  const int col = min(c0 + lane, W - 1);
  const int beg = colptr[b] + blockIdx.z, end = colptr[b + 1];
  double acc = 0.0;
  // lane i holds the index and the factor of row t + JT_SLICES i of the batch at t
  // (row 0 with factor 0 past the last)
  auto entry = [&](int t) { return t + JT_SLICES * lane < end ? (unsigned int)colrows[t + JT_SLICES * lane] : 0u; };
  auto factor = [&](int t, unsigned int e) { return t + JT_SLICES * lane < end ? x[e & 0x7fffffffu] : 0.0; };
  double v[2][8];
  auto load = [&](double (&q)[8], unsigned int ent, int i0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const unsigned int e = __shfl_sync(0xffffffffu, ent, i0 + i);
      const long long r = e & 0x7fffffffu;
      q[i] = __ldcs(((e >> 31) ? Js + (size_t)(r - m_int) * W : Jp + (size_t)r * W) + col);
    }
  };
  unsigned int ent = entry(beg);
  double xr = factor(beg, ent);
  load(v[0], ent, 0);
  for (int t = beg; t < end; t += 32 * JT_SLICES) {
    const int cnt = min(32, (end - t + JT_SLICES - 1) / JT_SLICES), tn = t + 32 * JT_SLICES;
    const unsigned int nent = entry(tn);
    double nxr = 0.0;
#pragma unroll
    for (int i0 = 0; i0 < 32; i0 += 8) {  // the next eight rows' loads, then this eight's products
      if (i0 < 24) {
        if (cnt > i0 + 8) load(v[(i0 / 8 + 1) & 1], ent, i0 + 8);
      } else if (tn < end) {
        load(v[0], nent, 0);
      }
      if (i0 == 8) nxr = factor(tn, nent);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i0 + i < cnt) acc += v[(i0 / 8) & 1][i] * __shfl_sync(0xffffffffu, xr, i0 + i);
    }
    ent = nent;
    xr = nxr;
  }
  if (c0 + lane < W) part[(size_t)blockIdx.z * n + (size_t)b * W + col] = acc;
}

__global__ void k_jtmv_sum(const double* __restrict__ part, long long n, const int* __restrict__ skip,
                           double* __restrict__ y) {
  if (skip && *skip) return;
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
#pragma unroll
  for (int z = 0; z < JT_SLICES; ++z) s += part[(size_t)z * n + i];
  y[i] = s;
}

// x = R^{-1} b (TRANS = 0) or R^{-T} b (TRANS = 1).
template <int TRANS>
__global__ void __launch_bounds__(256) k_trsv(const double* __restrict__ R, long long ldr, int n,
                                              const double* __restrict__ rhs, double* __restrict__ x,
                                              unsigned int* __restrict__ flags, const unsigned int* __restrict__ epoch_dev,
                                              unsigned int* __restrict__ ticket, unsigned int* __restrict__ err,
                                              const int* __restrict__ skip) {
  if (skip && *skip) return;
  const unsigned int epoch = *epoch_dev;  // set by k_trsv_prep, which ran before this launch
  __shared__ double sdiag[TB][TB + 1];
  __shared__ double sacc[8][TB];
  __shared__ double srec[TB];
  __shared__ int sblk;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nblk = (n + TB - 1) / TB;
  if (tid == 0) {
    const unsigned int t = atomicAdd(ticket, 1u);
    sblk = TRANS == 0 ? nblk - 1 - (int)t : (int)t;
  }
  __syncthreads();
  const int k = sblk;
  const int r0 = k * TB;
  const int rows = min(TB, n - r0);
  // diagonal tile (column-major in R)
  for (int idx = tid; idx < TB * TB; idx += 256) {
    const int rr = idx % TB, cc = idx / TB;
    sdiag[rr][cc] = (rr < rows && cc < rows) ? R[(size_t)(r0 + cc) * ldr + r0 + rr] : 0.0;
  }
  // reciprocals of the block's pivots, taken in parallel before any wait so the
  // dependency chain below only multiplies
  if (tid < TB) srec[tid] = tid < rows ? 1.0 / R[(size_t)(r0 + tid) * ldr + r0 + tid] : 0.0;
  double a0 = 0.0, a1 = 0.0;          // TRANS 0: rows lane, lane+32 of the block
  double pc[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // TRANS 1: columns w + 8 t of the block, partial over lanes
  if (TRANS == 0) {
    for (int j = nblk - 1; j > k; --j) {
      if (tid == 0) wait_flag(flags + j, epoch, err);
      __syncthreads();
      const int c0 = j * TB, cols = min(TB, n - c0);
      for (int cc = w; cc < cols; cc += 8) {
        const double xc = __ldcg(x + c0 + cc);
        const double* col = R + (size_t)(c0 + cc) * ldr + r0;
        if (lane < rows) a0 += col[lane] * xc;
        if (lane + 32 < rows) a1 += col[lane + 32] * xc;
      }
    }
    sacc[w][lane] = a0;
    sacc[w][lane + 32] = a1;
  } else {
    for (int j = 0; j < k; ++j) {
      if (tid == 0) wait_flag(flags + j, epoch, err);
      __syncthreads();
      const int q0 = j * TB;  // full block: j < k < nblk
      const double z0 = __ldcg(x + q0 + lane), z1 = __ldcg(x + q0 + 32 + lane);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int cc = w + 8 * t;
        if (cc < rows) {
          const double* col = R + (size_t)(r0 + cc) * ldr + q0;
          pc[t] += col[lane] * z0 + col[lane + 32] * z1;
        }
      }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const double v = warp_sum(pc[t]);
      if (lane == 0) sacc[0][w + 8 * t] = v;
    }
  }
  __syncthreads();
  if (w == 0) {
    double acc[2];
    for (int h = 0; h < 2; ++h) {
      const int rr = lane + 32 * h;
      double s = 0.0;
      if (TRANS == 0) {
        for (int q = 0; q < 8; ++q) s += sacc[q][rr];
      } else {
        s = sacc[0][rr];
      }
      acc[h] = rr < rows ? rhs[r0 + rr] - s : 0.0;
    }
    // solve the diagonal block in registers: lane owns entries lane, lane+32
    double xv[2] = {0.0, 0.0};
    if (TRANS == 0) {
      for (int i = rows - 1; i >= 0; --i) {
        const int h = i >> 5, ln = i & 31;
        const double num = __shfl_sync(0xffffffffu, acc[h], ln);
        const double xi = num * srec[i];
        if (lane == ln) xv[h] = xi;
        if (lane < i) acc[0] -= sdiag[lane][i] * xi;
        if (lane + 32 < i) acc[1] -= sdiag[lane + 32][i] * xi;
      }
    } else {
      for (int i = 0; i < rows; ++i) {
        const int h = i >> 5, ln = i & 31;
        const double num = __shfl_sync(0xffffffffu, acc[h], ln);
        const double xi = num * srec[i];
        if (lane == ln) xv[h] = xi;
        if (lane > i) acc[0] -= sdiag[i][lane] * xi;
        if (lane + 32 > i) acc[1] -= sdiag[i][lane + 32] * xi;
      }
    }
    if (lane < rows) x[r0 + lane] = xv[0];
    if (lane + 32 < rows) x[r0 + lane + 32] = xv[1];
    __threadfence();
    __syncwarp();
    if (lane == 0) st_release(flags + k, epoch);
  }
}

// ---------------------------------------------------------------------------
// Triangular solve by a chain cluster and helper CTAs (cooperative launch, all
// CTAs co-resident).  The 64-row blocks are solved in dependency order t = 0,
// 1, ... (block k = nblk-1-t for R^{-1}, block t for R^{-T}).  With Z_k the
// inverse of the diagonal block (k_trsv_dinv, once per factorisation) and C_d
// the couplings of block k to the blocks solved d = 1 .. CHAIN_D steps before,
//     y_t = (b_k - s_t) - sum_d C_d x_{t-d},    x_t = Z_k y_t,
// where s_t, the contributions of all earlier blocks, comes from a helper: it
// owns the targets t = h + H m, adds each published block's part and publishes
// the sum after its last one.
//
// What bounds a step is again FP64 instruction issue (31 ns per warp instruction
// and SM partition) and the exchanges: the four CTAs take 16 rows each, a thread
// 8 columns of one row, so a product is 8 instructions per warp, the sum over
// columns one shuffle and four shared-memory partials, and y_t and x_t go to all
// four CTAs through distributed shared memory with one cluster barrier each (0.2
// us).  Which columns a thread takes and how the partials are added is fixed by
// chain_col, not by the split: a row's sum is eight chains of eight products in
// the order that one CTA solving the chain alone would take, so the solution's
// bits do not depend on the cluster.  Only C_1 and Z_k wait for the step before; their tiles and the others are
// read from a copy in the threads' order (k_trsv_pack), two steps ahead.  One
// chain CTA that did both products alone took 3.7 to 4.6 us per step, this takes
// 2.1 (n = 4,096: 239 / 295 -> 135 us for R^{-1} / R^{-T}); from n = 16,384 on the
// helpers' FP64 work bounds it (n = 32,768: 2.55 / 2.89 -> 1.84 / 1.78 ms, with
// n^2 / 2 products worth 0.93 ms).  CHAIN_D = 2 gives a helper two to three steps
// between a block's publication and the chain's need of its sum; 3 measured the
// same.  (Z_k C_d formed once,
// which would leave one exchange per step, lost digits where Z_k is
// ill-conditioned: LSQR on a cond(R) = 1e9 problem took 44 steps for 41.)
//
// Published values are records {low, tag, high, tag} (rec_publish) whose tag is
// the solve's epoch, polled directly; nothing is reset between solves.  All sums
// are in a fixed order, so results are deterministic.  Waits are bounded.
constexpr int CHAIN_CL = 4;            // CTAs of the chain cluster (16 rows each)
constexpr int CHAIN_D = 2;             // distances 1 .. CHAIN_D are the chain's
constexpr int HMAXT = 5;               // targets per helper CTA
constexpr int ZLD = TB + 1;            // leading dimension of a tile in shared memory

template <int TRANS>
__device__ __forceinline__ int chain_block(int t, int nblk) { return TRANS == 0 ? nblk - 1 - t : t; }

// Inverse of each 64 x 64 diagonal block of R, block k stored column-major at
// Z + k * 4096: Z[k][c * 64 + r] = (R_kk^{-1})(r, c).  Entries below the
// diagonal and, in a ragged last block, rows and columns past n are zero.
// Column c solves R_kk z = e_c by back substitution (one warp per column, rows
// on the lanes, IEEE division by each pivot); sixteen CTAs share a block's
// columns, as a step is some twelve FP64 instructions of 31 ns.
__global__ void __launch_bounds__(128) k_trsv_dinv(const double* __restrict__ R, long long ldr, int n,
                                                   double* __restrict__ Z) {
  __shared__ double D[TB * ZLD];
  const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int r0 = k * TB, rows = min(TB, n - r0);
  for (int idx = tid; idx < TB * TB; idx += blockDim.x) {
    const int r = idx & (TB - 1), c = idx >> 6;
    D[c * ZLD + r] = (r <= c && c < rows) ? R[(size_t)(r0 + c) * ldr + r0 + r] : 0.0;
  }
  __syncthreads();
  double* out = Z + (size_t)k * TB * TB;
  const int j = blockIdx.y + 16 * w;  // columns spread over CTAs and warps
  double acc0 = lane == j ? 1.0 : 0.0, acc1 = lane + 32 == j ? 1.0 : 0.0;
  double z0 = 0.0, z1 = 0.0;
  if (j < rows) {
    for (int i = j; i >= 0; --i) {
      const double zi = __shfl_sync(0xffffffffu, i < 32 ? acc0 : acc1, i & 31) / D[i * ZLD + i];
      if (i < 32 && lane == i) z0 = zi;
      if (i >= 32 && lane == i - 32) z1 = zi;
      if (lane < i) acc0 -= D[i * ZLD + lane] * zi;
      if (i > 32 && lane + 32 < i) acc1 -= D[i * ZLD + lane + 32] * zi;
    }
  }
  out[j * TB + lane] = z0;
  out[j * TB + lane + 32] = z1;
}

// Column of the i-th product in chain g (0 .. 7) of row r of tile d.  The chains'
// sums are added as ((0+1) + (2+3)) + ((4+5) + (6+7)):
//  d = 0 (the inverse, a triangle): a pair of rows r, 63 - r is 65 terms dealt to
//        eight chains in turn, row min(r, 63 - r) first; the entries outside the
//        triangle are zeros in the same chains
//  d = 1: columns of equal remainder modulo 8, the even remainders before the odd
//        ones for R^{-T}
//  d = 2: every fourth column of a half
__device__ __forceinline__ int chain_col(int dir, int d, int r, int g, int i) {
  if (d == 2) return 32 * (g >> 2) + (g & 3) + 4 * i;
  if (d == 1) return 8 * i + (dir == 0 ? g : (g < 4 ? 2 * g : 2 * g - 7));
  const int pos = (g >> 1) + 4 * (g & 1);  // term's position modulo 8
  const int first = dir == 0 ? (r < TB / 2 ? pos + r : pos - 1) : (r < TB / 2 ? pos : pos + r);
  return 8 * i + (first & 7);
}

// Tiles of the chain, P[dir][k][d]: d = 0 the inverse (dir 0 Z_k, dir 1 Z_k^T),
// d >= 1 the couplings (dir 0 R_{k,k+d}, dir 1 R_{k-d,k}^T); zero where the
// neighbour does not exist or past n.
__global__ void __launch_bounds__(256) k_trsv_pack(const double* __restrict__ R, long long ldr, int n, int nblk,
                                                   const double* __restrict__ Z, double* __restrict__ P) {
  __shared__ double t[TB * ZLD];
  const int k = blockIdx.x, d = blockIdx.y, dir = blockIdx.z, tid = threadIdx.x;
  const int j = dir == 0 ? k + d : k - d;  // column block (dir 0) or row block (dir 1) of the coupling
  double* out = P + (((size_t)dir * nblk + k) * (CHAIN_D + 1) + d) * TB * TB;
  for (int idx = tid; idx < TB * TB; idx += 256) {
    const int lo = idx & (TB - 1), hi = idx >> 6;  // row and column of the tile as stored
    double v = 0.0;
    if (d == 0) {
      v = Z[(size_t)k * TB * TB + idx];
    } else if (j >= 0 && j < nblk) {
      const int gr = (dir == 0 ? k : j) * TB + lo, gc = (dir == 0 ? j : k) * TB + hi;
      if (gr < n && gc < n) v = R[(size_t)gc * ldr + gr];
    }
    t[dir == 0 ? hi * ZLD + lo : lo * ZLD + hi] = v;  // t[c * ZLD + r]
  }
  __syncthreads();
  // in the order the chain's threads read it: rank, the thread's i-th product, warp, lane
  for (int idx = tid; idx < TB * TB; idx += 256) {
    const int lane = idx & 31, w = (idx >> 5) & 3, i = (idx >> 7) & 7, q = idx >> 10;
    const int r = q * 16 + (lane & 15), c = chain_col(dir, d, r, w * 2 + (lane >> 4), i);
    out[idx] = t[c * ZLD + r];
  }
}

struct ChainArgs {
  const double* R;
  const double* P;            // the chain's tiles of this direction (k_trsv_pack)
  long long ldr;
  int n, nblk, H;
  const double* rhs;
  double* x;
  unsigned long long* hrec;   // [nblk][64] records of the helpers' sums
  unsigned long long* xrec;   // [nblk][64] records of x
  unsigned int* epoch;        // solves so far; this one's tag is the next number
  unsigned int* err;
  const int* skip;
};

// The chain: ranks 0-3 of cluster 0.  Warps 0-3 take a step's critical path,
// C_1 x_{t-1} and Z_k y_t; warps 4-7 meanwhile form the rest of the next step's
// right-hand side (C_2, the helper's sum), one warp of each group per SM
// partition, so that this product fills the FP64 units while the critical warps
// wait for an exchange.  Two cluster barriers a step: B (y_t is spread) and A
// (x_t is spread and the next right-hand side is ready).
template <int TRANS>
__device__ __forceinline__ void trsv_chain(const ChainArgs& a, unsigned int tag, RecWait& wait, double* sm) {
  double* xs = sm;                 // [4][64] x of the last steps, all rows
  double* ys = xs + 4 * TB;        // [64] y, all rows
  double* part = ys + TB;          // [3][4][16] the warps' partial sums: y, x, next right-hand side
  double* hs = part + 3 * 4 * 16;  // [2][16] this rank's rows of b - s - C_2 x, steps alternating
  const int tid = threadIdx.x, lane = tid & 31, w = (tid >> 5) & 3;
  const bool crit = tid < 128;
  const int rank = blockIdx.x, nblk = a.nblk, n = a.n;
  const int row = rank * 16 + (lane & 15), chain = w * 2 + (lane >> 4);
  int c0[3];  // first columns of this thread's chains in the three tiles
#pragma unroll
  for (int d = 0; d < 3; ++d) c0[d] = chain_col(TRANS, d, row, chain, 0);
  // tile d of step t
  auto fetch = [&](double (&q)[8], int t, int d) {
    if (t >= nblk) return;
    const double* src = a.P + ((size_t)chain_block<TRANS>(t, nblk) * (CHAIN_D + 1) + d) * TB * TB +
                        (rank * 8 * 4 + w) * 32 + lane;
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = __ldg(src + i * 128);
  };
  auto dot8 = [&](const double (&q)[8], const double* v, int d) {
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc = fma(q[i], v[c0[d] + (d == 2 ? 4 : 8) * i], acc);
    return acc;
  };
  // this thread's part of a row summed over its warp's columns, then the warps'
  auto row_part = [&](double acc, double* p) {
    acc += __shfl_xor_sync(0xffffffffu, acc, 16);
    if (lane < 16) p[w * 16 + lane] = acc;
    __syncwarp();
    if (crit) asm volatile("bar.sync 1, 128;" ::: "memory");
    else asm volatile("bar.sync 2, 128;" ::: "memory");
  };
  auto row_sum = [&](const double* p) {
    const int r = lane & 15;
    return (p[r] + p[16 + r]) + (p[32 + r] + p[48 + r]);
  };
  // row r of this rank to every rank: lanes 0-15 write to ranks 0, 1, lanes 16-31 to ranks 2, 3
  auto spread = [&](double* v, double val) {
    double* dst = v + rank * 16 + (lane & 15);
    st_cluster(dst, (lane >> 4) * 2, val);
    st_cluster(dst, (lane >> 4) * 2 + 1, val);
  };
  double m[2][2][8];
  if (crit) {
    for (int i = tid; i < 4 * TB; i += 128) xs[i] = 0.0;
    fetch(m[0][0], 0, 0);
    fetch(m[0][1], 0, 1);
    fetch(m[1][0], 1, 0);
    fetch(m[1][1], 1, 1);
    cluster_arrive();
    auto step = [&](double (&q)[2][8], int t) {
      const int k = chain_block<TRANS>(t, nblk);
      cluster_wait();  // A: x_{t-1} and hs of this step
      row_part(dot8(q[1], xs + ((t - 1) & 3) * TB, 1), part);
      if (w == 0) spread(ys, hs[(t & 1) * 16 + (lane & 15)] - row_sum(part));
      cluster_arrive();
      cluster_wait();  // B: y_t
      row_part(dot8(q[0], ys, 0), part + 64);
      if (w == 0) {
        const double xv = row_sum(part + 64);
        spread(xs + (t & 3) * TB, xv);
        if (lane < 16) {
          const int gi = k * TB + rank * 16 + lane;
          rec_publish(a.xrec + (size_t)gi * 2, xv, tag);
          if (gi < n) a.x[gi] = xv;
        }
      }
      cluster_arrive();
      fetch(q[0], t + 2, 0);
      fetch(q[1], t + 2, 1);
    };
    for (int t = 0; t < nblk; t += 2) {
      step(m[0], t);
      if (t + 1 < nblk) step(m[1], t + 1);
    }
  } else {
    // b - s - C_2 x_{t-2} of step t into hs
    auto prepare = [&](double (&q)[8], int t) {
      const int gi = t < nblk ? chain_block<TRANS>(t, nblk) * TB + rank * 16 + lane : 0;
      const bool own = w == 0 && lane < 16 && t < nblk;
      const bool summed = own && t > CHAIN_D;
      const unsigned long long* rec = a.hrec + (size_t)gi * 2;
      unsigned long long lo = 0, hi = 0;
      if (summed) rec_load(rec, lo, hi);
      double v = own && gi < n ? a.rhs[gi] : 0.0;
      row_part(dot8(q, xs + ((t - 2) & 3) * TB, 2), part + 128);
      if (w == 0) {
        const double near = row_sum(part + 128);
        if (summed) {
          unsigned int spins = 0;
          while (!rec_ready(lo, hi, tag) && wait.spin(spins)) rec_load(rec, lo, hi);
          v -= rec_value(lo, hi);
        }
        if (own) hs[(t & 1) * 16 + lane] = v - near;
      }
      fetch(q, t + 2, 2);
    };
    if (w == 0 && lane < 16) {
      const int gi = chain_block<TRANS>(0, nblk) * TB + rank * 16 + lane;
      hs[lane] = gi < n ? a.rhs[gi] : 0.0;
    }
    fetch(m[1][0], 1, 2);
    fetch(m[0][0], 2, 2);
    cluster_arrive();
    auto step = [&](double (&q)[8], int t) {
      cluster_wait();    // A: x_{t-1}
      cluster_arrive();  // B needs nothing of these warps
      if (t + 1 < nblk) prepare(q, t + 1);
      cluster_wait();
      cluster_arrive();
    };
    for (int t = 0; t < nblk; t += 2) {
      step(m[1][0], t);
      if (t + 1 < nblk) step(m[0][0], t + 1);
    }
  }
  cluster_wait();  // no rank leaves before the last remote store has landed
}

// Helper h: its targets t = h + H m, m < NT.
template <int TRANS, int NT>
__device__ __forceinline__ void trsv_helper(const ChainArgs& a, unsigned int tag, RecWait& wait, double* sm) {
  double* xs = sm;                   // [2][64] x of the source block
  double* sred = xs + 2 * TB;        // [8][64]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nblk = a.nblk, n = a.n, h = blockIdx.x - CHAIN_CL;
  int tg[NT], nt = 0;
#pragma unroll
  for (int m = 0; m < NT; ++m) {
    const int t = h + a.H * m;
    tg[m] = t < nblk ? t : -1;
    if (t < nblk) nt = m + 1;
  }
  if (nt == 0) return;
  const int tmax = h + a.H * (nt - 1);
  double pa[NT][2];   // TRANS 0: partial sums of target rows lane, lane+32 over this warp's sources
  double ptp[NT][8];  // TRANS 1: partial sums of target rows w + 8 q over this lane's sources
#pragma unroll
  for (int m = 0; m < NT; ++m) {
    pa[m][0] = pa[m][1] = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) ptp[m][q] = 0.0;
  }
  // the sum of target m's partial sums, published
  auto finish = [&](int m, const double (&p2)[2], const double (&p8)[8]) {
    unsigned long long* out = a.hrec + (size_t)chain_block<TRANS>(tg[m], nblk) * TB * 2;
    if (TRANS == 0) {
      sred[w * TB + lane] = p2[0];
      sred[w * TB + lane + 32] = p2[1];
      __syncthreads();
      if (tid < TB) {
        double sum = sred[tid];
#pragma unroll
        for (int q = 1; q < 8; ++q) sum += sred[q * TB + tid];
        rec_publish(out + 2 * tid, sum, tag);
      }
      __syncthreads();  // sred is rewritten by the next target
    } else {
      // sum of p8[q] over the lanes, lane q (< 8) ends with entry q
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = p8[q];
#pragma unroll
      for (int o = 4; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < o; ++q) {
          const double send = up ? v[q] : v[q + o];
          const double keep = up ? v[q + o] : v[q];
          v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], 8);
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
      if (lane < 8) rec_publish(out + 2 * (w + 8 * lane), v[0], tag);
    }
  };
  // tile entries of (source u, target m): TRANS 0 rows lane, lane+32 of R(k, j),
  // columns w + 8 q; TRANS 1 rows w + 8 q of R(j, k) (columns of block k), read
  // along j's rows
  auto load_tile = [&](double (&tv)[16], int u, int t) {
    const bool live = t >= u + CHAIN_D + 1;
    const int j = chain_block<TRANS>(u, nblk), k = live ? chain_block<TRANS>(t, nblk) : 0;
    const int c0 = j * TB, r0 = k * TB;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int y = w + 8 * q;
      if (TRANS == 0) {  // R(r0 + lane (+32), c0 + y)
        const bool ok = live && c0 + y < n;
        const double* col = a.R + (size_t)(c0 + y) * a.ldr + r0;
        tv[2 * q] = ok && r0 + lane < n ? __ldg(col + lane) : 0.0;
        tv[2 * q + 1] = ok && r0 + lane + 32 < n ? __ldg(col + lane + 32) : 0.0;
      } else {           // R(c0 + lane (+32), r0 + y): target row y
        const bool ok = live && r0 + y < n;
        const double* col = a.R + (size_t)(r0 + y) * a.ldr + c0;
        tv[2 * q] = ok ? __ldg(col + lane) : 0.0;
        tv[2 * q + 1] = ok ? __ldg(col + lane + 32) : 0.0;
      }
    }
  };
  // x_u by records: threads 0-63 load theirs for the next source ahead
  unsigned long long xlo = 0, xhi = 0;
  auto load_x = [&](int u) {
    if (tid < TB && u < nblk) rec_load(a.xrec + ((size_t)chain_block<TRANS>(u, nblk) * TB + tid) * 2, xlo, xhi);
  };
  const int last = tmax - CHAIN_D - 1;  // last source of the last target
  double t[NT][16];
  auto source = [&](int u) {
    double* xb = xs + (u & 1) * TB;
    if (tid < TB) {
      unsigned int spins = 0;
      while (!rec_ready(xlo, xhi, tag) && wait.spin(spins)) load_x(u);
      xb[tid] = rec_value(xlo, xhi);
    }
    __syncthreads();
    load_x(u + 1);
    double xv[8], z0 = 0.0, z1 = 0.0;
    if (TRANS == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q) xv[q] = xb[w + 8 * q];
    } else {
      z0 = xb[lane];
      z1 = xb[lane + 32];
    }
    // the targets in the order they are due (the first live one may be due now)
#pragma unroll
    for (int m = 0; m < NT; ++m) {
      if (!(m < nt && tg[m] >= u + CHAIN_D + 1)) continue;
      if (TRANS == 0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          pa[m][0] += t[m][2 * q] * xv[q];
          pa[m][1] += t[m][2 * q + 1] * xv[q];
        }
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) ptp[m][q] = fma(t[m][2 * q + 1], z1, fma(t[m][2 * q], z0, ptp[m][q]));
      }
      if (tg[m] == u + CHAIN_D + 1) finish(m, pa[m], ptp[m]);
      else load_tile(t[m], u + 1, tg[m]);  // in flight during the other targets and the wait for x_{u+1}
    }
  };
  load_x(0);
#pragma unroll
  for (int m = 0; m < NT; ++m)
    if (m < nt) load_tile(t[m], 0, tg[m]);
  for (int u = 0; u <= last; ++u) source(u);
}

constexpr size_t chain_smem_bytes() { return (size_t)(2 * TB + 8 * TB) * sizeof(double); }

template <int TRANS, int NT>
__global__ void __cluster_dims__(CHAIN_CL, 1, 1) __launch_bounds__(256, 1) k_trsv_chain(ChainArgs a) {
  if (a.skip && *a.skip) return;
  if (!in_cluster(CHAIN_CL, a.err)) return;
  extern __shared__ __align__(16) double csm[];
  unsigned int tag = __ldcg(a.epoch) + 1u;
  if (tag == 0u) tag = 1u;  // 0 is the records' initial tag
  RecWait wait(a.err, threadIdx.x);
  if (blockIdx.x < CHAIN_CL) {
    trsv_chain<TRANS>(a, tag, wait, csm);
    // every helper whose records the chain used has read the epoch; the others use no
    // tag (after a wait that gave up, k_clear_err drops what a late one leaves)
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.epoch = tag;
  } else {
    trsv_helper<TRANS, NT>(a, tag, wait, csm);
  }
}

// Next epoch for the block flags (never 0, their initial value) and a fresh ticket
// counter; runs before every k_trsv so that replays of a captured graph see a new
// epoch each time.
__global__ void k_trsv_prep(unsigned int* __restrict__ epoch, unsigned int* __restrict__ ticket) {
  unsigned int e = *epoch + 1u;
  *epoch = e == 0u ? 1u : e;
  *ticket = 0u;
}

__global__ void k_partial_norm2(const double* __restrict__ x, long long n, double* __restrict__ partial) {
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    acc += x[i] * x[i];
  __shared__ double sh[32];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    v = warp_sum(v);
    if (threadIdx.x == 0) partial[blockIdx.x] = v;
  }
}

__global__ void k_finish(const double* __restrict__ partial, int np, double* __restrict__ out) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < np; i += 32) acc += partial[i];
  acc = warp_sum(acc);
  if (threadIdx.x == 0) out[0] = sqrt(acc);
}

constexpr int kRedBlocks = 304;

}  // namespace

rfm_status rfm_norm2(cudaStream_t st, const double* x, long long n, double* partial, double* out_dev) {
  k_partial_norm2<<<kRedBlocks, 256, 0, st>>>(x, n, partial);
  RFM_CHECK_LAUNCH();
  k_finish<<<1, 32, 0, st>>>(partial, kRedBlocks, out_dev);
  RFM_CHECK_LAUNCH();
  return RFM_OK;
}

rfm_status rfm_launch_jmv(rfm_problem* p, const double* x, double* y) {
  ProfScope ps(PF_JMV, p->stream);
  rfm_prof_work(PF_JMV, 8.0 * ((double)(p->m + p->m_iface) * p->W + p->m + p->n));
  long long g = (p->m + 8 * JMV_ROWS - 1) / (8 * JMV_ROWS);
  if (g > 152 * 64) g = 152 * 64;
  k_jmv<<<(int)g, 256, 0, p->stream>>>(p->Jp, p->Js, p->rmeta, p->m, p->m_int, p->W, x, 1.0, 0.0, nullptr, p->skip,
                                       y);
  RFM_CHECK_LAUNCH();
  return RFM_OK;
}

rfm_status rfm_launch_jmv_axpby(rfm_problem* p, const double* x, double s1, double s2, double* y,
                                const double* s2dev) {
  ProfScope ps(PF_JMV, p->stream);
  rfm_prof_work(PF_JMV, 8.0 * ((double)(p->m + p->m_iface) * p->W + 2.0 * p->m + p->n));
  long long g = (p->m + 8 * JMV_ROWS - 1) / (8 * JMV_ROWS);
  if (g > 152 * 64) g = 152 * 64;
  k_jmv<<<(int)g, 256, 0, p->stream>>>(p->Jp, p->Js, p->rmeta, p->m, p->m_int, p->W, x, s1, s2, s2dev, p->skip, y);
  RFM_CHECK_LAUNCH();
  return RFM_OK;
}

rfm_status rfm_launch_jtmv(rfm_problem* p, const double* x, double* y) {
  ProfScope ps(PF_JTMV, p->stream);
  rfm_prof_work(PF_JTMV, 8.0 * ((double)(p->m + p->m_iface) * p->W + p->m + p->n));
  k_jtmv<<<dim3(p->G, (p->W + 127) / 128, JT_SLICES), 128, 0, p->stream>>>(p->Jp, p->Js, p->colptr, p->colrows,
                                                                          p->m_int, p->W, x, p->skip, p->jt_part, p->n);
  RFM_CHECK_LAUNCH();
  k_jtmv_sum<<<(unsigned)((p->n + 255) / 256), 256, 0, p->stream>>>(p->jt_part, p->n, p->skip, y);
  RFM_CHECK_LAUNCH();
  return RFM_OK;
}

namespace {
using ChainKernel = void (*)(ChainArgs);
ChainKernel chain_kernel(int trans, int nt) {
  static const ChainKernel k[2][4] = {
      {k_trsv_chain<0, 1>, k_trsv_chain<0, 2>, k_trsv_chain<0, 4>, k_trsv_chain<0, HMAXT>},
      {k_trsv_chain<1, 1>, k_trsv_chain<1, 2>, k_trsv_chain<1, 4>, k_trsv_chain<1, HMAXT>}};
  return k[trans ? 1 : 0][nt == 1 ? 0 : nt == 2 ? 1 : nt <= 4 ? 2 : 3];
}

// CTAs of the chain kernels that are resident together (whole clusters), per
// device; 0 on failure.
int chain_max_ctas() {
  static std::mutex mu;
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lk(mu);
  if (cached[dev] == 0) {
    int least = 1 << 30;
    for (int trans = 0; trans < 2; ++trans)
      for (int nt : {1, 2, 4, HMAXT}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CHAIN_CL);
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = chain_smem_bytes();
        int c = 0;
        const ChainKernel fn = chain_kernel(trans, nt);
        if (rfm_smem_attr((const void*)fn, (int)chain_smem_bytes()) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&c, fn, &cfg) != cudaSuccess) {
          cudaGetLastError();  // the caller takes k_trsv; no later check may find this error
          return 0;
        }
        least = std::min(least, c * CHAIN_CL);
      }
    // one CTA per SM: two would share the FP64 units the chain depends on
    cached[dev] = std::min(least, rfm_num_sms() / CHAIN_CL * CHAIN_CL);
  }
  return cached[dev];
}
}  // namespace

// Helper CTAs of the chain for nblk blocks; 0 where k_trsv solves instead.  Chain
// and helpers up to four blocks per SM (n = 38,800), a rule on n alone so that the
// solution's bits are those of one form; the helpers, fewer than the SMs, take a
// fifth target at the end of that range.
static int chain_helpers(int nblk) {
  const int H = std::min(chain_max_ctas() - CHAIN_CL, (nblk + CHAIN_CL - 1) / CHAIN_CL * CHAIN_CL);
  return H > 0 && nblk <= HMAXT * H && nblk - CHAIN_D - 1 <= 4 * (rfm_num_sms() - 1) ? H : 0;
}

// Inverses and tiles of R for the chain; their buffer comes with the first R, like
// the sketch's and the QR's.
rfm_status rfm_trsv_prepare(rfm_problem* p) {
  const int n = (int)p->n, nblk = (n + TB - 1) / TB;
  if (!p->R || chain_helpers(nblk) == 0) return RFM_OK;
  if (!p->dinv) {
    const size_t inv = (size_t)nblk * TB * TB, tiles = 2 * inv * (CHAIN_D + 1);
    double* buf = nullptr;
    if (cudaMalloc(&buf, (inv + tiles) * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      rfm_set_error("triangular solve: allocation of " + std::to_string((inv + tiles) * sizeof(double)) + " bytes failed");
      return RFM_ENOMEM;
    }
    p->dinv = buf;
    p->chain_tiles = buf + inv;
  }
  k_trsv_dinv<<<dim3(nblk, 16), 128, 0, p->stream>>>(p->R, p->ldr, n, p->dinv);
  RFM_CHECK_LAUNCH();
  k_trsv_pack<<<dim3(nblk, CHAIN_D + 1, 2), 256, 0, p->stream>>>(p->R, p->ldr, n, nblk, p->dinv, p->chain_tiles);
  RFM_CHECK_LAUNCH();
  p->dinv_of = p->R;
  return RFM_OK;
}

rfm_status rfm_launch_trsv(rfm_problem* p, int trans, const double* b, double* x) {
  const int n = (int)p->n;
  const int nblk = (n + TB - 1) / TB;
  if (nblk > RFM_SYNC_WORDS - SYNC_FLAGS) {
    rfm_set_error("trsv: too many blocks");
    return RFM_EINVAL;
  }
  const int H = chain_helpers(nblk);
  if (H > 0 && p->dinv_of != p->R) RFM_TRY(rfm_trsv_prepare(p));
  ProfScope ps(PF_TRSV, p->stream);
  rfm_prof_work(PF_TRSV, 8.0 * (double)n * (n + 1) / 2 + 16.0 * n);  // R read once, b and x
  if (H > 0) {
    ChainArgs a;
    a.R = p->R; a.P = p->chain_tiles + (trans ? (size_t)nblk * (CHAIN_D + 1) * TB * TB : 0);
    a.ldr = p->ldr; a.n = n; a.nblk = nblk; a.H = H; a.rhs = b; a.x = x;
    a.hrec = p->trsv_rec; a.xrec = p->trsv_rec + (size_t)nblk * TB * 2;
    a.epoch = p->sync + SYNC_EPOCH; a.err = p->sync + SYNC_ERR; a.skip = p->skip;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(CHAIN_CL + H));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = chain_smem_bytes();
    cfg.stream = p->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;  // all CTAs co-resident: helpers and the chain wait on each other
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    RFM_CUDA(cudaLaunchKernelEx(&cfg, chain_kernel(trans, (nblk + H - 1) / H), a));
    RFM_CHECK_LAUNCH();
    return RFM_OK;
  }
  k_trsv_prep<<<1, 1, 0, p->stream>>>(p->sync + SYNC_EPOCH, p->sync + SYNC_TICKET);
  RFM_CHECK_LAUNCH();
  if (trans == 0)
    k_trsv<0><<<nblk, 256, 0, p->stream>>>(p->R, p->ldr, n, b, x, p->sync + SYNC_FLAGS, p->sync + SYNC_EPOCH,
                                           p->sync + SYNC_TICKET, p->sync + SYNC_ERR, p->skip);
  else
    k_trsv<1><<<nblk, 256, 0, p->stream>>>(p->R, p->ldr, n, b, x, p->sync + SYNC_FLAGS, p->sync + SYNC_EPOCH,
                                           p->sync + SYNC_TICKET, p->sync + SYNC_ERR, p->skip);
  RFM_CHECK_LAUNCH();
  return RFM_OK;
}
