// k_inverse.cu -- FP64 in-place Gauss-Jordan inverse, one thread-block
// cluster per matrix (the from-scratch N of the initial build and of the
// periodic recompute, Eq. Zk: N = [e^V - g0 (e^V - 1)]^-1).
//
// A cluster of C blocks (16 for up to 6 matrices, else 8) shares one n x n
// matrix in global memory; row r belongs to block r % C.  The columns are taken
// in panels of B.  With J the rows of a panel after its row interchanges,
//   A_JJ <- A_JJ^-1,  A_Jk <- A_JJ^-1 A_Jk,  A_iJ <- -A_iJ A_JJ^-1,
//   A_ik <- A_ik - A_iJ A_JJ^-1 A_Jk,
// so the panel itself carries all factors: with P the panel after its own
// Gauss-Jordan steps and X the rows J of the other columns before, every row
// becomes A_ik = [i not in J] A_ik + sum_j P_ij X_jk.
//   1. The panel's rows sit in the shared memory of their blocks.  Per column
//      every block posts its largest |A[r][c]|, r >= c, with that panel row, and
//      the owner of row c posts row c; one cluster barrier; every block reads
//      the posts through distributed shared memory, takes the same pivot,
//      interchanges and eliminates in its own rows.
//   2. The interchanges are applied to the other columns (a slice per block, all
//      loads before the stores) and the rows J of them written to the scratch
//      X; cluster barrier.
//   3. Every block updates its own rows, X passing through shared memory.
// The row interchanges are undone at the end as one permutation of the
// columns.  The sign of det A comes from the pivots.
//
// Bound by FP64 issue (a warp-wide FP64 instruction holds its SM sub-partition's
// unit for 64 cycles): n^3 multiply-adds on 2 C per cycle.  A rank-1 pass over
// the matrix per column instead made it wait on L2 and on two cluster barriers
// a column: two matrices of order 500 (dca_fresh_N) 12.8 -> 4.33 ms a call on two
// clusters, and 3.21 with the updates on the whole device (below).
#include <cooperative_groups.h>

#include <cstdint>
#include <mutex>

#include "device_util.cuh"
#include "kernels.h"
#include "state.h"

namespace cg = cooperative_groups;

namespace dca {

namespace {

constexpr int GJ_THREADS = 1024;
constexpr int GJ_MAX_CTAS = 16;
constexpr int GJ_WIDE_MATS = 6;        // most matrices for clusters of 16
constexpr int GJ_XC = 256;             // columns of X in shared memory at a time
constexpr size_t GJ_SMEM = 208 * 1024;  // dynamic shared memory of a block, at most

template <int B>
struct GjPost {
  unsigned long long mag;  // bits of the largest |A[r][c]| of the block's rows r >= c, 0 if there is none
  int idx, pad;
  double row[B];           // that row of the panel
};

// Larger magnitude first, then the lower row.
__device__ __forceinline__ bool gj_better(unsigned long long m1, int i1, unsigned long long m2, int i2) {
  return m1 > m2 || (m1 == m2 && i1 < i2);
}

__device__ __forceinline__ bool gj_wants(const Config& cfg, int mode, int mat) {
  const WalkerDev& w = cfg.W[mat >> 1];
  if (mode == 0) return true;
  if (mode == 2) return w.rebuild_pending && w.status == ST_OK;
  return w.active && w.recompute_pending && w.status == ST_OK;
}

__host__ __device__ __forceinline__ int gj_rows(int n, int ctas) { return (n + ctas - 1) / ctas; }

__host__ __device__ __forceinline__ size_t gj_rp_bytes(int max_n, int B) {
  return B == 16 ? (sizeof(int) * (size_t)max_n + 15) & ~(size_t)15 : 0;
}

// Bytes of the panel rows and of X (the row buffers of the last step share them).
__host__ __device__ __forceinline__ size_t gj_work_bytes(int rows, int B) {
  return sizeof(double) * ((size_t)rows * (B + 1) + (size_t)B * GJ_XC);
}

// The whole inverse of one matrix (ONE = false), or (ONE) steps 1 and 2 of the
// panel at `first`: the panel factors then go to the scratch at 16 n for
// k_gj_update, the permutation is kept at 32 n for k_gj_finish.
template <int B, bool ONE>
__device__ void gj_matrix(const Config& cfg, int mode, int mat, int* sgn_out, cg::cluster_group& cluster, int max_n,
                          size_t work_bytes, int first = 0) {
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int wi = mat >> 1, sp = mat & 1;
  WalkerDev& w = cfg.W[wi];
  const int n = w.n, ld = w.cap;
  double* A = (cfg.prec == PREC_MIXED) ? w.Ascr[sp] : (double*)w.N[mode == 1 ? w.parity ^ 1 : w.parity][sp];
  double* X = w.gjX[sp];  // scratch [16][n]: rows J of the other columns; row buffers of the last step
  extern __shared__ __align__(16) unsigned char gj_smem[];
  // rp [n]: original row now at each position; in shared memory with panels of
  // 16, else one copy per block behind the first 8 rows of the scratch
  int* rp = ONE ? reinterpret_cast<int*>(X + 32 * (size_t)n)
                : (B == 16 ? reinterpret_cast<int*>(gj_smem)
                           : reinterpret_cast<int*>(X + 8 * (size_t)n) + (size_t)rank * n);
  double* pan = reinterpret_cast<double*>(gj_smem + (ONE ? 0 : gj_rp_bytes(max_n, B)));
  const int rows = n > rank ? (n - rank + C - 1) / C : 0;  // own rows rank, rank + C, ...
  double* xs = pan + (size_t)gj_rows(max_n, C) * (B + 1);
  constexpr int PS = B + 1;
  __shared__ GjPost<B> s_post[2];
  __shared__ double s_rowc[2][B];
  __shared__ double s_prow[B], s_old[B];
  __shared__ unsigned long long s_wmag[GJ_THREADS / 32];
  __shared__ int s_widx[GJ_THREADS / 32];
  __shared__ int s_piv[B], s_dst[2 * B], s_src[2 * B], s_p, s_bad, s_own;
  __shared__ double s_d;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr unsigned FULL = 0xffffffffu;
  int sign = 1;
  bool bad = false;
  if (ONE && first > 0 && sgn_out[mat] == 0) return;  // an earlier panel was singular (read before any barrier)
  if (!ONE || (first == 0 && rank == 0))
    for (int i = tid; i < n; i += GJ_THREADS) rp[i] = i;

  for (int c0 = first; c0 < n && !bad; c0 += B) {
    const int b = min(B, n - c0);
    __syncthreads();  // the own rows are up to date, the shared panel and X are free
    for (int e = tid; e < rows * B; e += GJ_THREADS) {
      const int r = e / B, j = e - r * B;
      pan[r * PS + j] = j < b ? A[(size_t)(rank + r * C) * ld + c0 + j] : 0.0;
    }
    __syncthreads();
    for (int s = 0; s < b; ++s) {
      const int c = c0 + s, par = s & 1;
      // pivot candidate of the own rows (NaN never wins)
      unsigned long long bm = 0ull;
      int bi = 0x7fffffff;
      for (int r = tid; r < rows; r += GJ_THREADS) {
        const int i = rank + r * C;
        const unsigned long long m = (unsigned long long)__double_as_longlong(pan[r * PS + s]) & 0x7fffffffffffffffull;
        if (i >= c && m <= 0x7ff0000000000000ull && gj_better(m, i, bm, bi)) {
          bm = m;
          bi = i;
        }
      }
      const int nw = min(GJ_THREADS / 32, (rows + 31) >> 5);  // warps that hold a candidate
      if (warp < nw) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const unsigned long long om = __shfl_xor_sync(FULL, bm, o);
          const int oi = __shfl_xor_sync(FULL, bi, o);
          if (gj_better(om, oi, bm, bi)) {
            bm = om;
            bi = oi;
          }
        }
        if (nw > 1 && lane == 0) {
          s_wmag[warp] = bm;
          s_widx[warp] = bi;
        }
      }
      if (nw > 1) __syncthreads();
      if (warp == 0) {
        if (nw > 1) {
          bm = lane < nw ? s_wmag[lane] : 0ull;
          bi = lane < nw ? s_widx[lane] : 0x7fffffff;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long om = __shfl_xor_sync(FULL, bm, o);
            const int oi = __shfl_xor_sync(FULL, bi, o);
            if (gj_better(om, oi, bm, bi)) {
              bm = om;
              bi = oi;
            }
          }
        }
        GjPost<B>& post = s_post[par];
        if (lane == 0) {
          post.mag = bi < n ? bm : 0ull;
          post.idx = bi;
        }
        if (lane < B && bi < n) post.row[lane] = pan[((bi - rank) / C) * PS + lane];
        if (lane < B && c % C == rank) s_rowc[par][lane] = pan[(c / C) * PS + lane];
      }
      cluster.sync();
      // every block takes the same pivot from all posts
      if (warp == 0) {
        unsigned long long m = 0ull;
        int idx = 0x7fffffff, own = lane;
        if (lane < C) {
          const GjPost<B>* q = cluster.map_shared_rank(&s_post[par], lane);
          m = q->mag;
          idx = m ? q->idx : 0x7fffffff;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const unsigned long long om = __shfl_xor_sync(FULL, m, o);
          const int oi = __shfl_xor_sync(FULL, idx, o), oo = __shfl_xor_sync(FULL, own, o);
          if (gj_better(om, oi, m, idx)) {
            m = om;
            idx = oi;
            own = oo;
          }
        }
        if (m > 0ull) {
          const GjPost<B>* q = cluster.map_shared_rank(&s_post[par], own);
          const double* rc = cluster.map_shared_rank(&s_rowc[par][0], c % C);
          const double pr = lane < B ? q->row[lane] : 0.0;
          const double d = __shfl_sync(FULL, pr, s), rd = 1.0 / d;
          if (lane < B) {
            s_prow[lane] = lane == s ? rd : pr * rd;
            s_old[lane] = rc[lane];
          }
          if (lane == 0) {
            s_d = d;
            s_p = idx;
            s_piv[s] = idx;
            if (!ONE || rank == 0) {
              const int t = rp[c];
              rp[c] = rp[idx];
              rp[idx] = t;
            }
          }
        }
        if (lane == 0) s_bad = m > 0ull ? 0 : 1;
      }
      __syncthreads();
      if (s_bad) {
        bad = true;  // every block reaches the same decision
        break;
      }
      const int p = s_p;
      if (p != c) sign = -sign;
      if (s_d < 0.0) sign = -sign;
      // interchange and eliminate in the own rows; the B entries of a row are in one warp
      for (int e0 = 0; e0 < rows * B; e0 += GJ_THREADS) {
        const int e = e0 + tid, r = e / B, j = e - r * B, i = rank + r * C;
        const bool in = e < rows * B;
        double v = 0.0, f = 0.0;
        if (in) {
          v = i == p ? s_old[j] : pan[r * PS + j];
          f = i == p ? s_old[s] : pan[r * PS + s];
        }
        __syncwarp();
        if (in) pan[r * PS + j] = i == c ? s_prow[j] : (j == s ? -f * s_prow[j] : fma(-f, s_prow[j], v));
      }
      __syncthreads();
    }
    if (bad) break;
    // the net interchange of rows: lanes 0 .. B - 1 hold the rows of J, the next
    // ones the distinct pivot rows outside it; each lane its position's source
    if (warp == 0) {
      int pos = lane < b ? c0 + lane : -1, src = pos, cnt = b;
      for (int s = 0; s < b; ++s) {
        const int p = s_piv[s];
        unsigned at = __ballot_sync(FULL, pos == p);
        if (!at) {
          if (lane == cnt) pos = src = p;
          at = 1u << cnt;
          ++cnt;
        }
        const int q = __ffs(at) - 1;
        const int x = __shfl_sync(FULL, src, s), y = __shfl_sync(FULL, src, q);
        if (lane == s) src = y;
        else if (lane == q) src = x;
      }
      if (lane < cnt) {
        s_dst[lane] = pos;
        s_src[lane] = src;
      }
      if (lane == 0) s_own = cnt;
    }
    __syncthreads();
    // slice of the other columns: 32 columns x (up to 32 rows), loads before stores
    const int cnt = s_own;
    const int k0 = (int)(((long long)n * rank) / C), k1 = (int)(((long long)n * (rank + 1)) / C);
    for (int kb = k0; kb < k1; kb += 32) {
      const int k = kb + lane;
      const bool in = warp < cnt && k < k1 && (k < c0 || k >= c0 + b);
      double v = 0.0;
      if (in) v = A[(size_t)s_src[warp] * ld + k];
      __syncthreads();
      if (in) {
        if (warp < b) X[(size_t)warp * n + k] = v;
        else A[(size_t)s_dst[warp] * ld + k] = v;
      }
    }
    if constexpr (ONE) {
      double* P = X + 16 * (size_t)n;
      for (int e = tid; e < rows * B; e += GJ_THREADS) {
        const int r = e / B, j = e - r * B;
        P[(size_t)(rank + r * C) * B + j] = pan[r * PS + j];
      }
    }
    cluster.sync();
    if constexpr (ONE) {
      if (rank == 0 && tid == 0) sgn_out[mat] = first == 0 ? sign : sign * sgn_out[mat];
      return;
    }
    // update of the own rows
    for (int kb = 0; kb < n; kb += GJ_XC) {
      const int m = min(GJ_XC, n - kb);
      __syncthreads();
      for (int e = tid; e < B * GJ_XC; e += GJ_THREADS) {
        const int j = e / GJ_XC, k = e - j * GJ_XC, col = kb + k;
        xs[e] = (j < b && k < m && (col < c0 || col >= c0 + b)) ? X[(size_t)j * n + col] : 0.0;
      }
      __syncthreads();
      // a warp's item: one row, 64 columns (two per lane)
      const int segs = (m + 63) >> 6;
      for (int it = warp; it < rows * segs; it += GJ_THREADS / 32) {
        const int r = it / segs, k = (it - r * segs) * 64 + lane, i = rank + r * C;
        double* Ar = A + (size_t)i * ld + kb;
        const bool inJ = i >= c0 && i < c0 + b;
        double a0 = 0.0, a1 = 0.0;
        if (!inJ) {
          if (k < m) a0 = Ar[k];
          if (k + 32 < m) a1 = Ar[k + 32];
        }
#pragma unroll
        for (int j = 0; j < B; ++j) {
          const double f = pan[r * PS + j];
          a0 = fma(f, xs[j * GJ_XC + k], a0);
          a1 = fma(f, xs[j * GJ_XC + k + 32], a1);
        }
        const int col = kb + k;
        if (k < m) Ar[k] = (col >= c0 && col < c0 + b) ? pan[r * PS + col - c0] : a0;
        if (k + 32 < m) Ar[k + 32] = (col + 32 >= c0 && col + 32 < c0 + b) ? pan[r * PS + col + 32 - c0] : a1;
      }
    }
  }
  if (bad) {
    cluster.sync();  // no block leaves while another may still read its posts
    if (rank == 0 && tid == 0) {
      set_status(w, ST_ERR_NUMERIC);
      sgn_out[mat] = 0;
    }
    return;
  }
  // undo the interchanges: column rp[k] of the inverse is the working column k;
  // rows pass through shared memory (or the block's row of the scratch), every
  // block being past its reads of X
  cluster.sync();
  const int fit = (int)(work_bytes / (sizeof(double) * (size_t)(n > 0 ? n : 1)));
  double* buf = fit > 0 ? pan : X + (size_t)rank * n;
  const int batch = fit > 0 ? fit : 1;
  for (int r0 = 0; r0 < rows; r0 += batch) {
    const int m = min(batch, rows - r0);
    __syncthreads();
    for (int r = 0; r < m; ++r) {
      const double* Ar = A + (size_t)(rank + (r0 + r) * C) * ld;
      for (int k = tid; k < n; k += GJ_THREADS) buf[(size_t)r * n + k] = Ar[k];
    }
    __syncthreads();
    for (int r = 0; r < m; ++r) {
      double* Ar = A + (size_t)(rank + (r0 + r) * C) * ld;
      for (int k = tid; k < n; k += GJ_THREADS) Ar[rp[k]] = buf[(size_t)r * n + k];
    }
  }
  if (rank == 0 && tid == 0) sgn_out[mat] = sign;
}

// mode 0: initial build / standalone; mode 1: periodic recompute (into the
// other buffer); mode 2: rebuild after a change of the bare propagator.
// Persistent grid of clusters fed by a work queue: the rank-0 block of a
// cluster takes the next matrix (walker * 2 + spin) from cfg.gj_next (reset to
// 0 by k_build_A before every launch), so clusters that drew small matrices
// take more of them.
template <int B>
__global__ void __launch_bounds__(GJ_THREADS) k_gj_cluster(Config cfg, int mode, int max_n, size_t work_bytes,
                                                           int* sgn_out) {
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ int s_next;
  // Nothing to do in most windows: every block sees the same records, so the
  // decision is uniform over the cluster.
  __shared__ int s_any;
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  for (int m = threadIdx.x; m < 2 * cfg.n_walkers && !s_any; m += blockDim.x)
    if (gj_wants(cfg, mode, m)) s_any = 1;
  __syncthreads();
  if (!s_any) return;
  const int rank = (int)cluster.block_rank();
  for (;;) {
    if (rank == 0 && threadIdx.x == 0) s_next = atomicAdd(cfg.gj_next, 1);
    cluster.sync();
    const int mat = *cluster.map_shared_rank(&s_next, 0);
    cluster.sync();  // every block has read s_next before it changes
    if (mat >= 2 * cfg.n_walkers) break;
    if (!gj_wants(cfg, mode, mat)) continue;
    gj_matrix<B, false>(cfg, mode, mat, sgn_out, cluster, max_n, work_bytes);
    cluster.sync();  // the next matrix reuses the shared posts and pivots
  }
}

// One matrix over the whole device, a kernel pair per panel (n known to the
// host): the panel's factors on one cluster, then the update of everything else
// by all SMs.  With the update on the cluster's 16 SMs as well, n^3 multiply-adds
// on 32 a cycle took half the time: dca_fresh_N of order 500 4.33 -> 3.21 ms.  At
// order 256 the two launches a panel still cost what the update saves (1.59 ms
// against 1.52 on the cluster), hence GW_MIN.  The panel stays on 16 blocks: with 8
// a call of order 500 takes 3.41 ms, with 4 3.72.
constexpr int GW_B = 16, GW_R = 8, GW_C = 64;  // panel; rows and columns of an update item
constexpr int GW_MIN = 320, GW_MAX = 4096;     // orders that take this path

__global__ void __launch_bounds__(GJ_THREADS) k_gj_panel(Config cfg, int first, int max_n, int* sgn_out) {
  cg::cluster_group cluster = cg::this_cluster();
  const int mat = blockIdx.x / (int)cluster.num_blocks();
  gj_matrix<GW_B, true>(cfg, 0, mat, sgn_out, cluster, max_n, 0, first);
}

__global__ void __launch_bounds__(256) k_gj_update(Config cfg, int c0, const int* sgn) {
  __shared__ double xs[GW_B][GW_C], ps[GW_R][GW_B];
  const int tid = threadIdx.x, k = tid & (GW_C - 1), rg = tid / GW_C;
  for_each_item(
      2 * cfg.n_walkers,
      [&](int s) -> long long {
        const int n = cfg.W[s >> 1].n;
        return c0 < n && sgn[s] != 0 ? blocks_of(n, GW_R) * blocks_of(n, GW_C) : 0;
      },
      [&](int s, int item) {
        const WalkerDev& w = cfg.W[s >> 1];
        const int sp = s & 1, n = w.n, ld = w.cap, b = min(GW_B, n - c0), cblocks = (n + GW_C - 1) / GW_C;
        const int i0 = (item / cblocks) * GW_R, k0 = (item % cblocks) * GW_C, col = k0 + k;
        double* A = cfg.prec == PREC_MIXED ? w.Ascr[sp] : (double*)w.N[w.parity][sp];
        const double* X = w.gjX[sp];
        const double* P = X + 16 * (size_t)n;
        __syncthreads();  // the previous item is done with the shared tiles
        for (int e = tid; e < GW_B * GW_C; e += 256) {
          const int j = e / GW_C, c = k0 + (e - j * GW_C);
          xs[j][e - j * GW_C] = (j < b && c < n && (c < c0 || c >= c0 + b)) ? X[(size_t)j * n + c] : 0.0;
        }
        if (tid < GW_R * GW_B) ps[tid / GW_B][tid % GW_B] = i0 + tid / GW_B < n ? P[(size_t)i0 * GW_B + tid] : 0.0;
        __syncthreads();
        if (col >= n) return;
        const bool in_panel = col >= c0 && col < c0 + b;
#pragma unroll
        for (int u = 0; u < GW_R / 4; ++u) {
          const int r = rg + 4 * u, i = i0 + r;
          if (i >= n) break;
          double* a = A + (size_t)i * ld + col;
          double v = (i >= c0 && i < c0 + b) ? 0.0 : *a;
#pragma unroll
          for (int j = 0; j < GW_B; ++j) v = fma(ps[r][j], xs[j][k], v);
          *a = in_panel ? ps[r][col - c0] : v;
        }
      });
}

// The interchanges undone: column rp[k] of the inverse is the working column k;
// one block per row.
__global__ void __launch_bounds__(256) k_gj_finish(Config cfg, const int* sgn) {
  extern __shared__ double row[];
  const int mat = blockIdx.y, sp = mat & 1, i = blockIdx.x;
  const WalkerDev& w = cfg.W[mat >> 1];
  if (i >= w.n || sgn[mat] == 0) return;
  const int* rp = reinterpret_cast<const int*>(w.gjX[sp] + 32 * (size_t)w.n);
  double* A = (cfg.prec == PREC_MIXED ? w.Ascr[sp] : (double*)w.N[w.parity][sp]) + (size_t)i * w.cap;
  for (int k = threadIdx.x; k < w.n; k += blockDim.x) row[k] = A[k];
  __syncthreads();
  for (int k = threadIdx.x; k < w.n; k += blockDim.x) A[rp[k]] = row[k];
}

template <int B>
cudaError_t gj_launch(const Config& cfg, int mode, int max_n, int ctas, int clusters, int* d_sgn, cudaStream_t st) {
  const size_t rp = gj_rp_bytes(max_n, B);
  size_t work = gj_work_bytes(gj_rows(max_n, ctas), B);
  // room for a batch of whole rows in the last step, up to 96 KB
  const size_t want = sizeof(double) * (size_t)max_n * 32 < 96 * 1024 ? sizeof(double) * (size_t)max_n * 32 : 96 * 1024;
  if (work < want) work = want;
  const size_t smem = rp + work;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(ctas * clusters);
  lc.blockDim = dim3(GJ_THREADS);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, k_gj_cluster<B>, cfg, mode, max_n, work, d_sgn);
}

// Kernel attributes (once per device) and the clusters of 16 that the device holds at once.
template <int B>
int gj_setup() {
  cudaFuncSetAttribute(k_gj_cluster<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GJ_SMEM);
  if (cudaFuncSetAttribute(k_gj_cluster<B>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(GJ_MAX_CTAS);
  lc.blockDim = dim3(GJ_THREADS);
  lc.dynamicSmemBytes = GJ_SMEM;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = GJ_MAX_CTAS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  int got = 0;
  if (cudaOccupancyMaxActiveClusters(&got, k_gj_cluster<B>, &lc) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return got;
}

size_t gw_smem(int n) { return sizeof(double) * (size_t)gj_rows(n, GJ_MAX_CTAS) * (GW_B + 1); }

cudaLaunchConfig_t gw_config(int n, int mats, cudaLaunchAttribute* at, cudaStream_t st) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(GJ_MAX_CTAS * mats);
  lc.blockDim = dim3(GJ_THREADS);
  lc.dynamicSmemBytes = gw_smem(n);
  lc.stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = GJ_MAX_CTAS;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  return lc;
}

// Whether clusters of 16 blocks of the panel kernel fit the device.
bool gw_setup() {
  cudaFuncSetAttribute(k_gj_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gw_smem(GW_MAX));
  int got = 0;
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t lc = gw_config(GW_MAX, 1, &at, nullptr);
  if (cudaFuncSetAttribute(k_gj_panel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&got, k_gj_panel, &lc) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return got > 0;
}

}  // namespace

size_t gj_wide_scratch(int n) { return sizeof(double) * 33 * (size_t)n; }

bool launch_gj_wide(const Config& cfg, int n, int* d_sgn, cudaStream_t st) {
  static std::mutex mu;
  static int state[64] = {0};  // per device: 0 unknown, 1 not available, 2 available
  if (n < GW_MIN || n > GW_MAX) return false;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (state[dev] == 0) state[dev] = gw_setup() ? 2 : 1;
    if (state[dev] != 2) return false;
  }
  const int mats = 2 * cfg.n_walkers;
  const long long items = (long long)mats * blocks_of(n, GW_R) * blocks_of(n, GW_C);
  const int grid = persist_grid((const void*)k_gj_update, items, 256);
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t lc = gw_config(n, mats, &at, st);
  for (int c0 = 0; c0 < n; c0 += GW_B) {
    cudaLaunchKernelEx(&lc, k_gj_panel, cfg, c0, n, d_sgn);
    k_gj_update<<<grid, 256, 0, st>>>(cfg, c0, d_sgn);
  }
  k_gj_finish<<<dim3(n, mats), 256, sizeof(double) * n, st>>>(cfg, d_sgn);
  return true;
}

void launch_gj(const Config& cfg, int mode, int max_n, int* d_sgn, cudaStream_t st) {
  static std::mutex mu;
  static int state[64] = {0};  // per device: 0 unknown, else 1 + the clusters of 16 it holds
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  int wide;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (state[dev] == 0) {
      const int a = gj_setup<16>();
      gj_setup<4>();
      gj_setup<1>();
      state[dev] = 1 + a;
    }
    wide = state[dev] - 1;
  }
  if (max_n < 1) max_n = 1;
  const int mats = 2 * cfg.n_walkers;
  // Panels of 16 columns while the panel rows of a block fit beside X (n up to
  // about 9000 on 8 blocks), else of 4 (about 40000) or single columns.  Up to
  // GJ_WIDE_MATS matrices take clusters of 16 blocks, so that one matrix has the
  // FP64 units of 16 SMs; more take clusters of 8 on all SMs, a second wave of
  // the larger ones being slower: a sweep's recompute of 2 / 6 / 8 / 10 matrices of
  // order 310 1478 / 1596 / 2744 / 2839 us on clusters of 16, 2119 / 2328 / 2406 / 2407
  // on 8; of order 50 262 / - / 383 / 586 against 272 / - / 272 / 477.
  auto fits = [&](int c, int B) { return gj_rp_bytes(max_n, B) + gj_work_bytes(gj_rows(max_n, c), B) <= GJ_SMEM; };
  const int ctas = mats <= wide && mats <= GJ_WIDE_MATS && fits(GJ_MAX_CTAS, 16) ? GJ_MAX_CTAS : 8;
  const int fit = device_sm_count() / ctas > 0 ? device_sm_count() / ctas : 1;
  const int clusters = mats < fit ? mats : fit;
  if (fits(ctas, 16)) gj_launch<16>(cfg, mode, max_n, ctas, clusters, d_sgn, st);
  else if (fits(ctas, 4)) gj_launch<4>(cfg, mode, max_n, ctas, clusters, d_sgn, st);
  else gj_launch<1>(cfg, mode, max_n, ctas, clusters, d_sgn, st);
}

}  // namespace dca
