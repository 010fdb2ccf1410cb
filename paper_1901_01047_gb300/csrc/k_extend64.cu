// k_extend64.cu -- candidate extension of the FP64 path (Sec. 2.3, "Submatrix
// updates"), three products of FP64 matrices, each output written once:
//   k_ext64   G_ext[i, n + c] = sum_j N[i, j] V[c, j]
//             X[c, j]         = sum_i U[c, i] N[i, j]
//   k_cc64    G_ext[n + c', n + c] = sum_j X[c', j] V[c, j] + g0(c', c)
// with V and U tabulated by k_cand_zero (zero on dead vertices).
//
// Bound: GB300 issues two FP64 multiply-adds per clock and SM, so what counts
// is that all 152 SMs get an equal share; everything else (shared-memory
// reads, staging from L2) fits beside that.  An item is 4 rows (or columns)
// times 16 candidates with the inner index split over four groups of 64
// threads: at order 50 that is 52 items for the two spins, at order 310 with
// 32 candidates 624.  Against 64 x 64 tiles of N with FP64 atomics (2 and 50
// items), both products of a window: order 56, 16 candidates 75 -> 7 us;
// order 311, 32 candidates 94 -> 38 us, its candidate block 66 -> 12 us.  One
// sweep of a 16-site walker (order 311) 2.46 -> 1.70 ms, four of the 2x2
// cluster (order 56) 2.01 -> 1.33 ms, of the atom 0.74 -> 0.48 ms, with the
// factor tables (k_cand_zero) spread over the SMs.
#include <cstdint>

#include "device_util.cuh"
#include "kernels.h"
#include "state.h"

namespace dca {

namespace {

constexpr int ER = 4;              // rows of the item
constexpr int EC = 16;             // candidates of the item
constexpr int EG = 256 / (ER * EC);  // groups sharing the inner index
constexpr int EK = 32 * EG;        // inner extent of a staged chunk: 32 per group
constexpr int EST = EK + 1;        // odd row stride: conflict-free rows of B

__device__ __forceinline__ long long ext64_blocks(const WalkerDev& w) {
  return (w.active && w.n_cand > 0) ? blocks_of(w.n, ER) * blocks_of(w.n_cand, EC) : 0;
}

__device__ __forceinline__ long long cc64_blocks(const WalkerDev& w) {
  return (w.active && w.n_cand > 0) ? blocks_of(w.n_cand, ER) * blocks_of(w.n_cand, EC) : 0;
}

struct Ext64Smem {
  double a[ER][EST];
  double b[EC][EST];
  double red[256];
};

// sum_{k < n} a(r, k) b(c, k) of the item's outputs, r < ER, c < EC: thread
// (group, r, c) sums its 32 inner indexes of every chunk, the next chunk's
// loads in flight in registers meanwhile; the group sums are added in a fixed
// order.  a(r, k) is read from A + r * sr + k * sk, zero for r >= nr; with
// sk = 1 consecutive threads read consecutive k, else consecutive r.  Threads
// below ER * EC return the sum of output (tid / EC, tid % EC).
__device__ __forceinline__ double ext64_tile(Ext64Smem& s, int n, const double* __restrict__ A, size_t sr, size_t sk,
                                             int nr, const double* __restrict__ B, int ld, int nb) {
  const int tid = threadIdx.x, c = tid & (EC - 1), r = (tid / EC) & (ER - 1), g = tid / (ER * EC);
  constexpr int PA = ER * EK / 256, PB = EC * EK / 256;
  double ra[PA], rb[PB];
  const bool rows = sk == 1;
  auto a_at = [&](int e, int& rr, int& kk) {
    rr = rows ? e / EK : e % ER;
    kk = rows ? e % EK : e / ER;
  };
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < PA; ++q) {
      int rr, kk;
      a_at(tid + 256 * q, rr, kk);
      ra[q] = (rr < nr && k0 + kk < n) ? A[(size_t)rr * sr + (size_t)(k0 + kk) * sk] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < PB; ++q) {
      const int e = tid + 256 * q, cc = e / EK, kk = e % EK;
      rb[q] = (cc < nb && k0 + kk < n) ? B[(size_t)cc * ld + k0 + kk] : 0.0;
    }
  };
  double acc = 0.0;
  if (n > 0) fetch(0);
  for (int k0 = 0; k0 < n; k0 += EK) {
    __syncthreads();  // the previous chunk (or item) is done with the shared tiles
#pragma unroll
    for (int q = 0; q < PA; ++q) {
      int rr, kk;
      a_at(tid + 256 * q, rr, kk);
      s.a[rr][kk] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < PB; ++q) {
      const int e = tid + 256 * q;
      s.b[e / EK][e % EK] = rb[q];
    }
    __syncthreads();
    if (k0 + EK < n) fetch(k0 + EK);
    // every EG-th inner index: a short last chunk is still shared by all groups
    const int len = min(EK, n - k0);
    const double* pa = s.a[r];
    const double* pb = s.b[c];
#pragma unroll 4
    for (int k = g; k < len; k += EG) acc = fma(pa[k], pb[k], acc);
  }
  __syncthreads();  // s.red of the previous item read
  s.red[tid] = acc;
  __syncthreads();
  double sum = 0.0;
  if (tid < ER * EC)
#pragma unroll
    for (int q = 0; q < EG; ++q) sum += s.red[tid + q * ER * EC];
  return sum;
}

}  // namespace

__global__ void __launch_bounds__(256) k_ext64(Config cfg) {
  __shared__ Ext64Smem sm;
  for_each_item(
      2 * cfg.n_walkers, [&](int s) -> long long { return 2 * ext64_blocks(cfg.W[s >> 1]); },
      [&](int s, int item) {
        const WalkerDev& w = cfg.W[s >> 1];
        const int sp = s & 1, n = w.n, nc_ = w.n_cand, ld = w.cap;
        const double* N = (const double*)w.N[w.parity][sp];
        const int blocks = (int)ext64_blocks(w), xb = item >= blocks ? 1 : 0, t = item - xb * blocks;
        const int rblocks = (n + ER - 1) / ER, cb = (t / rblocks) * EC, i0 = (t % rblocks) * ER;
        const double v = ext64_tile(sm, n, xb ? N + i0 : N + (size_t)i0 * ld, xb ? 1 : ld, xb ? ld : 1, n - i0,
                                    (xb ? w.Ub[sp] : w.Vb[sp]) + (size_t)cb * ld, ld, nc_ - cb);
        const int c = cb + (threadIdx.x & (EC - 1)), i = i0 + threadIdx.x / EC;
        if (threadIdx.x < ER * EC && c < nc_ && i < n) (xb ? w.Xr[sp] : w.Gc[sp])[(size_t)c * ld + i] = v;
      });
}

__global__ void __launch_bounds__(256) k_cc64(Config cfg) {
  __shared__ Ext64Smem sm;
  for_each_item(
      2 * cfg.n_walkers, [&](int s) -> long long { return cc64_blocks(cfg.W[s >> 1]); },
      [&](int s, int item) {
        const WalkerDev& w = cfg.W[s >> 1];
        const int sp = s & 1, n = w.n, nc_ = w.n_cand, ld = w.cap, par = w.parity;
        const int rblocks = (nc_ + ER - 1) / ER, cb = (item / rblocks) * EC, r0 = (item % rblocks) * ER;
        const double v = ext64_tile(sm, n, w.Xr[sp] + (size_t)r0 * ld, ld, 1, nc_ - r0, w.Vb[sp] + (size_t)cb * ld, ld,
                                    nc_ - cb);
        const int c = cb + (threadIdx.x & (EC - 1)), cp = r0 + threadIdx.x / EC;
        if (threadIdx.x < ER * EC && c < nc_ && cp < nc_) {
          const ProblemDev& pb = cfg.P[w.problem];
          const int rc = w.vsite[par][n + c];
          const double g = cp == c ? g0_diag(pb, sp, rc)
                                   : g0_pair(pb, sp, w.vsite[par][n + cp], w.vtau[par][n + cp], rc, w.vtau[par][n + c]);
          w.Gc[sp][(size_t)c * ld + n + cp] = v + g;
        }
      });
}

int launch_ext64(const Config& cfg, int max_cap, cudaStream_t st) {
  const long long S = 2LL * cfg.n_walkers, cb = blocks_of(cfg.ks, EC);
  k_ext64<<<persist_grid((const void*)k_ext64, 2 * S * cb * blocks_of(max_cap, ER), 256), 256, 0, st>>>(cfg);
  k_cc64<<<persist_grid((const void*)k_cc64, S * cb * blocks_of(cfg.ks, ER), 256), 256, 0, st>>>(cfg);
  return 2;
}

}  // namespace dca
