// ext_view.cuh -- entries of the extended G of a window (existing rows of N and
// the candidate rows / columns), and the bookkeeping that ends a Metropolis
// kernel.
#pragma once
#include "device_util.cuh"
#include "state.h"

namespace dca {

constexpr int METRO_SMEM_KS = 96;   // largest k_s whose B^-1 (both spins) lives in shared memory
constexpr int METRO_LIVE = 2048;    // live vertices whose rows and spins are staged in shared memory

template <typename T>
struct ExtView {
  const T* N;        // current N (ld)
  const T* X;        // candidate rows [c][ld] (stored like N)
  const double* Gc;  // candidate columns [c][ld]
  const int* vs;
  int n, ld;
};

template <typename T>
__device__ __forceinline__ ExtView<T> make_view(const WalkerDev& w, int sp) {
  ExtView<T> v;
  v.N = (const T*)w.N[w.parity][sp];
  v.X = reinterpret_cast<const T*>(w.Xr[sp]);
  v.Gc = w.Gc[sp];
  v.vs = w.vs[w.parity];
  v.n = w.n;
  v.ld = w.cap;
  return v;
}

// G_ext[x, y]; for an interacting existing column y, G = (N e^{V} - I) / (e^{V} - 1)
// column-wise, which follows from N = [I + G (e^V - I)] e^{-V}.
template <typename T>
__device__ __forceinline__ double g_ext(const ExtView<T>& v, const ProblemDev& pb, int sp, int x, int y) {
  if (y >= v.n) return v.Gc[(size_t)(y - v.n) * v.ld + x];
  const double nxy = ldN(x < v.n ? v.N : v.X, (size_t)(x < v.n ? x : x - v.n) * v.ld + y);
  const int sy = v.vs[y];
  const double ev = expV(pb, sp, sy);
  // (N e^V - 1) / (e^V - 1) with the reciprocal tabulated per spin (no FP64 division)
  return (nxy * ev - (x == y ? 1.0 : 0.0)) * pb.rexpVm1[sp][sy > 0 ? 1 : 0];
}

// G_ext[x, y] with the spin factors of column y given: e^{V_y} and
// 1 / (e^{V_y} - 1) (unused for a candidate column y >= n).
template <typename T>
__device__ __forceinline__ double g_ext_at(const ExtView<T>& v, int x, int y, double ev, double rv) {
  if (y >= v.n) return v.Gc[(size_t)(y - v.n) * v.ld + x];
  const double nxy = ldN(x < v.n ? v.N : v.X, (size_t)(x < v.n ? x : x - v.n) * v.ld + y);
  return (nxy * ev - (x == y ? 1.0 : 0.0)) * rv;
}

// Address of the stored entry g_ext_at reads for (x, y).
template <typename T>
__device__ __forceinline__ const void* g_ext_ptr(const ExtView<T>& v, int x, int y) {
  if (y >= v.n) return v.Gc + (size_t)(y - v.n) * v.ld + x;
  return (x < v.n) ? (const void*)(v.N + (size_t)x * v.ld + y) : (const void*)(v.X + (size_t)(x - v.n) * v.ld + y);
}

__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// End of the window's Metropolis (one thread): the counters of l accepted
// changes, nrem removals and nins insertions after `eval` of `len` proposals,
// and what the window still has to do (measurement, recompute).
__device__ __forceinline__ void metro_finish(const Config& cfg, WalkerDev& w, int n_live, int len, int l, int nrem,
                                             int nins, int eval, double sign) {
  w.n_acc = l;
  w.n_removed = nrem;
  w.n_ins = nins;
  w.n_eval = eval;
  w.aborted = (eval < len) && w.status == ST_OK;
  w.sign = sign;
  if (w.status == ST_OK) {
    w.q += (uint64_t)eval;
    w.sweep_pos += eval;
    w.n_windows++;
    if (w.aborted) w.n_aborts++;
    const int64_t sweep_no = w.sweeps_done;  // the sweep this window belongs to
    if (w.sweep_pos >= w.sweep_len_cur) {
      w.measure_pending = (w.sweeps_done >= cfg.warmup) ? 1 : 0;
      w.sweeps_done++;
      w.sweep_pos = 0;
    }
    w.windows_since_recompute++;
    if (cfg.recompute_every > 0 && w.windows_since_recompute >= cfg.recompute_every) {
      w.recompute_pending = 1;
      w.windows_since_recompute = 0;
    }
    // Batched schedule: every walker recomputes after the first window of
    // every recompute_sweeps-th sweep (the same window for all walkers).
    // (With N recomputed at every measurement the measured sweeps need no other.)
    if (cfg.recompute_sweeps > 0 && w.first_window && sweep_no > 0 && sweep_no % cfg.recompute_sweeps == 0 &&
        !(cfg.recompute_at_measure && sweep_no > cfg.warmup)) {
      w.recompute_pending = 1;
      w.windows_since_recompute = 0;
    }
    // Fresh N for every measurement: the recompute runs in the window that
    // ends the sweep, before the measurement.
    if (cfg.recompute_at_measure && w.measure_pending) {
      w.recompute_pending = 1;
      w.windows_since_recompute = 0;
    }
    // Algorithmic work per spin on the k live vertices after the window:
    // update 2 k^2 l + 2 k l^2 flop, reading and writing k^2 entries of N
    // plus the k x l factors; extension 4 k0^2 c flop and one read of N (both
    // candidate products need only that one read).
    const double b = cfg.prec == PREC_MIXED ? 4.0 : 8.0;
    const double kk = (double)(n_live - nrem + nins), ll = (double)l;
    if (l > 0) {
      w.flops += 2.0 * (2.0 * kk * kk * ll + 2.0 * kk * ll * ll);
      w.upd_bytes += 2.0 * (b * 2.0 * kk * kk + 8.0 * 2.0 * kk * ll);
    }
    const double k0 = (double)n_live, cc = (double)w.n_cand;
    if (w.n_cand > 0) {
      w.ext_flops += 2.0 * (4.0 * k0 * k0 * cc);
      w.ext_bytes += 2.0 * b * (k0 * k0);
    }
  } else {
    w.active = 0;
    w.n_acc = 0;
  }
}

}  // namespace dca
