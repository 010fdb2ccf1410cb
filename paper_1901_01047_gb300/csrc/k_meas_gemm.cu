// k_meas_gemm.cu -- the correction term of a measurement of G(tau),
//   C[(x, a), r'] = sum_i g0(x - r_i, tau_a - tau_i) b_i(r'),
// scattered to Gtmp[sp][x - r'][a] (FP64 atomics).  The g0 factor is
// interpolated on the fly while tiles of MK vertices pass through shared
// memory, so a tile costs one interpolation per (x, a, i) and nc products of
// it; the work item is a site x, a block of tau points and all vertices of one
// walker-spin (or VSEG of them).
#include <cstdint>

#include "device_util.cuh"
#include "kernels.h"
#include "state.h"

namespace dca {

namespace {

constexpr int MK = 32;    // vertices per tile
constexpr int MT = 128;   // tau points per item, FP32 kernel
constexpr int AST = MT + 4;
// Vertices per item of the FP32 kernel (SPLIT) where the items of a measurement are
// fewer than the SMs without it: one walker of 16 sites with 256 tau points is 64
// items (order 640, 114 -> 76 us; a sweep's measurement with 32 / 128 items, order 408,
// 230 / 244 -> 216 / 233 us, one of 36 sites, 72 items, 300 -> 281).  With items enough
// the split only adds flushes and atomics: 256 / 768 / 12288 items of 16 sites 252 /
// 400 / 2326 -> 267 / 438 / 3044 us, 576 of 36 sites 458 -> 491.  Clusters above 36
// sites, one block an SM, lose from 98 items on.
constexpr int VSEG = 256, VSEG_ITEMS = 152;
template <bool SPLIT>
__host__ __device__ constexpr int vseg() {
  return SPLIT ? VSEG : 1 << 30;
}
constexpr int DT = 16;    // tau points per item, FP64 kernel

__device__ __forceinline__ bool wants_gemm(const WalkerDev& w) { return w.active && w.measure_pending; }

// Reference-site classes of the kernels: one instance each, so that the
// registers of the small clusters do not follow those of the large ones.
__device__ __forceinline__ int site_class(int nc) { return nc <= 16 ? 0 : (nc <= 36 ? 1 : 2); }

// ---------------------------------------------------------------------------
// FP32 (mixed path).  A thread owns TA tau points times SR sites; NG site
// groups times MT / TA tau threads form a k group, and 256 / that many k
// groups share the vertices of a tile.  The site group is uniform over a warp,
// so the b reads are broadcasts: per vertex 1 vector read of g0 and SR / 4 of b
// feed TA SR multiply-adds (16 or 18 for 2 or 4 reads), where one tau point
// times MR / 4 sites a thread read 17 values for 16.  The table values of the
// next tile are loaded into registers and the vertex records of the one after
// prepared while a tile is multiplied: one barrier per tile.  What is left is
// the interpolation, as many instructions as the products for nc <= 16.  One
// measurement: 4 walkers of 36 sites, order 860, 2048 tau points 6.3 -> 2.4 ms;
// 256 walkers of 8 and 16 sites, 128 points 1.26 -> 1.09 ms (without the loads
// ahead 1.34).  FP32 sums run over 32 vertices and
// are added into double-float totals.
// ---------------------------------------------------------------------------
struct MeasRec {  // one vertex of a tile
  int lo, hi;     // offsets of the two interpolation rows in the phase table (lo < 0: dead vertex)
  int mb;         // m offset
  float w;        // weight of the upper row
};

template <int NG, int SR>
constexpr int bs_stride() {
  return NG * ((SR + 3) & ~3) + 4;  // rows of b: 16-byte aligned groups, odd multiple of 4 words or near it
}

// dynamic shared memory of a site class
constexpr int smem_class(int c) {
  return 4 * 2 * MK * (AST + (c == 0 ? bs_stride<4, 4>() : (c == 1 ? bs_stride<4, 9>() : bs_stride<4, 16>())));
}

struct MeasSmem {
  MeasRec rec[2][MK];
  GridTime gi[2][MK];
  int row[2][MK];
};

// acc -> (hi, lo), error free in hi
__device__ __forceinline__ void df_add(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x), bb = __fsub_rn(s, hi);
  lo += __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
  hi = s;
}

template <bool SPLIT, int NG, int SR, int TA>
__device__ __forceinline__ void meas_item_f(const Config& cfg, const WalkerDev& w, int sp, int item, MeasSmem& sm,
                                            float* dyn) {
  constexpr int TT = MT / TA;            // tau threads
  constexpr int TPG = TT * NG;           // threads of a k group
  constexpr int KG = 256 / TPG;          // k groups
  constexpr int KP = MK / KG;            // vertices of a tile per k group
  constexpr int PAD = (SR + 3) & ~3;
  constexpr int BST = bs_stride<NG, SR>();
  const ProblemDev& pb = cfg.P[w.problem];
  const int nc = pb.nc, ntm = cfg.n_tau_meas, par = w.parity, ld = w.cap, q = pb.meas_q;
  constexpr int VS = vseg<SPLIT>();
  const int tblocks = (ntm + MT - 1) / MT, segs = (int)blocks_of(w.n, VS);
  const int v0 = (item % segs) * VS, n = (int)min((long long)w.n, (long long)v0 + VS);  // the item's vertices v0 .. n - 1
  item /= segs;
  const int x = item / tblocks, a0 = (item - x * tblocks) * MT;
  const int tid = threadIdx.x, kg = tid / TPG, tg = tid - kg * TPG, sg = tg / TT, ta = tg - sg * TT;
  float* const As = dyn;                      // [2][MK][AST]
  float* const Bs = dyn + 2 * MK * AST;       // [2][MK][BST]
  const int* vsite = w.vsite[par];
  const double* vtau = w.vtau[par];
  const int* vs = w.vs[par];
  const float* bvec = reinterpret_cast<const float*>(w.bvec) + (size_t)sp * nc * ld;

  auto prep = [&](int i0, int b) {
    if (tid < MK) {
      const int i = i0 + tid;
      const bool live = i < n && vs[i] != 0;
      const int d = live ? __ldg(pb.site_sub + x * nc + vsite[i]) : -1;
      MeasRec r{-1, -1, 0, 0.0f};
      if (live) {
        const GridTime gi = grid_time(vtau[i], pb.tau_scale);
        if (q > 0) {
          // grid offset of tau_a - tau_i: l = q a + c, c = q/2 - gi.i - (gi.f > 0), weight 1 - gi.f
          const int c = q / 2 - gi.i - (gi.f > 0.0f ? 1 : 0);
          const int p = ((c % q) + q) % q, mrow = ntm + 1;
          r.lo = (p * nc + d) * mrow;
          r.hi = p + 1 < q ? r.lo + nc * mrow : d * mrow + 1;
          r.mb = (c - p) / q;
          r.w = gi.f > 0.0f ? 1.0f - gi.f : 0.0f;
        } else {
          sm.gi[b][tid] = gi;
        }
      }
      sm.rec[b][tid] = r;
      sm.row[b][tid] = d;
    }
  };
  // this thread's tau point in the fill
  const int al = tid & (MT - 1), fa = a0 + al, il0 = tid / MT;
  const GridTime ga = q > 0 ? GridTime{0, 0.0f}
                            : grid_time(((double)fa + 0.5) * pb.beta / (double)ntm, pb.tau_scale);
  const float* gm = pb.g0m + (size_t)sp * q * nc * ((size_t)ntm + 1);
  // The two table values of this thread's entries of stage b's tile, in flight
  // while the tile before is multiplied (phase-table path).
  constexpr int FE = MK * MT / 256;
  float flo[FE], fhi[FE];
  auto fetch = [&](int b) {
    if (q <= 0) return;
#pragma unroll
    for (int s = 0; s < FE; ++s) {
      const MeasRec r = sm.rec[b][il0 + (256 / MT) * s];
      int m = fa + r.mb;
      if (m < 0) m += ntm;  // tau_a - tau_i < 0: antiperiodic continuation
      const bool ok = r.lo >= 0 && fa < ntm;
      flo[s] = ok ? __ldg(gm + r.lo + m) : 0.0f;
      fhi[s] = ok ? __ldg(gm + r.hi + m) : 0.0f;
    }
  };
  auto fill = [&](int i0, int b) {
    float* A = As + (size_t)b * MK * AST + al;
    if (q > 0) {
#pragma unroll
      for (int s = 0; s < FE; ++s) {
        const int il = il0 + (256 / MT) * s;
        const float v = flo[s] + sm.rec[b][il].w * (fhi[s] - flo[s]);
        A[il * AST] = fa + sm.rec[b][il].mb < 0 ? -v : v;
      }
    } else {
      for (int s = 0; s < FE; ++s) {
        const int il = il0 + (256 / MT) * s, d = sm.row[b][il];
        A[il * AST] = (fa < ntm && d >= 0) ? g0_interp_grid(g0f_row(pb, sp, d), pb.n_tau, ga, sm.gi[b][il]) : 0.0f;
      }
    }
    float* B = Bs + (size_t)b * MK * BST;
    for (int e = tid; e < MK * NG * PAD; e += 256) {
      const int il = e & (MK - 1), slot = e / MK, g = slot / PAD, m = slot - g * PAD, rp = g * SR + m;
      B[il * BST + slot] = (m < SR && rp < nc && i0 + il < n) ? bvec[(size_t)rp * ld + i0 + il] : 0.0f;
    }
  };
  float acc[TA][SR], th[TA][SR], tl[TA][SR];
#pragma unroll
  for (int u = 0; u < TA; ++u)
#pragma unroll
    for (int m = 0; m < SR; ++m) acc[u][m] = th[u][m] = tl[u][m] = 0.0f;
  auto compute = [&](int b) {
    const float* A = As + (size_t)b * MK * AST + (size_t)kg * KP * AST + ta * TA;
    const float* B = Bs + (size_t)b * MK * BST + (size_t)kg * KP * BST + sg * PAD;
#pragma unroll 4
    for (int k = 0; k < KP; ++k) {
      float g[TA], bv[PAD];
      if constexpr (TA == 4) {
        const float4 v = *reinterpret_cast<const float4*>(A + k * AST);
        g[0] = v.x;
        g[1] = v.y;
        g[2] = v.z;
        g[3] = v.w;
      } else {
        const float2 v = *reinterpret_cast<const float2*>(A + k * AST);
        g[0] = v.x;
        g[1] = v.y;
      }
#pragma unroll
      for (int m = 0; m < PAD; m += 4) {
        const float4 v = *reinterpret_cast<const float4*>(B + k * BST + m);
        bv[m] = v.x;
        bv[m + 1] = v.y;
        bv[m + 2] = v.z;
        bv[m + 3] = v.w;
      }
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int m = 0; m < SR; ++m) acc[u][m] += g[u] * bv[m];
    }
  };
  auto flush = [&]() {
#pragma unroll
    for (int u = 0; u < TA; ++u)
#pragma unroll
      for (int m = 0; m < SR; ++m) {
        df_add(th[u][m], tl[u][m], acc[u][m]);
        acc[u][m] = 0.0f;
      }
  };

  __syncthreads();  // the previous item of this block is done with the shared tiles
  if (v0 < n) {
    prep(v0, 0);
    if (v0 + MK < n) prep(v0 + MK, 1);
    __syncthreads();
    fetch(0);
    fill(v0, 0);
    __syncthreads();
    for (int i0 = v0, t = 0; i0 < n; i0 += MK, ++t) {
      const int b = t & 1;
      if (i0 + MK < n) fetch(b ^ 1);
      compute(b);
      if ((t & (KG - 1)) == KG - 1) flush();      // every 32 vertices of this k group
      if (i0 + MK < n) fill(i0 + MK, b ^ 1);     // reads the records of stage b ^ 1
      if (i0 + 2 * MK < n) prep(i0 + 2 * MK, b);  // stage b's records were read one tile ago
      __syncthreads();
    }
    flush();
  }
  // totals of the k groups, through the g0 tiles (all reads of them are past the last barrier)
  if constexpr (KG > 1) {
    float2* R = reinterpret_cast<float2*>(dyn);  // [k group - 1][TA SR][TPG]
    static_assert((KG - 1) * TPG * TA * SR * 8 <= smem_class(0), "reduction buffer");
    if (kg > 0)
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int m = 0; m < SR; ++m)
          R[((size_t)(kg - 1) * TA * SR + u * SR + m) * TPG + tg] = make_float2(th[u][m], tl[u][m]);
    __syncthreads();
    if (kg == 0)
      for (int g = 0; g < KG - 1; ++g)
#pragma unroll
        for (int u = 0; u < TA; ++u)
#pragma unroll
          for (int m = 0; m < SR; ++m) {
            const float2 v = R[((size_t)g * TA * SR + u * SR + m) * TPG + tg];
            df_add(th[u][m], tl[u][m], v.x);
            tl[u][m] += v.y;
          }
  }
  if (kg == 0)
#pragma unroll
    for (int m = 0; m < SR; ++m) {
      const int rp = sg * SR + m;
      if (rp >= nc) continue;
      const int d = __ldg(pb.site_sub + x * nc + rp);
      double* out = w.Gtmp + ((size_t)sp * nc + d) * ntm;
#pragma unroll
      for (int u = 0; u < TA; ++u) {
        const int a = a0 + ta * TA + u;
        if (a < ntm) atomicAdd(out + a, (double)th[u][m] + (double)tl[u][m]);
      }
    }
}

}  // namespace

template <int CLASS, bool SPLIT>
__global__ void __launch_bounds__(256, CLASS == 2 ? 1 : 2) k_meas_gemm(Config cfg) {
  extern __shared__ __align__(16) float dyn[];
  __shared__ MeasSmem sm;
  for_each_item(
      2 * cfg.n_walkers,
      [&](int s) -> long long {
        const WalkerDev& w = cfg.W[s >> 1];
        const int nc = cfg.P[w.problem].nc;
        return (wants_gemm(w) && site_class(nc) == CLASS)
                   ? (long long)nc * blocks_of(cfg.n_tau_meas, MT) * blocks_of(w.n, vseg<SPLIT>()) : 0;
      },
      [&](int s, int item) {
        const WalkerDev& w = cfg.W[s >> 1];
        if constexpr (CLASS == 0) {
          if (cfg.P[w.problem].nc <= 8) meas_item_f<SPLIT, 2, 4, 4>(cfg, w, s & 1, item, sm, dyn);
          else meas_item_f<SPLIT, 4, 4, 4>(cfg, w, s & 1, item, sm, dyn);
        } else if constexpr (CLASS == 1) {
          meas_item_f<SPLIT, 4, 9, 2>(cfg, w, s & 1, item, sm, dyn);
        } else {
          meas_item_f<SPLIT, 4, 16, 2>(cfg, w, s & 1, item, sm, dyn);
        }
      });
}

// ---------------------------------------------------------------------------
// FP64.  Bound by the two FP64 lanes of an SM, so the count of FP64 operations
// and an even share of the SMs decide: items of DT = 16 tau points; on a
// commensurate grid (n_tau an even multiple of n_tau_meas) the table index of
// tau_a - tau_i is q a + c_i with one weight per vertex, two operations per
// value instead of about ten.  One walker of 16 sites, order 311, 256 points:
// 253 -> 135 us; 48 of 4 sites, order 41, 128 points: 230 -> 67 us (64 points
// an item: 32 to 128 items for 152 SMs).  Thread = tau point times site (rr of 16; NM
// sites 16 apart for nc > 16), the vertices of a tile shared by the 16 / P
// groups where P = the power of two holding nc.
// ---------------------------------------------------------------------------
template <int NM>
__global__ void __launch_bounds__(256) k_meas_gemm64(Config cfg) {
  __shared__ double As[MK][DT];
  __shared__ double Bs[MK][16 * NM];
  __shared__ double s_w[MK], s_t[MK], s_red[256];
  __shared__ int s_d[MK], s_c[MK];
  for_each_item(
      2 * cfg.n_walkers,
      [&](int s) -> long long {
        const WalkerDev& w = cfg.W[s >> 1];
        const int nc = cfg.P[w.problem].nc;
        return (wants_gemm(w) && (nc > 16) == (NM > 1)) ? (long long)nc * blocks_of(cfg.n_tau_meas, DT) : 0;
      },
      [&](int s, int item) {
        const WalkerDev& w = cfg.W[s >> 1];
        const ProblemDev& pb = cfg.P[w.problem];
        const int sp = s & 1, nc = pb.nc, ntm = cfg.n_tau_meas, n = w.n, par = w.parity, ld = w.cap, np1 = pb.n_tau + 1;
        const int tblocks = (ntm + DT - 1) / DT, x = item / tblocks, a0 = (item - x * tblocks) * DT;
        const int q1 = pb.n_tau % ntm == 0 ? pb.n_tau / ntm : 0, q = (q1 & 1) ? 0 : q1;
        const int tid = threadIdx.x, al = tid & (DT - 1), rr = tid / DT, a = a0 + al;
        int lp = 4;  // log2 of the sites side by side
        if (NM == 1)
          while (lp > 0 && (1 << (lp - 1)) >= nc) --lp;
        const int r = rr & ((1 << lp) - 1), g = rr >> lp, G = 16 >> lp;
        const double ta = ((double)a + 0.5) * pb.beta / (double)ntm;
        const double* tab = pb.g0 + (size_t)sp * nc * np1;
        const double* bvec = w.bvec + (size_t)sp * nc * ld;
        double acc[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) acc[m] = 0.0;
        for (int i0 = 0; i0 < n; i0 += MK) {
          __syncthreads();  // the previous tile (or item) is done with the shared tiles
          if (tid < MK) {
            const int i = i0 + tid;
            const bool live = i < n && w.vs[par][i] != 0;
            s_d[tid] = live ? __ldg(pb.site_sub + x * nc + w.vsite[par][i]) : -1;
            if (live) {
              const double ti = w.vtau[par][i];
              s_t[tid] = ti;
              // grid offset of tau_a - tau_i: q a + c, c = q/2 - floor(x_i) - (f > 0), weight 1 - f
              const double xg = ti * pb.tau_scale, fl = floor(xg), f = xg - fl;
              s_c[tid] = q / 2 - (int)fl - (f > 0.0 ? 1 : 0);
              s_w[tid] = f > 0.0 ? 1.0 - f : 0.0;
            }
          }
          for (int e = tid; e < MK * 16 * NM; e += 256) {
            const int il = e & (MK - 1), rp = e / MK;
            Bs[il][rp] = (rp < nc && i0 + il < n) ? bvec[(size_t)rp * ld + i0 + il] : 0.0;
          }
          __syncthreads();
#pragma unroll
          for (int u = 0; u < MK * DT / 256; ++u) {
            const int il = rr + (256 / DT) * u, d = s_d[il];
            double v = 0.0;
            if (d >= 0 && a < ntm) {
              const double* row = tab + (size_t)d * np1;
              if (q > 0) {
                int l = q * a + s_c[il];
                const bool neg = l < 0;  // antiperiodic continuation
                if (neg) l += pb.n_tau;
                const double lo = __ldg(row + l), hi = __ldg(row + l + 1);
                v = fma(s_w[il], hi - lo, lo);
                if (neg) v = -v;
              } else {
                v = g0_interp(row, pb.n_tau, pb.beta, pb.tau_scale, ta - s_t[il]);
              }
            }
            As[il][al] = v;
          }
          __syncthreads();
          const int len = min(MK, n - i0);
          if (r < nc)
#pragma unroll 4
            for (int k = g; k < len; k += G) {
              const double v = As[k][al];
#pragma unroll
              for (int m = 0; m < NM; ++m) acc[m] = fma(v, Bs[k][r + 16 * m], acc[m]);
            }
        }
        if (NM == 1 && G > 1) {
          __syncthreads();  // s_red of the previous item read
          s_red[tid] = acc[0];
          __syncthreads();
          if (g == 0)
            for (int h = 1; h < G; ++h) acc[0] += s_red[tid + h * (DT << lp)];
        }
        if (g == 0 && a < ntm)
#pragma unroll
          for (int m = 0; m < NM; ++m) {
            const int rp = r + 16 * m;
            if (rp < nc)
              atomicAdd(&w.Gtmp[((size_t)sp * nc + __ldg(pb.site_sub + x * nc + rp)) * ntm + a], acc[m]);
          }
      });
}

cudaError_t setup_meas_gemm() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* fn, int c) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_class(c));
  };
  set((const void*)k_meas_gemm<0, false>, 0);
  set((const void*)k_meas_gemm<0, true>, 0);
  set((const void*)k_meas_gemm<1, false>, 1);
  set((const void*)k_meas_gemm<1, true>, 1);
  set((const void*)k_meas_gemm<2, false>, 2);
  return e;
}

template <int CLASS, bool SPLIT>
static void gemm_f(const Config& cfg, long long items, cudaStream_t st) {
  constexpr int sm = smem_class(CLASS);
  const void* fn = (const void*)k_meas_gemm<CLASS, SPLIT>;
  k_meas_gemm<CLASS, SPLIT><<<persist_grid(fn, items, 256, sm), 256, sm, st>>>(cfg);
}

int launch_meas_gemm(const Config& cfg, int max_cap, int max_nc, cudaStream_t st) {
  const long long S = 2LL * cfg.n_walkers;
  if (cfg.prec == PREC_MIXED) {
    const long long items = S * max_nc * blocks_of(cfg.n_tau_meas, MT);
    // walkers that measure in one window: all under the lockstep schedule, else about
    // one of the windows that a sweep takes
    const long long at_once = cfg.pooled ? blocks_of(cfg.n_walkers, 8) : cfg.n_walkers;
    auto split = [&](int nc) { return 2 * at_once * nc * blocks_of(cfg.n_tau_meas, MT) < VSEG_ITEMS; };
    const long long parts = items * blocks_of(max_cap, VSEG);
    if (split(max_nc < 16 ? max_nc : 16)) gemm_f<0, true>(cfg, parts, st);
    else gemm_f<0, false>(cfg, items, st);
    if (max_nc > 16) {
      if (split(max_nc < 36 ? max_nc : 36)) gemm_f<1, true>(cfg, parts, st);
      else gemm_f<1, false>(cfg, items, st);
    }
    if (max_nc > 36) gemm_f<2, false>(cfg, items, st);
    return 1 + (max_nc > 16) + (max_nc > 36);
  }
  const long long items = S * max_nc * blocks_of(cfg.n_tau_meas, DT);
  k_meas_gemm64<1><<<persist_grid((const void*)k_meas_gemm64<1>, items, 256), 256, 0, st>>>(cfg);
  if (max_nc > 16) k_meas_gemm64<4><<<persist_grid((const void*)k_meas_gemm64<4>, items, 256), 256, 0, st>>>(cfg);
  return 1 + (max_nc > 16);
}

}  // namespace dca
