// k_correct_tc.cu -- the terms of the Newton recompute N1 = N0 + N0 R (+ N0 R^2)
// on the 5th generation tensor cores (mixed precision):  D = N0 R,  R = I - A N0
// from the digit planes (k_refine_oz, which stores R^T split into two TF32
// planes), and where newton_second() asks for it D R.
// 3xTF32 as in the other products with N: hi = tf32(x), lo = tf32(x - hi) and
// hi hi + hi lo + lo hi.  The tensor cores truncate when they add to an accumulator,
// so the hi hi products of every 32 inner indexes go to an accumulator of their
// own, added in FP32 registers; the cross terms, 2^-12 of them, have one for the
// whole item.  Error of N0 R against 64 bits, relative, random matrices of order
// 40 / 129 / 300 / 900: 1.2e-7 / 1.4e-7 / 1.4e-7 / 1.7e-7, the FP32 kernel
// (k_refine_correct) 1.1e-7 / 2.1e-7 / 3.1e-7 / 5.4e-7, one accumulator for all
// 3.4e-7 / 1.0e-6 / 2.2e-6 / 6.4e-6 (below order 40 up to twice the FP32 kernel's,
// of a term that is then below the rounding of N1).  Time of one walker of order
// 670 / 900: 35.1 / 43.2 us with the second term's idle launch, with one
// accumulator 34.6 / 39.4, the FP32 kernel 94 / 117.
//
// Bound: 3 x 2 n^3 flop per spin at the TF32 rate (the FP32 pipes, where
// k_refine_correct runs at their peak, are 12 times slower); every 128 x 128
// tile of N1 re-reads 2 x 128 rows from L2.  256 walkers of orders 90 to 900:
// 1.84 -> 0.46 ms a recompute, and a pass of the batch 15.4 -> 13.9 ms; 4
// walkers of 36 sites 9.47 -> 8.95 ms (both with one accumulator).  The residual
// kernel pays 0.3 ms of it for storing R transposed and split.  Work item = one
// such tile of one walker-spin; the CTA (one per SM, 448 threads) streams the
// inner index 32 at a time through a three-stage ring:
//   warp 4 (TMA producer)   N0 (or D) box (128 rows x 32 columns), R^T hi and lo boxes;
//   warps 0-3 (converters)  split that box in place into hi and a lo plane,
//                           zeros outside the live rows and columns;
//   warp 5 (MMA issuer)     4 K steps x 3 tcgen05.mma kind::tf32 (M = N = 128):
//                           hi hi into one of two TMEM accumulators in turn,
//                           the cross terms into one of two others per item;
//   warps 6-13 (epilogue)   add the chunks up, store the sum at the item's end.
// Every wait is bounded; a timeout sets the walker's status to
// ST_ERR_TIMEOUT, lets the copies in flight land, frees the tensor memory and
// returns.
#include <cstdint>

#include "device_util.cuh"
#include "kernels.h"
#include "state.h"
#include "item_plan.cuh"
#include "tc_ptx.cuh"

namespace dca {

namespace {

constexpr int CB = 128;        // tile of the product
constexpr int CE = 64;         // its columns per epilogue warp
constexpr int CO_THREADS = 448;  // converters 0-3, producer 4, issuer 5, epilogue 6-13

struct CoLayout {
  static constexpr int BOX = CB * 128;     // 128 rows x 32 FP32 columns
  static constexpr int STAGE = 4 * BOX;    // N0 hi (as loaded, then split), N0 lo, R^T hi, R^T lo
  static constexpr int STAGES = 3;
  static constexpr int OFF_BAR = STAGES * STAGE;
  static constexpr int SMEM = OFF_BAR + 256 + 1024;
  static constexpr uint32_t TMEM_COLS = 4 * CB;
  static_assert(SMEM + sizeof(ItemPlan) + 1024 <= 232448, "shared memory (dynamic + the static item plan)");
};

template <bool SECOND>
__device__ __forceinline__ long long co_items(const Config& cfg, int s) {
  const WalkerDev& w = cfg.W[s >> 1];
  const long long t = (w.n + CB - 1) / CB;
  return (w.active && w.recompute_pending && w.status == ST_OK && (!SECOND || newton_second(w, s & 1))) ? t * t : 0;
}

template <bool SECOND>
struct CoIter {
  PlanWalk<ItemPlan> pw;
  __device__ void start(const ItemPlan& plan) { pw.start(plan); }
  __device__ bool next(const Config& cfg, int& set, int& i0, int& j0) {
    int sub = 0;
    if (!pw.next(2 * cfg.n_walkers, [&](int s) { return co_items<SECOND>(cfg, s); }, set, sub)) return false;
    const int t = (cfg.W[set >> 1].n + CB - 1) / CB;
    i0 = (sub / t) * CB;
    j0 = (sub % t) * CB;
    return true;
  }
};

}  // namespace

template <bool SECOND>
__global__ void __launch_bounds__(CO_THREADS, 1) k_correct_tc(Config cfg) {
  using L = CoLayout;
  constexpr int S = L::STAGES;
  extern __shared__ uint8_t co_raw[];
  const uint32_t raw = tc::smem_u32(co_raw);
  const uint32_t sb = (raw + 1023u) & ~1023u;  // 1024-byte aligned base (128-byte swizzle atoms)
  uint8_t* gb = co_raw + (sb - raw);
  const uint32_t bar = sb + L::OFF_BAR;
  // barriers: full[S], conv[S], empty[S], afull[2], aempty[2], fin
  auto full = [&](int st) { return bar + 8 * st; };
  auto conv = [&](int st) { return bar + 8 * (S + st); };
  auto empty = [&](int st) { return bar + 8 * (2 * S + st); };
  auto afull = [&](int b) { return bar + 8 * (3 * S + b); };
  auto aempty = [&](int b) { return bar + 8 * (3 * S + 2 + b); };
  const uint32_t fin = bar + 8 * (3 * S + 4);
  uint32_t* tmem_slot = (uint32_t*)(gb + L::OFF_BAR + 8 * (3 * S + 5));
  volatile int* abort_flag = (volatile int*)(gb + L::OFF_BAR + 8 * (3 * S + 5) + 4);
  static_assert(8 * (3 * S + 5) + 8 <= 256, "barrier area");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int st = 0; st < S; ++st) {
      tc::mbar_init(full(st), 1);
      tc::mbar_init(conv(st), 4);
      tc::mbar_init(empty(st), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(afull(b), 1);
      tc::mbar_init(aempty(b), 8);
    }
    tc::mbar_init(fin, 1);
    *abort_flag = 0;
    tc::fence_mbar_init();
  }
  if (warp == 5) {
    tc::tmem_alloc(tc::smem_u32(tmem_slot), L::TMEM_COLS);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  __shared__ ItemPlan plan;
  plan_items(plan, 2 * cfg.n_walkers, [&](int s) { return co_items<SECOND>(cfg, s); });

  CoIter<SECOND> it;
  it.start(plan);
  int set = 0, i0 = 0, j0 = 0;
  if (warp == 4) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      uint32_t g = 0;
      uint32_t armed[S] = {};
      bool ok = true;
      while (ok && it.next(cfg, set, i0, j0)) {
        const WalkerDev& w = cfg.W[set >> 1];
        const int n = w.n;
        const TmapDev* m = cfg.tmaps + (size_t)set * TMAPS_PER_SPIN;
        const void* mN = m + 2 + w.parity;
        const void* mN32 = SECOND ? m + 11 : m + 6 + w.parity;  // 32-row boxes: the last, partial row block
        const void* mRh = m + 2 + (w.parity ^ 1);   // R^T hi in the other buffer of N
        const void* mRl = m + 10;                   // R^T lo in the upper half of the FP64 work matrix
        const int nsub = n - i0 >= CB ? 4 : (n - i0 + 31) / 32;  // 32-row boxes that start below n
        for (int k0 = 0; k0 < n; k0 += 32, ++g) {
          const int st = (int)(g % S);
          const uint32_t u = g / S;
          if (u > 0 && !tc::mbar_wait(empty(st), (u - 1) & 1u, abort_flag, cfg.wait_cycles)) {
            ok = false;
            break;
          }
          const uint32_t s0 = sb + st * L::STAGE;
          tc::mbar_expect_tx(full(st), (uint32_t)(nsub * (L::BOX / 4) + 2 * L::BOX));
          armed[st] = u + 1;
          if (!SECOND && nsub == 4) {
            tc::tma_load_2d(s0, mN, k0, i0, full(st));
          } else {
            for (int q = 0; q < nsub; ++q) tc::tma_load_2d(s0 + q * (L::BOX / 4), mN32, k0, i0 + 32 * q, full(st));
          }
          tc::tma_load_2d(s0 + 2 * L::BOX, mRh, k0, j0, full(st));
          tc::tma_load_2d(s0 + 3 * L::BOX, mRl, k0, j0, full(st));
        }
      }
      if (!ok) {
        set_status(cfg.W[set >> 1], ST_ERR_TIMEOUT);
        // the loads already issued land before the CTA exits
        for (int st = 0; st < S; ++st)
          if (armed[st] > 0) tc::mbar_wait(full(st), (armed[st] - 1) & 1u, nullptr, 400000000LL);
      }
    }
  } else if (warp == 5) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      uint32_t g = 0, k = 0;  // chunks and items so far
      bool ok = true;
      constexpr uint32_t idesc = tc::idesc_tf32(CB, CB);
      while (ok && it.next(cfg, set, i0, j0)) {
        const int n = cfg.W[set >> 1].n;
        // read out two items ago, before that item's last chunk was released
        const uint32_t x = tmem + (uint32_t)(2 * CB + CB * (int)(k & 1u));
        for (int k0 = 0; k0 < n; k0 += 32, ++g) {
          const int st = (int)(g % S), b = (int)(g & 1u);
          const uint32_t u = g / S;
          if (g >= 2 && !tc::mbar_wait(aempty(b), ((g >> 1) - 1) & 1u, abort_flag, cfg.wait_cycles)) {
            ok = false;
            break;
          }
          if (!tc::mbar_wait(conv(st), u & 1u, abort_flag, cfg.wait_cycles)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t d = tmem + (uint32_t)(CB * b);
          const uint32_t s0 = sb + st * L::STAGE;
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // K step of 8 columns: 32 bytes inside the 128-byte swizzle row
            const uint64_t ah = tc::sdesc_k_sw128(s0 + 32 * q), al = tc::sdesc_k_sw128(s0 + L::BOX + 32 * q);
            const uint64_t bh = tc::sdesc_k_sw128(s0 + 2 * L::BOX + 32 * q);
            const uint64_t bl = tc::sdesc_k_sw128(s0 + 3 * L::BOX + 32 * q);
            tc::mma_tf32(d, ah, bh, idesc, q > 0 ? 1u : 0u);
            tc::mma_tf32(x, ah, bl, idesc, k0 + q > 0 ? 1u : 0u);
            tc::mma_tf32(x, al, bh, idesc, 1u);
          }
          tc::mma_commit(empty(st));
          tc::mma_commit(afull(b));  // the chunk (and, at the item's end, the cross terms)
        }
        ++k;
      }
      if (!ok) set_status(cfg.W[set >> 1], ST_ERR_TIMEOUT);
      // every MMA of this CTA has completed before the tensor memory is freed
      tc::mma_commit(fin);
      tc::mbar_wait(fin, 0u, nullptr, 400000000LL);
    }
  } else if (warp < 4) {
    // ---------------- converters: warps 0-3 ----------------
    uint32_t g = 0;
    bool stop = false;
    const int r = 32 * warp + lane;  // row of the box
    while (!stop && it.next(cfg, set, i0, j0)) {
      const int n = cfg.W[set >> 1].n;
      const bool row_ok = i0 + r < n;
      for (int k0 = 0; k0 < n; k0 += 32, ++g) {
        const int st = (int)(g % S);
        const uint32_t u = g / S;
        const bool mine = tc::mbar_wait(full(st), u & 1u, abort_flag, cfg.wait_cycles);
        if (!__all_sync(0xffffffffu, mine)) {
          stop = true;
          break;
        }
        // logical 16-byte chunk lc of row r sits at physical chunk lc ^ (r & 7)
        // (128-byte swizzle); walking logical chunks spreads a warp over all banks
        uint8_t* nrow = gb + st * L::STAGE + r * 128;
#pragma unroll
        for (int lc = 0; lc < 8; ++lc) {
          const int pc = lc ^ (r & 7);
          float4* ph = (float4*)(nrow + pc * 16);
          float4* pl = (float4*)(nrow + L::BOX + pc * 16);
          const float4 x = *ph;
          const int kc = k0 + 4 * lc;
          const float xv[4] = {x.x, x.y, x.z, x.w};
          float hv[4], lv[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) tc::tf32_split(row_ok && kc + q < n ? xv[q] : 0.f, hv[q], lv[q]);
          *ph = make_float4(hv[0], hv[1], hv[2], hv[3]);
          *pl = make_float4(lv[0], lv[1], lv[2], lv[3]);
        }
        tc::fence_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(conv(st));
      }
    }
    if (stop && lane == 0) set_status(cfg.W[set >> 1], ST_ERR_TIMEOUT);
    if (stop) *abort_flag = 1;
  } else {
    // ---------------- epilogue: warps 6-13, TMEM lanes 32 (warp % 4) .. +31, CE columns ----------------
    uint32_t g = 0, k = 0;  // chunks and items so far
    bool stop = false;
    const int sub = warp & 3, r = 32 * sub + lane, c0 = CE * ((warp - 6) >> 2);
    const uint32_t lanes = tmem + ((uint32_t)(32 * sub) << 16) + (uint32_t)c0;
    while (!stop && it.next(cfg, set, i0, j0)) {
      WalkerDev& w = cfg.W[set >> 1];
      const int sp = set & 1, n = w.n, ld = w.cap, i = i0 + r;
      float* out = SECOND ? (float*)w.OzN[sp] : (float*)w.Ascr[sp];
      uint32_t dmax = 0u;
      float acc[CE];
#pragma unroll
      for (int c = 0; c < CE; ++c) acc[c] = 0.0f;
      for (int k0 = 0; k0 < n; k0 += 32, ++g) {
        const int b = (int)(g & 1u);
        const bool mine = tc::mbar_wait(afull(b), (g >> 1) & 1u, abort_flag, cfg.wait_cycles);
        if (!__all_sync(0xffffffffu, mine)) {
          stop = true;
          break;
        }
        tc::fence_after_sync();
#pragma unroll
        for (int cb = 0; cb < CE; cb += 32) {
          float v[32];
          tc::tmem_ld32(lanes + (uint32_t)(CB * b + cb), v);
#pragma unroll
          for (int c = 0; c < 32; ++c) acc[cb + c] = __fadd_rn(acc[cb + c], v[c]);
        }
        if (k0 + 32 >= n) {
#pragma unroll
          for (int cb = 0; cb < CE; cb += 32) {
            float v[32];
            tc::tmem_ld32(lanes + (uint32_t)(2 * CB + CB * (int)(k & 1u) + cb), v);
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[cb + c] = __fadd_rn(acc[cb + c], v[c]);
          }
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(aempty(b));
      }
      if (stop) break;
      ++k;
      if (i < n) {
        const size_t o = (size_t)i * ld + j0 + c0;  // 16-byte aligned: ld and j0 are multiples of 32
#pragma unroll
        for (int q = 0; q < CE / 4; ++q) {
          const int j = j0 + c0 + 4 * q;
          if (j + 3 < n) {
            *reinterpret_cast<float4*>(out + o + 4 * q) =
                make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (j + e < n) out[o + 4 * q + e] = acc[4 * q + e];
          }
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (j + e < n) dmax = max(dmax, abs_bits(acc[4 * q + e]));
        }
      }
      newton_max(&w.newton_bits[sp][SECOND ? 2 : 1], dmax);
    }
    if (stop && lane == 0) set_status(cfg.W[set >> 1], ST_ERR_TIMEOUT);
    if (stop) *abort_flag = 1;
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // an aborted CTA may have left any of its items undone: stop every walker it served
    it.start(plan);
    while (it.next(cfg, set, i0, j0)) set_status(cfg.W[set >> 1], ST_ERR_TIMEOUT);
  }
  if (warp == 5) {
    __syncwarp();
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, L::TMEM_COLS);
  }
}

cudaError_t setup_correct_tc() {
  const cudaError_t e =
      cudaFuncSetAttribute(k_correct_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, CoLayout::SMEM);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_correct_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, CoLayout::SMEM);
}

void launch_correct_tc(const Config& cfg, cudaStream_t st) {
  k_correct_tc<false><<<device_sm_count(), CO_THREADS, CoLayout::SMEM, st>>>(cfg);
  k_correct_tc<true><<<device_sm_count(), CO_THREADS, CoLayout::SMEM, st>>>(cfg);
}

}  // namespace dca
