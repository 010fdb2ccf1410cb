// k_metropolis.cu -- Metropolis decisions of one window with FP64 Gamma
// (B^-1 and the Schur complements), one block per walker.
//
// The window is a serial chain of up to k_s decisions, so the kernel is bound
// by the latency of one decision.  On GB300 a warp-wide FP64 instruction holds
// the FP64 unit of its SM sub-partition for 64 cycles, whatever the number of
// lanes in use; the layout below keeps the number of FP64 warp instructions
// on the chain small and everything else off it:
//   - warps 0 to 3 (one per sub-partition) carry the FP64 work, two warps per
//     spin, the rows of B^-1 on 64 / l lanes each;
//   - warps 4 and 5 are the helpers: while the others evaluate proposal j,
//     each prepares proposal j + 1 for one outcome of j (warp 4 rejected, warp
//     5 accepted): its target, and its border entries loaded into shared
//     memory.  Warp 4 also keeps the lists, the log and the counters, warp 5
//     forms 1/d of an acceptance;
//   - the four FP64 warps evaluate the decision, each for itself; warp 0 hands
//     it to the helpers (named barrier 1).
// The border of B = I + (I - G) diag(a) against the accepted set P is taken as
// raw entries x of N, X and the candidate columns.  With e = e^{V_t}, the
// removal of t (a = 1/e - 1), its flip (a = 1/e^2 - 1) and an insertion
// (a = e - 1) have
//   column  B[P_p, t] = c x(P_p, t),   diagonal  B[t, t] = k0 + c x(t, t),
//   row     B[t, P_p] = r_p x(t, P_p), r_p the c of P_p when it was accepted,
//   c, k0 = 1, 0 (removal: x = N);  1 + 1/e, -1/e (flip: x = N);
//           1 - e, e (insertion: x = G_ext),
// from G = (N e - I)/(e - 1) on existing columns.  So
//   d = B_tt - row B^-1 col = k0 + c (x_tt - sum_pq r_p x_tp B^-1_pq x_qt)
// needs one sum over p and q (no separate t = B^-1 col), c once.  An entry of
// P whose total change became zero has r_p = 0, and a later proposal on that
// same existing row has x(t, t) - 1/e in its column entry.
//
// Per proposal (l accepted so far): 2 l^2 / 128 multiply-adds per lane and a
// five-step shuffle sum, barrier, decision; an acceptance adds s = row B^-1,
// 1/d and the rank-1 update with one barrier, and one of the FP64 warps alone
// (the helpers prepare meanwhile).  A window of 64 proposals, half of them
// accepted: one FP64 walker of order 311 138 us, one mixed walker of order 640
// 158 us.  With the border loaded by the FP64 warps behind a barrier of its own
// and one planner warp for both outcomes it took 176 and 184 us; the border
// loads have to start together and land across the barrier (loaded one after
// the other inside the evaluation: 200 us).
#include <cstdint>
#include <type_traits>

#include "device_util.cuh"
#include "ext_view.cuh"
#include "kernels.h"
#include "state.h"

namespace dca {

namespace {

constexpr int MW = 4;                     // FP64 warps
constexpr int MTHREADS = 32 * (MW + 2);   // and the helpers
constexpr unsigned FULL = 0xffffffffu;

// Kinds of a planned proposal: 0 insert, 1 remove, 3 flip, 2 rejected without
// a ratio, 4 / 5 remove / flip a vertex inserted in this window, 6 / 7 remove
// / flip one flipped in it, -1 end of the window.
struct Plan {
  int kind, target, rank, up, kcur, dupq, dupi, pad;
};

// FP64 value of an entry of N or X; FP32 is widened by integer operations
// (exact; a conversion would hold the FP64 unit).
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m == 0u) return __hiloint2double((int)u, 0);
  if (m < 0x00800000u || m >= 0x7f800000u) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
}

// Raw border entry x(x, y) of the extended matrix: N or X on existing columns
// (float or double), the candidate columns of G_ext elsewhere.  The address is
// selected first, so that the loads of several entries are in flight together.
template <typename T>
__device__ __forceinline__ const T* raw_ptr(const ExtView<T>& v, int x, int y) {
  return (x < v.n ? v.N + (size_t)x * v.ld : v.X + (size_t)(x - v.n) * v.ld) + y;
}

// Named barriers: 1 hands the decision from warp 0 to the two helpers, 2 the
// border entries of the next proposal from the helpers to the FP64 warps (and
// joins those after the update of B^-1).
__device__ __forceinline__ void bar_arrive_decision() { asm volatile("bar.arrive 1, 96;" ::: "memory"); }
__device__ __forceinline__ void bar_sync_decision() { asm volatile("bar.sync 1, 96;" ::: "memory"); }
__device__ __forceinline__ void bar_arrive_border() { asm volatile("bar.arrive 2, 192;" ::: "memory"); }
__device__ __forceinline__ void bar_sync_border() { asm volatile("bar.sync 2, 192;" ::: "memory"); }

// border entries in flight per lane: 8 of P a round and spin, side
constexpr int BORDER_ROUND = 5;

__device__ __forceinline__ double shfl_xor_d(double a, int o) { return __shfl_xor_sync(FULL, a, o); }

// Lanes per row of B^-1 (64 threads per spin): l G <= 64, at most 8.
__device__ __forceinline__ int lanes_log2(int l) { return l <= 8 ? 3 : (l <= 16 ? 2 : (l <= 32 ? 1 : 0)); }

}  // namespace

template <typename T>
__global__ void __launch_bounds__(MTHREADS) k_metropolis64(Config cfg) {
  WalkerDev& w = cfg.W[blockIdx.x];
  if (!w.active) return;
  const ProblemDev& pb = cfg.P[w.problem];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool helper = warp >= MW, keeper = warp == MW;  // keeper: lists, log and counters
  const int n = w.n, n_live = w.n_live, len = w.win_len;
  // the spin whose entries this thread reads: its warp's, or by lane in the helpers
  const int vsp = helper ? (lane >> 1) & 1 : warp >> 1;
  const ExtView<T> ev = make_view<T>(w, vsp);
  // B^-1 of both spins: in shared memory for k_s <= METRO_SMEM_KS (odd row
  // stride: row-wise reads without bank conflicts), else in the global buffers
  extern __shared__ double s_binv[];
  const bool in_smem = cfg.ks <= METRO_SMEM_KS;
  const int bst = in_smem ? (cfg.ks | 1) : KS_MAX;
  double* const B0 = in_smem ? s_binv : w.Binv[0];
  double* const B1 = in_smem ? s_binv + (size_t)cfg.ks * bst : w.Binv[1];

  __shared__ double s_u[KS_MAX];                  // Metropolis uniforms
  __shared__ int s_type[KS_MAX], s_slot[KS_MAX];  // proposal kind; slot of an insertion, index word otherwise
  __shared__ uint8_t s_up[KS_MAX], s_forced[KS_MAX];
  __shared__ int s_live[METRO_LIVE];              // 2 row + (s > 0) of the live vertex of each rank
  __shared__ double s_row[2][KS_MAX], s_t[2][KS_MAX], s_r[2][KS_MAX], s_aP[2][KS_MAX];
  // raw border entries [parity of the proposal][outcome of the one before][spin]; the diagonal entry at p = KS_MAX
  __shared__ double s_xr[2][2][2][KS_MAX], s_xc[2][2][2][KS_MAX + 1];
  __shared__ double s_quo[2][2 * KS_MAX + 2];     // K/(k+1) and k/K for k = k0 + index, k0 = max(n_live - len, 0)
  __shared__ double s_c[4][2][2], s_k0[4][2][2];  // c and k0: [kind][spin][s > 0]
  __shared__ double s_a[4][2][2], s_ie[2][2];     // a_t; e^{-V}
  __shared__ double s_part[2][MW], s_f[2], s_cf[2], s_coef[2], s_d[2], s_R;
  __shared__ Plan s_plan[2][2];                   // [parity of the proposal][outcome of the one before]
  __shared__ int s_P[KS_MAX], s_Pup[KS_MAX], s_gone[KS_MAX];
  __shared__ int s_removed[KS_MAX + 1], s_flipped[KS_MAX], s_flip_p[KS_MAX], s_ins_p[KS_MAX];
  __shared__ int s_dec, s_acc[2], s_end[5];       // outcomes; l, removals, insertions, flips, evaluated
  __shared__ double s_sign;

  const uint64_t q0 = w.q;
  const int64_t forced_n = w.forced_n, log_cap = w.log_cap;
  const int k0 = n_live > len ? n_live - len : 0;
  for (int j = tid; j < len; j += MTHREADS) {
    const Proposal& pr = w.prop[j];
    s_u[j] = pr.u;
    s_type[j] = pr.type;
    s_slot[j] = pr.type == 0 ? pr.slot : (int)pr.word;
    s_up[j] = pr.s > 0;
    const uint64_t q = q0 + (uint64_t)j;
    s_forced[j] = (int64_t)q < forced_n ? (uint8_t)(w.forced[q] & 1) : (uint8_t)2;
  }
  const bool live_smem = n_live <= METRO_LIVE;
  if (live_smem)
    for (int r = tid; r < n_live; r += MTHREADS) {
      const int x = w.live_idx[r];
      s_live[r] = 2 * x + (ev.vs[x] > 0 ? 1 : 0);
    }
  {
    const double K = pb.K;
    const int m = n_live + len - k0 + 1;  // <= 2 len + 1
    for (int i = tid; i < 2 * m; i += MTHREADS) {
      const int side = i >= m ? 1 : 0, k = k0 + i - side * m;
      s_quo[side][i - side * m] = (side ? (double)k : K) / (side ? K : (double)(k + 1));
    }
  }
  if (keeper && lane < 4) {
    const int sp = lane >> 1, up = lane & 1;
    const double e = pb.expV[sp][up], ie = pb.expV[sp][up ^ 1];
    s_ie[sp][up] = ie;
    s_a[0][sp][up] = e - 1.0;
    s_c[0][sp][up] = 1.0 - e;
    s_k0[0][sp][up] = e;
    s_a[1][sp][up] = ie - 1.0;
    s_c[1][sp][up] = 1.0;
    s_k0[1][sp][up] = 0.0;
    s_a[3][sp][up] = ie * ie - 1.0;
    s_c[3][sp][up] = 1.0 + ie;
    s_k0[3][sp][up] = -ie;
  }
  // the helpers' view of the chain state (uniform over their lanes)
  int nrem = 0, nins = 0, nflip = 0, n_eval = 0;
  int64_t c_acc = 0, c_ties = 0, c_negl = 0;
  double sign = w.sign;
  __syncthreads();

  // Plan of proposal j, the same in every lane of the calling warp.  cur, l: the
  // proposal before it is taken as accepted (as position l of P) when cur is
  // not null.
  auto plan = [&](int j, const Plan* cur, int l) -> Plan {
    Plan p{-1, -1, -1, 0, 0, -1, 0, 0};
    if (j >= len) return p;
    const int ck = cur ? cur->kind : -1;
    const int nold = n_live - nrem - (ck == 1 ? 1 : 0);
    p.kcur = nold + nins + (ck == 0 ? 1 : 0);
    if (s_type[j] == 0) {
      p.kind = 0;
      p.target = n + s_slot[j];
      p.up = s_up[j];
      return p;
    }
    if (p.kcur == 0) {
      p.kind = 2;
      return p;
    }
    const int idx = (int)scaled_index((uint32_t)s_slot[j], (uint32_t)p.kcur);
    const bool ins = idx >= nold;  // a vertex inserted in this window
    bool dup = ins;
    if (ins) {
      p.dupi = idx - nold;
      p.dupq = p.dupi < nins ? s_ins_p[p.dupi] : l;
    } else {
      // rank of the idx-th live vertex not removed yet: idx + r*, r* the number
      // of r with s_removed[r] - r <= idx (ascending and distinct); one more
      // removed rank at or below it moves on to the next one
      int want = idx;
      for (int pass = 0; pass < 2; ++pass) {
        int lo = 0;
        for (int b = 0; b < nrem; b += 32)
          lo += __popc(__ballot_sync(FULL, b + lane < nrem && s_removed[b + lane] - (b + lane) <= want));
        p.rank = want + lo;
        if (ck != 1 || cur->rank > p.rank || pass == 1) break;
        want = idx + 1;
      }
      for (int b = 0; b < nflip; b += 32) {
        const unsigned m = __ballot_sync(FULL, b + lane < nflip && s_flipped[b + lane] == p.rank);
        if (m) {
          dup = true;
          p.dupi = b + __ffs(m) - 1;
          p.dupq = s_flip_p[p.dupi];
        }
      }
      if (ck == 3 && cur->rank == p.rank) {
        dup = true;
        p.dupq = l;
        p.dupi = nflip;
      }
    }
    const bool flip = s_type[j] == 2;
    if (dup) {
      if (cfg.dup_rule == 1) {
        p.kind = 2;  // neglect rule: rejected
      } else if (cfg.dup_rule == 2) {
        p.kind = (ins ? 4 : 6) + (flip ? 1 : 0);
        p.target = p.dupq == l && cur ? cur->target : s_P[p.dupq];
        p.up = p.dupq == l && cur ? cur->up : s_Pup[p.dupq];
      }  // abort rule: the window ends here
      return p;
    }
    p.kind = flip ? 3 : 1;
    if (live_smem) {
      const int v = s_live[p.rank];
      p.target = v >> 1;
      p.up = v & 1;
    } else {
      p.target = w.live_idx[p.rank];
      p.up = ev.vs[p.target] > 0 ? 1 : 0;
    }
    return p;
  };
  // A helper warp prepares proposal j: its plan for outcome `out` of the
  // proposal before it (cur: accepted as position l) and its border entries
  // against P, each lane one spin and side.  prepare() starts the loads of the
  // first round (40 entries of P) and leaves them in flight; land() writes them
  // to shared memory.
  Plan np{-1, -1, -1, 0, 0, -1, 0, 0};  // the plan in flight
  T bx[BORDER_ROUND];
  double bg[BORDER_ROUND];
  int bP[BORDER_ROUND];
  const bool col = lane & 1;
  auto load_round = [&](int b, const Plan* cur, int l) {
    const int m = l + (cur ? 1 : 0), t = np.target;
#pragma unroll
    for (int u = 0; u < BORDER_ROUND; ++u) {
      const int q = b + 8 * u;  // q = m: the diagonal entry
      bP[u] = q < l ? s_P[q] : (q < m ? cur->target : t);
    }
#pragma unroll
    for (int u = 0; u < BORDER_ROUND; ++u) {
      const int q = b + 8 * u, x = col ? bP[u] : t, y = col ? t : bP[u];
      const bool want = q < m || (q == m && col);
      bx[u] = (T)0;
      bg[u] = 0.0;
      if (want && y < n) bx[u] = __ldg(raw_ptr(ev, x, y));
      if (want && y >= n) bg[u] = __ldg(ev.Gc + (size_t)(y - n) * ev.ld + x);
    }
  };
  auto store_round = [&](int b, int par, int out, const Plan* cur, int l) {
    const int m = l + (cur ? 1 : 0), t = np.target;
    double* const dst = col ? s_xc[par][out][vsp] : s_xr[par][out][vsp];
#pragma unroll
    for (int u = 0; u < BORDER_ROUND; ++u) {
      const int q = b + 8 * u;
      const bool cand = (col ? t : bP[u]) >= n;
      double v = cand ? bg[u] : widen(bx[u]);
      if (q < m) {
        if (col && bP[u] == t) v -= s_ie[vsp][np.up];
        dst[q] = v;
      } else if (q == m && col) {
        dst[KS_MAX] = v;
      }
    }
  };
  auto normal = [](int kind) { return kind == 0 || kind == 1 || kind == 3; };
  auto prepare = [&](int j, int out, const Plan* cur, int l) {
    np = plan(j, cur, l);
    if (lane == 0) s_plan[j & 1][out] = np;
    if (!normal(np.kind)) return;
    const int m = l + (cur ? 1 : 0);
    for (int b = (lane >> 2) + 8 * BORDER_ROUND; b <= m; b += 8 * BORDER_ROUND) {
      load_round(b, cur, l);
      store_round(b, j & 1, out, cur, l);
    }
    load_round(lane >> 2, cur, l);
  };
  auto land = [&](int j, int out, const Plan* cur, int l) {
    if (normal(np.kind)) store_round(lane >> 2, j & 1, out, cur, l);
  };
  // Sorted insertion of a rank into the removed ranks (the keeper; both helpers count it).
  auto add_removed = [&](int rank) {
    int pos = 0;
    for (int b = (nrem - 1) & ~31; b >= 0; b -= 32) {
      const int i = b + lane;
      const int v = i < nrem ? s_removed[i] : 0x7fffffff;
      __syncwarp();
      if (i < nrem && v > rank) s_removed[i + 1] = v;
      pos += __popc(__ballot_sync(FULL, v < rank));
      __syncwarp();
    }
    if (lane == 0) s_removed[pos] = rank;
    __syncwarp();
  };
  // Log and counters of a decided proposal (the keeper).
  auto decided = [&](int j, bool acc, double R) {
    const uint64_t q = q0 + (uint64_t)j;
    const int tie = fabs(fabs(R) - s_u[j]) < cfg.tie_eps ? 1 : 0;
    if (lane == 0 && (int64_t)q < log_cap) w.log[q] = (uint8_t)((acc ? 1 : 0) | (tie << 1));
    if (acc && R < 0.0) sign = -sign;
    n_eval = j + 1;
    c_ties += tie;
    c_acc += acc ? 1 : 0;
  };
  // An accepted second change of a spin, in the helpers' counts.
  auto second_change = [&](int kind) {
    if (kind == 4) --nins;
    if (kind >= 6) --nflip;
    if (kind == 6) ++nrem;
  };
  if (keeper) {
    prepare(0, 0, nullptr, 0);
    land(0, 0, nullptr, 0);
  }
  __syncthreads();

  int l = 0, sel = 0;
  for (int j = 0;; ++j) {
    const int par = j & 1;
    const Plan pl = s_plan[par][sel];  // a copy: the buffer is written again while a decision is still taken
    const int kind = pl.kind;
    if (kind < 0) break;
    if (kind == 2) {
      // a removal or flip from the empty configuration (ratio zero), or a
      // proposal dropped by the neglect rule
      if (keeper) {
        const uint64_t q = q0 + (uint64_t)j;
        if (lane == 0 && (int64_t)q < log_cap) w.log[q] = 0;
        c_negl += pl.kcur > 0 ? 1 : 0;
        n_eval = j + 1;
        prepare(j + 1, 0, nullptr, l);
        land(j + 1, 0, nullptr, l);
      }
      __syncthreads();
      sel = 0;
      continue;
    }
    if (kind >= 4) {
      // A spin changed earlier in this window changes again: column q of B
      // changes by c (B e_q - e_q), c = (a' - a) / a, so det B'/det B =
      // 1 + c (1 - (B^-1)_qq) and, by Sherman-Morrison, B'^-1 = B^-1 -
      // (c / rho) (e_q - B^-1 e_q) e_q^T B^-1.  Exact: the chain of single-spin
      // updates without ending the window.
      __syncthreads();  // B^-1 is up to date (the helpers do not wait for its last update)
      const int qp = pl.dupq;
      if (keeper) {
        const int sp = lane & 1, up = pl.up;
        const double a = s_aP[sp][qp];
        const double an = kind == 4 || kind == 7 ? 0.0 : (kind == 5 ? s_a[0][sp][up ^ 1] : s_a[1][sp][up]);
        const double c = an == a ? 0.0 : (an - a) / a;  // a = 0 only where every factor is (U = 0): no change
        const double rho = 1.0 + c * (1.0 - (sp ? B1 : B0)[(size_t)qp * bst + qp]);
        const double other = shfl_xor_d(rho, 1);
        const double R = ((kind & 1) ? 1.0 : s_quo[1][pl.kcur - k0]) * (sp ? other : rho) * (sp ? rho : other);
        int acc = -1;
        if (isfinite(R)) {
          acc = s_forced[j] < 2 ? s_forced[j] : (s_u[j] < fabs(R) ? 1 : 0);
          decided(j, acc != 0, R);
        }
        if (acc > 0) {
          __syncwarp();
          if (lane < 2) {
            s_coef[sp] = -c / rho;
            s_aP[sp][qp] = an;
            s_r[sp][qp] = kind == 5 ? -an : (kind == 6 ? 1.0 : 0.0);
          }
          const int di = pl.dupi, rank = pl.rank;
          if (kind == 4) {  // the inserted vertex goes: later insertions move up one place
            if (lane == 0) {
              for (int r = di; r + 1 < nins; ++r) s_ins_p[r] = s_ins_p[r + 1];
              s_gone[qp] = 1;
            }
          } else if (kind == 5) {  // the inserted vertex keeps its place with the other spin
            if (lane == 0) s_Pup[qp] ^= 1;
          } else {  // no longer a flipped vertex
            if (lane == 0)
              for (int r = di; r + 1 < nflip; ++r) {
                s_flipped[r] = s_flipped[r + 1];
                s_flip_p[r] = s_flip_p[r + 1];
              }
            if (kind == 6) add_removed(rank);
          }
          __syncwarp();
          second_change(kind);
        }
        if (lane == 0) s_acc[par] = acc;
        if (acc >= 0) {
          prepare(j + 1, 0, nullptr, l);
          land(j + 1, 0, nullptr, l);
        }
      }
      __syncthreads();
      const int acc = s_acc[par];
      sel = 0;
      if (helper && !keeper && acc > 0) second_change(kind);
      if (acc < 0) {
        if (tid == 0) set_status(w, ST_ERR_NUMERIC);
        break;
      }
      if (!acc) continue;
      for (int i = tid; i < 2 * l; i += MTHREADS) {
        const int sp = i >= l ? 1 : 0, p = i - sp * l;
        const double* B = sp ? B1 : B0;
        s_t[sp][p] = s_coef[sp] * ((p == qp ? 1.0 : 0.0) - B[(size_t)p * bst + qp]);
        s_row[sp][p] = B[(size_t)qp * bst + p];
      }
      __syncthreads();
      for (int i = tid; i < 2 * l * l; i += MTHREADS) {
        const int sp = i >= l * l ? 1 : 0, r = i - sp * l * l, p = r / l, c = r - p * l;
        double* B = (sp ? B1 : B0) + (size_t)p * bst + c;
        *B = fma(s_t[sp][p], s_row[sp][c], *B);
      }
      __syncthreads();  // s_row is written again at the top
      continue;
    }

    // 1. partial sums of row B^-1 col: thread (p, g) of a spin's 64 sums the
    // columns q = g mod G of row p (rows p and p + 64 for l > 64)
    const int t = pl.target, up = pl.up;
    const int lg = lanes_log2(l), G = 1 << lg;
    const int sp = vsp, ti = tid & 63, p0 = ti >> lg, g = ti & (G - 1);
    double* const Bs = sp ? B1 : B0;
    double a0 = 0.0, a1 = 0.0;
    const int ds = lane & 1;  // decision: even lanes form d of spin up, odd of down
    double xtt = 0.0, c = 0.0, k0d = 0.0, quo = 0.0, uj = 0.0;
    int forced = 2;
    if (!helper) {
      const double* xc = s_xc[par][sel][sp];
      const double* xr = s_xr[par][sel][sp];
      double part = 0.0;
      if (l > 0) {
        if (p0 < l) {
          const double row = s_r[sp][p0] * xr[p0];
          if (g == 0) s_row[sp][p0] = row;
          const double* B = Bs + (size_t)p0 * bst;
#pragma unroll 4
          for (int q = g; q < l; q += G) a0 = fma(B[q], xc[q], a0);
          part = a0 * row;
        }
        if (l > 64 && p0 + 64 < l) {
          const double row = s_r[sp][p0 + 64] * xr[p0 + 64];
          s_row[sp][p0 + 64] = row;
          const double* B = Bs + (size_t)(p0 + 64) * bst;
          for (int q = 0; q < l; ++q) a1 = fma(B[q], xc[q], a1);
          part = fma(a1, row, part);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += shfl_xor_d(part, o);
      }
      if (lane == 0) s_part[par][warp] = part;
      // operands of the decision, before the barrier
      xtt = s_xc[par][sel][ds][KS_MAX];
      c = s_c[kind][ds][up];
      k0d = s_k0[kind][ds][up];
      quo = kind == 3 ? 1.0 : s_quo[kind][pl.kcur - k0];
      uj = s_u[j];
      forced = s_forced[j];
    } else {
      prepare(j + 1, warp - MW, keeper ? nullptr : &pl, l);
    }
    __syncthreads();
    // 2. the decision, by every FP64 thread
    int acc;
    if (!helper) {
      const double d = fma(c, xtt - (s_part[par][2 * ds] + s_part[par][2 * ds + 1]), k0d);
      const double dx = shfl_xor_d(d, 1);
      const double R = quo * (ds ? dx : d) * (ds ? d : dx);
      const int rhi = __double2hiint(R) & 0x7fffffff;
      // u and |R| are not negative: they order like their bits
      acc = forced < 2 ? forced
                       : (__double_as_longlong(uj) < (__double_as_longlong(R) & 0x7fffffffffffffffll) ? 1 : 0);
      if (rhi >= 0x7ff00000) acc = -1;  // not finite
      if (warp == 0) {
        if (lane < 2) s_d[lane] = d;
        if (lane == 0) {
          s_dec = acc;
          s_R = R;
        }
        __syncwarp();
        bar_arrive_decision();
      }
      if (acc <= 0) bar_sync_border();
    } else {
      land(j + 1, warp - MW, keeper ? nullptr : &pl, l);
      __syncwarp();
      bar_arrive_border();
      bar_sync_decision();
      acc = s_dec;
    }
    if (acc < 0) {
      if (tid == 0) set_status(w, ST_ERR_NUMERIC);
      break;
    }
    sel = acc;
    if (!acc) {
      if (keeper) decided(j, false, s_R);
      continue;
    }
    // 3. acceptance: t = B^-1 col (from step 1), s = row B^-1, 1/d
    double ssum[2] = {0.0, 0.0};
    if (helper) {
      if (keeper) {
        if (lane == 0) {
          s_P[l] = t;
          s_Pup[l] = up;
          s_gone[l] = 0;
          if (kind == 0) s_ins_p[nins] = l;
          if (kind == 3) {
            s_flip_p[nflip] = l;
            s_flipped[nflip] = pl.rank;
          }
        }
        if (kind == 1) add_removed(pl.rank);
        decided(j, true, s_R);
      } else if (lane < 2) {
        const double f = __drcp_rn(s_d[lane]), cl = s_c[kind][lane][up];
        s_f[lane] = f;
        s_cf[lane] = f * cl;
        s_r[lane][l] = cl;
        s_aP[lane][l] = s_a[kind][lane][up];
      }
      if (kind == 0) ++nins;
      else if (kind == 3) ++nflip;
      else ++nrem;
    } else if (l > 0) {
      if (p0 < l)
#pragma unroll 4
        for (int p = g; p < l; p += G) ssum[0] = fma(s_row[sp][p], Bs[(size_t)p * bst + p0], ssum[0]);
      if (p0 + 64 < l)
        for (int p = 0; p < l; ++p) ssum[1] = fma(s_row[sp][p], Bs[(size_t)p * bst + p0 + 64], ssum[1]);
      for (int o = G >> 1; o > 0; o >>= 1) {
        a0 += shfl_xor_d(a0, o);
        ssum[0] += shfl_xor_d(ssum[0], o);
      }
      if (p0 < l && g == 0) s_t[sp][p0] = a0;
      if (p0 + 64 < l) s_t[sp][p0 + 64] = a1;
    }
    __syncthreads();
    // 4. bordered inverse: [[B^-1 + t s c/d, -t c/d], [-s/d, 1/d]], thread (q, g)
    // the rows p = g mod G of column q, four rows' loads before their stores
    if (!helper) {
      double* B = Bs;
      const double f = s_f[sp], cf = s_cf[sp];
      for (int h = 0; h < 2; ++h) {
        const int q = p0 + 64 * h;
        if (q < l) {
          const double sc = cf * ssum[h];
          if (g == 0) {
            B[(size_t)l * bst + q] = -f * ssum[h];
            B[(size_t)q * bst + l] = -cf * s_t[sp][q];
          }
          for (int p = g; p < l; p += 4 * G) {
            double b[4], tt[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int r = min(p + u * G, l - 1);
              b[u] = B[(size_t)r * bst + q];
              tt[u] = s_t[sp][r];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (p + u * G < l) B[(size_t)(p + u * G) * bst + q] = fma(tt[u], sc, b[u]);
          }
        }
      }
      if (ti == 0) B[(size_t)l * bst + l] = f;
      bar_sync_border();  // B^-1 is up to date too; the helpers already prepare the proposal after the next
    }
    ++l;
  }
  __syncthreads();

  // Epilogue: B^-1 for the update kernels (FP64, or FP32 pairs on the mixed
  // path), the accepted set and the counters.
  if (keeper && lane == 0) {
    s_end[1] = nrem;
    s_end[2] = nins;
    s_end[3] = nflip;
    s_end[4] = n_eval;
    s_sign = sign;
  }
  constexpr bool to_pairs = sizeof(T) == 4;
  __syncthreads();
  const int e_rem = s_end[1], e_ins = s_end[2], e_flip = s_end[3];
  if (keeper) {
    if (lane == 0) {
      w.n_flipped = e_flip;
      w.n_neglected += c_negl;
      w.n_prop += n_eval;
      w.n_ties += c_ties;
      w.n_accept += c_acc;
      metro_finish(cfg, w, n_live, len, l, e_rem, e_ins, s_end[4], s_sign);
    }
    __syncwarp();
    // the surviving insertions in order: their slots and positions in P
    int m = 0;
    for (int b = 0; b < l; b += 32) {
      const int p = b + lane;
      const bool in = p < l && s_P[p] >= n && !s_gone[p];
      const unsigned mask = __ballot_sync(FULL, in);
      if (in) {
        const int at = m + __popc(mask & ((1u << lane) - 1u));
        w.acc_slot[at] = s_P[p] - n;
        w.acc_p[at] = p;
        w.vs[w.parity][s_P[p]] = s_Pup[p] ? 1 : -1;  // its spin (a flip in the window may have changed it)
      }
      m += __popc(mask);
    }
    for (int p = lane; p < l; p += 32) {
      w.P[p] = s_P[p];
      w.aP[0][p] = s_aP[0][p];
      w.aP[1][p] = s_aP[1][p];
    }
    for (int r = lane; r < e_rem; r += 32) w.removed[r] = s_removed[r];
    for (int r = lane; r < e_flip; r += 32) w.flipped[r] = s_flipped[r];
  } else if (!helper && (in_smem || to_pairs)) {
    for (int i = tid; i < 2 * l * l; i += 32 * MW) {
      const int sp = i >= l * l ? 1 : 0, r = i - sp * l * l, p = r / l, q = r - p * l;
      const double b = (sp ? B1 : B0)[(size_t)p * bst + q];
      if (to_pairs) reinterpret_cast<float2*>(w.Binv[sp])[(size_t)p * KS_MAX + q] = df_split(b);
      else w.Binv[sp][(size_t)p * KS_MAX + q] = b;
    }
  }
}

static int metro64_smem(int ks) { return ks <= METRO_SMEM_KS ? (int)sizeof(double) * 2 * ks * (ks | 1) : 0; }

cudaError_t setup_metropolis64() {
  const int sm = metro64_smem(METRO_SMEM_KS);
  cudaError_t e = cudaFuncSetAttribute(k_metropolis64<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_metropolis64<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  return e;
}

void launch_metropolis64(const Config& cfg, cudaStream_t st) {
  const int sm = metro64_smem(cfg.ks);
  if (cfg.prec == PREC_MIXED) k_metropolis64<float><<<cfg.n_walkers, MTHREADS, sm, st>>>(cfg);
  else k_metropolis64<double><<<cfg.n_walkers, MTHREADS, sm, st>>>(cfg);
}

}  // namespace dca
