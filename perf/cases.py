"""Performance cases of the CT-AUX walker library.

A pass runs sweeps of a batch of walkers and reads their accumulated Green's
functions back (the inner loop of a solver run), or one step of the outer DCA
loop, or one standalone inverse.  Sizes are those of the named workloads in
paper_1901_01047_gb300/inputs.py and of the tests, or ranges around them.

The mixed-precision cases replay the decisions of an FP64 run of the same
chains for their first two passes (dca_walker_set_forced_decisions), so that
their outputs can be compared although the two precisions would part ways at
the first near-tie; later passes decide for themselves.  Results of the mixed
path are taken in the type of its N, FP32, and N is recomputed before every
measurement there (the mode whose G is within 1e-6 of FP64: without it the
drift of N between recomputes, not the code, decides the digits of G).
"""
import numpy as np
import torch

from paper_1901_01047_gb300 import inputs, walker

# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
_SWEEP = dict(kind="sweep", walkers=1, precision="fp64", tp=0.0, k_sub=64, sweeps=1, warmup=10, init=10, n_tau=4096,
              n_tau_meas=256, schedule="lockstep", recompute_every=64, recompute_sweeps=0, at_measure=False, n_omega=0,
              freq="nfft", n_w4=0, flips=0.0)


def _sweep(**kw):
    c = dict(_SWEEP)
    c.update(kw)
    return c


def listed():
    return [
        # the Hubbard atom: orders near 5, every launch latency bound
        _sweep(name="atom_fp64", nc=1, U_lo=4.0, U_hi=4.0, beta_lo=2.0, beta_hi=2.0, k_sub=8, sweeps=4, warmup=20),
        # 2x2 cluster, one chain in FP64: the run that is checked against exact diagonalisation
        _sweep(name="cluster4_fp64", nc=4, U_lo=4.0, U_hi=4.0, beta_lo=10.0, beta_hi=10.0, k_sub=32, sweeps=4,
               warmup=20),
        # the same cluster as a batch of short chains, with flips and M(i w_n) measured
        _sweep(name="cluster4_fp64_batch", nc=4, U_lo=4.0, U_hi=4.0, beta_lo=4.0, beta_hi=10.0, walkers=48, k_sub=32,
               sweeps=2, n_omega=64, flips=0.25, n_tau=2048, n_tau_meas=128),
        # 16 sites in FP64, one chain of order 300
        _sweep(name="cluster16_fp64", nc=16, tp=-0.15, U_lo=6.0, U_hi=6.0, beta_lo=8.0, beta_hi=8.0, init=100,
               warmup=24),
        # 16 sites, mixed precision, one chain of order 600, N recomputed every 8 windows too
        _sweep(name="cluster16_mixed", nc=16, tp=-0.15, U_lo=6.0, U_hi=6.0, beta_lo=16.0, beta_hi=16.0, init=250,
               precision="mixed", warmup=24, recompute_every=8, at_measure=True),
        # 256 uneven walkers sharing the sweep budget: the production batch (orders 90 to 900)
        _sweep(name="batch256", nc=0, U_lo=4.0, U_hi=7.0, beta_lo=5.0, beta_hi=25.0, walkers=256, precision="mixed",
               schedule="pooled", init=35, warmup=28, recompute_every=0, recompute_sweeps=8, n_tau=2048,
               n_tau_meas=128, at_measure=True),
        # a small batch under the lockstep schedule
        _sweep(name="batch24_lockstep", nc=8, U_lo=4.0, U_hi=7.0, beta_lo=5.0, beta_hi=12.0, walkers=24,
               precision="mixed", init=35, warmup=28, recompute_every=0, recompute_sweeps=8, at_measure=True,
               n_tau=2048, n_tau_meas=128),
        # M(i w_n) by the delayed NFFT beside G(tau)
        _sweep(name="batch64_nfft", nc=0, U_lo=4.0, U_hi=7.0, beta_lo=5.0, beta_hi=25.0, walkers=64, precision="mixed",
               schedule="pooled", sweeps=2, init=35, warmup=28, recompute_every=0, recompute_sweeps=8, n_tau=2048,
               n_tau_meas=128, n_omega=128, at_measure=True),
        # the two-particle function beside G(tau)
        _sweep(name="batch32_two_particle", nc=8, U_lo=4.0, U_hi=7.0, beta_lo=5.0, beta_hi=20.0, walkers=32,
               precision="mixed", schedule="pooled", sweeps=2, init=35, warmup=28, recompute_every=0,
               recompute_sweeps=8, n_tau=2048, n_tau_meas=128, n_w4=8, at_measure=True),
        # 36 sites: orders near 900 and a fine tau grid
        _sweep(name="cluster36_mixed", nc=36, U_lo=7.0, U_hi=7.0, beta_lo=8.0, beta_hi=8.0, walkers=4,
               precision="mixed", init=400, warmup=20, recompute_every=8, at_measure=True, n_tau_meas=2048),
        # one iteration of the outer loop: new self-energy, coarse-graining, new G0 table
        dict(kind="loop", name="outer_loop16", nc=16, beta=15.0, U=5.5, n_omega=128, n_fine=32, n_sets=64, n_tau=2048),
        # N of a stored configuration from scratch
        dict(kind="fresh", name="fresh500", nc=16, beta=20.0, U=6.0, n=500, n_tau=4096),
    ]


def _log_uniform(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    """One more case of the same ranges, costing no more than the largest above."""
    what = rng.choice(["small", "batch4", "one16", "mixed16", "batch", "batch", "lockstep", "nfft", "g4", "large",
                       "loop", "fresh"])
    U = round(rng.uniform(4.0, 7.0), 3)
    if what == "small":
        nc = rng.choice([1, 4])
        b = round(rng.uniform(2.0, 10.0), 3)
        return _sweep(nc=nc, U_lo=U, U_hi=U, beta_lo=b, beta_hi=b, k_sub=rng.choice([8, 16, 32]),
                      sweeps=rng.randint(2, 8), warmup=rng.randint(15, 25), n_tau_meas=rng.choice([64, 100, 256]))
    if what == "batch4":
        return _sweep(nc=4, U_lo=4.0, U_hi=U, beta_lo=3.0, beta_hi=round(rng.uniform(5.0, 10.0), 3),
                      walkers=rng.randint(5, 48), k_sub=rng.choice([16, 32]), sweeps=rng.randint(1, 3),
                      n_omega=rng.choice([0, 33, 64]), flips=rng.choice([0.0, 0.25]), n_tau=2048, n_tau_meas=128)
    if what == "one16":
        b = round(rng.uniform(4.0, 8.0), 3)
        return _sweep(nc=rng.choice([8, 16]), tp=-0.15, U_lo=U, U_hi=U, beta_lo=b, beta_hi=b, init=30, warmup=24,
                      k_sub=rng.choice([32, 64]))
    if what == "mixed16":
        b = round(rng.uniform(5.0, 12.0), 3)
        return _sweep(nc=16, tp=-0.15, U_lo=min(U, 6.0), U_hi=min(U, 6.0), beta_lo=b, beta_hi=b, init=int(15 * b),
                      precision="mixed", warmup=24, k_sub=rng.choice([48, 64]), recompute_every=8, at_measure=True)
    if what == "lockstep":
        return _sweep(nc=rng.choice([4, 8]), U_lo=4.0, U_hi=U, beta_lo=4.0, beta_hi=round(rng.uniform(6.0, 12.0), 3),
                      walkers=rng.randint(8, 24), precision="mixed", init=12, warmup=28, recompute_every=0,
                      recompute_sweeps=8, at_measure=True, n_tau=2048, n_tau_meas=rng.choice([64, 100, 128]))
    if what in ("batch", "nfft", "g4"):
        c = _sweep(nc=rng.choice([0, 8]), U_lo=4.0, U_hi=7.0, beta_lo=5.0, beta_hi=round(rng.uniform(10.0, 25.0), 3),
                   walkers=int(_log_uniform(rng, 12, 160 if what == "batch" else 48)), precision="mixed",
                   schedule="pooled", init=35, warmup=28, recompute_every=0, recompute_sweeps=8, n_tau=2048,
                   n_tau_meas=128, k_sub=rng.choice([48, 64, 64, 96]), at_measure=True)
        if what == "nfft":
            c.update(n_omega=rng.choice([50, 64, 128]), freq=rng.choice(["nfft", "dft"]))
        if what == "g4":
            c.update(nc=rng.choice([4, 8]), init=15, walkers=min(c["walkers"], 32), n_w4=rng.choice([4, 5, 8]))
        return c
    if what == "large":
        b = round(rng.uniform(3.0, 8.0), 3)
        return _sweep(nc=36, U_lo=U, U_hi=U, beta_lo=b, beta_hi=b, walkers=rng.randint(1, 4), precision="mixed",
                      init=int(30 * b), warmup=24, recompute_every=8, at_measure=True,
                      n_tau_meas=rng.choice([512, 1000, 2048]))
    if what == "loop":
        return dict(kind="loop", nc=rng.choice([4, 8, 16]), beta=round(rng.uniform(5.0, 25.0), 3), U=U,
                    n_omega=rng.choice([50, 64, 128]), n_fine=rng.randint(8, 32), n_sets=rng.randint(1, 64),
                    n_tau=rng.choice([1000, 2048]))
    return dict(kind="fresh", nc=rng.choice([4, 8, 16]), beta=round(rng.uniform(5.0, 20.0), 3), U=U,
                n=int(_log_uniform(rng, 20, 500)), n_tau=rng.choice([2048, 4096]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _bath(nc, tp, U, beta, n_tau):
    """A problem with the bath of the isolated cluster at half filling (mu = U/2)."""
    c = inputs.cluster(nc)
    kr = inputs.k_dot_r(c)
    eps = inputs.square_dispersion(c.kpts, 1.0 if nc > 1 else 0.0, tp)
    G0 = walker.g0_isolated_cluster(eps, kr, U / 2, U, beta, n_tau)
    return dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0, k_dot_r=kr, k_sub=c.k_sub)


def _problems(case):
    """(nc, U, beta) per walker: fixed by the case, uneven where it gives ranges (nc = 0: 8 and 16 in turn)."""
    if case["walkers"] == 1 or (case["U_lo"] == case["U_hi"] and case["beta_lo"] == case["beta_hi"]):
        return [(case["nc"], case["U_lo"], case["beta_lo"])]
    rng = np.random.default_rng(12345)
    out = []
    for w in range(case["walkers"]):
        beta = float(rng.uniform(case["beta_lo"], case["beta_hi"]))
        U = float(rng.uniform(case["U_lo"], case["U_hi"]))
        out.append((case["nc"] or (8, 16)[w % 2], U, beta))
    return out


def _order(nc, U, beta):
    """Mean expansion order, about 0.85 beta U nc / 2 + K."""
    return 0.85 * beta * U * nc / 2 + 1.0


def _chain_seed(seed):
    return (seed * 2654435761 + 97) % (1 << 62)


def prepare(case, seed):
    if case["kind"] == "loop":
        return _prepare_loop(case, seed)
    if case["kind"] == "fresh":
        return dict(case=case, problem=_bath(case["nc"], 0.0, case["U"], case["beta"], case["n_tau"]),
                    config=_config(case, seed))
    probs = [_bath(nc, case["tp"], U, beta, case["n_tau"]) for nc, U, beta in _problems(case)]
    common = dict(n_walkers=case["walkers"], k_sub=case["k_sub"], warmup_sweeps=case["warmup"],
                  n_tau_meas=case["n_tau_meas"], init_config_size=case["init"], seed=_chain_seed(seed),
                  schedule=case["schedule"], duplicate_rule="update", flip_fraction=case["flips"],
                  stream=torch.cuda.current_stream().cuda_stream)
    measured = dict(recompute_every=case["recompute_every"], recompute_sweeps=case["recompute_sweeps"],
                    recompute_at_measure=case["at_measure"], n_omega_meas=case["n_omega"], freq_method=case["freq"],
                    n_w4=case["n_w4"])
    logs = []
    if case["precision"] == "mixed":
        steps = case["warmup"] + 2 * case["sweeps"]
        cap = int(3.0 * (steps + 4) * max(_order(*p) for p in _problems(case))) + 4096
        with_log = walker.Walkers(probs, recompute_every=64, log_capacity=cap, **common)
        with_log.sweep(case["warmup"])
        with_log.sweep(case["sweeps"])
        with_log.sweep(case["sweeps"])
        logs = [with_log.decision_log(w) for w in range(case["walkers"])]
        with_log.close()
    gw = walker.Walkers(probs, precision=case["precision"], **measured, **common)
    for w, log in enumerate(logs):
        gw.set_forced_decisions(w, log)
    if logs:  # the random initial configurations are ill conditioned: N of the mixed path is kept fresh meanwhile
        gw.set_recompute(recompute_every=4)
    gw.sweep(case["warmup"])
    if logs:
        gw.set_recompute(case["recompute_every"], case["recompute_sweeps"], case["at_measure"])
    gw.reset_measurements()
    return dict(case=case, walkers=gw)


def run(state):
    case = state["case"]
    if case["kind"] == "loop":
        return _run_loop(state)
    if case["kind"] == "fresh":
        return walker.fresh_N(state["problem"], *state["config"])
    gw = state["walkers"]
    typ = np.float32 if case["precision"] == "mixed" else np.float64
    gw.sweep(case["sweeps"], sync=False)
    G, sign, count = gw.measure_G()
    out = {"G": _flat(G, typ), "sign": sign, "count": count}
    if case["n_omega"]:
        out["M"] = _flat(gw.measure_M()[0], np.complex64 if case["precision"] == "mixed" else np.complex128)
    if case["n_w4"]:
        acc = gw.measure_G4()[0]
        ctyp = np.complex64 if case["precision"] == "mixed" else np.complex128
        out["A"] = _flat([a for a, _ in acc], ctyp)
        out["D"] = _flat([d for _, d in acc], ctyp)
    return out


def _flat(arrays, typ):
    out = np.empty(sum(a.size for a in arrays), typ)
    at = 0
    for a in arrays:
        out[at:at + a.size] = a.reshape(-1)
        at += a.size
    return out


def work(case):
    if case["kind"] == "loop":
        nc, nw = case["nc"], case["n_omega"]
        return {"bytes": 16.0 * nc * nw * (2 * case["n_sets"] + 7) + 16.0 * nc * case["n_tau"],
                "flops": 20.0 * nc * nw * case["n_fine"] ** 2 + 16.0 * nc * nc * nw * case["n_sets"]
                + 4.0 * nc * case["n_tau"] * (nw + nc)}
    if case["kind"] == "fresh":
        n = case["n"]
        return {"bytes": 16.0 * n * n + 16.0 * case["nc"] * case["n_tau"], "flops": 4.0 * n ** 3}
    # per sweep of k proposals and spin: N read for the candidates, read and written by the update, once per window;
    # flops of the candidate products, the update (a quarter of the proposals accepted) and G(tau)
    probs = _problems(case)
    probs = [probs[w % len(probs)] for w in range(case["walkers"])]
    b = 4.0 if case["precision"] == "mixed" else 8.0
    nt, by, fl = case["n_tau_meas"], 0.0, 0.0
    for p in probs:
        k, nc = _order(*p), p[0]
        windows = max(1.0, k / case["k_sub"])
        by += case["sweeps"] * 2 * 3 * b * k * k * windows + 16.0 * nc * nt + 32.0 * nc * case["n_omega"]
        fl += case["sweeps"] * 2 * (2.0 * k ** 3 + 0.5 * k ** 3 + 2.0 * nc * k * (k + nc * nt))
        if case["at_measure"]:
            fl += case["sweeps"] * 8.0 * k ** 3
        if case["n_w4"]:
            S = 2.0 * nc * case["n_w4"]
            by += 16.0 * S * S
            fl += case["sweeps"] * 16.0 * (k * k * S + k * S * S)
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# The outer loop and the standalone inverse
# ---------------------------------------------------------------------------
def _loop_inputs(case, seed):
    rng = np.random.default_rng(seed)
    nc, nw, ns = case["nc"], case["n_omega"], case["n_sets"]
    wn = (2 * np.arange(nw) + 1) * np.pi / case["beta"]
    shape = 1.0 + 0.2 * rng.standard_normal((nc, 1))
    sigma = case["U"] / 2 + shape * case["U"] ** 2 / 4 / (1j * wn[None, :] + 0.3)
    counts = rng.integers(50, 200, ns).astype(np.float64)
    M = np.zeros((ns, 2, nc, nw), np.complex128)
    M[:, :, 0, :] = case["U"] ** 2 / 4 / (1j * wn + 0.5)
    M += 0.01 * (rng.standard_normal(M.shape) + 1j * rng.standard_normal(M.shape))
    return sigma, M * counts[:, None, None, None], counts


def _lattice(case):
    c = inputs.cluster(case["nc"])
    recip = 2.0 * np.pi * np.linalg.inv(np.array(c.vecs, np.float64)).T
    return c, inputs.k_dot_r(c), recip


def _prepare_loop(case, seed):
    c, kr, recip = _lattice(case)
    loop = walker.DCALoop(case["nc"], c.kpts, kr, recip, 1.0, 0.0, case["U"] / 2, case["U"], case["beta"],
                          case["n_fine"], case["n_omega"])
    sigma, M, counts = _loop_inputs(case, seed)
    g0s = loop.coarse_grain(sigma)[2]
    return dict(case=case, loop=loop, sigma=sigma, M=M, counts=counts, g0s=g0s)


def _run_loop(state):
    case, loop = state["case"], state["loop"]
    sigma = loop.sigma_update(state["g0s"], state["M"], state["counts"], state["sigma"], 0.7)
    gbar, g0, g0s, xi = loop.coarse_grain(sigma)
    table = loop.g0_table(g0s, xi, case["n_tau"])
    return {"sigma": sigma, "gbar": gbar, "g0": g0, "g0s": g0s, "xi": xi, "table": table}


def _config(case, seed):
    rng = np.random.default_rng(seed)
    n = case["n"]
    return (rng.integers(0, case["nc"], n).astype(np.int32), rng.random(n) * case["beta"],
            np.where(rng.random(n) < 0.5, 1, -1).astype(np.int32))


# ---------------------------------------------------------------------------
# The same results in plain 64-bit numpy
# ---------------------------------------------------------------------------
def exact(case, seed):
    if case["kind"] == "loop":
        return _exact_loop(case, seed)
    if case["kind"] == "fresh":
        nc, U, beta = case["nc"], case["U"], case["beta"]
        g0, sub = _table(nc, 0.0, U, beta, case["n_tau"])
        site, tau, s = _config(case, seed)
        mats, sign = [], 1.0
        for sp in (1, -1):
            A = _inverse_N(g0, sub, np.arccosh(1 + U * beta * nc / 2), beta, site, tau, s, sp)
            mats.append(np.linalg.inv(A))
            sign *= np.linalg.slogdet(A)[0]
        return mats[0], mats[1], None
    probs = _problems(case)
    probs = [probs[w % len(probs)] for w in range(case["walkers"])]
    cost = 0.0
    for p in probs:
        k = _order(*p)
        cost += (case["warmup"] + case["sweeps"]) * k * (1e-4 + 2e-9 * k * k) + case["n_omega"] * k * k * 4e-8
    if cost > 12.0 or case["n_w4"]:
        return None
    G, M, sign, count = [], [], [], []
    for w, (nc, U, beta) in enumerate(probs):
        g, m, sg = _chain(case, nc, U, beta, _chain_seed(seed), w)
        G.append(g)
        M.append(m)
        sign.append(sg)
    out = {"G": _flat(G, np.float64), "sign": np.array(sign, np.float64), "count": None}
    if case["n_omega"]:
        out["M"] = _flat(M, np.complex128)
    return out


def _table(nc, tp, U, beta, n_tau):
    """g0 = -G0(r, tau_l) of the isolated cluster (mu_eff = 0 at half filling) and the table of r_i - r_j."""
    c = inputs.cluster(nc)
    kx, ky = c.kpts[:, 0], c.kpts[:, 1]
    t = 1.0 if nc > 1 else 0.0
    xi = -2.0 * t * (np.cos(kx) + np.cos(ky)) - 4.0 * tp * np.cos(kx) * np.cos(ky)
    tau = np.arange(n_tau + 1) * (beta / n_tau)
    fk = np.exp(-tau[None, :] * xi[:, None] - np.logaddexp(0.0, -beta * xi)[:, None])
    phase = np.cos(c.kpts @ c.sites.T.astype(np.float64))
    return phase.T @ fk / nc, c.site_sub


def _interp(g0, d, beta, dt):
    """g0 at site differences d and times dt in (-beta, beta): linear, antiperiodic, 0 read as 0+."""
    n_tau = g0.shape[1] - 1
    sg = np.where(dt < 0, -1.0, 1.0)
    x = np.where(dt < 0, dt + beta, dt) * (n_tau / beta)
    i = np.clip(x.astype(np.int64), 0, n_tau - 1)
    a, b = g0[d, i], g0[d, i + 1]
    return sg * (a + (x - i) * (b - a))


def _inverse_N(g0, sub, gamma, beta, site, tau, s, sp):
    e = np.exp(sp * gamma * s)
    g = _interp(g0, sub[site[:, None], site[None, :]], beta, tau[:, None] - tau[None, :])
    return np.diag(e) - g * (e - 1.0)[None, :]


def _philox(c0, tag, key):
    """Philox4x32-10 blocks of counters (c0, tag) as uint64 arrays."""
    m32 = np.uint64(0xFFFFFFFF)
    v = [c0 & m32, c0 >> np.uint64(32), np.full_like(c0, tag), np.zeros_like(c0)]
    k = [int(key[0]), int(key[1])]
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * v[0], np.uint64(0xCD9E8D57) * v[2]
        v = [(p1 >> np.uint64(32)) ^ v[1] ^ np.uint64(k[0]), p1 & m32,
             (p0 >> np.uint64(32)) ^ v[3] ^ np.uint64(k[1]), p0 & m32]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    return v


def _u53(hi, lo):
    return ((hi << np.uint64(32) | lo) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _chain(case, nc, U, beta, seed, wi):
    """One chain by single-spin updates: (sum of sign G, sum of sign M, sum of signs) of the pass after the warm-up."""
    g0, sub = _table(nc, case["tp"], U, beta, case["n_tau"])
    gamma = np.arccosh(1.0 + U * beta * nc / 2)
    key = (seed & 0xFFFFFFFF, (seed >> 32) ^ wi)
    r = _philox(np.arange(case["init"], dtype=np.uint64), 2, key)
    site = ((r[1] * np.uint64(nc)) >> np.uint64(32)).astype(np.int64)
    tau = beta * _u53(r[2], r[3])
    s = np.where(r[0] & np.uint64(2), 1, -1)
    N = None
    sign, done = 1.0, 0

    def rebuild():
        return [np.linalg.inv(_inverse_N(g0, sub, gamma, beta, site, tau, s, sp)) for sp in (1, -1)]

    if case["init"]:
        for sp in (1, -1):
            sign *= np.linalg.slogdet(_inverse_N(g0, sub, gamma, beta, site, tau, s, sp))[0]
        N = rebuild()
    else:
        N = [np.zeros((0, 0)), np.zeros((0, 0))]
    words, have = None, 0

    def proposals(n):
        nonlocal words, have
        if done + n > have:
            have = done + n + 4096
            q = np.arange(done, have, dtype=np.uint64)
            words = (done, _philox(q, 0, key), _philox(q, 1, key))

    def remove(p):
        nonlocal site, tau, s
        for i in (0, 1):
            n = N[i]
            N[i] = np.delete(np.delete(n - np.outer(n[:, p], n[p, :]) / n[p, p], p, 0), p, 1)
        site, tau, s = np.delete(site, p), np.delete(tau, p), np.delete(s, p)

    def insertion(x, t, sx):
        """(ratio, parts) of an insertion at the end, per spin."""
        out = []
        for i, sp in enumerate((1, -1)):
            e = np.exp(sp * gamma * sx)
            col = -_interp(g0, sub[site, x], beta, tau - t) * (e - 1.0)
            row = -_interp(g0, sub[x, site], beta, t - tau) * (np.exp(sp * gamma * s) - 1.0)
            diag = e - g0[sub[x, x], 0] * (e - 1.0)
            nc_ = N[i] @ col
            out.append((diag - row @ nc_, nc_, row @ N[i]))
        return out

    def insert(x, t, sx, parts):
        nonlocal site, tau, s
        for i, (d, u, v) in enumerate(parts):
            n = N[i].shape[0]
            B = np.empty((n + 1, n + 1))
            B[:n, :n] = N[i] + np.outer(u, v) / d
            B[:n, n], B[n, :n], B[n, n] = -u / d, -v / d, 1.0 / d
            N[i] = B
        site, tau, s = np.append(site, x), np.append(tau, t), np.append(s, sx)

    thr = int(case["flips"] * 2 ** 30)
    wn = (2 * np.arange(case["n_omega"]) + 1) * np.pi / beta
    nt = case["n_tau_meas"]
    ta = (np.arange(nt) + 0.5) * beta / nt
    G, M, signs = np.zeros((2, nc, nt)), np.zeros((2, nc, wn.size), np.complex128), 0.0
    warm = []
    for sweep in range(case["warmup"] + case["sweeps"]):
        k = site.size
        if sweep < case["warmup"]:
            length = max(k, 1)
            warm.append(k)
        else:
            length = max(1, (2 * sum(warm) + len(warm)) // (2 * len(warm)))
        proposals(length)
        for _ in range(length):
            j = done - words[0]
            w0, w1, w2, w3 = (int(v[j]) for v in words[1])
            u = float(_u53(words[2][0][j:j + 1], words[2][1][j:j + 1])[0])
            done += 1
            k = site.size
            if not ((thr and (w0 >> 2) < thr) or w0 & 1):
                x, t = (w1 * nc) >> 32, beta * float(_u53(words[1][2][j:j + 1], words[1][3][j:j + 1])[0])
                sx = 1 if w0 & 2 else -1
                parts = insertion(x, t, sx)
                R = parts[0][0] * parts[1][0] / (k + 1)
                if u < abs(R):
                    insert(x, t, sx, parts)
                    sign = -sign if R < 0 else sign
            elif k:
                p = (w1 * k) >> 32
                if thr and (w0 >> 2) < thr:
                    # N^-1 column p changes by u = (I - g0)[:, p] (e' - e) with e = e^V; N^-1 N = 1 gives (I - g0) e_p
                    R, new = 1.0, []
                    for i, sp in enumerate((1, -1)):
                        e, en = np.exp(sp * gamma * s[p]), np.exp(-sp * gamma * s[p])
                        col = -_interp(g0, sub[site, site[p]], beta, tau - tau[p]) * (en - e)
                        col[p] += en - e
                        c = N[i] @ col
                        R *= 1.0 + c[p]
                        new.append(N[i] - np.outer(c, N[i][p, :]) / (1.0 + c[p]))
                    if u < abs(R):
                        N[:] = new
                        s = s.copy()
                        s[p] = -s[p]
                        sign = -sign if R < 0 else sign
                else:
                    R = N[0][p, p] * N[1][p, p] * k
                    if u < abs(R):
                        remove(p)
                        sign = -sign if R < 0 else sign
            if done % 64 == 0:
                N = rebuild()
        if sweep >= case["warmup"]:
            N = rebuild()
            signs += sign
            for i, sp in enumerate((1, -1)):
                f = np.exp(sp * gamma * s) - 1.0
                c = f[:, None] * N[i]
                gr = _interp(g0, sub[site, :], beta, np.broadcast_to(tau[:, None], (site.size, nc)))
                b = c @ gr
                for x in range(nc):
                    corr = _interp(g0, sub[x, site][None, :], beta, ta[:, None] - tau[None, :]) @ b
                    for rp in range(nc):
                        G[i, sub[x, rp]] -= sign * corr[:, rp] / nc
                for d in range(nc):
                    G[i, d] -= sign * _interp(g0, d, beta, ta)
                if wn.size:
                    ph = np.exp(1j * tau[:, None] * wn[None, :])
                    for d in range(nc):
                        pick = np.where(sub[site[:, None], site[None, :]] == d, c, 0.0)
                        M[i, d] += sign * np.sum(ph * (pick @ ph.conj()), 0) / (beta * nc)
    return G, M, signs


def _exact_loop(case, seed):
    c, kr, recip = _lattice(case)
    sigma0, Ms, counts = _loop_inputs(case, seed)
    nc, nw, beta, U, nf = case["nc"], case["n_omega"], case["beta"], case["U"], case["n_fine"]
    wn = (2 * np.arange(nw) + 1) * np.pi / beta
    x = (np.arange(nf) + 0.5) / nf - 0.5
    off = (x[:, None, None] * recip[0] + x[None, :, None] * recip[1]).reshape(-1, 2)
    k = c.kpts[:, None, :] + off[None]
    eps = -2.0 * (np.cos(k[..., 0]) + np.cos(k[..., 1]))

    def grain(sigma):
        z = 1j * wn + U / 2 - sigma
        gbar = np.stack([np.mean(1.0 / (z[K][:, None] - eps[K][None, :]), 1) for K in range(nc)])
        g0 = 1.0 / (1.0 / gbar + sigma)
        return gbar, g0, 1.0 / (1.0 / g0 - U / 2), eps.mean(1)

    g0s = grain(sigma0)[2]
    MK = np.einsum("kd,sdn->kn", np.exp(-1j * kr), Ms.sum(0)) / (2.0 * counts.sum())
    sigma = 0.7 * (1.0 / g0s + U / 2 - 1.0 / (g0s - g0s * g0s * MK)) + 0.3 * sigma0
    gbar, g0, g0s, xi = grain(sigma)
    tau = np.arange(case["n_tau"] + 1) * (beta / case["n_tau"])
    rest = g0s - 1.0 / (1j * wn[None, :] - xi[:, None])
    gk = (2.0 / beta) * np.real(rest @ np.exp(-1j * wn[:, None] * tau[None, :]))
    gk -= np.exp(-tau[None, :] * xi[:, None] - np.logaddexp(0.0, -beta * xi)[:, None])
    table = np.cos(kr).T @ gk / nc
    return {"sigma": sigma, "gbar": gbar, "g0": g0, "g0s": g0s, "xi": xi, "table": np.stack([table, table])}
