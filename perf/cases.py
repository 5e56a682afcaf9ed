"""The calls that users of the sampler make, at the sizes they make them, for timing.

Each case is one pass through the public binding: a sampling call (one launch and the histograms that
are read from it), a training round of the learned proposal, or a histogram of the caller's own data.
Models and sizes are those of the repository's workloads, tests and benchmark legs. A pass returns the
per-trajectory results (step counts, ln w, status), every histogram array and scalar, and for training
the updated parameters and Adam moments.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_13683_gb300 import fpt
from paper_2410_13683_gb300 import train as TR

NAN = float("nan")

# Potentials of the repository's workloads (dN = 1e-3 throughout).
EXP = dict(kind=fpt.FPT_POT_EXP, V0=1e-4, mu=0.01, phi_in=0.05, pi_in=-0.01, phi_end=0.0, dN=1e-3)
LINEAR = dict(kind=fpt.FPT_POT_PWLINEAR, V0=1e-4, a_plus=1e-2, a_minus=1e-2, phi_star=0.0, phi_in=0.05,
              pi_in=NAN, phi_end=0.0, dN=1e-3)
USR = dict(kind=fpt.FPT_POT_PWLINEAR, V0=2e-10, a_plus=1e-3, a_minus=1e-6, phi_star=1.0, bg_phi0=1.02,
           n_in=math.log(1.1), n_end=5.0, dN=1e-3)
BUMP = dict(kind=fpt.FPT_POT_BUMP, V0=7.76487e-11, bump_K=1.17e-3, bump_m=0.5, bump_width=1.59e-2,
            bump_phi0=2.18812, bg_phi0=2.6, n_in=1.2, n_end=5.2, dN=1e-3)
EXP_S = 1e-3                    # constant noise amplitude of the exponential model
AMPLITUDES = (0.5, 1.0, 2.0, 3.0, 4.0, 6.0, 8.0, 10.0)
N_12 = 152.5                    # e-folds where the sudden-transition tail is 1e-12

# Thread operations of one Euler-Maruyama step (noise, lookup, drift, update, passage test), counted in
# the source of the 1-D, full-rank and bump steppers.
OPS_1D, OPS_2D, OPS_BUMP = 60, 87, 66
# Operations of the 3 -> 64 -> 64 -> 2 network per state, forward, and forward with backward.
MLP_FWD, MLP_BWD = 8800, 26000


def listed():
    return [
        # First look at a model: a couple of thousand biased paths, a coarse histogram. Launch and latency.
        dict(name="quick_2k", kind="exp", n=2048, A=0.8, bins=32, max_steps=1 << 16),
        # The slow-roll check against the inverse-Gaussian law, at the size it is quoted on.
        dict(name="linear_16k", kind="linear", n=16384, A=0.0, bins=512, max_steps=1 << 16),
        # Direct sampling of the sudden transition: the plain method's production size.
        dict(name="usr_direct_4m", kind="usr", n=1 << 22, A=0.0, bins=512, max_steps=1 << 18),
        # The constant-bias sweep: eight amplitudes of uneven lengths in one launch, most paths capped.
        dict(name="usr_bias8", kind="bias", n=20011, runs=8, bins=512, max_steps=1 << 18),
        # The learned proposal as it is used for the far tail: long paths, a network every 128 steps.
        dict(name="usr_learned", kind="learned", n=1 << 18, alpha=0.45, segment=128, bins=512, max_steps=1 << 18),
        # Noise in global time, switched off after a window (the paper's production setting).
        dict(name="usr_window_1m", kind="window", n=1000003, A=1.0, bins=512, max_steps=1 << 18),
        # Full-rank noise from numerical matching.
        dict(name="usr_2d_1m", kind="noise2d", n=1 << 20, A=0.0, A2=0.0, bins=512, max_steps=1 << 18),
        # The smooth transition, biased into its upper tail (the sample of the eps2 fit).
        dict(name="bump_1m", kind="bump", n=1 << 20, A=2.0, bins=512, max_steps=1 << 18),
        # A sweep over 64 potentials in one launch, each with its own table and histogram.
        dict(name="family_64", kind="family", models=64, n=8192, A=0.5, points=256, bins=64, max_steps=1 << 17),
        # One training round of the learned proposal: paths with segment records, backward, Adam.
        dict(name="train_round", kind="train", n=1 << 15, alpha=0.45, segment=128, max_steps=1 << 18),
        # One training round of 64 proposals at once, a network per model.
        dict(name="train_batch_64", kind="batch", models=64, n=1024, alpha=0.2, segment=128, points=256,
             max_steps=1 << 17),
        # Histogram of a pooled job's own arrays, resident on the GPU.
        dict(name="hist_data_10m", kind="hist", n=10000019, bins=512),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["exp", "linear", "usr", "bias", "learned", "window", "noise2d", "bump", "family", "train",
                       "batch", "hist"])
    if kind == "exp":
        return dict(kind=kind, n=size(500, 60000), A=round(rng.uniform(0.0, 1.0), 3), bins=rng.randint(16, 128),
                    max_steps=1 << 16)
    if kind == "linear":
        return dict(kind=kind, n=size(2000, 500000), A=rng.choice([0.0, 0.5, -0.5]), bins=rng.randint(64, 1024),
                    max_steps=1 << 16)
    if kind == "usr":
        return dict(kind=kind, n=size(30000, 4000000), A=0.0, bins=rng.randint(64, 2048), max_steps=1 << 18)
    if kind == "bias":
        return dict(kind=kind, n=size(2000, 20000), runs=rng.randint(2, 8), bins=rng.randint(64, 1024),
                    max_steps=1 << 18)
    if kind == "learned":
        return dict(kind=kind, n=size(5000, 250000), alpha=round(rng.uniform(0.2, 0.45), 3),
                    segment=rng.choice([64, 128, 256]), bins=rng.randint(64, 1024), max_steps=1 << 18)
    if kind == "window":
        return dict(kind=kind, n=size(30000, 1000000), A=rng.choice([0.0, 0.5, 1.0]), bins=rng.randint(64, 1024),
                    max_steps=1 << 18)
    if kind == "noise2d":
        return dict(kind=kind, n=size(30000, 1000000), A=rng.choice([0.0, 0.2, 0.4]), A2=rng.choice([0.0, 0.3]),
                    bins=rng.randint(64, 1024), max_steps=1 << 17)
    if kind == "bump":
        return dict(kind=kind, n=size(30000, 1000000), A=rng.choice([0.0, 1.0, 2.0, 3.0]), bins=rng.randint(64, 1024),
                    max_steps=1 << 18)
    if kind == "family":
        return dict(kind=kind, models=rng.randint(2, 64), n=size(300, 8000), A=rng.choice([0.0, 0.25, 0.5]),
                    points=rng.choice([64, 128, 256]), bins=rng.randint(32, 256), max_steps=1 << 17)
    if kind == "train":
        return dict(kind=kind, n=size(1500, 32000), alpha=round(rng.uniform(0.1, 0.45), 3),
                    segment=rng.choice([64, 128]), max_steps=1 << 18)
    if kind == "batch":
        return dict(kind=kind, models=rng.randint(2, 64), n=size(100, 1000), alpha=round(rng.uniform(0.0, 0.2), 3),
                    segment=rng.choice([64, 128]), points=rng.choice([64, 256]), max_steps=1 << 17)
    return dict(kind=kind, n=size(20000, 10000000), bins=rng.randint(16, 4096))


# ---------------------------------------------------------------------------------------------------
def _family(count, max_steps):
    """The batched-sweep family: slopes, transition points and scales of each model."""
    rng = np.random.default_rng(5)
    a = 10.0 ** rng.uniform(-7.0, -4.0, 64)
    s = rng.uniform(0.9, 1.1, 64)
    v = 10.0 ** rng.uniform(-11.0, -9.0, 64)
    return [dict(USR, V0=float(v[i]), a_minus=float(a[i]), phi_star=float(s[i]), bg_phi0=float(s[i]) + 0.02,
                 max_steps=max_steps) for i in range(count)]


def _network(rng, alpha):
    """A proposal's weights: the initialisation of the tests, with outputs around a mean bias alpha as a
    trained network has (its own part of the bias is a fraction of the mean)."""
    H = 64
    return fpt.canonical_params(dict(
        W1=rng.normal(0.0, 1.0 / math.sqrt(3), (H, 3)), b1=np.zeros(H),
        W2=rng.normal(0.0, 1.0 / math.sqrt(H), (H, H)), b2=np.zeros(H),
        W3=rng.normal(0.0, 0.1 / math.sqrt(H), (2, H)), b3=np.array([alpha, 0.0])))


def _context(case, models, points=4096):
    ctx = fpt.fpt_init_model(models)
    k = case["kind"]
    for i in range(len(models)):
        if k == "exp":
            fpt.fpt_noise_table(ctx, i, fpt.FPT_TABLE_USER, 16, 1.0, -0.1, 0.2, np.full(16, EXP_S), np.zeros(16))
        elif k == "linear":
            fpt.fpt_noise_table(ctx, i, fpt.FPT_TABLE_DESITTER, points, 1.0, 0.0, 0.06)
        elif k == "window":
            fpt.fpt_noise_table(ctx, i, fpt.FPT_TABLE_BESSEL_N, points, 1.0, 0.0, USR["n_end"] - USR["n_in"])
        elif k == "noise2d":
            fpt.fpt_noise_table2(ctx, i, fpt.FPT_TABLE_NUMERIC, points, 1.0)
        else:
            fpt.fpt_noise_table(ctx, i, fpt.FPT_TABLE_BESSEL, points, 1.0)
    return ctx


def _proposals(ctx, case, rng, count):
    infos = [fpt.fpt_model_get_info(ctx, i) for i in range(count)]
    x_in = [f["phi_in"] - f["phi_end"] for f in infos]
    return TR.new_proposals(ctx, [_network(rng, case["alpha"]) for _ in range(count)],
                            [(math.log(x), 0.0, 0.0) for x in x_in],
                            [(0.2, 1.0 / abs(f["pi_in"]), 0.01) for f in infos], segment=case["segment"],
                            alpha_max=8.0, flags=fpt.FPT_MLP_LOG_X, x_floors=[x * 2.0 ** -14 for x in x_in])


def _hist_data(case, seed):
    """First-passage times with an exponential upper tail and the log-weights of a bias towards it."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["n"]
    N = 4.0 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64).log_().mul_(-8.0)
    lw = -0.25 * N + 0.5 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    status = (torch.rand(n, generator=g, device="cuda") < 1e-3).to(torch.uint8)
    return (N * 1e3).to(torch.int32), lw, status


HIST_RANGE = dict(N_lo=0.0, N_hi=64.0, N_tail=40.05)


def prepare(case, seed):
    k = case["kind"]
    rng = np.random.default_rng(seed)
    st = dict(case=case, seed=seed)
    if k == "hist":
        st["ctx"] = fpt.fpt_init_model([dict(EXP, max_steps=1 << 16)])
        st["data"] = _hist_data(case, seed)
        return st
    count = case.get("models", 1)
    base = {"exp": EXP, "linear": LINEAR, "bump": BUMP}.get(k, USR)
    models = _family(count, case["max_steps"]) if k in ("family", "batch") else [dict(base, max_steps=case["max_steps"])]
    ctx = st["ctx"] = _context(case, models, case.get("points", 4096))
    n = case["n"]
    if k in ("learned", "train", "batch"):
        props, P, B = _proposals(ctx, case, rng, count)
        st.update(props=props, P=P, B=B)
    if k in ("train", "batch"):
        # a training run in its third round: real Adam moments
        N_cut = 20.0
        if k == "train":
            TR.train(ctx, props[0], 0, rounds=2, n_traj=min(n, 2048), seed=seed, lam=0.25, N_cut=lambda r: N_cut, lr=3e-4)
            m, v = (x.reshape(1, -1) for x in props[0]._adam)
        else:
            TR.train_batch(ctx, props, P, B, list(range(count)), rounds=2, n_traj=min(n, 128), seed=seed, lam=0.25,
                           N_cuts=[N_cut] * count, lr=3e-4)
            m, v = P._adam
        torch.cuda.synchronize()
        st.update(N_cut=N_cut, live=(P, m, v, B), start=tuple(t.clone() for t in (P, m, v, B)),
                  runs=[props[i].desc(i, n, seed=seed, run_id=100 + i) for i in range(count)])
        return st
    if k == "learned":
        st["runs"] = [props[0].desc(0, n, seed=seed, run_id=0)]
    elif k == "bias":
        st["runs"] = [fpt.run_desc(0, n, seed=seed, run_id=r, A=A) for r, A in enumerate(AMPLITUDES[:case["runs"]])]
    else:
        st["runs"] = [fpt.run_desc(i, n, seed=seed, run_id=i, A=case["A"], A2=case.get("A2", 0.0)) for i in range(count)]
    total = n * len(st["runs"])
    st["out"] = dict(nsteps=torch.empty(total, dtype=torch.int32, device="cuda"),
                     logw=torch.empty(total, dtype=torch.float64, device="cuda"),
                     status=torch.empty(total, dtype=torch.uint8, device="cuda"))
    st["outs"] = [{f: t[r * n:(r + 1) * n] for f, t in st["out"].items()} for r in range(len(st["runs"]))]
    top = {"exp": 16.0, "linear": 8.0, "window": 16.0, "bump": 8.0, "usr": 30.0, "noise2d": 60.0, "family": 100.0}
    st["hist"] = dict(N_lo=0.0, N_hi=top.get(k, 400.0), n_bins=case["bins"],
                      N_tail=N_12 if k in ("bias", "learned") else NAN)
    return st


def _collect(hists):
    """The histograms of a call's runs, array by array."""
    keys = fpt.HIST_ARRAYS + fpt.HIST_SCALARS
    return {key: np.stack([np.asarray(h[key]) for h in hists]) for key in keys}


def run(st):
    case, ctx = st["case"], st["ctx"]
    k = case["kind"]
    if k == "hist":
        n, lw, status = st["data"]
        return fpt.fpt_histogram_data(ctx, n, lw, status, 1e-3, HIST_RANGE["N_lo"], HIST_RANGE["N_hi"], case["bins"],
                                      N_tail=HIST_RANGE["N_tail"])
    if k in ("train", "batch"):
        for live, start in zip(st["live"], st["start"]):
            live.copy_(start)
        P, m, v, B = st["live"]
        stream, adam = torch.cuda.current_stream(), dict(lr=3e-4, step=3)
        if k == "train":
            stats = [fpt.fpt_mlp_train_round(ctx, st["runs"][0], case["n"], 0.25, st["N_cut"], adam, P[0], m[0], v[0],
                                             B[0], stream=stream)]
        else:
            stats = fpt.fpt_mlp_train_batch(ctx, st["runs"], 0.25, [st["N_cut"]] * len(st["runs"]), adam, P, m, v, B,
                                            stream=stream)
        return dict(params=P, adam_m=m, adam_v=v, blob=B,
                    stats={key: np.array([s[key] for s in stats]) for key in stats[0]})
    fpt.fpt_run(ctx, st["runs"], st["outs"])
    hists = [fpt.fpt_histogram(ctx, r, **st["hist"]) for r in range(len(st["runs"]))]
    return dict(st["out"], hist=_collect(hists))


def _mean_steps(case):
    """Steps of a path on average (measured on the workloads; capped paths count the cap)."""
    k, cap = case["kind"], case.get("max_steps", 0)
    A = case.get("A", case.get("alpha", 0.0))
    if k == "exp":
        return min(cap, 50.0 / (0.01 - EXP_S * A))
    if k == "linear":
        return 5000.0
    if k in ("window", "bump"):
        return 5000.0 if k == "window" else 4300.0
    if k == "bias":
        r = case["runs"]
        return (60000.0 + (r - 1) * cap) / r
    # drift against noise in the sudden transition: lengths grow towards the cap as the bias does
    return min(0.8 * cap, 5000.0 * math.exp(5.0 * max(0.0, A)))


def work(case):
    k, n = case["kind"], case["n"]
    if k == "hist":
        return dict(bytes=13.0 * n + 8.0 * (10 * case["bins"] + 16), flops=12.0 * n)
    paths = n * case.get("models", 1) * case.get("runs", 1)
    steps = paths * _mean_steps(case)
    ops = {"noise2d": OPS_2D, "bump": OPS_BUMP}.get(k, OPS_1D)
    flops = steps * ops
    bytes_ = 13.0 * paths
    if k in ("learned", "train", "batch"):
        flops += steps / case["segment"] * MLP_FWD
    if k in ("train", "batch"):
        flops += steps / case["segment"] * MLP_BWD
        bytes_ += 2 * 32.0 * steps / case["segment"] + 4 * 4.0 * fpt.FPT_MLP_PARAMS * case.get("models", 1)
    else:
        bytes_ += 8.0 * 10 * case["bins"] * case.get("models", 1) * case.get("runs", 1)
    return dict(bytes=bytes_, flops=flops)


# ---------------------------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on arrays of counters."""
    M0, M1, mask = np.uint64(0xD2511F53), np.uint64(0xCD9E8D57), np.uint64(0xFFFFFFFF)
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    c = [np.asarray(x, np.uint64) for x in (c0, c1, c2, c3)]
    for _ in range(10):
        p0, p1 = M0 * c[0], M1 * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _normals(n, traj, seed):
    """The four normals of steps n .. n + 3."""
    c = _philox(np.full(traj.shape, n >> 2), traj, np.zeros_like(traj), np.zeros_like(traj), seed)
    u = [((x >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23 for x in c]
    z = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        rho = np.sqrt(-2.0 * np.log(a))
        z += [rho * np.cos(2.0 * np.pi * b), rho * np.sin(2.0 * np.pi * b)]
    return z


def _walk(case, seed):
    """Paths of the exponential or the linear model, stepped in 64 bits."""
    n, A, dN, cap = case["n"], case["A"], 1e-3, case["max_steps"]
    if case["kind"] == "exp":
        pi0, mu = -0.01, 0.01
        amp = lambda x: EXP_S
        vpv = lambda x: mu
    else:
        a, V0 = 1e-2, 1e-4
        pi0 = -a / (1.0 + a * 0.05)
        grid = np.linspace(0.0, 0.06, 4096)
        pa = a / (1.0 + a * grid)
        tab = np.sqrt(V0 * (1.0 + a * grid) / (3.0 - 0.5 * pa * pa)) / (2.0 * np.pi)
        amp = lambda x: np.interp(x, grid, tab)
        vpv = lambda x: a / (1.0 + a * x)
    nsteps, logw = np.full(n, cap, np.int32), np.zeros(n)
    idx = np.arange(n)
    x, p, lw = np.full(n, 0.05), np.full(n, pi0), np.zeros(n)
    sq = math.sqrt(dN)
    i = 0
    while len(idx) and i < cap:
        z4 = _normals(i, idx, seed)
        for z in z4:
            S = amp(x)
            dx = p * dN + S * (A * dN + z * sq)
            p = p + (0.5 * p * p - 3.0) * (p + vpv(x)) * dN
            lw = lw - (A * sq * z + 0.5 * A * A * dN)
            x = x + dx
            i += 1
            hit = x <= 0.0
            if hit.any():
                nsteps[idx[hit]], logw[idx[hit]] = i, lw[hit]
                keep = ~hit
                idx, x, p, lw = idx[keep], x[keep], p[keep], lw[keep]
                z4[:] = [w[keep] for w in z4]      # the group's later normals, for the paths that go on
            if i >= cap or not len(idx):
                break
    logw[idx] = lw
    return nsteps, logw


def exact(case, seed):
    k = case["kind"]
    if k == "hist":
        return _exact_hist(case, seed)
    if k not in ("exp", "linear") or case["n"] > 17000:
        return None
    nsteps, logw = _walk(case, seed)
    none = {key: None for key in fpt.HIST_ARRAYS + fpt.HIST_SCALARS}
    return dict(nsteps=nsteps, logw=logw, status=None, hist=none)


def _exact_hist(case, seed):
    nst, lw, status = (t.cpu().numpy() for t in _hist_data(case, seed))
    nb, n, G = case["bins"], case["n"], 32
    lo, db, tail = HIST_RANGE["N_lo"], (HIST_RANGE["N_hi"] - HIST_RANGE["N_lo"]) / nb, HIST_RANGE["N_tail"]
    N = nst.astype(np.float64) * 1e-3
    passed = status == 0
    q = (N - lo) / db
    inside = passed & (q >= 0.0) & (q < nb)
    b, w = np.floor(q[inside]).astype(np.int64), lw[inside]
    block = (np.arange(n, dtype=np.int64) * G // n)[inside]
    M = np.full(nb, -np.inf)
    np.maximum.at(M, b, w)
    M0 = np.where(np.isfinite(M), M, 0.0)
    e = np.exp(w - M0[b])

    def sums(v):
        return np.bincount(b, v, nb)

    cnt, S1, S2, L1, L2 = sums(np.ones_like(e)), sums(e), sums(e * e), sums(w), sums(w * w)
    some = cnt > 0
    with np.errstate(all="ignore"):
        out = dict(count=cnt.astype(np.int64), log_sum_w=np.where(some, M0 + np.log(S1), -np.inf),
                   log_sum_w2=np.where(some, 2.0 * M0 + np.log(S2), -np.inf), sum_lw=L1, sum_lw2=L2)
        out["pdf"] = np.where(some, np.exp(M0) * S1 / (n * db), 0.0)
        var = np.maximum(S2 - S1 * S1 / n, 0.0) / ((n - 1.0) * n)
        out["se_w"] = np.where(some, np.exp(M0) * np.sqrt(var) / db, 0.0)
        # variance of ln w about its mean, without the cancellation of the raw moments
        m = L1 / cnt
        s2 = sums((w - m[b]) ** 2) / (cnt - 1.0)
        two = cnt >= 2
        pl = (cnt / n) * np.exp(m + 0.5 * s2) / db
        cox = s2 / cnt + s2 * s2 / (2.0 * (cnt - 1.0))
        out["pdf_ln"] = np.where(two, pl, NAN)
        out["se_ln"] = np.where(two, pl * np.sqrt(cox + np.maximum(1.0 - cnt / n, 0.0) / cnt), NAN)
        per = np.bincount(block * nb + b, e, G * nb).reshape(G, nb)
        size = np.diff(np.array([-(-g * n // G) for g in range(G + 1)]))[:, None]
        jk = (S1 - per) / (n - size)
        out["se_jk"] = np.where(some, np.exp(M0) * np.sqrt((G - 1.0) / G * ((jk - jk.mean(0)) ** 2).sum(0)) / db, 0.0)
    lp, Np = lw[passed], N[passed]
    wt = np.exp(lp - lp.max())
    far = Np >= tail
    mt = lp[far].max() if far.any() else 0.0
    wf = np.exp(lp[far] - mt)
    out.update(n_total=n, n_passed=int(passed.sum()), n_under=int((passed & (q < 0)).sum()),
               n_over=int((passed & ~(q < nb)).sum()), n_capped=int((status == 1).sum()), n_tail=int(far.sum()),
               N_mean=float(Np.mean()), N_mean_w=float((wt * Np).sum() / wt.sum()),
               ess_tail=float(wf.sum() ** 2 / (wf * wf).sum()) if far.any() else 0.0,
               p_tail=float(math.exp(mt) * wf.sum() / n) if far.any() else 0.0, log_max_w=float(lp.max()), db=db)
    return out
