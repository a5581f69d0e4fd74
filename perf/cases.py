"""Workloads whose speed matters to a user of the sampler, with their inputs,
one pass through the public entry points, and the same results in FP64.

A case is one piece of a program written against the package: a call that
allocates nothing, a handle that is run again and again, a one-call batch, a
step of the downstream beta' search, a training step, the extreme field of an
ensemble.  `listed` gives the sizes of the repository's own workloads and
tests, `draw` more of the same ranges (odd mode numbers and ragged budgets
included).  Parameters follow workloads.py: C3/C2 = lambda / beta'.

`exact` evaluates the method from its definition in FP64 (Philox stream,
Box-Muller, H2, H3 by grid cubature, envelope), with torch and numpy only.

Integer statistics and the accepted records do not depend on the launch or on
the H3 form.  What only tells how a run was carried out (n_refined,
n_fallback, max_delta of the FP32 path, the record flags) is not returned.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_16952_gb300 as T
from paper_2411_16952_gb300 import matching

PROPOSALS = {"uniform": T.PROPOSAL_UNIFORM, "paper": T.PROPOSAL_PAPER, "learned": T.PROPOSAL_LEARNED}
FORMS = {"triad": T.H3_TRIAD_F32, "grid": T.H3_GRID_BF16X3, "auto": T.H3_AUTO}


# ---- the cases ---------------------------------------------------------------
def listed():
    return [
        # a latency-bound loop that may not allocate (sampler_run_static): the
        # statistics of one short range at the small configuration
        dict(name="static_k16", kind="static", K=16, proposal="paper", beta=20.0, lam=1500.0, n=1 << 16),
        # the small plain configuration: 2^20 proposals at acceptance ~1e-2,
        # statistics and the accepted fields read back
        dict(name="small_k16", kind="run", K=16, form="triad", proposal="paper", beta=20.0, beta_hi=20.0, points=1,
             lam=1500.0, n=1 << 20, grid_N=0, sir=False, keep=1 << 15),
        # the extreme-event regime on the tensor-core form, the form that AUTO
        # gives: eight beta' in one launch, streaming statistics
        dict(name="extreme_k32", kind="run", K=32, form="auto", proposal="paper", beta=20.0, beta_hi=60.0, points=8,
             lam=9000.0, n=1 << 24, grid_N=128, sir=False, keep=0),
        # the same regime in plain FP32 (the form to compare with, and the
        # only one beside SIR and static runs)
        dict(name="plain_k32", kind="run", K=32, form="triad", proposal="paper", beta=20.0, beta_hi=60.0, points=8,
             lam=9000.0, n=1 << 22, grid_N=0, sir=False, keep=0),
        # the naive baseline: uniform proposal, many proposals, the fields kept
        dict(name="naive_k32", kind="run", K=32, form="grid", proposal="uniform", beta=20.0, beta_hi=20.0, points=1,
             lam=3000.0, n=1 << 26, grid_N=128, sir=False, keep=1 << 16),
        # a parameter sweep in one call: beta' over two decades, two depth
        # ratios, uneven budgets; the call finds every point's envelope itself
        dict(name="batch_k32", kind="batch", K=32, form="auto", points=32, beta=6.0, beta_hi=600.0, log2_lo=18,
             log2_hi=24),
        # the 64-mode upstream ensemble with a learned correction, fields kept
        dict(name="upstream_k64", kind="run", K=64, form="grid", proposal="learned", beta=40.0, beta_hi=40.0, points=1,
             lam=24000.0, n=1 << 25, grid_N=256, sir=False, keep=1 << 13),
        # one step of the downstream beta' search at 64 modes: new candidates,
        # each with its own envelope, sampled in one launch
        dict(name="bisect_k64", kind="bisect", K=64, candidates=8, steps=1, n=1 << 22, lam=24000.0, r_scale=1.1,
             grid_N=256),
        # the cutoff of the speedup figure: 128 modes, acceptance ~0.28
        dict(name="speedup_k128", kind="run", K=128, form="triad", proposal="paper", beta=20.0, beta_hi=60.0, points=2,
             lam=9000.0, n=1 << 21, grid_N=0, sir=False, keep=0),
        # sampling-importance resampling in the extreme regime
        dict(name="sir_k32", kind="run", K=32, form="triad", proposal="paper", beta=20.0, beta_hi=60.0, points=8,
             lam=9000.0, n=1 << 21, grid_N=0, sir=True, keep=0),
        # a training step of the learned proposal on 2^20 fields per point
        dict(name="train_k32", kind="train", K=32, points=8, rows=1 << 20, beta=20.0, beta_hi=60.0, lam=9000.0,
             tau=0.5),
        # the 1-in-500 wave field of an ensemble of some hundred thousand
        dict(name="field_k32", kind="field", K=32, beta=20.0, lam=1000.0, n=1 << 20, m=500),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["static", "run", "run", "run", "warp", "sir", "batch", "bisect", "train", "field"])
    if kind == "static":
        K = rng.randint(4, 128)
        return dict(kind="static", K=K, proposal=rng.choice(["paper", "paper", "uniform"]),
                    beta=round(_logu(rng, 4.0, min(60.0, 0.6 * K * K)), 3),
                    lam=round(_lam(K) * rng.uniform(0.2, 0.8), 1), n=int(_logu(rng, 1 << 12, 1 << 18)))
    if kind in ("run", "sir", "warp"):
        K = rng.randint(65, 128) if kind == "warp" else rng.randint(4, 64)
        sir = kind == "sir"
        form = "triad" if sir or kind == "warp" else rng.choice(["triad", "grid", "auto"])
        pts = rng.randint(1, 8)
        top = min(60.0, 0.6 * K * K)
        # at most the work of the largest listed run (proposals x modes)
        cap = (1 << 22) * 128.0 if kind == "warp" else (1 << 30) * (0.25 if form == "triad" else 1.0)
        n = int(_logu(rng, 1 << 14, max(1 << 15, cap / (K * max(K, 16) / 32.0) / pts)))
        prop = "paper" if sir else rng.choice(["paper", "paper", "learned", "uniform"])
        return dict(kind="run", K=K, form=form, proposal=prop, beta=round(_logu(rng, 4.0, 0.6 * top), 3),
                    beta_hi=round(top, 3), points=pts, lam=round(_lam(K) * rng.uniform(0.2, 1.2), 1), n=n, grid_N=0,
                    sir=sir, keep=0 if sir or n > 1 << 17 else n * pts)
    if kind == "batch":
        K = rng.randint(8, 32)
        return dict(kind="batch", K=K, form=rng.choice(["auto", "triad"]), points=rng.randint(5, 32), beta=6.0,
                    beta_hi=round(0.58 * K * K, 3), log2_lo=rng.randint(14, 18), log2_hi=rng.randint(19, 23))
    if kind == "bisect":
        K = rng.randint(20, 64)
        return dict(kind="bisect", K=K, candidates=rng.randint(4, 8), steps=1, n=int(_logu(rng, 1 << 19, 1 << 22)),
                    lam=round(_lam(K), 1), r_scale=round(rng.uniform(0.95, 1.1), 3), grid_N=0)
    if kind == "train":
        return dict(kind="train", K=rng.randint(6, 64), points=rng.randint(1, 8), rows=int(_logu(rng, 1 << 14, 1 << 19)),
                    beta=8.0, beta_hi=20.0, lam=round(rng.uniform(500.0, 4000.0), 1), tau=rng.choice([0.5, 1.0, 0.0]))
    K = rng.randint(8, 64)
    return dict(kind="field", K=K, beta=round(_logu(rng, 10.0, 30.0), 3), lam=round(_lam(K) * 0.2, 1),
                n=int(_logu(rng, 1 << 17, 1 << 20)), m=rng.randint(50, 500))


def _lam(K):
    """beta' C3/C2 near the strongly nonlinear regime of K modes (1600 at 16, 4500 at 32, 13000 at 64)."""
    return 25.0 * K ** 1.5 if K <= 64 else 9000.0


# ---- points ---------------------------------------------------------------------
def _points(c):
    """[(beta', E0, C3/C2)] of a case."""
    if c["kind"] == "batch":  # the sweep of workloads.batch_k32: two depth ratios, E0 in [0.5, 2]
        g = np.random.default_rng(20241126)
        b = np.exp(g.uniform(np.log(c["beta"]), np.log(c["beta_hi"]), c["points"]))
        e = g.uniform(0.5, 2.0, c["points"])
        d = np.where(np.arange(c["points"]) % 2 == 0, 1.0, 0.24)
        return [(float(bb), float(ee), 4000.0 / math.sqrt(dd) / float(bb)) for bb, ee, dd in zip(b, e, d)]
    P = c.get("points", 1)
    betas = np.geomspace(c["beta"], c["beta_hi"], P) if P > 1 else [c["beta"]]
    return [(float(b), 1.0, c["lam"] / float(b)) for b in betas]


def _budgets(c):
    g = np.random.default_rng(7)
    return [int(2 ** g.uniform(c["log2_lo"], c["log2_hi"])) for _ in range(c["points"])]


def _correction(K):
    """A smooth mean-zero correction of a few per cent, as training gives."""
    k = np.arange(1, K + 1)
    t = 0.06 * np.cos(np.pi * k / K) + 0.02 * np.exp(-0.5 * k)
    return t - t.mean()


def _make(c, points, logM=None):
    corr = _correction(c["K"]) if c.get("proposal") == "learned" else None
    prop = PROPOSALS[c.get("proposal", "paper")]
    return [T.make_point(b, e, r, prop, point_id=p, logM=None if logM is None else logM[p], log_var_correction=corr)
            for p, (b, e, r) in enumerate(points)]


# ---- what a program holds before the call ---------------------------------------
def prepare(case, seed):
    c, K = case, case["K"]
    s = {"case": c, "seed": int(seed)}
    if c["kind"] == "static":
        (b, e, r), = _points(c)
        s2 = None if c["proposal"] == "uniform" else _sigma2(K, b, c["proposal"])
        s["logM"] = T.tkdv_log_M(K, b, e, r, s2)
        s["point"] = _make(c, [(b, e, r)], [s["logM"]])[0]
        s["stream"] = torch.cuda.current_stream()
    elif c["kind"] == "run":
        s["S"] = T.Sampler(K, _make(c, _points(c)), h3_mode=FORMS[c["form"]], grid_N=c["grid_N"],
                           sample_capacity=max(c["keep"], 16), stream=torch.cuda.current_stream(), sir=c["sir"])
        s["buf"] = torch.empty(c["keep"] * T.tkdv_record_bytes(K), dtype=torch.uint8, device="cuda")
    elif c["kind"] == "batch":
        s["points"] = _make(c, _points(c))
        s["options"] = T.make_options(K, h3_mode=FORMS[c["form"]], sample_capacity=1 << 16)
        s["budgets"] = np.array(_budgets(c), dtype=np.uint64)
    elif c["kind"] == "bisect":
        # the upstream ensemble gives the target of the search
        up = T.Sampler(K, [T.make_point(40.0, 1.0, c["lam"] / 40.0)], h3_mode=T.H3_GRID_BF16X3, grid_N=c["grid_N"],
                       sample_capacity=16)
        up.run(1 << 24, seed + 1)
        s["target"] = matching.mean_S(up.stats()[0], K)
        up.close()
    elif c["kind"] == "train":
        pts = _points(c)
        buf, n = _field_records(c, pts, seed)
        s["w0"] = _weights(seed)
        s["m"] = _Mlp(T.tkdv_mlp_create(0))
        feats = np.array([T.tkdv_mlp_features(K, b, e, r) for b, e, r in pts])
        w = [1.0 / _sigma2(K, b, "paper") for b, _, _ in pts]
        z = np.array([[b / (e * K * K), r] for b, e, r in pts])
        torch.cuda.synchronize()
        T.tkdv_mlp_set_data_records(s["m"].h, [K] * len(pts), feats, w, z, buf, n, K, c["rows"])
    else:
        s["S"] = T.Sampler(K, _make(dict(c, proposal="paper"), _points(c)), sample_capacity=c["n"],
                           stream=torch.cuda.current_stream())
        s["S"].run(c["n"], seed)
        s["S"].sync()
    return s


class _Mlp:
    def __init__(self, h):
        self.h = h

    def __del__(self):
        T.tkdv_mlp_destroy(self.h)


def _weights(seed):
    """Network weights part of the way through a training."""
    return (0.12 * np.random.default_rng(seed).standard_normal(T.MLP_NPARAM)).astype(np.float32)


def _field_records(c, points, seed):
    """Sampler records of `rows` fields per point, drawn from the paper's proposal."""
    K, n = c["K"], c["rows"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    words = T.tkdv_record_bytes(K) // 4
    buf = torch.zeros(len(points) * n, words, dtype=torch.float32, device="cuda")
    k = torch.arange(1, K + 1, device="cuda", dtype=torch.float32)
    N = 4 * K
    for p, (b, e, _) in enumerate(points):
        sig = torch.tensor(np.sqrt(_sigma2(K, b, "paper")), dtype=torch.float32, device="cuda")
        for o in range(0, n, 1 << 18):
            m = min(1 << 18, n - o)
            x = torch.randn(m, 2, K, generator=g, device="cuda") * sig
            x /= x.square().sum((1, 2), keepdim=True).sqrt()
            rows = buf[p * n + o:p * n + o + m]
            rows[:, 4] = e * (x.square().sum(1) * k * k).sum(1)
            u = torch.fft.irfft(torch.cat([torch.zeros(m, 1, device="cuda", dtype=torch.complex64),
                                           torch.complex(x[:, 0], -x[:, 1])], 1), n=N, norm="forward")
            # irfft gives 2 U; H3 = 2 pi (E0/2pi)^(3/2) T, T = (4/(3N)) sum U^3
            rows[:, 5] = 2 * math.pi * (e / (2 * math.pi)) ** 1.5 * (u / 2).pow(3).sum(1) * (4.0 / (3 * N))
            rows[:, 8:8 + 2 * K] = x.reshape(m, 2 * K)
        buf.view(torch.int32)[p * n:(p + 1) * n, 2] = p
    return buf, len(points) * n


# ---- one pass -------------------------------------------------------------------
def run(state):
    c, K = state["case"], state["case"]["K"]
    if c["kind"] == "static":
        st, _ = T.sampler_run_static(K, state["point"], 0, c["n"], state["seed"], stream=state["stream"])
        return {"stats": _stats([st], K, False)}
    if c["kind"] == "run":
        S = state["S"]
        S.reset()
        S.run(c["n"], state["seed"])
        out = {"stats": _stats(S.stats(), K, c["sir"])}
        if c["keep"]:
            out["records"] = _records(state["buf"], S.samples(c["keep"], device_dst=state["buf"]), K, c["keep"])
        return out
    if c["kind"] == "batch":
        return {"stats": _stats(T.sampler_batch_run(state["points"], state["options"], state["budgets"],
                                                    state["seed"]), K, False)}
    if c["kind"] == "bisect":
        d = matching.bisect_beta(K, 1.0, c["r_scale"] * c["lam"] / 40.0, matching.mean_S, state["target"], 30.0, 50.0,
                                 n_candidates=c["candidates"], n_steps=c["steps"], proposals_per_candidate=c["n"],
                                 seed=state["seed"], h3_mode=T.H3_GRID_BF16X3, grid_N=c["grid_N"])
        return {"beta": d["beta"], "bracket": d["bracket"], "history": [list(h) for h in d["history"]]}
    if c["kind"] == "train":
        T.tkdv_mlp_set_params(state["m"].h, state["w0"])
        loss, grad = T.tkdv_mlp_step(state["m"].h, lr=2e-2, tau=c["tau"], update=True, want_grad=True)
        return {"loss": loss, "grad": grad}
    return state["S"].extreme_field(m=c["m"])


def _stats(stats, K, sir):
    """The statistics of all points, one array per field."""
    ints = ["n_proposals", "n_accepted", "n_near_threshold", "n_envelope_violations", "n_dropped", "n_kept"]
    out = {"counts": np.array([[s[f] for f in ints] for s in stats], dtype=np.int64),
           "hist": np.array([s["hist"] for s in stats]).astype(np.int64),
           "exceed": np.array([s["exceed"] for s in stats]).astype(np.int64),
           "spectrum": np.array([s["spectrum"][:K] for s in stats]),
           "sum_u0": np.array([s["sum_u0"] for s in stats]),
           "moments": np.array([[s[f] for f in ("mean", "var", "skew", "kurt")] for s in stats])}
    if sir:
        out["sir"] = np.array([[s["sir_sum_w"], s["sir_sum_w2"], s["sir_sum_wS"], *s["sir_sum_w_u0"]] for s in stats])
    return out


def _records(buf, n, K, keep):
    """The accepted fields in the order of their proposals, on the device, in
    arrays of `keep` rows (index -1 and zeros after the last field)."""
    rec = buf[:n * T.tkdv_record_bytes(K)].view(n, T.tkdv_record_bytes(K))
    key = torch.full((keep,), -1, dtype=torch.int64, device=buf.device)
    idx = rec[:, 0:8].contiguous().view(torch.int64).reshape(n)
    point = rec[:, 8:12].contiguous().view(torch.int32).reshape(n)
    key[:n], order = torch.sort(idx + point.long() * _POINT)
    vals = torch.zeros(keep, 4 + 2 * K, device=buf.device)
    vals[:n] = rec[:, 16:32 + 8 * K].view(torch.float32)[order]
    return {"key": key, "H2": vals[:, 0], "H3": vals[:, 1], "u0": vals[:, 2], "delta": vals[:, 3], "xhat": vals[:, 4:]}


_POINT = 1 << 48  # key of a field: its point and its index in the point's stream


# ---- the least a pass can do ------------------------------------------------------
def work(case):
    """bytes: inputs read and results written once.  flops: FP32 and integer
    operations of the method per proposal: ten Philox rounds of eight
    operations per block, about forty per mode for the two normals and the
    mode sums, and the cubature by a fast transform onto 4K points."""
    c, K = case, case["K"]
    op = 80.0 * (K / 2 + 1) + 40.0 * K + 10.0 * K * math.log2(4 * K) + 12.0 * K
    rb = 32 + 8 * K
    if c["kind"] == "static":
        return {"bytes": 3400.0, "flops": c["n"] * op}
    if c["kind"] == "run":
        return {"bytes": c["points"] * 3400.0, "flops": c["points"] * c["n"] * op}
    if c["kind"] == "batch":
        return {"bytes": c["points"] * 3400.0, "flops": float(sum(_budgets(c))) * op}
    if c["kind"] == "bisect":
        return {"bytes": c["candidates"] * c["steps"] * 3400.0, "flops": c["candidates"] * c["steps"] * c["n"] * op}
    if c["kind"] == "train":
        rows = c["points"] * c["rows"]
        return {"bytes": rows * 4.0 * (K + 1) + 4.0 * T.MLP_NPARAM * 6, "flops": rows * (4.0 * K + 40)}
    return {"bytes": c["n"] * 0.1 * rb, "flops": c["n"] * 0.1 * 10.0 * K * math.log2(2 * K)}


# ---- the same results in FP64 -----------------------------------------------------
def _alpha(K, beta):
    k = np.arange(1, K + 1, dtype=np.float64)

    def f(a):
        return 1.0 - a / K * np.sum(1.0 / (1.0 + a * beta * k * k / K ** 3))
    lo, hi = 0.0, 1.0
    while f(hi) > 0:
        lo, hi = hi, 2 * hi
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if f(mid) > 0 else (lo, mid)
    return 0.5 * (lo + hi)


def _sigma2(K, beta, proposal):
    if proposal == "uniform":
        return np.ones(K)
    k = np.arange(1, K + 1, dtype=np.float64)
    s2 = 1.0 / (1.0 + _alpha(K, beta) * beta * k * k / K ** 3)
    return s2 * np.exp(_correction(K)) if proposal == "learned" else s2


def _coef(K, b, e, r, uniform):
    h3s = 2 * math.pi * (e / (2 * math.pi)) ** 1.5
    return -b / K ** 2, b * r / (e * K ** 2) * h3s, 0.0 if uniform else float(K), h3s


def _log_m(K, b, e, r, s2, uniform):
    """max of log f/g.  |Re v_k v_l conj v_{k+l}| <= |v_k v_l v_{k+l}|, so the
    maximum is at real amplitudes of one sign; L-BFGS over those from
    Dirichlet-like, flat and narrow starts."""
    cS, cH, cQ, _ = _coef(K, b, e, r, uniform)
    k = torch.arange(1, K + 1, dtype=torch.float64)
    w = torch.tensor(1.0 / s2, dtype=torch.float64)
    N = 4 * K

    def f(y):
        x = y / y.norm()
        U = torch.fft.irfft(torch.cat([x.new_zeros(1), x]) + 0j, n=N, norm="forward") / 2
        v = cS * (k * k * x * x).sum() + abs(cH) * (4.0 / (3 * N)) * U.pow(3).sum()
        return v + cQ * torch.log((w * x * x).sum()) if cQ else v
    best = -math.inf
    one = torch.zeros(K, dtype=torch.float64)
    one[0] = 1.0
    for start in [torch.exp(-g * k * k / K ** 2) for g in (0.0, 2.0, 8.0, 32.0)] + [one + 1e-3, one.flip(0) + 1e-3]:
        y = (start / start.norm()).requires_grad_(True)
        opt = torch.optim.LBFGS([y], max_iter=600, history_size=30, tolerance_grad=1e-12, tolerance_change=1e-16,
                                line_search_fn="strong_wolfe")

        def closure():
            opt.zero_grad()
            loss = -f(y)
            loss.backward()
            return loss
        opt.step(closure)
        best = max(best, float(f(y.detach())))
    return best


def _philox(c0, lo, hi, pid, seed):
    m = 0xFFFFFFFF
    c = [c0 & m, lo & m, hi & m, pid & m]
    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # low 64 bits; the sign is masked away
        c = [((p1 >> 32) & m) ^ c[1] ^ k0, p1 & m, ((p0 >> 32) & m) ^ c[3] ^ k1, p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c


def _u(w):
    return ((w >> 8) | 1).double() * 2.0 ** -24


def _u_tail(w, g, lo, hi, pid, seed):
    """The uniform of word w at stream position g, its lowest bucket refined."""
    u = _u(w)
    rows = torch.nonzero(w < 512, as_tuple=True)
    if rows[0].numel():
        l, h, gg = lo.expand_as(w)[rows], hi.expand_as(w)[rows], g.expand_as(w)[rows]
        w1 = _philox(0x80000000 + (1 << 24) + gg, l, h, torch.full_like(l, pid), seed)[0]
        w2 = _philox(0x80000000 + (2 << 24) + gg, l, h, torch.full_like(l, pid), seed)[0]
        u[rows] = torch.where(w1 >= 512, 2.0 ** -23 * _u(w1), 2.0 ** -46 * _u(w2))
    return u


def _proposals(K, s2, cf, logM, E0, pid, seed, idx):
    """log f/(Mg), ln U and the fields of the listed proposals."""
    cS, cH, cQ, h3s = cf
    dev = idx.device
    lo, hi = (idx & 0xFFFFFFFF)[:, None], (idx >> 32)[:, None]
    j = torch.arange((K + 1) // 2, device=dev)[None, :]
    one = torch.ones_like(lo + j)
    w = torch.stack(_philox(j * one, lo * one, hi * one, pid * one, seed), -1).reshape(len(idx), -1, 2)[:, :K]
    g = 2 * torch.arange(K, device=dev)[None, :]
    rho = -2.0 * torch.log(_u_tail(w[..., 0], g, lo, hi, pid, seed))
    ang = 2 * math.pi * _u(w[..., 1])
    sig = torch.tensor(np.sqrt(s2), device=dev)
    x, y = sig * rho.sqrt() * torch.cos(ang), sig * rho.sqrt() * torch.sin(ang)
    nrm2 = (x * x + y * y).sum(1)
    inv = nrm2.rsqrt()
    x, y = x * inv[:, None], y * inv[:, None]
    k = torch.arange(1, K + 1, device=dev, dtype=torch.float64)
    S = (k * k * (x * x + y * y)).sum(1)
    N = 4 * K
    U = torch.fft.irfft(torch.cat([torch.zeros(len(idx), 1, device=dev, dtype=torch.complex128),
                                   torch.complex(x, -y)], 1), n=N, norm="forward") / 2
    t3 = (4.0 / (3 * N)) * U.pow(3).sum(1)
    delta = cS * S + cH * t3 - logM
    if cQ:
        delta = delta + cQ * torch.log(rho.sum(1) / nrm2)
    b = (K + 1) // 2
    wa = _philox(torch.full_like(lo, b), lo, hi, torch.full_like(lo, pid), seed)[0]
    lnU = torch.log(_u_tail(wa, torch.full_like(lo, 4 * b), lo, hi, pid, seed))[:, 0]
    u0 = 2 * math.sqrt(E0 / (2 * math.pi)) * x.sum(1)
    return delta, lnU, E0 * S, h3s * t3, u0, torch.cat([x, y], 1)


def _copies(u, lam):
    """#{k >= 1 : u < P(N >= k)}, N ~ Poisson(lam), from the upper tail."""
    n = 0
    while n < 4000:
        lead = math.exp((n + 1) * math.log(lam) - lam - math.lgamma(n + 2.0))
        term = total = 1.0
        for i in range(1, 400):
            term *= lam / (n + 1 + i)
            total += term
            if term < 1e-17 * total:
                break
        if not u < lead * total:
            break
        n += 1
    return n


def _moments(s, n):
    if n == 0:
        return [math.nan] * 4
    m = [v / n for v in s]
    var = m[1] - m[0] ** 2
    return [m[0], var, (m[2] - 3 * m[0] * m[1] + 2 * m[0] ** 3) / var ** 1.5,
            (m[3] - 4 * m[0] * m[2] + 6 * m[0] ** 2 * m[1] - 3 * m[0] ** 4) / var ** 2]


def _ensemble(c, points, counts, seed, sir=False):
    """The statistics and records of all points by the method's definition."""
    K, prop = c["K"], c.get("proposal", "paper")
    uni = prop == "uniform"
    stat = {"counts": None, "hist": None, "exceed": None, "spectrum": [], "sum_u0": [], "moments": [], "sir": []}
    recs = []
    for p, (b, e, r) in enumerate(points):
        s2 = _sigma2(K, b, prop)
        cf = _coef(K, b, e, r, uni)
        logM = _log_m(K, b, e, r, s2, uni)
        spec, q, w7, n = torch.zeros(K, dtype=torch.float64, device="cuda"), np.zeros(4), np.zeros(7), 0
        step = (1 << 23) // K
        for o in range(0, counts[p], step):
            idx = torch.arange(o, min(o + step, counts[p]), device="cuda", dtype=torch.int64)
            d, lnU, H2, H3, u0, xh = _proposals(K, s2, cf, logM, e, p, seed, idx)
            if sir:
                w = d.exp()
                w7 += np.array([float(v) for v in (w.sum(), (w * w).sum(), (w * H2 / e).sum(), *((w * u0 ** i).sum()
                                                                                               for i in (1, 2, 3, 4)))])
                sel = torch.nonzero(lnU < torch.log(-torch.expm1(-w)) + 1e-6)[:, 0]
                cp = [_copies(math.exp(a), math.exp(f)) for a, f in zip(lnU[sel].tolist(), d[sel].tolist())]
                cp = torch.tensor(cp, dtype=torch.float64, device="cuda")
            else:
                sel = torch.nonzero(lnU < d)[:, 0]
                cp = torch.ones(len(sel), dtype=torch.float64, device="cuda")
                recs.append([v[sel] for v in (H2, H3, u0, d, xh)])
            n += int(cp.sum())
            q += np.array([float((cp * u0[sel] ** i).sum()) for i in (1, 2, 3, 4)])
            spec += (cp[:, None] * (xh[sel, :K] ** 2 + xh[sel, K:] ** 2)).sum(0)
        stat["spectrum"].append(spec.cpu().numpy())
        stat["sum_u0"].append(q)
        stat["moments"].append(_moments(q, n))
        stat["sir"].append(w7)
    out = {"stats": {f: v if v is None else np.array(v) for f, v in stat.items() if sir or f != "sir"}}
    if c.get("keep"):
        out["records"] = {"key": None}
        for i, f in enumerate(("H2", "H3", "u0", "delta", "xhat")):
            v = torch.cat([x[i] for x in recs])
            out["records"][f] = torch.cat([v, v.new_zeros(c["keep"] - len(v), *v.shape[1:])])
    return out


def _train_exact(c, seed):
    K, pts, tau = c["K"], _points(c), c["tau"]
    buf, _ = _field_records(c, pts, seed)
    w0 = torch.tensor(_weights(seed)).bfloat16().double().requires_grad_(True)
    sizes = [(64, 4), (64,), (64, 64), (64,), (64, 64), (64,)]
    par, o = [], 0
    for sh in sizes:
        par.append(w0[o:o + math.prod(sh)].reshape(sh))
        o += math.prod(sh)
    loss = 0.0
    for p, (b, e, r) in enumerate(pts):
        ft = torch.tensor([math.log(max(b, 1e-3)) / math.log(100.0), math.log(e),
                           math.log1p(max(b * r, 0.0) / 100.0) / math.log(100.0), K / 64.0], dtype=torch.float64)
        h = torch.tanh(par[2] @ torch.tanh(par[0] @ ft + par[1]) + par[3])
        cc = (par[4] @ h + par[5])[:K]
        cc = (cc - cc.mean()).cuda()
        wp = torch.tensor(1.0 / _sigma2(K, b, "paper"), device="cuda") * torch.exp(-cc)
        rows = buf[p * c["rows"]:(p + 1) * c["rows"]].double()
        xh = rows[:, 8:8 + 2 * K]
        Q = (xh[:, :K] ** 2 + xh[:, K:] ** 2) @ wp
        ell = K * torch.log(Q) - torch.log(wp).sum()
        z = -b / (e * K * K) * (rows[:, 4] - r * rows[:, 5])
        J = tau * (torch.logsumexp((z + ell) / tau, 0) - math.log(len(Q))) if tau > 0 else ell.mean()
        loss = loss + J.cpu()
    loss.backward()
    return {"loss": float(loss), "grad": w0.grad.numpy()}


def exact(case, seed):
    c = case
    if c["kind"] == "static":
        return _ensemble(c, _points(c), [c["n"]], seed)
    if c["kind"] == "run":
        if c["points"] * c["n"] * c["K"] > 1 << 32:
            return None
        return _ensemble(c, _points(c), [c["n"]] * c["points"], seed, c["sir"])
    if c["kind"] == "batch":
        if sum(_budgets(c)) * c["K"] > 1 << 32:
            return None
        return _ensemble(c, _points(c), _budgets(c), seed)
    if c["kind"] == "train":
        return _train_exact(c, seed)
    if c["kind"] == "field":
        # the first m accepted fields of the stream, on the 2K-point grid
        K, (b, e, r) = c["K"], _points(c)[0]
        s2 = _sigma2(K, b, "paper")
        cf, logM = _coef(K, b, e, r, False), _log_m(K, b, e, r, s2, False)
        got, o = [], 0
        while sum(len(g) for g in got) < c["m"] and o < c["n"]:
            idx = torch.arange(o, min(o + (1 << 16), c["n"]), device="cuda", dtype=torch.int64)
            d, lnU, *_, xh = _proposals(K, s2, cf, logM, e, 0, seed, idx)
            got.append(xh[lnU < d])
            o += 1 << 16
        xh = torch.cat(got)[:c["m"]]
        if len(xh) < c["m"]:
            return None
        k = torch.arange(1, K + 1, device="cuda", dtype=torch.float64)
        xi = -math.pi + math.pi * torch.arange(2 * K, device="cuda", dtype=torch.float64) / K
        u = 2 * math.sqrt(e / (2 * math.pi)) * (xh[:, :K] @ torch.cos(k[:, None] * xi)
                                                + xh[:, K:] @ torch.sin(k[:, None] * xi))
        i, jj = divmod(int(u.argmax()), 2 * K)
        return {"idx": None, "umax": float(u[i, jj]), "xi": float(xi[jj]), "xhat": xh[i].cpu().numpy()}
    return None
