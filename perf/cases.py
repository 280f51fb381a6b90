"""Performance cases of the sampler library: what its users have it compute, as
calls of its public entry points.

Three kinds of work stand here.  Whole sampler runs (`run`): a handle is
restarted with a new seed, runs some iterations and gives back its particles,
log-weights and evidence estimate.  Single moves (`leapfrog`, `flow_move`) of
programs that drive their own loop: every particle's leapfrog trajectory under
one of the targets, in one of the precisions.  And the stages around them
(`normalise`, `resample`, `flow_grad`).  Sizes are those of the configurations
in `workloads`, of the benchmark and of the tests, and ranges around them.

All inputs are made from the seed alone; model data are FP32 values (the
library computes in FP32), so that the 64-bit results of `exact` are for the
very same inputs.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2504_02627_gb300 import _binding as B

PREC = {"fp32": B.PREC_FP32, "bf16x3": B.PREC_BF16X3, "bf16x2": B.PREC_BF16X2, "bf16c": B.PREC_BF16C,
        "bf16": B.PREC_BF16}
LOG_2PI = math.log(2.0 * math.pi)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest call: one SMC run of 256 particles on a 10-d correlated
        # Gaussian, 20 iterations; latency of the stages is what a user waits for.
        {"name": "run_gauss10", "op": "run", "model": "gauss", "dim": 10, "particles": 256, "runs": 1, "iters": 20,
         "precision": "fp32", "eps": 0.1, "len0": 5.0, "init_scale": 2.0, "cond": 100.0},
        # Many independent runs of uneven size in one handle: 64 runs of 512 to
        # 8192 particles on the 52-d hierarchical normal model.
        {"name": "run_hier64", "op": "run", "model": "hier", "dim": 52, "particles": 8192, "runs": 64, "iters": 3,
         "precision": "fp32", "eps": 0.01, "len0": 1.0, "init_scale": 1.0},
        # Ten seeds of the n = 1000 logistic regression in one handle, in the
        # precision that the benchmark chooses for regressions.
        {"name": "run_logistic10", "op": "run", "model": "logistic", "n": 1000, "dim": 25, "particles": 4096,
         "runs": 10, "iters": 2, "precision": "bf16c", "eps": 1e-3, "len0": 5.0, "init_scale": 1.0},
        # One move of the same regression in plain FP32, jittered step counts.
        {"name": "leapfrog_logistic_fp32", "op": "leapfrog", "model": "logistic", "n": 1000, "dim": 25,
         "particles": 4096, "steps": 40, "ragged": True, "precision": "fp32", "eps": 1e-3},
        # The largest call: a move of the n = 1e5, 100-d regression.
        {"name": "leapfrog_logistic_large", "op": "leapfrog", "model": "logistic", "n": 100000, "dim": 100,
         "particles": 16384, "steps": 8, "ragged": False, "precision": "bf16c", "eps": 5e-4},
        # The ill-conditioned 100-d Gaussian: plain FP32, and on tensor cores.
        {"name": "leapfrog_gauss100_fp32", "op": "leapfrog", "model": "gauss", "dim": 100, "particles": 8192,
         "steps": 20, "ragged": False, "precision": "fp32", "eps": 0.005, "cond": 1e4},
        {"name": "leapfrog_gauss100_bf16x3", "op": "leapfrog", "model": "gauss", "dim": 100, "particles": 8191,
         "steps": 50, "ragged": True, "precision": "bf16x3", "eps": 0.005, "cond": 1e4},
        # The 50-d banana: a cheap gradient, long trajectories, ragged.
        {"name": "leapfrog_banana50", "op": "leapfrog", "model": "banana", "dim": 50, "particles": 8192, "steps": 100,
         "ragged": True, "precision": "fp32", "eps": 0.02},
        # The learned transport map: a move in its latent space, and the
        # gradient of its training loss, with BF16 products.
        {"name": "flow_move_bf16", "op": "flow_move", "dim": 100, "hidden": 128, "layers": 4, "particles": 8192,
         "steps": 4, "precision": "bf16", "eps": 0.005},
        {"name": "flow_grad_bf16", "op": "flow_grad", "dim": 100, "hidden": 128, "layers": 4, "particles": 8192,
         "precision": "bf16"},
        # Weights and ancestors for loops that resample on their own, an odd
        # number of particles and a large one.
        {"name": "normalise_100k", "op": "normalise", "particles": 100003, "spread": 3.0},
        {"name": "resample_1m", "op": "resample", "particles": 1048576, "spread": 1.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["run", "run", "leapfrog", "leapfrog", "leapfrog", "leapfrog", "flow_move", "flow_grad",
                     "normalise", "resample"])
    if op == "normalise":
        return {"op": op, "particles": _log_int(rng, 256, 4194304), "spread": round(rng.uniform(0.5, 6.0), 2)}
    if op == "resample":
        return {"op": op, "particles": _log_int(rng, 256, 4194304), "spread": round(rng.uniform(0.5, 4.0), 2)}
    if op in ("flow_move", "flow_grad"):
        dim = 2 * rng.randint(5, 50)
        c = {"op": op, "dim": dim, "hidden": 16 * rng.randint(max(2, (dim + 31) // 32), 8), "layers": rng.randint(2, 4),
             "particles": _log_int(rng, 500, 8192), "precision": rng.choice(["bf16", "bf16", "fp32"])}
        if op == "flow_move":
            c.update(steps=rng.randint(1, 6), eps=0.005)
        return c
    if op == "run":
        model = rng.choice(["gauss", "gauss", "hier", "logistic"])
        if model == "gauss":
            return {"op": op, "model": model, "dim": rng.randint(2, 30), "particles": _log_int(rng, 200, 4000),
                    "runs": rng.choice([1, 1, 10]), "iters": rng.randint(5, 20), "precision": "fp32", "eps": 0.1,
                    "len0": 5.0, "init_scale": 2.0, "cond": 100.0}
        if model == "hier":
            return {"op": op, "model": model, "dim": rng.randint(8, 60), "particles": _log_int(rng, 600, 8192),
                    "runs": rng.randint(2, 64), "iters": rng.randint(2, 4), "precision": "fp32", "eps": 0.01,
                    "len0": 1.0, "init_scale": 1.0}
        return {"op": op, "model": model, "n": _log_int(rng, 300, 5000), "dim": rng.randint(5, 60),
                "particles": _log_int(rng, 500, 4096), "runs": rng.randint(1, 10), "iters": 2, "precision": "bf16c",
                "eps": 1e-3, "len0": 5.0, "init_scale": 1.0}
    model = rng.choice(["logistic", "logistic", "linear", "gauss", "gauss", "banana", "hier"])
    c = {"op": op, "model": model, "particles": _log_int(rng, 250, 16384), "steps": _log_int(rng, 4, 100),
         "ragged": rng.random() < 0.5, "precision": "fp32"}
    if model in ("logistic", "linear"):
        c["precision"] = rng.choice(["fp32", "bf16c", "bf16c", "bf16x2"])
        c["n"] = _log_int(rng, 200, 100000 if c["precision"] == "bf16c" else 20000)
        c["dim"] = rng.randint(4, 100)
        c["eps"] = 2.5e-4
        # keep the move below the largest listed one (FP32 runs at a
        # twentieth of the tensor cores' rate)
        most = 4e12 if c["precision"] == "bf16c" else 1e12 if c["precision"] == "bf16x2" else 1.5e11
        c["steps"] = max(1, min(c["steps"], int(most / (4.0 * c["n"] * c["dim"] * c["particles"]))))
        c["particles"] = max(64, min(c["particles"], int(most / (8.0 * c["n"] * c["dim"]))))
    elif model == "gauss":
        c.update(dim=_log_int(rng, 5, 128), eps=0.01, cond=1e3)
        c["precision"] = rng.choice(["fp32", "fp32", "bf16x3"])
    elif model == "banana":
        c.update(dim=2 * rng.randint(1, 32), eps=0.02)
    else:
        c.update(dim=rng.randint(5, 64), eps=0.01)
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _f32(t):
    """The FP32 values of t, in 64 bits: what the library is given."""
    return t.float().double()


def _data(case, g):
    """The target's data, on the GPU in 64 bits (FP32 values)."""
    D = case["dim"]
    kind = case.get("model", "gauss")
    if kind == "gauss":
        # N(0, Q diag(lam) Q'), lam geometric over the condition number
        cond = case.get("cond", 1e4)
        lam = torch.logspace(0.0, -math.log10(cond), D, dtype=torch.float64, device="cuda")
        Q, R = torch.linalg.qr(_randn(g, D, D))
        Q = Q * torch.sign(torch.diagonal(R))[None, :]
        P = (Q / lam[None, :]) @ Q.T
        return {"P": _f32(0.5 * (P + P.T)), "mu": torch.zeros(D, dtype=torch.float64, device="cuda"),
                "root": Q * lam.sqrt()[None, :]}
    if kind in ("logistic", "linear"):
        n = case["n"]
        X = _randn(g, n, D)
        if n >= 5000:   # the large regressions have correlated features
            X = math.sqrt(0.7) * X + math.sqrt(0.3) * _randn(g, n, 1)
        else:
            X[:, 0] = 1.0
        X = _f32(X)
        beta = _randn(g, D)
        if kind == "linear":
            return {"X": X, "beta": beta, "y": _f32(X @ beta + 0.5 * _randn(g, n))}
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        return {"X": X, "beta": beta, "y": (u < torch.sigmoid(X @ beta)).double()}
    if kind == "hier":
        G, obs = D - 2, 20
        mu, lt = _randn(g, 1), _randn(g, 1)
        y = mu + lt.exp() * _randn(g, G, 1) + _randn(g, G, obs)
        ybar = y.mean(1)
        return {"ybar": _f32(ybar), "n_g": torch.full((G,), float(obs), dtype=torch.float64, device="cuda"),
                "ss": _f32(((y - ybar[:, None]) ** 2).sum(1)), "mu": mu, "lt": lt}
    return {}


def _model(case, d):
    host = lambda k: d[k].cpu().numpy()  # noqa: E731
    kind, D = case.get("model", "gauss"), case["dim"]
    if kind == "gauss":
        return B.ModelData(B.GAUSS_DENSE, D, mu=host("mu"), prec=host("P"))
    if kind == "logistic":
        return B.ModelData(B.LOGISTIC, D, case["n"], X=host("X"), y=host("y"), hyper=(1.0,))
    if kind == "linear":
        return B.ModelData(B.LINEAR_GAUSS, D, case["n"], X=host("X"), y=host("y"), hyper=(0.5, 1.0))
    if kind == "hier":
        return B.ModelData(B.HIER_NORMAL, D, D - 2, group_mean=host("ybar"), group_n=host("n_g"),
                           group_ss=host("ss"), hyper=(1.0,))
    return B.ModelData(B.BANANA, D, hyper=(10.0, 0.1))


def _positions(case, d, g):
    """Particles where a sampler has them: around the target's mass."""
    D, N = case["dim"], case["particles"]
    kind = case.get("model", "gauss")
    z = _randn(g, D, N)
    if kind == "gauss":
        th = d["root"] @ z
    elif kind in ("logistic", "linear"):
        th = d["beta"][:, None] + (2.0 / math.sqrt(case["n"])) * z
    elif kind == "hier":
        th = z
        th[0] = d["mu"] + 0.3 * z[0]
        th[1] = d["lt"] + 0.15 * z[1]
    else:
        th = z
        th[0::2] *= math.sqrt(10.0)
        th[1::2] += 0.1 * (th[0::2] ** 2 - 10.0)
    return th.float()


def _steps(case, g):
    N, S = case["particles"], case["steps"]
    if not case.get("ragged"):
        return torch.full((N,), S, dtype=torch.int32, device="cuda")
    return torch.randint(1, S + 1, (N,), generator=g, device="cuda", dtype=torch.int32)


def _flow_params(case, g):
    """Parameters of a partly trained map: hidden weights of variance
    1 / fan-in, a small last layer."""
    D, H, L = case["dim"], case["hidden"], case["layers"]
    parts = []
    for _ in range(L):
        parts += [_randn(g, H * (D // 2)) / math.sqrt(D // 2), 0.1 * _randn(g, H), _randn(g, H * H) / math.sqrt(H),
                  0.1 * _randn(g, H), 0.1 * _randn(g, D * H) / math.sqrt(H), 0.1 * _randn(g, D) / math.sqrt(H)]
    return torch.cat(parts).float()


def _logw(case, g):
    """Log-weights after a move: a normal spread about a large offset."""
    return case["spread"] * _randn(g, case["particles"]) - 300.0


def _move_inputs(case, seed):
    g = _gen(seed)
    d = _data(case, g)
    th = _positions(case, d, g)
    p = _randn(g, case["dim"], case["particles"]).float()
    return g, d, th, p, _steps(case, g)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    op, N = case["op"], case["particles"]
    st = {"case": case}
    if op == "run":
        d = _data(case, _gen(seed))
        R = case["runs"]
        sizes = [N] * R
        if case["model"] == "hier":   # uneven runs
            sizes = np.random.default_rng(4242).integers(min(512, N), N + 1, size=R).tolist()
        cfgs = [B.make_config(n, max(20, case["iters"]), max(10, case["iters"] // 2), case["eps"], case["len0"],
                              seed=int(seed) * 1000 + r, init_scale=case["init_scale"],
                              precision=PREC[case["precision"]]) for r, n in enumerate(sizes)]
        smp = B.Sampler(_model(case, d), cfgs if R > 1 else cfgs[0], _stream())
        st.update(smp=smp, seed=int(seed) * 1000 + 500,
                  theta=torch.empty(case["dim"], smp.n_total, device="cuda"),
                  logw=torch.empty(smp.n_total, dtype=torch.float64, device="cuda"))
        return st
    if op == "normalise":
        one = lambda: torch.empty(1, dtype=torch.float64, device="cuda")  # noqa: E731
        st.update(logw=_logw(case, _gen(seed)), W=torch.empty(N, dtype=torch.float64, device="cuda"), lse=one(),
                  ess=one())
        return st
    if op == "resample":
        W = torch.softmax(_logw(case, _gen(seed)), 0)
        nb = B.lib().smc_k_resample_scratch_bytes(N)
        st.update(W=W, r64=(int(seed) * 0x9E3779B97F4A7C15 + 12345) % (1 << 64),
                  q=torch.empty(N, dtype=torch.int64, device="cuda"),
                  anc=torch.empty(N, dtype=torch.int32, device="cuda"),
                  status=torch.empty(1, dtype=torch.int32, device="cuda"),
                  scratch=torch.empty(nb, dtype=torch.uint8, device="cuda"))
        return st
    if op == "flow_grad":
        g = _gen(seed)
        par = _flow_params(case, g)
        st.update(par=par, theta=_randn(g, case["dim"], N).float(),
                  W=torch.softmax(0.5 * _randn(g, N), 0), grad=torch.empty_like(par))
        return st
    g, d, th, p, steps = _move_inputs(case, seed)
    dm = B.DevModel(_model(case, d), _stream())
    gr = torch.zeros_like(th)
    lp = torch.zeros(N, dtype=torch.float64, device="cuda")
    tprec = B.PREC_FP32 if op == "flow_move" else PREC[case["precision"]]
    B.check(B.lib().smc_k_target(dm.h, th.data_ptr(), N, N, lp.data_ptr(), gr.data_ptr(), tprec, _stream()),
            "smc_k_target")
    # the move is in place: the program keeps the state before it
    st.update(dm=dm, before=(th, p, gr, lp), after=tuple(torch.empty_like(t) for t in (th, p, gr, lp)), steps=steps)
    if op == "flow_move":
        st.update(par=_flow_params(case, g), z0=torch.empty_like(th), z1=torch.empty_like(th),
                  dH=torch.empty(N, dtype=torch.float64, device="cuda"))
    torch.cuda.current_stream().synchronize()
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    op, N, lib, s = case["op"], case["particles"], B.lib(), _stream()
    if op == "run":
        smp = st["smp"]
        smp.reset(st["seed"])
        smp.run(case["iters"])
        B.check(lib.smc_get_particles(smp.h, ctypes.c_void_p(st["theta"].data_ptr()),
                                      ctypes.c_void_p(st["logw"].data_ptr()), 1), "smc_get_particles", smp.h)
        return {"theta": st["theta"], "logw": st["logw"], "log_z": smp.log_evidence()}
    if op == "normalise":
        B.check(lib.smc_k_normalise(st["logw"].data_ptr(), N, st["W"].data_ptr(), st["lse"].data_ptr(),
                                    st["ess"].data_ptr(), s), "smc_k_normalise")
        return {"W": st["W"], "lse": st["lse"], "ess": st["ess"]}
    if op == "resample":
        B.check(lib.smc_k_resample(st["W"].data_ptr(), N, st["r64"], st["q"].data_ptr(), st["anc"].data_ptr(),
                                   st["status"].data_ptr(), st["scratch"].data_ptr(), s), "smc_k_resample")
        return {"q": st["q"], "ancestors": st["anc"], "status": st["status"]}
    if op == "flow_grad":
        B.check(lib.smc_k_flow_loss_grad(case["dim"], case["hidden"], case["layers"], st["par"].data_ptr(),
                                         st["theta"].data_ptr(), st["W"].data_ptr(), N, N, st["grad"].data_ptr(),
                                         PREC[case["precision"]], s), "smc_k_flow_loss_grad")
        return {"grad": st["grad"]}
    for a, b in zip(st["after"], st["before"]):
        a.copy_(b)
    th, p, gr, lp = st["after"]
    out = {"theta": th, "p": p, "grad": gr, "logpi": lp}
    if op == "leapfrog":
        B.check(lib.smc_k_leapfrog(st["dm"].h, th.data_ptr(), p.data_ptr(), gr.data_ptr(), lp.data_ptr(),
                                   st["steps"].data_ptr(), case["eps"], N, N, PREC[case["precision"]], s),
                "smc_k_leapfrog")
        return out
    B.check(lib.smc_k_flow_leapfrog(st["dm"].h, case["hidden"], case["layers"], st["par"].data_ptr(), th.data_ptr(),
                                    p.data_ptr(), gr.data_ptr(), lp.data_ptr(), st["steps"].data_ptr(), case["eps"],
                                    N, N, st["z0"].data_ptr(), st["z1"].data_ptr(), st["dH"].data_ptr(),
                                    PREC[case["precision"]], s), "smc_k_flow_leapfrog")
    out.update(z0=st["z0"], z1=st["z1"], dH=st["dH"])
    return out


# ------------------------------------------------------------------ the work
def work(case):
    op, N = case["op"], case["particles"]
    if op == "normalise":   # log-weights in, weights out; an exponential each
        return {"bytes": 16.0 * N, "flops": 20.0 * N}
    if op == "resample":    # weights in, fixed-point weights and ancestors out
        return {"bytes": 20.0 * N, "flops": 4.0 * N}
    D = case["dim"]
    if op in ("flow_move", "flow_grad"):
        H, L = case["hidden"], case["layers"]
        Dh = D // 2
        mac = Dh * H + H * H + H * D          # one conditioner evaluation
        npar = L * (mac + 2 * H + D)
        if op == "flow_grad":   # forward, transposed products, weight gradients
            return {"bytes": 4.0 * (2 * npar + D * N) + 8.0 * N, "flops": 8.0 * L * mac * N}
        return {"bytes": 4.0 * (npar + D * D + 8 * D * N) + 28.0 * N,
                "flops": (4.0 * L * mac + 2.0 * D * D) * N * (case["steps"] + 1)}
    kind = case["model"]
    n = case.get("n", 0)
    grad = {"gauss": 2.0 * D * D, "logistic": 4.0 * n * D, "linear": 4.0 * n * D, "hier": 9.0 * D,
            "banana": 5.0 * D}[kind]
    end = {"gauss": 2.0 * D, "logistic": 2.0 * n * D, "linear": 2.0 * n * D, "hier": 8.0 * D, "banana": 4.0 * D}[kind]
    data = 4.0 * {"gauss": D * D, "logistic": n * D, "linear": n * D, "hier": 3 * D, "banana": 2}[kind]
    if op == "run":
        # jittered lengths: on average half of the first iteration's longest
        S = 0.5 * min(500.0, case["len0"] / case["eps"])
        total = N * case["runs"] * (0.53 if kind == "hier" else 1.0)
        per = S * (grad + 4.0 * D) + end + 10.0 * D
        return {"bytes": case["iters"] * total * (20.0 * D + 40.0) + data, "flops": case["iters"] * total * per}
    S = case["steps"] * (0.5 if case["ragged"] else 1.0)
    return {"bytes": 24.0 * D * N + 20.0 * N + data, "flops": N * (S * (grad + 4.0 * D) + end)}


# ------------------------------------------------------------------ 64 bits
def _target64(case, d):
    """log pi and its gradient at theta [D x N], in 64 bits."""
    kind, D = case.get("model", "gauss"), case["dim"]
    if kind == "gauss":
        def f(th):
            g = -(d["P"] @ (th - d["mu"][:, None]))
            return 0.5 * ((th - d["mu"][:, None]) * g).sum(0), g
        return f
    if kind in ("logistic", "linear"):
        X, y = d["X"], d["y"]

        def f(th, chunk=4096):
            lp = torch.zeros(th.shape[1], dtype=torch.float64, device="cuda")
            g = -th.clone()   # prior scale one
            for i in range(0, X.shape[0], chunk):
                Xc, yc = X[i:i + chunk], y[i:i + chunk, None]
                eta = Xc @ th
                if kind == "logistic":
                    lp += (yc * eta - torch.nn.functional.softplus(eta, threshold=1e9)).sum(0)
                    r = yc - torch.sigmoid(eta)
                else:
                    r = (yc - eta) * 4.0
                    lp += -0.5 * ((yc - eta) * 2.0).square().sum(0)
                g += Xc.T @ r
            lp += -0.5 * th.square().sum(0) - 0.5 * D * LOG_2PI
            if kind == "linear":
                lp += -0.5 * X.shape[0] * (LOG_2PI + 2.0 * math.log(0.5))
            return lp, g
        return f
    if kind == "hier":
        yb, ng, ss = d["ybar"][:, None], d["n_g"][:, None], d["ss"][:, None]
        const = -LOG_2PI - 0.5 * float(d["n_g"].sum()) * LOG_2PI - 0.5 * (D - 2) * LOG_2PI

        def f(th):
            mu, lt, eta = th[0:1], th[1:2], th[2:]
            tau = lt.exp()
            dev = yb - mu - tau * eta
            r = ng * dev
            g = torch.cat([r.sum(0, keepdim=True) - mu, (r * tau * eta).sum(0, keepdim=True) - lt, r * tau - eta])
            lp = (-0.5 * mu.square() - 0.5 * lt.square())[0] - (0.5 * (ng * dev.square() + ss) + 0.5 * eta.square()).sum(0)
            return lp + const, g
        return f

    def f(th):
        xo, xe = th[0::2], th[1::2]
        u = xe - 0.1 * (xo.square() - 10.0)
        g = torch.empty_like(th)
        g[0::2] = -xo / 10.0 + 0.2 * u * xo
        g[1::2] = -u
        lp = (-xo.square() / 20.0 - 0.5 * u.square()).sum(0)
        return lp - (D // 2) * (0.5 * (LOG_2PI + math.log(10.0)) + 0.5 * LOG_2PI), g
    return f


def _leapfrog64(f, th, p, steps, eps):
    """Each particle's own number of steps; returns theta, p, grad, log pi."""
    lp, g = f(th)
    for s in range(int(steps.max())):
        on = steps > s
        ph = p + 0.5 * eps * g
        t1 = th + eps * ph
        lp1, g1 = f(t1)
        p = torch.where(on, ph + 0.5 * eps * g1, p)
        th, g, lp = torch.where(on, t1, th), torch.where(on, g1, g), torch.where(on, lp1, lp)
    return th, p, g, lp


def _flow_layers(case, par):
    D, H, L = case["dim"], case["hidden"], case["layers"]
    Dh, o, out = D // 2, 0, []
    for _ in range(L):
        lay = []
        for rows, cols in ((H, Dh), (H, 1), (H, H), (H, 1), (D, H), (D, 1)):
            lay.append(par[o:o + rows * cols].reshape(rows, cols))
            o += rows * cols
        out.append(lay)
    return out


def _flow_st(lay, a, Dh):
    W1, b1, W2, b2, W3, b3 = lay
    o = W3 @ torch.tanh(W2 @ torch.tanh(W1 @ a + b1) + b2) + b3
    return 2.0 * torch.tanh(o[:Dh]), o[Dh:]


def _flow_fwd(layers, z):
    """theta = T(z) and log|det dT/dz|."""
    Dh, ld = z.shape[0] // 2, 0.0
    for l, lay in enumerate(layers):
        a, b = (z[:Dh], z[Dh:]) if l % 2 == 0 else (z[Dh:], z[:Dh])
        s, t = _flow_st(lay, a, Dh)
        b = b * s.exp() + t
        z = torch.cat([a, b]) if l % 2 == 0 else torch.cat([b, a])
        ld = ld + s.sum(0)
    return z, ld


def _flow_inv(layers, th):
    """z = T^-1(theta) and log|det dT^-1/dtheta|."""
    Dh, ld = th.shape[0] // 2, 0.0
    for l in range(len(layers) - 1, -1, -1):
        a, b = (th[:Dh], th[Dh:]) if l % 2 == 0 else (th[Dh:], th[:Dh])
        s, t = _flow_st(layers[l], a, Dh)
        b = (b - t) * (-s).exp()
        th = torch.cat([a, b]) if l % 2 == 0 else torch.cat([b, a])
        ld = ld - s.sum(0)
    return th, ld


def exact(case, seed):
    op = case["op"]
    if op in ("run", "resample"):
        # a run draws its own momenta and takes discrete decisions (ancestors,
        # step counts); ancestors and fixed-point weights are whole numbers
        return None
    if op == "normalise":
        lw = _logw(case, _gen(seed))
        lse = torch.logsumexp(lw, 0)
        W = (lw - lse).exp()
        return {"W": W, "lse": lse.reshape(1), "ess": (1.0 / W.square().sum()).reshape(1)}
    if op == "flow_grad":
        g = _gen(seed)
        par = _flow_params(case, g).double().requires_grad_()
        th = _randn(g, case["dim"], case["particles"]).float().double()
        W = torch.softmax(0.5 * _randn(g, case["particles"]), 0)
        z, ld = _flow_inv(_flow_layers(case, par), th)
        (W * (0.5 * z.square().sum(0) - ld)).sum().backward()
        return {"grad": par.grad}
    g, d, th, p, steps = _move_inputs(case, seed)
    f = _target64(case, d)
    th, p = th.double(), p.double()
    if op == "leapfrog":
        th, p, gr, lp = _leapfrog64(f, th, p, steps, case["eps"])
        return {"theta": th, "p": p, "grad": gr, "logpi": lp}
    layers = _flow_layers(case, _flow_params(case, g).double())

    def fz(z):
        z = z.detach().requires_grad_()
        t, ld = _flow_fwd(layers, z)
        lp, gt = f(t)
        # d/dz [log pi(T(z)) + log det] by the chain rule through T
        gz, = torch.autograd.grad((t * gt.detach()).sum() + ld.sum(), z)
        return (lp + ld).detach(), gz

    z0 = _flow_inv(layers, th)[0]
    z1, p, _, _ = _leapfrog64(fz, z0, p, steps, case["eps"])
    t1 = _flow_fwd(layers, z1)[0]
    lp, gr = f(t1)
    # the energy error of a trajectory is that of its own rounded gradients
    return {"theta": t1, "p": p, "grad": gr, "logpi": lp, "z0": z0, "z1": z1, "dH": None}
