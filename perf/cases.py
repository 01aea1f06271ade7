"""The work that a user of the sampler has it do, one case per kind of call and
size: whole inferences, batches of runs on a kept handle, and the step-level
calls that a program with its own loop makes.  Every input is made from the
case and the seed alone."""
import math

import numpy as np
import torch

from paper_2608_28514_gb300 import _native as nat
from paper_2608_28514_gb300 import workloads as W

DEV = "cuda"

# How each kind of case runs:
#   infer    ns_create_batch, ns_run, ns_result of every run, ns_destroy: a
#            program that wants the evidence and the posterior samples.
#   batch    a kept handle, ns_reset, ns_run (or ns_step for `iters`
#            iterations where a whole run takes minutes), the summaries and
#            the live sets.
#   slice    ns_slice_replace on a live set in the middle of a run.
#   cluster  ns_cluster of a live set.
#   select   ns_select_worst over several runs' live sets.
#   loglike  ns_loglike of many points (samples re-evaluated, a prior scan).
#   mlp      ns_mlp_loglike of a batch of candidates of the emulator network.
EMULATOR = "27-512-512-512-512-2000"


def listed():
    return [
        # the quick start: one sequential run (the paper's sampler setting) on a
        # 2-D Gaussian; latency of one walker is everything
        dict(name="infer_gauss2_m1", kind="infer", family="iso", d=2, sigma=0.5, box=5.0, runs=1, N=100, m=1),
        # the same setting as in the comparison study: 50 seeds side by side, one
        # walker each, 8-D unit Gaussian on [-7, 7]^8
        dict(name="infer_gauss8_m1_50runs", kind="infer", family="iso", d=8, sigma=1.0, box=7.0, runs=50, N=200, m=1),
        # one batched inference of the 10-D correlated Gaussian, m / N = 0.1
        dict(name="infer_corr10_m100", kind="infer", family="corr", d=10, sigma=1.0, box=10.0, runs=1, N=1000, m=100),
        # one multimodal inference with the cluster tree (4 modes in 5-D, depth 3)
        dict(name="infer_mixture5_m200_tree", kind="infer", family="mix", d=5, sigma=0.1, box=5.0, runs=1, N=2000,
             m=200, depth=3),
        # throughput: as many of those 10-D runs as fill the GPU, to convergence
        dict(name="batch_corr10_m100_608runs", kind="batch", family="corr", d=10, sigma=1.0, box=10.0, runs=608,
             N=1000, m=100, iters=0),
        # uneven runs in one call: d 2..30, N 100..2000, four likelihoods; the
        # first iterations (a whole batch takes seconds)
        dict(name="batch_mixed_256runs", kind="batch", family="mixed", d=30, sigma=1.0, box=7.0, runs=256, N=2000,
             m=100, iters=60),
        # the emulator likelihood: one inference at m / N = 0.1 in BF16 with the
        # FP32 re-evaluation, its first iteration (a whole run takes minutes)
        dict(name="batch_emulator27_m150", kind="batch", family="mlp", d=27, sigma=1.0, box=1.0, runs=1, N=1500,
             m=150, iters=1, precision=1, net=EMULATOR),
        # one replacement step for a caller's own loop, ragged sizes
        dict(name="slice_corr10_m100", kind="slice", family="corr", d=10, sigma=1.0, box=10.0, N=1000, m=100,
             spread=2.0),
        # the cluster tree of one live set at the depth the multimodal tests use
        dict(name="cluster_d10_N2000_depth6", kind="cluster", d=10, N=2000, depth=6, blobs=6, spread=0.02),
        # posterior samples of a run re-evaluated
        dict(name="loglike_corr10_1M", kind="loglike", family="corr", d=10, sigma=1.0, box=10.0, n=1000003),
        # emulator predictions for a large sample in BF16 on the tensor cores
        dict(name="mlp_bf16_155648", kind="mlp", n=155648, precision=1, net=EMULATOR),
        # and a moderate, ragged one at FP32 accuracy
        dict(name="mlp_fp32_3001", kind="mlp", n=3001, precision=2, net=EMULATOR),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(_log(rng, lo, hi)))))


def draw(rng):
    kind = rng.choice(["infer", "infer", "batch", "batch", "slice", "cluster", "select", "loglike", "mlp", "mlp"])
    family = rng.choice(["iso", "corr", "rosen", "mix"])
    box = {"iso": 7.0, "corr": 10.0, "rosen": 5.0, "mix": 5.0}[family]
    sigma = {"mix": 0.1}.get(family, 1.0)
    if kind == "infer":
        d = rng.randint(2, 8)
        N = _logint(rng, 60, 500)
        m = rng.choice([1, max(1, N // 20), max(1, N // 10)])
        return dict(kind=kind, family=family, d=d, sigma=sigma, box=box, runs=_logint(rng, 1, 40), N=N, m=m,
                    depth=rng.choice([0, 0, 3]) if family == "mix" else 0)
    if kind == "batch":
        if rng.random() < 0.25:
            return dict(kind=kind, family="mlp", d=27, sigma=1.0, box=1.0, runs=rng.randint(1, 2),
                        N=_logint(rng, 200, 1000), m=rng.randint(10, 90), iters=1, precision=rng.choice([1, 1, 2]),
                        net=EMULATOR)
        N = _logint(rng, 200, 2000)
        return dict(kind=kind, family=rng.choice([family, "mixed"]), d=rng.randint(2, 30), sigma=sigma, box=box,
                    runs=_logint(rng, 10, 600), N=N, m=max(1, min(256, int(N * rng.choice([0.01, 0.05, 0.1])))),
                    iters=rng.randint(4, 20))
    if kind == "slice":
        N = _logint(rng, 100, 4000)
        return dict(kind=kind, family=family, d=rng.randint(2, 32) if family != "rosen" else rng.randint(2, 10),
                    sigma=sigma, box=box, N=N, m=max(1, min(256, int(N * rng.choice([0.01, 0.05, 0.1])))),
                    spread=rng.uniform(1.0, 3.0))
    if kind == "cluster":
        return dict(kind=kind, d=rng.randint(2, 24), N=_logint(rng, 200, 4000), depth=rng.choice([0, 0, 1, 3, 4]),
                    blobs=rng.randint(1, 8), spread=rng.uniform(0.01, 0.05))
    if kind == "select":
        N = _logint(rng, 100, 65536)
        return dict(kind=kind, runs=_logint(rng, 1, 256), N=N, m=max(1, min(256, N // rng.choice([10, 20, 100]))))
    if kind == "loglike":
        return dict(kind=kind, family=family, d=rng.randint(2, 32), sigma=sigma, box=box, n=_logint(rng, 100, 1000000))
    return dict(kind="mlp", n=_logint(rng, 1, 40000) if rng.random() < 0.7 else _logint(rng, 1, 300),
                precision=rng.choice([1, 1, 2, 3]), net=EMULATOR)


# --------------------------------------------------------------------------
# Problems
# --------------------------------------------------------------------------
def _problem(family, d, sigma, box, seed):
    if family == "iso":
        r = np.random.default_rng([11, seed])
        p = W.gauss_iso(d, sigma, -box, box)
        p.mean = r.uniform(-0.1 * box, 0.1 * box, size=d)
        return p
    if family == "corr":
        return W.gauss_corr(d, seed, box=box)
    if family == "rosen":
        return W.rosenbrock(d, box=box)
    return W.mixture(d, seed, sigma=sigma, box=box)


_NETS = {}


def _emulator(net):
    """The network of a program: loaded once, whatever points it is asked for."""
    if net not in _NETS:
        _NETS[net] = W.mlp_emulator(1, widths=tuple(int(v) for v in net.split("-")))
    return _NETS[net]


def _runs(case, seed):
    """The runs of a case as ns_create_batch takes them, and its options."""
    fam, opt = case["family"], nat.ns_default_options(depth=int(case.get("depth", 0)))
    if fam == "mlp":
        opt.precision = int(case["precision"])
        p = _emulator(case["net"])
        return [(p, case["N"], case["m"], 5 * p.d, 1e-3, seed * 1000 + r) for r in range(case["runs"])], opt
    if fam == "mixed":
        # the sizes are the case's, the problems and the draws the seed's
        many = W.batched_runs(case["runs"], seed=1, d_hi=case["d"], n_lo=100, n_hi=max(101, case["N"]),
                              frac=case["m"] / case["N"])
        again = {W.GAUSS_ISO: lambda d, s: W.gauss_iso(d, 1.0, -7.0, 7.0), W.GAUSS_CORR: W.gauss_corr,
                 W.ROSENBROCK: lambda d, s: W.rosenbrock(d), W.MIXTURE: W.mixture}
        return [(again[p.kind](p.d, seed * 1000 + r), N, min(m, 256), 5 * p.d, 1e-3, seed * 1000 + r)
                for r, (p, N, m, _) in enumerate(many)], opt
    p = _problem(fam, case["d"], case["sigma"], case["box"], seed)
    return [(p, case["N"], case["m"], 5 * case["d"], 1e-3, seed * 1000 + r) for r in range(case["runs"])], opt


def _shell_points(p, family, n, spread, rng):
    """Unit-cube points as a live set in the middle of a run has them: uniform
    inside a likelihood contour about `spread` standard deviations out."""
    d, lo, span = p.d, np.asarray(p.lo), np.asarray(p.hi) - np.asarray(p.lo)
    if family == "rosen":
        th = rng.uniform(p.lo, p.hi, size=(40 * n, d))
        return ((th - lo) / span)[np.argsort(-_ll64(p, th))[:n]][rng.permutation(n)]
    out = np.empty((0, d))
    while len(out) < n:
        g = rng.standard_normal((2 * n, d))
        g *= (spread * math.sqrt(d) * rng.uniform(size=(2 * n, 1)) ** (1.0 / d)) / np.linalg.norm(g, axis=1, keepdims=True)
        if family == "corr":
            th = p.mean + np.linalg.solve(p.prec_chol.T, g.T).T
        elif family == "iso":
            th = p.mean + p.sigma * g
        else:
            th = p.centres[rng.integers(0, len(p.centres), size=2 * n)] + p.sigma * g
        u = (th - lo) / span
        out = np.concatenate([out, u[np.all((u > 0) & (u < 1), axis=1)]])
    return out[:n]


def _ll64(p, th):
    """log L in 64 bits."""
    if p.kind == W.GAUSS_ISO:
        return -0.5 * np.sum(((th - p.mean) / p.sigma) ** 2, axis=1)
    if p.kind == W.GAUSS_CORR:
        return -0.5 * np.sum(((th - p.mean) @ p.prec_chol) ** 2, axis=1)
    if p.kind == W.ROSENBROCK:
        return -np.sum((p.a - th[:, :-1]) ** 2 + p.b * (th[:, 1:] - th[:, :-1] ** 2) ** 2, axis=1)
    e = np.stack([-np.sum((th - c) ** 2, axis=1) / (2 * p.sigma**2) for c in p.centres])
    mx = e.max(axis=0)
    return mx + np.log(np.exp(e - mx).sum(axis=0)) - math.log(len(p.centres))


def _dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dtype)


# --------------------------------------------------------------------------
# prepare / run
# --------------------------------------------------------------------------
def prepare(case, seed):
    kind, seed = case["kind"], int(seed) % (1 << 31)
    rng = np.random.default_rng([seed, 3])
    if kind == "infer":
        runs, opt = _runs(case, seed)
        # room for the samples: dead points are the run's compression, at most
        # about 35 N over these families and sizes, and the last live points
        R, rows = len(runs), 60 * case["N"] + 8 * case["m"]
        return dict(kind=kind, runs=runs, opt=opt, samples=dict(
            dead_x=np.zeros((R, rows, case["d"]), np.float32), dead_l=np.zeros((R, rows), np.float32),
            dead_logw=np.zeros((R, rows), np.float64)))
    if kind == "batch":
        runs, opt = _runs(case, seed)
        return dict(kind=kind, h=nat.ns_create_batch(runs, opt), n=len(runs), iters=case["iters"])
    if kind == "slice":
        p = _problem(case["family"], case["d"], case["sigma"], case["box"], seed)
        d, N, m, n_steps = p.d, case["N"], case["m"], 5 * p.d
        n_pad = (N + 31) // 32 * 32
        u = _shell_points(p, case["family"], N, case["spread"], rng).astype(np.float32)
        ll = _ll64(p, p.lo + (p.hi - p.lo) * u.astype(np.float64)).astype(np.float32)
        order = np.argsort(ll, kind="stable")
        x = np.zeros((d, n_pad), np.float32)
        x[:, :N] = u.T
        chol = np.linalg.cholesky(np.atleast_2d(np.cov(u.T.astype(np.float64))) + 1e-12 * np.eye(d))
        f, i32 = torch.float32, torch.int32
        out = dict(new_x=torch.zeros(m, d, device=DEV), new_l=torch.zeros(m, device=DEV),
                   hist_l=torch.zeros(m, 64, device=DEV), hist_x=torch.zeros(m, 64, d, device=DEV),
                   hist_len=torch.zeros(m, dtype=i32, device=DEV),
                   evals=torch.zeros(m, dtype=torch.int64, device=DEV),
                   flags=torch.zeros(m, dtype=i32, device=DEV))
        scratch = torch.empty((nat.ns_slice_scratch_bytes(d, m, n_steps) + 3) // 4, dtype=f, device=DEV)
        return dict(kind=kind, args=(p, N, n_pad, m, n_steps, nat.ns_default_options(), seed, 7, _dev(x, f), _dev(ll, f),
                                     _dev(rng.choice(order[m:], size=m), i32), _dev(ll[order[:m]], f), _dev(chol, f),
                                     torch.zeros(N, dtype=i32, device=DEV)), out=out, scratch=scratch)
    if kind == "cluster":
        d, N, depth = case["d"], case["N"], case["depth"]
        n_pad, n_nodes = (N + 31) // 32 * 32, (1 << (depth + 1)) - 1
        x = np.zeros((d, n_pad), np.float32)
        x[:, :N] = _blobs(case, seed).T
        i32 = dict(dtype=torch.int32, device=DEV)
        out = dict(centres=torch.zeros(n_nodes, d, device=DEV), chol=torch.zeros(n_nodes, d, d, device=DEV),
                   chol64=torch.zeros(n_nodes, d, d, dtype=torch.float64, device=DEV),
                   logvol=torch.zeros(n_nodes, device=DEV), count=torch.zeros(n_nodes, **i32),
                   split=torch.zeros(n_nodes, **i32), mask=torch.zeros(n_nodes, **i32), cid=torch.zeros(N, **i32))
        scratch = torch.empty(nat.ns_cluster_scratch_bytes(N, n_pad, d), dtype=torch.uint8, device=DEV)
        return dict(kind=kind, args=(N, n_pad, d, _dev(x, torch.float32), nat.ns_default_options(depth=depth), seed, 3),
                    out=out, scratch=scratch)
    if kind == "select":
        ll = _select_input(case, seed)
        R, m = case["runs"], case["m"]
        return dict(kind=kind, ll=_dev(ll, torch.float32), m=m, seeds=[seed + r for r in range(R)],
                    out=dict(worst=torch.zeros(R, m, dtype=torch.int32, device=DEV), W=torch.zeros(R, m, device=DEV),
                             seed_slot=torch.zeros(R, m, dtype=torch.int32, device=DEV)))
    if kind == "loglike":
        p, u = _loglike_input(case, seed)
        return dict(kind=kind, p=p, x=u, out=torch.zeros(case["n"], device=DEV))
    p = _emulator(case["net"])
    nb = nat.ns_mlp_image_bytes(p)
    raw = torch.empty(nb + 1024, dtype=torch.uint8, device=DEV)
    o = -raw.data_ptr() % 1024
    image = raw[o:o + nb]
    nat.ns_mlp_pack(p, image)
    return dict(kind=kind, p=p, image=image, x=_mlp_input(case, seed), out=torch.zeros(case["n"], device=DEV),
                precision=case["precision"])


def _blobs(case, seed):
    """A live set over a few modes of uneven shape, in the unit cube."""
    r = np.random.default_rng([seed, 5])
    d, N, k = case["d"], case["N"], case["blobs"]
    c = r.uniform(0.2, 0.8, size=(k, d))
    sd = case["spread"] * np.exp(r.uniform(-0.7, 0.7, size=(k, d)))
    lab = r.integers(0, k, size=N)
    return np.clip(c[lab] + sd[lab] * r.standard_normal((N, d)), 0, 1).astype(np.float32)


def _select_input(case, seed):
    r = np.random.default_rng([seed, 6])
    # log L of a live set: chi^2-like, of a run's own scale
    scale = np.exp(r.uniform(0.0, 6.0, size=(case["runs"], 1)))
    return (-scale * r.chisquare(10, size=(case["runs"], case["N"]))).astype(np.float32)


def _loglike_input(case, seed):
    p = _problem(case["family"], case["d"], case["sigma"], case["box"], seed)
    g = torch.Generator(device=DEV).manual_seed(seed)
    # most points near the middle of the box, as samples are, the others over all of it
    u = torch.rand(case["n"], p.d, generator=g, device=DEV)
    s = torch.rand(case["n"], 1, generator=g, device=DEV)
    return p, (0.5 + (u - 0.5) * torch.where(s < 0.8, 0.3, 1.0)).contiguous()


def _mlp_input(case, seed):
    p = _emulator(case["net"])
    g = torch.Generator(device=DEV).manual_seed(seed)
    # candidates of a run: from prior-wide to posterior-narrow about the truth
    th = torch.from_numpy(p.mlp.theta_star).to(DEV, torch.float32)
    s = torch.exp(-4.6 * torch.rand(case["n"], 1, generator=g, device=DEV))
    u = torch.rand(case["n"], p.d, generator=g, device=DEV)
    return (th + (u - th) * s).clamp(0.0, 1.0).contiguous()


SCALARS = ("log_z", "log_z_err", "info")
COUNTS = ("n_dead", "n_evals", "n_iter", "n_relaxed", "n_reeval", "n_capped", "status")


def _table(res):
    out = {k: np.array([r[k] for r in res], dtype=np.float64) for k in SCALARS}
    out.update({k: np.array([r[k] for r in res], dtype=np.int64) for k in COUNTS})
    return out


def run(state):
    kind = state["kind"]
    if kind == "infer":
        h = nat.ns_create_batch(state["runs"], state["opt"])
        nat.ns_run(h, check=False)
        res = [nat.ns_result(h, r) for r in range(len(state["runs"]))]
        nat.ns_destroy(h)
        for k, into in state["samples"].items():
            for r, one in enumerate(res):
                into[r, :one["n_dead"]] = one[k]
        return {**_table(res), **state["samples"]}
    if kind == "batch":
        h = state["h"]
        nat.ns_reset(h)
        if state["iters"]:
            nat.ns_step(h, state["iters"])
        else:
            nat.ns_run(h)
        out = _table([nat.ns_summary(h, r) for r in range(state["n"])])
        for k in ("live_x", "live_l"):
            out[k] = np.concatenate([nat.ns_copy_run_buffer(h, r, k) for r in range(state["n"])])
        return out
    if kind == "slice":
        nat.ns_slice_replace(*state["args"], **state["out"], dir_scratch=state["scratch"])
        return state["out"]
    if kind == "cluster":
        nat.ns_cluster(*state["args"], **state["out"], scratch=state["scratch"])
        return state["out"]
    if kind == "select":
        nat.ns_select_worst(state["ll"], state["m"], state["seeds"], 5, **state["out"])
        return state["out"]
    if kind == "loglike":
        nat.ns_loglike(state["p"], state["x"], state["out"])
        return state["out"]
    nat.ns_mlp_loglike(state["p"], state["image"], state["x"], state["out"], precision=state["precision"])
    return state["out"]


# --------------------------------------------------------------------------
# work / exact
# --------------------------------------------------------------------------
def _eval_flops(family, d):
    return {"iso": 4 * d, "corr": d * (d + 1) + 2 * d, "rosen": 9 * d, "mix": 16 * d + 40,
            "mixed": (d * (d + 1) + 31 * d + 40) / 4}.get(family, 0) + 2 * d


def _mlp_flops(net):
    w = [int(v) for v in net.split("-")]
    return 2 * sum(a * b for a, b in zip(w[:-1], w[1:]))


def work(case):
    kind, d = case["kind"], case.get("d", 0)
    if kind in ("infer", "batch"):
        R, N, m = case["runs"], case["N"], case["m"]
        dm = d if case["family"] != "mixed" else (2 + d) / 2
        if case.get("iters"):
            iters = case["iters"]
        else:  # compression from the prior to the stopping rule, about (H + 7) N / m
            h = dm * max(0.5, math.log(2 * case["box"] / (4.13 * case["sigma"] * (0.32 if case["family"] == "corr" else 1))))
            iters = (h + 7) * N / m
        # a slice step takes about 6 evaluations: two ends that fail, one
        # expansion or two, the shrink draws
        evals = R * (N + iters * m * 5 * dm * 6)
        f = _mlp_flops(case["net"]) if case["family"] == "mlp" else _eval_flops(case["family"], dm)
        # samples out (x, log L, weight), once each
        return {"bytes": R * (N + (0 if case.get("iters") else iters * m)) * (4 * dm + 12), "flops": evals * f}
    if kind == "slice":
        return {"bytes": 4 * case["N"] + 4 * case["m"] * (2 * d + 8 + 4 * (d + 1)),
                "flops": case["m"] * 5 * d * 6 * _eval_flops(case["family"], d)}
    if kind == "cluster":
        N, lv = case["N"], case["depth"]
        # per level: ten Lloyd passes of two distances, the covariance
        return {"bytes": 4 * N * (d + 1), "flops": N * d * d + lv * N * (10 * 6 * d + d * d)}
    if kind == "select":
        return {"bytes": case["runs"] * 4 * (case["N"] + 3 * case["m"]), "flops": case["runs"] * case["N"]}
    if kind == "loglike":
        return {"bytes": case["n"] * 4 * (d + 1), "flops": case["n"] * _eval_flops(case["family"], d)}
    w = [int(v) for v in case["net"].split("-")]
    return {"bytes": case["n"] * 4 * (w[0] + 1) + 2 * sum(a * b for a, b in zip(w[:-1], w[1:])),
            "flops": case["n"] * _mlp_flops(case["net"])}


def exact(case, seed):
    kind, seed = case["kind"], int(seed) % (1 << 31)
    if kind == "select":
        w = np.sort(_select_input(case, seed).astype(np.float64), axis=1, kind="stable")[:, :case["m"]]
        return dict(worst=None, W=torch.from_numpy(w.copy()), seed_slot=None)
    if kind == "loglike":
        p, u = _loglike_input(case, seed)
        th = p.lo + (p.hi - p.lo) * u.cpu().numpy().astype(np.float64)
        return torch.from_numpy(_ll64(p, th))
    if kind == "cluster" and case["depth"] == 0:
        x = _blobs(case, seed).astype(np.float64)
        d = x.shape[1]
        c = np.atleast_2d(np.cov(x.T, bias=True))
        L = np.linalg.cholesky(c + 1e-10 * np.trace(c) / d * np.eye(d))[None]
        return dict(centres=torch.from_numpy(x.mean(axis=0)[None]), chol=torch.from_numpy(L), chol64=torch.from_numpy(L),
                    logvol=None, count=None, split=None, mask=None, cid=None)
    if kind == "mlp":
        p = _emulator(case["net"])
        h = _mlp_input(case, seed).double()
        n_layers = len(p.mlp.weights)
        data, sig = (torch.from_numpy(np.asarray(a, dtype=np.float32)).to(DEV).double()
                     for a in (p.mlp.data, p.mlp.sigma_out))
        out = torch.empty(len(h), dtype=torch.float64, device=DEV)
        for i0 in range(0, len(h), 8192):
            a = h[i0:i0 + 8192]
            for i, (Wi, Bi) in enumerate(zip(p.mlp.weights, p.mlp.biases)):
                a = a @ torch.from_numpy(Wi).to(DEV).double().T + torch.from_numpy(Bi).to(DEV).double()
                if i + 1 < n_layers:
                    a = a * torch.sigmoid(a)
            out[i0:i0 + 8192] = -0.5 * (((a - data) / sig) ** 2).sum(dim=1)
        return out
    return None
