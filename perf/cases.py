"""Timed workloads of the sparsity-path-analysis library, through its public Python API.

Each case is one call (or one forward and backward) that a user of the package makes: a
whole SMC sweep over the prior scale for one hit region (`Region.run`), a prepared batch of
regions (`Batch.run`), the particle log-likelihood and its gradient on device tensors, and
the MAP path. Sizes come from `synth.WORKLOADS`, from the batched regions' ranges and from
the tests. Inputs are synthetic regions of the package's own generator.

    listed()             the fixed cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  the region(s), schedule and device buffers a program has before the call
    run(state)           one call and all its outputs
    work(case)           bytes and operations that one call cannot do without
    exact(case, seed)    the outputs in 64 bits, where they are deterministic functions
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1106_0322_gb300 as spa
from paper_1106_0322_gb300 import synth

CAUSAL = (0.3, 0.5, -0.4)


def listed():
    return [
        # the smallest complete sweep (the tutorial-sized region): launches and latency count
        dict(name="sweep_rw_plain_small", kind="sweep", move="rw", precision="split_bf16", n=200, p=10, N=1024, T=50,
             M=5, nu=1.0, rho=0.9, init="prior_is", burn_in=0, descend=False, map_path=False),
        # the flagship: one hit region with random-walk moves, sparse to diffuse
        dict(name="sweep_rw_hit_region", kind="sweep", move="rw", precision="split_bf16", n=2000, p=200, N=8192, T=200,
             M=10, nu=1.0, rho=0.95, init="prior_is", burn_in=0, descend=False, map_path=False),
        # the largest region and particle count of the package's workloads, a shorter schedule
        dict(name="sweep_rw_split_large", kind="sweep", move="rw", precision="split_bf16", n=5000, p=500, N=16384, T=20,
             M=10, nu=1.0, rho=0.95, init="prior_is", burn_in=0, descend=False, map_path=False),
        # the paper's direction (diffuse to sparse, MCMC start) under the double-exponential
        # prior, with odd sizes, recording each step's best particle for the MAP path
        dict(name="sweep_rw_ragged_de", kind="sweep", move="rw", precision="split_bf16", n=1859, p=183, N=5003, T=40,
             M=5, nu=math.inf, rho=0.95, init="resample_move", burn_in=3, descend=True, map_path=True),
        # the hit region with gradient-driven moves
        dict(name="sweep_mala_hit_region", kind="sweep", move="mala", precision="split_bf16", n=2000, p=200, N=8192,
             T=100, M=5, nu=2.0, rho=0.95, init="prior_is", burn_in=0, descend=False, map_path=False),
        # gradient-driven moves on a mid-sized region of the batched workload's range, odd sizes
        dict(name="sweep_mala_mid_ragged", kind="sweep", move="mala", precision="split_bf16", n=1234, p=77, N=4096,
             T=60, M=5, nu=4.0, rho=0.9, init="prior_is", burn_in=0, descend=False, map_path=False),
        # the paper's own kernel on its 18q-shaped region, a short schedule
        dict(name="sweep_site_paper_18q", kind="sweep", move="site", precision="split_bf16", n=1859, p=184, N=8192, T=6,
             M=5, nu=4.0, rho=0.95, init="resample_move", burn_in=1, descend=True, map_path=False),
        # the plain FP32 option, for users who want no split-BF16 operand
        dict(name="sweep_rw_fp32", kind="sweep", move="rw", precision="fp32", n=1000, p=100, N=4096, T=30, M=5, nu=1.0,
             rho=0.95, init="prior_is", burn_in=0, descend=False, map_path=False),
        # uneven regions side by side in one prepared batch
        dict(name="batch_mala", kind="batch", move="mala", R=8, n_lo=1000, n_hi=5000, p_lo=20, p_hi=500, N=4096, T=20,
             M=5),
        # the log-likelihood of a few particles: one call's latency
        dict(name="loglik_small", kind="loglik", precision="split_bf16", n=500, p=50, N=128),
        # log-likelihood and gradient of many particles as a differentiable torch function
        dict(name="grad_large", kind="grad", precision="split_bf16", n=5000, p=500, N=4096),
        # the MAP path from given starts on the paper's small data set's shape
        dict(name="map_path_paper_small", kind="map", n=500, p=50, T=64, nu=1.0),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# A drawn case costs no more than the largest listed one of its kind: operations of the
# likelihood (and adjoint) contractions, or coordinate updates x individuals.
_MOST = {"rw": 1.3e13, "mala": 1.2e13, "site": 1.5e11, "fp32": 7e10, "batch": 2e13, "loglik": 8e10, "grad": 4e10}


def draw(rng):
    kind = rng.choice(["rw", "rw", "rw", "mala", "mala", "site", "fp32", "batch", "loglik", "grad", "map"])
    while True:
        if kind in ("rw", "mala", "fp32"):
            c = dict(kind="sweep", move="mala" if kind == "mala" else "rw",
                     precision="fp32" if kind == "fp32" else "split_bf16", n=_log_int(rng, 150, 5000),
                     p=_log_int(rng, 5, 500), N=_log_int(rng, 256, 16384), T=rng.randint(5, 60), M=rng.randint(1, 10),
                     nu=rng.choice([1.0, 2.0, 4.0, 16.0, math.inf]), rho=round(rng.uniform(0.8, 0.97), 3),
                     init="prior_is", burn_in=0, descend=False, map_path=False)
            if rng.random() < 0.25:
                c.update(init="resample_move", burn_in=rng.randint(1, 4), descend=True, map_path=rng.random() < 0.5)
        elif kind == "site":
            c = dict(kind="sweep", move="site", precision="split_bf16", n=_log_int(rng, 150, 1900),
                     p=_log_int(rng, 5, 200), N=_log_int(rng, 512, 8192), T=rng.randint(3, 12), M=rng.randint(1, 5),
                     nu=rng.choice([1.0, 4.0]), rho=round(rng.uniform(0.8, 0.97), 3), init="resample_move",
                     burn_in=rng.randint(0, 2), descend=True, map_path=False)
        elif kind == "batch":
            n_lo, p_lo = _log_int(rng, 200, 2000), _log_int(rng, 10, 100)
            c = dict(kind="batch", move=rng.choice(["mala", "rw"]), R=rng.randint(2, 8), n_lo=n_lo,
                     n_hi=min(5000, n_lo * rng.randint(1, 4)), p_lo=p_lo, p_hi=min(500, p_lo * rng.randint(1, 6)),
                     N=_log_int(rng, 512, 4096), T=rng.randint(5, 20), M=rng.randint(1, 5))
        elif kind in ("loglik", "grad"):
            c = dict(kind=kind, precision=rng.choice(["split_bf16", "split_bf16", "fp32"]), n=_log_int(rng, 150, 5000),
                     p=_log_int(rng, 5, 500), N=_log_int(rng, 64, 16384))
        else:
            c = dict(kind="map", n=_log_int(rng, 150, 600), p=_log_int(rng, 5, 60), T=rng.randint(8, 64),
                     nu=rng.choice([1.0, 4.0]))
        if kind == "map" or _cost(c) <= _MOST[kind]:
            return c


def _regions_sizes(case):
    """The uneven (n, p) of a batch: even n spread over [n_lo, n_hi], p over [p_lo, p_hi]."""
    R = case["R"]
    out = []
    for r in range(R):
        f, g = (r + 0.5) / R, ((r * 5) % R + 0.5) / R
        out.append((int(case["n_lo"] + f * (case["n_hi"] - case["n_lo"])) // 2 * 2,
                    int(case["p_lo"] + g * (case["p_hi"] - case["p_lo"]))))
    return out


def _evaluations(case):
    """Likelihood evaluations of a sweep: the start's, then one a move."""
    return 1 + case["M"] * (case["T"] + case.get("burn_in", 0))


def _cost(case):
    return work(case)["flops"]


def work(case):
    k = case["kind"]
    if k == "sweep":
        n, p, N, T = case["n"], case["p"], case["N"], case["T"]
        per = 2.0 * N * n * p  # one contraction of all particles with the genotypes
        if case["move"] == "site":
            # a cycle of p updates changes the n linear predictors of a particle p times
            flops = per + 2.0 * N * n * p * case["M"] * (T + case["burn_in"])
        else:
            flops = per * _evaluations(case) * (2.0 if case["move"] == "mala" else 1.0)
        return {"bytes": float(n * p + n + T * (p * 6 + 3) * 8 + T), "flops": flops}
    if k == "batch":
        b = f = 0.0
        for n, p in _regions_sizes(case):
            f += 2.0 * case["N"] * n * p * (1 + case["M"] * case["T"]) * (2.0 if case["move"] == "mala" else 1.0)
            b += n * p + n + case["T"] * (p * 6 + 3) * 8 + case["T"]
        return {"bytes": b, "flops": f}
    if k in ("loglik", "grad"):
        n, p, N = case["n"], case["p"], case["N"]
        g = 1 if k == "grad" else 0
        return {"bytes": float(n * p + n + 4 * N * p + 8 * N + g * 4 * N * p), "flops": 2.0 * N * n * p * (1 + g)}
    # MAP path: at least one solve a step, each at least one evaluation of the two products
    return {"bytes": float(case["n"] * case["p"] + case["n"] + 8 * case["T"] * (case["p"] + 2)),
            "flops": 4.0 * case["T"] * case["n"] * case["p"]}


def _schedule(case):
    return synth.geometric_schedule(case["T"], sparse_to_diffuse=not case.get("descend", False))


def _particles(case, seed):
    """Sparse Laplace particles of moderate scale, with some exact zeros, on the device."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    N, p = case["N"], case["p"]
    u = torch.rand((N, p), generator=g, device="cuda", dtype=torch.float32) - 0.5
    B = -0.1 * torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp(max=0.49999))
    B[torch.rand((N, p), generator=g, device="cuda") < 0.05] = 0.0
    return B.contiguous()


def _region(case, seed, rho=0.95):
    return synth.make_region(case["n"], case["p"], case.get("rho", rho), CAUSAL, seed)


def prepare(case, seed):
    k = case["kind"]
    if k == "sweep":
        reg = _region(case, seed)
        cfg = spa.make_config(move=case["move"], precision=case["precision"], init=case["init"],
                              burn_in_steps=case["burn_in"], map_path=case["map_path"])
        return dict(case=case, region=spa.Region(reg.G, reg.y, case["nu"], config=cfg), schedule=_schedule(case),
                    seed=seed + 1)
    if k == "batch":
        regions = []
        for r, (n, p) in enumerate(_regions_sizes(case)):
            reg = synth.make_region(n, p, 0.8 + 0.02 * (r % 8), CAUSAL[: 1 + r % 3], 100 * seed + r)
            regions.append(spa.Region(reg.G, reg.y, (1.0, 2.0, 4.0, 16.0)[r % 4], config=spa.make_config(move=case["move"])))
        R = len(regions)
        batch = spa.Batch(regions, [_schedule(case)] * R, [case["N"]] * R, [case["M"]] * R,
                          [seed + 1 + r for r in range(R)])
        return dict(case=case, regions=regions, batch=batch)
    reg = _region(case, seed)
    if k == "map":
        rng = np.random.default_rng(seed)
        best = rng.laplace(0.0, 0.1, size=(case["T"], case["p"])).astype(np.float32)
        return dict(case=case, region=spa.Region(reg.G, reg.y, case["nu"]), best=best,
                    schedule=synth.geometric_schedule(case["T"], -4.0, 0.0, sparse_to_diffuse=False))
    region = spa.Region(reg.G, reg.y, 1.0, config=spa.make_config(precision=case["precision"]))
    B = _particles(case, seed)
    if k == "loglik":
        return dict(case=case, region=region, B=B, out=torch.empty(case["N"], dtype=torch.float64, device="cuda"))
    return dict(case=case, region=region, B=B.requires_grad_(True))


def run(state):
    case = state["case"]
    k = case["kind"]
    if k == "sweep":
        return state["region"].run(state["schedule"], case["N"], case["M"], state["seed"])
    if k == "batch":
        return state["batch"].run()
    if k == "map":
        modes, logpost = state["region"].map_path_given(state["schedule"], state["best"], max_em=100)
        return {"map": modes, "logpost": logpost}
    if k == "loglik":
        state["region"].loglik_device(state["B"], state["out"], torch.cuda.current_stream().cuda_stream)
        return {"loglik": state["out"]}
    ll = spa.loglik_autograd(state["B"], state["region"])
    (g,) = torch.autograd.grad(ll.sum(), state["B"])
    return {"loglik": ll.detach(), "grad": g}


def exact(case, seed):
    """The log-likelihood and its gradient in 64 bits. A sweep's and a MAP path's outputs follow
    from many accept or convergence decisions and have no such value."""
    if case["kind"] not in ("loglik", "grad"):
        return None
    reg = _region(case, seed)
    G = torch.from_numpy(reg.G).cuda().double()
    y = torch.from_numpy(reg.y).cuda().double()
    X = (G - G.mean(0)) / G.std(0, unbiased=False)
    B = _particles(case, seed).double()
    ll, grad = [], []
    for i in range(0, B.shape[0], 2048):
        eta = B[i : i + 2048] @ X.T
        ll.append(eta @ y - torch.logaddexp(eta, torch.zeros_like(eta)).sum(1))
        if case["kind"] == "grad":
            grad.append((y - torch.sigmoid(eta)) @ X)
    out = {"loglik": torch.cat(ll)}
    if case["kind"] == "grad":
        out["grad"] = torch.cat(grad)
    return out
