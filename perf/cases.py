"""The force evaluations that users of this library wait for, as measurable cases.

A case is a dict of plain values; ``prepare`` makes what a program has in hand before the call
(particles on the GPU, a context with its parameters), ``run`` is one call of a public entry
point and returns everything that it computes, ``work`` the operations and bytes the call cannot
do without, ``exact`` the plain direct sum in 64 bits where that takes seconds.

Sizes and parameters are those of the benchmark's workloads, the crossover table and the tests
(odd and ragged sizes among them); the models are the benchmark's Plummer spheres and gamma = 1.5
cusps.  The order p, eps, the leaf size and the direct-sum threshold p2p_c are the parameters a
user tunes, so they vary over the range in which the tuner looks.
"""
import math

import numpy as np
import torch

from paper_1405_2255_gb300 import gb3fmm as g
from paper_1405_2255_gb300 import inputs

DEV = "cuda:0"


def listed():
    return [
        # an embedded small system: a plugin that may not allocate evaluates a few thousand
        # bodies per call; latency and launches are all there is
        {"name": "noalloc_2k", "kind": "noalloc", "model": "plummer", "n": 2039, "p": 8, "eps": 1e-6, "leaf": 32,
         "c": 4.0, "mac": 0, "mixed": True},
        # a star cluster in the making: the smallest system for which the FMM beats direct summation
        {"name": "mixed_10k", "kind": "evaluate", "model": "plummer", "n": 10000, "p": 14, "eps": 2.3e-7, "leaf": 48,
         "c": 1.0, "mac": 0, "mixed": True},
        # an ordinary cluster with the library's defaults for leaf size, order and threshold
        {"name": "mixed_100k_default", "kind": "evaluate", "model": "plummer", "n": 100003, "p": 8, "eps": 1e-6,
         "leaf": 64, "c": 8.0, "mac": 0, "mixed": True},
        # the benchmark's workload: a Plummer sphere of 1e6 at rms 1e-7
        {"name": "mixed_1m", "kind": "evaluate", "model": "plummer", "n": 1000000, "p": 14, "eps": 2.3e-7, "leaf": 80,
         "c": 1.0, "mac": 0, "mixed": True},
        # the largest: a galactic nucleus, a cusp with a central point mass (deep tree)
        {"name": "cusp_3m", "kind": "evaluate", "model": "cusp", "n": 2999999, "p": 14, "eps": 2.6e-7, "leaf": 80,
         "c": 1.0, "mac": 0, "mixed": True},
        # an ensemble of independent clusters of 1e3 .. 1e5 stars in one forest
        {"name": "ensemble_48", "kind": "ensemble", "model": "plummer", "n": 48, "p": 14, "eps": 3.6e-7, "leaf": 48,
         "c": 1.0, "mac": 0, "mixed": True},
        # block time steps: a few per cent of the particles are active, the tree is re-cycled
        {"name": "block_step_1m", "kind": "block", "model": "plummer", "n": 1000000, "p": 14, "eps": 2.3e-7,
         "leaf": 80, "c": 1.0, "mac": 0, "mixed": True, "fraction": 0.03},
        # a Hermite-type integrator's step: forces with the tidal tensor
        {"name": "tidal_150k", "kind": "tidal", "model": "plummer", "n": 150001, "p": 14, "eps": 2.3e-7, "leaf": 64,
         "c": 1.0, "mac": 0, "mixed": True},
        # the paper's Table 2 row (p = 10, eps = 10^-6.25, the f criterion) in full FP64
        {"name": "fp64_100k_f", "kind": "evaluate", "model": "plummer", "n": 100000, "p": 10, "eps": 5.623e-7,
         "leaf": 64, "c": 1.0, "mac": 1, "mixed": False},
        # FP64 at the reference accuracy: what the mixed mode is checked against
        {"name": "fp64_cusp_60k", "kind": "evaluate", "model": "cusp", "n": 60013, "p": 14, "eps": 3e-7, "leaf": 80,
         "c": 1.0, "mac": 0, "mixed": False},
        # the parity configuration of the tests and of a small production check: 4096 bodies, FP64
        {"name": "fp64_4k", "kind": "evaluate", "model": "plummer", "n": 4096, "p": 6, "eps": 1e-6, "leaf": 32,
         "c": 1.0, "mac": 0, "mixed": False},
        # the truth sample of the parameter tuner: 4096 sinks against every particle in FP64
        {"name": "direct_4096_300k", "kind": "direct", "model": "plummer", "n": 300000, "sinks": 4096, "f": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mixed", "mixed", "mixed", "fp64", "fp64", "ensemble", "block", "tidal", "direct", "noalloc"])
    model = rng.choice(["plummer", "plummer", "cusp"])
    if kind == "direct":
        n = _log_int(rng, 4000, 300000)
        return {"kind": "direct", "model": model, "n": n, "sinks": min(n, _log_int(rng, 500, 4096)),
                "f": rng.random() < 0.3}
    if kind == "noalloc":
        return {"kind": "noalloc", "model": model, "n": _log_int(rng, 300, 8192), "p": rng.randint(6, 10),
                "eps": 10 ** rng.uniform(-6.0, -5.0), "leaf": rng.randint(28, 64), "c": rng.choice([4.0, 8.0]),
                "mac": rng.choice([0, 0, 1]), "mixed": rng.random() < 0.7}
    c = {"kind": "evaluate", "model": model, "p": rng.randint(10, 16), "leaf": rng.randint(32, 96),
         "eps": 10 ** rng.uniform(-6.7, -5.5), "c": rng.choice([1.0, 1.0, 2.0, 4.0]), "mac": 0, "mixed": True}
    if kind == "mixed":
        c["n"] = _log_int(rng, 3000, 2000000)
    elif kind == "fp64":
        c.update(n=_log_int(rng, 1000, 60000), mixed=False, p=rng.randint(4, 14), leaf=rng.randint(16, 80),
                 mac=rng.choice([0, 0, 1]), eps=10 ** rng.uniform(-6.3, -5.0))
    elif kind == "ensemble":
        c.update(kind="ensemble", model="plummer", n=rng.randint(2, 60), leaf=rng.randint(32, 64))
    elif kind == "block":
        c.update(kind="block", n=_log_int(rng, 20000, 1000000), fraction=round(10 ** rng.uniform(-2.5, -0.5), 4))
    else:
        c.update(kind="tidal", n=_log_int(rng, 5000, 150000))
    return c


def _particles(case, seed):
    """Host arrays; an ensemble also has its offsets."""
    s = inputs.BASE_SEED + 7919 * (int(seed) % 1000003)
    if case["kind"] == "ensemble":
        sizes = inputs.ensemble_sizes(case["n"], 20140509 + case["n"])  # the sizes are the case's, not the seed's
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        x = np.empty((off[-1], 3))
        mu = np.empty(off[-1])
        for k, n in enumerate(sizes):
            sk = inputs.system_seed(s, k)
            x[off[k]:off[k + 1]] = inputs.plummer(int(n), sk)[0]
            mu[off[k]:off[k + 1]] = inputs.kroupa_masses(int(n), sk)
        return x, mu, off
    x, mu = (inputs.dehnen if case["model"] == "cusp" else inputs.plummer)(case["n"], s)
    return x, mu, None


def _active(case, x, seed):
    """The active particles of a block step: the innermost ones (short time steps) and a few others."""
    r = np.linalg.norm(x, axis=1)
    k = max(1, int(0.8 * case["fraction"] * len(r)))
    a = r <= np.partition(r, k - 1)[k - 1]
    a |= inputs.uniforms(int(seed), 11, len(r)) < 0.2 * case["fraction"]
    return a


def _drift(x, seed):
    """Positions a short time after the tree was built."""
    d = np.stack([inputs.uniforms(int(seed), 12 + k, len(x)) - 0.5 for k in range(3)], axis=1)
    return x + 2e-4 * d * (0.1 + np.linalg.norm(x, axis=1, keepdims=True))


def _params(case):
    return {"p": case["p"], "eps": case["eps"], "leaf_size": case["leaf"], "p2p_c": case["c"], "mac": case["mac"],
            "precision": g.FMM_PREC_MIXED if case["mixed"] else g.FMM_PREC_FP64}


def _sinks(case, seed):
    return np.sort(np.random.default_rng(int(seed)).choice(case["n"], case["sinks"], replace=False)).astype(np.int64)


def prepare(case, seed):
    g.load()
    x, mu, off = _particles(case, seed)
    st = {"kind": case["kind"], "x": torch.from_numpy(x).to(DEV), "mu": torch.from_numpy(mu).to(DEV)}
    if case["kind"] == "direct":
        st.update(ctx=g.Context(), sinks=torch.from_numpy(_sinks(case, seed)).to(DEV), f=case["f"])
        return st
    if case["kind"] == "noalloc":
        params = g.fmm_default_params()
        for k, v in _params(case).items():
            setattr(params, k, v)
        st["params"] = params
        return st
    st["ctx"] = g.Context(**_params(case))
    if case["kind"] == "ensemble":
        st.update(off=off, G=np.ones(len(off) - 1))
    if case["kind"] == "block":
        # the last full step, whose tree the block step re-cycles
        st["ctx"].fmm_evaluate(st["x"], st["mu"])
        x1 = _drift(x, seed)
        st.update(x=torch.from_numpy(x1).to(DEV), active=torch.from_numpy(_active(case, x1, seed).astype(np.uint8)).to(DEV),
                  psi=torch.full((len(mu),), float("nan"), dtype=torch.float64, device=DEV),
                  acc=torch.full((len(mu), 3), float("nan"), dtype=torch.float64, device=DEV))
    return st


def run(st):
    kind = st["kind"]
    if kind == "evaluate":
        return st["ctx"].fmm_evaluate(st["x"], st["mu"])
    if kind == "ensemble":
        return st["ctx"].fmm_evaluate_batch(st["off"], st["x"], st["mu"], st["G"])
    if kind == "block":
        return st["ctx"].fmm_evaluate_active(st["x"], st["mu"], st["active"], psi=st["psi"], acc=st["acc"],
                                             reuse_tree=True)
    if kind == "tidal":
        return st["ctx"].fmm_evaluate_active(st["x"], st["mu"], tidal=True)
    if kind == "noalloc":
        return g.fmm_evaluate_noalloc(st["x"], st["mu"], params=st["params"])
    return st["ctx"].fmm_direct(st["x"], st["mu"], sinks=st["sinks"], want_f=st["f"])


def work(case):
    """Bytes: positions and masses in, potential and acceleration out (FP64), each once.  Flops: 20
    per direct pair; an FMM evaluation has about 84 leaf_size pairs per particle and 230 / leaf_size
    M2L interactions of 4.2 p^3 flops (the lists of the benchmark's sphere at its accuracy)."""
    n = case["n"]
    if case["kind"] == "direct":
        s = case["sinks"]
        return {"bytes": 32.0 * n + (40.0 + 8.0 * case["f"]) * s, "flops": 20.0 * n * s}
    if case["kind"] == "ensemble":
        n = int(inputs.ensemble_sizes(n, 20140509 + n).sum())
    sinks = n * case.get("fraction", 1.0)
    near = min(84.0 * case["leaf"], n - 1.0) * (60.0 if case["kind"] == "tidal" else 20.0)
    far = 230.0 / case["leaf"] * 4.2 * case["p"] ** 3
    return {"bytes": 32.0 * n + (80.0 if case["kind"] == "tidal" else 32.0) * sinks, "flops": sinks * (near + far)}


def _direct(xs, x, mu, tidal=False, f=False):
    """Potential, acceleration [, tidal tensor | f] of the sinks xs by plain summation in 64 bits."""
    psi, acc, more = [], [], []
    chunk = max(1, 6000000 // max(1, len(x)))
    for b in range(0, len(xs), chunk):
        d = x.T[:, None, :] - xs[b:b + chunk].T[:, :, None]
        r2 = (d[0] * d[0]).addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        ri = torch.where(r2 > 0, torch.rsqrt(r2), torch.zeros((), dtype=torch.float64, device=x.device))
        q = ri * mu
        psi.append(q.sum(1))
        if f:
            more.append((q * ri).sum(1))
        ri *= ri
        q *= ri
        acc.append(torch.einsum("dij,ij->id", d, q))
        if tidal:
            tr = q.sum(1)
            q *= ri
            t = [3.0 * (q * d[i] * d[j]).sum(1) - (tr if i == j else 0.0) for i in range(3) for j in range(i, 3)]
            more.append(torch.stack(t, 1))
    out = [torch.cat(psi), torch.cat(acc)]
    return out + [torch.cat(more)] if tidal or f else out


def exact(case, seed):
    x, mu, off = _particles(case, seed)
    if case["kind"] == "ensemble":
        pairs = float((np.diff(off).astype(float) ** 2).sum())
    else:
        pairs = float(case["n"]) * (case["sinks"] if case["kind"] == "direct" else
                                    1.3 * case["fraction"] * case["n"] if case["kind"] == "block" else case["n"])
    if pairs > (3e10 if case["kind"] == "tidal" else 4e10):
        return None
    if case["kind"] == "block":
        x = _drift(x, seed)
    xt, mt = torch.from_numpy(x).to(DEV), torch.from_numpy(mu).to(DEV)
    if case["kind"] == "direct":
        return tuple(_direct(xt[torch.from_numpy(_sinks(case, seed)).to(DEV)], xt, mt, f=case["f"]))
    if case["kind"] == "ensemble":
        parts = [_direct(xt[a:b], xt[a:b], mt[a:b]) for a, b in zip(off[:-1], off[1:])]
        return torch.cat([q[0] for q in parts]), torch.cat([q[1] for q in parts])
    if case["kind"] == "block":
        a = torch.from_numpy(_active(case, x, seed)).to(DEV)
        psi = torch.full((len(mu),), float("nan"), dtype=torch.float64, device=DEV)
        acc = torch.full((len(mu), 3), float("nan"), dtype=torch.float64, device=DEV)
        psi[a], acc[a] = _direct(xt[a], xt, mt)
        return psi, acc
    return tuple(_direct(xt, xt, mt, tidal=case["kind"] == "tidal"))
