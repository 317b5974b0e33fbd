"""The workloads that the library's speed is measured on, each one pass through its public
entry points as a particle filter's program calls them.

Three kinds:

* ``resample``: one ``rs_resample`` call on one filter's log-weights (the synthetic weight sets
  of the paper's Section 4.1, log w = -(x - y)^2 / 2 with x ~ N(0, 1)), any of the five
  schemes, binary32 or binary64 log-weights in any precision mode, with or without Permute.
* ``batched``: one ``rs_resample_batched`` call on many filters of uneven sizes (CSR layout,
  sizes log-uniform, an own y per filter), Metropolis with its B per filter from Eq. B.
* ``smc``: a whole bootstrap filter on the linear-Gaussian state-space model
  (``smc.lgssm_bootstrap_launch``): resample with Permute, copy in place, propagate and weight,
  log weight total, T steps, compensated sums (the module's default).

The handle, its scratch, the output buffers and (for a batch) the filters' offsets and B are
what a program keeps from call to call; the log-weights are the new input of every call.
"""
import math

import numpy as np
import torch

import paper_1301_4019_gb300 as rs
from paper_1301_4019_gb300 import smc

PREC = {"plain": rs.PREC_PLAIN, "compensated": rs.PREC_COMPENSATED, "binary64": rs.PREC_BINARY64}
PHI, SIGMA_X, SIGMA_Y = 0.9, 1.0, 0.5  # the state-space model of the SMC cases


def _beta(y):
    """beta = E(w) / w_max of the synthetic weights (Section 4.1)."""
    return math.exp(-0.25 * y * y) / math.sqrt(2.0)


def _eq_b(y, eps=0.01):
    """Metropolis steps of Eq. B."""
    return max(1, math.ceil(math.log(eps) / math.log1p(-_beta(y))))


def _resample(name, scheme, dtype, N, y, prec="plain", permute=True):
    c = {"kind": "resample", "scheme": scheme, "dtype": dtype, "prec": prec, "N": int(N),
         "y": float(y), "B": _eq_b(y) if scheme == "metropolis" else 0, "permute": bool(permute)}
    if name:
        c["name"] = name
    return c


def _batched(name, scheme, dtype, F, n_min, n_max, sizes_seed, permute=True):
    c = {"kind": "batched", "scheme": scheme, "dtype": dtype, "prec": "plain", "F": int(F),
         "n_min": int(n_min), "n_max": int(n_max), "sizes_seed": int(sizes_seed),
         "permute": bool(permute)}
    if name:
        c["name"] = name
    return c


def _smc(name, scheme, N, T, B=0):
    c = {"kind": "smc", "scheme": scheme, "dtype": "f32", "N": int(N), "T": int(T), "B": int(B)}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest filter for which a GPU is worth its while (2^10 in the paper): launches
        # and dependent steps, as in a filter run at a high rate
        _resample("systematic_f32_1k", "systematic", "f32", 1000, 2.0),
        # the benchmark's size, the scheme most filters use
        _resample("systematic_f32_1m", "systematic", "f32", 1 << 20, 2.0),
        # the largest size of the size sweep: the memory-bound end
        _resample("systematic_f32_16m", "systematic", "f32", 1 << 24, 2.0),
        # binary64 log-weights with the default double-float sums, a size that fills no tile
        _resample("stratified_f64_3m", "stratified", "f64", 3000001, 2.0),
        # IEEE binary64 sums and weights, asked for where the last bits matter; the ancestry
        # itself (no Permute), as a program that gathers into new storage takes it
        _resample("systematic_f64_ieee_700k", "systematic", "f64", 700001, 1.0,
                  prec="binary64", permute=False),
        # the classic multinomial bootstrap filter
        _resample("multinomial_f32_1m", "multinomial", "f32", 1 << 20, 2.0),
        # the collective-free resamplers: Metropolis at Eq. B's B, in both types (a small odd
        # filter in binary64), and rejection under the a-priori bound
        _resample("metropolis_f32_1m", "metropolis", "f32", 1 << 20, 2.0),
        _resample("metropolis_f64_200k", "metropolis", "f64", 200003, 2.0),
        _resample("rejection_f32_1m", "rejection", "f32", 1 << 20, 2.0),
        # a whole particle filter
        _smc("smc_systematic_1m", "systematic", 1 << 20, 10),
        # a bank of 4096 filters of 256 .. 65536 particles (the batched benchmark's layout)
        _batched("batched_systematic_4096", "systematic", "f32", 4096, 256, 65536, 20130115),
        _batched("batched_metropolis_4096", "metropolis", "f32", 4096, 256, 65536, 20130115),
    ]


def _log_uniform(rng, lo, hi):
    return int(math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


_SCHEMES = ["systematic", "stratified", "multinomial", "metropolis", "rejection"]


def draw(rng):
    kind = rng.choice(["resample"] * 5 + ["batched"] * 2 + ["smc"])
    if kind == "resample":
        scheme = rng.choice(_SCHEMES)
        dtype = rng.choice(["f32", "f32", "f64"])
        y = rng.choice([0.0, 0.5, 1.0, 1.5, 2.0, 2.5, 3.0, 3.5, 4.0])
        prec, hi = "plain", 1 << 24
        if scheme in ("metropolis", "rejection"):
            steps = _eq_b(y) if scheme == "metropolis" else 1.0 / _beta(y)
            hi = min(hi, int((1 << 26) / steps))
        else:
            prec = rng.choice(["plain", "plain", "compensated" if dtype == "f32" else "binary64"])
            if scheme == "multinomial":
                hi = 1 << 23
            if prec == "binary64":
                hi = 1 << 22
        return _resample("", scheme, dtype, _log_uniform(rng, 256, hi), y, prec=prec,
                         permute=rng.random() < 0.75)
    if kind == "batched":
        scheme = rng.choice(_SCHEMES)
        dtype = rng.choice(["f32", "f32", "f64"])
        F = _log_uniform(rng, 64, 3000 if dtype == "f32" else 1000)
        n_max = _log_uniform(rng, 4096, 65536)
        return _batched("", scheme, dtype, F, rng.choice([1, 64, 256]), n_max,
                        rng.randrange(1 << 30), permute=rng.random() < 0.75)
    scheme = rng.choice(["systematic", "systematic", "stratified", "metropolis", "rejection"])
    return _smc("", scheme, _log_uniform(rng, 1 << 12, 1 << 20), rng.randint(2, 12),
                B=16 if scheme == "metropolis" else 0)


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _sizes_and_y(case):
    """Sizes and observation of every filter of a batch: the layout, the same for every seed."""
    g = np.random.Generator(np.random.PCG64(case["sizes_seed"]))
    u = g.uniform(math.log(case["n_min"]), math.log(case["n_max"]), size=case["F"])
    sizes = np.clip(np.floor(np.exp(u)), case["n_min"], case["n_max"]).astype(np.int64)
    return sizes, g.uniform(0.0, 4.0, size=case["F"])


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    st = {"case": case, "seed": seed & 0xFFFFFFFF, "scheme": rs.SCHEMES[case["scheme"]]}
    if case["kind"] == "smc":
        r = np.random.Generator(np.random.PCG64(seed))
        T, x = case["T"], r.standard_normal() * SIGMA_X / math.sqrt(1.0 - PHI * PHI)
        ys = []
        for _ in range(T):
            ys.append(x + SIGMA_Y * r.standard_normal())
            x = PHI * x + SIGMA_X * r.standard_normal()
        st["y"] = ys
        st["bufs"] = smc.LgssmBuffers(case["N"], T)
        st["h"] = rs.Handle(case["N"])
        return st
    if case["kind"] == "batched":
        sizes, y = _sizes_and_y(case)
        offsets = np.zeros(case["F"] + 1, np.int64)
        np.cumsum(sizes, out=offsets[1:])
        N = int(offsets[-1])
        st["offsets"] = torch.from_numpy(offsets).to(dev)
        yy = torch.repeat_interleave(torch.from_numpy(y).to(dev),
                                     torch.from_numpy(sizes).to(dev), output_size=N)
        st["B"] = torch.tensor([_eq_b(v) for v in y], dtype=torch.int32, device=dev)
    else:
        N, yy = case["N"], case["y"]
    x = torch.randn(N, generator=g, device=dev, dtype=torch.float64)
    st["logw"] = (-0.5 * (x - yy) ** 2).to(_dtype(case)).contiguous()
    st["out"] = torch.empty(N, dtype=torch.int32, device=dev)
    st["h"] = rs.Handle(N)
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "smc":
        b = smc.lgssm_bootstrap_launch(state["h"], state["y"], c["N"], state["scheme"], PHI,
                                       SIGMA_X, SIGMA_Y, seed=state["seed"], B=c["B"],
                                       bufs=state["bufs"])
        return {"x": b.x, "logw": b.logw, "ancestors": b.c, "log_total": b.log_total}
    if c["kind"] == "batched":
        return rs.rs_resample_batched(state["h"], state["scheme"], state["logw"],
                                      state["offsets"],
                                      B_per_filter=state["B"] if c["scheme"] == "metropolis" else None,
                                      seed=state["seed"], step=1, out=state["out"],
                                      permute=c["permute"], prec=PREC[c["prec"]])
    return rs.rs_resample(state["h"], state["scheme"], state["logw"], B=c["B"],
                          seed=state["seed"], step=1, out=state["out"], permute=c["permute"],
                          prec=PREC[c["prec"]])


def work(case):
    """Log-weights read once and ancestors written once; a Metropolis or rejection step reads
    one more log-weight. Arithmetic: an exponential (about ten operations) per weight formed
    and the sums over them. An SMC step reads and writes the states and writes the weights."""
    if case["kind"] == "smc":
        # per step: state read and written, log-weight written and read, ancestor written
        n = case["N"] * case["T"]
        return {"bytes": 20 * n, "flops": 40 * n}
    S = 4 if case["dtype"] == "f32" else 8
    if case["kind"] == "batched":
        sizes, y = _sizes_and_y(case)
        n = int(sizes.sum())
        if case["scheme"] == "metropolis":
            steps = float(np.dot(sizes, [_eq_b(v) for v in y]))
        elif case["scheme"] == "rejection":
            steps = float(np.dot(sizes, [1.0 / _beta(v) for v in y]))
        else:
            steps = n
    else:
        n = case["N"]
        if case["scheme"] == "metropolis":
            steps = n * case["B"]
        elif case["scheme"] == "rejection":
            steps = n / _beta(case["y"])
        else:
            steps = n
    return {"bytes": n * (S + 4), "flops": 12 * steps}


def exact(case, seed):
    """Ancestors are whole numbers, and a filter's states follow from them and from the
    library's own random numbers: no output has a value of its own in 64-bit arithmetic."""
    return None
