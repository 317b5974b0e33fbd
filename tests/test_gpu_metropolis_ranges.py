"""GPU test of the Metropolis chains where their quick decisions do not hold or did not: large
log-weights, whose binary32 truncations are too coarse (unnormalised log-likelihoods), rises above
66 (the exponential overflows), many zero weights, the type's lowest value. Ancestors equal the
oracle's, from one filter and from a batch."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _weights(kind, N, dtype):
    x = np.random.default_rng(len(kind)).standard_normal(N)
    lw = -0.5 * (x - 2.0) ** 2
    if kind.startswith("spread"):
        lw = float(kind[6:]) * x
    elif kind.startswith("near"):
        lw = lw + float(kind[4:])
    elif kind.startswith("zero"):
        lw[np.random.default_rng(1).random(N) < float(kind[4:])] = -np.inf
    elif kind == "lowest":
        lw[::2] = np.finfo(dtype).min
        lw[::3] = -np.inf
    return lw.astype(dtype)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["spread100", "spread1e4", "spread1e5", "near-41943", "near-1e6", "near1e6",
                                  "zero0.5", "zero0.99", "lowest"])
def test_chains_equal_oracle(rs, dtype, kind):
    for N, B in ((4099, 30), (20000, 7)):
        lw = _weights(kind, N, dtype)
        t = torch.from_numpy(lw).to(DEV)
        st, want = oracle.metropolis(lw, B, seed=5, step=2)
        assert st == oracle.OK
        off = torch.tensor([0, N], dtype=torch.int64, device=DEV)
        with rs.Handle(N) as h:
            a = rs.rs_resample(h, rs.METROPOLIS, t, B=B, seed=5, step=2).cpu().numpy()
            assert rs.rs_last_error(h) == rs.RS_OK and np.array_equal(a, want), (N, B)
            b = rs.rs_resample_batched(h, rs.METROPOLIS, t, off, B=B, seed=5, step=2).cpu().numpy()
            assert rs.rs_last_error(h) == rs.RS_OK and np.array_equal(b, want), (N, B)
