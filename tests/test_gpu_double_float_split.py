"""GPU test of the double-float split of binary64 log-weights where it changes form: magnitudes
on both sides of 2^-73, zeros of both signs, subnormals, large magnitudes and -inf among ordinary
ones, below a maximum of either form. Cumulative offspring within the rounding bound of the
double-double oracle."""
import numpy as np
import pytest
import torch

import oracle
from parity_tools import cumulative_mismatches

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("top", [0.0, -0.0, 2.0 ** -140, 2.0 ** -73 * (1 - 2.0 ** -53), 2.0 ** -73, 1.0,
                                 -2.0 ** -72])
def test_split_ranges(rs, top):
    rng = np.random.default_rng(73)
    N = 20000
    lw = -0.5 * rng.normal(2.0, 1.0, N) ** 2
    lw[::5] = -2.0 ** rng.uniform(-76.0, -70.0, len(lw[::5]))
    lw[1::50] = -2.0 ** -73
    lw[2::50] = -2.0 ** -73 * (1 - 2.0 ** -53)
    lw[3::50] = -2.0 ** 127
    lw[4::50] = -2.0 ** 127 * (1 - 2.0 ** -53)
    lw[6::50] = rng.choice([-5e-324, -2.0 ** -126, -2.0 ** -149, -2.0 ** 100, -np.inf], len(lw[6::50]))
    lw = np.minimum(lw, top)
    lw[N // 2] = top
    t = torch.from_numpy(lw).to(DEV)
    with rs.Handle(N) as h:
        for sch, f in ((rs.SYSTEMATIC, oracle.systematic), (rs.STRATIFIED, oracle.stratified)):
            a = rs.rs_resample(h, sch, t, seed=31, step=1, prec=0)
            assert rs.rs_last_error(h) == rs.RS_OK
            O_k = np.cumsum(np.bincount(a.cpu().numpy(), minlength=N))
            st, O_o, _ = f(lw, 31, step=1, prec=1)
            assert st == oracle.OK
            n, bad = cumulative_mismatches("f64", sch, lw, O_k, O_o, seed=31, step=1,
                                           oracle_is_sequential=False)
            assert bad == 0, (sch, n)
