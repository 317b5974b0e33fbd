"""GPU test of the rejection resampler where lanes share particles (the end of a warp's run): the
ancestors and statuses equal the oracle's, whichever lane makes an attempt."""
import numpy as np
import pytest
import torch

import oracle
import workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# one particle (32 lanes on it), the group sizes 16 .. 1, partial warps, several runs per warp
SIZES = [1, 2, 3, 5, 8, 9, 16, 17, 31, 33, 65, 1000, 20011]


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("N", SIZES)
def test_shared_attempts_equal_oracle(rs, dtype, N):
    lw = workload.synthetic_logw(N, 4.0, seed=N, dtype=dtype)
    t = torch.from_numpy(lw).to(DEV)
    # the a-priori bound; one that the largest weights exceed (flagged, accepted at once); caps on
    # the trials at and around the attempts of one round of 1 .. 32 lanes
    tight = float(np.sort(lw)[max(0, N - 1 - N // 4)]) - 1.0
    for wmax, caps in ((0.0, (1 << 20, 1, 2, 3, 31, 32, 33, 63, 64, 65, 129)), (tight, (1 << 20, 5))):
        for cap in caps:
            with rs.Handle(N) as h:
                for mode in (rs.LAUNCH_AUTO, rs.LAUNCH_SEPARATE):
                    rs.rs_set_launch_mode(h, mode)
                    a = rs.rs_resample(h, rs.REJECTION, t, seed=11, step=2, log_wmax=wmax,
                                       max_trials=cap).cpu().numpy()
                    got = rs.rs_last_error(h)
                    st, want = oracle.rejection(lw, wmax, seed=11, step=2, max_trials=cap)
                    assert np.array_equal(a, want), (wmax, cap, mode)
                    assert got == st, (wmax, cap, mode)
                off = torch.tensor([0, N], dtype=torch.int64, device=DEV)
                b = rs.rs_resample_batched(h, rs.REJECTION, t, off, seed=11, step=2, log_wmax=wmax,
                                           max_trials=cap).cpu().numpy()
                assert rs.rs_last_error(h) == got and np.array_equal(a, b), (wmax, cap)
