"""GPU test of offsets that do not ascend in a batched call: reported as RS_ERR_ARG, no index out
of range (csrc/ragged.cuh, checked on the host in test_ragged_host.py), and the handle's next call
is right."""
import numpy as np
import pytest
import torch

import workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("shift", [-1000, 1000])
def test_one_wrong_offset_is_reported(rs, shift):
    """4000 filters of 64, one offset moved over its neighbours: the windows of the binary32
    Metropolis chains hold a filter that begins before or ends after them."""
    sizes = np.full(4000, 64, np.int64)
    offsets, lw, _ = workload.ragged_logw(sizes, seed=2, dtype=np.float32)
    t = torch.from_numpy(lw).to(DEV)
    good = torch.from_numpy(offsets).to(DEV)
    bad = good.clone()
    bad[1005] += shift
    with rs.Handle(lw.size) as h:
        want = rs.rs_resample_batched(h, rs.METROPOLIS, t, good, B=16, seed=3)
        assert rs.rs_last_error(h) == rs.RS_OK
        out = torch.zeros_like(want)
        rs.rs_resample_batched(h, rs.METROPOLIS, t, bad, B=16, seed=3, out=out)
        assert rs.rs_last_error(h) == rs.RS_ERR_ARG
        again = rs.rs_resample_batched(h, rs.METROPOLIS, t, good, B=16, seed=3)
        assert rs.rs_last_error(h) == rs.RS_OK
        assert torch.equal(want, again)
