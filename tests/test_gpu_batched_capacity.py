"""GPU test of batches on handles larger than they are: the forms that follow the batch's size
(rejection runs, slots per lane of Permute) and the surplus of the grids give the ancestors of a
handle of the batch's own size, at sizes on both sides of the lines."""
import numpy as np
import pytest
import torch

import workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("total", [1, 4099, (1 << 18) - 1, 1 << 18, (1 << 20) - 3, 1 << 20])
@pytest.mark.parametrize("scheme", [0, 2, 3, 4])
def test_results_do_not_depend_on_the_capacity(rs, total, scheme):
    rng = np.random.default_rng(total)
    cuts = np.sort(rng.integers(0, total + 1, 40))
    sizes = np.diff(np.concatenate([[0], cuts, [total]]))
    offsets, lw, _ = workload.ragged_logw(sizes, seed=3, dtype=np.float32)
    t = torch.from_numpy(lw).to(DEV)
    off = torch.from_numpy(offsets).to(DEV)
    flags = torch.from_numpy((rng.random(sizes.size) < 0.8).astype(np.uint8)).to(DEV)
    got = []
    for cap in (total, 3 * total + 5000, 1 << 23):
        with rs.Handle(cap) as h:
            for kw in ({}, {"resample": flags}):
                for permute in (False, True):
                    got.append(rs.rs_resample_batched(h, scheme, t, off, B=6, seed=8, permute=permute,
                                                      **kw))
            assert rs.rs_last_error(h) == rs.RS_OK
    for k in range(4):
        assert torch.equal(got[k], got[k + 4]) and torch.equal(got[k], got[k + 8])
