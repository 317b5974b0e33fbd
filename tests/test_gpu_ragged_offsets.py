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


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("scheme", range(5))
def test_descending_offsets_write_nothing_past_the_last(rs, scheme, dtype):
    """Offsets that run ahead of offsets[F] and fall back, and ones that give every second filter
    the whole batch (more tiles than the scratch holds): RS_ERR_ARG with and without Permute and in
    both launch modes, nothing written past offsets[F], and the next call is right."""
    n = 20000
    good = torch.tensor([0, 300, 9000, n], dtype=torch.int64, device=DEV)
    ahead = torch.tensor([0, 300, 19000, 9000, 12000], dtype=torch.int64, device=DEV)
    many = torch.tensor([0, n] * 500 + [0, 12000], dtype=torch.int64, device=DEV)
    t = torch.from_numpy(workload.synthetic_logw(n, 2.0, seed=1, dtype=dtype)).to(DEV)
    with rs.Handle(n) as h:
        for mode in (rs.LAUNCH_AUTO, rs.LAUNCH_SEPARATE):
            rs.rs_set_launch_mode(h, mode)
            for permute in (False, True):
                want = rs.rs_resample_batched(h, scheme, t, good, B=5, seed=1, permute=permute)
                assert rs.rs_last_error(h) == rs.RS_OK
                for off in (ahead, many):
                    out = torch.full((n,), -7, dtype=torch.int32, device=DEV)
                    rs.rs_resample_batched(h, scheme, t, off, B=5, seed=1, permute=permute, out=out)
                    assert rs.rs_last_error(h) == rs.RS_ERR_ARG
                    assert bool((out[12000:] == -7).all())
                got = rs.rs_resample_batched(h, scheme, t, good, B=5, seed=1, permute=permute)
                assert rs.rs_last_error(h) == rs.RS_OK and torch.equal(got, want)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_first_offset_above_zero(rs, dtype):
    """Positions before offsets[0] belong to no filter: the per-particle schemes report them,
    binary32 Metropolis from either of its kernels; the filters' own results are not affected."""
    n = 5000
    t = torch.from_numpy(workload.synthetic_logw(n, 2.0, seed=1, dtype=dtype)).to(DEV)
    off = torch.tensor([3, 1200, n], dtype=torch.int64, device=DEV)
    kernel = rs.BATCHED_METROPOLIS_F64 if dtype == np.float64 else rs.BATCHED_METROPOLIS_F32
    with rs.Handle(n) as h:
        got = []
        for shape in ((256, 1), (128, 2)):
            rs.rs_set_batched_launch(h, kernel, *shape)
            got.append(rs.rs_resample_batched(h, rs.METROPOLIS, t, off, B=9, seed=1))
            assert rs.rs_last_error(h) == rs.RS_ERR_ARG
        assert torch.equal(got[0][3:], got[1][3:])
        rs.rs_resample_batched(h, rs.REJECTION, t, off, seed=1)
        assert rs.rs_last_error(h) == rs.RS_ERR_ARG
