"""GPU test of the Code-11 scatter (warp_runs) at the sizes where its window changes form: the
offspring of one warp's 256 particles below, at and above 256 (one part), 320 (a short rest), 512
(one window) and several windows, with the output at every alignment of its 32-byte sectors.
Integer work: equal to numpy's repeat."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("shift", [0, 1, 3, 7])
@pytest.mark.parametrize("spread", ["even", "first", "last", "random"])
def test_code11_windows(rs, shift, spread):
    rng = np.random.default_rng(shift)
    per = [0, 1, 255, 256, 257, 263, 264, 265, 319, 320, 321, 327, 511, 512, 513, 520, 1023, 1500, 7,
           8, 9, 0, 2000, 0, 0]
    per += [0] * (sum(per) // 256 + 1 - len(per))  # enough particles that the counts sum to N
    N = 256 * len(per)
    o = np.zeros(N, np.int64)
    for s, k in enumerate(per):
        seg = o[256 * s:256 * (s + 1)]
        if spread == "even":
            seg += k // 256
            seg[:k % 256] += 1
        elif spread == "random":
            seg += np.bincount(rng.integers(0, 256, k), minlength=256)
        else:
            seg[0 if spread == "first" else 255] += k
    o[rng.integers(0, N)] += N - o.sum()  # (one long run takes what is left)
    assert o.sum() == N and o.min() >= 0
    O = torch.from_numpy(np.cumsum(o).astype(np.int32)).to(DEV)
    buf = torch.full((N + 8,), -7, dtype=torch.int32, device=DEV)
    with rs.Handle(N) as h:
        rs.rs_cumulative_offspring_to_ancestors(h, O, a=buf[shift:shift + N])
        assert rs.rs_last_error(h) == rs.RS_OK
    got = buf.cpu().numpy()
    assert np.array_equal(got[shift:shift + N], np.repeat(np.arange(N), o))
    assert np.all(got[:shift] == -7) and np.all(got[shift + N:] == -7)
