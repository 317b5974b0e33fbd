"""CPU test of the ragged batches' index arithmetic (csrc/ragged.cuh). The staged windows of the
batched Metropolis kernel: with ascending offsets every particle is run once, from staged values
where its filter fits; with offsets that descend, overlap or leave the batch (which the call
reports as RS_ERR_ARG) no index that a chain may form leaves the staged values or the log-weights.
The plans: whatever the offsets, the accepted filters hold no more than the handle's particles and
none beyond offsets[F], so tiles and segments fit the scratch."""
import ctypes as C

import numpy as np
import pytest

import host_build

CAP = 57344  # staged values of the kernel
MAX_FILTER = 1 << 20


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_build.load("ragged", tmp_path_factory.mktemp("host"))


def _ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def _run(lib, off, total, B, chunks, cap=CAP):
    """All chunks of the batch, cut at equal shares of the work as the kernel cuts them."""
    off = np.asarray(off, np.int64)
    F = off.size - 1
    n = np.diff(off)
    ok = (off[:-1] >= 0) & (n >= 0) & (off[1:] <= total) & (n <= MAX_FILTER)
    per = np.broadcast_to(np.asarray(B, np.int64) + 8, F)
    work = np.concatenate([[0], np.cumsum(np.where(ok, n * per, 0))]).astype(np.int64)
    cuts = []
    for x in [work[-1] * k // chunks for k in range(chunks)] if work[-1] else []:
        f = int(np.searchsorted(work, x, side="right")) - 1
        cuts.append((f, int((x - work[f]) // per[f]) & -32))
    cuts.append((F, 0))
    visits, staged = np.zeros(total, np.int32), np.zeros(total, np.int32)
    st = 0
    for (f, i), (fe, ie) in zip(cuts, cuts[1:]):
        st = st or lib.chain_chunk(_ptr(off), F, C.c_int64(total), _ptr(work), f, i, fe, ie, cap,
                                   _ptr(visits), _ptr(staged))
    return st, visits, staged


@pytest.mark.parametrize("sizes,chunks", [([64] * 4000, 152), ([1, 0, 300, 57344, 57345, 2, 0, 131077, 17], 5),
                                          ([4096], 3), ([200, 1, 0, 70000, 5] * 40, 37)])
def test_ascending_offsets_run_every_particle_once(lib, sizes, chunks):
    off = np.concatenate([[0], np.cumsum(sizes)])
    total = int(off[-1])
    st, visits, staged = _run(lib, off, total, 16, chunks)
    assert st == 0 and np.all(visits == 1)
    fits = np.repeat(np.asarray(sizes) <= CAP, sizes)
    assert np.array_equal(staged == 1, fits)  # (a chunk's cut lies inside a staged filter)


@pytest.mark.parametrize("shift", [-1000, -64, -1, 1, 63, 64, 1000, 57343, 200000, -200000])
@pytest.mark.parametrize("at", [1, 1003, 1005, 1010, 2000, 3999])
def test_one_wrong_offset_stays_in_range(lib, at, shift):
    off = np.arange(4001, dtype=np.int64) * 64
    off[at] += shift
    st, _, _ = _run(lib, off, 4000 * 64, 16, 152)
    assert st == 0


def test_wide_wrong_offsets_stay_in_range(lib):
    total = 300300
    st, _, _ = _run(lib, [0, 100, 60000, 200, 300, total], total, np.array([1, 1, 1, 1, 400]), 2)
    assert st == 0
    rng = np.random.default_rng(4)
    for k in range(300):
        F = int(rng.integers(1, 60))
        total = int(rng.integers(1, 200000))
        off = np.sort(rng.integers(0, total + 1, F + 1))
        for _ in range(int(rng.integers(1, 6))):
            off[rng.integers(0, F + 1)] = rng.integers(-50, total + 200)
        st, _, _ = _run(lib, off, total, rng.integers(0, 60, F), int(rng.integers(1, 20)),
                        cap=int(rng.choice([64, 1000, CAP])))
        assert st == 0, (k, off.tolist())


@pytest.mark.parametrize("max_n", [1, 4096, 300000])
def test_accepted_filters_fit_the_scratch(lib, max_n):
    rng = np.random.default_rng(max_n)
    F_max = max(1024, max_n // 16)
    cases = [np.tile([0, max_n], 600)[:1025],                     # every other filter holds all
             np.array([0, max_n, max_n // 2]),                     # past offsets[F]
             np.array([0, 1, max_n + 1, max_n + 2]), np.array([-1, 1, max_n])]
    cases += [rng.integers(-2, max_n + 3, rng.integers(2, F_max + 1)) for _ in range(50)]
    cases += [np.sort(rng.integers(0, max_n + 1, rng.integers(2, F_max + 1))) for _ in range(50)]
    for off in cases:
        off = off.astype(np.int64)
        F = off.size - 1
        n = np.empty(F, np.int64)
        st = lib.batch_sizes(_ptr(off), F, C.c_int64(max_n), _ptr(n))
        d = np.diff(off)
        good = off[0] >= 0 and np.all(d >= 0) and off[-1] <= max_n and np.all(d <= MAX_FILTER)
        assert (st == 0) == bool(good)
        assert np.array_equal(n, d) or not good
        # the scratch holds max_n / 2048 + max_filters + 1 tiles of 8 segments of 256 particles
        tiles, segs = (n + 2047) // 2048, (n + 255) // 256
        assert tiles.sum() <= max_n // 2048 + F_max + 1 and segs.sum() <= 8 * (max_n // 2048 + F_max + 1)
        assert np.all((n == 0) | ((off[:-1] >= 0) & (off[:-1] + n <= min(max_n, off[-1]))))
