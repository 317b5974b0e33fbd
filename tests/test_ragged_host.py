"""CPU test of the batched Metropolis kernel's staged windows (csrc/ragged.cuh): with ascending
offsets every particle is run once, from staged values where its filter fits; with offsets that
descend, overlap or leave the batch (which the call reports as RS_ERR_ARG) no index that a chain
may form leaves the staged values or the log-weights."""
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
