"""CPU test of Code 11 by a warp (csrc/runs.cuh), its 32 lanes run on the host: the positions of a
segment's runs at the sizes where the window changes form, at every alignment, at the start of a
sequence and at the end of the longest one accepted (2^31 - 1 particles), against numpy's repeat;
and the counts of two-float sums, which need not ascend with the cumulative weights."""
import ctypes as C

import numpy as np
import pytest

import host_build

LAST = (1 << 31) - 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_build.load("runs", tmp_path_factory.mktemp("host"))


def _ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def _segment(lib, O, before, b0, n, shift, two_float=0):
    """(status, positions before .. the last count, guards untouched, claimed bits)"""
    O = np.asarray(O, np.int64)
    cnt = min(256, n - b0)
    end = n if b0 + cnt == n else int(O[cnt - 1])
    G = 4096
    buf = np.full(max(end - before, 0) + 2 * G + 16, -7, np.int32)
    # position `before` at a place of buf whose address gives position 0 the alignment `shift`
    at = G + next(k for k in range(8) if (buf.ctypes.data // 4 + G + k - before) % 8 == shift)
    bits = np.zeros(32, np.uint8)
    st = lib.segment_runs(two_float, _ptr(O.astype(np.int32)), before, b0, n, C.c_int64(before), _ptr(buf[at:]),
                          shift, _ptr(bits))
    m = max(end - before, 0)
    clean = np.all(buf[:at] == -7) and np.all(buf[at + m:] == -7)
    return st, buf[at:at + m], bool(clean), np.unpackbits(bits, bitorder="little")


def _check(lib, o, before, b0, n, shift):
    o = np.asarray(o, np.int64)
    cnt = min(256, n - b0)
    O = before + np.cumsum(o)
    st, got, clean, bits = _segment(lib, O, before, b0, n, shift)
    want = o.copy()
    want[cnt:] = 0
    if b0 + cnt == n:
        want[cnt - 1] = n - before - want[:cnt - 1].sum()
    assert st == 0 and clean
    assert np.array_equal(got, np.repeat(b0 + np.arange(256), want))
    assert np.array_equal(bits, want > 0)


TOTALS = [0, 1, 7, 8, 9, 255, 256, 257, 263, 319, 320, 321, 511, 512, 513, 520, 1023, 1500]


@pytest.mark.parametrize("place", ["start", "middle", "end"])
@pytest.mark.parametrize("spread", ["even", "first", "last", "random"])
def test_runs_of_a_segment(lib, place, spread):
    rng = np.random.default_rng(len(place) + len(spread))
    for k in TOTALS:
        o = np.zeros(256, np.int64)
        if spread == "even":
            o += k // 256
            o[:k % 256] += 1
        elif spread == "random":
            o += np.bincount(rng.integers(0, 256, k), minlength=256)
        else:
            o[0 if spread == "first" else 255] = k
        for shift in range(8):
            before = {"start": 0, "middle": 1000003 + shift, "end": LAST - 300 - k}[place]
            _check(lib, o, before, {"start": 0, "middle": 5120, "end": LAST - 256 - 255}[place], LAST,
                   shift)


@pytest.mark.parametrize("valid", [1, 2, 7, 8, 9, 127, 248, 249, 255, 256])
@pytest.mark.parametrize("n", [LAST, LAST - 1, LAST - 300, 100000])
def test_last_segment(lib, n, valid):
    """The segment that holds the sequence's last particle, its counts ending at n: what lies past
    the end, and the last windows, may pass 2^31 - 1."""
    rng = np.random.default_rng(valid)
    for k in (0, 1, 8, 255, 256, 505, 512, 513, 1100):
        o = np.zeros(256, np.int64)
        o[:valid] += np.bincount(rng.integers(0, valid, k), minlength=valid)
        for shift in (0, 3, 7):
            _check(lib, o, n - k, n - valid, n, shift)


def _f(x):
    return np.asarray(x, np.float32)


def test_two_float_counts_can_fall(lib):
    """Two-float products do not preserve order: neighbouring cumulative weights on the two sides
    of a step of the high word whose counts fall, and the runs of a segment around them."""
    rng = np.random.default_rng(7)
    n, found = 1 << 20, 0
    for _ in range(3000):
        S = rng.uniform(1.0, n)
        hi = np.float32(rng.uniform(0.01, 1.0) * S)
        up = np.nextafter(hi, np.float32(np.inf), dtype=np.float32)
        half = (np.float64(up) - np.float64(hi)) / 2
        W = np.empty((256, 2), np.float32)  # ascending: half of them below the step, half above
        W[:128, 0], W[:128, 1] = hi, half * (1.0 - 2.0 ** -22 * np.arange(127, -1, -1))
        W[128:, 0], W[128:, 1] = up, -half * (1.0 - 2.0 ** -22 * np.arange(128))
        exact = W[:, 0].astype(np.float64) + W[:, 1]
        assert np.all(np.diff(exact) >= 0)
        c = n / S
        c2 = _f([c, c - np.float64(np.float32(c))])
        r = exact[127] * c
        u = np.ceil(r) - r  # (the count steps between the two halves)
        u2 = _f([u, u - np.float64(np.float32(u))])
        O = np.empty(256, np.int32)
        lib.two_float_counts(_ptr(W), 256, _ptr(c2), _ptr(u2), _ptr(O))
        if np.all(np.diff(O) >= 0):
            continue
        found += 1
        for before, last in ((O[0], O[-1]), (int(O.min()), int(O.max())), (int(O.max()), int(O.min()))):
            X = O.copy()
            X[-1] = last  # (the counts at the segment's two prefixes, whichever way they fall)
            st, got, clean, bits = _segment(lib, X, int(before), 0, n, 3, two_float=1)
            assert st == 0 and clean
            assert np.all((got >= 0) & (got < 256)) and np.all(np.diff(got) >= 0)
            assert bits.sum() == np.unique(got).size
    assert found > 10


def test_falling_counts_stay_in_the_window(lib):
    """Counts that fall by one anywhere, at ranges that fill the window exactly and begin at its
    first position: no write outside the window or the range, every position written."""
    rng = np.random.default_rng(8)
    for total in (1, 8, 255, 256, 257, 505, 511, 512, 513, 900):
        for k in range(40):
            O = 8000 + np.sort(rng.integers(0, total + 1, 256))
            O[-1] = 8000 + total
            i = rng.integers(0, 255, 9)
            O[i] += rng.integers(-1, 2, 9)
            if k % 4 == 0:
                O[0], O[200] = 7999, 8000 + total + 1
            st, got, clean, bits = _segment(lib, O, 8000, 512, 1 << 20, 0, two_float=1)
            assert st == 0 and clean and got.size == total
            assert np.all((got >= 512) & (got < 768)) and np.all(np.diff(got) >= 0)
            assert np.array_equal(np.nonzero(bits)[0] + 512, np.unique(got))
