"""CPU test of Code 11 by a warp (csrc/runs.cuh), its 32 lanes run on the host: the positions of a
segment's runs at the sizes where the window changes form, at every alignment, at the start of a
sequence and at the end of the longest one accepted (2^31 - 1 particles), against numpy's repeat."""
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


def _segment(lib, O, before, b0, n, shift):
    """(status, positions before .. the last count, guards untouched, claimed bits)"""
    O = np.asarray(O, np.int64)
    cnt = min(256, n - b0)
    end = n if b0 + cnt == n else int(O[cnt - 1])
    G = 4096
    buf = np.full(max(end - before, 0) + 2 * G + 16, -7, np.int32)
    # position `before` at a place of buf whose address gives position 0 the alignment `shift`
    at = G + next(k for k in range(8) if (buf.ctypes.data // 4 + G + k - before) % 8 == shift)
    bits = np.zeros(32, np.uint8)
    st = lib.segment_runs(_ptr(O.astype(np.int32)), before, b0, n, C.c_int64(before), _ptr(buf[at:]),
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
