"""The radix sort's shares of the key's bits (csrc/sort_digits.h, compiled for the host) and its passes' integer
arithmetic restated with them: for every key width the digits tile the key, one mask serves the counts and the scatter,
and every pass's destinations are a stable permutation of [0, n)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2607_14513_gb300", "csrc")


@pytest.fixture(scope="module")
def shares(tmp_path_factory):
    d = tmp_path_factory.mktemp("digits")
    src, lib = str(d / "digits.cpp"), str(d / "digits.so")
    with open(src, "w") as f:
        f.write('#include "sort_digits.h"\n'
                'extern "C" int passes_of(int bits) { return sort_passes(bits); }\n'
                'extern "C" void digit_of(int bits, int p, int* o) {\n'
                '  const SortDigit d = sort_digit(bits, p);\n'
                '  o[0] = d.shift; o[1] = d.bits; o[2] = (int)d.mask; o[3] = d.ballots;\n}\n')
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib])
    L = C.CDLL(lib)

    def of(key_bits):
        out = []
        for p in range(L.passes_of(key_bits)):
            o = (C.c_int * 4)()
            L.digit_of(key_bits, p, o)
            out.append(tuple(o))
        return out
    return of


def _pass(keys, shift, mask, ballots, tile=4096):
    """Destinations of one pass: digit counts per tile (k_rs_count), their rows' and the digits' prefixes (k_rs_rows,
    k_rs_scatter), ranks inside the tile among the items whose low `ballots` digit bits agree."""
    n = keys.shape[0]
    d = ((keys >> np.uint64(shift)) & np.uint64(mask)).astype(np.int64)
    nt = -(-n // tile)
    counts = np.zeros((256, nt), np.int64)
    np.add.at(counts, (d, np.arange(n) // tile), 1)
    before = np.cumsum(counts, axis=1) - counts
    total = counts.sum(axis=1)
    start = np.cumsum(total) - total
    dst = np.empty(n, np.int64)
    for t in range(nt):
        s = slice(t * tile, min((t + 1) * tile, n))
        told = d[s] & ((1 << ballots) - 1)     # what the ballots compare
        order = np.argsort(told, kind="stable")
        rank = np.empty(order.shape[0], np.int64)
        first = np.searchsorted(told[order], told[order], side="left")
        rank[order] = np.arange(order.shape[0]) - first
        dst[s] = start[d[s]] + before[d[s], t] + rank
    return dst


@pytest.mark.parametrize("key_bits", range(1, 65))
def test_shares_and_destinations(shares, key_bits):
    digits = shares(key_bits)
    at = 0
    for shift, bits, mask, ballots in digits:
        assert shift == at and 1 <= bits <= 8 and mask == (1 << bits) - 1
        assert ballots == max(bits, 4)
        at += bits
    assert at == key_bits
    rng = np.random.default_rng(key_bits)
    n = 9001
    keys = rng.integers(0, 2 ** 64, n, dtype=np.uint64) >> np.uint64(64 - key_bits)
    keys[::3] = keys[0]
    k, v = keys.copy(), np.arange(n)
    for shift, bits, mask, ballots in digits:
        dst = _pass(k, shift, mask, ballots)
        assert np.array_equal(np.sort(dst), np.arange(n))
        k2, v2 = np.empty_like(k), np.empty_like(v)
        k2[dst], v2[dst] = k, v
        k, v = k2, v2
    want = np.argsort(keys, kind="stable")
    assert np.array_equal(v, want) and np.array_equal(k, keys[want])
