"""The host rule that says before anything is built whether strips can serve a
list of items: item numbers that do not fit 32 bits are refused without a walk
over the items, and nothing is refused that the count on the device would
take."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2606_27086_gb300 import build as pkbuild

SRC = r"""
#include "strip_rule.h"
extern "C" int possible(const long long* blocks, int n, const long long* len, long long* calls, int pbytes,
                        long long entries) {
    std::vector<long long> b(blocks, blocks + n);
    auto at = [&](size_t, long long i) { ++*calls; return len[i]; };
    return suppy::strips_possible(b, at, pbytes, entries);
}
extern "C" int pays(long long packets, long long most, int pbytes, long long entries) {
    return suppy::strips_pay(packets, most, pbytes, entries);
}
"""
PBYTES = 16 + 256 + 512   # FP32 packets without a scatter


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    src = os.path.join(d, "rule.cpp")
    with open(src, "w") as f:
        f.write(SRC)
    so = os.path.join(d, "rule.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", pkbuild.CSRC, src, "-o", so])
    return ctypes.CDLL(so)


def _possible(rule, blocks, lens, entries, pbytes=PBYTES):
    b = np.asarray(blocks, np.int64)
    ln = np.ascontiguousarray(lens, np.int64)
    calls = ctypes.c_longlong(0)
    ptr = ctypes.POINTER(ctypes.c_longlong)
    got = rule.possible(b.ctypes.data_as(ptr), len(b), ln.ctypes.data_as(ptr), ctypes.byref(calls), pbytes,
                        ctypes.c_longlong(entries))
    return bool(got), calls.value


def _pays(rule, packets, most, entries, pbytes=PBYTES):
    return bool(rule.pays(ctypes.c_longlong(packets), ctypes.c_longlong(most), pbytes, ctypes.c_longlong(entries)))


@pytest.mark.parametrize("n,blocks", [(2048 * 2048, 512), (4096 * 4096, 128), (2**31 - 1, 2)])
def test_item_numbers_beyond_int32_are_refused_unread(rule, n, blocks):
    first = np.arange(blocks + 1, dtype=np.int64) * n
    assert first[-1] >= 2**31
    assert _possible(rule, first, np.zeros(1), 10**9) == (False, 0)


def test_items_longer_than_half_the_ring(rule):
    """A strip is copied in one piece of at most half the ring: 80 KB are 104
    packets, items of up to 3328 entries."""
    most = (160 * 1024 // 2) // PBYTES
    assert _possible(rule, [0, 4], [32 * most, 1, 1, 1], 32 * most + 3)[0]
    assert not _possible(rule, [0, 4], [32 * most + 1, 1, 1, 1], 32 * most + 4)[0]


def test_empty_items(rule):
    assert not _possible(rule, [0, 5], np.zeros(5), 0)[0]
    assert _possible(rule, [0, 5], [0, 0, 0, 0, 1], 1)[0]


@pytest.mark.parametrize("seed", range(20))
def test_never_refuses_what_the_count_takes(rule, seed):
    """Any packing that the rule on the counted packets takes has at least the
    packets of the lengths alone."""
    rng = np.random.default_rng(seed)
    nseg = int(rng.integers(1, 5))
    sizes = rng.integers(0, 4000, nseg)
    blocks = np.concatenate([[0], np.cumsum(sizes)])
    lens = rng.integers(0, int(rng.choice([3, 40, 400, 4096])), blocks[-1]) * (rng.random(blocks[-1]) < rng.random())
    least = most = 0
    for a, b in zip(blocks[:-1], blocks[1:]):
        for i in range(a, b, 4):
            p = -(-int(lens[i:min(i + 4, b)].max()) // 32)
            least, most = least + p, max(most, p)
    entries = int(lens.sum())
    got = _possible(rule, blocks, lens, entries)[0]
    assert got == _pays(rule, least, most, entries)
    for extra in (0, 1, 7, 1000, 10**6):
        if _pays(rule, least + extra, most + min(extra, 3), entries):
            assert got
