"""The persistent backward's items on the CPU: their barriers and their placement.

An mbarrier's parity wait passes when the phase of that parity is the one before
the current one. The producer of csrc/attn_bwd_tc.cu asks for item k - 2 (and on a
change of kind for item k - 1) before it loads item k, when item k - 1 may or may
not be done: both waits must pass exactly when the item they ask for is done.
"""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_20940_gb300", "csrc")

SOURCE = r"""
#include "bwd_items.h"
extern "C" int bars() { return msf::kDoneBars; }
extern "C" int bar(int k) { return msf::done_bar(k); }
extern "C" int parity(int k) { return (int)msf::done_parity(k); }
// n classes of (count, ns): the CTA of every item, or 0 if they are not placed
extern "C" int place(const int* count, const int* ns, int n, int ctas, int* cta) {
    static msf::BwdOrder o;
    msf::ItemClass cl[2 * MSF_MAX_GROUPS];
    int total = 0;
    for (int i = 0; i < n; ++i) {
        cl[i] = {0, i, count[i], 0, ns[i], total};
        total += count[i];
    }
    msf::place_items(o, cl, n, total, ctas);
    if (!o.on) return 0;
    for (int x = 0; x < total; ++x) cta[x] = -1;
    for (int c = 0; c < ctas; ++c)
        for (int k = o.first[c]; k < o.first[c + 1]; ++k) {
            if (o.item[k] >= total || cta[o.item[k]] != -1) return -1;  // no item, or one twice
            cta[o.item[k]] = c;
        }
    return o.first[ctas] == total ? 1 : -2;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("bwd_items")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _passes(rule, item, done):
    """Whether the wait for `item` passes once items 0 .. done - 1 are done."""
    phase = sum(rule.bar(i) == rule.bar(item) for i in range(done))  # the barrier's current phase
    return (phase & 1) != rule.parity(item)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 100, 101])
def test_waits_before_item_k(rule, k):
    # every item before k may be done, item k is not loaded; items up to k - 3 were waited for
    for done in range(max(k - 2, 0), k + 1):
        for item in {k - 2, k - 1} - {-1}:
            if item == k - 1 and done < k - 1:
                continue  # asked only once item k - 2 is done
            assert _passes(rule, item, done) == (done > item), (k, item, done)


def test_every_bar_is_used_in_range(rule):
    assert all(0 <= rule.bar(k) < rule.bars() for k in range(64))


def _place(rule, classes, ctas):
    n = sum(c for c, _ in classes)
    cta = (ctypes.c_int * max(n, 1))()
    arr = ctypes.c_int * len(classes)
    on = rule.place(arr(*(c for c, _ in classes)), arr(*(t for _, t in classes)), len(classes), ctas, cta)
    return on, list(cta[:n])


def _rounds_end(classes, ctas):
    load, x = [0] * ctas, 0
    for count, ns in classes:
        for _ in range(count):
            r, c = divmod(x, ctas)
            load[ctas - 1 - c if r & 1 else c] += ns
            x += 1
    return max(load)


CLASSES = [
    [(153, 9000)], [(100, 20000), (300, 7000)], [(80, 15000), (80, 14000), (160, 3000), (7, 900)],
    [(1, 90000), (2047, 1200)], [(160, 30000), (170, 1500)], [(300, 5000), (200, 8000)], [(2048, 1500)],
    [(1000, 3700), (500, 2100), (300, 11000), (240, 800)],
]


@pytest.mark.parametrize("ctas", [152, 148, 160, 13])
@pytest.mark.parametrize("classes", CLASSES, ids=str)
def test_every_item_is_placed_once(rule, classes, ctas):
    on, cta = _place(rule, classes, ctas)
    assert on in (0, 1)
    if on:
        assert all(0 <= c < ctas for c in cta)
        load, x = [0] * ctas, 0
        for count, ns in classes:
            for _ in range(count):
                load[cta[x]] += ns
                x += 1
        gain = _rounds_end(classes, ctas) - max(load)
        assert gain >= 1000 and 100 * gain >= _rounds_end(classes, ctas)


def test_some_are_placed_and_some_not(rule):
    placed = {i: _place(rule, c, 152)[0] for i, c in enumerate(CLASSES)}
    assert set(placed.values()) == {0, 1}, placed
    assert _place(rule, [(2049, 1500)], 152)[0] == 0   # more items than the order holds
    assert _place(rule, [(152, 1500)], 152)[0] == 0    # one each
    assert _place(rule, [(900, 1500), (3, 90000)], 161)[0] == 0  # more CTAs than it holds
