"""The persistent backward's item barriers on the CPU.

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
