"""Host rules of csrc/sched.h on the CPU."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_20940_gb300", "csrc")

SOURCE = r"""
#include "sched.h"
extern "C" int idle(long long ctas, int sms, long long total, long long two_four, long long one_three) {
    const msf::IdleTasks t = msf::idle_tasks(ctas, sms, total, two_four, one_three);
    return 10 * t.one + t.more;
}
"""


@pytest.fixture(scope="module")
def sched(tmp_path_factory):
    d = tmp_path_factory.mktemp("sched")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    lib = ctypes.CDLL(str(d / "t.so"))
    lib.idle.argtypes = [ctypes.c_longlong, ctypes.c_int] + [ctypes.c_longlong] * 3
    return lib


# CTAs, tasks, the two shares, and what was faster than no sharing (us without / one and three / two and four)
@pytest.mark.parametrize("ctas,total,two_four,one_three,want", [
    (468, 93600, 16896, 10368, 0),      # 15.2 / 16.1 / 16.7
    (488, 101376, 15232, 9280, 0),      # 14.1 / 14.8 / 15.1
    (558, 120960, 12992, 7744, 0),      # 13.2 / 13.8 / 14.6
    (816, 177408, 18624, 10656, 0),     # 18.3 / 18.2 / 19.0: a tenth of the tasks
    (795, 149760, 34560, 21120, 24),    # the 480p window with the history: 16.2 / 16.1 / 14.7
    (1006, 74880, 34560, 21120, 13),    # two 480p streams, window only
    (933, 162864, 51328, 32320, 0),     # a third, and a fifth less one
    (1580, 322560, 52480, 33600, 24),   # 30.8 / 30.4 / 30.5
    (14468, 3244800, 294912, 163840, 24),  # 294 / 284 / 285
    (2888, 460800, 156672, 87040, 13),  # 72.4 / 70.1
    (4000, 1000, 900, 500, 0),          # more than a third of the tasks
])
def test_idle_tasks(sched, ctas, total, two_four, one_three, want):
    assert sched.idle(ctas, 152, total, two_four, one_three) == want
