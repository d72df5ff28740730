"""Placement of the bf16 backward's items on the CTAs.

Every item (a query tile's dq, a key tile's dk/dv) is computed by one CTA, so
which CTA takes it changes no bit: a call of several streams equals the calls of
its streams, which are not placed, on the same forward results. Cases: placed by
time at both head widths, just below the largest number of items that is placed,
above it, and a call whose gain lies below the line.
"""
import dataclasses

import pytest
import torch

from paper_2607_20940_gb300 import synth

from helpers import BF16, bind, device_inputs, make_plan, msf, routes
from test_gpu_backward import _run

pytestmark = pytest.mark.gpu

D128 = synth.Workload("items_d128", 2, (1, 1), 8, 39, 12, 128, 250, 1, 1, 4, 61)
CASES = {  # workload, items, placed
    "d128": (synth.Workload("d128", 2, (1, 1), 20, 16, 2, 128, 0, 1, 1, 16, 62), 320, 1),
    "d64": (synth.Workload("d64", 2, (1, 1), 30, 52, 3, 64, 0, 1, 1, 2, 63), 300, 1),
    "d64_most": (synth.Workload("d64_most", 2, (1, 2), 34, 36, 5, 64, 250, 1, 1, 13, 64), 2015, 1),
    "no_gain": (D128, 480, 0),
    "too_many": (dataclasses.replace(D128, batch=18), 2160, 0),
}


@pytest.mark.parametrize("name", CASES)
def test_items_placed_anywhere_same_bits(name):
    w, items, placed = CASES[name]
    one = dataclasses.replace(w, batch=1)
    r = routes(make_plan(w))
    assert (r["items"], r["placed"]) == (items, placed) and routes(make_plan(one))["placed"] == 0
    x, dout, out, lse, g, _ = _run(w, BF16)
    for b in (0, w.batch - 1):
        dx = device_inputs({k: v[b:b + 1].contiguous() for k, v in x.items()}, w.history_capacity)
        plan = make_plan(one, BF16)
        bind(plan, dx)
        plan.kv_resample(dx["k_win"], dx["v_win"])
        h = {k: torch.full_like(dx["q"], float("nan")) for k in g}
        plan.mssa_backward(dx["q"], dx["k_win"], dx["v_win"], out[b:b + 1].contiguous(), dout[b:b + 1].cuda(),
                           lse[b:b + 1].clone(), h["dq"], h["dk"], h["dv"], plan.backward_workspace())
        torch.cuda.synchronize()
        assert plan.device_status() == msf().MSF_OK
        for k in g:
            assert torch.equal(h[k][0], g[k][b]), (b, k)
