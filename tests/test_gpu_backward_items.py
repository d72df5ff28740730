"""Placement of the bf16 backward's items on the CTAs.

Every item (a query tile's dq, a key tile's dk/dv) is computed by one CTA, so
which CTA takes it changes no bit: a call of several streams equals the calls of
its parts that have no more items than an SM count and so are not placed, on the
same forward results. Sizes: placed by time at both head widths, just below
and just above the largest number of items that is placed.
"""
import dataclasses

import pytest
import torch

from paper_2607_20940_gb300 import synth

from helpers import BF16, bind, device_inputs, make_plan, msf
from test_gpu_backward import _run

pytestmark = pytest.mark.gpu

D128 = synth.Workload("items_d128", 2, (1, 1), 8, 39, 12, 128, 250, 1, 1, 4, 61)     # 120 items a stream
D64 = synth.Workload("items_d64", 4, (1, 2, 2, 4), 12, 60, 5, 64, 130, 1, 1, 2, 62)  # 140 items a stream


@pytest.mark.parametrize("w", [D128, dataclasses.replace(D128, batch=17), dataclasses.replace(D128, batch=18), D64],
                         ids=["d128_480", "d128_2040", "d128_2160", "d64_280"])
def test_items_placed_anywhere_same_bits(w):
    x, dout, out, lse, g, _ = _run(w, BF16)
    one = dataclasses.replace(w, batch=1)
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
