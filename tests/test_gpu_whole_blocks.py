"""Attention calls of the persistent kernel that take whole 256-row blocks
instead of an even split of the tile sequence (no partial results, no merge):
one and several groups, one to three blocks a CTA, both head widths, ragged last
blocks, and the pyramid built in the same launch. Tolerances as for the other
bf16 attention tests: |err| <= 2e-2, mean <= 2e-3 for unit-variance inputs; the
row log-sum-exp 2e-3; a second launch gives the same bits.
"""
import numpy as np
import pytest
import torch

from helpers import BF16, bind, device_inputs, err_stats, make_plan, msf, oracle_mssa, routes
from oracle import mssa as omssa
from paper_2607_20940_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [
    synth.Workload("one_group", 2, (1, 1), 13, 32, 9, 128, 2, 1, 1, 3, 71),           # 108 blocks
    synth.Workload("three_groups", 3, (1, 2, 4), 24, 16, 13, 128, 53, 3, 3, 4, 72),    # 208 blocks, two or three a CTA
    synth.Workload("d64", 3, (1, 1, 2), 10, 8, 11, 64, 61, 2, 2, 8, 73),               # one-tile groups
    synth.Workload("six_states", 6, (1, 1, 2, 2, 4, 4), 8, 56, 13, 128, 187, 0, 1, 2, 74),
]


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
def test_whole_blocks(w):
    x = synth.attention_inputs(w, BF16)
    dx = device_inputs(x, w.history_capacity)
    plan = make_plan(w, BF16)
    taken = routes(plan)
    assert taken["whole"] == 1 and taken["cluster"] == 0, taken
    bind(plan, dx)
    B, N = dx["q"].shape[:2]
    outs = [torch.full_like(dx["q"], float("nan")) for _ in range(3)]
    lse = torch.full((B, w.heads, N), float("nan"), dtype=torch.float32, device="cuda")
    plan.kv_resample(dx["k_win"], dx["v_win"])
    plan.mssa_forward_lse(dx["q"], dx["k_win"], dx["v_win"], outs[0], lse)
    plan.mssa_forward(dx["q"], dx["k_win"], dx["v_win"], outs[1])
    plan.mssa_forward_resample(dx["q"], dx["k_win"], dx["v_win"], outs[2])
    torch.cuda.synchronize()
    assert plan.device_status() == msf().MSF_OK
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    heads = [0, w.heads - 1]
    mx, mean = err_stats(outs[0], oracle_mssa(x, w, heads=heads), heads=heads)
    assert mx <= 2e-2 and mean <= 2e-3, (mx, mean)
    f = synth.to_f64
    ref = omssa.mssa_lse(f(x["q"]), f(x["k_win"]), f(x["k_sink"]), f(x["k_hist"]), w.scales, w.grid_h, w.grid_w, 0,
                         heads=heads, frames=w.frames)
    assert np.abs(lse.double().cpu().numpy()[:, heads] - ref[:, heads]).max() <= 2e-3
