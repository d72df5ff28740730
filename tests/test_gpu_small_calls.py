"""Attention calls on either side of the small-call rule.

Small calls give every 128-row query tile its own thread-block cluster (1, 2, 4
or 8 CTAs over its context) and merge over distributed shared memory; larger
ones run the persistent kernel, whose split blocks merge in place (up to eight
pieces) or from the partial slots. Every case says which form it is there for, and
the call must take it. Tolerances as for the other bf16 attention tests: |err| <=
2e-2, mean <= 2e-3 for unit-variance inputs.
"""
import dataclasses

import pytest
import torch

from helpers import BF16, bind, device_inputs, err_stats, make_plan, msf, oracle_mssa, routes
from paper_2607_20940_gb300 import synth

pytestmark = pytest.mark.gpu

W = synth.Workload("small", 1, (1,), 8, 16, 1, 64, 0, 0, 0, 1, 60)
CASES = {
    # ---- one tile (whole blocks); clusters: edges of 128, fewer tiles than CTAs would take
    "one_key": dataclasses.replace(W, grid_h=1, grid_w=1),
    "one_tile_d128": dataclasses.replace(W, head_dim=128, heads=3),
    "tile_and_a_few_d128": dataclasses.replace(W, T=2, scales=(1, 2), heads=3, head_dim=128, sink_tokens=1),
    "tile_and_a_row": dataclasses.replace(W, grid_h=3, grid_w=43, sink_tokens=1, heads=2),
    "cluster8_long": dataclasses.replace(W, head_dim=128, heads=2, sink_tokens=6000),
    "cluster8_ragged": dataclasses.replace(W, T=2, scales=(1, 2), grid_h=10, grid_w=14, heads=1, sink_tokens=5333),
    "cluster4_ragged": dataclasses.replace(W, T=2, scales=(1, 2), grid_h=10, grid_w=14, heads=4, sink_tokens=2333),
    "cluster4_groups": dataclasses.replace(W, T=4, scales=(1, 2, 2, 4), grid_h=12, grid_w=20, heads=4, head_dim=128,
                                           sink_tokens=77, history_frames=2, history_capacity=3),
    "cluster2_streams": dataclasses.replace(W, T=3, scales=(1, 2, 2), grid_h=18, grid_w=26, heads=6, sink_tokens=33,
                                            history_frames=1, history_capacity=1, batch=2),
    "cluster1_full": dataclasses.replace(W, T=2, scales=(1, 1), grid_h=16, grid_w=16, heads=19, head_dim=128,
                                         sink_tokens=100, batch=2),  # 152 query tiles
    # ---- the persistent kernel: merges in place, from the slots, whole blocks
    "in_place": dataclasses.replace(W, grid_w=32, heads=15, head_dim=128, sink_tokens=3600, batch=4),
    "in_place_long_d64": dataclasses.replace(W, grid_w=32, heads=15, sink_tokens=7400, batch=4),
    "in_place_d64": dataclasses.replace(W, T=3, scales=(1, 1, 2), grid_h=20, grid_w=20, heads=12, sink_tokens=700,
                                        batch=3),
    "from_slots": dataclasses.replace(W, grid_h=16, grid_w=16, heads=9, head_dim=128, sink_tokens=30000),
    "from_slots_d64": dataclasses.replace(W, grid_h=16, grid_w=16, heads=9, sink_tokens=30000),
    "whole": dataclasses.replace(W, T=2, scales=(1, 1), grid_h=16, grid_w=20, heads=17, head_dim=128,
                                 sink_tokens=900, batch=2),
}


def takes(name, r):
    """Whether the forms r (helpers.routes) are those that the case is there for."""
    form = name.split("_")[0]
    if form.startswith("cluster"):
        return r["cluster"] == int(form[-1])
    if form == "tile":
        return r["cluster"] > 0
    if form in ("one", "whole"):
        return r["cluster"] == 0 and r["whole"] == 1
    few = 2 <= r["pieces"] <= 8
    return r["cluster"] == 0 and r["whole"] == 0 and r["rounds"] == 0 and few == (form == "in") and r["pieces"] > 1


def _run(w):
    x = synth.attention_inputs(w, BF16)
    plan = make_plan(w, BF16)
    taken = routes(plan)
    dx = device_inputs(x, w.history_capacity)
    ws = bind(plan, dx)
    plan.kv_resample(dx["k_win"], dx["v_win"])
    outs = [torch.full_like(dx["q"], float("nan")) for _ in range(4)]
    L = torch.full((w.batch, w.heads, plan.info.n_tokens), float("nan"), device="cuda")
    plan.mssa_forward(dx["q"], dx["k_win"], dx["v_win"], outs[0])
    plan.mssa_forward_lse(dx["q"], dx["k_win"], dx["v_win"], outs[1], L)
    plan.mssa_forward_resample(dx["q"], dx["k_win"], dx["v_win"], outs[2])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plan.mssa_forward(dx["q"], dx["k_win"], dx["v_win"], outs[3])
    outs[3].fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert plan.device_status() == msf().MSF_OK
    del ws
    return x, outs, L, taken


@pytest.mark.parametrize("name", CASES)
def test_small_and_first_large_calls(name):
    w = CASES[name]
    x, outs, lse, taken = _run(w)
    assert takes(name, taken), taken
    for o in outs[1:]:
        assert torch.equal(outs[0], o)
    heads = None if w.heads <= 4 else [0, w.heads - 1]
    mx, mean = err_stats(outs[0], oracle_mssa(x, w, heads=heads), heads)
    assert mx <= 2e-2 and mean <= 2e-3, (mx, mean)
    if max(w.scales) == 1 and w.history_frames == 0:
        # fp32 sums of bf16 products: 1e-5 of a log-sum-exp of up to ~12
        q, k = x["q"].double(), torch.cat([x["k_sink"], x["k_win"]], 1).double()
        s = torch.einsum("bqhd,bkhd->bhqk", q[:, :, :1], k[:, :, :1]) * w.head_dim ** -0.5
        assert (lse[:, :1].double().cpu() - torch.logsumexp(s, -1)).abs().max() <= 1.2e-4


@pytest.mark.parametrize("dim", [64, 128])
def test_scores_that_outgrow_the_first_tile(dim):
    """The running maximum lags: later tiles hold much larger scores, so O, l
    and P are rescaled on the way (both warpgroups, several CTAs). With one
    dominant key per tile the bf16 rounding of P and of the output is all that
    is left: 2^-8 of values up to ~4."""
    w = dataclasses.replace(W, head_dim=dim, heads=2, sink_tokens=1500)
    assert routes(make_plan(w))["cluster"] > 1
    x = synth.attention_inputs(w, BF16)
    for i, t in enumerate(range(100, 1500, 128)):
        x["k_sink"][:, t] = (x["q"][:, 5] * (1 + i)).to(BF16)
    plan = make_plan(w, BF16)
    dx = device_inputs(x, w.history_capacity)
    ws = bind(plan, dx)
    out = torch.empty_like(dx["q"])
    plan.mssa_forward(dx["q"], dx["k_win"], dx["v_win"], out)
    torch.cuda.synchronize()
    assert plan.device_status() == msf().MSF_OK
    mx, _ = err_stats(out, oracle_mssa(x, w))
    assert mx <= 4e-2, mx
    del ws
