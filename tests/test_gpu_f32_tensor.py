"""fp32 attention on the tensor cores (three bf16 planes per value): tile edges
of every segment, both head sizes, whole and split query tiles, against the
fp64 oracle, and the operands the planes cannot hold.

Tolerance: scores of a 128-wide dot product of unit normals scaled by 1/sqrt(D)
carry an absolute error of a few 2^-24 times their size (up to ~6 here), the
probabilities the same relative error, and the output is a convex combination
of values up to ~5: 5 * 8 * 2^-24 * 6 = 1.5e-5 covers the worst element. The
log-sum-exp (up to ~10) rounds to 2^-24 of itself twice: 2e-6.
"""
import dataclasses

import pytest
import torch

from helpers import F32, bind, device_inputs, err_stats, make_plan, msf, oracle_mssa
from paper_2607_20940_gb300 import synth

pytestmark = pytest.mark.gpu

BASE = synth.Workload("f32", 3, (1, 1, 2), 8, 8, 2, 64, 0, 0, 0, 1, 50)
CASES = [
    # one query tile, one to three context tiles, single rows past an edge
    dataclasses.replace(BASE, T=1, scales=(1,), grid_h=1, grid_w=1, heads=1, sink_tokens=0),
    dataclasses.replace(BASE, T=1, scales=(1,), grid_h=1, grid_w=127, heads=3, sink_tokens=1, head_dim=128),
    dataclasses.replace(BASE, T=1, scales=(1,), grid_h=8, grid_w=16, heads=1, sink_tokens=129),
    dataclasses.replace(BASE, T=1, scales=(1,), grid_h=3, grid_w=43, heads=2, sink_tokens=128, head_dim=128),
    # every segment ragged, several groups, streams and history frames
    dataclasses.replace(BASE, T=4, scales=(1, 2, 2, 4), grid_h=12, grid_w=20, heads=3, head_dim=128, sink_tokens=77,
                        history_frames=2, history_capacity=3, batch=2),
    dataclasses.replace(BASE, T=3, scales=(1, 2, 4), grid_h=16, grid_w=28, heads=5, sink_tokens=33, history_frames=1,
                        history_capacity=1, batch=3),
    # few query tiles over a long context: the most units per tile
    dataclasses.replace(BASE, T=2, scales=(1, 2), grid_h=4, grid_w=6, heads=1, head_dim=128, sink_tokens=5000),
    # more query tiles than one round of the SMs: several rounds, mixed unit lengths
    dataclasses.replace(BASE, T=5, scales=(1, 1, 2, 2, 2), grid_h=30, grid_w=52, heads=3, head_dim=128,
                        sink_tokens=200, history_frames=1, history_capacity=2),
]


def _forward(w, x):
    plan = make_plan(w, F32)
    d = device_inputs(x, w.history_capacity)
    ws = bind(plan, d)
    out = torch.full_like(d["q"], float("nan"))
    lse = torch.full((w.batch, w.heads, plan.info.n_tokens), float("nan"), device="cuda")
    plan.kv_resample(d["k_win"], d["v_win"])
    plan.mssa_forward_lse(d["q"], d["k_win"], d["v_win"], out, lse)
    again = torch.empty_like(out)
    plan.mssa_forward(d["q"], d["k_win"], d["v_win"], again)
    simt = torch.empty_like(out)
    plan.mssa_forward_simt(d["q"], d["k_win"], d["v_win"], simt)
    torch.cuda.synchronize()
    assert plan.device_status() == msf().MSF_OK
    assert torch.equal(out, again) or torch.isnan(out).any()
    del ws
    return out, lse, simt


@pytest.mark.parametrize("w", CASES, ids=[f"{w.scales}-{w.grid_h}x{w.grid_w}-h{w.heads}-d{w.head_dim}" for w in CASES])
def test_f32_tensor_attention(w):
    x = synth.attention_inputs(w, F32)
    out, lse, simt = _forward(w, x)
    ref = oracle_mssa(x, w)
    mx, _ = err_stats(out, ref)
    assert mx <= 1.5e-5, mx
    # no further from the oracle than the CUDA-core kernel, on average (both
    # are near fp32's rounding; small windows differ by chance)
    assert err_stats(out, ref)[1] <= 1.5 * err_stats(simt, ref)[1] + 2e-8
    assert torch.isfinite(lse).all()


def test_f32_tensor_attention_lse():
    w = CASES[3]
    x = synth.attention_inputs(w, F32)
    _, lse, _ = _forward(w, x)
    q, k = x["q"].double(), torch.cat([x["k_sink"], x["k_win"]], 1).double()
    ref = torch.logsumexp(torch.einsum("bqhd,bkhd->bhqk", q, k) * w.head_dim ** -0.5, -1)
    assert (lse.double().cpu() - ref).abs().max() <= 2e-6


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), torch.finfo(F32).min, 2.0 ** 127])
@pytest.mark.parametrize("where", ["q", "k_win", "v_sink"])
def test_f32_values_the_planes_cannot_hold(value, where):
    """Such a call gives exactly what the CUDA-core kernel gives."""
    w = CASES[4]
    x = synth.attention_inputs(w, F32)
    x[where][1, 3, 1, 5] = value
    out, _, simt = _forward(w, x)
    assert torch.equal(torch.nan_to_num(out, nan=123.0), torch.nan_to_num(simt, nan=123.0))


def test_f32_tensor_attention_small_and_large_values():
    """Magnitudes far from one keep fp32's relative precision."""
    w = CASES[2]
    x = synth.attention_inputs(w, F32)
    x = {k: v * (2.0 ** 40 if k.startswith("q") else 2.0 ** -40 if k.startswith("k") else 2.0 ** -60)
         for k, v in x.items()}
    out, _, _ = _forward(w, x)
    mx, _ = err_stats(out * 2.0 ** 60, oracle_mssa(x, w) * 2.0 ** 60)
    assert mx <= 1.5e-5, mx
