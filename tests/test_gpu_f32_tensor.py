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


def _forward(w, x, plan=None):
    plan = plan or make_plan(w, F32)
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


# ---- magnitudes on both sides of csrc/f32_range.h. Outside, the call gives exactly
# what the CUDA-core kernel gives; on both sides fp32's precision is kept (the same
# bounds as above, of results scaled back: powers of two change no rounding).
def _scaled(w, uq=0, uk=0, uv=0):
    x = synth.attention_inputs(w, F32)
    u = {"q": uq, "k": uk, "v": uv}
    return {k: t * 2.0 ** u[k[0]] for k, t in x.items()}


@pytest.mark.parametrize("uq,uk,uv", [(40, -40, -90), (-40, 40, 90), (0, 0, -112), (0, 0, -118), (55, -55, 99),
                                      (-112, 112, 0), (112, -112, 0), (-105, 105, -105)])
@pytest.mark.parametrize("w", [CASES[3], CASES[4]], ids=["one_group", "groups"])
def test_f32_attention_magnitudes(w, uq, uk, uv):
    out, _, simt = _forward(w, _scaled(w, uq, uk, uv))
    if max(abs(uq), abs(uk), abs(uv)) > 97:
        assert torch.equal(out, simt)
    mx, _ = err_stats(out.double() * 2.0 ** -uv, oracle_mssa(_scaled(w), w))
    assert mx <= 1.5e-5, mx


@pytest.mark.parametrize("u", [-97, -112])
def test_f32_attention_one_small_head(u):
    """One head's values far below the others': it keeps its own precision."""
    w = CASES[4]
    x = synth.attention_inputs(w, F32)
    ref = oracle_mssa(x, w)
    for k in ("v_win", "v_sink", "v_hist"):
        x[k][..., 1, :] *= 2.0 ** u
    out, _, _ = _forward(w, x)
    out = out.double()
    out[..., 1, :] *= 2.0 ** -u
    mx, _ = err_stats(out, ref)
    assert mx <= 1.5e-5, mx


def test_f32_attention_scores_past_fp32_before_the_scale():
    """q k reaches 2^130, the scaled scores 2^5."""
    w = CASES[3]
    m = msf()
    plan = m.Plan(m.make_desc(w.scales, w.grid_h, w.grid_w, w.heads, w.head_dim, w.sink_tokens, 0, dtype=m.MSF_DTYPE_F32,
                              softmax_scale=2.0 ** -126 * w.head_dim ** -0.5 * 4))
    out, lse, simt = _forward(w, _scaled(w, 62, 62), plan)
    assert torch.equal(out, simt)
    mx, _ = err_stats(out, oracle_mssa(_scaled(w), w))
    assert mx <= 1.5e-5 and torch.isfinite(lse).all(), mx


def test_f32_attention_score_below_fp32():
    """A key whose score is minus infinity has no weight (after a first key that has)."""
    w = dataclasses.replace(CASES[0], sink_tokens=300)
    x = synth.attention_inputs(w, F32)
    x["q"] *= 2.0 ** 40
    x["k_sink"] *= 2.0 ** -40
    x["k_win"] *= 2.0 ** -40
    x["k_sink"][:, 130:290] = -2.0 ** 100 * torch.sign(x["q"])
    out, _, simt = _forward(w, x)
    assert torch.isfinite(out).all() and torch.equal(out, simt)


@pytest.mark.parametrize("uv,ug", [(0, -30), (-30, -30), (0, -112), (-45, -45), (-40, -60), (45, 45), (99, -40)])
def test_f32_backward_magnitudes(uv, ug):
    from oracle import mssa_bwd as obwd
    w = CASES[4]
    dout, (got, _, simt) = _backward(w, _scaled(w, uv=uv), scale=2.0 ** ug)
    if uv + ug < -70 or uv + ug > 80 or max(abs(uv), abs(ug)) > 97:
        assert all(torch.equal(a, b) for a, b in zip(got, simt))
    f = synth.to_f64
    x = synth.attention_inputs(w, F32)
    ref = obwd.mssa_backward(f(x["q"]), f(x["k_win"]), f(x["v_win"]), f(x["k_sink"]), f(x["v_sink"]), f(x["k_hist"]),
                             f(x["v_hist"]), f(dout), w.scales, w.grid_h, w.grid_w)
    for g, key, u in zip(got, ("dq", "dk_win", "dv_win"), (uv + ug, uv + ug, ug)):
        e = abs(g.double().cpu().numpy() * 2.0 ** -u - ref[key]).max() / abs(ref[key]).max()
        assert e <= 1e-5, (key, e)


def _backward(w, x, seed=9, scale=1.0):
    plan = make_plan(w, F32)
    d = device_inputs(x, w.history_capacity)
    ws = bind(plan, d)
    out = torch.empty_like(d["q"])
    lse = torch.empty((w.batch, w.heads, plan.info.n_tokens), device="cuda")
    dout = torch.randn(d["q"].shape, generator=torch.Generator().manual_seed(seed))
    plan.kv_resample(d["k_win"], d["v_win"])
    plan.mssa_forward_lse(d["q"], d["k_win"], d["v_win"], out, lse)
    bws = plan.backward_workspace()
    got = []
    for fn in (plan.mssa_backward, plan.mssa_backward, plan.mssa_backward_simt):
        g = [torch.full_like(d["q"], float("nan")) for _ in range(3)]
        fn(d["q"], d["k_win"], d["v_win"], out, (dout * scale).cuda(), lse, *g, bws)
        got.append(g)
    torch.cuda.synchronize()
    assert plan.device_status() == msf().MSF_OK
    del ws
    return dout, got


# Gradients: sums of up to a few thousand products P * (dP - delta) * k with
# |P| <= 1 and dP around sqrt(D); fp32 sums of them in any order differ by less
# than 2^-24 times the terms' absolute sum, well below 1e-5 of the largest
# gradient (the CUDA-core kernels show up to 2e-6 of it).
@pytest.mark.parametrize("w", CASES[:7], ids=[f"{w.scales}-{w.grid_h}x{w.grid_w}-h{w.heads}-d{w.head_dim}" for w in CASES[:7]])
@pytest.mark.parametrize("mode", [0, 1], ids=["avg", "strided"])
def test_f32_tensor_backward(w, mode):
    from oracle import mssa_bwd as obwd
    if mode and max(w.scales) == 1:
        pytest.skip("no pooling")
    x = synth.attention_inputs(w, F32)
    m = msf()
    desc = m.make_desc(w.scales, w.grid_h, w.grid_w, w.heads, w.head_dim, w.sink_tokens, w.history_frames,
                       history_capacity=w.history_capacity, batch=w.batch, dtype=m.MSF_DTYPE_F32, resample=mode)
    plan = m.Plan(desc)
    d = device_inputs(x, w.history_capacity)
    ws = bind(plan, d)
    out = torch.empty_like(d["q"])
    lse = torch.empty((w.batch, w.heads, plan.info.n_tokens), device="cuda")
    dout = torch.randn(d["q"].shape, generator=torch.Generator().manual_seed(9))
    plan.kv_resample(d["k_win"], d["v_win"])
    plan.mssa_forward_lse(d["q"], d["k_win"], d["v_win"], out, lse)
    bws = plan.backward_workspace()
    got = []
    for _ in range(2):
        g = [torch.full_like(d["q"], float("nan")) for _ in range(3)]
        plan.mssa_backward(d["q"], d["k_win"], d["v_win"], out, dout.cuda(), lse, *g, bws)
        got.append(g)
    torch.cuda.synchronize()
    assert plan.device_status() == m.MSF_OK
    assert all(torch.equal(a, b) for a, b in zip(*got))
    f = synth.to_f64
    ref = obwd.mssa_backward(f(x["q"]), f(x["k_win"]), f(x["v_win"]), f(x["k_sink"]), f(x["v_sink"]), f(x["k_hist"]),
                             f(x["v_hist"]), f(dout), w.scales, w.grid_h, w.grid_w, mode=mode)
    for g, key in zip(got[0], ("dq", "dk_win", "dv_win")):
        e = abs(g.double().cpu().numpy() - ref[key]).max() / max(abs(ref[key]).max(), 1e-30)
        # one key in all (a 1 x 1 window without a cache): dS is 0 in exact arithmetic
        assert e <= 1e-5 or abs(ref[key]).max() < 1e-12, (key, e)
    del ws


@pytest.mark.parametrize("D,keys", [(64, 12), (64, 13), (64, 24), (64, 25), (128, 10), (128, 11), (128, 18), (128, 19)])
def test_f32_few_keys(D, keys):
    """On either side of the number of keys from which the tensor cores are ahead."""
    from oracle import mssa_bwd as obwd
    w = dataclasses.replace(CASES[0], grid_w=keys - 5, sink_tokens=5, heads=3, head_dim=D, batch=2)
    x = synth.attention_inputs(w, F32)
    out, lse, simt = _forward(w, x)
    if keys <= (24 if D == 64 else 18):
        assert torch.equal(out, simt)
    mx, _ = err_stats(out, oracle_mssa(x, w))
    assert mx <= 1.5e-5 and torch.isfinite(lse).all(), mx
    dout, (got, again, simt) = _backward(w, x)
    assert all(torch.equal(a, b) for a, b in zip(got, again))
    if keys <= (12 if D == 64 else 10):
        assert all(torch.equal(a, b) for a, b in zip(got, simt))
    f = synth.to_f64
    ref = obwd.mssa_backward(f(x["q"]), f(x["k_win"]), f(x["v_win"]), f(x["k_sink"]), f(x["v_sink"]), f(x["k_hist"]),
                             f(x["v_hist"]), f(dout), w.scales, w.grid_h, w.grid_w)
    for g, key in zip(got, ("dq", "dk_win", "dv_win")):
        e = abs(g.double().cpu().numpy() - ref[key]).max() / abs(ref[key]).max()
        assert e <= 1e-5, (key, e)


@pytest.mark.parametrize("value", [float("inf"), float("nan"), torch.finfo(F32).min])
@pytest.mark.parametrize("where", ["q", "k_win", "v_sink"])
def test_f32_backward_values_the_planes_cannot_hold(value, where):
    w = CASES[4]
    x = synth.attention_inputs(w, F32)
    x[where][1, 3, 1, 5] = value
    _, (got, _, simt) = _backward(w, x)
    for a, b in zip(got, simt):
        assert torch.equal(torch.nan_to_num(a, nan=123.0), torch.nan_to_num(b, nan=123.0))
