"""fp32 attention calls of one plan on several streams, from several threads and
on the branches of one capture: each gives the bits that it gives alone.

The operands' planes lie in the plan's workspace, so the calls have to run one
after the other on the device. The inputs are larger than one wave of units, and
the streams start together behind a busy kernel, so that unordered calls would meet.
"""
import ctypes
import threading

import pytest
import torch

from helpers import F32, bind, device_inputs, make_plan, msf
from paper_2607_20940_gb300 import synth

pytestmark = pytest.mark.gpu

W = synth.Workload("streams", 4, (1, 1, 2, 2), 24, 40, 6, 128, 300, 1, 1, 1, 81)
N_STREAMS, ROUNDS = 3, 6


def _setup():
    x = synth.attention_inputs(W, F32)
    plan = make_plan(W, F32)
    d = device_inputs(x, W.history_capacity)
    ws = bind(plan, d)
    plan.kv_resample(d["k_win"], d["v_win"])
    g = torch.Generator(device="cuda").manual_seed(4)
    calls = []
    for i in range(N_STREAMS):
        q = torch.randn(d["q"].shape, generator=g, device="cuda")
        c = {"q": q, "out": torch.empty_like(q), "dout": torch.randn(q.shape, generator=g, device="cuda"),
             "lse": torch.empty((1, W.heads, plan.info.n_tokens), device="cuda"),
             "grads": [torch.empty_like(q) for _ in range(3)], "bws": plan.backward_workspace(),
             "stream": torch.cuda.Stream()}
        calls.append(c)
    torch.cuda.synchronize()
    return plan, d, ws, calls


def _pass(plan, d, c):
    plan.mssa_forward_lse(c["q"], d["k_win"], d["v_win"], c["out"], c["lse"])
    plan.mssa_backward(c["q"], d["k_win"], d["v_win"], c["out"], c["dout"], c["lse"], *c["grads"], c["bws"])


def _results(c):
    return [c["out"], c["lse"], *c["grads"]]


def _alone(plan, d, calls):
    ref = []
    for c in calls:
        _pass(plan, d, c)
        torch.cuda.synchronize()
        ref.append([t.clone() for t in _results(c)])
        for t in _results(c):
            t.fill_(float("nan"))
    torch.cuda.synchronize()
    return ref


def _check(plan, calls, ref):
    torch.cuda.synchronize()
    assert plan.device_status() == msf().MSF_OK
    for c, r in zip(calls, ref):
        assert all(torch.equal(a, b) for a, b in zip(_results(c), r))


def test_streams():
    plan, d, ws, calls = _setup()
    ref = _alone(plan, d, calls)
    for _ in range(ROUNDS):
        torch.cuda._sleep(2_000_000)  # the current stream; the others queue up behind it
        start = torch.cuda.Event()
        start.record()
        for c in calls:
            c["stream"].wait_event(start)
        for c in calls:
            with torch.cuda.stream(c["stream"]):
                _pass(plan, d, c)
        _check(plan, calls, ref)
    del ws


def test_stream_that_is_gone():
    """The stream of an earlier call may be destroyed before the next one, its work still running."""
    plan, d, ws, calls = _setup()
    ref = _alone(plan, d, calls)
    rt = torch.cuda.cudart()
    for _ in range(ROUNDS):
        for c in calls:
            s = ctypes.c_void_p()
            assert int(rt.cudaStreamCreate(ctypes.addressof(s))) == 0
            with torch.cuda.stream(torch.cuda.ExternalStream(s.value)):
                _pass(plan, d, c)
            assert int(rt.cudaStreamDestroy(s.value)) == 0
        _check(plan, calls, ref)
    del ws


def test_threads():
    plan, d, ws, calls = _setup()
    ref = _alone(plan, d, calls)
    errors = []

    def work(c):
        try:
            with torch.cuda.stream(c["stream"]):
                for _ in range(ROUNDS):
                    _pass(plan, d, c)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    _check(plan, calls, ref)
    del ws


def test_branches_of_a_capture():
    plan, d, ws, calls = _setup()
    ref = _alone(plan, d, calls)
    main = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        for c in calls:
            c["stream"].wait_stream(main)
        for c in calls:
            with torch.cuda.stream(c["stream"]):
                _pass(plan, d, c)
        for c in calls:
            main.wait_stream(c["stream"])
    for _ in range(2):
        for c in calls:
            for t in _results(c):
                t.fill_(float("nan"))
        torch.cuda.synchronize()
        graph.replay()
        _check(plan, calls, ref)
    # calls outside the capture again
    for c in calls:
        with torch.cuda.stream(c["stream"]):
            _pass(plan, d, c)
    _check(plan, calls, ref)
    del ws


def test_while_another_stream_captures():
    """Calls on a stream that is not captured, the plan's first among them, go on
    while another one is, and neither side waits on the other's events."""
    plan, d, ws, calls = _setup()
    fresh, fd, fws, fcalls = _setup()
    ref = _alone(plan, d, calls)
    graph, main = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=main):
        _pass(plan, d, calls[0])
        for p, pd, c in ((plan, d, calls[1]), (fresh, fd, fcalls[2])):
            with torch.cuda.stream(c["stream"]):
                _pass(p, pd, c)
        _pass(plan, d, calls[0])
    torch.cuda.synchronize()
    _check(plan, calls[1:2], ref[1:2])
    _check(fresh, fcalls[2:], ref[2:])
    graph.replay()
    _check(plan, calls[:1], ref[:1])
    del ws, fws
