"""The GPU tests that are there for one form of the bf16 attention or gradient, on the
CPU: on 152 SMs every case takes the form that it names (the tests assert the same
on their device)."""
import dataclasses

import pytest

import test_gpu_backward_items as items
import test_gpu_forward_resample as resample
import test_gpu_merge_paths as merges
import test_gpu_merge_rest as rest
import test_gpu_small_calls as small
import test_gpu_whole_blocks as whole
from helpers import make_plan, routes

SMS = 152


@pytest.mark.parametrize("name", small.CASES)
def test_small_calls(name):
    r = routes(make_plan(small.CASES[name]), SMS)
    assert small.takes(name, r), r


@pytest.mark.parametrize("name", merges.CASES)
def test_merges(name):
    w, _, takes = merges.CASES[name]
    r = routes(make_plan(w), SMS)
    assert takes(r), r


@pytest.mark.parametrize("name,w", resample.CASES, ids=[c[0] for c in resample.CASES])
def test_one_launch(name, w):
    r = routes(make_plan(w), SMS)
    assert (w.head_dim == 128 and not r["cluster"] and not r["whole"]) == (name in resample.ONE), r


@pytest.mark.parametrize("w", whole.CASES, ids=lambda w: w.name)
def test_whole_blocks(w):
    r = routes(make_plan(w), SMS)
    assert r["whole"] == 1 and r["cluster"] == 0, r


@pytest.mark.parametrize("w", rest.CASES, ids=lambda w: w.name)
def test_rest(w):
    r = routes(make_plan(w), SMS)
    assert rest.takes_a_round_in(w, r), r


@pytest.mark.parametrize("name", items.CASES)
def test_backward_items(name):
    w, n, placed = items.CASES[name]
    r = routes(make_plan(w), SMS)
    assert (r["items"], r["placed"]) == (n, placed), r
    assert routes(make_plan(dataclasses.replace(w, batch=1)), SMS)["placed"] == 0
