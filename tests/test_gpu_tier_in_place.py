"""De-embedding with a latent residual whose output lies over its own input:
the state's latent is replaced in place (one stream, or one state), or the output
covers another part of the window latent. Bits as with separate buffers.
"""
import dataclasses

import pytest
import torch

from paper_2607_20940_gb300 import synth

from helpers import BF16, msf
from test_gpu_tier import SMALL, _setup

pytestmark = pytest.mark.gpu

CASES = {
    "small": (dataclasses.replace(SMALL, batch=1), 2),
    "480p": (synth.LAYER_480P, 4),  # more tiles than run at once
    "streams_one_state": (dataclasses.replace(SMALL, T=1, scales=(2,), batch=3), 0),
}


@pytest.mark.parametrize("shift", [0, 1], ids=["over_its_input", "over_part_of_it"])
@pytest.mark.parametrize("name", CASES)
def test_unpatchify_tier_over_its_input(name, shift):
    w, pos = CASES[name]
    plan, mi, dev, mods, _ = _setup(w, 16)
    lat = mi["latent"].cuda()
    B, C = w.batch, w.latent_channels
    n = lat[0, 0].numel()
    tok = torch.randn(B, plan.info.n_tokens, w.embed_dim, generator=torch.Generator().manual_seed(5)).to(BF16).cuda()
    apart = torch.full((B * n,), float("nan"), dtype=BF16, device="cuda")
    s = w.scales[pos]
    plan.unpatchify_tier(pos, tok, lat, mods[s], apart)
    # the window latent with room behind it; the output starts on the state's own
    # latent, or half a state later
    room = torch.zeros(lat.numel() + n, dtype=BF16, device="cuda")
    room[:lat.numel()] = lat.flatten()
    at = pos * n + shift * (n // 16 * 8)
    over = room[at:at + B * n]
    plan.unpatchify_tier(pos, tok, room[:lat.numel()].view_as(lat), mods[s], over)
    torch.cuda.synchronize()
    assert plan.device_status() == msf().MSF_OK
    assert torch.equal(over, apart)
