"""De-embedding with and without a tier's extras at every cluster size, with
rings that wrap several times before the gathered residual chunks, and patch
edges of every gather width. Tolerance as in test_gpu_tier.py: 2^-7 of the
output's range (bf16 output rounding, one rounding of the codes).
"""
import dataclasses

import pytest

from paper_2607_20940_gb300 import synth

from test_gpu_tier import SMALL, _check_window

pytestmark = pytest.mark.gpu

CASES = {
    # clusters of eight (one 128-token tile), many chunks per CTA
    "e4096_one_tile": dataclasses.replace(SMALL, embed_dim=4096, batch=1),
    # sixteen to 72 clusters: four CTAs, six token chunks before the residual's
    "four": dataclasses.replace(synth.LAYER_480P, heads=2, batch=2),
    # four with a short contraction, two (73 clusters and more)
    "four_short": dataclasses.replace(synth.LAYER_480P, heads=2, batch=3, embed_dim=512),
    "two": dataclasses.replace(synth.LAYER_480P, heads=2, batch=5, embed_dim=512),
    "two_many": dataclasses.replace(synth.LAYER_480P, heads=1, batch=10, embed_dim=256),
    # one token chunk: no split, a tile column of 64 and no whole 192
    "e64": dataclasses.replace(SMALL, embed_dim=64),
    # patch edges 8 (16-byte gathers) and 16 (pixel by pixel)
    "patch4": dataclasses.replace(SMALL, patch=4, scales=(1, 2, 4, 4), latent_channels=4),
    "three_scales": dataclasses.replace(SMALL, scales=(1, 2, 4, 4), grid_h=16, grid_w=24, batch=3),
}


@pytest.mark.parametrize("name", CASES)
def test_tier_cluster_sizes(name):
    _check_window(CASES[name], 24)


def test_adapter_or_residual_alone():
    _check_window(CASES["two_many"], 64, lora=True, residual=False)
    _check_window(CASES["two_many"], 64, lora=False, residual=True)
    _check_window(CASES["e64"], 64, lora=True, residual=False)  # one CTA per tile
