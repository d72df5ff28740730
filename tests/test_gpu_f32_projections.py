"""fp32 patch embedding and de-embedding on the tensor cores: tile edges, K
chunk remainders, cluster splits, shared and separate tier weights, streams,
chunks of frames, and operands the bf16 planes cannot hold.

Tolerance against fp64: products are exact to 2^-24 of themselves and sums of K
unit-variance terms (weights N(0, 1/K)) round to a few 2^-24 of values up to
~5: 5e-6 covers the worst element.
"""
import pytest
import torch

from helpers import F32, msf
from paper_2607_20940_gb300 import synth

pytestmark = pytest.mark.gpu

#        scales      grid      E    C  patch batch frames
SHAPES = [
    ((1,), (1, 1), 64, 16, 2, 1, 1),        # one token, one K chunk
    ((1, 2), (6, 22), 192, 3, 2, 2, 1),     # K = 12 and 48: part of a chunk; N a tile and a half
    ((1, 1, 2, 2, 4), (16, 24), 200, 16, 2, 1, 1),  # N not a tile's multiple, runs of states, K = 1024
    ((2, 2, 4), (12, 20), 1536, 16, 2, 1, 2),       # coarse only, frames per state
    ((1, 2, 2), (30, 52), 1536, 16, 2, 2, 1),       # several tiles each way, two streams
    ((1, 1), (10, 13), 4100, 16, 1, 1, 1),          # de-embedding: 64 tokens' K remainder, N = 16
]


# The ways into the latent: one, two (a token per thread) and four CTAs a tile (a
# token's features over the threads), stores of 1, 2 and 4 pixels, 64- and 128-wide
# tiles, a last tile of few tokens and features.
INTO_LATENT = [
    ((1, 2), (6, 22), 64, 3, 1, 2, 1),      # edge 1 and 2; N = 3 x 1 and 12: not vectors of four, then one
    ((1, 2), (10, 14), 64, 4, 3, 1, 1),     # edge 3 and 6
    ((1, 2, 4), (16, 24), 64, 16, 2, 3, 1),  # edge 2, 4, 8; N = 64, 256, 1024
    ((1, 2), (12, 20), 320, 16, 3, 1, 2),   # two CTAs; N = 144 and 576
    ((2, 4), (12, 20), 576, 5, 2, 2, 1),    # four CTAs; N = 80 and 320
]


def _run(shape, edit=None):
    scales, (gh, gw), E, C, patch, B, F = shape
    w = synth.Workload("p", len(scales), scales, gh, gw, 1, 64, 0, 0, 0, B, 70, latent_channels=C, patch=patch,
                       embed_dim=E, frames=F)
    m = msf()
    plan = m.Plan(m.make_desc(scales, gh, gw, 1, 64, 0, 0, batch=B, dtype=m.MSF_DTYPE_F32, latent_channels=C,
                              patch=patch, embed_dim=E, frames_per_state=F))
    ws = plan.workspace()
    plan.bind(ws, None, None, None, None)
    g = torch.Generator().manual_seed(7)
    lat = torch.randn(B, len(scales), C, F, gh * patch, gw * patch, generator=g)
    wt = {s: torch.randn(E, C * (patch * s) ** 2, generator=g) * (C * (patch * s) ** 2) ** -0.5 for s in set(scales)}
    wo = {s: torch.randn(C * (patch * s) ** 2, E, generator=g) * E ** -0.5 for s in set(scales)}
    N = plan.info.n_tokens
    h = torch.randn(B, N, E, generator=g)
    if edit:
        edit(lat, wt, h, wo)
    dev = {s: v.cuda() for s, v in wt.items()}
    tok = torch.full((B, N, E), float("nan"), device="cuda")
    plan.patchify(lat.cuda(), [dev[s] for s in scales], tok)
    back, hd = [], h.cuda()
    for l, s in enumerate(scales):
        y = torch.full(lat[:, l].shape, float("nan"), device="cuda")
        plan.unpatchify(l, hd, wo[s].cuda(), y)
        back.append(y.cpu())
    torch.cuda.synchronize()
    assert plan.device_status() == m.MSF_OK
    del ws
    toks, lats, off = [], [], 0
    for l, s in enumerate(scales):
        P = patch * s
        x = lat[:, l].double().reshape(B, C, F * gh // s, P, gw // s, P)
        n = F * (gh // s) * (gw // s)
        rows = x.permute(0, 2, 4, 1, 3, 5).reshape(B, n, C * P * P)
        toks.append(rows @ wt[s].double().T)
        y = (h[:, off:off + n].double() @ wo[s].double().T).reshape(B, F * gh // s, gw // s, C, P, P)
        lats.append(y.permute(0, 3, 1, 4, 2, 5).reshape(lat[:, l].shape))
        off += n
    return tok.cpu(), torch.cat(toks, 1), back, lats


@pytest.mark.parametrize("shape", SHAPES + INTO_LATENT,
                         ids=[f"{s[0]}-{s[1]}-E{s[2]}-C{s[3]}" for s in SHAPES + INTO_LATENT])
def test_f32_projections(shape):
    tok, ref, back, lats = _run(shape)
    assert (tok.double() - ref).abs().max() <= 5e-6
    for y, r in zip(back, lats):
        assert (y.double() - r).abs().max() <= 5e-6


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), torch.finfo(F32).min])
def test_f32_projections_of_values_the_planes_cannot_hold(value):
    def edit(lat, wt, h, wo):
        lat[0, 1, 2, 0, 3, 5] = value
        h[1, 7, 11] = value
    tok, ref, back, lats = _run(SHAPES[1], edit)
    ref32 = ref.float()  # fp64 sums of |value| up to fp32's range round to it or to infinity
    for a, b in [(tok, ref32)] + list(zip(back, [x.float() for x in lats])):
        assert torch.equal(torch.isnan(a), torch.isnan(b))
        assert torch.equal(torch.isinf(a), torch.isinf(b)) and torch.equal(a[torch.isinf(a)], b[torch.isinf(b)])
        f = torch.isfinite(b)
        assert ((a[f] - b[f]).abs() <= 5e-6 * b[f].abs().clamp(min=1.0)).all()


@pytest.mark.parametrize("ua,ub", [(-40, 40), (-112, 112), (112, -112), (-112, 0), (0, -105), (-60, -55), (60, 60)])
def test_f32_projections_magnitudes(ua, ub):
    """fp32's precision on both sides of csrc/f32_range.h (powers of two change no rounding)."""
    def edit(lat, wt, h, wo):
        lat *= 2.0 ** ua
        h *= 2.0 ** ua
        for x in (wt, wo):
            for s in x:
                x[s] *= 2.0 ** ub
    tok, ref, back, lats = _run(SHAPES[1], edit)
    u = 2.0 ** -(ua + ub)
    assert ((tok.double() - ref) * u).abs().max() <= 5e-6
    for y, r in zip(back, lats):
        assert ((y.double() - r) * u).abs().max() <= 5e-6


@pytest.mark.parametrize("shape", [SHAPES[2], SHAPES[4]], ids=["runs", "two_streams"])
def test_f32_unpatchify_over_its_tokens(shape):
    """A latent written over the tokens (or the weight) that it is computed from
    has the bits of one written elsewhere."""
    scales, (gh, gw), E, C, patch, B, F = shape
    m = msf()
    plan = m.Plan(m.make_desc(scales, gh, gw, 1, 64, 0, 0, batch=B, dtype=m.MSF_DTYPE_F32, latent_channels=C,
                              patch=patch, embed_dim=E, frames_per_state=F))
    ws = plan.workspace()
    plan.bind(ws, None, None, None, None)
    g = torch.Generator(device="cuda").manual_seed(3)
    n = C * F * gh * gw * patch * patch
    for pos in (0, len(scales) - 1):
        h = torch.randn(B, plan.info.n_tokens, E, generator=g, device="cuda")
        w = torch.randn(C * (patch * scales[pos]) ** 2, E, generator=g, device="cuda")
        apart = torch.full((B * n,), float("nan"), device="cuda")
        plan.unpatchify(pos, h, w, apart)
        for over_tokens in (True, False):
            src = h if over_tokens else w
            room = torch.zeros(max(src.numel(), B * n) + 64, device="cuda")
            room[32:32 + src.numel()] = src.flatten()
            x = room[32:32 + src.numel()].view_as(src)
            y = room[:B * n]
            plan.unpatchify(pos, x if over_tokens else h, w if over_tokens else x, y)
            torch.cuda.synchronize()
            assert plan.device_status() == m.MSF_OK
            assert torch.equal(y, apart)
    del ws
