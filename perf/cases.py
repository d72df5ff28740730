"""Performance cases of the window pass: what a program does with this library.

A case is one call sequence of such a program, at a size of its range:

  window   K/V pyramid + multi-scale attention of one layer (`kv_resample`, `mssa_forward`)
  step     one denoising step of a layer: patchify + embedding, pyramid, attention,
           de-embedding of the emitted head (bf16: the one-launch embedding + pyramid with
           the history head staged; fp32: the separate calls)
  rollout  the first steps of a new stream: `step` with the history growing from nothing to
           the ring's capacity and past it
  train    attention forward with the row log-sum-exp, and its gradient
  tiers    embedding and de-embedding with the coarse tiers' modules (LoRA, latent residual)

Sizes are the repository's workloads (`synth.py`): the 480p layer (T = 5, 30 x 52 tokens,
12 heads x 128), its three-frame chunks, the three-scale 48 x 80 window and the tiny window,
and generic ones with ragged segments, 64-wide heads, odd head counts and no history.
"""
import math

import torch

from paper_2607_20940_gb300 import msf

CHANNELS, PATCH = 16, 2  # the latent's channels and the native patch edge of every workload


def _case(name, op, scales, grid, heads, dim, sink, hist, batch=1, frames=1, dtype="bf16", mode="avg", steps=1,
          fused=0, rank=0):
    c = {"op": op, "scales": ",".join(str(s) for s in scales), "gh": grid[0], "gw": grid[1], "heads": heads,
         "dim": dim, "sink": sink, "hist": hist, "batch": batch, "frames": frames, "dtype": dtype, "mode": mode,
         "steps": steps, "fused": fused, "rank": rank}
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # The smallest call: latency and launches are all there is.
        _case("window_tiny", "window", (1, 1, 2), (8, 8), 2, 64, 64, 1),
        # One layer of the 480p window, the library's ordinary call.
        _case("window_480p", "window", (1, 1, 2, 2, 2), (30, 52), 12, 128, 1560, 2),
        # A larger grid with three patch sizes: a deep pyramid, few fine queries.
        _case("window_3scale", "window", (1, 1, 2, 2, 4, 4), (48, 80), 16, 128, 3840, 2),
        # Nothing a multiple of a tile: ragged segments, odd head count, 64-wide heads, strided keys.
        _case("window_ragged_d64", "window", (1, 2, 2, 4), (36, 44), 5, 64, 77, 1, batch=2, mode="strided"),
        # One denoising step of a layer with the history update folded in.
        _case("step_480p", "step", (1, 1, 2, 2, 2), (30, 52), 12, 128, 1560, 2, fused=1),
        # Two streams from their first frame on, past the ring's capacity.
        _case("rollout_480p_b2", "rollout", (1, 1, 2, 2, 2), (30, 52), 12, 128, 1560, 3, batch=2, steps=5, fused=1),
        # Training through the window at 480p, ...
        _case("train_480p", "train", (1, 1, 2, 2, 2), (30, 52), 12, 128, 1560, 2),
        # ... at a small ragged window with 64-wide heads, ...
        _case("train_small_d64", "train", (1, 2, 2), (18, 26), 6, 64, 33, 1, batch=2),
        # ... and in the layout of the streaming model, whose states are chunks of three frames.
        _case("train_chunk3", "train", (1, 1, 2, 2, 2), (30, 52), 12, 128, 4680, 1, frames=3),
        # The coarse tiers' own embedding and de-embedding.
        _case("tiers_480p", "tiers", (1, 1, 2, 2, 2), (30, 52), 12, 128, 1560, 2, rank=32),
        # fp32 plans: a whole step (the run that a bf16 result is checked with) and a small training window.
        _case("step_480p_f32", "step", (1, 1, 2, 2, 2), (30, 52), 12, 128, 1560, 2, dtype="f32"),
        _case("train_small_f32", "train", (1, 2, 4), (16, 24), 4, 128, 70, 1, frames=2, dtype="f32"),
    ]


def draw(rng):
    """One more case: the same calls over the whole range of sizes, odd ones included."""
    while True:
        op = rng.choice(["window"] * 4 + ["train"] * 4 + ["step"] * 2 + ["rollout", "tiers"])
        dtype = "f32" if op in ("window", "step", "train") and rng.random() < 0.2 else "bf16"
        scales = rng.choice([(1, 1), (1, 2), (1, 1, 1), (1, 1, 2), (1, 2, 2), (1, 2, 4), (1, 2, 2, 4), (1, 1, 2, 2),
                             (1, 1, 2, 2, 2), (1, 1, 2, 2, 4), (1, 1, 2, 2, 4, 4)])
        top = scales[-1]
        side = lambda: max(1, round(math.exp(rng.uniform(math.log(8), math.log(64))) / top)) * top  # noqa: E731
        dim = rng.choice([64, 128, 128])
        sink = rng.choice([0, rng.randint(1, 200), rng.randint(200, 4000)])
        hist = rng.randint(0, 4)
        fused = rng.randint(0, 1)
        steps = rng.randint(3, 6) if op == "rollout" else 1
        if op == "rollout" or (op == "step" and fused):
            hist = max(hist, 1)
        c = _case(None, op, scales, (side(), side()), rng.randint(1, 16), dim, sink, hist,
                  batch=rng.choice([1, 1, 1, 2, 3, 4]), frames=rng.choice([1, 1, 1, 2, 3]), dtype=dtype,
                  mode=rng.choice(["avg", "avg", "strided"]), steps=steps,
                  fused=fused if op in ("step", "rollout") and dtype == "bf16" else 0,
                  rank=rng.choice([8, 16, 32, 64]) if op == "tiers" else 0)
        w = work(c)
        most = 3e12 if dtype == "bf16" else 2e10 if op == "train" else 1e11
        if w["flops"] <= most and w["bytes"] <= 1.5e9:
            return c


# --------------------------------------------------------------- shapes

def _scales(c):
    return [int(s) for s in c["scales"].split(",")]


def _sizes(c):
    """Fine tokens, tokens of each state, their offsets and the window's tokens."""
    G = c["frames"] * c["gh"] * c["gw"]
    n = [G // (s * s) for s in _scales(c)]
    off = [sum(n[:i]) for i in range(len(n) + 1)]
    return G, n, off


def _groups(c):
    """(scale, first state, one past the last) of each query group."""
    s, out = _scales(c), []
    for i, v in enumerate(s):
        if i and v == s[i - 1]:
            out[-1][2] = i + 1
        else:
            out.append([v, i, i + 1])
    return out


def _live(c, step):
    """Live history frames at a step (a rollout starts with none)."""
    return min(step, c["hist"]) if c["op"] == "rollout" else c["hist"]


def _embeds(c):
    return c["op"] in ("step", "rollout", "tiers")


def work(case):
    c = case
    s = _scales(c)
    G, n, off = _sizes(c)
    H, D, B, N = c["heads"], c["dim"], c["batch"], off[-1]
    e = 4 if c["dtype"] == "f32" else 2
    row = H * D * e
    flops = bytes_ = 0
    E = H * D
    lat = CHANNELS * PATCH * PATCH * G  # latent values of a state
    if c["op"] != "tiers":
        for step in range(c["steps"]):
            h = _live(c, step)
            for g, a, z in _groups(c):
                nq = off[z] - off[a]
                win = sum(G // (max(g, v) ** 2) for v in s)
                nkv = c["sink"] + h * G // (g * g) + win
                flops += 4 * D * H * B * nq * nkv
                if c["op"] == "train":
                    flops += B * H * nq * (6 * D * nkv + 4 * D * win)
            bytes_ += 4 * B * N * row + 2 * B * (c["sink"] + h * G) * row  # q, k, v, out; the cache's k, v
            if c["op"] == "train":
                bytes_ += 4 * B * N * row + 4 * B * H * N  # dout, dq, dk, dv; the log-sum-exp
            if c["op"] == "rollout" or c["fused"]:
                bytes_ += 2 * B * G * row  # the head's k, v into the ring
    if _embeds(c):
        weights = sum(CHANNELS * (PATCH * v) ** 2 * E for v in set(s))
        flops_t = sum(2 * B * m * CHANNELS * (PATCH * v) ** 2 * E for v, m in zip(s, n))
        back = _emitted(c)
        for _ in range(c["steps"]):
            flops += flops_t + sum(2 * B * lat * E for _ in back)
            bytes_ += B * len(s) * lat * e + B * N * E * e + weights * e  # latent in, tokens out
            bytes_ += len(back) * B * lat * e + sum(CHANNELS * (PATCH * v) ** 2 * E * e for v in {s[p] for p in back})
        if c["op"] == "tiers":
            r = c["rank"]
            bytes_ += sum(B * n[p] * E * e for p in back)  # the backbone's tokens
            for v, m in zip(s, n):
                K = CHANNELS * (PATCH * v) ** 2
                if v > 1:
                    flops += 2 * B * m * (2 * r * (K + E) + K * K)
            for v in set(s):
                K = CHANNELS * (PATCH * v) ** 2
                if v > 1:
                    bytes_ += (2 * r * (K + E) + K * K) * e
    return {"bytes": bytes_, "flops": flops}


def _emitted(c):
    """Window positions that are de-embedded: the head, or every state for the tiers."""
    return list(range(len(_scales(c)))) if c["op"] == "tiers" else [0]


# -------------------------------------------------------------- the program

def _dtype(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _inputs(c, seed):
    """Everything the call reads. Heads differ in how peaked their attention is, as after
    the normalised q/k projections of a trained model: q is scaled by 0.5 to 2 per head."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = _dtype(c)

    def randn(*shape, std=1.0):
        return (torch.randn(*shape, generator=gen, device="cuda") * std).to(dt)

    G, n, off = _sizes(c)
    H, D, B, N, E = c["heads"], c["dim"], c["batch"], off[-1], c["heads"] * c["dim"]
    x = {}
    if c["op"] != "tiers":
        gain = torch.exp2(torch.rand(H, 1, generator=gen, device="cuda") * 2 - 1)
        x["q"] = [(torch.randn(B, N, H, D, generator=gen, device="cuda") * gain).to(dt) for _ in range(c["steps"])]
        x["k"] = [randn(B, N, H, D) for _ in range(c["steps"])]
        x["v"] = [randn(B, N, H, D) for _ in range(c["steps"])]
    if c["op"] == "train":
        x["dout"] = randn(B, N, H, D)
    x["k_sink"], x["v_sink"] = randn(B, max(c["sink"], 1), H, D), randn(B, max(c["sink"], 1), H, D)
    slots = max(c["hist"] + c["fused"], 1)
    x["k_hist"], x["v_hist"] = randn(B, slots, G, H, D), randn(B, slots, G, H, D)
    if _embeds(c):
        s = _scales(c)
        lat = (B, len(s), CHANNELS, c["frames"], c["gh"] * PATCH, c["gw"] * PATCH)
        x["latent"] = [randn(*lat) for _ in range(c["steps"])]
        for v in sorted(set(s)):
            K = CHANNELS * (PATCH * v) ** 2
            x["w%d" % v] = randn(E, K, std=K ** -0.5)
            x["o%d" % v] = randn(K, E, std=E ** -0.5)
            if c["op"] == "tiers" and v > 1:
                r = c["rank"]
                x["ad%d" % v], x["au%d" % v] = randn(r, K, std=K ** -0.5), randn(E, r, std=r ** -0.5)
                x["bd%d" % v], x["bu%d" % v] = randn(r, E, std=E ** -0.5), randn(K, r, std=r ** -0.5)
                x["res%d" % v] = randn(K, K, std=K ** -0.5)
        if c["op"] == "tiers":
            x["h"] = randn(B, N, E)  # the backbone's output tokens
    return x


def prepare(case, seed):
    c = case
    x = _inputs(c, seed)
    G, n, off = _sizes(c)
    H, D, B, N = c["heads"], c["dim"], c["batch"], off[-1]
    dt = _dtype(c)
    rolls = c["op"] == "rollout"
    plan = msf.Plan(msf.make_desc(
        _scales(c), c["gh"], c["gw"], H, D, c["sink"], 0 if rolls else c["hist"], history_capacity=c["hist"], batch=B,
        dtype=msf.MSF_DTYPE_F32 if c["dtype"] == "f32" else msf.MSF_DTYPE_BF16,
        resample=msf.MSF_RESAMPLE_STRIDED if c["mode"] == "strided" else msf.MSF_RESAMPLE_AVG,
        latent_channels=CHANNELS, patch=PATCH, embed_dim=H * D, frames_per_state=c["frames"], fused_append=c["fused"]))
    plan.bind(plan.workspace(), x["k_sink"], x["v_sink"], x["k_hist"], x["v_hist"])
    st = {"case": c, "plan": plan, "x": x}
    if c["op"] != "tiers":
        st["out"] = [torch.empty_like(q) for q in x["q"]]
    if c["op"] == "train":
        st["lse"] = torch.empty((B, H, N), dtype=torch.float32, device="cuda")
        st["grads"] = [torch.empty_like(x["q"][0]) for _ in range(3)]
        st["bws"] = plan.backward_workspace()
    if _embeds(c):
        s = _scales(c)
        st["w"] = [x["w%d" % v] for v in s]
        st["tokens"] = [torch.empty((B, N, H * D), dtype=dt, device="cuda") for _ in range(c["steps"])]
        shape = (B, CHANNELS, c["frames"], c["gh"] * PATCH, c["gw"] * PATCH)
        st["emitted"] = [torch.empty(shape, dtype=dt, device="cuda") for _ in range(max(c["steps"], len(_emitted(c))))]
    if c["op"] == "tiers":
        mods = {}
        for v in set(s):
            if v == 1:
                mods[v] = msf.tier_module(x["w1"], x["o1"])
            else:
                mods[v] = msf.tier_module(x["w%d" % v], x["o%d" % v], x["ad%d" % v], x["au%d" % v], x["bd%d" % v],
                                          x["bu%d" % v], x["res%d" % v], lora_rank=c["rank"], lora_scale=0.5)
        st["tiers"] = [mods[v] for v in s]
    if rolls:
        st["empty"] = plan.history_state()
    return st


def _step(st, i, flags):
    """Embedding and pyramid, attention, de-embedding of the emitted head."""
    plan, x, c = st["plan"], st["x"], st["case"]
    q, k, v, out, tok = x["q"][i], x["k"][i], x["v"][i], st["out"][i], st["tokens"][i]
    if c["dtype"] == "f32":
        plan.patchify(x["latent"][i], st["w"], tok)
        plan.kv_resample(k, v, flags)
    else:
        plan.patchify_resample(x["latent"][i], st["w"], tok, k, v, flags)
    plan.mssa_forward(q, k, v, out)
    plan.unpatchify(0, out, x["o%d" % _scales(c)[0]], st["emitted"][i])


def run(state):
    st = state
    plan, x, c = st["plan"], st["x"], st["case"]
    op = c["op"]
    if op == "window":
        plan.kv_resample(x["k"][0], x["v"][0])
        plan.mssa_forward(x["q"][0], x["k"][0], x["v"][0], st["out"][0])
        return {"out": st["out"][0]}
    if op == "step":
        _step(st, 0, msf.MSF_RESAMPLE_FULL)
        return {"tokens": st["tokens"][0], "out": st["out"][0], "latent": st["emitted"][0]}
    if op == "rollout":
        plan.set_history_state(st["empty"])
        for i in range(c["steps"]):
            _step(st, i, msf.MSF_RESAMPLE_WINDOW_ONLY)
            if c["fused"]:
                plan.history_commit()
            else:
                plan.history_append(x["k"][i], x["v"][i])
        return {"out": st["out"], "latent": st["emitted"], "tokens": st["tokens"][-1],
                "ring": [x["k_hist"][:, :c["hist"]], x["v_hist"][:, :c["hist"]]]}
    if op == "train":
        q, k, v = x["q"][0], x["k"][0], x["v"][0]
        plan.kv_resample(k, v)
        plan.mssa_forward_lse(q, k, v, st["out"][0], st["lse"])
        plan.mssa_backward(q, k, v, st["out"][0], x["dout"], st["lse"], *st["grads"], st["bws"])
        return {"out": st["out"][0], "lse": st["lse"], "dq": st["grads"][0], "dk": st["grads"][1], "dv": st["grads"][2]}
    plan.patchify_tiers(x["latent"][0], st["tiers"], st["tokens"][0])
    for p in range(len(st["tiers"])):
        plan.unpatchify_tier(p, x["h"], x["latent"][0], st["tiers"][p], st["emitted"][p])
    return {"tokens": st["tokens"][0], "latent": st["emitted"]}


# ---------------------------------------------------------------- 64 bits

def _pool(c, x, gw, f):
    """x [B, rows * gw, H, D] pooled f x f (rows of all frames stacked: f divides one frame's)."""
    if f == 1:
        return x
    B, n, H, D = x.shape
    y = x.reshape(B, n // gw // f, f, gw // f, f, H, D)
    y = y[:, :, 0, :, 0] if c["mode"] == "strided" else y.mean(dim=(2, 4))
    return y.reshape(B, -1, H, D)


def _context(c, g, win, sink, frames):
    """Keys (or values) that a query of scale g attends to."""
    s = _scales(c)
    G, n, off = _sizes(c)
    parts = [sink] if c["sink"] else []
    parts += [_pool(c, f, c["gw"], g) for f in frames]
    for i, v in enumerate(s):
        parts.append(_pool(c, win[:, off[i]:off[i + 1]], c["gw"] // v, max(1, g // v)))
    return torch.cat(parts, 1)


def _attend(c, q, k, v, sink_k, sink_v, hk, hv, dout=None):
    """Eq. 4 in 64 bits, head by head; with dout its gradients too."""
    G, n, off = _sizes(c)
    out, lse = torch.zeros_like(q), torch.zeros(q.shape[0], q.shape[2], q.shape[1], dtype=q.dtype, device=q.device)
    grads = None
    if dout is not None:
        k, v = k.requires_grad_(), v.requires_grad_()
        dq = torch.zeros_like(q)
    scale = c["dim"] ** -0.5
    for g, a, z in _groups(c):
        ck = _context(c, g, k, sink_k, hk)
        cv = _context(c, g, v, sink_v, hv)
        dk, dv = (torch.zeros_like(ck), torch.zeros_like(cv)) if dout is not None else (None, None)
        with torch.no_grad():
            for b in range(q.shape[0]):
                for h in range(q.shape[2]):
                    K, V = ck[b, :, h].contiguous(), cv[b, :, h].contiguous()
                    for r in range(off[a], off[z], 2048):
                        t = slice(r, min(r + 2048, off[z]))
                        Q = q[b, t, h]
                        S = (Q @ K.T) * scale
                        L = torch.logsumexp(S, 1)
                        P = torch.exp_(S.sub_(L[:, None]))
                        lse[b, h, t] = L
                        out[b, t, h] = P @ V
                        if dout is not None:
                            dO = dout[b, t, h]
                            dv[b, :, h] += P.T @ dO
                            dS = P.mul_((dO @ V.T).sub_((dO * out[b, t, h]).sum(1)[:, None])).mul_(scale)
                            dq[b, t, h] = dS @ K
                            dk[b, :, h] += dS.T @ Q
        if dout is not None:
            torch.autograd.backward([ck, cv], [dk, dv])
    if dout is not None:
        grads = (dq, k.grad, v.grad)
    return out.detach(), lse, grads


def _patches(c, state, s):
    """A state [B, C, F, Hl, Wl] as patch vectors [B, tokens, C * P * P]."""
    B, P = state.shape[0], PATCH * s
    y = state.reshape(B, CHANNELS, c["frames"] * c["gh"] // s, P, c["gw"] // s, P)
    return y.permute(0, 2, 4, 1, 3, 5).reshape(B, -1, CHANNELS * P * P)


def _unpatch(c, rows, s):
    B, P = rows.shape[0], PATCH * s
    y = rows.reshape(B, c["frames"] * c["gh"] // s, c["gw"] // s, CHANNELS, P, P)
    return y.permute(0, 3, 1, 4, 2, 5).reshape(B, CHANNELS, c["frames"], c["gh"] * PATCH, c["gw"] * PATCH)


def exact(case, seed):
    c = case
    x = {k: [t.double() for t in v] if isinstance(v, list) else v.double() for k, v in _inputs(c, seed).items()}
    s = _scales(c)
    G, n, off = _sizes(c)

    def tokens(i):
        return torch.cat([_patches(c, x["latent"][i][:, l], v) @ x["w%d" % v].T for l, v in enumerate(s)], 1)

    if c["op"] in ("window", "step", "train"):
        hk = [x["k_hist"][:, f] for f in range(c["hist"])]
        hv = [x["v_hist"][:, f] for f in range(c["hist"])]
        out, lse, grads = _attend(c, x["q"][0], x["k"][0], x["v"][0], x["k_sink"], x["v_sink"], hk, hv, x.get("dout"))
        if c["op"] == "window":
            return {"out": out}
        if c["op"] == "train":
            return {"out": out, "lse": lse, "dq": grads[0], "dk": grads[1], "dv": grads[2]}
        return {"tokens": tokens(0), "out": out,
                "latent": _unpatch(c, out[:, :n[0]].flatten(2) @ x["o%d" % s[0]].T, s[0])}
    if c["op"] == "rollout":
        outs, latents, frames = [], [], []  # frames: (k, v) of the heads so far
        for i in range(c["steps"]):
            live = frames[-c["hist"]:]
            out, _, _ = _attend(c, x["q"][i], x["k"][i], x["v"][i], x["k_sink"], x["v_sink"], [f[0] for f in live],
                                [f[1] for f in live])
            outs.append(out)
            latents.append(_unpatch(c, out[:, :n[0]].flatten(2) @ x["o%d" % s[0]].T, s[0]))
            frames.append((x["k"][i][:, :G], x["v"][i][:, :G]))
        return {"out": outs, "latent": latents, "tokens": tokens(c["steps"] - 1), "ring": [None, None]}
    E = c["heads"] * c["dim"]
    toks, lats = [], []
    for l, v in enumerate(s):
        p = _patches(c, x["latent"][0][:, l], v)
        h = x["h"][:, off[l]:off[l + 1]]
        t, y = p @ x["w%d" % v].T, h @ x["o%d" % v].T
        if v > 1:
            t = t + 0.5 * (p @ x["ad%d" % v].T) @ x["au%d" % v].T
            y = y + 0.5 * (h @ x["bd%d" % v].T) @ x["bu%d" % v].T + p @ x["res%d" % v].T
        toks.append(t)
        lats.append(_unpatch(c, y, v))
    return {"tokens": torch.cat(toks, 1), "latent": lats}


def tolerance(case):
    # Four times the distance from exact() over the listed and ten drawn cases: bf16 up to 0.0029 (max 0.079 of the
    # rms, a gradient's few large elements), fp32 up to 2.3e-6 (max 4e-5: sums over up to 9000 keys).
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 2e-4}
    return {"rel": 1.2e-2, "max": 0.32}
