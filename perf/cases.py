"""The work that users of this library have it do, as cases to be timed: a step of one attention block, a step of a whole
compute block, a step of a stack of blocks as one CUDA graph, and a step on host buffers.

A case is a dict of plain values.  `kind` says which public entry point it goes through:

    step        astraea_step: score, select, sparse attention of the selected tokens, refresh of the reference inputs
    block       astraea_block_step: the same inside a whole block (projections, cross-attention, MLP on the selected rows)
    generation  ModelSchedule: one denoising step of L blocks that share one selection, captured as one CUDA graph
    host        Session.step_host: the first (dense) step of a generation whose tensors live in pinned host memory

Sizes: B batch elements, H heads of d channels, N_v selectable (video) tokens, N_t always-kept (text) tokens behind them,
theta the keep-ratio in permille; blocks also have `hidden` MLP channels and N_text text keys of the cross-attention.
Values follow the synthetic latents of the workloads: N(0, 1) tensors, an input that drifted by 0.05 since the reference,
LSE around ln N + 0.5, zero to three skipped steps; `lognormal` scales every token by LogNormal(0, lognormal).

A pass hands the step a copy of the previous step's LSE cache, so that the same selection is made whatever the rounding of
the attention before it; the other state (reference inputs, skip counters, output caches) is carried from pass to pass, and
the input alternates between two latents.
"""
import math

import torch

from paper_2506_05096_b200 import binding as A

W_ALPHA, W_BETA, EPS = 1.0, 1.0, 1e-6


def _case(name, kind, B, H, d, N_v, N_t, theta, **more):
    c = {"kind": kind, "B": B, "H": H, "d": d, "N_v": N_v, "N_t": N_t, "theta": theta, "lognormal": 0.0,
         "delta_mode": A.DELTA_MEAN_ABS, "lse_mode": A.LSE_SUM_EXP}
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # a toy latent of 4 x 8 x 8 tokens: the smallest call, where launches and latencies are the whole cost
        _case("step_tiny", "step", 1, 2, 64, 256, 0, 500),
        # a short low-resolution clip with a ragged token count and a few text tokens, one wide-headed block
        _case("step_short_clip_d128", "step", 1, 24, 128, 3517, 77, 300),
        # the CogVideoX shape (13 x 30 x 45 latent, 226 text tokens) at the two keep-ratios that a budget search hands out most
        _case("step_cogvideox_500", "step", 1, 48, 64, 17550, 226, 500),
        _case("step_cogvideox_250", "step", 1, 48, 64, 17550, 226, 250),
        # the Open-Sora shape: a batch of two (conditional and unconditional), 72-channel heads, skewed token norms
        _case("step_opensora_400", "step", 2, 16, 72, 16384, 0, 400, lognormal=0.5),
        # the lowest budget of the keep-ratio sweep: 65536 keys, a twentieth of the tokens as queries
        _case("step_sweep_050", "step", 1, 24, 128, 65536, 0, 50),
        # the HunyuanVideo shape (33 x 45 x 80 latent): the largest call
        _case("step_hunyuan_300", "step", 1, 24, 128, 118800, 0, 300),
        # whole compute blocks: the CogVideoX shape at half the budget, the Open-Sora shape at its own
        _case("block_cogvideox_500", "block", 1, 48, 64, 17550, 226, 500, hidden=12288, N_text=226, select_qk=False),
        _case("block_opensora_400", "block", 2, 16, 72, 16384, 0, 400, lognormal=0.5, hidden=4608, N_text=226, select_qk=False),
        # the variant that also drops the keys and values of the unselected tokens
        _case("block_cogvideox_250_qk", "block", 1, 48, 64, 17550, 226, 250, hidden=12288, N_text=226, select_qk=True),
        # one denoising step of a small model, four blocks behind one selection, replayed as a CUDA graph
        _case("generation_small", "generation", 1, 24, 64, 4050, 226, 400, hidden=6144, N_text=226, L=4),
        # host buffers in and out: the dense first step of a session on one half of the Open-Sora batch
        _case("host_opensora_dense", "host", 1, 16, 72, 16384, 0, 1000),
    ]


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n | 1 if rng.random() < 0.5 else n

    kind = rng.choice(["step"] * 6 + ["block"] * 3 + ["generation", "host"])
    d = rng.choice([64, 72, 128])
    B = rng.choice([1, 1, 2])
    theta = rng.choice([1000, size(50, 999), size(50, 999), size(50, 999)])
    n_t = rng.choice([0, 0, 77, 226, size(8, 300)])
    more = {"lognormal": rng.choice([0.0, 0.0, 0.5]),
            "delta_mode": rng.choice([A.DELTA_MEAN_ABS, A.DELTA_MEAN_ABS, A.DELTA_MEAN_SQ]),
            "lse_mode": rng.choice([A.LSE_SUM_EXP, A.LSE_SUM_EXP, A.LSE_LOG])}
    if kind == "step":
        return _case("", kind, B, rng.choice({64: [2, 12, 24, 48], 72: [4, 9, 16], 128: [3, 12, 24]}[d]), d, size(200, 60000 // B), n_t, theta, **more)
    if kind == "host":
        return _case("", kind, B, rng.choice([2, 8, 16]), d, size(200, 16000), n_t, 1000, **more)
    H = rng.choice({64: [12, 24, 48], 72: [8, 16], 128: [12, 24]}[d])
    hidden = 64 * rng.randint(H * d // 32, H * d // 16)
    if kind == "generation":
        return _case("", kind, B, H, d, size(300, 6000 // B), n_t, theta, hidden=hidden, N_text=size(20, 300), L=rng.randint(2, 4), **more)
    return _case("", kind, B, H, d, size(300, 18000 // B), n_t, theta, hidden=hidden, N_text=size(20, 300), select_qk=rng.random() < 0.25, **more)


def _sizes(c):
    N, k = c["N_v"] + c["N_t"], A.astraea_budget_to_k(c["N_v"], c["theta"])
    return N, k, k + c["N_t"], c["H"] * c["d"]


# ------------------------------------------------------------------ inputs
def _latents(c, g):
    """What every kind starts from: reference input, two drifted inputs, LSE cache, skip counters, a draw function."""
    B, H, N_v = c["B"], c["H"], c["N_v"]
    N, _, _, D = _sizes(c)
    norms = torch.exp(c["lognormal"] * torch.randn(B, N, 1, device="cuda", generator=g)) if c["lognormal"] else None

    def draw(scaled=True):
        t = torch.randn(B, N, D, device="cuda", dtype=torch.bfloat16, generator=g)
        return t.mul_(norms) if scaled and norms is not None else t

    x_ref = draw()
    x = [x_ref + 0.05 * draw(), x_ref + 0.05 * draw()]
    lse = torch.randn(B, H, N, device="cuda", generator=g).mul_(0.25).add_(math.log(N) + 0.5)
    n_skip = torch.randint(0, 4, (B, N_v), device="cuda", dtype=torch.int32, generator=g)
    return {"x_ref": x_ref, "x": x, "lse_prev": lse, "n_skip": n_skip}, draw


def _weights(c, g):
    D, hid, B = c["H"] * c["d"], c["hidden"], c["B"]

    def mat(rows, cols):
        return torch.randn(rows, cols, device="cuda", dtype=torch.bfloat16, generator=g).mul_(1.0 / math.sqrt(cols))

    def vec(*shape):
        return torch.randn(*shape, device="cuda", dtype=torch.bfloat16, generator=g).mul_(0.1)

    w = {n: mat(D, D) for n in ("wq", "wk", "wv", "wo", "wq2", "wo2")}
    w.update(w1=mat(hid, D), w2=mat(D, hid), b1=vec(hid))
    w.update({n: vec(D) for n in ("bq", "bk", "bv", "bo", "bq2", "bo2", "b2")})
    w.update({n: vec(B, D) for n in ("s1", "t1", "s3", "t3")})
    w.update({n: vec(B, D).add_(0.5) for n in ("g1", "g3")})
    text = [torch.randn(B, c["N_text"], D, device="cuda", dtype=torch.bfloat16, generator=g) for _ in range(2)]
    return w, text


def _inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s, draw = _latents(c, g)
    if c["kind"] in ("step", "host"):
        s["q"], s["k"], s["v"] = draw(), draw(), draw()
        s["out"] = draw(False)
    else:
        L = c.get("L", 1)
        s["blocks"] = [_weights(c, g) + (draw(False),) for _ in range(L)]
    return s


def _selection_buffers(c):
    B, N_v = c["B"], c["N_v"]
    _, k, M, _ = _sizes(c)
    return {"score": torch.zeros(B, N_v, device="cuda"),
            "idx_sel": torch.zeros(B, M, dtype=torch.int32, device="cuda"),
            "idx_rem": torch.zeros(B, N_v - k, dtype=torch.int32, device="cuda")}


def prepare(case, seed):
    c = case
    B, H, d, N_v = c["B"], c["H"], c["d"], c["N_v"]
    N, k, M, D = _sizes(c)
    s = _inputs(c, seed)
    s.update(case=c, turn=0)
    if c["kind"] == "host":
        for n in ("q", "k", "v", "out"):
            s[n] = s[n].cpu().pin_memory()
        s["x"] = [t.cpu().pin_memory() for t in s["x"]]
        s["session"] = A.Session(B, H, N, N_v, d)
        return s
    s["lse"] = s["lse_prev"].clone()
    s.update(_selection_buffers(c))
    if c["kind"] == "step":
        s["ws"] = A.new_workspace(A.OP_STEP, B, H, N, M, d)
        return s
    hid = c["hidden"]
    s["ws"] = torch.zeros(A.astraea_block_workspace_bytes(B, H, N, d, hid), dtype=torch.uint8, device="cuda")
    if c["kind"] == "block":
        w, (s["text_k"], s["text_v"]), s["y"] = s["blocks"][0]
        s["weights"] = A.block_weights(w, hid)
        return s
    states = []
    for i, (_, _, y) in enumerate(s["blocks"]):
        st = _selection_buffers(c) if i else {n: s[n] for n in ("score", "idx_sel", "idx_rem")}
        # only the first block selects, the others' selection state is never read
        st.update(x_ref=s["x_ref"], lse_cache=s["lse"] if i == 0 else s["lse_prev"].clone(), n_skip=s["n_skip"], y_cache=y)
        states.append(st)
    s["states"] = states
    s["graphs"] = [A.ModelSchedule([k], [x], [(w, hid) for w, _, _ in s["blocks"]], states, [t[0] for _, t, _ in s["blocks"]],
                                   [t[1] for _, t, _ in s["blocks"]], c["N_text"], B, H, N, N_v, d, W_ALPHA, W_BETA, c["delta_mode"],
                                   c["lse_mode"], EPS, A.VARIANT_FIXED_TOKEN, s["ws"]) for x in s["x"]]
    return s


def run(state):
    s, c = state, state["case"]
    B, H, d, N_v = c["B"], c["H"], c["d"], c["N_v"]
    N, k, _, _ = _sizes(c)
    turn = s["turn"]
    s["turn"] = turn ^ 1
    x = s["x"][turn]
    if c["kind"] == "host":
        s["session"].step_host(x, s["q"], s["k"], s["v"], s["out"], k, W_ALPHA, W_BETA, c["delta_mode"], c["lse_mode"])
        return {"out": s["out"]}
    s["lse"].copy_(s["lse_prev"])
    outs = {n: s[n] for n in ("score", "idx_sel", "idx_rem", "n_skip", "x_ref", "lse")}
    if c["kind"] == "step":
        A.astraea_step(x, s["x_ref"], s["lse"], s["n_skip"], s["q"], s["k"], s["v"], s["out"], s["score"], s["idx_sel"], s["idx_rem"],
                       B, H, N, N_v, d, k, W_ALPHA, W_BETA, c["delta_mode"], c["lse_mode"], s["ws"])
        outs["out"] = s["out"]
    elif c["kind"] == "block":
        A.astraea_block_step(x, s["weights"], s["x_ref"], s["lse"], s["n_skip"], s["y"], s["text_k"], s["text_v"], c["N_text"],
                             s["score"], s["idx_sel"], s["idx_rem"], B, H, N, N_v, d, k, W_ALPHA, W_BETA, c["delta_mode"], c["lse_mode"],
                             EPS, A.BLOCK_SELECT_QK if c["select_qk"] else 0, s["ws"])
        outs["y"] = s["y"]
    else:
        s["graphs"][turn].launch()
        outs["y"] = [st["y_cache"] for st in s["states"]]
        outs["lse_blocks"] = [st["lse_cache"] for st in s["states"][1:]]
    return outs


# ------------------------------------------------------------------ work
def work(case):
    c = case
    B, H, d, N_v = c["B"], c["H"], c["d"], c["N_v"]
    N, k, M, D = _sizes(c)
    row = 2 * D
    if c["kind"] == "host":      # four tensors in, one out
        return {"bytes": 5 * B * N * row, "flops": 4 * B * H * M * N * d}
    # the score reads two rows and H LSE values a token, the selection writes its lists and counters; the refresh writes M rows
    select = B * (N_v * (2 * row + 4 * H) + 4 * N_v + 8 * N_v + 4 * (M + N_v - k)) + B * M * row
    if c["kind"] == "step":
        return {"bytes": select + B * (2 * M + 2 * N) * row + 4 * B * H * M, "flops": 4 * B * H * M * N * d}
    hid, L = c["hidden"], c.get("L", 1)
    keys = M if c.get("select_qk") else N
    weights = 2 * (6 * D * D + 2 * D * hid)
    flops = 2 * B * (2 * keys * D * D + 4 * M * D * D + 2 * M * D * hid) + 4 * B * H * M * d * (keys + c["N_text"])
    return {"bytes": select + L * (weights + B * (keys + M + 2 * c["N_text"]) * row + 4 * B * H * M), "flops": L * flops}


def tolerance(case):
    # bf16 results of fp32 sums, LSE values that carry the bf16 rounding of the probabilities; whole values are the same
    return {"rel": 1e-2, "max": 0.2, "differ": 0.0}


# ------------------------------------------------------------------ 64 bits
def _select64(c, x, s):
    B, H, N_v = c["B"], c["H"], c["N_v"]
    N, k, M, D = _sizes(c)
    delta = torch.empty(B, N_v, device="cuda", dtype=torch.float64)
    for b in range(B):
        for i in range(0, N_v, 8192):
            e = slice(i, min(i + 8192, N_v))
            diff = x[b, e].double() - s["x_ref"][b, e].double()
            delta[b, e] = {A.DELTA_MEAN_ABS: diff.abs, A.DELTA_MEAN_SQ: diff.square}.get(c["delta_mode"], diff.clone)().mean(1)
    lse = s["lse_prev"][:, :, :N_v].double()
    s_lse = (lse.clamp(max=80.0).exp() if c["lse_mode"] == A.LSE_SUM_EXP else lse).mean(1)
    score = W_ALPHA * s_lse * delta + W_BETA * s["n_skip"].double().exp()
    order = torch.sort(score, dim=1, descending=True, stable=True).indices[:, :k]
    always = torch.arange(N_v, N, device="cuda").expand(B, N - N_v)
    return score, torch.cat([order.sort(1).values, always], 1)


def _attention64(q, k, v, H, d):
    """q [M, H*d], k, v [N, H*d] -> rows [M, H*d] and LSE [H, M], in 64 bits."""
    M, N = q.shape[0], k.shape[0]
    out, lse = torch.empty(M, H * d, device="cuda", dtype=torch.float64), torch.empty(H, M, device="cuda", dtype=torch.float64)
    rows = max(1, min(M, (1 << 28) // N))
    for h in range(H):
        e = slice(h * d, (h + 1) * d)
        kk, vv = k[:, e].double(), v[:, e].double()
        for i in range(0, M, rows):
            z = (q[i:i + rows, e].double() @ kk.T).mul_(1.0 / math.sqrt(d))
            l = z.logsumexp(1)
            lse[h, i:i + rows] = l
            out[i:i + rows, e] = z.sub_(l[:, None]).exp_() @ vv
    return out, lse


def _norm64(x, scale=None, shift=None):
    y = (x - x.mean(1, keepdim=True)) * torch.rsqrt(x.var(1, unbiased=False, keepdim=True) + EPS)
    return y if scale is None else y * (1.0 + scale) + shift


def _block64(c, x, w, text, rows, b):
    """The listed rows of one block's output and their LSE, for batch element b; x [N, D] in 64 bits."""
    H, d = c["H"], c["d"]
    p = {n: t[b].double() if n in ("s1", "t1", "g1", "s3", "t3", "g3") else t.double() for n, t in w.items()}
    lin = lambda a, n: a @ p["w" + n].T + p["b" + n]  # noqa: E731
    h = _norm64(x, p["s1"], p["t1"])
    keys = h[rows] if c.get("select_qk") else h
    att, lse = _attention64(lin(h[rows], "q"), lin(keys, "k"), lin(keys, "v"), H, d)
    x1 = x[rows] + p["g1"] * lin(att, "o")
    cross, _ = _attention64(lin(_norm64(x1), "q2"), text[0][b], text[1][b], H, d)
    x2 = x1 + lin(cross, "o2")
    u = torch.nn.functional.gelu(lin(_norm64(x2, p["s3"], p["t3"]), "1"))
    return x2 + p["g3"] * lin(u, "2"), lse


def exact(case, seed):
    c = case
    if work(c)["flops"] > 6e13:
        return None
    B, H, d = c["B"], c["H"], c["d"]
    s = _inputs(c, seed)
    x = s["x"][0]
    score, rows = _select64(c, x, s)
    lse, x_ref = s["lse_prev"].double(), s["x_ref"].clone()
    for b in range(B):
        x_ref[b, rows[b]] = x[b, rows[b]]
    outs = {"score": score, "idx_sel": None, "idx_rem": None, "n_skip": None, "x_ref": x_ref.double(), "lse": lse}
    if c["kind"] in ("step", "host"):
        out = s["out"].double()
        for b in range(B):
            r = rows[b]
            out[b, r], l = _attention64(s["q"][b, r], s["k"][b], s["v"][b], H, d)
            lse[b][:, r] = l
        if c["kind"] == "host":
            return {"out": out.cpu()}
        outs["out"] = out
        return outs
    ys, lses = [], []
    h = x.double()
    for i, (w, text, y) in enumerate(s["blocks"]):
        y, l = y.double(), lse if i == 0 else s["lse_prev"].double()
        for b in range(B):
            y[b, rows[b]], l[b][:, rows[b]] = _block64(c, h[b], w, text, rows[b], b)
        ys.append(y)
        lses.append(l)
        h = y
    if c["kind"] == "block":
        outs["y"] = ys[0]
    else:
        outs["y"], outs["lse_blocks"] = ys, lses[1:]
    return outs
