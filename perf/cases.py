"""The calls whose speed matters: the block step of an interactive world model and its parts.

Every case is one call (or one site of a transformer block) as a serving loop makes it, through
paper_2609_34144_gb300.native, on seeded synthetic inputs made on the GPU.  Shapes are those of
the two backbones of synthetic/workloads.py (Matrix-Game-shaped: 8 frames of 30x52 tokens, 12
heads of 128; HY-World-shaped: 16 frames of 44x80 tokens, 24 heads of 128), of the PAR sweep and
of the smallest configuration, plus one ragged size with heads of 64.

A case is a dict of plain values; "kind" names the call:
  attention  routed anchor attention            route   pooling, omission scores, TopK, refinement
  par        Phase-Aware Reconstruction         ffn     the anchor FFN site with its PAR
  select     control-aware frame selection      block   routing -> attention -> (W_O) -> PAR
"""
import math

import torch

from paper_2609_34144_gb300 import native as cast

DEV = "cuda"


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest configuration (4 frames of 8x8, f32 residuals, band 2): what a call costs
        # when there is next to nothing to compute
        dict(name="block_tiny_f32", kind="block", frames=4, Hg=8, Wg=8, H=2, d=64, anchors="0,3",
             hist="blocks", hist_n=4, K=2, refine=True, gram=False, w_o=False, out="f32", band=2.0),
        # a small latent with odd sides and heads of 64: low-resolution preview, short history
        dict(name="attention_ragged_d64", kind="attention", frames=5, Hg=13, Wg=27, H=8, d=64,
             anchors="0,2,4", hist="blocks", hist_n=6, K=2, out="bf16", lse=True),
        # Matrix-Game-shaped chunk against 4 of 16 frame-sized history blocks
        dict(name="attention_mg", kind="attention", frames=8, Hg=30, Wg=52, H=12, d=128,
             anchors="0,2,4,6", hist="blocks", hist_n=16, K=4, out="bf16", lse=False),
        # the same chunk at the paper's KV granularity: 90 of 448 (1,8,8) blocks
        dict(name="attention_mg64", kind="attention", frames=8, Hg=30, Wg=52, H=12, d=128,
             anchors="0,2,4,6", hist="frames", hist_n=16, K=90, out="bf16", lse=False),
        # HY-World-shaped routing with the paper's two refinement passes
        dict(name="route_hy", kind="route", frames=16, Hg=44, Wg=80, H=24, d=128,
             anchors="0,3,7,12,15", hist="blocks", hist_n=32, K=8, refine=True, gram=False),
        # Matrix-Game-shaped routing over (1,8,8) blocks
        dict(name="route_mg64", kind="route", frames=8, Hg=30, Wg=52, H=12, d=128,
             anchors="0,2,4,6", hist="frames", hist_n=16, K=90, refine=True, gram=False),
        # reconstruction of 11 skipped frames, bf16 residuals (a serving step)
        dict(name="par_hy_bf16", kind="par", frames=16, Hg=44, Wg=80, C=3072, anchors="0,3,7,12,15",
             dtype="bf16", weights=False, band=-1.0),
        # reconstruction with f32 residuals, channel weights and a band cut (the PAR sweep)
        dict(name="par_sweep_f32", kind="par", frames=16, Hg=44, Wg=80, C=3072,
             anchors="0,3,6,9,12,15", dtype="f32", weights=True, band=4.0),
        # the FFN site of a Matrix-Game-shaped block
        dict(name="ffn_mg", kind="ffn", frames=8, Hg=30, Wg=52, D=1536, D_ff=6144,
             anchors="0,2,4,6", bias=True, out="bf16"),
        # anchors of the next block from two control branches
        dict(name="select_mg", kind="select", frames=8, elems=30 * 52 * 1536, branches=2,
             dtype="bf16", K_f=4),
        # a whole attention site: routing with the Gram matrices of W_O, attention, the output
        # projection, PAR of the projected residual and the residual update
        dict(name="block_mg_projected", kind="block", frames=8, Hg=30, Wg=52, H=12, d=128,
             anchors="0,2,4,6", hist="blocks", hist_n=16, K=4, refine=True, gram=True, w_o=True,
             out="bf16", band=-1.0),
        # the largest block step
        dict(name="block_hy", kind="block", frames=16, Hg=44, Wg=80, H=24, d=128,
             anchors="0,3,7,12,15", hist="blocks", hist_n=32, K=8, refine=True, gram=False,
             w_o=False, out="bf16", band=-1.0),
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))
    return max(lo, min(hi, int(v // step * step)))


def _spaced(rng, frames, most):
    """Anchors every 1..4 frames from the first (at least two, at most `most`)."""
    sp = rng.randint(1, 4)
    got = list(range(0, frames, sp))[:most]
    if len(got) < 2:
        got = [0, frames - 1]
    return got


def _draw(rng):
    kind = rng.choice(["attention", "route", "par", "ffn", "select", "block"])
    frames = rng.randint(2, 16)
    Hg, Wg = _log_int(rng, 6, 44), _log_int(rng, 8, 80)
    c = dict(kind=kind, frames=frames)
    if kind == "select":
        c.update(frames=rng.randint(2, 32), elems=8 * _log_int(rng, 2000, 1500000),
                 branches=rng.randint(1, 2), dtype=rng.choice(["bf16", "bf16", "f32"]))
        c["K_f"] = rng.randint(1, c["frames"])
        return c
    c.update(Hg=Hg, Wg=Wg)
    if kind in ("par", "ffn"):
        if frames < 3:
            c["frames"] = frames = 3
        anchors = _spaced(rng, frames, 8)
        if len(anchors) == frames:
            anchors = list(range(0, frames, 2))
        c["anchors"] = ",".join(map(str, anchors))
        if kind == "par":
            c.update(C=_log_int(rng, 64, 3072, 8), dtype=rng.choice(["bf16", "bf16", "f32"]),
                     weights=rng.random() < 0.3, band=rng.choice([-1.0, -1.0, 2.0, 4.0]))
        else:
            D = _log_int(rng, 128, 3072, 8)
            c.update(D=D, D_ff=min(12288, 8 * int(D * rng.uniform(2.5, 4.0) / 8)),
                     bias=rng.random() < 0.7, out="bf16")
        return c
    hist = rng.choice(["blocks", "blocks", "frames"])
    hist_n = _log_int(rng, 4, 32)
    M = hist_n if hist == "blocks" else hist_n * (-(-Hg // 8)) * (-(-Wg // 8))
    anchors = _spaced(rng, frames, max(2, min(8, 9600 // M)))
    c.update(H=rng.randint(2, 24), d=rng.choice([64, 128, 128]), anchors=",".join(map(str, anchors)),
             hist=hist, hist_n=hist_n, K=max(1, math.ceil(M * rng.uniform(0.15, 0.4))))
    if kind == "attention":
        c.update(out="bf16", lse=rng.random() < 0.3)
    else:
        c.update(refine=rng.random() < 0.8, gram=M <= 64 and rng.random() < 0.3)
    if kind == "block":
        # f32 residuals belong to the smallest configuration
        small = frames * Hg * Wg <= 1024
        c.update(w_o=rng.random() < 0.3, out="f32" if small and rng.random() < 0.5 else "bf16",
                 band=rng.choice([-1.0, 2.0]))
    return c


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def draw(rng):
    top = _cost(listed()[-1])
    while True:
        c = _draw(rng)
        if _cost(c) <= top:
            return c


# --------------------------------------------------------------------------- inputs
def _anchors(c):
    return [int(t) for t in c["anchors"].split(",")]


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _tokens(g, groups, rows, H, d):
    """bf16 [groups, rows, H, d]: N(0,1) tokens plus one N(0,1) d-vector per (group, head)."""
    out = torch.empty((groups, rows, H, d), dtype=torch.bfloat16, device=DEV)
    for i in range(groups):
        off = torch.randn((1, H, d), generator=g, device=DEV)
        out[i] = torch.randn((rows, H, d), generator=g, device=DEV) + off
    return out


def _history_frames(g, n, Hg, Wg, H, d):
    """bf16 [n, Hg, Wg, H, d]: N(0,1) tokens plus one N(0,1) d-vector per (frame, 8x8 patch, head)."""
    out = torch.empty((n, Hg, Wg, H, d), dtype=torch.bfloat16, device=DEV)
    for i in range(n):
        off = torch.randn((-(-Hg // 8), -(-Wg // 8), H, d), generator=g, device=DEV)
        off = off.repeat_interleave(8, 0).repeat_interleave(8, 1)[:Hg, :Wg]
        out[i] = torch.randn((Hg, Wg, H, d), generator=g, device=DEV) + off
    return out


def _blur(n, ell=4.0):
    """Circulant matrix of a Gaussian of standard deviation ell / sqrt(2) over n tokens."""
    i = torch.arange(n, device=DEV, dtype=torch.float32)
    dist = (i[:, None] - i[None, :]).abs()
    dist = torch.minimum(dist, n - dist)
    m = torch.exp(-dist * dist / (ell * ell))
    return m / m.sum(1, keepdim=True)


def _fields(g, frames, Hg, Wg, C, dtype):
    """[frames, Hg, Wg, C]: one smooth random field per channel (correlation length 4 tokens)
    under a camera that moves 0-3 tokens a frame, the amplitude growing by 1 % a frame."""
    steps = torch.randint(0, 4, (frames, 2), generator=g, device=DEV).tolist()
    ch, cw = Hg + 3 * frames, Wg + 3 * frames
    white = torch.randn((ch, cw, C), generator=g, device=DEV)
    canvas = (_blur(ch) @ white.reshape(ch, -1)).reshape(ch, cw, C)
    del white
    canvas = torch.matmul(_blur(cw), canvas)
    canvas /= canvas.std()
    out = torch.empty((frames, Hg, Wg, C), dtype=dtype, device=DEV)
    y = x = 0
    for t in range(frames):
        if t:
            y, x = y + steps[t][0], x + steps[t][1]
        out[t] = canvas[y:y + Hg, x:x + Wg] * (1.01 ** t)
    return out


def _dtype(text):
    return torch.bfloat16 if text == "bf16" else torch.float32


def _sequence_inputs(c, g):
    """Queries, current keys and values and the history of one attention site."""
    N, S, H, d = c["frames"], c["Hg"] * c["Wg"], c["H"], c["d"]
    s = dict(anchors=_anchors(c))
    s["q"] = _tokens(g, N, S, H, d)
    if c["kind"] != "route":
        s["k"], s["v"] = _tokens(g, N, S, H, d), _tokens(g, N, S, H, d)
    if c["hist"] == "frames":
        s["kh"], s["vh"] = (_history_frames(g, c["hist_n"], c["Hg"], c["Wg"], H, d) for _ in range(2))
    else:
        s["kh"], s["vh"] = (_tokens(g, c["hist_n"], S, H, d) for _ in range(2))
    return s


def _n_blocks(c):
    return c["hist_n"] * ((-(-c["Hg"] // 8)) * (-(-c["Wg"] // 8)) if c["hist"] == "frames" else 1)


def _weight(g, rows, cols):
    return (torch.randn((rows, cols), generator=g, device=DEV) / math.sqrt(cols)).to(torch.bfloat16)


def _gram(w_o, H, d):
    """G_h = P_h^T P_h of the head slices P_h = W_O[:, h d : (h + 1) d]."""
    p = w_o.float().reshape(-1, H, d)
    return torch.einsum("ohi,ohj->hij", p, p).contiguous()


def _workspace(nbytes):
    return torch.empty(max(int(nbytes), 256), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    c, g = case, _gen(seed)
    kind = c["kind"]
    if kind == "select":
        N = c["frames"]
        dl = []
        for _ in range(c["branches"]):
            amp = 0.2 + 1.8 * torch.rand((N, 1), generator=g, device=DEV)
            x = torch.empty((N, c["elems"]), dtype=_dtype(c["dtype"]), device=DEV)
            for i in range(N):
                x[i] = torch.randn((c["elems"],), generator=g, device=DEV) * amp[i]
            dl.append(x)
        ages = torch.randint(0, 4, (N,), generator=g, device=DEV, dtype=torch.int32)
        mask = torch.zeros(N, dtype=torch.uint8, device=DEV)
        mask[torch.randperm(N, generator=g, device=DEV)[:c["K_f"]]] = 1
        ws = _workspace(cast.select_workspace_size(dl, ages, mask, c["K_f"]))
        return dict(kind=kind, deltas=dl, ages=ages, mask=mask, K_f=c["K_f"], ws=ws)
    if kind == "par":
        r = _fields(g, c["frames"], c["Hg"], c["Wg"], c["C"], _dtype(c["dtype"]))
        a = _anchors(c)
        mask = [1 if t in a else 0 for t in range(c["frames"])]
        for t in range(c["frames"]):
            if not mask[t]:
                r[t] = 0
        wc = torch.rand((c["C"],), generator=g, device=DEV) if c["weights"] else None
        p = cast.par_params(band_radius=c["band"])
        return dict(kind=kind, r=r, mask=mask, wc=wc, params=p,
                    ws=_workspace(cast.par_workspace_size(r, mask, p)))
    if kind == "ffn":
        S, D, Df = c["Hg"] * c["Wg"], c["D"], c["D_ff"]
        x = _fields(g, c["frames"], c["Hg"], c["Wg"], D, torch.bfloat16).reshape(c["frames"], S, D)
        w1, w2 = _weight(g, Df, D), _weight(g, D, Df)
        b1 = b2 = None
        if c["bias"]:
            b1 = (0.1 * torch.randn((Df,), generator=g, device=DEV)).to(torch.bfloat16)
            b2 = (0.1 * torch.randn((D,), generator=g, device=DEV)).to(_dtype(c["out"]))
        r = torch.zeros((c["frames"], S, D), dtype=_dtype(c["out"]), device=DEV)
        a = _anchors(c)
        grid = (c["Hg"], c["Wg"])
        ws = _workspace(cast.ffn_workspace_size(x, a, w1, b1, w2, b2, grid, r))
        return dict(kind=kind, x=x, anchors=a, w1=w1, b1=b1, w2=w2, b2=b2, grid=grid, r=r, ws=ws)
    s = _sequence_inputs(c, g)
    s.update(kind=kind, K=min(c["K"], _n_blocks(c)))
    N, S, H, d = s["q"].shape
    if kind == "attention":
        M = _n_blocks(c)
        pick = torch.rand((len(s["anchors"]), H, M), generator=g, device=DEV).argsort(-1)[..., :s["K"]]
        s["idx"] = pick.sort(-1).values.to(torch.int32).contiguous()
        s["o"] = torch.empty((len(s["anchors"]), S, H * d), dtype=_dtype(c["out"]), device=DEV)
        s["lse"] = c["lse"]
        s["ws"] = _workspace(cast.attention_workspace_size(s["q"], s["k"], s["v"], s["anchors"], s["kh"],
                                                           s["vh"], s["idx"]))
        return s
    w_o = _weight(g, H * d, H * d) if c["gram"] or c.get("w_o") else None
    s["gram"] = _gram(w_o, H, d) if c["gram"] else None
    s["refine"] = cast.REFINE_PAPER if c["refine"] else None
    if kind == "route":
        s["ws"] = _workspace(cast.route_workspace_size(s["q"], s["anchors"], s["kh"], s["vh"], s["K"],
                                                       refine=s["refine"]))
        return s
    dt = _dtype(c["out"])
    s["grid"] = (c["Hg"], c["Wg"])
    s["r"] = torch.zeros((N, S, H * d), dtype=dt, device=DEV)
    s["idx"] = torch.zeros((len(s["anchors"]), H, s["K"]), dtype=torch.int32, device=DEV)
    more = dict(gram=s["gram"], refine=s["refine"], params=cast.par_params(band_radius=c["band"]))
    if c["w_o"]:
        # the hidden state the site updates, and its projection
        s["x"] = _tokens(g, N, S, H, d).reshape(N, S, H * d).to(dt)
        more.update(w_o=w_o, b_o=(0.1 * torch.randn((H * d,), generator=g, device=DEV)).to(dt))
    else:
        s["x"] = None
    s["more"] = more
    args = cast.block_args(s["q"], s["k"], s["v"], s["anchors"], s["kh"], s["vh"], s["K"], s["grid"], s["r"],
                           s["x"], s["idx"], **more)
    s["ws"] = _workspace(cast.block_workspace_size(args))
    return s


# --------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "block":
        cast.cast_block_step(s["q"], s["k"], s["v"], s["anchors"], s["kh"], s["vh"], s["K"], s["grid"], s["r"],
                             x=s["x"], idx_out=s["idx"], workspace=s["ws"], **s["more"])
        out = {"r": s["r"], "idx": s["idx"]}
        if s["x"] is not None:
            out["x"] = s["x"]
        return out
    if kind == "attention":
        got = cast.cast_anchor_attention(s["q"], s["k"], s["v"], s["anchors"], s["kh"], s["vh"], s["idx"],
                                         want_lse=s["lse"], out=s["o"], workspace=s["ws"])
        return {"o": got[0], "lse": got[1]} if s["lse"] else {"o": got}
    if kind == "route":
        idx, u, (qb, kb, vb) = cast.cast_route_topk(
            s["q"], s["anchors"], s["kh"], s["vh"], s["K"], gram=s["gram"], want_u=True, want_pooled=True,
            workspace=s["ws"], refine=s["refine"])
        return {"idx": idx, "u": u, "qbar": qb, "kbar": kb, "vbar": vb}
    if kind == "par":
        return {"r": cast.cast_par_reconstruct(s["r"], s["mask"], channel_weight=s["wc"], params=s["params"],
                                               workspace=s["ws"])}
    if kind == "ffn":
        return {"r": cast.cast_ffn_step(s["x"], s["anchors"], s["w1"], s["b1"], s["w2"], s["b2"], s["grid"],
                                        s["r"], workspace=s["ws"])}
    anchors, ages, mask, rms, score = cast.cast_select_frames(
        s["deltas"], s["ages"], s["mask"], s["K_f"], want_rms=True, want_score=True, workspace=s["ws"])
    return {"anchors": anchors, "ages": ages, "mask": mask, "rms": rms, "score": score}


# --------------------------------------------------------------------------- what a pass needs
def _key_tokens(c):
    """History tokens one (anchor, head) attends to (the mean block size for (1,8,8) blocks)."""
    S = c["Hg"] * c["Wg"]
    return c["K"] * (S if c["hist"] == "blocks" else c["hist_n"] * S / _n_blocks(c))


def work(case):
    c = case
    kind = c["kind"]
    if kind == "select":
        n = c["branches"] * c["frames"] * c["elems"]
        return {"bytes": n * (2 if c["dtype"] == "bf16" else 4), "flops": 2 * n}
    S, N, a = c["Hg"] * c["Wg"], c["frames"], len(_anchors(c))
    if kind == "par":
        # per element: two tile transforms' share and the blend, about 30 operations
        return {"bytes": N * S * c["C"] * (2 if c["dtype"] == "bf16" else 4), "flops": 30 * N * S * c["C"]}
    if kind == "ffn":
        return {"bytes": a * S * c["D"] * 2 + 4 * c["D"] * c["D_ff"] + N * S * c["D"] * 2,
                "flops": 4 * a * S * c["D"] * c["D_ff"]}
    H, d = c["H"], c["d"]
    D, hist = H * d, c["hist_n"] * S
    if kind == "route":
        return {"bytes": (a * S + 2 * hist) * D * 2, "flops": (a * S + 2 * hist) * D + 6 * a * _n_blocks(c) * D}
    elt = 2 if c["out"] == "bf16" else 4
    flops = 4 * a * S * (N * S + _key_tokens(c)) * D
    if kind == "attention":
        # queries, current keys and values, every routed block once (at most the whole history), O
        routed = min(hist, a * _key_tokens(c))
        return {"bytes": (a * S + 2 * N * S + 2 * routed) * D * 2 + a * S * D * elt, "flops": flops}
    nbytes = (a * S + 2 * N * S + 2 * hist) * D * 2 + N * S * D * elt
    if c["w_o"]:
        flops += 2 * a * S * D * D
        nbytes += 2 * D * D + 2 * N * S * D * elt
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------- 64-bit values
_MOST_FLOPS = 8e11   # of the attention or GEMMs: what 64 bits do within some seconds


def _block_tokens(c, x):
    """The history as a list of M [tokens, H, d] blocks."""
    if c["hist"] == "blocks":
        return list(x)
    out = []
    for f in x:
        for y in range(0, c["Hg"], 8):
            for z in range(0, c["Wg"], 8):
                b = f[y:y + 8, z:z + 8]
                out.append(b.reshape(-1, *b.shape[2:]))
    return out


def _pooled64(c, s):
    """The mean queries [anchors, H, d], keys and values [M, H, d]."""
    qb = torch.stack([s["q"][i].double().mean(0) for i in s["anchors"]])
    kb = torch.stack([b.double().mean(0) for b in _block_tokens(c, s["kh"])])
    vb = torch.stack([b.double().mean(0) for b in _block_tokens(c, s["vh"])])
    return qb, kb, vb


def _scores64(c, s, qb, kb, vb):
    """u [anchors, H, M] of Eq. (omission) in 64 bits."""
    d = c["d"]
    pi = torch.softmax(torch.einsum("ahd,mhd->ahm", qb, kb) / math.sqrt(d), -1)
    ob = torch.einsum("ahm,mhd->ahd", pi, vb)
    delta = (pi / (1 - pi + 1e-8))[..., None] * (ob[:, :, None] - vb.transpose(0, 1)[None])
    if s["gram"] is None:
        return delta.square().sum(-1)
    return torch.einsum("ahmi,hij,ahmj->ahm", delta, s["gram"].double(), delta)


def _topk(key, K):
    """0/1 mask of the K largest, ties to the lower index."""
    order = torch.sort(key, descending=True, stable=True).indices[:K]
    x = torch.zeros_like(key)
    x[order] = 1
    return x


def _routed64(c, s, u):
    """Block sets [anchors, H, K] of Alg. (routing) on scores u (CPU, 64 bits)."""
    u = u.cpu()
    an, N, K = s["anchors"], c["frames"], s["K"]
    na, H, M = u.shape
    A, B, C = [0.0] * na, [0.0] * na, [0.0] * na
    sets = []   # (i, j, coefficients) of every interval and boundary set

    def coef(x0, x1, ts):
        al = [(t - x0) / (x1 - x0) for t in ts]
        return (sum((1 - v) ** 2 for v in al), sum(v * v for v in al), sum(abs(v * (1 - v)) for v in al))

    for j in range(1, na):
        sets.append((j - 1, j, coef(an[j - 1], an[j], range(an[j - 1] + 1, an[j]))))
    if na >= 2:
        sets.append((0, 1, coef(an[0], an[1], range(0, an[0]))))
        sets.append((na - 2, na - 1, coef(an[-2], an[-1], range(an[-1] + 1, N))))
    out = torch.zeros((na, H, K), dtype=torch.int64)
    for h in range(H):
        x = torch.stack([_topk(u[i, h], K) for i in range(na)])
        if s["refine"] and 0 < K < M:
            lam_a, lam_r, tol = s["refine"]["lambda_anc"], s["refine"]["lambda_rec"], s["refine"]["tol"]

            def J():
                v = lam_a * ((1 - x) * u[:, h]).sum()
                for p, q, (a, b, cc) in sets:
                    xp, xq = 1 - x[p], 1 - x[q]
                    v = v + lam_r * (a * xp * u[p, h] + b * xq * u[q, h]
                                     + 2 * cc * xp * xq * (u[p, h] * u[q, h]).sqrt()).sum()
                return float(v)

            for k in range(1, s["refine"]["passes"] + 1):
                changed = False
                for i in (range(na) if k % 2 else range(na - 1, -1, -1)):
                    rec = torch.zeros(M, dtype=torch.float64)
                    for p, q, (a, b, cc) in sets:
                        if i in (p, q):
                            o = q if i == p else p
                            rec += (a if i == p else b) * u[i, h] + 2 * cc * (1 - x[o]) * (u[p, h] * u[q, h]).sqrt()
                    gain = lam_a * u[i, h] + lam_r * rec
                    new = _topk(gain, K)
                    if float((gain * (new - x[i])).sum()) > tol * max(J(), 1e-8):
                        x[i] = new
                        changed = True
                if not changed:
                    break
        for i in range(na):
            out[i, h] = x[i].nonzero().flatten()
    return out


def _attention64(c, s, idx):
    """O [anchors, S, H, d] and the log-sum-exp [anchors, H, S]."""
    N, S, H, d = s["q"].shape
    kh, vh = _block_tokens(c, s["kh"]), _block_tokens(c, s["vh"])
    na = len(s["anchors"])
    O = torch.empty((na, S, H, d), dtype=torch.float64, device=DEV)
    L = torch.empty((na, H, S), dtype=torch.float64, device=DEV)
    idx = idx.tolist()
    for h in range(H):
        kc, vc = s["k"][:, :, h].reshape(-1, d).double(), s["v"][:, :, h].reshape(-1, d).double()
        for i, f in enumerate(s["anchors"]):
            K = torch.cat([kc] + [kh[m][:, h].double() for m in idx[i][h]])
            V = torch.cat([vc] + [vh[m][:, h].double() for m in idx[i][h]])
            for r in range(0, S, 2048):
                lg = s["q"][f, r:r + 2048, h].double() @ K.T / math.sqrt(d)
                L[i, h, r:r + 2048] = torch.logsumexp(lg, -1)
                O[i, r:r + 2048, h] = torch.softmax(lg, -1) @ V
    return O, L


def _par64(r, anchors, wc, band):
    """Every frame [F, Hg, Wg, C] in 64 bits with the skipped ones reconstructed (default gate)."""
    F, Hg, Wg, C = r.shape
    w8 = torch.ones(C, dtype=torch.float64, device=DEV) if wc is None else wc.double()
    pairs = []
    for j in range(1, len(anchors)):
        a, b = anchors[j - 1], anchors[j]
        ts = list(range(a + 1, b))
        if j == 1:
            ts = list(range(0, a)) + ts
        if j == len(anchors) - 1:
            ts = ts + list(range(b + 1, F))
        if ts:
            pairs.append((a, b, ts))
    for y0 in range(0, Hg, 8):
        for x0 in range(0, Wg, 8):
            h, w = min(8, Hg - y0), min(8, Wg - x0)
            ky, kx = torch.arange(h, device=DEV), torch.arange(w // 2 + 1, device=DEV)
            kys = torch.where(ky <= (h - 1) // 2, ky, ky - h).double()[:, None]
            kxs = kx.double()[None, :]
            rad = torch.sqrt((kys / h) ** 2 + (kxs / w) ** 2)
            rmax = math.sqrt(((h // 2) / h) ** 2 + ((w // 2) / w) ** 2)
            tau = 0.25 + 0.5 * (rad / rmax if rmax > 0 else rad) ** 2
            edge = (kx == 0) | ((w % 2 == 0) & (kx == w // 2))
            kap = torch.where(edge, 1.0, 2.0).double()[None, :].expand(h, -1).clone()
            kap[0, 0] = 0
            selfc = edge[None, :] & ((ky == 0) | ((h % 2 == 0) & (2 * ky == h)))[:, None]
            mirror = edge[None, :] & ~selfc & (2 * ky > h)[:, None]
            flip = (-ky) % h
            cut = torch.sqrt((kys * 8 / h) ** 2 + (kxs * 8 / w) ** 2) > band if band >= 0 else None
            spec = {t: torch.fft.rfft2(r[t, y0:y0 + h, x0:x0 + w].double(), dim=(0, 1), norm="ortho")
                    for t in anchors}
            for a, b, ts in pairs:
                Fa, Fb = spec[a], spec[b]
                Z = (Fb * Fa.conj() * w8).sum(-1)
                W = (Fb.abs() * Fa.abs() * w8).sum(-1)
                eta = 1e-6 * W.max() + 1e-8
                rel = (W > eta) & (Z.abs() > eta)
                theta = torch.angle(Z)
                rel = torch.where(mirror, rel[flip], rel)
                theta = torch.where(mirror, -theta[flip], theta)
                theta = torch.where(selfc | ~rel, torch.zeros_like(theta), theta)
                on = rel & (kap > 0)
                num, den = (kap * Z.abs())[on].sum(), (kap * W)[on].sum()
                conf = num / (den + 1e-8) if bool(on.any()) else torch.zeros((), dtype=torch.float64, device=DEV)
                gate = torch.sigmoid((conf - tau) / 0.10)
                if cut is not None:
                    gate = torch.where(cut, torch.zeros_like(gate), gate)
                for t in ts:
                    al = (t - a) / (b - a)
                    ph = gate * theta
                    Ft = (1 - al) * Fa * torch.exp(1j * al * ph)[..., None] \
                        + al * Fb * torch.exp(-1j * (1 - al) * ph)[..., None]
                    r[t, y0:y0 + h, x0:x0 + w] = torch.fft.irfft2(Ft, s=(h, w), dim=(0, 1), norm="ortho")
    return r


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind in ("attention", "block", "ffn") and work(c)["flops"] > _MOST_FLOPS:
        return None
    if kind == "par" and work(c)["bytes"] > 1e9:
        return None
    s = prepare(case, seed)
    if kind == "select":
        r = torch.stack([x.double().square().mean(1).sqrt() for x in s["deltas"]])
        lo, hi = r.min(1, keepdim=True).values, r.max(1, keepdim=True).values
        dd = ((r - lo) / (hi - lo + 1e-8)).mean(0)
        age = torch.where(s["mask"] != 0, 0, s["ages"] + 1)
        score = dd + 0.5 * age.double() / math.ceil(c["frames"] / c["K_f"])
        return {"anchors": None, "ages": None, "mask": None, "rms": r, "score": score}
    if kind == "par":
        return {"r": _par64(s["r"].double(), _anchors(c), s["wc"], c["band"])}
    if kind == "ffn":
        F, S, D = s["r"].shape
        r = torch.zeros((F, S, D), dtype=torch.float64, device=DEV)
        for a in s["anchors"]:
            hid = s["x"][a].double() @ s["w1"].double().T
            if s["b1"] is not None:
                hid += s["b1"].double()
            hid = 0.5 * hid * (1 + torch.tanh(math.sqrt(2 / math.pi) * (hid + 0.044715 * hid ** 3)))
            r[a] = hid @ s["w2"].double().T
            if s["b2"] is not None:
                r[a] += s["b2"].double()
        return {"r": _par64(r.reshape(F, *s["grid"], D), s["anchors"], None, -1.0).reshape(F, S, D)}
    if kind == "route":
        qb, kb, vb = _pooled64(c, s)
        return {"idx": None, "u": _scores64(c, s, qb, kb, vb), "qbar": qb, "kbar": kb, "vbar": vb}
    N, S, H, d = s["q"].shape
    if kind == "attention":
        O, L = _attention64(c, s, s["idx"])
        O = O.reshape(-1, S, H * d)
        return {"o": O, "lse": L} if c["lse"] else {"o": O}
    O, _ = _attention64(c, s, _routed64(c, s, _scores64(c, s, *_pooled64(c, s))))
    O = O.reshape(-1, S, H * d)
    if c["w_o"]:
        O = O @ s["more"]["w_o"].double().T + s["more"]["b_o"].double()
    r = torch.zeros((N, S, H * d), dtype=torch.float64, device=DEV)
    r[s["anchors"]] = O
    if len(s["anchors"]) < N:
        r = _par64(r.reshape(N, *s["grid"], H * d), s["anchors"], None, c["band"]).reshape(N, S, H * d)
    out = {"r": r, "idx": None}
    if s["x"] is not None:
        out["x"] = s["x"].double() + r
    return out
