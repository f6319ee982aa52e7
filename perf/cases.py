"""Performance cases of the K-interval attention operator.

Each case is one pass a user's program makes through the public entry points: a training
step of one attention layer (``kint.forward`` and ``kint.backward`` with the buffers a training
loop keeps, or the differentiable ``kint_attention``), a forward through ``kint.forward`` or the
allocation-free ``kint_attn_fwd_noalloc``, or a whole ``KIntSelfAttention`` layer.  ``listed()`` holds the fixed cases, ``draw(rng)`` one more of
the same ranges; ``prepare`` makes what the program has in hand, ``run`` is the pass,
``work`` its compulsory bytes and operations, ``exact`` its outputs in 64 bits.
"""
from __future__ import annotations

import math

import torch

from paper_2609_33591_gb300 import kint
from paper_2609_33591_gb300.attention import KIntSelfAttention, kint_attention

CALIB = {"minmax": kint.CALIB_MINMAX, "fwm": kint.CALIB_FWM, "softmax": kint.CALIB_SOFTMAX}
RECON = {"lerp": kint.RECON_LERP, "nearest": kint.RECON_NEAREST}
STE = {"weight": kint.STE_WEIGHT, "prob": kint.STE_PROB}
GRAD = {"full": kint.GRAD_FULL, "detach": kint.GRAD_DETACH}
PREC = {"tf32": kint.PREC_TF32, "3xtf32": kint.PREC_3XTF32}

# The largest case's score elements times head size (B H T^2 d): no drawn case exceeds it.
WORK_MAX = 16 * 16384 ** 2 * 128


def _case(name, kind, B, H, T, d, calib, K, recon, ste, grad="full", prec="tf32", tau=8.0, peaked=0.0):
    c = dict(kind=kind, B=B, H=H, T=T, d=d, calib=calib, K=K, recon=recon, ste=ste, grad=grad, prec=prec, tau=tau,
             peaked=peaked)
    if name:
        c = dict(name=name, **c)
    return c


def listed():
    return [
        # the smallest training call: one short sequence, two heads, fp32-accurate products, through autograd
        _case("tiny_train_3x", "autograd", 1, 2, 128, 64, "minmax", 4, "lerp", "weight", prec="3xtf32"),
        # a short ragged batch (fine-tuning on prompts that do not fill the context)
        _case("short_ragged_train", "train", 1, 12, 197, 64, "fwm", 8, "nearest", "weight"),
        # a prompt prefill in a serving loop that must not allocate (one sequence, odd length)
        _case("prefill_noalloc", "noalloc", 1, 12, 333, 64, "fwm", 4, "nearest", "weight"),
        # a whole small GPT-2-style layer: projections, head split, attention, and their gradients
        _case("layer_train_small", "layer", 2, 4, 160, 64, "fwm", 4, "nearest", "prob"),
        # GPT-2-small attention, the paper's main training recipe (batch 8, context 1024)
        _case("gpt2_train", "train", 8, 12, 1024, 64, "fwm", 4, "nearest", "prob"),
        # the same layer with fp32-accurate products (parity and debugging runs)
        _case("gpt2_train_3x", "train", 8, 12, 1024, 64, "fwm", 4, "nearest", "prob", prec="3xtf32"),
        # the softmax comparator every experiment trains beside it
        _case("gpt2_train_softmax", "train", 8, 12, 1024, 64, "softmax", 4, "lerp", "weight"),
        # validation pass of the same layer: forward only, fp32-accurate (the paper evaluates with TF32 off)
        _case("gpt2_eval_3x", "forward", 8, 12, 1024, 64, "fwm", 4, "nearest", "weight", prec="3xtf32"),
        # MinMax side of the variant sweep: per-row grids, both extremum channels
        _case("sweep_minmax_train", "train", 4, 12, 1024, 64, "minmax", 8, "nearest", "prob"),
        # detached-extrema control of the sweep, fine grid, ragged sequence length
        _case("sweep_fwm_detach_ragged", "train", 4, 12, 1000, 64, "fwm", 16, "lerp", "weight", grad="detach"),
        # a 1B-scale layer: head size 128, context 2048, 5% of the rows peaked
        _case("1b_train", "train", 4, 16, 2048, 128, "fwm", 4, "nearest", "weight", peaked=0.05),
        # long-context training: one sequence of 16384, fine per-row grids
        _case("long_train", "train", 1, 16, 16384, 128, "minmax", 16, "lerp", "weight"),
    ]


def draw(rng):
    """One more case: sequence lengths over the logarithm of 1 .. 16384, odd ones among them."""
    kind = rng.choices(["train", "autograd", "forward", "noalloc", "layer"], [5, 1, 2, 1, 1])[0]
    d = 64 if kind == "layer" else rng.choice([64, 64, 128])
    prec = "3xtf32" if (d == 64 and rng.random() < 0.3) else "tf32"
    T = int(round(math.exp(rng.uniform(math.log(16), math.log(2048 if kind in ("layer", "noalloc") else 16384)))))
    T = max(1, T + rng.choice([0, 1, -1, 7]) if rng.random() < 0.5 else -(-T // 64) * 64)
    cap = WORK_MAX // (3 if prec == "3xtf32" else 1) // (T * T * d)
    if kind == "noalloc":  # the forward scratch of the library holds 32 MiB
        cap = min(cap, (32 << 20) // (d * 4 * (-(-T // 32) * 32) * (6 if prec == "3xtf32" else 1)))
    cap = max(1, min(cap, (1 << 20) // T, 128))
    bh = max(1, int(round(math.exp(rng.uniform(0.0, math.log(cap))))))
    H = min(bh, rng.choice([1, 4, 12, 16]))
    B = max(1, bh // H)
    if kind == "layer":
        B, H = min(B, 8), rng.choice([2, 4, 12])
    calib = rng.choice(["fwm", "fwm", "fwm", "minmax", "minmax", "softmax"])
    return _case(None, kind, B, H, T, d, calib, rng.choice([4, 8, 16]), rng.choice(["lerp", "nearest", "nearest"]),
                 rng.choice(["weight", "prob"]), rng.choice(["full", "full", "detach"]), prec,
                 rng.choice([6.0, 8.0]), 0.05 if rng.random() < 0.2 else 0.0)


def _config(c):
    return kint.Config(Kint=c["K"], calib=CALIB[c["calib"]], tau=c["tau"], recon=RECON[c["recon"]],
                       ste=STE[c["ste"]], grad=GRAD[c["grad"]])


def _inputs(c, seed):
    """Q, K, V, dO i.i.d. N(0, 1) fp32; with ``peaked``, that share of the query rows is moved
    along one of its causal keys so that this score rises by 12."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B, H, T, d = c["B"], c["H"], c["T"], c["d"]
    q, k, v, do = (torch.randn(B, H, T, d, generator=gen, device="cuda") for _ in range(4))
    if c["peaked"] > 0:
        hit = torch.rand(B, H, T, generator=gen, device="cuda") < c["peaked"]
        i = torch.arange(T, device="cuda", dtype=torch.float32)
        j = (torch.rand(B, H, T, generator=gen, device="cuda") * (i + 1)).long().clamp(max=T - 1)
        j = torch.minimum(j, torch.arange(T, device="cuda"))
        kj = torch.gather(k, 2, j.unsqueeze(-1).expand(B, H, T, d))
        step = 12.0 * math.sqrt(d) * kj / (kj * kj).sum(-1, keepdim=True)
        q = torch.where(hit.unsqueeze(-1), q + step, q).contiguous()
    return q, k, v, do


def _layer_inputs(c, seed):
    """x, dy N(0, 1); weights of the GPT-2 initialisation scaled so that the scores spread over
    the window as those of unit-variance queries and keys do."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    C = c["H"] * c["d"]
    x = torch.randn(c["B"], c["T"], C, generator=gen, device="cuda")
    dy = torch.randn(c["B"], c["T"], C, generator=gen, device="cuda")
    wa = torch.randn(3 * C, C, generator=gen, device="cuda") / math.sqrt(C)
    wp = torch.randn(C, C, generator=gen, device="cuda") / math.sqrt(C)
    ba = 0.02 * torch.randn(3 * C, generator=gen, device="cuda")
    bp = 0.02 * torch.randn(C, generator=gen, device="cuda")
    return x, dy, wa, ba, wp, bp


def prepare(case, seed):
    cfg, prec = _config(case), PREC[case["prec"]]
    if case["kind"] == "layer":
        x, dy, wa, ba, wp, bp = _layer_inputs(case, seed)
        layer = KIntSelfAttention(x.shape[-1], case["H"], cfg, prec).cuda()
        with torch.no_grad():
            for p, w in zip((layer.c_attn.weight, layer.c_attn.bias, layer.c_proj.weight, layer.c_proj.bias),
                            (wa, ba, wp, bp)):
                p.copy_(w)
        return dict(kind="layer", layer=layer, x=x.requires_grad_(True), dy=dy, params=list(layer.parameters()))
    q, k, v, do = _inputs(case, seed)
    state = dict(kind=case["kind"], q=q, k=k, v=v, cfg=cfg, prec=prec)
    if case["kind"] == "autograd":
        for t in (q, k, v):
            t.requires_grad_(True)
        state["do"] = do
    elif case["kind"] in ("train", "noalloc"):
        # training and serving loops keep their output, row-statistics and workspace buffers
        state["O"] = torch.empty_like(q)
        state["stats"] = kint.alloc_rowstats(*q.shape, q.device, cfg.prob)
    if case["kind"] == "train":
        state["do"], state["grads"] = do, tuple(torch.empty_like(q) for _ in range(3))
        state["wf"], state["wb"] = (kint.workspace(*q.shape, prec, is_bwd, q.device) for is_bwd in (0, 1))
    return state


def run(state):
    kind = state["kind"]
    if kind == "layer":
        y = state["layer"](state["x"])
        g = torch.autograd.grad(y, [state["x"], *state["params"]], state["dy"])
        return {"y": y.detach(), "dx": g[0], "dparams": list(g[1:])}
    q, k, v = state["q"], state["k"], state["v"]
    if kind == "autograd":
        o = kint_attention(q, k, v, state["cfg"], state["prec"])
        dq, dk, dv = torch.autograd.grad(o, (q, k, v), state["do"])
        return {"O": o.detach(), "dQ": dq, "dK": dk, "dV": dv}
    if kind == "train":
        cfg, prec = state["cfg"], state["prec"]
        o, st = kint.forward(q, k, v, cfg, prec, O=state["O"], stats=state["stats"], ws=state["wf"])
        dq, dk, dv = kint.backward(q, k, v, o, state["do"], st, cfg, prec, grads=state["grads"], ws=state["wb"])
        return {"O": o, "dQ": dq, "dK": dk, "dV": dv}
    if kind == "forward":
        o, st = kint.forward(q, k, v, state["cfg"], state["prec"])
    else:
        o, st, cfg = state["O"], state["stats"], state["cfg"]
        B, H, T, d = q.shape
        rc = kint.kint_attn_fwd_noalloc(q, k, v, o, st, B, H, T, d, cfg.Kint, cfg.calib, cfg.tau, cfg.recon, cfg.ste,
                                        cfg.grad, 1, state["prec"])
        if rc != 0:
            raise kint.KintError(rc, "kint_attn_fwd_noalloc")
    return {"O": o, "W": st["W"], "row_max": st["row_max"], "arg_max": st["arg_max"], "n_max": st["n_max"]}


def work(case):
    """Compulsory traffic (each input read once, each output written once) and the operator's
    2 (forward) or 6 (forward and backward) causal T x T x d contractions."""
    B, H, T, d = case["B"], case["H"], case["T"], case["d"]
    n, rows, u = 4 * B * H * T * d, 4 * B * H * T, 2 * B * H * d * T * (T + 1) // 2
    if case["kind"] in ("forward", "noalloc"):
        return {"bytes": 4 * n + 4 * rows, "flops": 2 * u}
    if case["kind"] in ("train", "autograd"):  # Q, K, V, dO in; O, dQ, dK, dV out
        return {"bytes": 8 * n, "flops": 6 * u}
    C = H * d
    weights = 4 * (4 * C * C + 4 * C)
    return {"bytes": 4 * n + 2 * weights, "flops": 6 * u + 3 * 2 * B * T * 4 * C * C}


def _weights64(s, ok, c):
    """Row quantities of one block of rows in 64 bits: the reconstructed weights of the forward
    and of the surrogate, the secant slopes and, for MinMax, dw/dm."""
    inf = float("inf")
    M = s.masked_fill(~ok, -inf).amax(-1, keepdim=True)
    if c["calib"] == "softmax":
        w = torch.exp(s - M).masked_fill(~ok, 0.0)
        return w, w, w, None, M, None
    K = c["K"]
    if c["calib"] == "fwm":
        m, live = M - c["tau"], None
        h = torch.full_like(M, c["tau"] / K)
    else:
        m = s.masked_fill(~ok, inf).amin(-1, keepdim=True)
        live = (M - m) > 1e-12
        h = torch.where(live, M - m, torch.ones_like(M)) / K
    u = (s - m) / h
    r = u.floor().clamp(0, K - 1)
    t = (u - r).clamp(0.0, 1.0)
    er = torch.exp((m - M) + r * h)
    er1 = torch.exp((m - M) + (r + 1) * h)
    de = er1 - er
    wl = er + t * de
    wn = torch.where(t >= 0.5, er1, er)
    slope = de / h
    dm = None
    if c["calib"] == "fwm":
        dead = ~ok | (u < 0)
    else:
        dm = (1 - r / K) * er + t * ((1 - (r + 1) / K) * er1 - (1 - r / K) * er) + slope * (u / K - 1)
        wl, wn = (torch.where(live, w, torch.ones_like(w)) for w in (wl, wn))
        dm = dm.masked_fill(~ok | ~live, 0.0)
        slope = slope.masked_fill(~live, 0.0)
        dead = ~ok
    wl, wn, slope = (x.masked_fill(dead, 0.0) for x in (wl, wn, slope))
    if c["recon"] == "lerp":
        return wl, wl, slope, dm, M, m
    return wn, (wl if c["ste"] == "prob" else wn), slope, dm, M, m


def _attention64(q, k, v, do, c):
    """O, W, M and (with do) dQ, dK, dV in 64 bits, blocks of rows of one head at a time."""
    B, H, T, d = q.shape
    scale = 1.0 / math.sqrt(d)
    O, W, Mx = torch.empty_like(q), q.new_empty(B, H, T), q.new_empty(B, H, T)
    dQ, dK, dV = (torch.zeros_like(q) for _ in range(3)) if do is not None else (None, None, None)
    step = max(1, (1 << 25) // T)
    for b in range(B):
        for h in range(H):
            for i0 in range(0, T, step):
                i1 = min(T, i0 + step)
                Q, K, V = q[b, h, i0:i1], k[b, h, :i1], v[b, h, :i1]
                s = (Q @ K.T) * scale
                ok = torch.arange(i1, device=q.device)[None, :] <= torch.arange(i0, i1, device=q.device)[:, None]
                w, ws, slope, dm, M, m = _weights64(s, ok, c)
                Wf, Ws = w.sum(-1, keepdim=True), ws.sum(-1, keepdim=True)
                P = w / Wf
                O[b, h, i0:i1] = P @ V
                W[b, h, i0:i1], Mx[b, h, i0:i1] = Wf[:, 0], M[:, 0]
                if do is None:
                    continue
                G = do[b, h, i0:i1]
                g = G @ V.T
                gam = (g - (ws * g).sum(-1, keepdim=True) / Ws) / Ws
                ds = gam * slope
                if c["calib"] != "softmax" and c["grad"] == "full":
                    cm = (gam * dm).sum(-1, keepdim=True) if dm is not None else 0.0
                    cM = -ds.sum(-1, keepdim=True) - cm
                    top = (s == M) & ok
                    ds = ds + top * (cM / top.sum(-1, keepdim=True))
                    if dm is not None:
                        low = (s == m) & ok
                        ds = ds + low * (cm / low.sum(-1, keepdim=True))
                        ds = ds * ((M - m) > 1e-12)
                dQ[b, h, i0:i1] = scale * (ds @ K)
                dK[b, h, :i1] += scale * (ds.T @ Q)
                dV[b, h, :i1] += P.T @ G
    return O, W, Mx, dQ, dK, dV


def exact(case, seed):
    if case["kind"] == "layer":
        x, dy, wa, ba, wp, bp = (t.double() for t in _layer_inputs(case, seed))
        B, T, C = x.shape
        H, d = case["H"], case["d"]
        q, k, v = (t.view(B, T, H, d).transpose(1, 2).contiguous() for t in (x @ wa.T + ba).split(C, dim=2))
        dz = dy @ wp
        do = dz.view(B, T, H, d).transpose(1, 2).contiguous()
        O, _, _, dQ, dK, dV = _attention64(q, k, v, do, case)
        z = O.transpose(1, 2).reshape(B, T, C)
        dqkv = torch.cat([t.transpose(1, 2).reshape(B, T, C) for t in (dQ, dK, dV)], dim=2).view(B * T, 3 * C)
        rows = dy.reshape(B * T, C)
        return {"y": z @ wp.T + bp, "dx": (dqkv @ wa).view(B, T, C),
                "dparams": [dqkv.T @ x.reshape(B * T, C), dqkv.sum(0), rows.T @ z.reshape(B * T, C), rows.sum(0)]}
    q, k, v, do = (t.double() for t in _inputs(case, seed))
    train = case["kind"] in ("train", "autograd")
    O, W, M, dQ, dK, dV = _attention64(q, k, v, do if train else None, case)
    if train:
        return {"O": O, "dQ": dQ, "dK": dK, "dV": dV}
    return {"O": O, "W": W, "row_max": M, "arg_max": None, "n_max": None}
