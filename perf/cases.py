"""The work that users of this library have it do, as measured cases.

A case is one pass of a user's program through the public entry points:

* ``train``: a training step of one group through ``Group.forward`` and ``Group.backward``, with the
  caller's sublayer outputs and gradients; the gradient of the group's output is handed over by the
  layer above (a copy into ``dX``), parameter gradients accumulate over the micro-batches.
* ``forward``: prefill or evaluation through ``Group.forward``; with ``halo`` a later chunk of its
  sequences (chunked prefill, context parallelism), slot by slot with the previous chunk's last
  sublayer outputs.
* ``decode``: one new token for each of ``B`` sequences through ``Group.forward_decode``, called
  eagerly or replayed as a captured CUDA graph of the step, as a serving loop does.
* ``stack``: a small model under autograd (``XhcStack``): the streams' expansion, one group around the
  model's own sublayers, the sum of the streams, forward and backward.

State and sublayer outputs are N(0, 1) in bf16, weights and biases N(0, 0.02) in fp32, gating scalars
0.01, conv taps N(0, 1 / kappa): the distributions of this repository's workloads.  Tokens whose routing
is a near tie are drawn anew, as the tests do: either choice would be right there.
"""
import math

import torch
from torch import nn

from paper_2607_14530_gb300.model import XhcStack
from paper_2607_14530_gb300.xhc import FLASH, FULL, MHC, Config, Group

DEV = "cuda"
F64 = torch.float64
CONV = (4, 8, 12)
EPS = 1e-5
VARIANT = {"mhc": MHC, "full": FULL, "flash": FLASH}


def _case(name, kind, variant, N, k, m, C, G, mlp, B, S, **more):
    """``mlp``: the augmentation mask of the slots; ``B`` sequences of ``S`` tokens (decode: one token
    each, at positions around ``S``)."""
    c = dict(kind=kind, variant=variant, N=N, k=k, m=m, C=C, G=G, mlp=mlp, B=B, S=S, router="sigmoid",
             sparse_read=False, halo=False, graph=False)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the training workload that the benchmark quotes: one micro-batch of 8 x 4096 tokens
        _case("train_flash4", "train", "flash", 16, 4, 2, 4096, 4, 0xA, 8, 4096),
        # the widest state of the expansion sweep
        _case("train_flash4_n32", "train", "flash", 32, 4, 2, 4096, 4, 0xA, 2, 8192),
        # one full-xHC MLP sublayer with temporal augmentation, two long sequences
        _case("train_full_mlp", "train", "full", 16, 4, 2, 2048, 1, 0x1, 2, 8192),
        # the dense mHC baseline: every stream active, no router, no augmentation
        _case("train_mhc", "train", "mhc", 4, 4, 4, 2048, 1, 0x0, 1, 8192),
        # an xHC-Flash block on ragged sequences (lengths that no tile divides)
        _case("train_flash2_ragged", "train", "flash", 8, 4, 2, 1536, 2, 0x2, 3, 701),
        # a small model's step, where launches and latency count
        _case("train_small", "train", "full", 16, 4, 2, 256, 1, 0x1, 1, 512),
        # eight active streams and a width that no tile divides
        _case("train_k8_odd_width", "train", "full", 12, 8, 3, 1160, 1, 0x1, 2, 500),
        # prefill of one prompt
        _case("prefill_flash4", "forward", "flash", 16, 4, 2, 4096, 4, 0xA, 1, 4096),
        # a middle chunk of a chunked prefill of several prompts
        _case("prefill_chunk", "forward", "flash", 16, 4, 2, 2048, 4, 0xA, 3, 512, halo=True),
        # interactive decoding of one sequence
        _case("decode_1", "decode", "flash", 16, 4, 2, 4096, 4, 0xA, 1, 1000),
        # a serving batch, the step replayed as a CUDA graph
        _case("decode_256_graph", "decode", "flash", 16, 4, 2, 4096, 4, 0xA, 256, 4096, graph=True),
        # a small model under autograd, forward and backward
        _case("stack_train", "stack", "flash", 8, 4, 2, 1024, 4, 0xA, 2, 1024),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["train", "train", "train", "forward", "forward", "decode", "decode", "stack"])
    variant = rng.choice(["flash", "flash", "flash", "full", "full", "mhc"])
    G, mlp = 1, rng.choice([0x1, 0x1, 0x0])
    N, k = rng.choice([4, 8, 12, 16, 16, 16, 24, 32]), 4
    if kind == "stack" or variant == "flash":
        variant = "flash"
        G = rng.choice([2, 4, 4])
        mlp = 0x2 if G == 2 else 0xA
    if variant == "mhc":
        N = k = rng.choice([2, 4, 4])
        m, mlp, G = N, 0, 1
    else:
        if rng.random() < 0.1 and N >= 8:
            k = 8
        m = rng.choice([2, 2, 2, 1, 0, k])
    # hidden sizes: mostly multiples of 128, now and then any multiple of 8
    C = log(2, 32) * 128 if rng.random() < 0.8 else log(32, 512) * 8
    more = {}
    if variant != "mhc" and m < k and rng.random() < 0.15:
        more["router"] = "softmax"
    if variant != "mhc" and rng.random() < 0.1:
        more["sparse_read"] = True
    if kind == "decode":
        B, S = log(1, 512), log(8, 8192)
        more["graph"] = rng.random() < 0.5
    else:
        tokens = log(64, 32768) if kind == "train" else log(64, 16384)
        # a pass that costs no more than the largest listed one (eight active streams, and widths that
        # the matrix units' tiles do not divide, cost several times as much for each byte)
        much = (4 if k == 8 else 1) * (8 if C % 128 else 1)
        tokens = max(1, min(tokens, 32768 * 16 * 4096 // (N * C * much)))
        if kind == "stack":
            tokens, C = min(tokens, 4096), min(C, 2048)
        B = max(1, min(tokens // 16, rng.choice([1, 1, 2, 3, 8])))
        S = max(1, tokens // B)
        if kind == "forward" and mlp and rng.random() < 0.3:
            more["halo"] = True
    return _case("", kind, variant, N, k, m, C, G, mlp, B, S, **more)


# ---- inputs ------------------------------------------------------------------------------------


def _cfg(case):
    conv = () if case["variant"] == "mhc" else CONV
    seq = 0 if case["kind"] == "decode" else case["S"]
    return Config(VARIANT[case["variant"]], case["N"], case["k"], case["m"], case["C"], case["G"], case["mlp"],
                  conv, seq_len=seq, router=case["router"], sparse_read=case["sparse_read"])


def _tokens(case):
    return case["B"] if case["kind"] == "decode" else case["B"] * case["S"]


def _normal(gen, *shape, std=1.0, dtype=torch.bfloat16):
    out = torch.empty(shape, dtype=dtype, device=DEV)
    flat, step = out.view(-1), 1 << 27
    for i in range(0, flat.numel(), step):
        n = min(step, flat.numel() - i)
        flat[i:i + n] = torch.randn(n, generator=gen, dtype=torch.float32, device=DEV) * std
    return out


def _params(cfg, gen):
    P = {}
    for name, shape in cfg.param_shapes().items():
        if name.startswith("alpha"):
            P[name] = torch.full(shape, 0.01, dtype=torch.float32, device=DEV)
        else:
            std = 1.0 / math.sqrt(shape[0]) if name.startswith("conv_w") else 0.02
            P[name] = _normal(gen, *shape, std=std, dtype=torch.float32)
    return P


def _near_ties(case, X, W):
    """Tokens of X for which two routed logits that the selection separates are nearly equal."""
    m, n = case["m"], case["k"] - case["m"]
    found = []
    for i in range(0, X.shape[0], 2048):
        x = X[i:i + 2048].reshape(-1, W.shape[0]).float()
        mu = x.mean(1, keepdim=True)
        z = (x @ W - mu * W.sum(0)) / x.var(1, unbiased=False, keepdim=True).add(EPS).sqrt()
        s = z[:, m:].sort(1, descending=True).values
        s = s[:, :min(n + 1, s.shape[1])]
        if s.shape[1] > 1:
            gap = (s[:, :-1] - s[:, 1:]).amin(1)
            found.append(i + (gap < 1e-3 * z.abs().amax(1).clamp(min=1.0)).nonzero()[:, 0])
    return torch.cat(found) if found else torch.empty(0, dtype=torch.int64, device=DEV)


def _state(case, T, W, gen, streams):
    """A state [T, streams, C]; with one stream, the hidden vectors that are expanded to N."""
    X = _normal(gen, T, streams, case["C"])
    if W is not None:
        def ties(x):
            return _near_ties(case, x.expand(x.shape[0], case["N"], case["C"]), W)

        rows = ties(X)
        while rows.numel():
            X[rows] = _normal(gen, rows.numel(), streams, case["C"])
            rows = rows[ties(X[rows])]
    return X


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    cfg, T, C = _cfg(case), _tokens(case), case["C"]
    s = {"case": case, "cfg": cfg, "T": T}
    if case["kind"] == "stack":
        s["stack"] = XhcStack(cfg, 1, lambda l, t: _Gain(C), seed=int(seed) % 1000003).to(DEV)
        W = getattr(s["stack"].groups[0], "W_r", None)
        s["hidden"] = _state(case, T, None if W is None else W.detach(), gen, 1).reshape(T, C).requires_grad_(True)
        s["dy"] = _normal(gen, T, C)
        return s
    s["P"] = _params(cfg, gen)
    s["X"] = _state(case, T, s["P"].get("W_r"), gen, case["N"])
    s["outs"] = [_normal(gen, T, C) for _ in range(case["G"])]
    R = max(CONV) - 1
    conv = [t for t in range(case["G"]) if cfg.K(t) > 1]
    if case["kind"] == "train":
        s["dX_up"] = _normal(gen, T, case["N"], C)
        s["d_inputs"] = [_normal(gen, T, C) for _ in range(case["G"])]
    elif case["kind"] == "decode":
        # each sequence at a position of its own, its last R sublayer outputs in the slot's ring
        spread = torch.randint(0, 16, (case["B"],), generator=gen, device=DEV)
        s["pos"] = (case["S"] + spread).to(torch.int64)
        s["rings"] = [_normal(gen, T, R, C) if t in conv else None for t in range(case["G"])]
    elif case["halo"]:
        s["halos"] = [_normal(gen, case["B"], R, C) if t in conv else None for t in range(case["G"])]
    return s


def _grad_buffers(cfg):
    """Zeroed gradients: one tensor for each weight, and the small vectors (gating scalars and biases)
    as views of one buffer, the way an optimizer's bucket keeps them."""
    shapes = cfg.param_shapes()
    small = [n for n in shapes if n.startswith(("alpha", "b_"))]
    room = {n: -(-math.prod(shapes[n]) // 4) * 4 for n in small}
    flat = torch.zeros(sum(room.values()), dtype=torch.float32, device=DEV)
    grads, at = {}, 0
    for n in shapes:
        if n in room:
            grads[n] = flat[at:at + math.prod(shapes[n])].view(shapes[n])
            at += room[n]
        else:
            grads[n] = torch.zeros(shapes[n], dtype=torch.float32, device=DEV)
    return grads, flat


class _Gain(nn.Module):
    """A stand-in for a sublayer, whose own cost is not the library's: a gain for each channel."""

    def __init__(self, C):
        super().__init__()
        self.gain = nn.Parameter(torch.linspace(0.5, 1.5, C))

    def forward(self, x):
        return x * self.gain.to(x.dtype)


def prepare(case, seed):
    s = _inputs(case, seed)
    cfg, T, C = s["cfg"], s["T"], case["C"]
    if case["kind"] == "stack":
        return s
    g = s["g"] = Group(cfg)
    s["saved"], s["ws"] = g.alloc(T)

    def rows():
        return [torch.empty(T, C, dtype=torch.bfloat16, device=DEV) for _ in range(cfg.G)]

    s["inputs"] = rows()
    if case["kind"] == "train":
        s["dX"], s["d_outs"] = torch.empty_like(s["dX_up"]), rows()
        s["grads"], s["small"] = _grad_buffers(cfg)
    if case["kind"] == "decode":
        s["ring_bytes"] = [None if r is None else r.view(-1).view(torch.uint8) for r in s["rings"]]
    if case["graph"]:
        keep = {n: s[n].clone() for n in ("X", "pos")}
        rings = [None if r is None else r.clone() for r in s["rings"]]
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode(s)
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _decode(s)
        for n, v in keep.items():
            s[n].copy_(v)
        for r, v in zip(s["rings"], rings):
            if r is not None:
                r.copy_(v)
    return s


# ---- one pass ----------------------------------------------------------------------------------


def _decode(s):
    s["g"].forward_decode(s["P"], s["X"], s["outs"], s["ring_bytes"], s["pos"], s["saved"], s["ws"],
                          inputs=s["inputs"])


def run(state):
    s, case = state, state["case"]
    if case["kind"] == "stack":
        stack = s["stack"]
        stack.zero_grad(set_to_none=True)
        s["hidden"].grad = None
        y = stack(s["hidden"])
        y.backward(s["dy"])
        return {"y": y.detach(), "hidden": s["hidden"].grad, "grads": _stack_grads(stack)}
    g, P, X, saved, ws = s["g"], s["P"], s["X"], s["saved"], s["ws"]
    if case["kind"] == "train":
        s["dX"].copy_(s["dX_up"])
        g.forward(P, X, s["outs"], saved, ws, inputs=s["inputs"])
        g.backward(P, X, s["dX"], s["outs"], s["d_inputs"], s["grads"], saved, ws, d_outs=s["d_outs"])
        big = {n: v for n, v in s["grads"].items() if not n.startswith(("alpha", "b_"))}
        return {"inputs": s["inputs"], "X": X, "d_outs": s["d_outs"], "dX": s["dX"], "grads": big,
                "small": s["small"]}
    if case["kind"] == "decode":
        if case["graph"]:
            s["graph"].replay()
        else:
            _decode(s)
        return {"inputs": s["inputs"], "X": X, "rings": s["rings"], "pos": s["pos"]}
    if case["halo"]:
        pp = g.params(P)
        for t in range(case["G"]):
            g.pre_fwd(t, pp, X, s["inputs"][t], saved, ws)
            g.post_fwd(t, pp, X, s["outs"][t], saved, ws, halo=s["halos"][t])
    else:
        g.forward(P, X, s["outs"], saved, ws, inputs=s["inputs"])
    return {"inputs": s["inputs"], "X": X}


def _stack_grads(stack):
    """The weights' gradients one by one, and the others' as one vector: biases, gating scalars, the
    sublayers' gains, and the residual map's weights (the streams' sum cannot tell its rows apart, so
    their gradient is zero and holds nothing but rounding)."""
    return _by_name({n: p.grad for n, p in stack.groups[0].named_parameters()})


def _by_name(grads):
    big = {n: v for n, v in grads.items() if n.startswith(("W_r", "W_p", "conv_w")) and n != "W_res"}
    return dict(big, others=torch.cat([v.reshape(-1) for n, v in grads.items() if n not in big]))


# ---- what a pass cannot do without -------------------------------------------------------------


def _widths(case):
    """Columns of the full-state projection and of each slot's active-state projection."""
    k, G = case["k"], case["G"]
    full = (case["N"] if case["m"] < k else 0) + G * case["N"]
    act = [k * (1 + len(CONV) if (case["mlp"] >> t) & 1 else 1) + (k * k if t == G - 1 else 0) for t in range(G)]
    return full, act


def work(case):
    T, N, k, C, G = _tokens(case), case["N"], case["k"], case["C"], case["G"]
    full, act = _widths(case)
    state, row, active = 2 * T * N * C, 2 * T * C, 2 * T * k * C
    taps = C * sum(CONV) * bin(case["mlp"]).count("1")
    weights = 4 * (N * C * full + k * C * sum(act) + taps)
    # forward: state, sublayer outputs and weights read, sublayer inputs and active rows written
    b = state + G * row + weights + G * row + active
    f = 2.0 * T * (N * C * full + k * C * sum(act))
    if case["kind"] == "decode":
        conv = bin(case["mlp"]).count("1")
        b += conv * (max(CONV) - 1) * row + conv * row  # the rings' rows read, one row written
    if case["kind"] in ("train", "stack"):
        # backward: gradient of the state and of the inputs read, that of the state and of the
        # sublayer outputs written, weight gradients read and written
        b += 2 * state + 2 * G * row + 2 * weights
        f *= 3
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    # bf16 results, among them sums whose bf16 intermediate states may round the other way: measured
    # against exact(), 1.6e-3 to 2.2e-3 for every bf16 result and what follows from one; up to 9e-3
    # for the gradients of a model, in which bf16 sublayers feed the next slot
    if case["kind"] == "stack":
        return {"rel": 3e-2, "max": 0.9}
    return {"rel": 1e-2, "max": 0.3}


# ---- the same in 64 bits -----------------------------------------------------------------------


def _conv64(out, w, hist):
    """Causal depthwise conv of sequences [B, S, C] with taps w [kappa, C]; hist [B, R, C] or None
    holds the outputs before each sequence."""
    B, S, C = out.shape
    R = max(CONV) - 1
    ext = torch.cat([torch.zeros(B, R, C, dtype=F64, device=DEV) if hist is None else hist, out], 1)
    g = 0.0
    for i in range(w.shape[0]):
        g = g + w[i] * ext[:, R - i:R - i + S]
    return g


def _group64(case, P, X, outs, hists=None):
    """One group in 64 bits: ``outs[t]`` [B, S, C], or a function of the slot's input [T, C].
    Returns the inputs, the active streams and their new rows."""
    T, N, C = X.shape
    k, m, G = case["k"], case["m"], case["G"]
    x = X.reshape(T, N * C)
    nu = (x * x).mean(1, keepdim=True)
    rms = (nu + EPS).rsqrt()
    H = [torch.sigmoid(P["alpha_pre"][t] * rms * (x @ P["W_pre.%d" % t]) + P["b_pre"][t]) for t in range(G)]
    I, p = torch.arange(m, device=DEV).expand(T, m), torch.ones(T, m, dtype=F64, device=DEV)
    if m < k:
        mu = x.mean(1, keepdim=True)
        z = (x @ P["W_r"] - mu * P["W_r"].sum(0)) * (nu - mu * mu + EPS).rsqrt()
        s = torch.softmax(z, 1) if case["router"] == "softmax" else torch.sigmoid(z)
        top = z[:, m:].detach().sort(dim=1, descending=True, stable=True).indices[:, :k - m] + m
        I, p = torch.cat([I, top], 1), torch.cat([p, s.gather(1, top)], 1)
    A0 = X.gather(1, I[:, :, None].expand(T, k, C))
    A, inputs = A0, []
    for t in range(G):
        h = H[t].gather(1, I)
        if case["sparse_read"]:
            inputs.append(torch.einsum("tj,tjc->tc", h, A))
        else:
            inputs.append(torch.einsum("ti,tic->tc", H[t], X) + torch.einsum("tj,tjc->tc", h, A - A0))
        out = outs[t](inputs[t]) if callable(outs[t]) else outs[t]
        a = A.reshape(T, k * C)
        r = ((a * a).mean(1, keepdim=True) + EPS).rsqrt()
        v = [out.reshape(T, C)]
        if (case["mlp"] >> t) & 1:
            for j in range(len(CONV)):
                w = P["conv_w.%d.%d" % (t, j)]
                g = _conv64(out, w, None if hists is None else hists[t]).reshape(T, C)
                new = g
                for u in v:
                    new = new - (g * u).sum(1, keepdim=True) / ((u * u).sum(1, keepdim=True) + 1e-6 * C) * u
                v.append(new)
        y = P["alpha_post"][t] * r * (a @ P["W_post.%d" % t]) + P["b_post.%d" % t]
        E = p[:, :, None] * 2.0 * torch.sigmoid(y.reshape(T, k, len(v)))
        delta = sum(E[:, :, q, None] * v[q][:, None, :] for q in range(len(v)))
        if t == G - 1:
            M = torch.exp((P["alpha_res"] * r * (a @ P["W_res"]) + P["b_res"]).reshape(T, k, k))
            for _ in range(20):
                M = M / M.sum(2, keepdim=True)
                M = M / M.sum(1, keepdim=True)
            M = M / M.sum(2, keepdim=True).clamp(min=1.0)
            A = torch.einsum("tji,tic->tjc", M, A)
        A = A + delta
    return inputs, I, A


def _put_rows(X, I, A):
    return X.scatter(1, I[:, :, None].expand(*I.shape, X.shape[2]), A)


def exact(case, seed):
    if case["kind"] == "stack":
        return _exact_stack(case, seed)
    s = _inputs(case, seed)
    T, N, C, G = s["T"], case["N"], case["C"], case["G"]
    P = {n: v.to(F64).requires_grad_(case["kind"] == "train") for n, v in s["P"].items()}
    S = 1 if case["kind"] == "decode" else case["S"]
    hists = None
    if case["kind"] == "decode":
        hists = [None if r is None else _ring_history(r, s["pos"]) for r in s["rings"]]
    elif case["halo"]:
        hists = [None if h is None else h.to(F64) for h in s["halos"]]
    inputs, X_out = [torch.empty(T, C, dtype=F64, device=DEV) for _ in range(G)], torch.empty(T, N, C, dtype=F64, device=DEV)
    train = case["kind"] == "train"
    d_outs = [torch.empty(T, C, dtype=F64, device=DEV) for _ in range(G)] if train else None
    dX = torch.empty(T, N, C, dtype=F64, device=DEV) if train else None
    grads = {n: torch.zeros_like(v) for n, v in P.items()} if train else None
    # sequences do not meet but in the parameters' gradients: a few at a time
    step = max(1, min(case["B"], (1 << 28) // (N * C) // S))
    for b in range(0, case["B"], step):
        e = min(case["B"], b + step)
        r = slice(b * S, e * S)
        X = s["X"][r].to(F64).requires_grad_(train)
        outs = [o[r].to(F64).reshape(e - b, S, C).requires_grad_(train) for o in s["outs"]]
        hist = None if hists is None else [None if h is None else h[b:e] for h in hists]
        with torch.set_grad_enabled(train):
            ins, I, A = _group64(case, P, X, outs, hist)
        for t in range(G):
            inputs[t][r] = ins[t].detach()
        if not train:
            X_out[r] = _put_rows(X, I, A)
            continue
        X_out[r] = X.detach()  # the backward restores the entry state
        up = s["dX_up"][r].to(F64)
        rows = I[:, :, None].expand(*A.shape)
        loss = (A * up.gather(1, rows)).sum()
        for t in range(G):
            loss = loss + (ins[t] * s["d_inputs"][t][r].to(F64)).sum()
        names = list(P)
        got = torch.autograd.grad(loss, [X] + outs + [P[n] for n in names], allow_unused=True)
        dX[r] = got[0] + up.scatter(1, rows, 0.0)
        for t in range(G):
            d_outs[t][r] = got[1 + t].reshape(-1, C)
        for n, v in zip(names, got[1 + G:]):
            if v is not None:
                grads[n] += v
    if train:
        small = []
        for n, v in grads.items():
            if n.startswith(("alpha", "b_")):
                small.append(nn.functional.pad(v.reshape(-1), (0, -v.numel() % 4)))
        big = {n: v for n, v in grads.items() if not n.startswith(("alpha", "b_"))}
        return {"inputs": inputs, "X": X_out, "d_outs": d_outs, "dX": dX, "grads": big, "small": torch.cat(small)}
    if case["kind"] == "decode":
        R = max(CONV) - 1
        rings = [None if x is None else x.to(F64) for x in s["rings"]]
        for t, ring in enumerate(rings):
            if ring is not None:
                ring[torch.arange(T, device=DEV), s["pos"] % R] = s["outs"][t].to(F64)
        return {"inputs": inputs, "X": X_out, "rings": rings, "pos": s["pos"] + 1}
    return {"inputs": inputs, "X": X_out}


def _ring_history(ring, pos):
    """Ring [B, R, C] (row p mod R holds position p) as the R outputs before position pos, zero before
    the sequence's start."""
    B, R, C = ring.shape
    p = pos[:, None] - R + torch.arange(R, device=DEV)
    rows = ring.to(F64).gather(1, (p % R)[:, :, None].expand(B, R, C))
    return rows * (p >= 0)[:, :, None]


def _exact_stack(case, seed):
    s = _inputs(case, seed)
    T, N, C, G = s["T"], case["N"], case["C"], case["G"]
    # the parameters as the module draws them: its initialisation is part of the inputs
    grp = s["stack"].groups[0]
    hidden = s["hidden"].detach().to(F64).requires_grad_(True)
    P = {n: getattr(grp, n.replace(".", "_")).detach().to(F64).requires_grad_(True) for n in grp.names}
    gains = [f.gain.detach().to(F64).requires_grad_(True) for f in grp.sublayers]
    outs = [lambda x, w=w: (x * w).reshape(case["B"], case["S"], C) for w in gains]
    X = hidden[:, None, :].expand(T, N, C)
    _, I, A = _group64(case, P, X, outs)
    y = _put_rows(X, I, A).sum(1)
    got = torch.autograd.grad(y, [hidden] + list(P.values()) + gains, s["dy"].to(F64))
    named = {n.replace(".", "_"): v for n, v in zip(P, got[1:])}
    named.update({"sublayers.%d.gain" % t: v for t, v in enumerate(got[1 + len(P):])})
    return {"y": y.detach(), "hidden": got[0],
            "grads": _by_name({n: named[n] for n, _ in grp.named_parameters()})}
