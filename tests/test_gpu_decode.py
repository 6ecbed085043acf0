"""GPU parity of decoding (one new token per sequence, conv history in per-sequence rings).

B sequences are prefilled with S tokens through the ordinary forward, the rings are filled from
the prefill's sublayer outputs, then ND tokens are decoded one at a time.  The oracle runs the
plain forward on the whole sequences of S + ND tokens: every decoded token must give the oracle's
sublayer inputs, coefficients and new state rows at its position (tokens interact only through
the causal conv, whose history the rings carry).  S below max(kappa) - 1 exercises the zero
padding before the sequence start."""
import pytest
import torch

from paper_2607_14530_gb300 import synth
from paper_2607_14530_gb300.xhc import Config, Group

from xhc_cases import assert_bf16_close, assert_f32_close, flash_bases, run_oracle, tie_free

pytestmark = pytest.mark.gpu

ND = 3


def _cfg(N, k, m, C, G, S, **kw):
    if G == 1:
        return Config.full(N, k, m, C, True, seq_len=S, **kw)
    return Config.flash(N, k, m, C, G, seq_len=S, **kw)


@pytest.mark.parametrize("N,k,m,C,G,B,S", [
    (16, 4, 2, 256, 4, 3, 20),    # Flash-4sub, prefill longer than the ring
    (16, 4, 2, 256, 4, 2, 5),     # prefill shorter than the ring: zero padding
    (8, 4, 2, 128, 1, 4, 13),     # one full-xHC MLP sublayer
])
def test_decode_matches_the_whole_sequence_forward(N, k, m, C, G, B, S):
    L = S + ND
    cfg_o = _cfg(N, k, m, C, G, L)
    # seeded whole sequences without a routing near-tie (the oracle decides)
    for attempt in range(50):
        seed = 7 + 1000 * attempt
        inp = synth.group_inputs(B * L, N, C, G, seed)
        P = synth.params(cfg_o.param_shapes(), seed)
        if bool(tie_free(cfg_o, inp["X"], P["W_r"]).all()):
            break
    else:
        raise RuntimeError("no tie-free draw")
    ref = run_oracle(cfg_o, inp, P)
    aux = ref["aux"]
    bases = flash_bases(cfg_o, inp["X"], aux)

    pre_rows = torch.cat([torch.arange(b * L, b * L + S) for b in range(B)])

    def rows_at(p):
        return torch.tensor([b * L + p for b in range(B)])

    dev = torch.device("cuda", 0)
    Pd = {n: v.to(dev) for n, v in P.items()}
    # prefill: B sequences of S tokens
    gp = Group(_cfg(N, k, m, C, G, S))
    Xp = inp["X"][pre_rows].to(dev).contiguous()
    outs_p = [o[pre_rows].to(dev).contiguous() for o in inp["outs"]]
    saved, ws = gp.alloc(B * S)
    gp.forward(Pd, Xp, outs_p, saved, ws)
    rings = gp.alloc_rings(B)
    for t in range(G):
        if rings[t] is not None:
            gp.ring_fill(B, S, outs_p[t], rings[t])
    pos = torch.full((B,), S, dtype=torch.int64, device=dev)

    # decode ND tokens
    gd = Group(_cfg(N, k, m, C, G, 0))
    saved_d, ws_d = gd.alloc(B)
    errors = []

    def chk(fn, *a):
        try:
            fn(*a)
        except AssertionError as e:
            errors.append(str(e).split("\n")[0])

    for n in range(ND):
        r = rows_at(S + n)
        X = inp["X"][r].to(dev).contiguous()
        outs = [o[r].to(dev).contiguous() for o in inp["outs"]]
        ins = gd.forward_decode(Pd, X, outs, rings, pos, saved_d, ws_d)
        torch.cuda.synchronize()
        co = gd.coefficients(saved_d, B)
        tag = f"token {S + n}"
        if not torch.equal(co["I"].cpu().long(), aux["I"][r]):
            errors.append(f"{tag}: routing differs")
        for t in range(G):
            chk(assert_bf16_close, ins[t], ref["inputs"][t][r], f"{tag} input[{t}]",
                None if bases[t] is None else bases[t][r])
            chk(assert_f32_close, co["hpost"][t].cpu(), aux["H_post"][t][r], f"{tag} H_post[{t}]")
        chk(assert_f32_close, co["hres"].cpu(), aux["H_res"][r], f"{tag} H_res")
        chk(assert_bf16_close, X, ref["X"][r], f"{tag} X_out")
    assert gd.device_error(ws_d) == 0
    assert torch.equal(pos.cpu(), torch.full((B,), S + ND, dtype=torch.int64)), "pos not advanced"
    assert not errors, "\n".join(errors)


@pytest.mark.parametrize("cfg", [Config.flash(16, 4, 2, 1024, 4), Config.full(12, 8, 3, 264, True)], ids=["flash4", "k8"])
def test_batches_below_a_tile_have_the_same_bits(cfg):
    """A token decoded in a batch of any size below 128 (the tensor cores' tile) has the same routing,
    coefficients, sublayer inputs and state, bit by bit, as alone: batches on both sides of the sizes at which
    the projection takes more tokens a block or more blocks."""
    dev = torch.device("cuda", 0)
    n = 127
    inp = synth.group_inputs(n, cfg.N, cfg.C, cfg.G, 3)
    P = {k: v.to(dev) for k, v in synth.params(cfg.param_shapes(), 3).items()}
    g = Group(cfg)
    R = max(cfg.conv_k) - 1
    hist = [synth.normal_bf16((n, R, cfg.C), 17 + t).to(dev) for t in range(cfg.G)]

    def decode(rows):
        B = len(rows)
        X = inp["X"][rows].to(dev)
        outs = [o[rows].to(dev) for o in inp["outs"]]
        rings = g.alloc_rings(B)
        for t, r in enumerate(rings):
            if r is not None:
                r.view(torch.bfloat16).view(B, R, cfg.C).copy_(hist[t][rows])
        saved, ws = g.alloc(B)
        pos = torch.full((B,), 40, dtype=torch.int64, device=dev)
        ins = g.forward_decode(P, X, outs, rings, pos, saved, ws)
        co = g.coefficients(saved, B)
        return [X, *ins, *(co[k] for k in ("zfull", "stats", "I", "p", "hpre", "hres")), *co["hpost"]]

    whole = decode(list(range(n)))
    for first, B in ((0, 1), (126, 1), (3, 2), (5, 9), (0, 16), (40, 17), (1, 33), (20, 64), (9, 100)):
        for a, b in zip(decode(list(range(first, first + B))), whole):
            assert torch.equal(a, b[first:first + B]), (first, B)
