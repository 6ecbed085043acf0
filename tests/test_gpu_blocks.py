"""GPU parity at the block and tile edges of the per-token and write-back kernels, whose block sizes
and run lengths depend on the number of tokens: remainders on both sides of each switch, against the
oracle with the bounds of the parity suite."""
import dataclasses

import pytest
import torch

import test_gpu_parity as parity
import xhc_cases as cases
from paper_2607_14530_gb300 import synth
from paper_2607_14530_gb300.xhc import Config, Group

pytestmark = pytest.mark.gpu

# m = k (nothing routed): thousands of tokens have no draw without a routing near-tie
CASES = {
    # per-token kernels: 32-token blocks (k <= 4) from 9728 tokens on a 152-SM GPU, 8 below
    "coef_k4_T9731": (Config.flash(4, 4, 4, 16, 2, seq_len=9731), 9731, {}),
    # k > 4: 16-token blocks from 4864 tokens, 4 below; three streams with rows outside the matrix
    "coef_k7_T4867": (Config.full(8, 7, 7, 16, True, seq_len=4867), 4867, {}),
    "coef_k8_T611": (Config.full(8, 8, 8, 16, False), 611, {}),
    # Sinkhorn iterates that just fit the large block, just do not, fit only the small one, and none at all
    "coef_k8_iters43": (Config.full(8, 8, 8, 8, True, sinkhorn_iters=43, seq_len=4900), 4900, {}),
    "coef_k8_iters44": (Config.full(8, 8, 8, 8, True, sinkhorn_iters=44, seq_len=4900), 4900, {}),
    "coef_k8_iters64": (Config.full(8, 8, 8, 8, True, sinkhorn_iters=64, seq_len=4900), 4900, {}),
    "coef_k3_iters0": (Config.full(5, 3, 1, 32, True, sinkhorn_iters=0), 130, {}),
    # full-state dX on few blocks: the streams of a block in parts (of 2, 3 or all streams; fixed ones in
    # the first part, none, all), ragged token tiles
    "dx_split_N16_m3": (Config.flash(16, 4, 3, 64, 2, seq_len=150), 300, {}),
    "dx_split_N12_m0": (Config.full(12, 4, 0, 128, False), 131, {}),
    "dx_split_N9": (Config.full(9, 4, 2, 128, False), 200, {}),
    "dx_split_mhc": (Config.mhc(4, 128), 129, {}),
    # three and four units a CTA, those of the fixed streams alone (no d_input rows) before, between and after
    # the others; fixed streams only; a unit with one d_input tile
    "dx_split_N9_m3_units": (Config.full(9, 3, 3, 768, False), 1659, {}),
    "dx_units_mhc": (Config.mhc(4, 768), 1659, {}),
    "dx_split_N9_m2_units": (Config.full(9, 2, 2, 768, False), 1659, {}),
    # input gradients on widths that their channel tiles do not divide: last tiles of 8, 40, 72, 8 and 72 channels,
    # one or two stages of weight rows, eight active streams, no conv
    "dx_width_C72_N20": (Config.flash(20, 4, 4, 72, 4, seq_len=100), 200, {}),
    "dx_width_C40_mhc": (Config.mhc(4, 40), 131, {}),
    "dx_width_C200_k6": (Config.flash(8, 6, 6, 200, 2, seq_len=128), 128, {}),
    "dx_width_C1160_k8": (Config.full(12, 8, 3, 1160, True), 129, {}),
    "dx_width_C584_N16": (Config.flash(16, 4, 2, 584, 4, seq_len=257), 257, {}),
    # entry rows put back by the two-pair reductions (512-channel slices): a run that ends inside a block of 4
    "put_back_C1024": (Config.full(16, 4, 4, 1024, True, seq_len=67), 134, {}),
    # two components (a Gram-Schmidt basis smaller than its maximum), N with idle lanes
    "coef_N27_conv1": (Config.flash(27, 4, 2, 64, 2, conv_k=(4,), seq_len=131), 262, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_block_edges(name, monkeypatch):
    monkeypatch.setitem(parity.CASES, name, CASES[name])
    parity.test_forward_backward_parity(name)


# decode: batches at the switches of the projection for few tokens (1, 2, 4, 8, 16 tokens a block, the
# tensor cores from 128) and of the write-back's tokens per cluster; N and k with widths that are not a
# multiple of 4 (one column a load); slices that fill no whole CTA; other tap sets; positions below R
DECODE = {
    "B1": (Config.flash(16, 4, 2, 520, 4), 1, 3, False),
    "B3_N6": (Config.flash(6, 3, 1, 264, 2, conv_k=(2, 5)), 3, 40, False),
    "B9_k8": (Config.full(12, 8, 3, 776, True), 9, 15, False),
    "B17_no_gs": (Config.full(8, 4, 2, 64, True, gram_schmidt=False), 17, 11, False),
    # no conv in the last slot, several CTAs a token: pos is read and advanced by the first alone
    "B5_attn_wide": (Config.full(8, 4, 2, 2312, False), 5, 4, False),
    "B31_attn": (Config.full(8, 4, 2, 72, False), 31, 4, False),
    "B127": (Config.flash(8, 4, 2, 2312, 2, conv_k=(16,)), 127, 20, True),
    "B130": (Config.flash(8, 4, 2, 1024, 2), 130, 20, True),
}


@pytest.mark.parametrize("name", list(DECODE))
def test_decode_sizes(name):
    """One decoded token per sequence (positions S, S + 1, ...) against the forward of a sequence that
    ends there: the ring holds the outputs before it."""
    cfg, B, S, spread = DECODE[name]
    dev = torch.device("cuda", 0)
    R = max(cfg.conv_k) - 1
    # the oracle's sequences: the R history rows (their own states do not matter) and the new token
    seq = dataclasses.replace(cfg, seq_len=R + 1)
    for seed in range(5, 50):
        inp = synth.group_inputs(B * (R + 1), cfg.N, cfg.C, cfg.G, seed)
        P = synth.params(cfg.param_shapes(), seed)
        new = torch.arange(B) * (R + 1) + R
        if not cfg.has_router or bool(cases.tie_free(cfg, inp["X"][new], P["W_r"]).all()):
            break
    pos = S + (torch.arange(B) if spread else torch.zeros(B, dtype=torch.int64))
    for o in inp["outs"]:   # nothing before the start of a sequence shorter than the history
        v = o.view(B, R + 1, cfg.C)
        for b in range(B):
            v[b, :max(0, R - int(pos[b]))] = 0
    ref = cases.run_oracle(seq, inp, P)
    g = Group(cfg)
    saved, ws = g.alloc(B)
    rings = g.alloc_rings(B)
    for t, ring in enumerate(rings):
        if ring is None:
            continue
        r = ring.view(torch.bfloat16).view(B, R, cfg.C)
        r.fill_(float("nan"))   # rows that the conv must not read
        for b in range(B):
            for i in range(1, min(R, int(pos[b])) + 1):
                r[b, (int(pos[b]) - i) % R] = inp["outs"][t].view(B, R + 1, cfg.C)[b, R - i].to(dev)
    X = inp["X"][new].to(dev).contiguous()
    outs = [o[new].to(dev).contiguous() for o in inp["outs"]]
    dpos = pos.to(dev)
    ins = g.forward_decode({n: v.to(dev) for n, v in P.items()}, X, outs, rings, dpos, saved, ws)
    torch.cuda.synchronize()
    co = g.coefficients(saved, B)
    assert torch.equal(co["I"].cpu().long(), ref["aux"]["I"][new])
    bases = cases.flash_bases(cfg, inp["X"], ref["aux"])
    for t in range(cfg.G):
        cases.assert_bf16_close(ins[t], ref["inputs"][t][new], f"input[{t}]",
                                None if bases[t] is None else bases[t][new])
        cases.assert_f32_close(co["hpost"][t], ref["aux"]["H_post"][t][new], f"H_post[{t}]")
        if rings[t] is not None:
            r = rings[t].view(torch.bfloat16).view(B, R, cfg.C)
            assert torch.equal(r[torch.arange(B), (pos % R).to(dev)], outs[t])
    cases.assert_bf16_close(X, ref["X"][new], "X")
    assert torch.equal(dpos.cpu(), pos + 1)
    assert g.device_error(ws) == 0


def test_captured_step_equals_the_eager_one():
    """A forward and backward captured as a CUDA graph (no programmatic launches, the side stream forked
    and joined inside) gives the eager call's bits."""
    cfg, T = Config.flash(8, 4, 2, 512, 4, seq_len=150), 300
    inp, P, seed = cases.make_case(cfg, T, 1)
    gin = synth.group_grads(T, cfg.N, cfg.C, cfg.G, seed)
    g = Group(cfg)
    Pd = {n: v.cuda() for n, v in P.items()}
    X, X0 = inp["X"].cuda(), inp["X"].cuda()
    outs, d_in = [o.cuda() for o in inp["outs"]], [d.cuda() for d in gin["d_inputs"]]
    dX0 = gin["dX"].cuda()
    dX = torch.empty_like(dX0)
    gr = {n: torch.zeros_like(v) for n, v in Pd.items()}
    rows = [torch.empty(T, cfg.C, dtype=torch.bfloat16, device="cuda") for _ in range(2 * cfg.G)]
    saved, ws = g.alloc(T)

    def step():
        X.copy_(X0)
        dX.copy_(dX0)
        for v in gr.values():
            v.zero_()
        g.forward(Pd, X, outs, saved, ws, inputs=rows[:cfg.G])
        g.backward(Pd, X, dX, outs, d_in, gr, saved, ws, d_outs=rows[cfg.G:])

    step()
    torch.cuda.synchronize()
    want = [t.clone() for t in rows + [dX] + list(gr.values())]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(want, rows + [dX] + list(gr.values())):
        assert torch.equal(a, b)
    assert g.device_error(ws) == 0
