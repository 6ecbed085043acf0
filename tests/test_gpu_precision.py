"""The input gradients whose operands the tensor cores take in three bf16 parts keep what fp32 products keep.

The active-state gradient is fp32 and stays inside the library.  A sublayer output that is zero outside one channel a
token shows it: the gradient of the slot's post-map bias is then a sum of single elements of it."""
import pytest
import torch

import xhc_cases as cases
from paper_2607_14530_gb300 import synth
from paper_2607_14530_gb300.xhc import Config, Group

pytestmark = pytest.mark.gpu

# 16 fp32 roundoffs (the term bound of the gating scalars), on the 2-norm; two bf16 parts leave about 2^-18
REL = 2.0 ** -20

CASES = {
    "C72_k4": (Config.flash(8, 4, 4, 72, 2, conv_k=()), 150),
    "C1160_k4": (Config.flash(8, 4, 4, 1160, 2, conv_k=()), 129),
    "C256_k8": (Config.flash(8, 8, 8, 256, 2, conv_k=()), 130),
    "C256_k7_conv": (Config.flash(9, 7, 7, 256, 2, seq_len=65), 130),
}


def _backward(cfg, P, inp, gin, inject):
    g = Group(cfg)
    T = inp["X"].shape[0]
    Pd = {n: v.cuda() for n, v in P.items()}
    X, dX = inp["X"].cuda(), gin["dX"].cuda()
    outs, d_in = [o.cuda() for o in inp["outs"]], [d.cuda() for d in gin["d_inputs"]]
    grads = {n: torch.zeros_like(v) for n, v in Pd.items()}
    saved, ws = g.alloc(T)
    cases.group_forward(g, cfg, Pd, X, outs, saved, ws, [torch.empty_like(o) for o in outs], inject)
    g.backward(Pd, X, dX, outs, d_in, grads, saved, ws)
    torch.cuda.synchronize()
    assert g.device_error(ws) == 0
    return dX.cpu(), {n: v.cpu() for n, v in grads.items()}, g.coefficients(saved, T)


@pytest.mark.parametrize("name", list(CASES))
def test_active_gradient_keeps_fp32_products(name):
    cfg, T = CASES[name]
    tok, ch = torch.arange(T), (torch.arange(T) * 37) % cfg.C
    err = ref2 = 0.0
    for seed in range(4):
        inp, P, s = cases.make_case(cfg, T, seed)
        gin = synth.group_grads(T, cfg.N, cfg.C, cfg.G, s)
        # at the shown channels nothing but the projection's gradient reaches the active gradient
        shown = inp["outs"][0][tok, ch].clone()
        inp["outs"][0].zero_()
        inp["outs"][0][tok, ch] = shown
        gin["dX"][tok, :, ch] = 0
        gin["d_inputs"][1][tok, ch] = 0
        ref = cases.run_oracle(cfg, inp, P, gin)
        _, grads, _ = _backward(cfg, P, inp, gin, ref["aux"])
        n = [n for n in P if n.startswith("b_post")][0]
        err += float((grads[n].to(cases.F64) - ref["dP"][n]).pow(2).sum())
        ref2 += float(ref["dP"][n].pow(2).sum())
    assert err <= REL ** 2 * ref2, f"relative error {(err / ref2) ** 0.5:.2e}"


def test_infinite_gradient_stays_infinite():
    """One active stream, and an output that overflows the gradient of its post-map: the projection's gradient is
    infinite with the sign of the weight, not NaN."""
    cfg, T, t = Config.flash(4, 1, 1, 72, 2, conv_k=()), 130, 77
    inp, P, s = cases.make_case(cfg, T, 1)
    gin = synth.group_grads(T, cfg.N, cfg.C, cfg.G, s)
    P["b_post.0"][:] = -80.0   # a map of 2^-114: the output overflows the gradient, not the state
    inp["outs"][0][t] = 0
    inp["outs"][0][t, 5] = 2.0 ** 120
    gin["dX"][t] = 0
    gin["dX"][t, 0, 5] = 2.0 ** 30
    inp["outs"][1][t] = 0
    gin["d_inputs"][1][t] = 0
    dX, _, co = _backward(cfg, P, inp, gin, None)
    row = dX[t, 0].float()
    # dz is infinite, with dX's sign at the channel; the RMS term -cx x brings an infinity of its own
    w = P["W_post.0"][:, 0]
    x = co["xact"][0][t, 0].float().cpu()
    z = float((x * w).sum())
    agree = torch.sign(w) == -torch.sign(z * x)
    assert 10 < int(agree.sum()) < cfg.C
    assert torch.equal(row[agree], torch.sign(w[agree]) * float("inf"))
    assert torch.isfinite(dX[torch.arange(T) != t].float()).all()
