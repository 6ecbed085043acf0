"""Two host threads, each with a stream and buffers of its own, on calls of different sizes: the same kernels are
launched with different amounts of shared memory, and every call has to go through with its own results."""
import threading

import pytest
import torch

import xhc_cases as cases
from paper_2607_14530_gb300 import synth
from paper_2607_14530_gb300.xhc import Config, Group

pytestmark = pytest.mark.gpu

# the write-back reductions' runs of tokens and the projections' operand rings differ
SIZES = [(Config.flash(16, 4, 4, 512, 4, seq_len=300), 300), (Config.flash(8, 4, 4, 512, 4, seq_len=1400), 1400)]
STEPS = 2000


class Worker:
    def __init__(self, cfg, T):
        self.cfg, self.g = cfg, Group(cfg)
        inp, P, seed = cases.make_case(cfg, T, 1)
        gin = synth.group_grads(T, cfg.N, cfg.C, cfg.G, seed)
        self.P = {n: v.cuda() for n, v in P.items()}
        self.grads = {n: torch.zeros_like(v) for n, v in self.P.items()}
        self.pp, self.gg = self.g.params(self.P), self.g.params(self.grads)
        self.X0, self.dX0 = inp["X"].cuda(), gin["dX"].cuda()
        self.X, self.dX = torch.empty_like(self.X0), torch.empty_like(self.dX0)
        self.outs, self.d_in = [o.cuda() for o in inp["outs"]], [d.cuda() for d in gin["d_inputs"]]
        self.ins, self.d_outs = [[torch.empty_like(o) for o in self.outs] for _ in range(2)]
        self.saved, self.ws = self.g.alloc(T)
        self.stream = torch.cuda.Stream()
        self.error = None
        torch.cuda.synchronize()

    def step(self):
        """Forward and backward with as little as possible on the host around the calls."""
        g, X, dX, s, w, st = self.g, self.X, self.dX, self.saved, self.ws, self.stream
        X.copy_(self.X0)
        dX.copy_(self.dX0)
        torch._foreach_zero_(list(self.grads.values()))
        for t in range(self.cfg.G):
            g.pre_fwd(t, self.pp, X, self.ins[t], s, w, st)
            g.post_fwd(t, self.pp, X, self.outs[t], s, w, st)
        for t in reversed(range(self.cfg.G)):
            g.post_bwd(t, self.pp, X, dX, self.outs[t], self.d_outs[t], self.gg, s, w, st)
            g.pre_bwd(t, self.pp, X, self.d_in[t], dX, self.gg, s, w, st)

    def results(self):
        self.stream.synchronize()
        return self.ins + self.d_outs + [self.X, self.dX] + list(self.grads.values())

    def run(self, want):
        try:
            with torch.cuda.stream(self.stream):
                for _ in range(STEPS):
                    self.step()
                assert all(torch.equal(a, b) for a, b in zip(self.results(), want))
        except Exception as e:   # handed to the test's thread
            self.error = e


def test_two_threads_of_different_sizes():
    workers = [Worker(cfg, T) for cfg, T in SIZES]
    wants = []
    for w in workers:
        with torch.cuda.stream(w.stream):
            w.step()
            wants.append([r.clone() for r in w.results()])
        w.stream.synchronize()
    threads = [threading.Thread(target=w.run, args=(want,)) for w, want in zip(workers, wants)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for w in workers:
        if w.error is not None:
            raise w.error
        assert w.g.device_error(w.ws) == 0
