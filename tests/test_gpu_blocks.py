"""GPU parity at the block and tile edges of the per-token and write-back kernels, whose block sizes
and run lengths depend on the number of tokens: remainders on both sides of each switch, against the
oracle with the bounds of the parity suite."""
import pytest

import test_gpu_parity as parity
from paper_2607_14530_gb300.xhc import Config

pytestmark = pytest.mark.gpu

# m = k (nothing routed): thousands of tokens have no draw without a routing near-tie
CASES = {
    # per-token kernels: 32-token blocks (k <= 4) from 9728 tokens on a 152-SM GPU, 8 below
    "coef_k4_T9731": (Config.flash(4, 4, 4, 16, 2, seq_len=9731), 9731, {}),
    # k > 4: 16-token blocks from 4864 tokens, 4 below; three streams with rows outside the matrix
    "coef_k7_T4867": (Config.full(8, 7, 7, 16, True, seq_len=4867), 4867, {}),
    "coef_k8_T611": (Config.full(8, 8, 8, 16, False), 611, {}),
    # Sinkhorn iterates that fit only the small block, and none at all
    "coef_k8_iters64": (Config.full(8, 8, 8, 8, True, sinkhorn_iters=64, seq_len=4900), 4900, {}),
    "coef_k3_iters0": (Config.full(5, 3, 1, 32, True, sinkhorn_iters=0), 130, {}),
    # two conv components (a Gram-Schmidt basis smaller than its maximum), N with idle lanes
    "coef_N27_conv1": (Config.flash(27, 4, 2, 64, 2, conv_k=(4,), seq_len=131), 262, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_block_edges(name, monkeypatch):
    monkeypatch.setitem(parity.CASES, name, CASES[name])
    parity.test_forward_backward_parity(name)
