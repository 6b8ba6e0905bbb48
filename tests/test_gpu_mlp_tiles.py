"""The network's kernels at the edges of their tiles: 128 samples per cluster
(one short, full, one over, several clusters) and 256 samples per staged
chunk of the weight gradients (one over, a third chunk that reuses the first
buffer).  Against the FP64 oracle network, with test_gpu_mlp's bar for BF16
operands (relative L2 1e-2 per layer)."""
import numpy as np
import pytest

import oracle.mlp as M
from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import rel_l2, stream

pytestmark = pytest.mark.gpu

TOL = 1e-2


@pytest.mark.parametrize("S", [1, 127, 128, 129, 257, 600])
def test_forward_loss_and_gradient_at_tile_edges(S):
    p = I.mlp_init(3)
    x = I.warmstart_cases(S, S)
    y = 1.0 + 0.1 * np.random.default_rng(S).normal(size=(S, 64))
    m = iblb.iblb_mlp_create(p, S, stream())
    try:
        out = iblb.iblb_mlp_predict(m, x)
        g, loss = iblb.iblb_mlp_grad(m, x, y)
    finally:
        iblb.iblb_mlp_destroy(m)
    p64 = p.astype(np.float64)
    want, _ = M.forward(p64, x)
    assert rel_l2(out - 1.0, want - 1.0) < TOL
    assert abs(loss / M.loss(p64, x, y) - 1.0) < TOL
    go, at = M.grad(p64, x, y), 0
    for i, o in ((3, 256), (256, 256), (256, 256), (256, 64)):
        for n in (i * o, o):
            assert rel_l2(g[at:at + n], go[at:at + n]) < TOL, (i, o, n)
            at += n
