"""The warm-start network's kernels at sizes off their tiles: widths below, between and above the 64-wide
tiles and above the block's 256 threads, hidden sizes and point counts that are no multiple of four, one
sample, batches whose rows do not fill the splits, more modes than are staged at a time.  Against the FP64 reference network with the same
BF16-rounded weights; the tolerances of the network's own test."""
import numpy as np
import pytest

from oracle import nn as onn
from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb

from .test_gpu_nn import bf16_round, normalise, raw_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,L,H,P,B", [(8, 2, 1, 5, 9, 1), (20, 3, 2, 30, 50, 3), (64, 6, 4, 128, 256, 32), (96, 5, 2, 70, 65, 2),
                                         (33, 4, 3, 64, 64, 7), (300, 2, 1, 9, 30, 2), (1, 1, 2, 1, 8, 5), (70, 20, 2, 70, 70, 3)])
def test_sizes_off_the_tiles_match_fp64_reference(W, m, L, H, P, B):
    fbuild.build()
    kw = dict(P=P, W=W, m=m, L=L, H=H)
    lay, n = onn.layout(W, m, L, H)
    rng = np.random.default_rng(4)
    theta = np.zeros(n)
    for k, (o, s) in lay.items():
        cnt = int(np.prod(s))
        scale = 0.5 / W if k.startswith("r_") else 0.1 if len(s) == 1 else 1.0 / np.sqrt(s[0])
        theta[o:o + cnt] = bf16_round(scale * rng.uniform(-1, 1, cnt))
    raw = raw_params(B, 6)
    target = np.random.default_rng(7).normal(0, 1, (B, P, 4)).astype(np.float32)
    net = fdlb.WarmStartNet(W, m, L, H, P, max_batch=B + 1)
    net.set_params(theta.astype(np.float32))
    loss_o, grad_o, out_o = onn.loss_and_grad(theta, normalise(raw.astype(np.float64)), target.astype(np.float64), **kw)
    assert np.max(np.abs(net.forward(raw) - out_o)) <= 2e-4 * max(1.0, np.max(np.abs(out_o)))
    loss, grad = net.loss_grad(raw, target)
    assert loss == pytest.approx(loss_o, rel=1e-4)
    for k, (o, s) in lay.items():
        cnt = int(np.prod(s))
        assert np.max(np.abs(grad[o:o + cnt] - grad_o[o:o + cnt])) <= 2e-3 * max(np.max(np.abs(grad_o[o:o + cnt])), 1e-12), k
    net.close()


def test_a_narrow_network_leaves_a_wide_one_usable():
    """The kernels' shared memory limit is the function's, not the network's."""
    fbuild.build()
    wide = fdlb.WarmStartNet(512, 2, 1, 8, 16, max_batch=2)
    raw = raw_params(2, 6)
    before = wide.forward(raw)
    fdlb.WarmStartNet(8, 2, 1, 5, 9, max_batch=1).close()
    assert np.array_equal(wide.forward(raw), before)
    wide.close()
