"""Wide networks: the modes' mixing over several column tiles and more samples than a block takes at a time, widths
off the vector loads, many row tiles, against the FP64 reference network (the tolerances of the network's own
test); and the forward pass of a wide network with many modes at a tenth of the device's FP32 rate at least."""
import time

import numpy as np
import pytest

from oracle import nn as onn
from paper_2403_15051_gb300 import build as fbuild
from paper_2403_15051_gb300 import fdlb

from .test_gpu_nn import bf16_round, normalise, raw_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()


@pytest.mark.parametrize("W,m,L,H,P,B", [(130, 3, 2, 20, 200, 9), (512, 5, 1, 70, 64, 17), (200, 17, 1, 68, 130, 3),
                                         (36, 33, 2, 12, 1000, 1), (129, 2, 1, 64, 65, 8)])
def test_wide_sizes_match_fp64_reference(W, m, L, H, P, B):
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


def test_a_wide_network_runs_at_the_arithmetic_rate():
    # 0.7 ms at the FP32 rate for two layers of 512 channels, 32 modes, 8 row tiles, 64 samples; the mixing repeated
    # by every row tile took it to a twenty-eighth of the rate
    W, m, L, H, P, B = 512, 32, 2, 64, 512, 64
    net = fdlb.WarmStartNet(W, m, L, H, P, max_batch=B)
    net.init_params(1)
    raw = raw_params(B, 6)
    best = 1e9
    for _ in range(6):
        t = time.perf_counter()
        net.forward(raw)
        best = min(best, time.perf_counter() - t)
    net.close()
    flops = 2.0 * B * P * (6 * W + L * W * W + W * H + 4 * H) + L * (2 * 2.0 * B * 2 * m * W * P + 8.0 * B * m * W * W)
    assert flops / best > 0.1 * 1e12 * fdlb.fp32_fma_peak()[0]


def test_a_wide_networks_workspace_is_its_activations_and_parameters():
    # the activations of the passes, four parameter vectors and the BF16 copy; the rest (bases, spectral
    # coefficients, the splits of the weight gradients) a few dozen megabytes
    torch = pytest.importorskip("torch")
    W, m, L, H, P, B = 512, 2, 16, 512, 256, 64
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net = fdlb.WarmStartNet(W, m, L, H, P, max_batch=B)
    used = free - torch.cuda.mem_get_info()[0]
    lay, n = onn.layout(W, m, L, H)
    need = 18 * n + 4 * B * P * ((2 * L + 2) * W + 3 * H + 3 * 4 + 6)
    net.close()
    assert used <= need + (128 << 20)
