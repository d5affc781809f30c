"""Learned equaliser kernels at the edges of their launch shapes, against the FP64 oracle:
one segment, a few, and one more than the persistent forward grid holds (three CTAs per SM,
so that a CTA takes a second segment), with segment starts of either parity."""

import numpy as np
import pytest
import torch

import oracle
import paper_2010_14333_gb300 as rx
from paper_2010_14333_gb300 import cnn
from test_gpu_cnn import L0, S, gpu_grad

pytestmark = pytest.mark.gpu

# BF16 operands: weights and the three layers' activations carry a relative rounding of
# 2^-9 each; a handful of them in quadrature stays below 1e-2, doubled for the worst tensor
TOL = 2e-2


@pytest.mark.parametrize("nseg", [1, 5, 0])
def test_forward_and_gradient_at_grid_edges(nseg):
    nseg = nseg or 3 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    rng = np.random.default_rng(40 + nseg)
    params = cnn.init_params(4).astype(np.float64) + rng.standard_normal(rx.rx_cnn_nparams()) * 0.01
    y = (rng.standard_normal(6000) + 1j * rng.standard_normal(6000)) * 0.7
    seg = rng.integers(0, len(y) - L0, size=nseg)
    seg[0], seg[-1] = 0, len(y) - L0        # the first and the last samples of the input
    tgt = rng.standard_normal((nseg, S, 2)) * 0.7
    x = np.stack([np.stack([y[s:s + L0].real, y[s:s + L0].imag], axis=1) for s in seg])
    params = params.astype(np.float32)
    lo, go, oo = oracle.cnn_loss_grad(params, x, tgt)
    g, lg, og = gpu_grad(params, y, seg, tgt)
    assert np.linalg.norm(og - oo) < TOL * np.linalg.norm(oo)
    for s in (0, nseg // 2, nseg - 1):      # no segment is swapped or left out
        assert np.linalg.norm(og[s] - oo[s]) < 2 * TOL * np.linalg.norm(oo[s])
    assert abs(lg - lo) < TOL * lo
    assert np.linalg.norm(g - go) < TOL * np.linalg.norm(go)
