"""The FP8 block-Toeplitz FIR with one tap: a 16-symbol row reads 31 samples, so the last sample
of each group of 32 is read by no symbol and has no say in its block's scale."""

import numpy as np
import pytest

import paper_2010_14333_gb300 as rx
from test_gpu_precision import emulate, gpu_fir

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsym, sblk", [(16 * 130, 16), (2048 + 256, 256), (1 << 13, 2048)])
def test_fp8_scale_ignores_unread_samples(nsym, sblk):
    rng = np.random.default_rng(nsym)
    ny = 2 * nsym + 2
    y = (rng.standard_normal(ny) + 1j * rng.standard_normal(ny)) * 0.7
    y = y.astype(np.complex64).astype(complex)
    w = np.array([0.9 - 0.1j]).astype(np.complex64).astype(complex)
    z = gpu_fir(y, w, rx.RX_FIR_FP8, nsym, sblk)
    loud = y.copy()
    loud[31::32] *= 2.0 ** 13
    assert np.array_equal(gpu_fir(loud, w, rx.RX_FIR_FP8, nsym, sblk), z)
    # rounded operands, two exact products per part: FP32 rounding of one sum
    for k0 in range(0, nsym, sblk):     # a block's rows read 31 of every 32 samples
        seg = y[2 * k0: 2 * (k0 + sblk)].copy()
        seg[31::32] = 0
        ze = emulate(np.concatenate([seg, np.zeros(2)]), w, rx.RX_FIR_FP8, sblk, sblk)
        assert np.max(np.abs(z[k0:k0 + sblk] - ze)) <= 2.0 ** -23 * np.max(np.abs(ze)) * 2
