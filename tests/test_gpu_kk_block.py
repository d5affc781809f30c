"""The one-kernel KK front end of 4096-point blocks at the edges of its block grid, through
the allocation-free entry point, against the overlap-save field in FP64: a window that lies
almost wholly before the stream, one whole hop, an even and an odd number of blocks (the last
pair half empty), the smallest and the largest overlap, both pack orders."""

import numpy as np
import pytest
import torch

import paper_2010_14333_gb300 as rx
import synth
from parity_util import FIELD_TOL, rel_rms

pytestmark = pytest.mark.gpu
N = 4096


def field64(codes, v):
    inten = np.maximum(codes.astype(np.float64), 0.5)
    count, hop = len(codes) - v // 2, N - v
    u = 0.5 * np.log(np.concatenate([np.full(N, inten[0]), inten]))
    h = np.zeros(N, complex)
    h[1:N // 2], h[N // 2 + 1:] = -1j, 1j
    phi, blocks = np.empty(count), -(-count // hop)
    for j in range(blocks):
        start = len(codes) - N if j == blocks - 1 else j * hop - v // 2
        p = np.fft.ifft(np.fft.fft(u[start + N:start + 2 * N]) * h).real
        lo, hi = j * hop, min((j + 1) * hop, count)
        phi[lo:hi] = p[lo - start:hi - start]
    return np.sqrt(inten[:count]) * np.exp(1j * phi)


@pytest.mark.parametrize("nsamp, v", [(320, 512), (3840, 512), (7424, 512), (11_008, 512), (4096, 4032), (50_016, 64)])
@pytest.mark.parametrize("order", [0, 1])
def test_field_of_4096_point_blocks(nsamp, v, order):
    rng = np.random.default_rng(nsamp + v + order)
    codes = np.clip(rng.normal(1500, 350, nsamp), 0, 4095).astype(np.int64)
    packed = torch.from_numpy(synth.pack12(codes, order)).cuda()
    count = nsamp - v // 2
    out = torch.full((2 * count + 2,), float("nan"), dtype=torch.float32, device="cuda")
    rx.rx_kk_field_noalloc(packed.data_ptr(), nsamp, order, N, v, out.data_ptr(),
                           torch.cuda.current_stream().cuda_stream)
    got = out.cpu().numpy()
    assert np.all(np.isnan(got[-2:]))      # nothing is written past the field
    assert rel_rms(got[:-2].view(np.complex64), field64(codes, v)) <= FIELD_TOL


@pytest.mark.parametrize("n, v, nsamp", [(4096, 512, 41_984), (65536, 4096, 131_072)])
@pytest.mark.parametrize("at", [0, 4096])
def test_field_over_its_own_input(n, v, nsamp, at):
    """A field written over the packed samples it comes from is the field of a separate buffer,
    bit for bit."""
    rng = np.random.default_rng(nsamp + at)
    packed = torch.from_numpy(synth.pack12(rng.integers(0, 4096, nsamp), 0)).cuda()
    count, stream = nsamp - v // 2, torch.cuda.current_stream().cuda_stream
    want = torch.empty(2 * count, dtype=torch.float32, device="cuda")
    rx.rx_kk_field_noalloc(packed.data_ptr(), nsamp, 0, n, v, want.data_ptr(), stream)
    both = torch.empty(2 * count, dtype=torch.float32, device="cuda")
    src = both.view(torch.uint8)[at:at + len(packed)]
    src.copy_(packed)
    rx.rx_kk_field_noalloc(src.data_ptr(), nsamp, 0, n, v, both.data_ptr(), stream)
    assert torch.equal(both, want)
