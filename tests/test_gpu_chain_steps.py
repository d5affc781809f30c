"""Matched filter and demap kernels where their dispatch and their stores branch."""

import numpy as np
import pytest
import torch

import paper_2010_14333_gb300 as rx
from parity_util import Pair, make_stream

pytestmark = pytest.mark.gpu


# downshift periods in sample pairs: 40 (the default), 4 and 40 again with a longer table
# (both divide the filter's staging step of 120 pairs), 32 and 7 (which do not: the phases
# are looked up pair by pair)
@pytest.mark.parametrize("num, den", [(11, 80), (1, 8), (55, 400), (9, 64), (11, 77)])
def test_matched_filter_downshift_periods(num, den):
    nb = 65536 + 32 * 5
    g = make_stream(3, nb, 3, seed=den, fd_num=num, fd_den=den, truth=False)
    p = Pair(3, nb, ols_n=4096, ols_v=512, ntrain=4096, ncma=2048, amb_syms=1024, ds_num=num, ds_den=den)
    for b in g["packed"]:
        p.feed(b)           # matched-filter output within 1e-5 of the oracle's, then decisions and bits
    p.compare_stats()


@pytest.mark.parametrize("fmt", range(5))
def test_demap_stores_by_output_alignment(fmt):
    """Bits written in wide words (8-byte aligned pointers) and byte by byte are the same, and
    nothing is written past them, over calls whose window counts are no multiple of 64."""
    nb = 65536 + 32 * 33
    kw = dict(ols_n=4096, ols_v=512, ntrain=4096, ncma=2048, amb_syms=1024) if fmt >= 3 else dict(ntrain=4096)
    g = make_stream(fmt, nb, 3, seed=9 + fmt)
    bufs = [torch.from_numpy(b).cuda() for b in g["packed"]]
    runs = []
    for shift in (0, 1, 4):
        r = rx.Receiver(fmt, nb, **kw)
        out = torch.full((r.max_bits // 8 + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        bits = []
        for b in bufs:
            out.fill_(0xA5)
            n = rx.rx_process(r.h, b.data_ptr(), out.data_ptr() + shift, r.stream())
            got = out.cpu().numpy()
            assert n % 8 == 0 and np.all(got[:shift] == 0xA5) and np.all(got[shift + n // 8:] == 0xA5)
            bits.append(got[shift:shift + n // 8].copy())
        assert sum(len(b) for b in bits) > 0
        runs.append(np.concatenate(bits))
    assert np.array_equal(runs[0], runs[1]) and np.array_equal(runs[0], runs[2])
