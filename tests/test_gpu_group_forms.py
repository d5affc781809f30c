"""Receiver forms whose chains mix kernels launched as dependents with memsets, plain
launches and events (frozen and tensor-core equalisers, static filter with clock tracking,
resampler, symbol-by-symbol equaliser, learned equaliser, both transform lengths), in a
group round, plain and captured, and in a captured batch: the same bits, bit counts and
counters as each stream run call by call."""

import numpy as np
import pytest
import torch

import paper_2010_14333_gb300 as rx
from paper_2010_14333_gb300 import cnn
from parity_util import make_stream
from test_gpu_group import COUNTERS

pytestmark = pytest.mark.gpu

NB, ROUNDS = 1 << 17, 4
KK = dict(ntrain=4096, ncma=2048, amb_syms=1024)
SHORT = dict(KK, ols_n=4096, ols_v=512)
STEP = (1 << 32) + 40_000
FORMS = {
    "frozen": (4, dict(SHORT, fir_prec=rx.RX_FIR_FROZEN_F32)),
    "bf16": (4, dict(SHORT, fir_prec=rx.RX_FIR_BF16, eq_block=1024)),
    "fp8": (3, dict(SHORT, fir_prec=rx.RX_FIR_FP8, eq_block=1024)),
    "static filter": (4, dict(SHORT, mf_mode=rx.RX_MF_FD)),
    "clock tracking": (4, dict(SHORT, mf_mode=rx.RX_MF_FD, clk_track=1, rs_step=STEP)),
    "resampler": (3, dict(KK, rs_step=STEP)),
    "symbol by symbol": (4, dict(KK, eq_mode=rx.RX_EQ_DD_SYMBOL, ntaps=4)),
    "differential": (3, dict(SHORT, diff_code=1)),
    "learned": (4, KK),
    "cluster": (4, dict(KK, kk_front=1)),
    "pam": (1, dict(ntrain=4096)),
    "pam resampler": (2, dict(ntrain=4096, rs_step=STEP)),
    "pam static filter": (0, dict(ntrain=4096, mf_mode=rx.RX_MF_FD, clk_track=1)),
    "pam span": (1, dict(ntrain=4096, mf_span=8)),
}


@pytest.fixture(scope="module")
def streams():
    return {f: [torch.from_numpy(b).cuda() for b in make_stream(f, NB, ROUNDS, seed=70 + f)["packed"]] for f in range(5)}


@pytest.fixture(scope="module")
def network():
    h = rx.rx_cnn_create(1)
    rx.rx_cnn_set_params(h, cnn.init_params(5))
    yield h
    rx.rx_cnn_destroy(h)


def receiver(name, network):
    fmt, kw = FORMS[name]
    r = rx.Receiver(fmt, NB, **kw)
    if name == "learned":
        rx.rx_set_cnn(r.h, network)
    return r


def one_by_one(name, streams, network):
    r = receiver(name, network)
    bits = []
    for p in streams[FORMS[name][0]]:
        b, _ = r.process(p)
        bits.append(b.cpu().numpy().copy())
    return bits, r.stats()


def outputs(r, count):
    return [torch.zeros(r.max_bits // 8 + 16, dtype=torch.uint8, device="cuda") for _ in range(count)]


def same(bits, stats, want, swant, name):
    assert sum(len(b) for b in want) > 0
    for k in range(ROUNDS):
        assert np.array_equal(bits[k], want[k]), (name, k)
    for c in COUNTERS:
        assert stats[c] == swant[c], (name, c)


@pytest.mark.parametrize("flags", [0, rx.RX_GROUP_GRAPH])
def test_group_of_forms(streams, network, flags):
    recv = {n: receiver(n, network) for n in FORMS}
    outs = {n: outputs(r, 1)[0] for n, r in recv.items()}
    got = {n: [] for n in FORMS}
    g = rx.rx_group_create([r.h for r in recv.values()], flags)
    try:
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        for k in range(ROUNDS):
            ns = rx.rx_group_process(g, [streams[FORMS[n][0]][k].data_ptr() for n in FORMS],
                                     [o.data_ptr() for o in outs.values()], st.cuda_stream)
            st.synchronize()
            for n, bits in zip(FORMS, ns):
                got[n].append(outs[n][: (bits + 7) // 8].cpu().numpy().copy())
    finally:
        rx.rx_group_destroy(g)
    for n, r in recv.items():
        same(got[n], r.stats(), *one_by_one(n, streams, network), n)


@pytest.mark.parametrize("name", ["pam", "pam resampler", "pam span", "frozen", "static filter", "resampler"])
def test_captured_batch(streams, network, name):
    r = receiver(name, network)
    outs, st, graph = outputs(r, ROUNDS), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st, capture_error_mode="thread_local"):
        ns = rx.rx_process_batch(r.h, [p.data_ptr() for p in streams[FORMS[name][0]]], [o.data_ptr() for o in outs],
                                 st.cuda_stream)
    graph.replay()
    torch.cuda.synchronize()
    bits = [o[: (n + 7) // 8].cpu().numpy().copy() for o, n in zip(outs, ns)]
    same(bits, r.stats(), *one_by_one(name, streams, network), name)
