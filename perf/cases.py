"""Measured cases: the work that a program using the receiver library has it do.

Each case is one call (or the calls that belong together) through the public entry
points of ``paper_2010_14333_gb300``, on synthetic input of the kind the receiver meets:
12-bit intensity samples of a Kramers-Kronig QAM signal or of a direct-detection PAM
signal with noise, or the 2-sps samples that the equalisers see.  Kinds:

field        Kramers-Kronig field of one buffer (rx_kk_field_noalloc)
fir          block-Toeplitz FIR of the equaliser on the tensor cores (rx_fir_block)
cnn_forward  soft symbols of the learned equaliser (rx_cnn_forward)
cnn_train    one training step of the learned equaliser (rx_cnn_grad, rx_cnn_adam_step)
buffer       one buffer of a stream that a receiver follows (Receiver.process)
batch        consecutive buffers of a stream in one call (Receiver.process_batch)
host         the same from and to page-locked host memory (rx_process_host_batch)
group        one buffer of each of many streams (rx_group_process)

A receiver's program keeps its handle from buffer to buffer, so ``prepare`` makes the
handle and lets it take the stream's first buffers (its training); every pass is the
next buffers of that stream, which come round from a ring of distinct ones.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2010_14333_gb300 as rx
from paper_2010_14333_gb300 import cnn as rx_cnn_module

SEG = 64                                      # symbols per segment of the learned equaliser
BITS = {0: 1, 1: 2, 2: 3, 3: 2, 4: 4}         # per symbol and format: PAM-2/4/8, KK-QPSK, KK-16QAM


# --------------------------------------------------------------------- the cases
def listed():
    return [
        # a short capture with the 4096-point overlap-save transform: the smallest call,
        # for a caller that may not allocate (bound by launches)
        {"name": "field_small", "kind": "field", "nsamp": 41_984, "ols_n": 4096, "ols_v": 512, "pack_order": 0},
        # the largest buffer that entry point takes, with the workload's 2^16-point transform
        {"name": "field_large", "kind": "field", "nsamp": 1 << 19, "ols_n": 65536, "ols_v": 4096, "pack_order": 0},
        # the precision sweep's equaliser filter, one 2^22-sample buffer's symbols in BF16
        {"name": "fir_bf16", "kind": "fir", "prec": rx.RX_FIR_BF16, "nsym": 1 << 20, "ntaps": 31, "scale_block": 1024},
        # the same in FP8 with a scale per equaliser block, a ragged number of blocks
        {"name": "fir_fp8", "kind": "fir", "prec": rx.RX_FIR_FP8, "nsym": 777 * 1024, "ntaps": 31, "scale_block": 1024},
        # judging a trained learned equaliser on 2^18 symbols
        {"name": "cnn_forward", "kind": "cnn_forward", "nseg": 4096},
        # its training step: 64 segments of 64 symbols, gradient and Adam
        {"name": "cnn_train", "kind": "cnn_train", "nseg": 64},
        # the paper's buffer, one at a time: latency against the real-time budget
        {"name": "kk16qam_buffer", "kind": "buffer", "fmt": 4, "buf_len": 1 << 22, "ring": 4, "pack_order": 0,
         "ols_n": 65536, "ols_v": 4096, "fd": False},
        # the headline: consecutive 2^22-sample buffers in the pipelined call
        {"name": "kk16qam_batch", "kind": "batch", "fmt": 4, "buf_len": 1 << 22, "bufs": 16, "pack_order": 0,
         "ols_n": 65536, "ols_v": 4096, "fd": False, "cnn": False},
        # the receiver deciding through the learned equaliser
        {"name": "kk16qam_cnn", "kind": "batch", "fmt": 4, "buf_len": 1 << 22, "bufs": 4, "pack_order": 0,
         "ols_n": 65536, "ols_v": 4096, "fd": False, "cnn": True},
        # short ragged QPSK buffers end to end from host memory, in the paper's frequency-domain
        # form of the filter, big-endian ADC words
        {"name": "kkqpsk_fd_host", "kind": "host", "fmt": 3, "buf_len": 266_272, "bufs": 8, "pack_order": 1,
         "ols_n": 4096, "ols_v": 512, "fd": True, "cnn": False},
        # direct detection: the PAM-4 workload's 2^20-sample buffer
        {"name": "pam4_buffer", "kind": "buffer", "fmt": 1, "buf_len": 1 << 20, "ring": 4, "pack_order": 0,
         "ols_n": 0, "ols_v": 0, "fd": False},
        # 64 streams of mixed formats and buffer lengths in one captured round
        {"name": "group_64", "kind": "group", "members": 64, "log2_lo": 18, "log2_hi": 22, "ragged": False,
         "mix_seed": 2022, "graph": True},
    ]


def _log_uniform(rng, lo, hi, unit):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, unit * int(round(v / unit))))


def _receiver_options(rng, fmt, c):
    c["fmt"], c["pack_order"], c["fd"] = fmt, rng.randint(0, 1), rng.random() < 0.3
    if fmt >= 3 and rng.random() < 0.35:
        c["ols_n"], c["ols_v"] = 4096, 64 * rng.randint(4, 16)
    else:
        c["ols_n"], c["ols_v"] = (65536, 64 * rng.randint(16, 64)) if fmt >= 3 else (0, 0)
    return c


def draw(rng):
    kind = rng.choice(["field", "fir", "cnn_forward", "cnn_train", "buffer", "buffer", "batch", "batch", "host", "group"])
    if kind == "field":
        n = rng.choice([4096, 65536])
        return {"kind": kind, "nsamp": _log_uniform(rng, 1 << 15, 1 << 19, 32), "ols_n": n,
                "ols_v": 64 * (rng.randint(2, 16) if n == 4096 else rng.randint(16, 64)), "pack_order": rng.randint(0, 1)}
    if kind == "fir":
        block = 16 << rng.randint(2, 7)
        return {"kind": kind, "prec": rng.choice([rx.RX_FIR_BF16, rx.RX_FIR_FP16, rx.RX_FIR_FP8]),
                "nsym": _log_uniform(rng, 1 << 15, 1 << 21, block), "ntaps": rng.choice([7, 15, 23, 31]),
                "scale_block": block}
    if kind == "cnn_forward":
        return {"kind": kind, "nseg": _log_uniform(rng, 64, 4096, 1)}
    if kind == "cnn_train":
        return {"kind": kind, "nseg": _log_uniform(rng, 16, 512, 1)}
    if kind == "group":
        return {"kind": kind, "members": rng.randint(4, 40), "log2_lo": 18, "log2_hi": 22, "ragged": True,
                "mix_seed": rng.randint(1, 1 << 20), "graph": rng.random() < 0.5}
    fmt = rng.randint(0, 4)
    c = {"kind": kind, "buf_len": _log_uniform(rng, 1 << 17, 1 << 22, 32)}
    if kind == "buffer":
        c["ring"] = 4
    else:
        c["bufs"] = max(2, min(16, (1 << 25) // c["buf_len"]))
        c["cnn"] = fmt >= 3 and rng.random() < 0.25
    return _receiver_options(rng, fmt, c)


# ------------------------------------------------------------------------- inputs
def _prbs15(seed, count):
    """PRBS-15 bits (x^15 + x^14 + 1) as the receiver's BER reference has them for prbs_seed = seed."""
    r, period = seed % 32767 + 1, np.empty(32767, np.int64)
    for i in range(32767):
        b = ((r >> 13) ^ (r >> 14)) & 1
        r = ((r << 1) | b) & 0x7FFF
        period[i] = b
    return period[np.arange(count) % 32767]


def _levels(bits, nb):
    """Odd-integer levels of MSB-first Gray words of nb bits."""
    g = np.zeros(len(bits) // nb, np.int64)
    for i in range(nb):
        g = 2 * g + bits[i::nb]
    level = g.copy()
    for s in range(1, nb):
        level ^= g >> s
    return 2 * level - ((1 << nb) - 1)


def _rrc(sps, span, beta=0.1):
    t = np.arange(-sps * span // 2, sps * span // 2 + 1) / sps
    with np.errstate(divide="ignore", invalid="ignore"):
        h = (np.sin(np.pi * t * (1 - beta)) + 4 * beta * t * np.cos(np.pi * t * (1 + beta))) / (
            np.pi * t * (1 - (4 * beta * t) ** 2))
    edge = beta / np.sqrt(2) * ((1 + 2 / np.pi) * np.sin(np.pi / 4 / beta) + (1 - 2 / np.pi) * np.cos(np.pi / 4 / beta))
    h = np.where(np.abs(t) < 1e-9, 1 - beta + 4 * beta / np.pi, np.where(np.abs(np.abs(4 * beta * t) - 1) < 1e-9, edge, h))
    return h / np.sqrt(np.sum(h * h))


def _shape(symbols, pulse, sps):
    """Pulse-shaped samples of a symbol sequence (rows: real parts), symbol k centred on sample sps k."""
    rows, n = symbols.shape
    half = len(pulse) // 2
    reach = half // sps + 1
    padded = torch.nn.functional.pad(symbols, (reach, reach))
    out = torch.zeros(rows, n, sps, device="cuda")
    for phase in range(sps):
        for j in range(-reach, reach + 1):   # sample sps k + phase sees symbol k - j at pulse offset sps j + phase
            at = sps * j + phase + half
            if 0 <= at < len(pulse):
                out[:, :, phase] += float(pulse[at]) * padded[:, reach - j:reach - j + n]
    return out.view(rows, n * sps)


def _pack(intensity, full_scale, order):
    """12-bit codes of an intensity, two samples per three bytes."""
    q = torch.floor(intensity * (4095.0 / full_scale) + 0.5).clamp_(0, 4095).to(torch.int32).view(-1, 2)
    a, b = q[:, 0], q[:, 1]
    out = torch.empty(q.shape[0], 3, dtype=torch.uint8, device="cuda")
    if order == 0:
        out[:, 0], out[:, 1], out[:, 2] = a & 255, (a >> 8) | ((b & 15) << 4), b >> 4
    else:
        out[:, 0], out[:, 1], out[:, 2] = a >> 4, ((a & 15) << 4) | (b >> 8), b & 255
    return out.view(-1)


def _random(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _noise(shape, g):
    return torch.randn(shape, generator=g, device="cuda")


def _qam(fmt, bits):
    bps = BITS[fmt]
    both = np.stack([_levels(bits.reshape(-1, bps)[:, h * bps // 2:(h + 1) * bps // 2].reshape(-1), bps // 2) for h in (0, 1)])
    return torch.tensor(both / math.sqrt(2 if fmt == 3 else 10), dtype=torch.float32, device="cuda")


def _packed_stream(fmt, n, seed, order, snr_db):
    """n packed samples of a stream of the format, from its first symbol on."""
    g, snr = _random(seed), 10.0 ** (snr_db / 10.0)
    if fmt < 3:     # PAM at 2 samples/symbol: symbol-spaced ISI, intensity 1 + m s, noise on the detected intensity
        m = 2 ** BITS[fmt]
        s = torch.tensor(_levels(_prbs15(seed, BITS[fmt] * (n // 2)), BITS[fmt]) / (m - 1), dtype=torch.float32, device="cuda")
        pad = torch.nn.functional.pad(s, (1, 1))
        x = 0.5 * _shape((0.1 * pad[2:] + s + 0.2 * pad[:-2])[None], _rrc(2, 16), 2)[0]
        power = 0.25 * 0.5 * (m + 1) / (3.0 * (m - 1)) * 1.05
        return _pack(1.0 + x + math.sqrt(power / snr) * _noise((n,), g), 1.0 + 4.0 * math.sqrt(power), order)
    # KK at 4 samples/symbol: single sideband above a tone 10 dB over the signal, 100 kHz linewidth
    x = _shape(_qam(fmt, _prbs15(seed, BITS[fmt] * (n // 4))), _rrc(4, 16), 4)
    walk = (_noise((n,), g).double() * (math.sqrt(2 * math.pi * 1e5 / 4e9) * 2.0 ** 40)).to(torch.int64).cumsum(0)
    angle = walk.double() * 2.0 ** -40 + (2 * math.pi / 80) * ((11 * torch.arange(n, device="cuda")) % 80).double()
    c, s = torch.cos(angle).float(), torch.sin(angle).float()
    tone, sigma = math.sqrt(10.0 / 4), math.sqrt(0.5 / snr)
    re = tone + x[0] * c - x[1] * s + sigma * _noise((n,), g)
    im = x[0] * s + x[1] * c + sigma * _noise((n,), g)
    p = 0.25 + 2 * sigma * sigma
    return _pack(re * re + im * im, 2.5 + p + 4.0 * math.sqrt(5.0 * p + p * p), order)


def _ring(fmt, buf_len, count, seed, order, snr_db):
    stream = _packed_stream(fmt, buf_len * count, seed, order, snr_db)
    return [b.clone() for b in stream.view(count, -1)]


def _two_sps(n_sym, seed, snr_db=19.0):
    """Unit-power 16QAM symbols and their matched-filter output at 2 samples/symbol."""
    g = _random(seed)
    bits = torch.randint(0, 2, (4 * n_sym,), generator=g, device="cuda").cpu().numpy()
    symbols = _qam(4, bits)
    pulse = np.convolve(_rrc(2, 16), _rrc(2, 16))
    y = _shape(symbols, pulse, 2) + math.sqrt(0.5 * 10 ** (-snr_db / 10)) * _noise((2, 2 * n_sym), g)
    return symbols.t().contiguous(), y.t().contiguous()


# ------------------------------------------------------------------ prepare and run
class _Network:
    def __init__(self, max_seg, params):
        self.h = rx.rx_cnn_create(max_seg)
        rx.rx_cnn_set_params(self.h, params)

    def __del__(self):
        rx.rx_cnn_destroy(self.h)


class _Group:
    def __init__(self, receivers, flags):
        self.receivers = receivers
        self.h = rx.rx_group_create([r.h for r in receivers], flags)

    def __del__(self):
        rx.rx_group_destroy(self.h)


def _receiver(c, seed):
    more = {"prbs_seed": seed, "mf_mode": rx.RX_MF_FD if c["fd"] else rx.RX_MF_TIME, "pack_order": c["pack_order"]}
    if c["fmt"] >= 3:
        more |= {"ols_n": c["ols_n"], "ols_v": c["ols_v"]}
    return rx.Receiver(c["fmt"], c["buf_len"], **more)


def _acquire(receiver, ring):
    """The stream's first buffers, until the receiver has trained and emits payload."""
    count = max(1, -(-(1 << 18) // receiver.buf_len))
    for i in range(count):
        receiver.process(ring[i % len(ring)])
    return count


def _members(c):
    rng = random.Random(c["mix_seed"])
    for _ in range(c["members"]):
        fmt, length = rng.randint(0, 4), 1 << rng.randint(c["log2_lo"], c["log2_hi"])
        if c["ragged"]:
            length -= 32 * rng.randint(0, length // 128)
        yield {"fmt": fmt, "buf_len": length, "snr": rng.uniform(14.0, 22.0), "fd": False, "pack_order": 0,
               "ols_n": 65536, "ols_v": 4096}


def prepare(case, seed):
    c, s = case, {"case": case}
    if c["kind"] == "field":
        s["packed"] = _packed_stream(4, c["nsamp"], seed, c["pack_order"], 20.0)
        s["field"] = torch.zeros(c["nsamp"] - c["ols_v"] // 2, 2, device="cuda")
    elif c["kind"] == "fir":
        nt = c["ntaps"]
        _, y = _two_sps(c["nsym"] + 16, seed)
        g = _random(seed + 1)
        taps = 0.05 * _noise((nt, 2), g) * torch.exp(-0.3 * (torch.arange(nt, device="cuda") - nt // 2).abs())[:, None]
        taps[nt // 2, 0] += 1.0
        s["y"], s["taps"] = y, taps.contiguous()
        s["z"] = torch.zeros(c["nsym"], 2, device="cuda")
        s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    elif c["kind"] in ("cnn_forward", "cnn_train"):
        n = c["nseg"]
        symbols, s["y"] = _two_sps(max(1 << 16, SEG * (n + 2)), seed)
        s["net"] = _Network(n, rx_cnn_module.init_params(seed))
        if c["kind"] == "cnn_forward":
            k0 = torch.arange(n, device="cuda") * SEG + 8
            s["out"] = torch.zeros(n, SEG, 2, device="cuda")
        else:
            k0 = torch.randint(8, symbols.shape[0] - 2 * SEG, (n,), generator=_random(seed + 1), device="cuda")
            s["target"] = symbols[k0[:, None] + torch.arange(SEG, device="cuda")].contiguous()
            s["grad"] = torch.zeros(rx.rx_cnn_nparams(), device="cuda")
            s["loss"] = torch.zeros(1, device="cuda")
        s["start"] = (2 * k0 - 12).contiguous()
    elif c["kind"] == "group":
        members = list(_members(c))
        s["ins"] = [_ring(m["fmt"], m["buf_len"], 1, seed + i, 0, m["snr"])[0] for i, m in enumerate(members)]
        receivers = [_receiver(m, seed + i) for i, m in enumerate(members)]
        for r, b in zip(receivers, s["ins"]):
            _acquire(r, [b])
        torch.cuda.synchronize()
        s["group"] = _Group(receivers, rx.RX_GROUP_GRAPH if c["graph"] else 0)
        s["outs"] = [torch.zeros(r.max_bits // 8 + 16, dtype=torch.uint8, device="cuda") for r in receivers]
        s["stream"] = torch.cuda.Stream()
    else:
        count = c["ring"] if c["kind"] == "buffer" else c["bufs"]
        ring = _ring(c["fmt"], c["buf_len"], count, seed, c["pack_order"], 20.0 if c["fmt"] >= 3 else 18.0)
        r = s["receiver"] = _receiver(c, seed)
        s["at"] = _acquire(r, ring)
        if c.get("cnn"):
            s["net"] = _Network(1, rx_cnn_module.init_params(seed))
            rx.rx_set_cnn(r.h, s["net"].h)
        if c["kind"] == "host":
            s["ins"] = [b.cpu().pin_memory() for b in ring]
            s["outs"] = [torch.zeros(r.max_bits // 8 + 16, dtype=torch.uint8).pin_memory() for _ in ring]
        else:
            s["ins"] = ring
    return s


def run(s):
    c = s["case"]
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] == "field":
        rx.rx_kk_field_noalloc(s["packed"].data_ptr(), c["nsamp"], c["pack_order"], c["ols_n"], c["ols_v"],
                               s["field"].data_ptr(), stream)
        return s["field"]
    if c["kind"] == "fir":
        rx.rx_fir_block(s["y"].data_ptr(), s["y"].shape[0], s["taps"].data_ptr(), c["ntaps"], c["prec"], c["nsym"],
                        c["scale_block"], s["z"].data_ptr(), s["status"].data_ptr(), stream)
        return s["z"]
    if c["kind"] == "cnn_forward":
        rx.rx_cnn_forward(s["net"].h, s["y"].data_ptr(), s["start"].data_ptr(), c["nseg"], s["out"].data_ptr(), stream)
        return s["out"]
    if c["kind"] == "cnn_train":
        rx.rx_cnn_grad(s["net"].h, s["y"].data_ptr(), s["start"].data_ptr(), s["target"].data_ptr(), c["nseg"],
                       s["grad"].data_ptr(), s["loss"].data_ptr(), stream)
        rx.rx_cnn_adam_step(s["net"].h, 1e-3, stream)
        return s["grad"], s["loss"]
    if c["kind"] == "buffer":
        packed = s["ins"][s["at"] % len(s["ins"])]
        s["at"] += 1
        return s["receiver"].process(packed)
    if c["kind"] == "batch":
        return s["receiver"].process_batch(s["ins"])
    if c["kind"] == "host":
        n = rx.rx_process_host_batch(s["receiver"].h, [b.data_ptr() for b in s["ins"]],
                                     [o.data_ptr() for o in s["outs"]], stream)
        return [o[: (k + 7) // 8] for o, k in zip(s["outs"], n)]
    s["stream"].wait_stream(torch.cuda.current_stream())
    n = rx.rx_group_process(s["group"].h, [b.data_ptr() for b in s["ins"]], [o.data_ptr() for o in s["outs"]],
                            s["stream"].cuda_stream)
    torch.cuda.current_stream().wait_stream(s["stream"])
    return [o[: (k + 7) // 8] for o, k in zip(s["outs"], n)]


# ------------------------------------------------------------------ work and exact
def _stream_work(fmt, samples, ols_n, ols_v, cnn):
    """Packed samples in, bits out; the chain's arithmetic per sample."""
    if fmt < 3:     # normalise, 33-tap filter, 15-tap equaliser and its update per symbol
        flops = 66 + (30 + 30) / 2
    else:           # a forward and an inverse transform of two real blocks each, field, filter, equaliser
        flops = 5 * math.log2(ols_n) * ols_n / (ols_n - ols_v) + 20 + 130
        flops += 2 * 29_500 / 4 if cnn else (496 + 512) / 4
    return samples * (1.5 + BITS[fmt] / (16 if fmt < 3 else 32)), samples * flops


def work(case):
    c = case
    if c["kind"] == "field":
        n = c["nsamp"]
        return {"bytes": 9.5 * n, "flops": n * (5 * math.log2(c["ols_n"]) * c["ols_n"] / (c["ols_n"] - c["ols_v"]) + 20)}
    if c["kind"] == "fir":
        return {"bytes": 24 * c["nsym"], "flops": 8 * c["ntaps"] * c["nsym"]}
    if c["kind"].startswith("cnn_"):
        # multiply-adds per segment: 136, 128 and 64 positions of the three convolutions, the two dense layers
        macs = 136 * 32 * 18 + (128 + 64) * 32 * 288 + 64 * (64 * 32 + 2 * 64)
        train = c["kind"] == "cnn_train"
        return {"bytes": c["nseg"] * (152 * 8 + 8 + 512) + (2 + 6 * train) * 4 * rx.rx_cnn_nparams(),
                "flops": (6 if train else 2) * macs * c["nseg"]}
    if c["kind"] == "group":
        parts = [_stream_work(m["fmt"], m["buf_len"], 65536, 4096, False) for m in _members(c)]
    else:
        parts = [_stream_work(c["fmt"], c["buf_len"] * c.get("bufs", 1), c["ols_n"], c["ols_v"], c.get("cnn", False))]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def _exact_field(c, packed):
    b = packed.view(-1, 3).long()
    if c["pack_order"] == 0:
        codes = torch.stack([b[:, 0] | ((b[:, 1] & 15) << 8), (b[:, 1] >> 4) | (b[:, 2] << 4)], 1).reshape(-1)
    else:
        codes = torch.stack([(b[:, 0] << 4) | (b[:, 1] >> 4), ((b[:, 1] & 15) << 8) | b[:, 2]], 1).reshape(-1)
    intensity = codes.double().clamp_(min=0.5)
    n, v, total = c["ols_n"], c["ols_v"], c["nsamp"]
    count, hop = total - v // 2, n - v
    u = 0.5 * torch.log(torch.cat([intensity[:1].expand(n), intensity]))
    h = torch.zeros(n, dtype=torch.complex128, device="cuda")
    h[1:n // 2], h[n // 2 + 1:] = -1j, 1j
    phase = torch.empty(count, dtype=torch.float64, device="cuda")
    blocks = -(-count // hop)
    for j in range(blocks):     # every block but the last keeps its middle; the last one ends at the newest sample
        last = j == blocks - 1
        start = total - n if last else j * hop - v // 2
        p = torch.fft.ifft(torch.fft.fft(u[start + n:start + 2 * n]) * h).real
        lo, hi = j * hop, count if last else (j + 1) * hop
        phase[lo:hi] = p[lo - start:hi - start]
    a = torch.sqrt(intensity[:count])
    return torch.stack([a * torch.cos(phase), a * torch.sin(phase)], 1)


def _exact_network(params, y, start, nseg):
    """Soft symbols of the learned equaliser in 64 bits, [nseg, 64, 2]."""
    sizes = [(32, 9, 2), (32,), (32, 9, 32), (32,), (32, 9, 32), (32,), (64, 32), (64,), (2, 64), (2,)]
    parts, at = [], 0
    for shape in sizes:
        parts.append(params[at:at + math.prod(shape)].view(shape))
        at += math.prod(shape)
    w1, b1, w2, b2, w3, b3, m1, c1, m2, c2 = parts
    x = y.double()[start[:, None] + torch.arange(2 * SEG + 24, device=y.device)]
    for w, b in ((w1, b1), (w2, b2), (w3, b3)):
        x = x.unfold(1, 9, 1).permute(0, 1, 3, 2).reshape(nseg, x.shape[1] - 8, -1) @ w.reshape(32, -1).t() + b
        x = torch.nn.functional.gelu(x)
    return torch.nn.functional.gelu(x[:, ::2] @ m1.t() + c1) @ m2.t() + c2


def exact(case, seed):
    c = case
    if c["kind"] not in ("field", "fir", "cnn_forward", "cnn_train"):
        return None     # bits
    s = prepare(case, seed)
    if c["kind"] == "field":
        return _exact_field(c, s["packed"])
    if c["kind"] == "fir":
        y, w, n = torch.view_as_complex(s["y"].double()), torch.view_as_complex(s["taps"].double()), c["nsym"]
        z = torch.zeros(n, dtype=torch.complex128, device="cuda")
        for i in range(c["ntaps"]):
            z += w[i].conj() * y[c["ntaps"] - 1 - i:][: 2 * n:2]
        return torch.view_as_real(z)
    params = torch.tensor(rx_cnn_module.init_params(seed), dtype=torch.float64, device="cuda")
    if c["kind"] == "cnn_forward":
        return torch.cat([_exact_network(params, s["y"], s["start"][i:i + 256], len(s["start"][i:i + 256]))
                          for i in range(0, c["nseg"], 256)])
    params.requires_grad_()
    out = _exact_network(params, s["y"], s["start"], c["nseg"])
    loss = ((out - s["target"].double()) ** 2).sum() / (c["nseg"] * SEG)
    loss.backward()
    return params.grad, loss.detach().view(1)
