"""A CUDA call that fails inside a receiver call makes that call fail: nothing is reported as
decided from data that never arrived or out of order, and the handle refuses later buffers.
The receiver's host code runs against a stand-in for the CUDA runtime (fake_cudart.c)."""

import ctypes as C
import os
import subprocess

import pytest

import paper_2010_14333_gb300 as rx
from paper_2010_14333_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
RX_OK, RX_ECUDA, RX_ESTATE = 0, 3, 4
INVALID = 1      # cudaErrorInvalidValue
NB = 1 << 17


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    _build.build_library()
    objs = [os.path.join(_build.OBJ_DIR, s.replace(".cu", ".o")) for s in _build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        _build.build_library(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "librx_fake.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-x", "c", "-w", os.path.join(HERE, "fake_cudart.c"), "-x", "none",
                    *objs, "-o", out], check=True)
    L = C.CDLL(out)
    L.rx_default_config.argtypes = [C.c_int, C.POINTER(rx.RxConfig)]
    L.rx_create.argtypes = [C.c_int, C.c_double, C.c_double, C.c_int64, C.POINTER(rx.RxConfig), C.POINTER(C.c_void_p)]
    for f in (L.rx_process_host_batch, L.rx_process_batch):
        f.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p]
    L.rx_destroy.argtypes, L.rx_destroy.restype = [C.c_void_p], None
    L.fake_launches.restype = C.c_long
    return L


class Stream:
    def __init__(self, lib, fmt, **options):
        self.lib, cfg, h = lib, rx.RxConfig(), C.c_void_p()
        assert lib.rx_default_config(fmt, C.byref(cfg)) == RX_OK
        for k, v in options.items():
            setattr(cfg, k, v)
        assert lib.rx_create(fmt, 1e9 if fmt >= 3 else 2e9, 4e9, NB, C.byref(cfg), C.byref(h)) == RX_OK
        self.h = h
        self.ins = [(C.c_uint8 * (NB * 3 // 2 + 16))() for _ in range(3)]
        self.outs = [(C.c_uint8 * (NB // 2))() for _ in range(3)]

    def batch(self, host):
        align = lambda b: (C.addressof(b) + 15) & ~15
        ia = (C.c_void_p * 3)(*[align(b) for b in self.ins])
        oa = (C.c_void_p * 3)(*[C.addressof(b) for b in self.outs])
        f = self.lib.rx_process_host_batch if host else self.lib.rx_process_batch
        return f(self.h, ia, oa, 3, None, (C.c_int64 * 3)())

    def close(self):
        self.lib.fake_fail(b"", 0, 0)
        self.lib.rx_destroy(self.h)


PAM, KK = {"ntrain": 4096}, {"ols_n": 4096, "ols_v": 512, "ntrain": 4096, "ncma": 2048, "amb_syms": 1024}
FORMS = [(1, PAM, True), (1, PAM, False), (1, dict(PAM, mf_mode=1), True), (4, KK, True), (4, {}, False)]


@pytest.mark.parametrize("fmt, options, host", FORMS)
@pytest.mark.parametrize("name", ["cudaMemcpyAsync", "cudaEventRecord", "cudaStreamWaitEvent", "launch"])
def test_every_failed_call_fails_the_batch(lib, fmt, options, host, name):
    nth = 0
    while True:
        nth += 1
        s = Stream(lib, fmt, **options)
        try:
            assert s.batch(host) == RX_OK        # the stream's training
            before = lib.fake_launches()
            lib.fake_fail(name.encode(), nth, INVALID)
            status = s.batch(host)
            if lib.fake_pending():               # fewer than nth such calls in a batch
                assert status == RX_OK and lib.fake_launches() > before
                break
            assert status == RX_ECUDA, f"{name} {nth} failed unnoticed"
            if name == "cudaMemcpyAsync":
                assert s.batch(host) == RX_ESTATE
        finally:
            s.close()
    assert nth > (3 if host or name in ("cudaEventRecord", "cudaStreamWaitEvent", "launch") else 0)
