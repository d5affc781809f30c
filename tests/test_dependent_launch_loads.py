"""Kernels that start while the grid before them drains (they call pdl_wait or pdl_wait_late) may read data
that is still being written when they start.  ``__restrict__`` pointers and ``__ldg`` promise
the compiler data that nothing else writes while the kernel lives, and so allow loads above
the wait and through the read-only path: in these kernels, and in the device functions they
are built from, only tables that are written when a handle is made may carry that promise."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_14333_gb300", "csrc")
# twiddles, ln table, filter spectra and taps, downshift phases, reference bits
TABLES = {"gtab", "lnt", "twN2g", "tw", "H", "rrc", "ds_tab", "tab", "prbs_ext", "prbs_bits"}
FUNCTION = re.compile(r"__(?P<kind>global|device)__\s[^;{}]*?(?P<name>\w+)\((?P<args>[^{};]*)\)\s*\{")


def functions():
    """(file, kind, name, parameters, body) of every function with a body."""
    for fn in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, fn)).read())
        src = re.sub(r"__launch_bounds__\([^()]*\)|__cluster_dims__\([^()]*\)", "", src)
        for m in FUNCTION.finditer(src):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            yield fn, m.group("kind"), m.group("name"), m.group("args"), src[m.end():i]


def test_only_constant_tables_are_promised_read_only():
    every = list(functions())
    kernels = [f for f in every if f[1] == "global"]
    dependent = [f for f in kernels if "pdl_wait" in f[4]]
    ordinary = [f for f in kernels if "pdl_wait" not in f[4]]
    used = lambda name, fs: any(re.search(rf"\b{name}\b", f[4]) for f in fs)
    # device functions, but for those that only ordinary kernels call
    device = [f for f in every if f[1] == "device" and (used(f[2], dependent) or not used(f[2], ordinary))]
    assert len(dependent) >= 20
    bad = []
    for fn, _, name, args, body in dependent + device:
        bad += [(fn, name, p) for p in re.findall(r"__restrict__\s+(\w+)", args) if p not in TABLES]
        bad += [(fn, name, a) for a in re.findall(r"__ldg\(\s*([^)]*)", body) if not set(re.findall(r"\w+", a)) & TABLES]
    assert not bad, bad
