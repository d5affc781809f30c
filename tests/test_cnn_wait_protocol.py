"""What the learned receiver's kernel does when a bounded wait for its tensor-core work runs
out, shown on a model of one tile group that follows the kernel's source statement by
statement: whichever waits fail in whichever threads, the issuing thread issues nothing once
it gave up, and no tensor-core work is in flight when tensor memory is freed.
(A wait that runs out needs a hardware fault, so no run on a GPU shows it.)"""

import itertools
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_14333_gb300", "csrc",
                   "rx_cnn.cu")
TOKEN = re.compile(r"(?P<issue>if \(gtid == 0(?P<ok> && ok)?\))|(?P<wait>\bwait_mma\((?P<w>\w)\))"
                   r"|(?P<commit>umma_commit\(bar( \+ (?P<c>\w))?\))|(?P<meet>if \(!?group_and\(gbar, ok\)\))"
                   r"|(?P<bound>mbar_wait\(bar \+ 3)|(?P<free>tmem_dealloc)")
ROW_TILES = 3


def steps(text):
    """(kind, guarded) in source order; what stands in a loop over the row tiles three times."""
    out, guarded = [], False
    for t in TOKEN.finditer(text):
        kind = next(k for k in ("issue", "wait", "commit", "meet", "bound", "free") if t.group(k))
        if kind == "issue":
            guarded = bool(t.group("ok"))
            continue
        each = t.group("w") == "m" or t.group("c") == "m"
        out += [(kind, guarded)] * (ROW_TILES if each else 1)
    return out


def protocol():
    src = re.sub(r"//[^\n]*", "", open(SRC).read())
    body = src[src.index("k_cnn_rx_tc(const float"):src.index("cudaError_t prepare_cnn_rx")]
    loop = body.index("for (int t = t0; t < ntiles; t += tstep) {")
    end = body.index("\n    }\n", loop)
    return steps(body[loop:end]), steps(body[end:])


def run(tiles, fail, tile, leave):
    """The issuing thread (0) and another one (1); `fail` holds the (thread, wait) that run out.
    Work counts as completed only once a wait for it, or for later work, has succeeded."""
    ok, issued, done, waits = [True, True], 0, 0, 0
    for _ in range(tiles):
        if tile[0][0] == "meet" and not all(ok):
            break
        for kind, guarded in tile:
            if kind == "commit" and (ok[0] or not guarded):
                assert ok[0], "tensor-core work issued by a thread that gave up waiting for earlier work"
                issued += 1
            elif kind == "wait":
                waits += 1
                for i in (0, 1):
                    if ok[i] and ((i, waits) in fail or waits > issued):
                        ok[i] = False
                    elif ok[i]:
                        done = max(done, waits)     # commits complete in order
    for kind, _ in leave:
        if kind == "bound" and not all(ok):
            done = issued
        if kind == "free":
            assert done == issued, "tensor memory freed with work in flight"
    return issued, waits


def test_every_wait_may_run_out():
    tile, leave = protocol()
    per_tile = sum(k == "wait" for k, _ in tile)
    assert per_tile == sum(k == "commit" for k, _ in tile) == 2 * ROW_TILES + 3
    assert tile[0][0] == "meet" and leave[-1][0] == "free"
    assert run(2, set(), tile, leave) == (2 * per_tile, 2 * per_tile)
    waits = list(itertools.product((0, 1), range(1, 2 * per_tile + 1)))
    for fail in [{w} for w in waits] + [set(p) for p in itertools.combinations(waits, 2)]:
        for tiles in (1, 2):
            run(tiles, fail, tile, leave)
