"""Order of the accesses to distributed shared memory in the one-cluster panel kernel (csrc/sbr.cu, k_panel_qr with
CL > 0).  No GPU.

The barriers, the stores to the other blocks (st_peer) and the reads of what they sent are taken from the kernel's source
in program order; every block runs them, the ones of the column loop once per column.  A wait of the cluster barrier
completes only after all blocks have made the arrive that belongs to it, and nothing else orders two blocks.  From that
rule alone:
 * a store to a peer must follow the peer's start, and precede its exit;
 * the reads of column c must follow all stores of column c;
 * the stores of column c + 2 (same buffer, by parity) must follow all reads of column c."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_02460_gb300", "csrc")
TOKENS = [("arrive", r"barrier\.cluster\.arrive\S*aligned"), ("wait", r"barrier\.cluster\.wait\S*aligned"),
          ("store", r"\bst_peer\("), ("read", r"\+= cw\[|CL \? cp\[|CL \? cn\["), ("loop", r"for \(int c = 0; c < ncol; \+\+c\)"),
          ("end", r"---- write back")]


def program():
    """(prologue, column) event kinds in source order."""
    src = open(os.path.join(CSRC, "sbr.cu")).read()
    body = src[src.index("k_panel_qr(PanelArgs<T> a) {"):]
    body = re.sub(r"//(?! ---- write back).*", "", body)
    ev = sorted((m.start(), k) for k, rx in TOKENS for m in re.finditer(rx, body))
    kinds = [k for _, k in ev]
    loop, end = kinds.index("loop"), kinds.index("end")
    return kinds[:loop], kinds[loop + 1:end]


def run(prologue, column, ncol):
    """One block's events: (kind, column, waits completed before it, arrives made before it)."""
    out, waits, arrives = [], 0, 0
    for c, kinds in [(-1, prologue)] + [(c, column) for c in range(ncol)]:
        for k in kinds:
            out.append((k, c, waits, arrives))
            arrives += k == "arrive"
            waits += k == "wait"
    out.append(("exit", ncol, waits, arrives))
    return out


def before(a, b):
    """Event a of one block happens before event b of another: a precedes the block's arrive number i (its later events
    do, too), and b follows wait number i, which needs every block's arrive i."""
    return b[2] > a[3]


def faults(prologue, column, ncol=5):
    ev = run(prologue, column, ncol)
    start = ("start", -1, 0, 0)
    exit_ = ev[-1]
    stores = [e for e in ev if e[0] == "store"]
    reads = [e for e in ev if e[0] == "read"]
    assert stores and reads
    out = []
    out += [("store before the peer's start", s[1]) for s in stores if not before(start, s)]
    out += [("store after the peer's exit", s[1]) for s in stores if not before(s, exit_)]
    out += [("read before the store", r[1]) for r in reads for s in stores if s[1] == r[1] and not before(s, r)]
    out += [("store over a buffer still read", s[1]) for r in reads for s in stores
            if s[1] == r[1] + 2 and not before(r, s)]
    return out


@pytest.mark.parametrize("ncol", [1, 2, 3, 16, 64])
def test_every_remote_access_is_ordered(ncol):
    assert faults(*program(), ncol) == []


def test_missing_barriers_are_caught():
    prologue, column = program()
    assert ("store before the peer's start", 0) in faults([], column)
    assert faults(prologue, [k for k in column if k not in ("arrive", "wait")])
    late = [k for k in column if k != "store"]
    assert faults(prologue, late + ["store"])
