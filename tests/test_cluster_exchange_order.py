"""Order of the distributed shared-memory exchanges of the cluster kernels, checked on the
CPU from their source.

A CTA of a cluster writes into its peers' shared memory.  Between one CTA's access and
another's only the cluster barrier counts: x of CTA A comes before y of CTA B if A arrives at
some barrier after x whose wait in B comes before y.  (The barrier that ends a round of the
Jacobi sweeps joins CTAs of different clusters.)  Each kernel's loop body is reduced to its
sequence of cluster barriers and accesses to the exchanged arrays, run for a few rounds in
two CTAs; every remote write and every read by the owner that touch the same words must be
ordered one way or the other."""

import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2403_06218_gb300" / "csrc"

SYNC = r"cl\.sync\(\)|cluster_arrive\(\)|cluster_wait\(\)"


def _body(src, head, loop):
    """The braces' content after `loop` within the function whose definition follows `head`."""
    at = src.index(loop, src.index(head))
    i = src.index("{", at + len(loop) - 1)
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return re.sub(r"//[^\n]*", "", src[i:j])
    raise AssertionError("unbalanced braces")


def _events(body, arrays):
    """[(what, array, by_parity)] in source order; what: arrive, wait, write (remote) or read."""
    names = "|".join(map(re.escape, arrays))
    out = []
    for m in re.finditer(rf"{SYNC}|map_shared_rank\(&(?P<w>{names})\b(?P<wi>[^;]*?)\)|(?<![\w.])(?P<r>{names})\b"
                         rf"(?P<ri>(?:\[[^\]]*\])*)", body):
        t = m.group(0)
        if t.startswith("cl.sync"):
            out += [("arrive", None, False), ("wait", None, False)]
        elif t.startswith("cluster_"):
            out.append((t[8:-2], None, False))
        elif m.group("w"):
            out.append(("write", m.group("w"), "parity" in m.group("wi")))
        else:
            out.append(("read", m.group("r"), "parity" in m.group("ri")))
    return out


def _unordered(events, rounds=4):
    """Conflicting accesses of two CTAs that no cluster barrier orders."""
    seq, arrives, waits = [], 0, 0
    for rnd in range(rounds):
        for what, name, by_parity in events:
            if what == "arrive":
                arrives += 1
            elif what == "wait":
                if waits < arrives:  # the first round has nothing to wait for
                    waits += 1
            else:
                # arrives, waits: barriers arrived at before, and waited for before, this access
                seq.append((what, name, rnd % 2 if by_parity else 0, arrives, waits, rnd))
    bad = []
    for w in seq:
        for r in seq:
            if w[0] != "write" or r[0] != "read" or w[1:3] != r[1:3]:
                continue
            # x before y: barrier number x.arrives (the next one after x) has been waited for by y
            if not (r[4] > w[3] or w[4] > r[3]):
                bad.append((w[1], w[5], r[5]))
    return bad


KERNELS = [
    ("k_jacobi.cu", "jacobi32_kernel(int n", "for (int rnd = 0; rnd < nblk - 1;", ["s_in", "s_state"]),
    ("k_dense.cu", "chol_inv_cluster_kernel(int b", "for (int p0 = 0; p0 < b && bad == 0;", ["sm.Lp", "sm.Mp"]),
]


@pytest.mark.parametrize("file,head,loop,arrays", KERNELS, ids=["jacobi32", "cholesky"])
def test_exchanges_are_ordered_by_cluster_barriers(file, head, loop, arrays):
    ev = _events(_body((CSRC / file).read_text(), head, loop), arrays)
    for a in arrays:
        assert {w for w, n, _ in ev if n == a} == {"write", "read"}, (a, ev)
    assert _unordered(ev) == []


def test_the_model_finds_a_missing_barrier():
    one = [("write", "x", False), ("arrive", None, False), ("wait", None, False), ("read", "x", False)]
    assert _unordered(one)  # the next round's write against this round's read
    assert not _unordered([(w, n, True) for w, n, _ in one])  # two copies
    assert not _unordered([("wait", None, False)] + one + [("arrive", None, False)])  # split barrier
    assert not _unordered(one + [("arrive", None, False), ("wait", None, False)])  # whole barrier
