"""The named barriers of the sequential-commit kernel: in every order that a
CTA's scoring, lookup and inserting warps can run, each phase of a barrier
joins the arrivals it is meant for and every warp comes to its end.  The steps
at which a role waits or arrives are the kernel's own (csrc/seq_steps.h,
compiled for the host); a barrier is a count of arrivals, as on the device."""
import ctypes
import os
import subprocess

import pytest

from paper_2606_00946_gb300 import build as B

FNS = ["bar_looked_up(a)", "bar_inserted(a)", "waits_inserted(a, b)", "tells_inserted(a, b)", "bar_bids_look()",
       "tells_look(a, b)", "bar_bids_insert(a)"]


@pytest.fixture(scope="module")
def seq(tmp_path_factory):
    d = tmp_path_factory.mktemp("seq")
    src, lib = d / "seq.cpp", d / "libseq.so"
    src.write_text('#include "seq_steps.h"\n' + "".join(
        f'extern "C" int {f.split("(")[0]}(int a, int b) {{ (void)a; (void)b; return (int)ls::seq::{f}; }}\n'
        for f in FNS))
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", B.CSRC, "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(os.fspath(lib))


# warps of each role in the model (the kernel has 8, 6 and 2)
SCORE, LOOK, INSERT = 2, 1, 2


def programs(q, n):
    """Per role, its (kind, barrier, purpose) operations in order, as k_route_seq runs them for n requests.
    "sync" arrives and waits, "arrive" does not wait; the purpose names the phase the operation belongs to."""
    score, look, insert = [], [], []
    for s in range(n + 1):
        if s < n:
            score.append(("sync", q.bar_looked_up(s, n), ("looked up", s)))
        if q.waits_inserted(s, n):
            score.append(("sync", q.bar_inserted(s - 2, n), ("inserted", s - 2)))
        if q.tells_look(s, n):
            score.append(("arrive", q.bar_bids_look(), ("bids, lookups", s)))
        if s > 0:
            score.append(("arrive", q.bar_bids_insert(s, n), ("bids, inserts", s)))
        score.append(("sync", 1, ("scoring", s)))
    for s in range(-1, n - 1):
        if s > 0:
            look.append(("sync", q.bar_bids_look(), ("bids, lookups", s)))
        look.append(("arrive", q.bar_looked_up(s + 1, n), ("looked up", s + 1)))
    for s in range(n + 1):
        if s > 0:
            insert.append(("sync", q.bar_bids_insert(s, n), ("bids, inserts", s)))
        if q.tells_inserted(s, n):
            insert.append(("arrive", q.bar_inserted(s, n), ("inserted", s)))
    return [score] * SCORE + [look] * LOOK + [insert] * INSERT


def members(q, n):
    """Arrivals that complete a phase of each barrier."""
    m = {1: SCORE, q.bar_bids_look(): SCORE + LOOK}
    for s in range(n + 1):
        m[q.bar_looked_up(s, n)] = SCORE + LOOK
        m[q.bar_inserted(s, n)] = m[q.bar_bids_insert(s, n)] = SCORE + INSERT
    return m


def explore(q, n):
    """None, or what goes wrong in some order of the warps."""
    progs, count = programs(q, n), members(q, n)
    # state: next operation of each warp, those waiting, and each barrier's arrivals so far
    start = (tuple(0 for _ in progs), frozenset(), frozenset())
    todo, seen = [start], {start}
    while todo:
        pcs, waiting, bars = todo.pop()
        moves = 0
        for w, prog in enumerate(progs):
            if w in waiting or pcs[w] == len(prog):
                continue
            moves += 1
            kind, bar, purpose = prog[pcs[w]]
            at = dict(bars)
            inside = at.get(bar, ())
            if any(p != purpose for _, p in inside):
                return f"barrier {bar}: {purpose} joins {[p for _, p in inside]}"
            inside = tuple(sorted(inside + ((w, purpose),)))
            npc = list(pcs)
            nw = set(waiting)
            if kind == "sync":
                nw.add(w)
            else:
                npc[w] += 1
            if len(inside) == count[bar]:  # the phase completes: its waiting warps go on
                for v, _ in inside:
                    if v in nw and progs[v][npc[v]][1] == bar:
                        nw.discard(v)
                        npc[v] += 1
                at.pop(bar, None)
            else:
                at[bar] = inside
            st = (tuple(npc), frozenset(nw), frozenset(at.items()))
            if st not in seen:
                seen.add(st)
                todo.append(st)
        if not moves and any(pcs[w] < len(p) for w, p in enumerate(progs)):
            return f"warps wait forever: {[progs[w][pcs[w]] for w in waiting]}"
        if not moves and bars:
            return f"arrivals left over: {bars}"
    return None


@pytest.mark.parametrize("n", range(1, 11))
def test_every_order_ends(seq, n):
    assert explore(seq, n) is None
