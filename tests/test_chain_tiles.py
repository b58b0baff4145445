"""The one-launch training step's operand copies: the transposed tile that a
CTA stages in the copy its product has read lies inside it and apart from the
columns that the other CTA of its cluster may already be writing there for the
product after the next, for every sequence of layer widths that the step takes
(csrc/chain_tiles.h, compiled for the host)."""
import ctypes
import itertools
import os
import subprocess

import pytest

from paper_2606_00946_gb300 import build as B


@pytest.fixture(scope="module")
def chain(tmp_path_factory):
    d = tmp_path_factory.mktemp("chain")
    src, lib = d / "chain.cpp", d / "libchain.so"
    src.write_text('#include "chain_tiles.h"\nextern "C" {\n'
                   "int first_block(int r, int n) { return ls::chain::first_block(r, n); }\n"
                   "int stage_block(int c, int r, int n, int m) { return ls::chain::stage_block(c, r, n, m); }\n}\n")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", B.CSRC, "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(os.fspath(lib))


# hidden widths a cluster of CL CTAs takes: whole K-blocks of 64 in every part, at most 256
WIDTHS = {1: (64, 128, 192, 256), 2: (128, 256)}


@pytest.mark.parametrize("CL", (1, 2))
@pytest.mark.parametrize("layers", range(1, 6))
def test_staged_tile_meets_nothing_written_meanwhile(chain, CL, layers):
    for hidden in itertools.product(WIDTHS[CL], repeat=layers):
        # columns of the products in order: forward, then input gradients from the last hidden layer down
        N = [*hidden, *hidden[-2::-1]]
        NT = [n // CL for n in N]
        blocks = max(64, *hidden) // 64  # (a wider minibatch operand only adds room)
        for p, rank in itertools.product(range(len(N)), range(CL)):
            nxt = NT[p + 1] if p + 1 < len(N) else NT[p]
            at = chain.stage_block(CL, rank, NT[p], nxt)
            mine = set(range(at, at + NT[p] // 64))
            assert 0 <= at and max(mine) < blocks, (hidden, p, rank)
            if p + 1 < len(N) and CL > 1:
                first = chain.first_block(1 - rank, nxt)
                other = set(range(first, first + nxt // 64))
                assert not mine & other, (hidden, p, rank, sorted(mine), sorted(other))
