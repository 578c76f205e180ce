"""Places of a team's block sums (csrc/team_part.h) under every order of the
blocks that the team barrier allows.

Each block runs a random sequence of reductions and plain barriers, one access
to the shared array at a time, in an order drawn at random; a block may be
anywhere between two barriers while another has just passed the first.  With
the places of the header every block reads the same sums, the right ones.  With
one place for all reductions, as a control of the model, some order mixes two
reductions."""
import ctypes as C
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_08494_gb300", "csrc")
SOURCE = """
#include "team_part.h"
extern "C" int at(unsigned long long gen, int m, int nb, int b) { return lbeh::part_at(gen, m, nb, b); }
extern "C" long long doubles(int nb) { return lbeh::part_doubles(nb); }
extern "C" int sums() { return lbeh::kPartSums; }
"""


@pytest.fixture(scope="module")
def part(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("part")
    (d / "part.cpp").write_text(SOURCE)
    subprocess.run([gxx, "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "part.so"), str(d / "part.cpp")],
                   check=True, capture_output=True)
    lib = C.CDLL(str(d / "part.so"))
    lib.at.argtypes = [C.c_ulonglong, C.c_int, C.c_int, C.c_int]
    lib.doubles.argtypes = [C.c_int]
    lib.doubles.restype = C.c_longlong
    return lib


def _value(op, m, b):
    return 1 + 1000 * op + 10 * b + m


def _block(b, nb, ops, at, mem, out):
    """One block: ops[k] = values of the reduction, 0 for a barrier alone."""
    gen = 0
    for k, M in enumerate(ops):
        for m in range(M):
            mem[at(gen, m, nb, b)] = _value(k, m, b)
            yield "step"
        yield "barrier"
        gen += 1
        s = [0] * M
        for o in range(nb):
            for m in range(M):
                s[m] += mem[at(gen - 1, m, nb, o)]
                yield "step"
        out.append(s)


def _run(nb, ops, at, size, rng):
    """All blocks in a random order that respects the barriers; the sums each block read."""
    mem, outs = [0] * size, [[] for _ in range(nb)]
    blocks = [_block(b, nb, ops, at, mem, outs[b]) for b in range(nb)]
    arrived, passed, done = [0] * nb, [0] * nb, [False] * nb
    while not all(done):
        # a block waits at barrier g until every block has arrived there
        ready = [b for b in range(nb) if not done[b] and passed[b] == arrived[b]]
        for b in [b for b in range(nb) if not done[b] and arrived[b] > passed[b] and min(arrived) >= arrived[b]]:
            ready.append(b)
        b = rng.choice(ready)
        passed[b] = arrived[b]
        for _ in range(rng.choice((1, 1, 2, 50))):  # bursts let a block run ahead as far as it can
            e = next(blocks[b], "end")
            if e == "end":
                done[b] = True
                arrived[b] = passed[b] = len(ops)
                break
            if e == "barrier":
                arrived[b] += 1
                break
    return outs


def _wrong(nb, ops, at, size, rng):
    want = [[sum(_value(k, m, b) for b in range(nb)) for m in range(M)] for k, M in enumerate(ops)]
    return any(o != want for o in _run(nb, ops, at, size, rng))


@pytest.mark.parametrize("nb", [1, 2, 5, 16])
def test_every_block_reads_the_same_sums(part, nb):
    rng = random.Random(nb)
    size = int(part.doubles(nb))
    ms = range(part.sums())
    assert sorted({part.at(g, m, nb, b) for g in (0, 1) for m in ms for b in range(nb)}) == list(range(size))
    mixed = 0
    for _ in range(40):
        ops = [rng.choice((0, 1, 2, 3, 3)) for _ in range(rng.randint(2, 7))]
        assert not _wrong(nb, ops, part.at, size, rng), ops
        mixed += _wrong(nb, ops, lambda gen, m, nb, b: m * nb + b, size, rng)
    assert nb == 1 or mixed > 0
