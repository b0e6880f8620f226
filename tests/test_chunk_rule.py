"""The fused kernels' chunk rule (host code, compiled here by itself): the same
choices as trying every number of chunks, without its time (a launch plans its
own, so the rule runs once per launch)."""
import ctypes as C
import os
import random
import subprocess
import time

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1309_3452_gb300", "csrc")


@pytest.fixture(scope="module")
def rank(tmp_path_factory):
    with open(os.path.join(CSRC, "step_fused.cu")) as f:
        text = f.read()
    i = text.index("int rank_chunks(")
    src = tmp_path_factory.mktemp("rule") / "rule.cpp"
    src.write_text('extern "C" ' + text[i:text.index("\n}\n", i) + 3])
    lib = str(src)[:-4] + ".so"
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-o", lib, str(src)], check=True)
    fn = C.CDLL(lib).rank_chunks
    fn.argtypes = [C.c_longlong, C.c_int, C.c_longlong, C.c_int, C.c_double, C.POINTER(C.c_int), C.c_int]

    def call(tiles, levels, workers, min_chunk, restart, most):
        out = (C.c_int * most)()
        n = fn(tiles, levels, workers, min_chunk, restart, out, most)
        return list(out[:n])
    return call


def every_count(tiles, levels, workers, min_chunk, restart, most):
    """The rule as it is written down: every number of chunks in turn, best first, ties to fewer chunks."""
    best, seen = [], set()
    for c in range(1, levels + 1):
        n = -(-levels // c)
        if n < min_chunk and c > 1:
            break
        if n in seen:
            continue
        seen.add(n)
        rounds = -(-tiles * -(-levels // n) // workers)
        eff = tiles * levels / (float(rounds) * workers * (n + restart))
        pos = len(best)
        while pos and eff > best[pos - 1][0] * 1.0001:
            pos -= 1
        if pos < most:
            best.insert(pos, (eff, n))
            del best[most:]
    return [n for _, n in best] or [levels]


def test_same_choices(rank):
    rng = random.Random(5)
    cases = [(1, n, 3648, 2, 1.0, 6) for n in (1, 2, 3, 4, 5, 29, 30)]
    for _ in range(400):
        cases.append((rng.randint(1, 5000), int(2 ** rng.uniform(0, 13)), rng.choice((152, 2432, 3648)),
                      rng.choice((2, 4)), rng.choice((0.5, 1.0, 3.0)), rng.choice((1, 6))))
    for c in cases:
        assert rank(*c) == every_count(*c), c


def test_cost_grows_with_the_root_of_the_levels(rank):
    """2^24 levels have 8 190 different chunk lengths; 2^23 counts of chunks would take tens of milliseconds."""
    t = min(timed(rank) for _ in range(5))
    assert t < 5e-3


def timed(rank):
    t = time.perf_counter()
    rank(1, 1 << 24, 3648, 2, 1.0, 1)
    return time.perf_counter() - t
