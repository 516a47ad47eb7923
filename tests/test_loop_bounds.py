"""The bounds of the claim loops on the CPU.  walk_chunk bounds a chunk's claims: a model of
the warps' claims, in any order, stays within.  The row readers of k_hdeg2_cta and
k_hdeg2_peel bound a warp's steps: a model of one warp that reads a whole chunk alone, the
most steps a warp can take, stays within.  Every such loop has its bound."""
import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2112_06154_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def constant(name, *files):
    known = {}
    for f in files:
        for k, v in re.findall(r"constexpr int (\w+) = ([^;]+);", source(f)):
            try:
                known[k] = eval(v.replace("/", "//"), {}, known)  # noqa: S307 (our own source)
            except (NameError, SyntaxError):
                pass
    return known[name]


def steps_of_one_warp(buckets):
    """buckets: per bucket (in the order the warp takes them) its lane group size, words a
    lane and step, and the lists' lengths.  Iterations of the claim loop, as written."""
    n = 0
    for lanes, words, lens in buckets:
        groups = [None] * (32 // lanes)  # words left of each group's list
        todo = list(lens)
        while True:
            n += 1
            for i in range(len(groups)):
                if groups[i] is None and todo:
                    groups[i] = todo.pop()
            if all(g is None for g in groups):
                break  # this iteration ends the bucket
            for i, g in enumerate(groups):
                if g is not None:
                    groups[i] = g - lanes * words if g > lanes * words else None
    return n


def claims_of_a_chunk(rng, warps, lanes, lens):
    """The counter's value before each claim of one bucket, warps in any order: a warp claims
    for all its idle groups at once, a group that gets no list is done."""
    lists, cq, bases = list(lens), 0, []
    groups = [[0] * (32 // lanes) for _ in range(warps)]  # words left; -1: done
    running = set(range(warps))
    while running:
        w = rng.choice(sorted(running))
        g = groups[w]
        idle = [i for i, left in enumerate(g) if left == 0]
        if idle:
            bases.append(cq)
            for k, i in enumerate(idle):
                g[i] = lists[cq + k] if cq + k < len(lists) else -1
            cq += len(idle)
        if all(left == -1 for left in g):
            running.discard(w)
        groups[w] = [left if left < 0 else max(0, left - 4 * lanes) for left in g]
    return bases


@pytest.mark.parametrize("seed", range(6))
def test_walk_chunk(seed):
    rng = random.Random(seed)
    rows, most = (constant(c, "kh_internal.cuh", "kh_sampled.cu") for c in ("kLuThreads", "kMaxM"))
    bound = constant("kMaxClaims", "kh_internal.cuh", "kh_sampled.cu")
    lens = {0: [most] * rows, 1: [rng.randint(1, most) for _ in range(rows)], 2: [1] * rows, 3: [most] + [1] * (rows - 1),
            4: [rng.choice([1, 7, 8, 9, 64, 65, 128, 129]) for _ in range(rows)], 5: [5] * (rows // 3)}[seed]
    for lanes in (2, 8, 32):
        bases = claims_of_a_chunk(rng, rows // 32, lanes, lens)
        assert max(bases) < bound
    assert max(claims_of_a_chunk(rng, rows // 32, 2, [])) < bound


@pytest.mark.parametrize("rows", [128, 256, 512])
def test_row_readers(rows):
    expr = re.search(r"constexpr int row_steps\(int rows\) \{ return ([^;]+); \}",
                     source("kh_internal.cuh")).group(1)
    bound = eval(expr, {}, {"rows": rows})  # noqa: S307
    for a, b, c in ((rows, 0, 0), (0, rows, 0), (0, 0, rows), (rows // 3, rows // 3, rows // 3)):
        assert steps_of_one_warp([(32, 4, [511] * c), (8, 4, [32] * b), (2, 4, [8] * a)]) <= bound


def test_every_claim_loop_has_its_bound():
    walk = source("kh_sampled.cu")
    assert walk.count("if (base >= kMaxClaims)") == walk.count("atomicAdd(&sh.cq[") == 1
    for name in ("kh_hdeg2.cu", "kh_exact.cu"):
        text = source(name)
        assert text.count("if (step > row_steps(") == 1
    for text in (walk, source("kh_hdeg2.cu"), source("kh_exact.cu")):
        assert "atomicOr(c.err, kErrLoop)" in text or "atomicOr(a.err, kErrLoop)" in text
