"""Rows of the tuner's table (KH_TUNE_FILE) that a graph cannot use are passed over: a
slice count that fits another graph of the same shape class, values no build writes.
Each process reads the table once, so the calls run in one of their own."""
import math
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from paper_2112_06154_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# one slice holds the first size and not the second; both are of one shape class
SMALL, LARGE = 1_100_000, 1_700_000
CODE = """
import sys; sys.path.insert(0, %r)
import numpy as np
from paper_2112_06154_gb300 import graphgen as gg, khcore as K
K.load()
n, out = int(sys.argv[1]), sys.argv[2]
rp, cl = gg.chung_lu(%d, 12, 2.4, 1200, 31)
rp = np.concatenate([rp, np.full(n + 1 - rp.size, rp[-1], np.int64)])
c = K.kh_ctx_create(0)
G = K.kh_graph_load_csr(c, rp, cl)
np.save(out, K.kh_hdegree_exact(G))
print(*K.kh_get_variant(G)[:3])
G.close(); c.close()
"""
LINKED = 40000


def run(table, n, out, timeout=300):
    pytest.importorskip("torch")
    r = subprocess.run([sys.executable, "-c", CODE % (ROOT, LINKED), str(n), str(out)],
                       env=dict(os.environ, KH_TUNE_FILE=str(table)), capture_output=True, text=True,
                       timeout=timeout)
    assert r.returncode == 0, r.stderr[-2000:]
    rp, cl = gg.chung_lu(LINKED, 12, 2.4, 1200, 31)
    deg = np.load(str(out))
    assert np.array_equal(deg[:LINKED], O.hdegree_exact(rp, cl, 2)) and not deg[LINKED:].any()
    return [int(x) for x in r.stdout.split()]


# variant, slices, threads, ms, sweep bin: sliced in one slice; a layout that needs the
# bitmap of all nodes; values outside every range
@pytest.mark.parametrize("row", ["2 1 1024 1.0 0", "3 1 256 1.0 0", "1 0 256 1.0 0", "2 2 100 1.0 0",
                                 "2 0 256 1.0 0", "7 2 256 1.0 0", "2 2 256 1.0 99"])
def test_unusable_rows_are_passed_over(tmp_path, row):
    table = tmp_path / "tune.txt"
    rp, cl = gg.chung_lu(LINKED, 12, 2.4, 1200, 31)
    assert len({(int(math.log2(n)), int(math.log2(np.diff(rp).max() * n / cl.size)))
                for n in (SMALL, LARGE)}) == 1
    first = run(table, SMALL, tmp_path / "a.npy")
    assert first[0] in (2, 3) and first[1] >= 1
    key = table.read_text().split("|")[0].strip()
    table.write_text("%s | %s\n" % (key, row))
    variant, slices, threads = run(table, LARGE, tmp_path / "b.npy")
    assert variant in (2, 3) and slices >= 2 and threads in (256, 512, 1024)


def test_a_usable_row_is_used(tmp_path):
    table = tmp_path / "tune.txt"
    run(table, SMALL, tmp_path / "a.npy")
    key = table.read_text().split("|")[0].strip()
    table.write_text("%s | 2 5 128 1.0 0\n" % key)  # (the tuner offers no 128 threads)
    assert run(table, LARGE, tmp_path / "b.npy") == [2, 5, 128]


def test_rows_without_this_version_are_not_used(tmp_path):
    table = tmp_path / "tune.txt"
    run(table, SMALL, tmp_path / "a.npy")
    key = table.read_text().split("|")[0].split()
    assert key[0] == "hdeg2" and key[1].startswith("v")
    # as the first builds wrote it, and another version's
    rows = [" ".join(key[:1] + key[2:]), " ".join([key[0], key[1] + "9"] + key[2:])]
    table.write_text("".join("%s | 2 5 128 1.0 0\n" % k for k in rows))
    assert run(table, LARGE, tmp_path / "b.npy")[2] in (256, 512, 1024)
