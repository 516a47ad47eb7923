"""Edges of what the peels take: n on both sides of the bitmap that an exact peel keeps
in shared memory, and two contexts that run split graphs at once."""
import threading

import numpy as np
import pytest

import oracle as O
from paper_2112_06154_gb300 import graphgen as gg
from paper_2112_06154_gb300 import khcore as K

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    K.load(build_if_missing=True)
    c = K.kh_ctx_create(0)
    yield c
    c.close()


def spread(rp, cl, n):
    """The graph's nodes at ids 0, .. and .., n - 1 among n - (rp.size - 1) isolated ones."""
    m = rp.size - 1
    ids = np.concatenate([np.arange(m // 2), np.arange(n - (m - m // 2), n)])
    deg = np.diff(rp)
    return ids, deg, ids[cl].astype(np.int32)


# n <= 819,200: the search without a queue, a bitmap of all nodes in shared memory
@pytest.mark.parametrize("n", [819_169, 819_200, 819_201])
def test_exact_core_around_the_bitmap_limit(ctx, n):
    rp, cl = gg.with_hubs(900, (600, 512), 5, avg_deg=5)
    ids, deg, col = spread(rp, cl, n)
    rowptr = np.zeros(n + 1, np.int64)
    rowptr[ids + 1] = deg
    rowptr = np.cumsum(rowptr)
    G = K.kh_graph_load_csr(ctx, rowptr, col)
    try:
        K.kh_set_h(G, 2)
        core = K.kh_core_exact(G)
        assert np.array_equal(core[ids], O.core_exact(rp, cl, 2)[0])
        assert core.sum() == core[ids].sum()
    finally:
        G.close()


def test_two_contexts_with_split_graphs_at_once(ctx):
    graphs = [gg.with_hubs(6001, (4097, 2049, 1500), 23), gg.with_hubs(5003, (2600, 2100, 1025), 29)]
    want = [O.core_sampled(rp, cl, O.ranks(rp.size - 1, 1), 2, 24)[0] for rp, cl in graphs]
    got, errors = [[], []], []

    def work(q):
        try:
            c = K.kh_ctx_create(0)
            G = K.kh_graph_load_csr(c, *graphs[q])
            K.kh_set_h(G, 2)
            K.kh_set_sampling(G, seed=1, M=24)
            for _ in range(6):
                got[q].append(K.kh_core_sampled(G))
            G.close()
            c.close()
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(q,)) for q in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for q in (0, 1):
        assert len(got[q]) == 6 and all(np.array_equal(x, want[q]) for x in got[q])
