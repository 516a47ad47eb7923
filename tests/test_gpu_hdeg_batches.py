"""Exact h-degrees at h >= 3 by bit-parallel batches of 1024 sources, against the
oracle: ragged last batches, isolated nodes, rows at the edges of the kernels'
row pieces (128 entries), one to four pulls, and a graph of small balls that
keeps the search per source."""
import numpy as np
import pytest

import oracle as O
from paper_2112_06154_gb300 import graphgen as gg
from paper_2112_06154_gb300 import khcore as K

pytestmark = pytest.mark.gpu

GRAPHS = {
    "rmat12": lambda: gg.rmat(12, 16, 0.57, 0.19, 0.19, 5),   # about a third isolated
    "cl5k": lambda: gg.chung_lu(5003, 20, 2.5, 400, 17),
    "rows": lambda: gg.with_hubs(3100, (127, 128, 129, 255, 256, 257, 1500), 19, avg_deg=16),
}


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    K.load(build_if_missing=True)
    c = K.kh_ctx_create(0)
    yield c
    c.close()


@pytest.mark.parametrize("h", [3, 4, 5])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_batches_match_the_oracle(ctx, name, h):
    rp, cl = GRAPHS[name]()
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        K.kh_set_h(G, h)
        want = O.hdegree_exact(rp, cl, h)
        before = K.kh_launch_count(G)
        assert np.array_equal(K.kh_hdegree_exact(G), want)
        assert K.kh_launch_count(G) - before > 12  # batches, not one search kernel
        assert np.array_equal(K.kh_hdegree_exact(G), want)  # the masks are clean again
        # the counts and the other h go their own ways on the same graph
        cnt = K.kh_sampled_counts(G, 0, 3)
        assert np.array_equal(cnt[:, 0], want)
        K.kh_set_h(G, 2)
        assert np.array_equal(K.kh_hdegree_exact(G), O.hdegree_exact(rp, cl, 2))
    finally:
        G.close()


def test_small_balls_keep_the_search(ctx):
    rp, cl = gg.grid(90, 70, 0.01, 3)
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        K.kh_set_h(G, 3)
        assert np.array_equal(K.kh_hdegree_exact(G), O.hdegree_exact(rp, cl, 3))
        before = K.kh_launch_count(G)
        K.kh_hdegree_exact(G)
        assert K.kh_launch_count(G) - before == 1
    finally:
        G.close()


def test_no_memory_for_masks_or_entry_ranks(ctx):
    """The passes that need extra arrays fall back on the search per source."""
    rp, cl = GRAPHS["cl5k"]()
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        for h in (3, 4):
            K.kh_set_h(G, h)
            if h == 4:
                K.kh_debug_fail_alloc(ctx, 1)  # h = 3 has all but the third mask array
            assert np.array_equal(K.kh_hdegree_exact(G), O.hdegree_exact(rp, cl, h))
        K.kh_debug_fail_alloc(ctx, 0)
        assert np.array_equal(K.kh_hdegree_exact(G), O.hdegree_exact(rp, cl, 4))
        K.kh_set_h(G, 2)
        want = O.hdegree_exact(rp, cl, 2)
        K.kh_debug_fail_alloc(ctx, 1)  # the ranks of the row entries
        assert np.array_equal(K.kh_sampled_counts(G, 0, 3)[:, 0], want)
        K.kh_debug_fail_alloc(ctx, 0)
        assert np.array_equal(K.kh_sampled_counts(G, 0, 3)[:, 0], want)
    finally:
        K.kh_debug_fail_alloc(ctx, 0)
        G.close()


@pytest.mark.parametrize("h", [3, 4])
@pytest.mark.parametrize("m", [1501, 1506, 3000])  # around a mean degree of 5
def test_exact_cores_by_wide_searches(ctx, m, h):
    rp, cl = gg.erdos_renyi(601, m, 8)
    want, wround, steps = O.core_exact(rp, cl, h)
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        K.kh_set_h(G, h)
        assert np.array_equal(K.kh_core_exact(G), want)
        ro, rounds, _ = K.kh_peel_info(G)
        assert np.array_equal(ro, wround) and rounds == steps
    finally:
        G.close()
