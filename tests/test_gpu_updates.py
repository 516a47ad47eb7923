"""kh_peel_info's count of completed (re)computations on graphs where it can be
counted by hand: nodes that the early stop (Sec. 5) assigns are not recomputed."""
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


def path(n):
    return gg.csr_from_edges(n, np.arange(n - 1), np.arange(1, n))


# A path of 5 at h = 2: 2-degrees 2, 3, 4, 3, 2.  All five lower bounds are 2, the first
# threshold: five searches.  The ends leave with c = 2; three nodes are left, and
# c >= 3 - 1 assigns them.  The middle node, two hops from both ends, would have lost 2.
def test_path_of_five(ctx):
    rp, cl = path(5)
    want, wround, steps = O.core_exact(rp, cl, 2)
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        K.kh_set_h(G, 2)
        assert np.array_equal(K.kh_core_exact(G), want)
        ro, rounds, updates = K.kh_peel_info(G)
        assert np.array_equal(ro, wround) and rounds == steps
        assert updates == 5
    finally:
        G.close()


# Beside it in a batch, a path of 7: 2-degrees 2, 3, 4, 4, 4, 3, 2, lower bounds 2:
# seven searches.  The ends leave; five nodes are left (c = 2 < 4), the nodes next to the
# ends are searched again (2-degree 2), the nodes two hops away lose one each (to 3): 2 + 2.
# Those two leave; three are left and c >= 3 - 1 assigns them.
def test_paths_in_a_batch(ctx):
    graphs = [path(5), path(7)]
    off, rp, cl = gg.pack_batch(graphs)
    G = K.kh_graph_load_batch(ctx, off, rp, cl, [2, 2])
    try:
        core = K.kh_core_exact(G)
        _, _, updates = K.kh_peel_info(G)
        for q, (r, c) in enumerate(graphs):
            assert np.array_equal(core[off[q]:off[q + 1]], O.core_exact(r, c, 2)[0])
        assert updates == 5 + 7 + 4
    finally:
        G.close()
