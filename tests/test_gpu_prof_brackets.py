"""The brackets of a kernel class do not overlap: their algorithmic bytes add up to the
class's counter and their times to no more than the call took, also where a pass runs
kernels beside each other (the large sources of the one-CTA-per-source layout)."""
import time

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


@pytest.mark.parametrize("counts", [False, True])
def test_two_degree_brackets(ctx, counts):
    rp, cl = gg.chung_lu(20000, 20, 2.5, 1500, 1102)
    work = np.add.reduceat(np.diff(rp)[cl], rp[:-1][np.diff(rp) > 0])
    assert work.max() >= 2 ** 14  # some sources take a large CTA on the second stream
    want = O.hdegree_exact(rp, cl, 2)
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        K.kh_set_h(G, 2)
        K.kh_set_variant(G, K.KH_VAR_CTA)
        K.kh_set_variant(G, K.KH_SWEEP_OFF, op=K.KH_OP_HDEG2_SWEEP)
        call = (lambda: K.kh_sampled_counts(G, 0, 3)[:, 0]) if counts else lambda: K.kh_hdegree_exact(G)
        assert np.array_equal(call(), want)
        K.kh_prof_enable(G, True)
        t = time.perf_counter()
        assert np.array_equal(call(), want)
        wall = 1e3 * (time.perf_counter() - t)
        ms, launches, alg = K.kh_prof_read(G, K.KH_PROF_BFS)
        trace = K.kh_prof_trace_bytes(G, K.KH_PROF_BFS)
        assert trace.size == launches > 0 and alg > 0
        assert int(trace.sum()) == int(alg)
        assert 0.0 < ms <= wall
        K.kh_prof_enable(G, False)
    finally:
        G.close()
