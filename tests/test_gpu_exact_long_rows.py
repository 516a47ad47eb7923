"""Exact (k,2)-cores of graphs with rows on both sides of the length that the peel's
searches read by the whole CTA (512), searches that stop early among them, against
the oracle."""
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


@pytest.mark.parametrize("n,hubs,avg", [(2500, (511, 512, 513), 4), (1400, (1025, 600, 512), 6),
                                        (3001, (2047, 1300, 900, 700, 512, 511), 3)])
def test_rows_around_the_whole_cta_length(ctx, n, hubs, avg):
    rp, cl = gg.with_hubs(n, hubs, 19, avg_deg=avg)
    assert (np.diff(rp) >= 512).sum() >= len(hubs) - 1
    want, wround, steps = O.core_exact(rp, cl, 2)
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        for _ in range(2):  # the second peel replays the captured rounds
            assert np.array_equal(K.kh_core_exact(G), want)
            ro, rounds, _ = K.kh_peel_info(G)
            assert np.array_equal(ro, wround) and rounds == steps
    finally:
        G.close()
