"""Exact cores on both sides of the lines that the peel's searches are chosen by, against
the oracle: at h = 2 rows around the length that the whole CTA reads (512), searches
that stop early among them; at h >= 3 graphs whose balls take wide searches and
lattices and sparse graphs whose balls do not."""
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


def lattice3(a, b, c):
    idx = np.arange(a * b * c).reshape(a, b, c)
    u = [idx[:-1].ravel(), idx[:, :-1].ravel(), idx[:, :, :-1].ravel()]
    v = [idx[1:].ravel(), idx[:, 1:].ravel(), idx[:, :, 1:].ravel()]
    return gg.csr_from_edges(a * b * c, np.concatenate(u), np.concatenate(v))


@pytest.mark.parametrize("make", [lambda: lattice3(9, 8, 7), lambda: gg.grid(25, 20, 0.01, 3),
                                  lambda: gg.erdos_renyi(700, 1400, 5), lambda: gg.erdos_renyi(700, 1000, 5),
                                  lambda: gg.chung_lu(900, 3, 2.5, 60, 8)])
@pytest.mark.parametrize("h", [3, 4])
def test_searches_of_both_widths(ctx, make, h):
    rp, cl = make()
    want, wround, steps = O.core_exact(rp, cl, h)
    G = K.kh_graph_load_csr(ctx, rp, cl)
    try:
        K.kh_set_h(G, 2)
        K.kh_hdegree_exact(G)  # the arrays of a peel may come from an earlier call
        K.kh_set_h(G, h)
        for _ in range(2):
            assert np.array_equal(K.kh_core_exact(G), want)
            ro, rounds, _ = K.kh_peel_info(G)
            assert np.array_equal(ro, wround) and rounds == steps
    finally:
        G.close()
