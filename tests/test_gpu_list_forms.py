"""The forms a list and a union can take in the level recursion, each against
the oracle: dense lists (bitmap words, balls above n/32), the hash form of the
union (more than 131072 positions at its starting level) with and without
compactions, levels that fall during a peel (the union is done again from its
lowest level), hubs in parts on both sides of the part sizes, and batches whose
graphs have positions of their own."""
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


def load(ctx, rp, cl, h, M, seed=3):
    G = K.kh_graph_load_csr(ctx, rp, cl)
    K.kh_set_h(G, h)
    K.kh_set_sampling(G, seed=seed, M=M)
    return G


# n, h, M: dense lists of one word to hundreds, with ragged last words; M below
# and above n; the hash form (n = 140k, 200k) with M at the largest 4096-slot
# table (1638) and one above it
@pytest.mark.parametrize("make,h,M", [
    (lambda: gg.erdos_renyi(6001, 30005, 5), 3, 535), (lambda: gg.erdos_renyi(6001, 30005, 5), 4, 64),
    (lambda: gg.erdos_renyi(333, 1500, 6), 4, 40), (lambda: gg.erdos_renyi(333, 1500, 6), 3, 400),
    (lambda: gg.star(95), 2, 7), (lambda: gg.rmat(11, 16, 0.57, 0.19, 0.19, 9), 4, 100),
    (lambda: gg.with_hubs(140001, (9000, 3000, 2049, 2048, 513), 21), 2, 1638),
    (lambda: gg.with_hubs(140001, (9000, 3000, 2049, 2048, 513), 21), 2, 1639),
    (lambda: gg.with_hubs(200001, (6000, 5000), 22), 3, 97)])
def test_estimates(ctx, make, h, M):
    rp, cl = make()
    G = load(ctx, rp, cl, h, M)
    try:
        want = O.estimate_dp(rp, cl, O.ranks(rp.size - 1, 3), h, M)
        for x, y in zip(K.kh_estimate(G), want):
            assert np.array_equal(x, y)
    finally:
        G.close()


@pytest.mark.parametrize("make,h,M", [
    (lambda: gg.erdos_renyi(1501, 6003, 5), 3, 100), (lambda: gg.erdos_renyi(1501, 6003, 5), 4, 9),
    (lambda: gg.with_hubs(6001, (4097, 2049, 2048), 23), 3, 33),
    (lambda: gg.rmat(10, 16, 0.57, 0.19, 0.19, 9), 3, 61)])
def test_cores_with_falling_levels(ctx, make, h, M):
    rp, cl = make()
    G = load(ctx, rp, cl, h, M)
    try:
        want, wround, steps = O.core_sampled(rp, cl, O.ranks(rp.size - 1, 3), h, M)
        core = K.kh_core_sampled(G)
        ro, rounds, _ = K.kh_peel_info(G)
        assert np.array_equal(core, want) and np.array_equal(ro, wround) and rounds == steps
    finally:
        G.close()


def test_batch_positions(ctx):
    graphs = [gg.erdos_renyi(n, 4 * n, n) for n in (33, 1000, 31, 2049)]
    off, rp, cl = gg.pack_batch(graphs)
    hs = [4, 3, 2, 4]
    G = K.kh_graph_load_batch(ctx, off, rp, cl, hs)
    K.kh_set_sampling(G, seed=3, M=50)
    try:
        est, lvl, bs = K.kh_estimate(G)
        core = K.kh_core_sampled(G)
        for q, (r, c) in enumerate(graphs):
            sl = slice(off[q], off[q + 1])
            rk = O.ranks(r.size - 1, 3)
            we, wl, wb = O.estimate_dp(r, c, rk, hs[q], 50)
            assert np.array_equal(est[sl], we) and np.array_equal(lvl[sl], wl) and np.array_equal(bs[sl], wb)
            assert np.array_equal(core[sl], O.core_sampled(r, c, rk, hs[q], 50)[0])
    finally:
        G.close()
