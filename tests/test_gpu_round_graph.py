"""Cores of one graph with other calls between them: the captured rounds of a peel hold
the addresses of its arrays and its settings, and what such a call allocates again or
sets (levels, M, BFS scratch, the union's schedule) must not leave them in use.  Every
result against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2112_06154_gb300 import graphgen as gg
from paper_2112_06154_gb300 import khcore as K

pytestmark = pytest.mark.gpu

GRAPHS = {"er": lambda: gg.erdos_renyi(1501, 6003, 5),
          "hubs": lambda: gg.with_hubs(5001, (2500, 1100), 23, avg_deg=4)}  # with part slots


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    K.load(build_if_missing=True)
    c = K.kh_ctx_create(0)
    yield c
    c.close()


@pytest.fixture(params=sorted(GRAPHS))
def loaded(ctx, request):
    rp, cl = GRAPHS[request.param]()
    G = K.kh_graph_load_csr(ctx, rp, cl)
    yield rp, cl, G
    G.close()


def check_core(G, rp, cl, h, M):
    K.kh_set_h(G, h)
    K.kh_set_sampling(G, seed=1, M=M)
    want, wround, steps = O.core_sampled(rp, cl, O.ranks(rp.size - 1, 1), h, M)
    assert np.array_equal(K.kh_core_sampled(G), want)
    ro, rounds, _ = K.kh_peel_info(G)
    assert np.array_equal(ro, wround) and rounds == steps


def check_estimate(G, rp, cl, h, M):
    K.kh_set_h(G, h)
    K.kh_set_sampling(G, seed=1, M=M)
    want = O.estimate_dp(rp, cl, O.ranks(rp.size - 1, 1), h, M)
    for x, y in zip(K.kh_estimate(G), want):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("h,M", [(2, 16), (3, 24)])
def test_more_levels_between_two_cores(loaded, h, M):
    rp, cl, G = loaded
    check_core(G, rp, cl, h, M)
    check_estimate(G, rp, cl, h + 1, M)
    check_core(G, rp, cl, h, M)
    check_estimate(G, rp, cl, h + 2, M)
    check_core(G, rp, cl, h + 1, M)
    check_core(G, rp, cl, h, M)


def test_larger_slots_between_two_cores(loaded):
    rp, cl, G = loaded
    check_core(G, rp, cl, 2, 16)
    check_estimate(G, rp, cl, 2, 300)
    check_core(G, rp, cl, 2, 16)
    check_core(G, rp, cl, 2, 300)


def test_exact_and_sampled_in_turn(loaded):
    rp, cl, G = loaded
    for h in (3, 2, 3) if rp.size < 2000 else (2, 1, 2):  # (the oracle's exact cores at h = 3)
        K.kh_set_h(G, h)
        assert np.array_equal(K.kh_core_exact(G), O.core_exact(rp, cl, h)[0])
        K.kh_set_h(G, 3)
        assert np.array_equal(K.kh_hdegree_exact(G), O.hdegree_exact(rp, cl, 3))
        check_core(G, rp, cl, 2, 24)


def test_schedule_set_between_two_cores(loaded):
    rp, cl, G = loaded
    launches = []
    for mode in (K.KH_LEVELU_GROUPED, K.KH_LEVELU_FREE, K.KH_LEVELU_GROUPED):
        K.kh_set_variant(G, mode, op=K.KH_OP_LEVEL_UNION)
        check_core(G, rp, cl, 3, 24)
        before = K.kh_launch_count(G)
        check_core(G, rp, cl, 3, 24)  # nothing changed: the same rounds again
        launches.append(K.kh_launch_count(G) - before)
    assert len(set(launches)) == 1
