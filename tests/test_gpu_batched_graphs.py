"""What an untuned batch of chains keeps between calls: nothing for an argument set that comes once
(a disorder average has new seeds in every call), a captured graph for one that comes again, and at
most 4096 kernel nodes of them in all.  Enqueued, captured and replayed chains are the same launches:
equal moments bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")

DIMS = [(48, 44, 40), (36, 52, 41), (57, 40, 40)]
R = 16


def _batch(M):
    lats = [pv.Lattice.ti(d, (1, 0, 1), disorder=(1.5, i)) for i, d in enumerate(DIMS)]
    mu = torch.empty((3, R, M), dtype=torch.float64, device="cuda")
    work = pv.work_buffer(pv.batched_work_bytes(lats, R, pv.C64, M))

    def call(seed):
        return pv.kpm_moments_batched(lats, M, [10.0] * 3, [0.1] * 3, R=R, prec=pv.C64,
                                      seeds=[seed, seed + 1, seed + 2], mu=mu, work=work)
    return lats[0], call


def test_new_seeds_keep_no_graph():
    lat, call = _batch(40)
    for s in range(9):
        call(10 * s)
        assert pv.debug_graph_cache(lat) == (0, 0)


def test_a_repeated_call_replays_a_graph_with_the_same_moments():
    lat, call = _batch(41)
    first = call(3).clone()
    for s in range(3):  # others in between: the set is still among the last four
        call(100 + 10 * s)
    for _ in range(3):
        assert torch.equal(call(3), first)
        graphs, nodes = pv.debug_graph_cache(lat)
        assert graphs == 1 and nodes >= 3 * 21
    assert pv.device_error() == 0


def test_graphs_are_bounded_in_nodes():
    lat, call = _batch(1000)  # 3 x 502 kernels a call
    for s in range(4):
        call(10 * s)
        call(10 * s)
        assert 0 < pv.debug_graph_cache(lat)[1] <= 4096 + 200
    lat, call = _batch(2800)  # 3 x 1402: more than the cache holds
    a = call(1).clone()
    assert torch.equal(call(1), a) and torch.equal(call(1), a)
    assert pv.debug_graph_cache(lat) == (0, 0)
