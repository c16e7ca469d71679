"""A tuning that is read back selects the same sweeps when it is set again, on the same lattice or an
identical one, tuned or not: equal route, equal moments bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")

# (model, dims, R, precision, route without an entry)
CASES = [("ti", (64, 48, 20), 4, pv.C64, 7), ("ti", (61, 45, 30), 8, pv.C64, 7), ("ti", (12, 10, 6), 2, pv.C64, 0),
         ("ti", (66, 64, 33), 8, pv.C128, 7), ("ti", (16, 16, 16), 1, pv.C128, 0),
         ("wsm", (64, 32, 32), 16, pv.C64, 7), ("wsm", (8, 6, 5), 4, pv.C64, 1), ("wsm", (48, 20, 20), 4, pv.C128, 1),
         ("graphene", (60, 40), 2, pv.C64, 0), ("graphene", (60, 40), 2, pv.C128, 0)]


def _lattice(model, dims):
    if model == "graphene":
        return pv.Lattice.graphene(dims, (1, 0))
    return getattr(pv.Lattice, model)(dims, (1, 0, 1), disorder=(1.0, 3))


def _shape(lat, R, prec):
    return {k: v for k, v in lat.get_tuning(R, prec).items() if k != "time_ms"}


@pytest.mark.parametrize("model,dims,R,prec,route", CASES)
def test_setting_what_was_read_changes_nothing(model, dims, R, prec, route):
    lat, same = _lattice(model, dims), _lattice(model, dims)
    assert pv.debug_route(lat, R, prec) == route
    shape = _shape(lat, R, prec)
    mu = pv.kpm_moments(lat, 12, 10.0, 0.1, R=R, prec=prec, seed=4)
    for l in (lat, same):
        l.set_tuning(R, prec, **shape)
        assert pv.debug_route(l, R, prec) == route and _shape(l, R, prec) == shape
        assert torch.equal(pv.kpm_moments(l, 12, 10.0, 0.1, R=R, prec=prec, seed=4), mu)
    lat.set_tuning(R, prec, threads=64, zslab=2)
    lat.set_tuning(R, prec, **shape)
    assert torch.equal(pv.kpm_moments(lat, 12, 10.0, 0.1, R=R, prec=prec, seed=4), mu)


def test_the_untuned_winner_of_an_autotuner(tmp_path, monkeypatch):
    R, cache = 8, tmp_path / "tune"
    monkeypatch.setenv("PVSC_TUNE_CACHE", str(cache))
    dims = (61, 45, 30)
    _lattice("ti", dims).autotune(R, pv.C64)
    key = cache.read_text().split("|")[0]
    cache.write_text(f"{key}|0 0 0 0.5 0 0 0 0\n")  # an untuned winner, as cache files hold it
    lat, same = _lattice("ti", dims), _lattice("ti", dims)
    best = lat.autotune(R, pv.C64)
    assert best.pop("time_ms") == 0.5 and best == _shape(lat, R, pv.C64)
    same.set_tuning(R, pv.C64, threads=128)
    same.set_tuning(R, pv.C64, **best)
    assert pv.debug_route(lat, R, pv.C64) == pv.debug_route(same, R, pv.C64) == 7


def test_a_batch_keeps_its_form():
    R, M = 16, 13
    lats = [_lattice("ti", d) for d in ((33, 30, 25), (50, 41, 30), (64, 64, 40))]
    nb = pv.batched_work_bytes(lats, R, pv.C64, M)
    assert pv.debug_batched_route(lats, R, pv.C64, nb)
    shape = _shape(lats[0], R, pv.C64)
    mu = pv.kpm_moments_batched(lats, M, [10.0] * 3, [0.1] * 3, R=R, prec=pv.C64)
    lats[0].set_tuning(R, pv.C64, **shape)
    assert pv.batched_work_bytes(lats, R, pv.C64, M) == nb and pv.debug_batched_route(lats, R, pv.C64, nb)
    assert torch.equal(pv.kpm_moments_batched(lats, M, [10.0] * 3, [0.1] * 3, R=R, prec=pv.C64), mu)


def test_other_kernel_numbers_stay_refused():
    lat = _lattice("ti", (16, 16, 8))
    for kernel in (-2, 9):
        with pytest.raises(pv.PvscError):
            lat.set_tuning(4, pv.C64, kernel=kernel)
    with pytest.raises(pv.PvscError):
        lat.set_tuning(4, pv.Q64, threads=128, vpt=1, kernel=-1)
