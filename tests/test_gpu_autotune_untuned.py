"""The autotuners time the untuned sweeps wherever no entry selects them (on one lattice: any Lx, complex128
tiles, a series' mix of warp counts), so tuning never leaves a lattice slower than not tuning it, and no
shape twice."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("dims,R,prec,op,offered", [
    ((64, 48, 20), 8, pv.C64, pv.OP_SERIES, True), ((64, 48, 20), 8, pv.C64, pv.OP_KPM, False),
    ((64, 48, 20), 8, pv.C64, pv.OP_APPLY, False), ((61, 45, 30), 8, pv.C64, pv.OP_KPM, True),
    ((61, 45, 30), 8, pv.C64, pv.OP_SERIES, True), ((66, 64, 33), 8, pv.C128, pv.OP_KPM, True),
    ((66, 64, 33), 8, pv.C128, pv.OP_SERIES, True), ((12, 10, 6), 2, pv.C64, pv.OP_SERIES, False)])
def test_the_untuned_sweeps_are_a_candidate(dims, R, prec, op, offered):
    lat = pv.Lattice.ti(dims, (1, 0, 1))
    cands = [tuple(sorted(c.items())) for c in pv.debug_autotune_candidates(lat, R, prec, op)]
    assert len(set(cands)) == len(cands)
    kernels = [dict(c)["kernel"] for c in cands]
    assert kernels.count(pv.UNTUNED) == int(offered)
    spread = {(dict(c)["threads"], dict(c)["tile_y"]) for c in cands
              if dict(c)["kernel"] == 7 and dict(c)["zslab"] == 0 and dict(c)["blocks_per_sm"] == 1}
    assert not spread  # automatic chunks spread anyway


def test_results_hold_whatever_wins():
    R = 16
    lat = pv.Lattice.ti((64, 48, 20), (1, 0, 1), disorder=(1.0, 3))
    x = pv.random_vectors(lat, R, pv.C128, 1)
    c = [0.5, 0.3, 0.2, 0.1, -0.4, 0.6, 0.1]
    ref = pv.cheb_series(lat, x, c, 10.0, 0.1, prec=pv.C64)
    best = lat.autotune(R, pv.C64, pv.OP_SERIES)
    assert best["time_ms"] > 0 and best["kernel"] == lat.get_tuning(R, pv.C64)["kernel"]
    # whatever the order of a shape's fp32 operations: 6 sweeps of about 20 of them, 120 * 2**-24 < 1e-5
    y = pv.cheb_series(lat, x, c, 10.0, 0.1, prec=pv.C64)
    assert (torch.linalg.norm(y - ref) / torch.linalg.norm(ref)).item() < 1e-5
    lats = [pv.Lattice.ti(d, (1, 0, 1), disorder=(1.5, i)) for i, d in enumerate([(36, 30, 25), (64, 64, 40)])]
    args = dict(R=R, prec=pv.C64, seeds=[1, 2])
    mu = pv.kpm_moments_batched(lats, 13, [10.0] * 2, [0.1] * 2, **args)
    best = pv.autotune_batched(lats, 8, [10.0] * 2, [0.1] * 2, **args)
    assert best["time_ms"] > 0 and best["kernel"] == lats[0].get_tuning(R, pv.C64)["kernel"]
    assert torch.max(torch.abs(pv.kpm_moments_batched(lats, 13, [10.0] * 2, [0.1] * 2, **args) - mu)).item() < 1e-12
