"""A chain of KPM sweeps leaves the rows of its dot products to the next sweep; a call of one
sweep sums its own.  Both give the same moments: only the order of at most 2432 rows' sum
differs, 2432 * 2**-53 < 3e-13 of a sum of terms of total at most 1, doubled by 2 s - mu_0."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")

TI, WSM, GR = "ti", "wsm", "graphene"


def _lattice(model, dims):
    if model == GR:
        return pv.Lattice.graphene(dims[:2], (1, 0))
    make = pv.Lattice.ti if model == TI else pv.Lattice.wsm
    return make(dims, (1, 0, 1), disorder=(1.0, 3))


@pytest.mark.parametrize("model,dims", [(TI, (4, 4, 2)), (TI, (8, 12, 9)), (TI, (40, 36, 30)), (WSM, (8, 6, 5)),
                                        (WSM, (64, 30, 21)), (GR, (5, 3, 1)), (GR, (300, 170, 1))])
@pytest.mark.parametrize("R", [1, 4, 32, 64])
@pytest.mark.parametrize("prec", [pv.C128, pv.C64])
@pytest.mark.parametrize("tuning", [None, dict(kernel=1), dict(kernel=7)])
def test_chained_sweeps_equal_single_sweep_calls(model, dims, R, prec, tuning):
    lat = _lattice(model, dims)
    if tuning is not None:
        if model == GR or (tuning["kernel"] == 7 and prec == pv.C128):
            pytest.skip("no such kernel here")
        lat.set_tuning(R, prec, **tuning)
    M = 10
    r0 = pv.random_vectors(lat, R, prec, 5)
    w = [r0.clone(), torch.empty_like(r0)]
    single = torch.full((R, M), np.nan, dtype=torch.float64, device="cuda")
    for k in range(M // 2):
        pv.kpm_sweeps(lat, k, k + 1, w[0], w[1], 10.0, 0.0, single)
    w = [r0.clone(), torch.empty_like(r0)]
    parts = torch.full((R, M), np.nan, dtype=torch.float64, device="cuda")
    for k0, k1 in ((0, 2), (2, 5)):
        pv.kpm_sweeps(lat, k0, k1, w[0], w[1], 10.0, 0.0, parts)
    whole = pv.kpm_moments(lat, M, 10.0, 0.0, r0=r0)
    assert torch.max(torch.abs(single - parts)).item() < 1e-12
    assert torch.max(torch.abs(single - whole)).item() < 1e-12
