"""The hopping sum of complex128 TI sweeps on the staged tiles, which read the neighbours from shared
memory twice: every scale of values, subnormal, huge and non-finite ones, against exact rational sums at the bound
of tests/test_gpu_hop_int.py, at sites on tile edges and open and periodic boundaries."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from test_gpu_hop_int import _block, _check_rows

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")

# 2^20 site-vectors; tiles of 8x8 (R = 8, 16: the latter in slices) and 16x8 sites, remainders on both axes
CASES = [((61, 54, 40), (1, 0, 1), 8), ((45, 37, 41), (0, 1, 0), 16), ((94, 72, 40), (1, 1, 0), 4)]


def _setup(dims, per, R):
    n = int(np.prod(dims))
    V = W.disorder_potential(n, 1.0, 2)
    lat = pv.Lattice.ti(dims, per, V=V)
    assert pv.debug_route(lat, R, pv.C128) == 7
    return n, lat, O.ti_hamiltonian(dims, per, 1.0, 2.0, V)


@pytest.mark.parametrize("kind", ["normal", "scales", "far", "sparse", "real", "tiny", "subnormal", "huge", "integers"])
@pytest.mark.parametrize("dims,per,R", CASES)
def test_each_part_of_the_hopping_sum(kind, dims, per, R):
    n, lat, H = _setup(dims, per, R)
    rng = np.random.default_rng(17)
    x = _block(kind, (4 * n, R), rng)
    y = pv.apply_H(lat, torch.from_numpy(x).cuda()).cpu().numpy()
    corners = [4 * (xx + dims[0] * (yy + dims[1] * zz)) for xx in (0, 7, 8, dims[0] - 1) for yy in (0, 7, 8, dims[1] - 1)
               for zz in (0, dims[2] // 2, dims[2] - 1)]
    rows = [c + o for c in corners for o in range(4)] + list(rng.integers(0, 4 * n, 200))
    _check_rows(H, x, y, rows, 0)
    _check_rows(H, x, y, rows, R - 1)
    assert pv.device_error() == 0


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("dims,per,R", CASES[:2])
def test_non_finite_values_stay_at_their_neighbours(bad, dims, per, R):
    n, lat, H = _setup(dims, per, R)
    x = _block("normal", (4 * n, R), np.random.default_rng(3))
    T = H.T.tocsr()
    touched = np.zeros((4 * n, R), dtype=bool)
    ref_in = x.copy()
    for site, r in ((0, 0), (n // 2 + 3, R - 1)):
        col = 4 * site + 1
        x[col, r] = complex(bad, 0.5)
        ref_in[col, r] = 0.0
        touched[T.indices[T.indptr[col]:T.indptr[col + 1]], r] = True
    y = pv.apply_H(lat, torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.all(np.isfinite(y[~touched])) and not np.any(np.isfinite(y[touched]))
    assert np.max(np.abs((y - H @ ref_in)[~touched])) < 1e-13
