"""complex128 graphene sweeps, one value per thread: every sweep kind against the oracle at block
edges, single rows and columns (periodic lengths 1 and 2), blocks of several vectors."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("cells,per", [((1, 1), (1, 1)), ((2, 1), (1, 0)), ((1, 2), (0, 1)), ((7, 9), (0, 0)),
                                       ((16, 4), (1, 1)), ((65, 3), (1, 0))])
@pytest.mark.parametrize("R", [1, 2, 16])
def test_apply_and_series_match_the_oracle(cells, per, R):
    n = 4 * cells[0] * cells[1]
    V = W.disorder_potential(n, 0.7, 3)
    lat = pv.Lattice.graphene(cells, per, V=V)
    H = O.graphene_hamiltonian(cells, per, 1.0, V)
    x = W.gaussian_block(n, R, 1)
    xd = torch.from_numpy(x).cuda()
    assert np.linalg.norm(pv.apply_H(lat, xd).cpu().numpy() - H @ x) <= 1e-12 * np.linalg.norm(H @ x)
    y = xd.clone()
    pv.cheb_step(lat, xd, y, [0.3] * R, [0.1] * R, [0.7] * R)  # a general gamma
    ref = 0.3 * (H @ x - 0.1 * x) + 0.7 * x
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    a, b = 3.6, 0.05
    for K in (2, 3, 4, 5, 6, 7):  # every number of terms in the first and the last accumulator touch
        for c in ([0.3 + 0.1 * k for k in range(K)], [(0.2 + 0.1 * k) * (-1j) ** k for k in range(K)],
                  [0.2 - 0.3j + 0.1j * k for k in range(K)], [0.0] * (K - 1) + [1.0]):
            f = pv.cheb_series(lat, xd, c, a, b, phase=0.6 + 0.8j).cpu().numpy()
            ref = (0.6 + 0.8j) * O.cheb_series(H, x, c, a, b)
            assert np.linalg.norm(f - ref) <= 1e-12 * max(np.linalg.norm(ref), np.linalg.norm(x)), (K, c)
