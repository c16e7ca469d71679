"""complex128 graphene sweeps start with programmatic dependent launch, each waiting for the one before ahead
of its first access to global memory: propagations and gradients, hundreds of sweeps that write over one
another's vectors, are the same bits with and without it."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("cells", [(40, 30), (300, 170), (700, 500)])
def test_dependent_launch_changes_no_bit(monkeypatch, cells):
    n = 4 * cells[0] * cells[1]
    V0 = torch.from_numpy(W.disorder_potential(n, 0.4, 5)).cuda()
    psi0 = torch.from_numpy(W.gaussian_block(n, 1, 2)[:, 0]).cuda()
    psi0 /= torch.linalg.norm(psi0)
    mask = (torch.arange(n, device="cuda") % 7 < 3).to(torch.float64)
    out = {}
    for off in ("0", "1"):
        monkeypatch.setenv("PVSC_NO_PDL", off)
        lat = pv.Lattice.graphene(cells, (1, 0), V=V0)
        y = pv.cheb_propagate(lat, psi0.clone().reshape(n, 1), 1.0, 6, 3.4, 0.1)
        V, psi = V0.clone().requires_grad_(True), psi0.clone().requires_grad_(True)
        end = pv.propagate_with_grad(V, psi, lat, 1.0, 6, 3.4, 0.1, every=3)
        gV, gpsi = torch.autograd.grad((end.abs() ** 2 * mask).sum(), (V, psi))
        out[off] = [t.detach().cpu().numpy() for t in (y, end, gV, gpsi)]
    for a, b in zip(out["0"], out["1"]):
        assert np.array_equal(a, b)
