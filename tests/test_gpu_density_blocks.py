"""Spectral densities in every block size the launch picks (64, 128 and 256 threads, by the energies, the
vectors and the spectra of a call), at the blocks' edges: an energy's value does not depend on the others of
its call."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("R,M", [(1, 40), (8, 1030), (64, 33)])
@pytest.mark.parametrize("NE", [63, 64, 65, 9728, 9729, 19457, 38912, 38913, 300001])
@pytest.mark.parametrize("kernel", [pv.KERNEL_JACKSON, pv.KERNEL_LORENTZ, pv.KERNEL_NONE])
def test_each_block_size_gives_the_same_values(R, M, NE, kernel):
    g = torch.Generator(device="cuda").manual_seed(R)
    mu = torch.randn((R, M), generator=g, dtype=torch.float64, device="cuda")
    E = torch.linspace(-2.2, 2.2, NE, dtype=torch.float64, device="cuda")
    rho = pv.kpm_density(mu, E, 2.0, 0.1, kernel=kernel)
    few = torch.unique(torch.cat([torch.arange(0, min(NE, 40)), torch.arange(max(NE - 300, 0), NE),
                                  torch.randint(0, NE, (200,))])).cuda()
    assert torch.equal(rho[few], pv.kpm_density(mu, E[few], 2.0, 0.1, kernel=kernel))
    assert torch.all(rho[(E - 0.1).abs() >= 2.0] == 0)
