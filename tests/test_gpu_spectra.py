"""Several spectra in one launch: the same arithmetic as one call per spectrum, around the block
(64 energies) and the chunk (1024 coefficients) of the kernel; Bloch states at every width."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("n,R,M,NE", [(1, 1, 1, 1), (3, 2, 1025, 65), (16, 4, 256, 1000), (2, 3, 1024, 64)])
@pytest.mark.parametrize("kernel", [pv.KERNEL_JACKSON, pv.KERNEL_LORENTZ, pv.KERNEL_NONE])
def test_spectra_of_one_launch_equal_one_call_each(n, R, M, NE, kernel):
    rng = np.random.default_rng(n + M)
    mu = rng.standard_normal((n * R, M))
    E = np.linspace(-2.1, 2.1, NE)
    mud, Ed = torch.from_numpy(mu).cuda(), torch.from_numpy(E).cuda()
    rho = torch.empty((n, NE), dtype=torch.float64, device="cuda")
    vp = ctypes.c_void_p
    rc = pv.lib().pvsc_kpm_spectra(n, R, M, vp(mud.data_ptr()), kernel, 4.0, 2.0, 0.1, 1.0, NE, vp(Ed.data_ptr()),
                                   vp(rho.data_ptr()), vp(torch.cuda.current_stream().cuda_stream))
    assert rc == pv.PVSC_OK
    for i in range(n):
        rows = mud[i * R:(i + 1) * R].clone()
        assert torch.equal(rho[i], pv.kpm_density(rows, Ed, 2.0, 0.1, kernel=kernel))
    if kernel == pv.KERNEL_JACKSON:
        ref = O.kpm_density(mu[:R], E, 2.0, 0.1, O.jackson_kernel(M))
        assert np.max(np.abs(rho[0].cpu().numpy() - ref)) <= 1e-12 * max(1.0, np.max(np.abs(ref)))


@pytest.mark.parametrize("nk", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("prec,tol", [(pv.C128, 1e-15), (pv.C64, 1e-8)])
def test_bloch_states_at_every_width(nk, prec, tol):
    dims = (5, 7, 3)
    ks = [(0.3 * q, -0.2 * q, 0.7) for q in range(nk)]
    psi = pv.bloch_vectors(pv.Lattice.ti(dims, (1, 1, 1)), ks, prec).cpu().numpy()
    for q, k in enumerate(ks):
        assert np.max(np.abs(psi[:, 4 * q:4 * q + 4] - O.bloch_vectors(dims, k))) < tol
