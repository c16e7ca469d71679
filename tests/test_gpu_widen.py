"""Accumulating complex64 sweeps add fp32 sums to an fp64 accumulator through a conversion made of
integer operations.  With H = 0 the Chebyshev vectors are x, 0, -x, 0, x, 0, -x, 0, and with the weights
1, 1, 1, 1, 3, 1, 1, 1 the touches add x, 2 x and -x: 2 x in all, exactly, where x has few bits (every
product and sum is then representable), down to the smallest subnormal numbers and zero."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("dims", [(4, 3, 2), (32, 32, 9)])
@pytest.mark.parametrize("R", [1, 4, 32])
@pytest.mark.parametrize("kernel", [None, 0, 1, 7])
def test_zero_subnormal_and_extreme_values_reach_the_accumulator(dims, R, kernel):
    lat = pv.Lattice.ti(dims, (1, 1, 1), t=0.0, m=0.0)
    if kernel is not None:
        lat.set_tuning(R, pv.C64, kernel=kernel)
    exps = np.concatenate([[0.0], np.ldexp(1.0, np.arange(-149, 124)), np.arange(1, 8) * 2.0**-149,
                           np.array([5, 2**20 + 1]) * 2.0**-149, [(2.0 - 2.0**-20) * 2.0**-127]])
    vals = np.concatenate([exps, -exps])
    rng = np.random.default_rng(4)
    x = (rng.choice(vals, (lat.D, R)) + 1j * rng.choice(vals, (lat.D, R))).astype(np.complex128)
    assert np.array_equal(x.astype(np.complex64).astype(np.complex128), x)
    y = pv.cheb_filter(lat, torch.from_numpy(x).cuda(), [1, 1, 1, 1, 3, 1, 1, 1], 1.0, 0.0, prec=pv.C64)
    assert np.array_equal(y.cpu().numpy(), 2.0 * x)
