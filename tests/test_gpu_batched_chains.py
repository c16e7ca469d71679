"""An untuned batch of large lattices runs as chains of sweeps beside one another; a work buffer of
the persistent launch's size still gets that launch.  The vectors are the same bit for bit, the
moments differ in the order of at most 2432 fp64 row sums (< 1e-12)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("dims,R", [([(33, 30, 25), (40, 36, 20), (50, 41, 3), (64, 64, 40)], 16),
                                    ([(90, 60, 60), (5, 4, 3)], 4), ([(64, 65, 66)], 1)])
def test_chains_of_an_untuned_batch_equal_the_persistent_launch(dims, R):
    n, M = len(dims), 13
    lats = [pv.Lattice.ti(d, (1, 0, 1), disorder=(1.5, i)) for i, d in enumerate(dims)]
    args = dict(R=R, prec=pv.C64, seeds=list(range(7, 7 + n)))
    a, b = [10.0] * n, [0.1] * n
    nb = pv.batched_work_bytes(lats, R, pv.C64, M)
    mu = pv.kpm_moments_batched(lats, M, a, b, **args)
    again = pv.kpm_moments_batched(lats, M, a, b, **args)
    lats[0].set_tuning(R, pv.C64, threads=256, kernel=0)
    small = pv.batched_work_bytes(lats, R, pv.C64, M)
    ref = pv.kpm_moments_batched(lats, M, a, b, **args)
    fresh = [pv.Lattice.ti(d, (1, 0, 1), disorder=(1.5, i)) for i, d in enumerate(dims)]
    tight = pv.kpm_moments_batched(fresh, M, a, b, work=pv.work_buffer(small), **args)
    assert small <= nb and torch.equal(mu, again)
    assert torch.max(torch.abs(mu - ref)).item() < 1e-12
    assert torch.max(torch.abs(tight - ref)).item() < 1e-12
    assert pv.device_error() == 0
