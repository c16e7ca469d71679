"""What a batched call without a kernel 7 entry promises, in the form that runs large batches as
chains of sweeps too: its stream is done when it returns, a wait that ran out is an error of the
call, a stream under capture is refused."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")

R, M = 16, 400


def _batch():
    dims = [(48, 44, 40), (36, 52, 41), (57, 40, 40)]
    lats = [pv.Lattice.ti(d, (1, 0, 1), disorder=(1.5, i)) for i, d in enumerate(dims)]
    mu = torch.empty((3, R, M), dtype=torch.float64, device="cuda")
    work = pv.work_buffer(pv.batched_work_bytes(lats, R, pv.C64, M))
    return lats, dict(a=[10.0] * 3, b=[0.1] * 3, R=R, prec=pv.C64, seeds=[5, 6, 7], mu=mu, work=work)


@pytest.mark.parametrize("side", [False, True])
def test_the_stream_is_done_when_the_call_returns(side):
    lats, args = _batch()
    stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
    torch.cuda.synchronize()
    for _ in range(3):
        pv.kpm_moments_batched(lats, M, stream=stream, **args)
        assert stream.query()


def test_a_wait_that_ran_out_is_an_error_of_the_call():
    lats, args = _batch()
    ref = pv.kpm_moments_batched(lats, M, **args).clone()
    pv.inject_stall(True)
    try:
        with pytest.raises(pv.PvscError) as e:
            pv.kpm_moments_batched(lats, M, **args)
        assert e.value.code == pv.PVSC_ERR_TIMEOUT
    finally:
        pv.inject_stall(False)
    assert torch.equal(pv.kpm_moments_batched(lats, M, **args), ref)
    assert pv.device_error() == 0


def test_a_stream_under_capture_is_refused():
    lats, args = _batch()
    ref = pv.kpm_moments_batched(lats, M, **args).clone()
    g = torch.cuda.CUDAGraph()
    with pytest.raises(pv.PvscError):
        with torch.cuda.graph(g):
            pv.kpm_moments_batched(lats, M, **args)
    assert torch.equal(pv.kpm_moments_batched(lats, M, **args), ref)
