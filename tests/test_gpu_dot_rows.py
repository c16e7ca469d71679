"""cheb_step's dot products: a kernel after the sweep sums the rows its blocks left and writes
the selected outputs only.  The reference is the fp64 sum over the vectors the call returns.  fp64
vectors: at most 2**21 terms in any order, 2**21 * 2**-53 < 2.4e-10 of the terms' magnitudes in the
worst case; summed pairwise over blocks and threads it is below 1e-12.  fp32 vectors: at most 64
products are summed in fp32 before fp64, 64 * 2**-24 < 4e-6."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


@pytest.mark.parametrize("model,dims", [("ti", (2, 2, 2)), ("ti", (33, 5, 7)), ("ti", (64, 64, 20)),
                                        ("wsm", (16, 17, 9)), ("graphene", (3, 2)), ("graphene", (250, 90))])
@pytest.mark.parametrize("R", [1, 2, 16, 64])
@pytest.mark.parametrize("prec", [pv.C128, pv.C64])
@pytest.mark.parametrize("tuning", [None, dict(kernel=1), dict(kernel=7)])
def test_selected_dots_of_a_step(model, dims, R, prec, tuning):
    lat = pv.Lattice.graphene(dims, (1, 1)) if model == "graphene" else getattr(pv.Lattice, model)(
        dims, (1, 1, 0), disorder=(0.7, 11))
    if tuning is not None:
        if model == "graphene" or (tuning["kernel"] == 7 and (prec == pv.C128 or dims[0] % 4)):
            pytest.skip("no such kernel here")
        lat.set_tuning(R, prec, **tuning)
    x = pv.random_vectors(lat, R, prec, 1)
    y0 = pv.random_vectors(lat, R, prec, 2)
    work = pv.work_buffer(lat.work_bytes(pv.OP_CHEB_STEP, R, prec))
    tol = 1e-12 if prec == pv.C128 else 1e-5
    for flags in (1, 2, 4, 5, 7):
        y = y0.clone()
        out = torch.full((4, R), np.nan, dtype=torch.float64, device="cuda")
        ptr = [ctypes.c_void_p(t.data_ptr()) for t in (x, y, out, work)]
        coef = [(ctypes.c_double * R)(*[c] * R) for c in (0.3, 0.1, -0.9)]
        rc = pv.lib().pvsc_cheb_step(lat.handle, R, prec, ptr[0], ptr[1], None, *coef, None, flags, ptr[2], ptr[3],
                                     work.numel(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        xd, yd = x.to(torch.complex128).reshape(-1, R), y.to(torch.complex128).reshape(-1, R)
        xx, yy = (xd.abs() ** 2).sum(0), (yd.abs() ** 2).sum(0)
        xy = (yd.conj() * xd).sum(0)
        for d, (bit, ref) in enumerate(((1, xx), (2, xy.real), (2, xy.imag), (4, yy))):
            if flags & bit:
                assert torch.max((out[d] - ref).abs() / torch.sqrt(xx * yy)).item() < tol, (flags, d)
            else:
                assert torch.isnan(out[d]).all(), (flags, d)
