"""Which kernels untuned calls take (pvsc_debug_route), at the sizes at which the tests of the staged tiles and
of the batch's chains compare them with the register sweeps and the persistent launch: all but one of those run
them, complex128 blocks of 32 vectors, which are compared here."""
import pytest
import torch

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")


# more than 2^16 (TI) or 2^17 (Weyl) site-vectors; tiles of 32x32, 32x16, 16x16, 16x8, 8x8 for R = 1 .. 16 at least
# half full (Weyl, R >= 8 and at most 2^21: 0.85)
@pytest.mark.parametrize("model,dims,tiles", [("ti", (61, 45, 30), (1, 2, 4, 8, 16, 32)), ("ti", (50, 33, 51), (2, 4, 8, 16, 32)),
                                              ("ti", (127, 96, 7), (1, 2, 4, 8, 16, 32)), ("ti", (36, 65, 41), (4, 8, 16, 32)),
                                              ("ti", (16, 16, 16), (32,)), ("wsm", (62, 45, 30), (2, 4, 8, 16, 32))])
def test_complex64(model, dims, tiles):
    lat = getattr(pv.Lattice, model)(dims, (1, 0, 1))
    got = tuple(R for R in (1, 2, 4, 8, 16, 32) if pv.debug_route(lat, R, pv.C64) == 7)
    assert got == tiles


@pytest.mark.parametrize("dims,R,route", [((61, 45, 30), 16, 7), ((50, 33, 51), 32, 0), ((127, 96, 7), 64, 7),
                                          ((90, 72, 41), 4, 7), ((66, 64, 33), 8, 7), ((129, 128, 66), 1, 7),
                                          ((112, 96, 50), 2, 7), ((64, 64, 32), 4, 0), ((101, 87, 119), 1, 0)])
def test_complex128(dims, R, route):
    assert pv.debug_route(pv.Lattice.ti(dims, (1, 0, 1)), R, pv.C128) == route


def test_complex128_blocks_of_32_vectors_equal_the_march():
    dims, R, per = (50, 38, 45), 32, (0, 1, 0)
    lat, ref = (pv.Lattice.ti(dims, per, disorder=(1.5, 4), delta1=0.3) for _ in range(2))
    ref.set_tuning(R, pv.C128, threads=128, kernel=0)
    assert pv.debug_route(lat, R, pv.C128) == 7 and pv.debug_route(ref, R, pv.C128) == 0
    x, y = (pv.random_vectors(lat, R, pv.C128, s) for s in (1, 2))
    out = []
    for l in (lat, ref):
        y1 = y.clone()
        d = pv.cheb_step(l, x, y1, [0.2] * R, [0.1] * R, [-0.7] * R, dots=7)
        f = pv.cheb_series(l, x, [0.5, 0.3j, 0.2, 0.1, -0.4 + 0.1j, 0.6, 0.1], 10.0, 0.1)
        out.append((pv.apply_H(l, x), y1, f, d, pv.kpm_moments(l, 9, 10.0, 0.1, r0=x)))
    for a, b in list(zip(*out))[:3]:
        assert torch.equal(a, b)
    for a, b in list(zip(*out))[3:]:  # the order of at most 2432 fp64 row sums
        assert torch.max(torch.abs(a - b)).item() < 1e-12


@pytest.mark.parametrize("dims,R,chains", [([(33, 30, 25), (40, 36, 20), (50, 41, 3), (64, 64, 40)], 16, True),
                                           ([(90, 60, 60), (5, 4, 3)], 4, True), ([(64, 65, 66)], 1, True),
                                           ([(64, 64, 63)], 1, False), ([(20, 20, 20), (24, 24, 24)], 16, False)])
def test_batches(dims, R, chains):
    lats = [pv.Lattice.ti(d, (1, 0, 1)) for d in dims]
    nb = pv.batched_work_bytes(lats, R, pv.C64, 13)
    assert pv.debug_batched_route(lats, R, pv.C64, nb) is chains
    assert not pv.debug_batched_route(lats, R, pv.C64, 4096)
    assert not pv.debug_batched_route(lats, R, pv.C128, nb * 4)
    lats[0].set_tuning(R, pv.C64, threads=256, kernel=0)
    assert not pv.debug_batched_route(lats, R, pv.C64, nb)
