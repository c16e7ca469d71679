"""Untuned complex64 sweeps run on the TMA-staged tiles where these pay, for any Lx (a stored
potential whose rows are no multiple of 16 bytes is kept a second time in padded rows).  The
tiles' arithmetic is the z-march's and the cell sweeps', so vectors are equal bit for bit; the
moments differ only in the order of the blocks' fp64 sums (at most 2432 rows, < 1e-12)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")

# Lx mod 4 = 1, 2, 3, 0; tiles with remainders on both axes; short and long z; all boundary mixes
SHAPES = [((61, 45, 30), (1, 0, 1)), ((50, 33, 51), (0, 1, 0)), ((127, 96, 7), (1, 1, 0)), ((36, 65, 41), (0, 0, 1))]


def _lattice(model, dims, per, pot):
    dims = (dims[0] + dims[0] % 2,) + dims[1:] if model == "wsm" else dims  # Weyl cells: an even Lx
    n = int(np.prod(dims))
    kw = {"stored": dict(V=W.disorder_potential(n, 1.5, 4)), "none": {},
          "hashed": dict(disorder=(1.5, 4), on_the_fly=True)}[pot]
    if model == "ti" and pot == "stored":
        kw["delta1"] = 0.3
    return (pv.Lattice.ti if model == "ti" else pv.Lattice.wsm)(dims, per, **kw)


@pytest.mark.parametrize("dims,per", SHAPES)
@pytest.mark.parametrize("R", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("model", ["ti", "wsm"])
@pytest.mark.parametrize("pot", ["stored", "none", "hashed"])
def test_default_sweeps_equal_the_march(dims, per, R, model, pot):
    lat, ref = _lattice(model, dims, per, pot), _lattice(model, dims, per, pot)
    ref.set_tuning(R, pv.C64, threads=128, kernel=0)
    x = pv.random_vectors(lat, R, pv.C64, 1)
    y = pv.random_vectors(lat, R, pv.C64, 2)
    z = pv.random_vectors(lat, R, pv.C64, 3)
    out = []
    for l in (lat, ref):
        h = pv.apply_H(l, x)
        y1, z1 = y.clone(), z.clone()
        d = pv.cheb_step(l, x, y1, [0.2] * R, [0.1] * R, [-0.7] * R, z1, [0.3] * R, dots=7)
        f = pv.cheb_series(l, x.to(torch.complex128), [0.5, 0.3, 0.2, 0.1, -0.4, 0.6, 0.1], 10.0, 0.1, prec=pv.C64)
        mu = pv.kpm_moments(l, 9, 10.0, 0.1, r0=x)
        out.append((h, y1, z1, f, d, mu))
    a, b = out
    for k in range(4):
        assert torch.equal(a[k], b[k]), k
    assert torch.max(torch.abs(a[4] - b[4])).item() < 1e-12
    assert torch.max(torch.abs(a[5] - b[5])).item() < 1e-12
    assert pv.device_error() == 0


# at least 2^20 site-vectors; odd Lx (potential read per site), remainders, slices of 8 vectors
@pytest.mark.parametrize("dims,per,R", [((61, 45, 30), (1, 0, 1), 16), ((50, 33, 51), (0, 1, 0), 32),
                                        ((127, 96, 7), (1, 1, 0), 64), ((90, 72, 41), (0, 0, 1), 4),
                                        ((66, 64, 33), (1, 1, 1), 8), ((129, 128, 66), (0, 1, 1), 1),
                                        ((112, 96, 50), (1, 0, 0), 2)])
@pytest.mark.parametrize("pot", ["stored", "none", "hashed"])
def test_default_complex128_sweeps_equal_the_march(dims, per, R, pot):
    lat, ref = _lattice("ti", dims, per, pot), _lattice("ti", dims, per, pot)
    ref.set_tuning(R, pv.C128, threads=128, kernel=0)
    x = pv.random_vectors(lat, R, pv.C128, 1)
    y = pv.random_vectors(lat, R, pv.C128, 2)
    z = pv.random_vectors(lat, R, pv.C128, 3)
    out = []
    for l in (lat, ref):
        h = pv.apply_H(l, x)
        y1, z1 = y.clone(), z.clone()
        d = pv.cheb_step(l, x, y1, [0.2] * R, [0.1] * R, [-0.7] * R, z1, [0.3] * R, dots=7)
        f = pv.cheb_series(l, x, [0.5, 0.3j, 0.2, 0.1, -0.4 + 0.1j, 0.6, 0.1], 10.0, 0.1)
        mu = pv.kpm_moments(l, 9, 10.0, 0.1, r0=x)
        out.append((h, y1, z1, f, d, mu))
    a, b = out
    for k in range(4):
        assert torch.equal(a[k], b[k]), k
    assert torch.max(torch.abs(a[4] - b[4])).item() < 1e-12
    assert torch.max(torch.abs(a[5] - b[5])).item() < 1e-12
    assert pv.device_error() == 0


def test_new_potential_reaches_the_padded_rows():
    dims, R = (61, 45, 30), 4
    lat = pv.Lattice.ti(dims, (1, 0, 1))
    x = pv.random_vectors(lat, R, pv.C64, 1)
    pv.apply_H(lat, x)
    V = torch.from_numpy(W.disorder_potential(lat.n_sites, 2.0, 9)).cuda()
    for v in (V, 2.0 * V):
        lat.set_potential(v)
        ref = pv.Lattice.ti(dims, (1, 0, 1), V=v)
        ref.set_tuning(R, pv.C64, threads=128, kernel=0)
        assert torch.equal(pv.apply_H(lat, x), pv.apply_H(ref, x))
