"""complex128 TI sweeps form the hopping sum from integers aligned to the largest of a part's twelve
inputs.  Every real part of H x is compared with the exact rational sum: the aligned sum is off by
at most 12 * 2**-58 of twice the largest input, its conversion and the two fused operations of the
update round once each, so the error is below 4 * 2**-53 of the sum of the absolute values of the
thirteen terms (an fp64 sum of them may lose 12 * 2**-53), whatever the scales of the others."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

pv = pytest.importorskip("paper_1708_09689_gb300")

U = 2.0 ** -53


def _block(kind, shape, rng):
    x = rng.standard_normal(shape + (2,))
    if kind == "scales":
        x *= 2.0 ** rng.integers(-45, 46, x.shape)
    elif kind == "far":  # more than 64 binary places apart
        x *= 2.0 ** (70.0 * rng.integers(-3, 4, x.shape))
    elif kind == "sparse":
        x *= rng.integers(0, 4, x.shape) == 0
    elif kind == "real":
        x[..., 1] = 0.0
    elif kind == "tiny":  # below the exponents that are aligned
        x *= 1e-300
    elif kind == "subnormal":
        x = np.ldexp(rng.integers(-9, 10, x.shape).astype(np.float64), -1074)
    elif kind == "huge":
        x *= 2.0 ** 900
    elif kind == "integers":  # exact in fp64
        x = rng.integers(-2 ** 30, 2 ** 30, x.shape).astype(np.float64)
    return x[..., 0] + 1j * x[..., 1]


def _check_rows(H, x, y, rows, r):
    for row in rows:
        lo, hi = H.indptr[row], H.indptr[row + 1]
        re = im = Fraction(0)
        mag_re = mag_im = 0.0
        for c, h in zip(H.indices[lo:hi], H.data[lo:hi]):
            v = x[c, r]
            pr = [Fraction(h.real) * Fraction(v.real), -Fraction(h.imag) * Fraction(v.imag)]
            pi = [Fraction(h.real) * Fraction(v.imag), Fraction(h.imag) * Fraction(v.real)]
            re += sum(pr)
            im += sum(pi)
            mag_re += float(sum(map(abs, pr)))
            mag_im += float(sum(map(abs, pi)))
        for got, ref, mag in ((y[row, r].real, re, mag_re), (y[row, r].imag, im, mag_im)):
            assert abs(Fraction(float(got)) - ref) <= 4 * U * mag + 8 * 2.0 ** -1074, (row, got, float(ref), mag)


@pytest.mark.parametrize("kind", ["normal", "scales", "far", "sparse", "real", "tiny", "subnormal", "huge", "integers"])
@pytest.mark.parametrize("dims,per,R", [((4, 3, 5), (1, 0, 1), 2), ((64, 48, 30), (0, 1, 1), 4)])
def test_each_part_of_the_hopping_sum(kind, dims, per, R):
    n = int(np.prod(dims))
    V = W.disorder_potential(n, 1.0, 2)
    lat = pv.Lattice.ti(dims, per, V=V)
    H = O.ti_hamiltonian(dims, per, 1.0, 2.0, V)
    rng = np.random.default_rng(17)
    x = _block(kind, (4 * n, R), rng)
    y = pv.apply_H(lat, torch.from_numpy(x).cuda()).cpu().numpy()
    rows = range(4 * n) if n < 100 else rng.integers(0, 4 * n, 300)
    _check_rows(H, x, y, rows, R - 1)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("dims,R", [((4, 3, 5), 1), ((64, 48, 30), 4)])
def test_non_finite_values_stay_at_their_neighbours(bad, dims, R):
    n = int(np.prod(dims))
    lat = pv.Lattice.ti(dims, (1, 1, 1))
    H = O.ti_hamiltonian(dims, (1, 1, 1), 1.0, 2.0, np.zeros(n))
    x = _block("normal", (4 * n, R), np.random.default_rng(3))
    col = 4 * (n // 2) + 1
    x[col, 0] = complex(bad, 0.5)
    y = pv.apply_H(lat, torch.from_numpy(x).cuda()).cpu().numpy()
    touched = np.zeros((4 * n, R), dtype=bool)
    touched[H.T.tocsr().indices[H.T.tocsr().indptr[col]:H.T.tocsr().indptr[col + 1]], 0] = True
    assert np.all(np.isfinite(y[~touched])) and not np.any(np.isfinite(y[touched]))
    clean = x.copy()
    clean[col, 0] = 0.0
    ref = H @ clean
    assert np.max(np.abs((y - ref)[~touched])) < 1e-13
