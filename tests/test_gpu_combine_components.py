"""Combinations element by element, where some elements of the vectors are far
below the others: the fixed point of the tensor-core form is relative to a
vector's largest component and to an output's largest coefficient."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 8)


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


def _vectors(kind, L, N, seed):
    g = synthetic.rng(seed)
    V = synthetic.volume(DIMS)
    y = g.standard_normal((L, N, V, 4, 3)) + 1j * g.standard_normal((L, N, V, 4, 3))
    site = (L, 1, V, 4, 3)
    if kind == "one":  # a single element
        y[:, :, V // 3, 2, 1] *= 2.0 ** -40
    elif kind == "half_percent":  # fewer than the list of such elements holds
        y *= np.where(g.random(site) < 0.005, 2.0 ** -30, 1.0)
    elif kind == "four_percent":  # more
        y *= np.where(g.random(site) < 0.04, 2.0 ** -30, 1.0)
    elif kind == "grades":  # the list's threshold among them
        y *= 2.0 ** -np.where(g.random(site) < 0.01, g.integers(0, 60, site), 0).astype(float)
    elif kind == "imaginary":  # one part of the elements only
        y = y.real + 1j * y.imag * np.where(g.random(site) < 0.005, 2.0 ** -30, 1.0)
    elif kind == "sizes":  # vectors of different sizes, zero vectors, one of them with the largest coefficient
        y *= (10.0 ** -g.integers(0, 30, N).astype(float))[None, :, None, None, None]
        y[:, [0, N // 2]] = 0.0
        y[:, :, 5] *= 2.0 ** -35
    elif kind == "real":
        y = y.real.astype(np.complex128)
    elif kind == "apart":  # the vectors with large coefficients are zero where the others are not
        y[:, : N // 2, : V // 100] = 0.0
    return y


KINDS = ["one", "half_percent", "four_percent", "grades", "imaginary", "real", "apart"]


@pytest.mark.parametrize("L,N,M", [(1, 32, 8), (2, 20, 16), (1, 70, 21), (1, 16, 12)])
@pytest.mark.parametrize("kind,coefs", [(k, c) for k in KINDS for c in ("complex", "real", "steep")] + [("sizes", "complex")])
def test_every_element(ss, kind, L, N, M, coefs):
    y = _vectors(kind, L, N, 1)
    t = np.linspace(-1, 1, N)
    w = np.exp(0.3j * t) * (1 + 0.1 * t)
    zeta = t + 0.3j * (-1.0) ** np.arange(N)
    if coefs == "real":
        w, zeta = (1.2 + t).astype(np.complex128), (0.5 + 0.4 * t).astype(np.complex128)
    elif coefs == "steep":  # over twelve decades and more
        w = w * 10.0 ** -np.linspace(0, 12, N)
    lat = ss.create_lattice(DIMS, 0.12, -1)
    got = ss.moments(lat, w, zeta, y, M)
    coef = w[:, None] * zeta[:, None] ** np.arange(M)
    ref = np.einsum("jm,ljvsc->lmvsc", coef, y)
    # a part of a result by its own terms
    re, im = np.abs(y.real), np.abs(y.imag)
    cr, ci = np.abs(coef.real), np.abs(coef.imag)
    size_re = np.einsum("jm,ljvsc->lmvsc", cr, re) + np.einsum("jm,ljvsc->lmvsc", ci, im)
    size_im = np.einsum("jm,ljvsc->lmvsc", cr, im) + np.einsum("jm,ljvsc->lmvsc", ci, re)
    # 2 N products, each rounded at 2^-54.7 of the output's scale at most (vector,
    # coefficient and the dropped levels of digits); the part's largest term is at least 2^-11 of it.
    # The reference and the powers of zeta: FP64 sums of N terms.
    tol = 2 * N * 2.0 ** -43.7 + (2 * N + 2 * M + 16) * 2.0 ** -53
    assert np.all(np.abs(got.real - ref.real) <= tol * size_re)
    assert np.all(np.abs(got.imag - ref.imag) <= tol * size_im)
    # and in the norm as FP64
    assert np.linalg.norm(got - ref) <= 4e-15 * np.linalg.norm(np.hypot(size_re, size_im))
