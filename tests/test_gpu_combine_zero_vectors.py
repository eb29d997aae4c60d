"""Vectors of zeros have no share in a combination, however large their
coefficients: the other vectors' sum keeps its bits."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("large", [1e3, 1e60, 1e300])
@pytest.mark.parametrize("M", [4, 12])
def test_zero_vector_with_a_large_coefficient(large, M):
    ss = gpu_module()
    dims, L, N = (8, 8, 8, 8), 1, 48
    g = synthetic.rng(7)
    V = synthetic.volume(dims)
    y = g.standard_normal((L, N, V, 4, 3)) + 1j * g.standard_normal((L, N, V, 4, 3))
    y[:, [0, 20]] = 0.0
    t = np.linspace(-1, 1, N)
    w, zeta = np.exp(0.3j * t), t + 0.3j * (-1.0) ** np.arange(N)
    w[[0, 20]] = large * (1 - 0.5j)
    lat = ss.create_lattice(dims, 0.12, -1)
    got = ss.moments(lat, w, zeta, y, M)
    coef = w[:, None] * zeta[:, None] ** np.arange(M)
    keep = [j for j in range(N) if j not in (0, 20)]
    ref = np.einsum("jm,ljvsc->lmvsc", coef[keep], y[:, keep])
    size = np.einsum("jm,ljvsc->lmvsc", np.abs(coef[keep]), np.abs(y[:, keep]))
    # FP64 sums of N terms, or the fixed point at 2^-50 of a moment's largest
    tol = (2 * N + 2 * M + 16) * 2.0 ** -53
    assert np.all(np.abs(got - ref) <= tol * size.max(axis=(2, 3, 4), keepdims=True))
