"""More sources than a grid dimension of the tensor-core combination holds."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,M", [(65539, 4, 4), (100000, 9, 3)])  # more than 8 million terms
def test_moments_of_many_sources(L, N, M):
    ss = gpu_module()
    lat = ss.create_lattice((1, 1, 1, 1), 0.12, -1)
    g = synthetic.rng(2)
    y = g.standard_normal((L, N, 1, 4, 3)) + 1j * g.standard_normal((L, N, 1, 4, 3))
    t = np.linspace(-1, 1, N)
    w, zeta = np.exp(0.3j * t), t + 0.3j * (-1.0) ** np.arange(N)
    got = ss.moments(lat, w, zeta, y, M)
    coef = w[:, None] * zeta[:, None] ** np.arange(M)
    ref = np.einsum("jm,ljvsc->lmvsc", coef, y)
    size = np.einsum("jm,ljvsc->lmvsc", np.abs(coef), np.abs(y))
    # FP64 sums of N terms, or the fixed point at 2^-50 of a source's largest
    tol = (2 * N + 2 * M + 16) * 2.0 ** -53
    assert np.all(np.abs(got - ref) <= tol * size.max(axis=(2, 3, 4), keepdims=True))
