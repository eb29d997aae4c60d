"""Sources of one shifted-CG run that stop hundreds of iterations apart, one of
them at once: the counts of live shifts that its kernels read while others
change them.  Every run gives the same bits, and every source what it gives
alone."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


# groups of 16 sites x sources: four warps a group (324 of them), one (1024)
@pytest.mark.parametrize("dims", [(6, 6, 6, 6), (8, 8, 8, 8)])
def test_sources_that_stop_far_apart(ss, dims):
    kappa, tol = 0.12, 1e-12
    V = synthetic.volume(dims)
    U = np.broadcast_to(np.eye(3, dtype=np.complex128), (4, V, 3, 3)).copy()  # unit links
    v = synthetic.gaussian_sources(dims, 4, seed=3)
    # a plane wave: A^2 is a number on it, so that its recurrence ends with the second step
    t = np.arange(V) // (dims[0] * dims[1] * dims[2])
    v[1] = np.exp(1j * np.pi * t / dims[3])[:, None, None] * v[0, 0]
    v[2] = 0.0
    # a low eigenvector and little else stops between the two
    v[3] = v[1][:, ::-1] + 1e-6 * v[3]
    z = 0.05 + 0.02 * np.arange(16) + 0.03j * (-1.0) ** np.arange(16)
    lat = ss.create_lattice(dims, kappa, -1)
    ss.upload_gauge(lat, U)
    code, y, iters, _, _ = ss.shifted_cg(lat, z, v, tol=tol)
    assert code == ss.OK
    assert np.all(iters[2] == 0) and np.all(y[2] == 0)
    assert iters[1].max() <= 4 and iters[0].max() >= 10 * iters[1].max()
    A = lambda x: wilson.apply_H(U, x, kappa, dims, -1)
    for l in range(4):
        for j in range(0, 16, 5):
            r = v[l] - (z[j] * y[l, j] - A(y[l, j]))
            # the stop, and the roundings of the recurrence's steps
            drift = 8 * iters[l, j] * 2.2e-16 * 2.1 * np.linalg.norm(y[l, j])
            assert np.linalg.norm(r) <= tol * np.linalg.norm(v[l]) + drift
    for _ in range(10):
        code, y2, iters2, _, _ = ss.shifted_cg(lat, z, v, tol=tol)
        assert code == ss.OK and np.array_equal(iters, iters2) and np.array_equal(y, y2)
    for l in (0, 1, 3):
        code, y1, _, _, _ = ss.shifted_cg(lat, z, v[l:l + 1], tol=tol)
        assert code == ss.OK
        for j in range(16):  # two solutions to tol
            gap = 2 * tol * np.linalg.norm(v[l]) / abs(z[j].imag)
            assert np.linalg.norm(y1[0, j] - y[l, j]) <= gap + 1e-13 * np.linalg.norm(y[l, j])
