"""A bound on the iterations that no run reaches costs nothing: neither memory
for as many, nor a call refused."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_iter", [10 ** 6, 10 ** 9, 2 ** 31 - 1])
def test_large_max_iter(max_iter):
    import torch
    ss = gpu_module()
    dims, N, L = (8, 8, 8, 8), 8, 2
    lat = ss.create_lattice(dims, 0.125, -1)
    ss.upload_gauge(lat, synthetic.gauge_field(dims, "smooth", seed=5, eps=0.3))
    v = synthetic.gaussian_sources(dims, L, seed=6)
    z = 0.11 + 0.002 * np.arange(N) + 0.02j * (-1.0) ** np.arange(N)
    code, ref, iters, _, it = ss.shifted_cg(lat, z, v, tol=1e-10)
    assert code == ss.OK
    before = torch.cuda.mem_get_info()[0]
    code, y, iters2, _, it2 = ss.shifted_cg(lat, z, v, tol=1e-10, max_iter=max_iter)
    assert code == ss.OK and it == it2
    assert np.array_equal(y, ref) and np.array_equal(iters, iters2)
    assert before - torch.cuda.mem_get_info()[0] <= 64 << 20  # the first call's pool serves
    res = ss.ss_solve(lat, (0.105, 0.120), 16, 8, v, beta=0.6, nprime=8, max_iter=max_iter)
    assert res.status == ss.OK, res.error
