"""reliable_every belongs to the mixed precisions: the others run as without it."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu


# stored residuals (N L n = 0.8 million), updates (0.1 million)
@pytest.mark.parametrize("N,L", [(8, 2), (2, 1)])
@pytest.mark.parametrize("precision", ["FP64", "FP64_DFSHIFT", "FP64_SHIFT32"])
def test_no_effect_outside_the_mixed_precisions(precision, N, L):
    ss = gpu_module()
    dims = (8, 8, 8, 8)
    lat = ss.create_lattice(dims, 0.12, -1)
    ss.upload_gauge(lat, synthetic.gauge_field(dims, "smooth", seed=5, eps=0.3))
    v = synthetic.gaussian_sources(dims, L, seed=6)
    z = 0.11 + 0.002 * np.arange(N) + 0.02j * (-1.0) ** np.arange(N)
    out = [ss.shifted_cg(lat, z, v, tol=1e-10, precision=getattr(ss, precision), reliable_every=k) for k in (0, 32)]
    assert out[0][0] == out[1][0] == ss.OK
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])
