"""A scheduled request that reaches max_iter before its shifts have stopped
fails with SSQCD_ERR_NOCONV, and the server goes on."""
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu


# within the chunks in flight at the start, a whole number of chunks of sixteen iterations, and not
@pytest.mark.parametrize("max_iter", [5, 16, 40, 160, 203])
def test_request_that_reaches_max_iter(max_iter):
    ss = gpu_module()
    dims = (4, 4, 4, 4)
    lat = ss.create_lattice(dims, 0.13, -1)
    ss.upload_gauge(lat, synthetic.gauge_field(dims, "haar", seed=1))
    src = synthetic.gaussian_sources(dims, 2, seed=100)
    srv = ss.Server()
    rid = srv.submit(lat, (0.374, 0.3930), 16, 8, src, beta=0.3, nprime=14, max_iter=max_iter)
    for _ in range(1000):
        srv.progress(wait=True)
        if srv.status(rid)[0] != srv.RUNNING:
            break
    assert srv.status(rid)[0] == srv.FAILED
    try:
        code = srv.take(rid).status
    except ss.SsqcdError as e:
        code = e.code
    assert code == ss.ERR_NOCONV
    assert srv.counts() == (0, 0, 0)
    srv.close()
