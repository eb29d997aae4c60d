"""A gauge field uploaded while a request on the lattice is running: the
request ends in its own way (its kernels keep valid memory, whichever links
they see), and the lattice then gives what a fresh one gives."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


@pytest.mark.parametrize("precision", ["FP64", "DF"])
def test_upload_of_other_links_during_a_request(ss, precision):
    dims, kappa, interval = (4, 4, 4, 4), 0.13, (0.374, 0.3930)
    U = synthetic.gauge_field(dims, "haar", seed=1)
    W = U.copy()
    W[1, 5] *= 1 + 2.0 ** -9  # a link that the integer stencil does not take
    src = synthetic.gaussian_sources(dims, 3, seed=100)
    lat = ss.create_lattice(dims, kappa, -1, precision=getattr(ss, precision))
    for links, other in ((U, W), (W, U)):
        ss.upload_gauge(lat, links)
        srv = ss.Server()
        # iterations that no whole number of chunks makes up
        rid = srv.submit(lat, interval, 16, 8, src, beta=0.3, nprime=14, max_iter=1003)
        srv.progress(wait=True)
        assert srv.status(rid)[0] == srv.RUNNING
        ss.upload_gauge(lat, other)
        while srv.status(rid)[0] == srv.RUNNING:
            srv.progress(wait=True)
        try:  # it may end early or late, out of two operators
            srv.take(rid)
        except ss.SsqcdError as e:
            assert e.code in (ss.ERR_NOCONV, ss.ERR_BREAKDOWN)
        srv.close()
        fresh = ss.create_lattice(dims, kappa, -1, precision=getattr(ss, precision))
        ss.upload_gauge(fresh, other)
        assert np.array_equal(ss.apply_H(lat, src), ss.apply_H(fresh, src))
        out = []
        for x in (lat, fresh):
            res = ss.ss_solve(x, interval, 16, 8, src, beta=0.3, nprime=14)
            assert res.status == ss.OK, res.error
            out.append(ss.ss_eigpairs(res, want_vectors=False)[0])
        assert np.array_equal(out[0], out[1])
