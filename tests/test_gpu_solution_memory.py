"""The memory that shifted_cg takes for stored residuals: runs of several
segments, runs on a device with little left, what is given back, and the bound
that the caller sets."""
import ctypes

import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu

DIMS, KAPPA, TOL = (8, 8, 8, 8), 0.12, 1e-11


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


def _system(ss, L, N, dims=DIMS):
    import torch
    lat = ss.create_lattice(dims, KAPPA, -1)
    ss.upload_gauge(lat, synthetic.gauge_field(dims, "smooth", seed=5, eps=0.3))
    v = torch.from_numpy(synthetic.gaussian_sources(dims, L, seed=6)).cuda()
    z = 0.11 + 0.1 * np.arange(N) / N + 0.01j * (-1.0) ** np.arange(N)
    return lat, v, z


def _close(y, ref, v, z):
    """Two solutions with residuals up to TOL, and the recurrence's drift."""
    import torch
    gap = torch.linalg.vector_norm((y - ref).flatten(2), dim=2)
    size = torch.linalg.vector_norm(ref.flatten(2), dim=2)
    vn = torch.linalg.vector_norm(v.flatten(1), dim=1)
    bound = 2 * TOL * vn[:, None] / torch.from_numpy(np.abs(z.imag)).to(y.device)[None] + 1e-10 * size
    return bool((gap <= bound).all())


def _trim_pool():
    """Give the idle memory of the stream-ordered pool back, so that the free memory is what a call can have."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rt = ctypes.CDLL("libcudart.so.13")
    pool = ctypes.c_void_p()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert rt.cudaMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0


@pytest.mark.parametrize("precision", ["FP64", "FP64_DFSHIFT"])
def test_bound_set_by_the_caller(ss, precision):
    L, N = 2, 8
    lat, v, z = _system(ss, L, N)
    p = getattr(ss, precision)
    code, ref, iters, _, it = ss.shifted_cg(lat, z, v, tol=TOL, precision=p)
    assert code == ss.OK and it > 400
    block = 16 * 16 * 12 * synthetic.volume(DIMS) * L
    again = ss.shifted_cg(lat, z, v, tol=TOL, precision=p)[1]
    assert bool((again == ref).all())
    # none, too little for them, segments of 12 and 20 blocks of sixteen iterations, all in one
    for nbytes in (-1, 5 * block, 13 * block, 21 * block, 200 * block):
        ss.set_residual_bytes(lat, nbytes)
        code, y, iters2, _, _ = ss.shifted_cg(lat, z, v, tol=TOL, precision=p)
        assert code == ss.OK
        assert int((iters2 - iters).abs().max()) <= 0.02 * it
        assert _close(y, ref, v, z)
    ss.set_residual_bytes(lat, 0)
    assert bool((ss.shifted_cg(lat, z, v, tol=TOL, precision=p)[1] == ref).all())


@pytest.mark.parametrize("room", [60e6, 100e6, 130e6, 160e6, 200e6, 300e6, 500e6, 1000e6])
def test_little_memory_left(ss, room):
    # y and p-hat: 510 MB, where the update form needs some 30 MB beside them; a
    # block of sixteen iterations 9 MB, its coefficients 0.5 MB
    import torch
    L, N = 2, 512
    lat, v, z = _system(ss, L, N, (6, 6, 6, 6))
    ss.set_residual_bytes(lat, -1)
    code, ref, iters, _, it = ss.shifted_cg(lat, z, v, tol=TOL)
    assert code == ss.OK
    ss.set_residual_bytes(lat, 0)
    ref, iters = ref.cpu(), iters.cpu()
    y = torch.empty((L, N, lat.V, 4, 3), dtype=torch.complex128, device="cuda")
    _trim_pool()
    free = torch.cuda.mem_get_info()[0]
    rest = torch.empty(int(free - 2 * y.nbytes - room), dtype=torch.uint8, device="cuda")
    it_d = torch.empty((L, N), dtype=torch.int32, device="cuda")
    zz = np.ascontiguousarray(z, dtype=np.complex128)
    for _ in range(2):  # and again, with what the first call left in the pool
        code = ss.lib().ssqcd_shifted_cg(lat.handle, N, zz.ctypes.data, L, v.data_ptr(), 1, 0.0, TOL, 100000, ss.FP64, 0,
                                         y.data_ptr(), it_d.data_ptr(), None, None)
        assert code == ss.OK, ss.lib().ssqcd_last_error()
        torch.cuda.synchronize()
        assert _close(y.cpu(), ref, v.cpu(), z)
    del rest


def test_memory_given_back(ss):
    import torch
    dims = (12, 12, 12, 12)
    lat, v, z = _system(ss, 4, 32, dims)
    _trim_pool()
    free = torch.cuda.mem_get_info()[0]
    code, y, _, _, it = ss.shifted_cg(lat, z, v, tol=TOL)
    assert code == ss.OK
    assert it * 16 * lat.n * 4 > 6e9  # the residuals took more than may stay
    torch.cuda.synchronize()
    left = free - torch.cuda.mem_get_info()[0]
    assert left <= y.nbytes + (4 << 30) + (600 << 20)  # the links' digits and work spaces among them


def test_segments_of_residuals_that_keep_the_fp64_sum(ss):
    # diagonal links keep the colours apart: a source of one colour leaves zeros
    # in every residual, so that each segment's FP64 sum is added to the last one's
    import torch
    L, N = 2, 8
    lat = ss.create_lattice(DIMS, 0.15, -1)
    phases = synthetic.rng(8).uniform(-1.0, 1.0, (4, synthetic.volume(DIMS), 3))
    ss.upload_gauge(lat, np.exp(1j * phases)[..., None] * np.eye(3))
    v = synthetic.gaussian_sources(DIMS, L, seed=6)
    v[:, :, :, 1:] = 0.0
    v = torch.from_numpy(v).cuda()
    z = 0.01 + 0.002 * np.arange(N) + 0.002j * (-1.0) ** np.arange(N)
    ss.set_residual_bytes(lat, -1)
    code, ref, iters, _, it = ss.shifted_cg(lat, z, v, tol=TOL)
    assert code == ss.OK and it > 300  # two segments
    block = 16 * 16 * 12 * synthetic.volume(DIMS) * L
    for nbytes in (13 * block, 200 * block):
        ss.set_residual_bytes(lat, nbytes)
        code, y, iters2, _, _ = ss.shifted_cg(lat, z, v, tol=TOL)
        assert code == ss.OK
        assert bool((y[..., 1:] == 0).all())
        assert int((iters2 - iters).abs().max()) <= 0.02 * it + 2
        assert _close(y, ref, v, z)
