"""Moments written over the solutions they are formed from: the same as into a
buffer of their own, on the tensor cores and on the FP64 pipe."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic

pytestmark = pytest.mark.gpu


# 12.6 million terms (tensor cores), the same with a point-like vector (FP64), few terms (FP64)
@pytest.mark.parametrize("dims,L,N,M,point", [((8, 8, 8, 8), 2, 16, 8, False), ((8, 8, 8, 8), 2, 16, 8, True),
                                              ((4, 4, 4, 4), 3, 6, 4, False)])
@pytest.mark.parametrize("shift", [0, 1, 7])  # vectors from the solutions' start, the moments' from theirs if negative
@pytest.mark.parametrize("ahead", [False, True])
def test_moments_over_the_solutions(dims, L, N, M, point, shift, ahead):
    import torch
    ss = gpu_module()
    n = 12 * synthetic.volume(dims)
    g = torch.Generator(device="cuda").manual_seed(1)
    buf = torch.randn((L * N + 7) * n, generator=g, device="cuda", dtype=torch.complex128)
    lat = ss.create_lattice(dims, 0.12, -1)
    t = np.linspace(-1, 1, N)
    w, zeta = np.exp(0.3j * t), t + 0.3j * (-1.0) ** np.arange(N)
    w, zeta = np.ascontiguousarray(w), np.ascontiguousarray(zeta)
    at_y, at_s = (7 * n, (7 - shift) * n) if ahead else (0, shift * n)
    y = buf[at_y:at_y + L * N * n]
    if point:
        y[:n] = 0
        y[5] = 1.0
    want = ss.moments(lat, w, zeta, y.clone().reshape(L, N, -1, 4, 3), M)
    torch.cuda.synchronize()
    code = ss.lib().ssqcd_moments(lat.handle, N, M, L, w.ctypes.data, zeta.ctypes.data, y.data_ptr(),
                                  buf[at_s:].data_ptr(), 1)
    assert code == ss.OK
    torch.cuda.synchronize()
    assert torch.equal(buf[at_s:at_s + L * M * n], want.reshape(-1))
