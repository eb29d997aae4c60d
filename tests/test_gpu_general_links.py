"""Links that the integer stencil does not take (rows and columns off unit
length by 2^-9): the FP64 and float-float stencils serve the operator, the CG
loop and Rayleigh-Ritz, with what they did for all links once."""
import os
import subprocess
import sys

import numpy as np
import pytest

from tests._lib import ROOT, gpu_module

import synthetic
from oracle import contour, shifted_cg as oscg, wilson

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


def _links(dims, kind="haar", seed=1):
    return synthetic.gauge_field(dims, kind, seed=seed) * (1 + 2.0 ** -9)


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 4), 1), ((5, 3, 4, 6), 3), ((8, 8, 8, 8), 4)])
def test_operator(ss, dims, nrhs):
    U, psi = _links(dims), synthetic.gaussian_sources(dims, nrhs, seed=2)
    ref = wilson.apply_H(U, psi, 0.13, dims, -1)
    lat = ss.create_lattice(dims, 0.13, -1, precision=ss.DF)
    ss.upload_gauge(lat, U)
    # float-float: 150 operations of 2^-47 each on a component's terms
    assert np.linalg.norm(ss.apply_H_mixed(lat, psi) - ref) <= 150 * 2.0 ** -47 * np.linalg.norm(ref)
    assert np.linalg.norm(ss.apply_H(lat, psi) - ref) <= 150 * 2.0 ** -53 * np.linalg.norm(ref)


# updates (N L n below 0.4 million) and stored residuals
@pytest.mark.parametrize("dims,N,L", [((2, 2, 2, 4), 8, 2), ((4, 4, 4, 6), 32, 4)])
@pytest.mark.parametrize("precision", ["FP64", "FP64_DFSHIFT", "DF"])
def test_shifted_cg(ss, dims, N, L, precision):
    kappa, tol = 0.12, 1e-11
    U, v = _links(dims, "smooth", 5), synthetic.gaussian_sources(dims, L, seed=6)
    z = contour.line_nodes(0.3, 0.05, 0.8, N)
    p = getattr(ss, precision)
    lat = ss.create_lattice(dims, kappa, -1, precision=ss.DF if precision == "DF" else ss.FP64)
    ss.upload_gauge(lat, U)
    code, y, iters, _, it = ss.shifted_cg(lat, z, v, tol=tol, precision=p)
    assert code == ss.OK
    A = lambda x: wilson.apply_H(U, x, kappa, dims, -1)
    # the operator's own rounding acts on a solution as a residual of that relative size
    eps = 2.0 ** -44 if precision == "DF" else 2.0 ** -50
    for l in range(L):
        ref = oscg.shifted_cg(A, v[l], z, tol=tol)
        for j in range(N):
            # two residuals of tol and the drift of the recurrences' steps
            res = 2.5 * tol * np.linalg.norm(v[l]) + 8 * it * eps * np.linalg.norm(ref["y"][j])
            assert np.linalg.norm(y[l, j] - ref["y"][j]) <= res / abs(z[j].imag)


@pytest.mark.parametrize("precision,block", [("FP64", 0), ("FP64", 1), ("DF", 0), ("DF", 1)])
@pytest.mark.parametrize("M", [8, 12])  # float-float moments on the FP32 pipes, on the tensor cores
def test_solve(ss, precision, block, M):
    dims, kappa = (2, 2, 2, 4), 0.13
    U, v = _links(dims), synthetic.gaussian_sources(dims, 2, seed=2)
    lat = ss.create_lattice(dims, kappa, -1, precision=getattr(ss, precision))
    ss.upload_gauge(lat, U)
    lam = np.linalg.eigvalsh(wilson.dense_H(U, kappa, dims, -1))
    pos = np.sort(lam[lam > 0])
    a, b = pos[0] - 0.01, 0.5 * (pos[3] + pos[4])
    res = ss.ss_solve(lat, (a, b), 16, M, v, beta=0.3, nprime=12, source_block=block)
    assert res.status == ss.OK, res.error
    ev, _, rs, _ = ss.ss_eigpairs(res)
    exact = lam[(lam >= a) & (lam <= b)]
    near = np.abs(ev[:, None] - exact[None]).min(axis=0)
    assert np.max(near / exact) <= 1e-10
    assert np.sum(rs <= 1e-8) == len(exact)


def test_solve_loop_with_the_plain_stencil(ss):
    """SSQCD_STENCIL_SITES=32: the FP64 stencil of 32 sites a block, in a process of its own."""
    env = dict(os.environ, SSQCD_STENCIL_SITES="32")
    out = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider", __file__, "-k",
                          "test_shifted_cg and FP64 and not DFSHIFT"], cwd=ROOT, env=env, capture_output=True, text=True,
                         timeout=300)
    assert out.returncode == 0 and "2 passed" in out.stdout, out.stdout[-2000:]
