"""Combinations with complex coefficients on the tensor cores, through
ssqcd_moments and a solve that reaches its memory cap: vectors that fill no
tile of 64 elements, one to 100 of them (a K-step is 16, the short form ends
at 64), outputs on both sides of a launch's eight, several blocks, and vectors
that the fixed point does not suit, which keep the FP64 sum."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


def _inputs(dims, L, N, seed=1):
    g = synthetic.rng(seed)
    V = synthetic.volume(dims)
    y = g.standard_normal((L, N, V, 4, 3)) + 1j * g.standard_normal((L, N, V, 4, 3))
    t = np.linspace(-1, 1, N)
    return np.exp(0.3j * t) * (1 + t), t + 0.3j * (-1.0) ** np.arange(N), y


def _reference(w, zeta, y, M):
    coef = w[:, None] * zeta[:, None] ** np.arange(M)
    return np.einsum("jm,ljvsc->lmvsc", coef, y), np.einsum("jm,ljvsc->lmvsc", np.abs(coef), np.abs(y))


# terms L N M 12 V on both sides of the eight million where the tensor cores take over
@pytest.mark.parametrize("dims,L,N,M", [
    ((8, 8, 8, 8), 1, 32, 4), ((8, 8, 8, 8), 1, 32, 8), ((8, 8, 8, 8), 2, 16, 9), ((7, 9, 5, 11), 3, 20, 5),
    ((7, 9, 5, 11), 1, 64, 16), ((7, 9, 5, 11), 1, 65, 17), ((5, 7, 3, 11), 2, 100, 7), ((3, 5, 7, 4), 4, 100, 16),
    ((16, 8, 8, 9), 1, 1, 90), ((16, 8, 8, 9), 1, 17, 7), ((4, 4, 4, 4), 1, 8, 3),
])
@pytest.mark.parametrize("device", [False, True])
def test_moments_of_vectors(ss, dims, L, N, M, device):
    import torch
    w, zeta, y = _inputs(dims, L, N)
    lat = ss.create_lattice(dims, 0.12, -1)
    got = ss.moments(lat, w, zeta, torch.from_numpy(y).cuda() if device else y, M)
    got = got.cpu().numpy() if device else got
    ref, size = _reference(w, zeta, y, M)
    # both sums round at most N + 8 times at 2^-53 of the terms' sizes (the
    # powers of zeta take M products more); the fixed point at 2^-50 of the
    # largest component, 8 times a component's rms at most
    assert np.all(np.abs(got - ref) <= (N + M + 16) * 2.0 ** -53 * np.max(size, axis=(2, 3, 4), keepdims=True))


# more than eight outputs: 16 a pass, chunks of 96 vectors in two accumulators
@pytest.mark.parametrize("dims,L,N,M", [
    ((5, 7, 3, 11), 1, 95, 9), ((5, 7, 3, 11), 1, 96, 16), ((5, 7, 3, 11), 2, 97, 25), ((3, 5, 7, 4), 2, 193, 24),
    ((4, 4, 4, 5), 3, 289, 11), ((16, 8, 8, 9), 1, 2, 40), ((3, 3, 3, 5), 2, 600, 33),
])
def test_wide_passes(ss, dims, L, N, M):
    w, zeta, y = _inputs(dims, L, N, seed=2)
    lat = ss.create_lattice(dims, 0.12, -1)
    got = ss.moments(lat, w, zeta, y, M)
    ref, size = _reference(w, zeta, y, M)
    assert np.all(np.abs(got - ref) <= (N + M + 16) * 2.0 ** -53 * np.max(size, axis=(2, 3, 4), keepdims=True))


@pytest.mark.parametrize("kind", ["point", "wide", "inf", "nan", "zero vector", "inf weight"])
def test_vectors_that_keep_the_fp64_sum(ss, kind):
    dims, L, N, M = (8, 8, 8, 8), 2, 32, 8
    w, zeta, y = _inputs(dims, L, N)
    g = synthetic.rng(5)
    if kind == "point":  # decaying from one site
        y *= np.exp(-40.0 * np.arange(y.shape[2]) / y.shape[2])[None, None, :, None, None]
    elif kind == "wide":
        y *= 2.0 ** g.integers(-40, 40, y.shape)
    elif kind == "inf":
        y[1, 3, 77, 2, 1] = np.inf
    elif kind == "nan":
        y[0, 5, 9, 0, 0] = complex(1.0, np.nan)
    elif kind == "zero vector":
        y[0, 4] = 0
    else:
        w = w.copy()
        w[3] = np.inf
    lat = ss.create_lattice(dims, 0.12, -1)
    got = ss.moments(lat, w, zeta, y, M)
    with np.errstate(all="ignore"):
        ref, size = _reference(w, zeta, y, M)
    if kind in ("inf", "nan"):
        # only the component that the value reaches
        hit = np.zeros(ref.shape, bool)
        hit[(1, slice(None), 77, 2, 1) if kind == "inf" else (0, slice(None), 9, 0, 0)] = True
        assert np.all(np.isfinite(got[~hit]))
        assert np.all(~np.isfinite(got[hit]))
        got, ref, size = got[~hit], ref[~hit], size[~hit]
    if kind == "inf weight":
        assert np.all(~np.isfinite(got))
        return
    # componentwise, as FP64 gives it
    assert np.all(np.abs(got - ref) <= (N + M + 16) * 2.0 ** -53 * size)


# a cap of a few blocks of stored residuals: y and p-hat come from the
# combination and the run goes on with updates; a cap of nine or more: it goes
# on in segments, several of them here (~370 and more iterations)
@pytest.mark.parametrize("blocks", [6.5, 9.5, 11.5])
@pytest.mark.parametrize("dims,L", [((5, 4, 3, 8), 2), ((8, 8, 8, 8), 1)])
def test_solutions_formed_at_the_memory_cap(ss, dims, L, blocks):
    U = synthetic.gauge_field(dims, "smooth", seed=5, eps=0.3)
    v = synthetic.gaussian_sources(dims, L, seed=6)
    lat = ss.create_lattice(dims, 0.12, -1)
    ss.upload_gauge(lat, U)
    n = 12 * synthetic.volume(dims)
    block = 16 * 16 * n * L + 2 * 16 * 16 * 16 * L + 4096
    base, st0 = ss.ss_moments(lat, (0.10, 0.13), 16, 4, v, basis=0)
    got, st1 = ss.ss_moments(lat, (0.10, 0.13), 16, 4, v, basis=1, basis_max_bytes=blocks * block)
    assert st0["basis"] == 0 and st1["basis"] == 2
    for l in range(L):
        for k in range(4):
            assert np.linalg.norm(got[l, k] - base[l, k]) <= 1e-8 * np.linalg.norm(base[l, k])


@pytest.mark.parametrize("dims,L,N", [((8, 8, 8, 8), 1, 8), ((8, 8, 8, 8), 1, 9), ((8, 8, 8, 9), 2, 12)])
def test_shifted_solutions_from_stored_residuals(ss, dims, L, N):
    # both sides of the size from which shifted_cg forms the solutions from the
    # residuals; a source of zeros, frozen from the start, beside the others
    U = synthetic.gauge_field(dims, "smooth", seed=5, eps=0.3)
    v = synthetic.gaussian_sources(dims, L, seed=6)
    if L > 1:
        v[0] = 0
    z = 0.11 + 0.02 * np.linspace(-1, 1, N) + 0.01j * (-1.0) ** np.arange(N)
    lat = ss.create_lattice(dims, 0.12, -1)
    ss.upload_gauge(lat, U)
    code, y, iters, xi, seed_iters = ss.shifted_cg(lat, z, v, tol=1e-10)
    assert code == ss.OK and seed_iters == iters.max()
    for l in range(L):
        for j in range(N):
            if not v[l].any():
                assert not y[l, j].any() and iters[l, j] == 0
                continue
            r = v[l] - (z[j] * y[l, j] - wilson.apply_H(U, y[l, j], 0.12, dims, -1))
            # the stopping rule and the drift of the indefinite seed's recurrence, whose
            # residual passes peaks of a hundred ||v||: 100 it 2^-52 ||A|| ||y||
            drift = 100 * seed_iters * 2.0 ** -52 * 2.1 * np.linalg.norm(y[l, j])
            assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(v[l]) + drift
    # stopped early: the last iterate, as the update form leaves it
    code, y1, it1, _, _ = ss.shifted_cg(lat, z, v, tol=1e-10, max_iter=40)
    assert code == ss.ERR_NOCONV and it1.max() == 40
    live = v[-1]
    code, y2, it2, _, _ = ss.shifted_cg(lat, z[:3], live[None], tol=1e-10, max_iter=40)  # three points: updates
    assert code == ss.ERR_NOCONV
    for j in range(3):
        assert np.linalg.norm(y1[-1, j] - y2[0, j]) <= 1e-10 * np.linalg.norm(y2[0, j])


# float-float residuals: the update form's moments come from float-float shift
# vectors of the same seed recurrence.  Point sources: their first residuals
# keep the FP32 pipes' combination; a source of zeros; 16 and 17 moments are on
# both sides of what the tensor cores take.
@pytest.mark.parametrize("kind", ["gauss", "point", "zero"])
@pytest.mark.parametrize("dims,L,M", [((5, 4, 3, 8), 3, 5), ((8, 8, 8, 8), 1, 8), ((3, 3, 5, 8), 2, 16), ((3, 3, 5, 8), 2, 17)])
def test_moments_of_floatfloat_residuals(ss, dims, L, M, kind):
    U = synthetic.gauge_field(dims, "smooth", seed=5, eps=0.3)
    v = synthetic.gaussian_sources(dims, L, seed=6)
    if kind == "point":
        v[:] = 0
        for l in range(L):
            v[l, 3 * l + 1, l, 0] = 1.0
    elif kind == "zero":
        v[-1] = 0
    lat = ss.create_lattice(dims, 0.12, -1, precision=ss.DF)
    ss.upload_gauge(lat, U)
    base, st0 = ss.ss_moments(lat, (0.10, 0.13), 20, M, v, basis=0)
    got, st1 = ss.ss_moments(lat, (0.10, 0.13), 20, M, v, basis=1)
    assert st0["basis"] == 0 and st1["basis"] == 1
    for l in range(L):
        for k in range(M):
            # the stopping rule's residual, as for the FP64 solutions above
            assert np.linalg.norm(got[l, k] - base[l, k]) <= 1e-8 * np.linalg.norm(base[l, k])
