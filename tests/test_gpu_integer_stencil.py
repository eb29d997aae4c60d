"""The integer form of the FP64 stencil (60-bit fixed point, one exponent a
site) at the sizes where it can go wrong: every split of the hops over warps,
tiles of 16 sites that the lattice does not fill, wraps and extents of one,
blocks of right-hand sides that a block of the grid does not fill, fields
whose sites differ by hundreds of binades, values it does not hold, and links
it does not take."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

# 2^-53 per operation on the result's norm: the link products are exact but
# for roundings at 2^-58 of the site maximum (at most 6 times the rms of a
# Gaussian site), so the two roundings of the diagonal term dominate
NORM_TOL = 2.5e-16


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


def _case(ss, dims, nrhs, bc=-1, seed=3):
    U = synthetic.gauge_field(dims, "haar", seed=seed)
    psi = synthetic.gaussian_sources(dims, nrhs, seed=seed + 1)
    lat = ss.create_lattice(dims, 0.13, bc)
    ss.upload_gauge(lat, U)
    return U, psi, lat


# groups of 16 sites x rhs: below 304 (eight warps a group), below 608 (four), above (one)
@pytest.mark.parametrize("dims,nrhs,bc", [
    ((1, 1, 1, 1), 1, -1), ((1, 3, 1, 5), 2, -1), ((2, 2, 2, 2), 3, 1), ((5, 3, 1, 1), 1, -1), ((4, 4, 4, 4), 1, -1),
    ((3, 7, 5, 9), 4, -1), ((3, 7, 5, 9), 6, 1), ((3, 7, 5, 9), 9, -1), ((3, 7, 5, 9), 11, -1),
    ((8, 8, 8, 8), 1, -1), ((8, 8, 8, 8), 2, -1), ((8, 8, 8, 8), 3, 1), ((8, 8, 8, 8), 5, -1), ((16, 6, 5, 7), 7, -1),
])
def test_matches_oracle(ss, dims, nrhs, bc):
    U, psi, lat = _case(ss, dims, nrhs, bc)
    got = ss.apply_H(lat, psi)
    ref = wilson.apply_H(U, psi, 0.13, dims, bc)
    for f in range(nrhs):
        # the oracle's own FP64 sums of up to 150 terms are off by a few 2^-53
        assert np.linalg.norm(got[f] - ref[f]) <= (NORM_TOL + 4 * 2.0 ** -53) * np.linalg.norm(ref[f])
    # the same field alone and in the block, whatever the split: the integer sums have no order
    for f in range(nrhs):
        assert np.array_equal(ss.apply_H(lat, psi[f:f + 1])[0], got[f])


def test_site_magnitudes_and_zero_sites(ss):
    # sites of 2^-300 .. 2^300 beside zero sites: the error is relative to the
    # largest of the site and its neighbours, as in FP64
    dims = (5, 4, 3, 6)
    U, psi, lat = _case(ss, dims, 1)
    V = psi.shape[1]
    rng = synthetic.rng(9)
    scale = 2.0 ** rng.integers(-300, 300, V).astype(float)
    scale[rng.random(V) < 0.3] = 0.0
    x = psi * scale[None, :, None, None]
    got, ref = ss.apply_H(lat, x)[0], wilson.apply_H(U, x, 0.13, dims, -1)[0]
    fwd, bwd, _, _ = wilson.neighbours(dims, -1)
    big = np.abs(x[0]).reshape(V, -1).max(axis=1)
    near = np.maximum(big, np.max(np.maximum(big[fwd], big[bwd]), axis=0))
    assert np.all(np.abs(got - ref).reshape(V, -1).max(axis=1) <= 1e-14 * near)
    e = np.zeros_like(x)
    e[0, 17, 2, 1] = 1.0  # a point source: zero wherever nothing reaches
    got, ref = ss.apply_H(lat, e), wilson.apply_H(U, e, 0.13, dims, -1)
    assert np.array_equal(got == 0, ref == 0)
    assert np.max(np.abs(got - ref)) <= 2.0 ** -53


@pytest.mark.parametrize("dims,nrhs", [((3, 4, 2, 5), 1), ((8, 8, 8, 8), 2), ((8, 8, 8, 8), 3)])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e300, 1e-310, 5e-324])
def test_values_beyond_the_digits(ss, dims, nrhs, value):
    # links off unit length by 2^-9 take the FP64 kernel: its pattern of
    # infinities and NaN is the one to give
    U, psi, lat = _case(ss, dims, nrhs)
    psi[0, 3, 2, 1] = value
    psi[-1, 20, 0, 0] = complex(1.0, value)
    other = ss.create_lattice(dims, 0.13, -1)
    ss.upload_gauge(other, U * (1 + 2.0 ** -9))
    got, ref = ss.apply_H(lat, psi), ss.apply_H(other, psi)
    assert np.array_equal(np.isnan(got.real), np.isnan(ref.real))
    assert np.array_equal(np.isnan(got.imag), np.isnan(ref.imag))
    ok = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), ok)
    # one part in 2^9 of the hops apart, sites at 1e300 and their neighbours by their own size
    big = np.abs(ref) > 1e200
    for part in (ok & ~big, ok & big):
        if part.any():
            assert np.max(np.abs(got[part] - ref[part])) <= 2.0 ** -8 * np.max(np.abs(ref[part]))


def test_tiny_and_large_fields_scale(ss):
    # a field times a power of two: the same digits, the result times the same
    dims = (4, 3, 5, 4)
    U, psi, lat = _case(ss, dims, 2)
    base = ss.apply_H(lat, psi)
    for e in (-900, -200, 600):
        assert np.array_equal(ss.apply_H(lat, psi * 2.0 ** e), base * 2.0 ** e)


@pytest.mark.parametrize("factor", [1 + 2.0 ** -9, 0.5, 3.0, 1e-200])
def test_links_of_other_length_are_used_as_given(ss, factor):
    dims = (4, 4, 3, 6)
    U, psi, lat = _case(ss, dims, 2)
    V = U.shape[1]
    W = U.copy()
    W[2, V // 2] *= factor  # one link is enough
    ss.upload_gauge(lat, W)
    got = ss.apply_H(lat, psi)
    ref = wilson.apply_H(W, psi, 0.13, dims, -1)
    assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)
    ss.upload_gauge(lat, U)  # and back
    ref = wilson.apply_H(U, psi, 0.13, dims, -1)
    assert np.linalg.norm(ss.apply_H(lat, psi) - ref) <= (NORM_TOL + 4 * 2.0 ** -53) * np.linalg.norm(ref)


@pytest.mark.parametrize("dims,L", [((3, 4, 5, 6), 1), ((8, 8, 8, 8), 1), ((4, 8, 8, 8), 3), ((8, 8, 8, 8), 3)])
def test_seed_recurrence_with_the_integer_stencil(ss, dims, L):
    # every split inside the CG loop: true residuals by the oracle
    U = synthetic.gauge_field(dims, "smooth", seed=5, eps=0.3)
    v = synthetic.gaussian_sources(dims, L, seed=6)
    z = np.array([0.11 + 0.01j, 0.11 - 0.01j, 0.02j])
    lat = ss.create_lattice(dims, 0.12, -1)
    ss.upload_gauge(lat, U)
    code, y, iters, xi, it = ss.shifted_cg(lat, z, v, tol=1e-11)
    assert code == ss.OK
    for l in range(L):
        for j in range(len(z)):
            r = v[l] - (z[j] * y[l, j] - wilson.apply_H(U, y[l, j], 0.12, dims, -1))
            drift = 8 * it * 2.2e-16 * 2.1 * np.linalg.norm(y[l, j])
            assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(v[l]) + drift
