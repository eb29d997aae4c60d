"""The stand-alone operator component by component: fields in which some
components are far below their site's or their neighbours' largest, so that
the integer stencil's fixed point, which is relative to those, has no bits for
them.  Links that do not mix colours keep them apart in the result as well."""
import numpy as np
import pytest

from tests._lib import gpu_module

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

KAPPA, DIMS = 0.13, (5, 4, 3, 6)


@pytest.fixture(scope="module")
def ss():
    return gpu_module()


def _reference(U, psi, bc):
    """A psi and the sum of its terms' sizes, in more than 64 bits."""
    U, psi = U.astype(np.clongdouble), psi.astype(np.clongdouble)
    gam, g5 = wilson.gamma_matrices()
    fwd, bwd, sfwd, sbwd = wilson.neighbours(DIMS, bc)
    out, size = psi.copy(), np.abs(psi)
    kappa = np.longdouble(KAPPA)
    for mu in range(4):
        for nb, sg, u, g in ((fwd, sfwd, U[mu], np.eye(4) - gam[mu]),
                             (bwd, sbwd, np.conj(np.swapaxes(U[mu][bwd[mu]], 1, 2)), np.eye(4) + gam[mu])):
            p = psi[:, nb[mu]]
            t = np.einsum("sab,lsib->lsia", u, p * sg[mu][:, None, None])
            out -= kappa * np.einsum("ij,lsja->lsia", g.astype(np.clongdouble), t)
            size += kappa * np.einsum("ij,lsja->lsia", np.abs(g).astype(np.longdouble),
                                      np.einsum("sab,lsib->lsia", np.abs(u), np.abs(p)))
    return out * np.diag(g5).real[:, None], size


def _fields(nrhs):
    psi = synthetic.gaussian_sources(DIMS, nrhs, seed=4)
    V = psi.shape[1]
    g = synthetic.rng(5)
    colours = psi * 10.0 ** np.array([0, -20, -35])
    spins = psi * 10.0 ** np.array([0, -18, -18, -25])[:, None]
    slope = psi * 2.0 ** -(8.0 * wilson.site_coords(DIMS)[:, 0] + 1.0)[:, None, None] * 2.0 ** -np.array([0, 9, 30])
    mixed = psi * 2.0 ** -g.integers(0, 60, psi.shape).astype(float)
    few = psi * np.where(g.random(psi.shape) < 0.04, 2.0 ** -30, 1.0)
    dilute = psi.copy()
    dilute[:, :, [0, 1, 3]] = 0.0  # one spin
    dilute[:, :, 2, 2] *= 2.0 ** -50
    wall = psi * np.where(wilson.site_coords(DIMS)[:, 2] == 1, 1.0, 2.0 ** -45)[:, None, None]
    return dict(gaussian=psi, colours=colours, spins=spins, slope=slope, mixed=mixed, few=few, dilute=dilute, wall=wall)


# 23 groups of 16 sites a field: four warps a group, and with 27 fields one
@pytest.mark.parametrize("nrhs", [1, 2, 27])
@pytest.mark.parametrize("links", ["unit", "haar", "diagonal"])
def test_every_component(ss, links, nrhs):
    V = synthetic.volume(DIMS)
    if links == "haar":
        U = synthetic.gauge_field(DIMS, "haar", seed=3)
    else:
        ph = np.zeros((4, V, 3)) if links == "unit" else synthetic.rng(8).uniform(-3, 3, (4, V, 3))
        U = np.exp(1j * ph)[..., None] * np.eye(3)
    lat = ss.create_lattice(DIMS, KAPPA, -1)
    ss.upload_gauge(lat, U)
    for name, psi in _fields(nrhs).items():
        got = ss.apply_H(lat, psi)
        ref, size = _reference(U, psi, -1)
        # FP64 sums of 150 terms lie within ~2^-48 of the sizes; where the fixed
        # point serves, its roundings are at most 48 of the 2^52 units that a
        # component's terms have
        bad = np.abs(got - ref) > 2.0 ** -46 * size
        assert not bad.any(), (name, int(bad.sum()), float(np.max(np.abs(got - ref) / size)))
        # and zero where every term is
        assert np.all(got[size == 0] == 0), name
