"""Measurements take the stored matrices as they are: fields off SU(3) against the
oracle's full products, in every format (12-real links are their rows 0, 1 and
conj(row0 x row1))."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS = [[2, 4, 2, 6], [6, 4, 8, 10]]


def _field(orc, dims, prec):
    """A thermalised field plus noise of 0.02 an entry, as the format holds it."""
    U = orc.init_links(dims, 1, seed=31)
    orc.update_chain(U, dims, 5.9, 31, 0, 0, 3, 1, 1)
    rng = np.random.default_rng(7)
    U = U + 0.02 * (rng.standard_normal(U.shape) + 1j * rng.standard_normal(U.shape))
    if prec != "f64":
        U = U.astype(np.complex64).astype(np.complex128)
    if prec == "f32c12":
        U[..., 2, :] = np.conj(np.cross(U[..., 0, :], U[..., 1, :]))
    return U


# A chain of up to 12 products of 3-term sums, 12 x 3 x 2^-24 = 2.2e-6, of matrices whose norms grow by up to 2 over
# the chain; the charges sum over the sites, E over six planes.  Rebuilding row 2 anywhere moves the values by O(0.02)
TOL = {"f64": 1e-12, "f32": 4.4e-6, "f32c12": 4.4e-6}


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec", ["f64", "f32", "f32c12"])
def test_charges_off_su3(gpu, orc, dims, prec):
    U, tol, V = _field(orc, dims, prec), TOL[prec], int(np.prod(dims))
    lat = gpu.Lattice(dims, prec)
    lat.from_numpy(U)
    E, Q = gpu.mgq_topo_charge(lat)
    Er, Qr = orc.clover_EQ(U, dims)
    assert abs(E - Er) < 10 * tol and abs(Q - Qr) < tol * np.sqrt(V)
    assert np.max(np.abs(gpu.mgq_topo_charge_improved(lat) - orc.topo_charge_improved(U, dims))) < tol * np.sqrt(V)


# 15 products per plane and three planes after the clover's ten: 75 x 3 x 2^-24 = 1.3e-5 of the largest entry
@pytest.mark.parametrize("prec", ["f32", "f32c12"])
@pytest.mark.parametrize("obs", ["E", "Q"])
def test_clover_gradient_off_su3(gpu, orc, prec, obs):
    dims = DIMS[1]
    U = _field(orc, dims, prec)
    grads = {}
    for p in ("f64", prec):
        lat = gpu.Lattice(dims, p)
        lat.from_numpy(U)
        lam = lat.new_alg_field()
        gpu.mgq_clover_vjp(lat, obs, 1.0, lam)
        grads[p] = gpu.alg_to_numpy(lat, lam)
    assert np.max(np.abs(grads[prec] - grads["f64"])) < 1.3e-5 * np.max(np.abs(grads["f64"]))


# a 4x3 loop is a chain of 14 products and a trace, 15 x 3 x 2^-24 = 2.7e-6 of matrices grown by up to 2, averaged over
# sites and planes; h takes three times the largest single loop's
@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec", ["f64", "f32", "f32c12"])
def test_loops_off_su3(gpu, orc, dims, prec):
    U, tol = _field(orc, dims, prec), 1e-12 if prec == "f64" else 5.4e-6
    lat = gpu.Lattice(dims, prec)
    lat.from_numpy(U)
    for m, n in [(1, 1), (2, 1), (2, 3), (1, 5), (4, 3)]:
        assert abs(gpu.mgq_wilson_loop(lat, m, n) - orc.wilson_loop(U, dims, m, n)) < tol
    assert np.max(np.abs(gpu.mgq_partial_loops(lat) - orc.partial_loops(U, dims))) < 3 * tol
