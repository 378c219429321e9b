"""Measurements on extents the lines of 2 and 3 links wrap around (extent 2), and
clover gradients in the FP32 formats against FP64, at volumes below a block and
with a partly filled last block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS = [[2, 2, 2, 2], [2, 4, 2, 6], [4, 2, 6, 4], [6, 4, 2, 10]]


def _field(orc, dims):
    U = orc.init_links(dims, 1, seed=21)
    orc.update_chain(U, dims, 5.9, 21, 0, 0, 3, 1, 1)
    return U


# FP64: sums of at most 6 V ~ 3000 terms of O(1); FP32: a chain of up to 12 products of 3-term sums, 12 x 3 x 2^-24,
# averaged in the loops and summed over the sites (V ~ 480) in the charges
@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec,tol", [("f64", 1e-13), ("f32", 2.2e-6), ("f32c12", 2.2e-6)])
def test_loops_and_charges_on_short_extents(gpu, orc, dims, prec, tol):
    U = _field(orc, dims)
    lat = gpu.Lattice(dims, prec)
    lat.from_numpy(U)
    V = int(np.prod(dims))
    for m, n in [(1, 1), (2, 1), (3, 2), (1, 5), (4, 3)]:
        assert abs(gpu.mgq_wilson_loop(lat, m, n) - orc.wilson_loop(U, dims, m, n)) < tol
    assert np.max(np.abs(gpu.mgq_partial_loops(lat) - orc.partial_loops(U, dims))) < 3 * tol
    ref = orc.topo_charge_improved(U, dims)
    assert np.max(np.abs(gpu.mgq_topo_charge_improved(lat) - ref)) < tol * np.sqrt(V) + 1e-12
    E, Q = gpu.mgq_topo_charge(lat)
    Er, Qr = orc.clover_EQ(U, dims)
    assert abs(E - Er) < 10 * tol and abs(Q - Qr) < tol * np.sqrt(V) + 1e-12
    assert np.max(np.abs(lat.to_numpy() - U)) < 1e-6  # measuring leaves the links alone


# 15 products per plane and three planes: 45 x 3 x 2^-24 = 8e-6 of the largest entry
@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("obs", ["E", "Q"])
def test_clover_gradient_fp32_against_fp64(gpu, orc, dims, obs):
    U = _field(orc, dims)
    grads = {}
    for prec in ("f64", "f32", "f32c12"):
        lat = gpu.Lattice(dims, prec)
        lat.from_numpy(U)
        lam = lat.new_alg_field()
        gpu.mgq_clover_vjp(lat, obs, 0.5, lam)
        gpu.mgq_clover_vjp(lat, obs, 0.5, lam)  # adds
        grads[prec] = gpu.alg_to_numpy(lat, lam)
    top = np.max(np.abs(grads["f64"]))
    for prec in ("f32", "f32c12"):
        assert np.max(np.abs(grads[prec] - grads["f64"])) < 8e-6 * top
