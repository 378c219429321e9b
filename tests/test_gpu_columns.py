"""FP64 sub-sweeps with a column of each link per lane: the same bits as one thread
per link (the batched driver's form) at the edges of a warp's and a block's links,
for both lane counts, and the plaquette record to rounding."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# V/2 = 8 (less than a block), 32, 192, 648 and 1152 (six lanes per link, ragged ends), 3456 and
# 5120 (three lanes), 12288 (one thread)
DIMS = [[2, 2, 2, 2], [2, 4, 2, 4], [4, 2, 6, 8], [6, 6, 6, 6], [12, 6, 4, 8], [12, 12, 6, 8], [8, 8, 10, 16],
        [16, 8, 12, 16]]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("n_hb", [1, 3])
def test_columns_equal_one_thread_per_link(gpu, dims, n_hb):
    a = gpu.Lattice(dims, "f64", seed=9, lattice_id=2)
    gpu.mgq_init_links(a, 1)
    b = gpu.copy_lattice(a)
    plaq = gpu.mgq_update_sweeps(a, 5.8, 3, 2, n_hb, 2, plaq_out=True)
    # beside a lattice large enough that the launches take one thread per link
    filler = gpu.Lattice([16, 16, 16, 16], "f64", seed=1)
    gpu.mgq_init_links(filler, 0)
    batch = gpu.Batch([b, filler], [5.8, 5.8], max_sweeps=2)
    rec = batch.plaquette_buffer(2)
    gpu.mgq_update_sweeps_batched(batch, 3, 2, n_hb, 2, plaq_out=rec)
    assert torch.equal(a.links, b.links)
    # sums of at most 6 V terms of O(1), each to 2^-53 relative
    assert abs(rec.cpu().numpy()[:, 0] - plaq).max() < 1e-14
    assert abs(gpu.mgq_plaquette(a) - plaq[-1]) < 1e-13


@pytest.mark.parametrize("dims", [[2, 2, 2, 2], [4, 2, 6, 8], [6, 6, 6, 6], [8, 8, 8, 12], [12, 12, 12, 14]])
def test_force_and_plaquette_by_columns(gpu, orc, dims):
    """Force (written and accumulated) and plaquette around the limits of the lane counts, against the oracle."""
    import numpy as np

    U = orc.init_links(dims, 1, seed=5)
    orc.update_chain(U, dims, 5.8, 5, 0, 0, 1, 1, 1)
    lat = gpu.Lattice(dims, "f64", with_mom=True)
    lat.from_numpy(U)
    ref = orc.force(U, dims, 6.0)
    F = lat.new_alg_field()
    gpu.mgq_hmc_force(lat, 6.0, F)
    assert np.max(np.abs(gpu.alg_to_numpy(lat, F) - ref)) < 1e-13
    P = np.random.default_rng(3).standard_normal(ref.shape)
    lat.mom.view(torch.float64).copy_(gpu.alg_from_numpy(lat, P))
    gpu.mgq_hmc_momentum_step(lat, 6.0, 0.25)
    assert np.max(np.abs(lat.mom_numpy() - (P + 0.25 * ref))) < 1e-13
    assert abs(gpu.mgq_plaquette(lat) - orc.plaquette(U, dims)) < 1e-14
