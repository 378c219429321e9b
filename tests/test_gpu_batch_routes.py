"""The routes of a batched launch by its total of links, each against single-lattice
runs: the same bits, and the plaquette record."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _compare(gpu, prec, shapes, n_hb, n_or=2):
    betas = [5.7 + 0.05 * i for i in range(len(shapes))]
    singles = [gpu.Lattice(d, prec, seed=17, lattice_id=i) for i, d in enumerate(shapes)]
    for a in singles:
        gpu.mgq_init_links(a, 1)
    copies = [gpu.copy_lattice(a) for a in singles]
    batch = gpu.Batch(copies, betas, max_sweeps=2)
    rec = batch.plaquette_buffer(2)
    gpu.mgq_update_sweeps_batched(batch, 5, 2, n_hb, n_or, plaq_out=rec)
    # averages of O(1) terms in other groupings: 2^-53 or 2^-24 times a few roundings
    tol = 1e-14 if prec == "f64" else 1e-7
    for i, (a, b) in enumerate(zip(singles, copies)):
        plaq = gpu.mgq_update_sweeps(a, betas[i], 5, 2, n_hb, n_or, plaq_out=True)
        assert torch.equal(a.links, b.links), i
        assert np.max(np.abs(rec.cpu().numpy()[:, i] - plaq)) < tol, i


# 1640 links in all (few-link routes) and 69632 (a thread per link)
@pytest.mark.parametrize("prec", ["f32", "f32c12"])
@pytest.mark.parametrize("shapes", [[[6, 6, 6, 6], [2, 4, 6, 8], [4, 4, 10, 10]], [[16, 16, 16, 32], [8, 8, 8, 16]]])
def test_several_attempts(gpu, prec, shapes):
    _compare(gpu, prec, shapes, 3)


# 130 lattices: three launches a step; the partial sums' layout follows the whole call, the bits are those of one alone
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_prolongation_of_many_lattices(gpu, prec):
    shapes = [[2, 2, 2, 2], [2, 4, 2, 4], [4, 4, 4, 2]]
    coarse = []
    for i in range(130):
        c = gpu.Lattice(shapes[i % 3], prec, seed=23, lattice_id=i)
        gpu.mgq_init_links(c, 1)
        coarse.append(c)
    fine = [gpu.Lattice([2 * v for v in c.dims], prec) for c in coarse]
    batch = gpu.ProlongBatch(coarse, fine)
    gpu.mgq_prolongate_batched(batch, 0.05, 0.0, 3)
    iters, sd = batch.iters.cpu().numpy(), batch.sd.cpu().numpy()
    for i in (0, 1, 62, 63, 64, 65, 127, 128, 129):
        alone = gpu.Lattice(fine[i].dims, prec)
        it, s = gpu.mgq_prolongate(coarse[i], alone, 0.05, 0.0, 3)
        assert torch.equal(alone.links, fine[i].links) and list(iters[i]) == it
        # sums of at most 3 V terms of O(1) in other groupings
        assert np.max(np.abs(sd[i] - np.array(s))) < 1e-11 * max(1.0, np.max(np.abs(s)))


# 18-real: 32768 links (three warps per 32); 12-real: 36864 (three) and 53248 (three, packed); FP64: 3912 (three lanes)
@pytest.mark.parametrize("prec,shapes", [("f32", [[16, 16, 16, 8], [16, 16, 8, 16]]), ("f32c12", [[16, 16, 16, 8], [16, 16, 16, 10]]),
                                         ("f32c12", [[16, 16, 16, 14], [16, 16, 16, 12]]), ("f64", [[8, 8, 8, 12], [6, 6, 6, 6], [2, 4, 4, 4], [4, 4, 4, 4]])])
@pytest.mark.parametrize("n_hb", [1, 3])
def test_launches_over_few_links(gpu, prec, shapes, n_hb):
    _compare(gpu, prec, shapes, n_hb)


# 45056 links (a thread per link, ragged last blocks); FP64: 12288.  The batch's plaquettes are summed in other groupings
@pytest.mark.parametrize("prec,dims", [("f32", [16, 16, 16, 22]), ("f64", [16, 8, 12, 16])])
def test_block_sizes_do_not_change_results(gpu, prec, dims):
    from paper_1510_04675_gb300 import tune

    names = ("heatbath", "overrelax", "heatbath_batched", "overrelax_batched")
    lat = gpu.Lattice(dims, prec, seed=29)
    assert all(tune.launch_threads(k, [lat])[1] for k in names)
    gpu.mgq_init_links(lat, 1)
    small = gpu.Lattice([2, 4, 6, 2], prec, seed=30)
    gpu.mgq_init_links(small, 1)
    before, results = {k: tune.get_block_size(k, prec) for k in names}, []
    try:
        for bs in (128, 32, 64, 96):
            for k in names:
                tune.set_block_size(k, prec, bs)
            a, b, c = gpu.copy_lattice(lat), gpu.copy_lattice(lat), gpu.copy_lattice(small)
            plaq = gpu.mgq_update_sweeps(a, 5.9, 2, 2, 1, 2, plaq_out=True)
            batch = gpu.Batch([b, c], [5.9, 5.9], max_sweeps=2)
            rec = batch.plaquette_buffer(2)
            gpu.mgq_update_sweeps_batched(batch, 2, 2, 1, 2, plaq_out=rec)
            assert torch.equal(a.links, b.links)
            results.append((a.links, c.links, np.concatenate([plaq, rec.cpu().numpy().ravel()])))
    finally:
        for k in names:
            tune.set_block_size(k, prec, before[k])
    tol = 1e-14 if prec == "f64" else 1e-7
    for r in results[1:]:
        assert torch.equal(r[0], results[0][0]) and torch.equal(r[1], results[0][1])
        assert np.max(np.abs(r[2] - results[0][2])) < tol
