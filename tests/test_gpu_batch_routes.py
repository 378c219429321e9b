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
