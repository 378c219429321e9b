"""FP32 sub-sweeps with a staple term per warp: the same bits as the batched driver's
one thread per link, at volumes below and around a block's 32 links, on both sides
of the sizes where six warps give way to three and three to a thread per link, and
with the plaquette record."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# V/2 = 8, 32, 48, 648, 16128 and 16384 (six / three warps), 39936 and 40960 (18-real limit), 49152
# (packed from here on), 61440 and 65536 (12-real limit)
DIMS = [[2, 2, 2, 2], [2, 4, 2, 4], [4, 2, 6, 2], [6, 6, 6, 6], [8, 14, 12, 24], [8, 16, 16, 16], [16, 16, 4, 78],
        [16, 16, 16, 20], [16, 16, 16, 24], [16, 16, 16, 30], [16, 16, 16, 32]]


@pytest.mark.parametrize("prec", ["f32", "f32c12"])
@pytest.mark.parametrize("dims", DIMS)
def test_terms_equal_one_thread_per_link(gpu, prec, dims):
    a = gpu.Lattice(dims, prec, seed=11, lattice_id=4)
    gpu.mgq_init_links(a, 1)
    b = gpu.copy_lattice(a)
    plaq = gpu.mgq_update_sweeps(a, 5.9, 7, 2, 1, 2, plaq_out=True)
    # beside a lattice large enough that the launches take one thread per link
    filler = gpu.Lattice([24, 24, 24, 24], prec, seed=1)
    gpu.mgq_init_links(filler, 0)
    batch = gpu.Batch([b, filler], [5.9, 5.9], max_sweeps=2)
    rec = batch.plaquette_buffer(2)
    gpu.mgq_update_sweeps_batched(batch, 7, 2, 1, 2, plaq_out=rec)
    assert torch.equal(a.links, b.links)
    # FP32 plaquettes of O(1) in other groupings: 2^-24 x a few roundings each, averaged
    assert np.max(np.abs(rec.cpu().numpy()[:, 0] - plaq)) < 1e-7
    assert abs(gpu.mgq_plaquette(a) - plaq[-1]) < 1e-6


# 4096 links in all (six warps), 40960 (three), 49152 (three, packed)
@pytest.mark.parametrize("prec", ["f32", "f32c12"])
@pytest.mark.parametrize("dims", [[[8, 8, 8, 8], [8, 8, 8, 8]], [[16, 16, 16, 12], [16, 16, 16, 8]], [[16, 16, 16, 12], [16, 16, 16, 12]]])
def test_batched_terms_equal_single(gpu, prec, dims):
    singles = [gpu.Lattice(d, prec, seed=11, lattice_id=i) for i, d in enumerate(dims)]
    for a in singles:
        gpu.mgq_init_links(a, 1)
    copies = [gpu.copy_lattice(a) for a in singles]
    for a in singles:
        gpu.mgq_update_sweeps(a, 5.9, 7, 2, 1, 2)
    batch = gpu.Batch(copies, [5.9] * len(copies), max_sweeps=2)
    gpu.mgq_update_sweeps_batched(batch, 7, 2, 1, 2)
    for a, b in zip(singles, copies):
        assert torch.equal(a.links, b.links)
