"""Import and export of the canonical array at 16-byte and at only 8-byte aligned
addresses: the same bytes either way, at volumes below and beyond a block's links."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32", "f32c12"])
@pytest.mark.parametrize("dims", [[2, 2, 2, 2], [4, 2, 6, 10]])
def test_canonical_array_at_either_alignment(gpu, prec, dims):
    lat = gpu.Lattice(dims, prec, seed=3)
    gpu.mgq_init_links(lat, 1)
    n = lat.volume * 72
    buf = torch.full((2 * n + 8,), float("nan"), dtype=torch.float64, device="cuda")
    even, odd = buf[2:2 + n], buf[n + 5:2 * n + 5]
    assert even.data_ptr() % 16 == 0 and odd.data_ptr() % 16 == 8
    gpu.mgq_export_links(lat, even)
    gpu.mgq_export_links(lat, odd)
    assert torch.equal(even, odd) and bool(torch.isfinite(even).all())
    assert torch.isnan(buf).sum() == buf.numel() - 2 * n  # nothing outside the two arrays
    for src in (even, odd):
        other = gpu.Lattice(dims, prec)
        gpu.mgq_import_links(other, src)
        assert torch.equal(other.links, lat.links)
    U = even.cpu().numpy().view(np.complex128).reshape(-1, 3, 3)
    tol = 1e-14 if prec == "f64" else 8 * 2.0 ** -24  # row 2 of a link against the rounded rows 0, 1
    assert np.max(np.abs(U[:, 2] - np.conj(np.cross(U[:, 0], U[:, 1])))) < tol
