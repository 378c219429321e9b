"""Which launches the block-size setting applies to, and that the autotuner leaves the
others alone."""
import ctypes

import pytest


def _lats(prec, dims_list):
    from paper_1510_04675_gb300._lib import MgqLattice

    arr = (MgqLattice * len(dims_list))()
    for c, dims in zip(arr, dims_list):
        c.dims[:] = list(dims)
        c.prec = prec
    return arr


def _shape(lib, kernel, prec, dims_list):
    t = ctypes.c_int(7)
    n = lib.mgq_launch_threads(kernel, _lats(prec, dims_list), len(dims_list), ctypes.byref(t))
    return n, t.value


F64, F32, C12 = 0, 1, 2
# 8192, 40448, 40960, 65536 links
D = {8192: (8, 8, 16, 16), 40448: (4, 4, 16, 316), 40960: (16, 16, 16, 20), 65536: (16, 16, 16, 32)}


@pytest.mark.parametrize("kernel", [0, 1])
def test_shapes_of_single_lattice_launches(mgqlib, kernel):
    assert _shape(mgqlib, kernel, F32, [D[8192]]) == (192, 0)
    assert _shape(mgqlib, kernel, F32, [D[40448]]) == (96, 0)
    assert _shape(mgqlib, kernel, F32, [D[40960]]) == (128, 1)
    assert _shape(mgqlib, kernel, C12, [D[40960]]) == (96, 0)
    assert _shape(mgqlib, kernel, C12, [D[65536]]) == (128, 0)
    assert _shape(mgqlib, kernel, F64, [(8, 8, 8, 8)]) == (32, 0)
    assert _shape(mgqlib, kernel, F64, [(16, 8, 12, 16)]) == (128, 1)
    assert mgqlib.mgq_set_block_size(kernel, F32, 64) == 0
    assert _shape(mgqlib, kernel, F32, [D[40960]]) == (64, 1) and _shape(mgqlib, kernel, F32, [D[8192]]) == (192, 0)
    assert mgqlib.mgq_set_block_size(kernel, F32, 128) == 0


def test_shapes_of_batches_and_invalid_arguments(mgqlib):
    small = (8, 8, 8, 8)
    assert _shape(mgqlib, 2, F32, [small] * 3) == (192, 0)
    assert _shape(mgqlib, 3, F32, [small] * 20) == (128, 1)          # 40960 links
    assert _shape(mgqlib, 3, F32, [(2, 2, 2, 2)] * 128 + [D[40960]]) == (128, 1)  # the second launch of the call
    assert _shape(mgqlib, 3, C12, [small] * 40) == (128, 0)
    assert _shape(mgqlib, 4, C12, [small]) == (128, 1)
    for bad in [(5, F32, [small]), (-1, F32, [small]), (0, F32, [small, small]), (2, 3, [small]), (2, F32, [(3, 4, 4, 4)])]:
        assert _shape(mgqlib, *bad) == (0, 0)
    assert mgqlib.mgq_launch_threads(0, _lats(F32, [small]), 1, None) == 192


@pytest.mark.gpu
@pytest.mark.parametrize("prec,dims", [("f32", (8, 8, 8, 8)), ("f64", (6, 6, 6, 6)), ("f32c12", (4, 4, 4, 4)), ("f32c12", D[65536])])
def test_autotuner_times_only_what_the_setting_changes(gpu, tmp_path, monkeypatch, prec, dims):
    from paper_1510_04675_gb300 import tune

    def timed(*a):
        raise AssertionError("nothing to time here")

    monkeypatch.setattr(tune, "_time", timed)
    lat = gpu.Lattice(list(dims), prec)
    cache = str(tmp_path / "tune.json")
    names = ("heatbath", "overrelax", "heatbath_batched", "overrelax_batched")
    before = {k: tune.get_block_size(k, prec) for k in names}
    try:
        for k in names:
            tune.set_block_size(k, prec, 64)
        for _ in range(2):  # measured, then from the cache
            assert tune.autotune(lat, cache_path=cache) == {"heatbath": 64, "overrelax": 64}
            assert tune.autotune_batched(gpu.Batch([lat], [6.0]), cache_path=cache) == {"heatbath_batched": 64, "overrelax_batched": 64}
        assert all(tune.get_block_size(k, prec) == 64 for k in names)
    finally:
        for k in names:
            tune.set_block_size(k, prec, before[k])
