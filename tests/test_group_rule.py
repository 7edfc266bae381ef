"""The automatic velocity-group count, from handles that are not bound, and the default
tile shape (no GPU)."""
import ctypes

import pytest

from paper_2208_09132_gb300 import cdugks, tune, workloads as wl


def automatic(cfg, prec, tile, recon=0):
    lib = cdugks.load()
    g, v, p = cdugks.describe(cfg, prec)
    h, info = ctypes.c_void_p(), cdugks.Info()
    assert lib.cdugks_create(ctypes.byref(g), ctypes.byref(v), ctypes.byref(p), ctypes.byref(h)) == 0
    assert lib.cdugks_set_reconstruction(h, recon) == 0
    assert lib.cdugks_set_tile(h, tile) == 0 and lib.cdugks_info(h, ctypes.byref(info)) == 0
    lib.cdugks_destroy(h)
    return info.velocity_groups


SIZES = [((256,), (64,)), ((4096,), (128,)), ((20000,), (100,)), ((64, 64), (16, 16)), ((100, 100), (21, 22)),
         ((256, 256), (16, 16)), ((16, 16, 16), (8, 8, 8)), ((20, 21, 22), (10, 10, 10))]


@pytest.mark.parametrize("n,nv", SIZES)
def test_fp64_sweeps_without_the_face_store_take_four_waves(n, nv):
    D = len(n)
    cfg, _ = wl.random_smooth(dim=D, n=n, nv=nv, seed=1)
    chunks = 1
    for m in nv:
        chunks *= m
    chunks = -(-chunks // 4)
    seen = 0
    for t in range(cdugks.load().cdugks_tile_count(cdugks.FP64, D)):
        cells, mode = cdugks.tile_shape(cdugks.FP64, D, t)
        if mode & 4:
            continue
        tiles = 1
        for a in range(D):
            tiles *= -(-n[a] // cells[a])
        run = -(-chunks // min(-(-1216 // tiles), chunks, 64))       # chunks of a group: equal runs
        assert automatic(cfg, cdugks.FP64, t) == -(-chunks // run), (cells, mode)
        seen += 1
    assert seen >= 1


@pytest.mark.parametrize("n,nv,cells,mode,groups",
                         [((24, 24, 24), (12, 12, 12), (8, 4, 4), 2, 8), ((20, 21, 22), (10, 10, 10), (8, 4, 4), 2, 8),
                          ((100, 100), (21, 22), (32, 8), 0, 17), ((128, 128), (24, 24), (32, 8), 0, 14)])
def test_fp32_sweeps_without_the_face_store_fill_both_sweeps(n, nv, cells, mode, groups):
    """The fastest of every count timed at these sizes (within 1 %)."""
    cfg, _ = wl.random_smooth(dim=len(n), n=n, nv=nv, seed=1)
    assert automatic(cfg, cdugks.FP32, cdugks.find_tile(cdugks.FP32, len(n), cells, mode)) == groups


@pytest.mark.parametrize("n,nv,groups", [((4096,), (128,), 32), ((128, 128), (24, 24), 7)])
def test_fp64_face_gradient_takes_at_least_four_waves(n, nv, groups):
    cfg, _ = wl.random_smooth(dim=len(n), n=n, nv=nv, seed=1)
    t = next(t for t in range(cdugks.load().cdugks_tile_count(cdugks.FP64, len(n)))
             if cdugks.tile_shape(cdugks.FP64, len(n), t)[1] & 8)
    assert automatic(cfg, cdugks.FP64, t, recon=1) == groups


@pytest.mark.parametrize("n", [(3, 3), (10, 10), (11, 23), (16, 16), (40, 20), (256, 256)])
def test_default_shape_of_2d_fp32_has_256_threads(n):
    """Also on grids of fewer cells than any tile has."""
    cfg, _ = wl.random_smooth(dim=2, n=n, nv=(9, 9), seed=1)
    assert cdugks.tile_shape(cdugks.FP32, 2, tune.default_choice(cfg, cdugks.FP32)[0])[0] == (32, 8, 1)
