"""Routes of the face-store sweeps beside those of test_gpu_sweeps: against the FP64
oracle with the repository's targets (1e-5 FP32, 1e-12 FP64)."""
import numpy as np
import pytest

from paper_2208_09132_gb300 import cdugks, workloads as wl
from paper_2208_09132_gb300.tune import has_zero_node
from test_gpu_parity import _bc
from test_gpu_sweeps import CASES, check

pytestmark = pytest.mark.gpu

P, S, DI = wl.BC_PERIODIC, wl.BC_SPECULAR, wl.BC_DIRICHLET


@pytest.mark.parametrize("prec", [cdugks.FP32, cdugks.FP64])
@pytest.mark.parametrize("nv", [(10, 6), (9, 7), (3, 5), (6, 5, 4), (3, 4, 5), (2, 3, 3)])
def test_force_along_several_axes_on_rows_that_are_not_whole_chunks(oracle_mod, nv, prec):
    """The force gradients of sweep B lane by lane: a chunk's lanes in one, two or
    three velocity rows, padding, the ends of every axis, walls that leave out the
    normal component."""
    D = len(nv)
    cfg, f = wl.random_smooth(dim=D, n=(17, 9, 5), nv=nv, seed=7, amp=0.1, kn=3e-3, vmax=4.0)
    cfg = _bc(cfg, [(S, S), (P, P), (S, S)][:D])
    cfg["accel"] = [0.3, -0.4, 0.2][:D] + [0.0] * (3 - D)
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(3)
    for groups in (1, 3):
        s = cdugks.Solver(cfg, precision=prec, velocity_groups=groups)
        s.init(f)
        s.step(3)
        check(s, o, prec, groups)


STORED = [(prec, collision, case) for prec in (cdugks.FP32, cdugks.FP64) for collision in (0, 1) for case in CASES
          if len(case[0]) == 3 or (len(case[0]) == 2 and prec == cdugks.FP32 and not collision)]
STORED = [x for x in STORED if not any(DI in b for b in x[2][2])]      # (they take no Dirichlet ends)


@pytest.mark.parametrize("prec,collision,case", STORED, ids=[
    f"{'fp64' if p == cdugks.FP64 else 'fp32'}_{'shakhov_' if c else ''}{'x'.join(map(str, k[0]))}_nv{'x'.join(map(str, k[1]))}"
    for p, c, k in STORED])
def test_stored_face_store_at_tile_edges_matches_oracle(oracle_mod, prec, collision, case):
    """Stored slopes and face store: sweep B with exchanged fluxes on its own tile,
    in FP64 3D among them (the only face-store shapes of the default model there)."""
    n, nv, bc = case
    cfg, f = wl.random_smooth(dim=len(n), n=n, nv=nv, seed=sum(n) + nv[0], amp=0.2, kn=3e-3, vmax=5.0)
    cfg = _bc(cfg, bc)
    cfg["collision"] = collision
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(3)
    checked = 0
    for t in range(cdugks.load().cdugks_tile_count(prec, len(n))):
        mode = cdugks.tile_shape(prec, len(n), t)[1]
        if mode & ~16 != 6 or bool(mode & 16) != bool(collision):
            continue
        for groups in (1, 3, 64):
            s = cdugks.Solver(cfg, precision=prec, tile_id=t, velocity_groups=groups)
            s.init(f)
            s.step(3)
            check(s, o, prec, (t, groups))
        checked += 1
    assert checked >= 1


@pytest.mark.parametrize("prec,D,cells,mode", [(cdugks.FP32, 1, (128,), 0), (cdugks.FP32, 2, (32, 8), 0), (cdugks.FP64, 1, (128,), 0),
                                               (cdugks.FP64, 2, (8, 8), 12)])
def test_wait_hook_on_sweeps_that_stage_in_production(oracle_mod, prec, D, cells, mode):
    """The bounded wait of the sweeps that steps of these shapes run (the shapes with
    upwind owners have no such wait and run the staging sweep under the hook only)."""
    cfg, f = wl.random_smooth(dim=D, n=(1030,) if D == 1 else (72, 28), nv=(8, 8), seed=1, amp=0.3, kn=3e-3)
    cfg["recon"] = 1 if mode & 8 else 0
    lib = cdugks.load()
    t = next(t for t in range(lib.cdugks_tile_count(prec, D))
             if cdugks.tile_shape(prec, D, t) == (cells + (1,) * (3 - D), mode))
    s = cdugks.Solver(cfg, precision=prec, tile_id=t)
    s.init(f)
    assert lib.cdugks_test_wait_timeout(s._h, 1) == 0
    s.step(1)
    assert s.sync_status() == cdugks.ERR_TIMEOUT
    assert lib.cdugks_test_wait_timeout(s._h, 0) == 0
    s.init(f)
    s.step(3)
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(3)
    check(s, o, prec, t)


# velocity ranges per axis: one sign only, a node at 0 at an end, uneven about 0
RANGES = [((7,), [(0.1, 4.5)], [(P, P)], (11,)), ((32,), [(-4.5, -0.2)], [(DI, DI)], (70,)), ((9,), [(0.0, 4.0)], [(P, P)], (5,)),
          ((7, 4), [(0.1, 4.5), (-4.5, 4.5)], [(P, P), (DI, DI)], (1, 2)), ((16, 9), [(-5.9, -0.2), (-5.9, 5.9)], [(P, P), (P, P)], (3, 19)),
          ((8, 12), [(-3.8, 5.5), (-5.5, 5.5)], [(DI, DI), (S, DI)], (3, 8)), ((8, 5), [(-5.5, 3.3), (-5.5, 5.5)], [(DI, DI), (DI, S)], (12, 27)),
          ((10, 13), [(-4.4, 4.4), (0.0, 4.4)], [(P, P), (DI, DI)], (1, 3)),
          ((8, 8, 8), [(0.1, 5.5), (-5.5, 5.5), (-3.9, 5.5)], [(P, P), (S, S), (P, P)], (13, 2, 1)),
          ((3, 8, 2), [(0.1, 4.8), (-4.8, -0.2), (-4.8, 4.8)], [(P, P), (P, P), (DI, DI)], (2, 11, 6)),
          ((2, 8, 8), [(-3.8, 3.8), (-3.8, -0.2), (-3.8, 3.8)], [(DI, DI), (DI, DI), (S, S)], (3, 6, 2))]


@pytest.mark.parametrize("prec", [cdugks.FP32, cdugks.FP64])
@pytest.mark.parametrize("nv,ranges,bc,n", RANGES, ids=["x".join(map(str, r[0])) + "_n" + "x".join(map(str, r[3])) for r in RANGES])
def test_velocity_ranges_of_one_sign_in_a_workspace_of_nans(oracle_mod, nv, ranges, bc, n, prec):
    """Groups that lack a sign along an axis, alone and with others of several
    classes: every partial sum and face value that is read has been written."""
    import torch
    D = len(nv)
    cfg, f = wl.random_smooth(dim=D, n=n, nv=nv, seed=3, amp=0.1, kn=1e-2, vmax=4.0)
    cfg = _bc(cfg, bc)
    cfg["vlo"], cfg["vhi"] = [r[0] for r in ranges] + [-1.0] * (3 - D), [r[1] for r in ranges] + [1.0] * (3 - D)
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(2)
    checked = 0
    for t in range(cdugks.load().cdugks_tile_count(prec, D)):
        mode = cdugks.tile_shape(prec, D, t)[1]
        if not mode & 4 or mode & (8 | 16 | 32) or (mode & 128 and has_zero_node(cfg)) or (mode & 3 == 2 and DI in sum(bc, ())):
            continue
        checked += 1
        for groups in (0, 1, 2, 3, 5, 6, 7, 64):
            size = cdugks.Solver(cfg, precision=prec, tile_id=t, velocity_groups=groups).workspace_bytes
            ws = torch.full((size + 256,), 255, dtype=torch.uint8, device="cuda:0")
            s = cdugks.Solver(cfg, precision=prec, tile_id=t, velocity_groups=groups, workspace=ws)
            s.init(f)
            s.step(2)
            check(s, o, prec, (t, groups))
    assert checked or (D == 3 and prec == cdugks.FP64 and DI in sum(bc, ()))


@pytest.mark.parametrize("prec", [cdugks.FP32, cdugks.FP64])
@pytest.mark.parametrize("physics", ["plain", "shakhov", "force"])
@pytest.mark.parametrize("D,axis,vmax,nodes", [(1, 0, 3.675, 7), (1, 0, 3.88, 7), (2, 0, 3.727, 11), (2, 1, 3.962, 11), (2, 1, 3.675, 7),
                                               (2, 0, 5.964, 13), (3, 0, 3.88, 7), (3, 1, 3.675, 7), (3, 2, 3.88, 7)])
def test_walls_on_odd_grids_whose_middle_node_rounds_off_zero(oracle_mod, D, axis, vmax, nodes, physics, prec):
    """The middle node of -v .. v is 4e-16 or 9e-16 off 0 to either side: its mirror
    image is itself, of the same sign, so a wall's ghost is not the image of the
    cell's upwind side there."""
    middle = -vmax + 2 * vmax * (nodes // 2) / (nodes - 1)
    assert 0 < abs(middle) < 1e-15
    nv = [8, 6, 4][:D]
    nv[axis] = nodes
    cfg, f = wl.random_smooth(dim=D, n=(19, 11, 6), nv=nv, seed=9, amp=0.1, kn=3e-3, vmax=vmax)
    cfg = _bc(cfg, [(S, S) if a == axis else (P, P) for a in range(D)])
    cfg["collision"] = 1 if physics == "shakhov" else 0
    if physics == "force":
        cfg["accel"] = [0.2 if a == axis else -0.1 for a in range(D)] + [0.0] * (3 - D)
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(3)
    checked = 0
    for t in range(cdugks.load().cdugks_tile_count(prec, D)):
        mode = cdugks.tile_shape(prec, D, t)[1]
        if not mode & 4 or mode & 8 or bool(mode & 16) != (physics == "shakhov") or bool(mode & 32) != (physics == "force"):
            continue
        checked += 1
        for groups in (0, 1, 5):
            s = cdugks.Solver(cfg, precision=prec, tile_id=t, velocity_groups=groups)
            s.init(f)
            s.step(3)
            check(s, o, prec, (t, groups))
    assert checked
