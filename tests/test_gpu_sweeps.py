"""The face-store sweeps where their kernels branch: cell counts at the edges of
the tiles of sweep A and of sweep B, velocity grids whose visits are pure
(whole chunks of one sign), mixed, unaligned (rows that are not whole chunks) and
with a node at 0, velocity groups that hold one sign pattern and several, every
boundary kind, and the acceleration's pre-pass along lines of each axis.

Against the FP64 oracle with the repository's targets: relative L-infinity 1e-5
(FP32) and 1e-12 (FP64) of rho, u (one scale), T and of every distribution value
against the largest one."""
import numpy as np
import pytest

from paper_2208_09132_gb300 import cdugks, workloads as wl
from paper_2208_09132_gb300.tune import has_zero_node
from test_gpu_parity import _bc, rel_linf

pytestmark = pytest.mark.gpu

P, S, DI = wl.BC_PERIODIC, wl.BC_SPECULAR, wl.BC_DIRICHLET
TOL = {cdugks.FP32: 1e-5, cdugks.FP64: 1e-12}

# (cells, velocities, boundaries per axis)
CASES = [
    ((1,), (8,), [(P, P)]), ((2,), (6,), [(S, S)]), ((127,), (9,), [(DI, DI)]), ((129,), (12,), [(S, DI)]),
    ((257,), (64,), [(P, P)]),
    ((1, 3), (8, 4), [(P, P), (S, S)]), ((33, 5), (8, 8), [(P, P), (P, P)]), ((64, 8), (12, 6), [(S, S), (P, P)]),
    ((31, 17), (10, 9), [(P, P), (S, S)]), ((65, 9), (6, 4), [(DI, DI), (S, S)]), ((32, 4), (5, 7), [(S, S), (S, S)]),
    ((9, 5, 3), (8, 4, 4), [(P, P), (P, P), (P, P)]), ((8, 4, 4), (12, 4, 6), [(S, S), (P, P), (S, S)]),
    ((17, 9, 5), (10, 4, 4), [(P, P), (S, S), (P, P)]), ((7, 8, 9), (6, 4, 4), [(S, S), (S, S), (S, S)]),
    ((16, 3, 4), (12, 4, 4), [(P, P), (DI, DI), (S, S)]),
]


def check(s, o, prec, what):
    assert s.sync_status() == 0
    assert np.all(rel_linf(s.moments(), o.moments()) <= TOL[prec]), what
    for got, ref in zip(s.distributions(), o.distributions()):
        assert np.abs(got - ref).max() <= TOL[prec] * np.abs(ref).max(), what


@pytest.mark.parametrize("prec", [cdugks.FP32, cdugks.FP64])
@pytest.mark.parametrize("n,nv,bc", CASES, ids=["x".join(map(str, c[0])) + "_nv" + "x".join(map(str, c[1])) for c in CASES])
def test_branches_match_oracle(oracle_mod, n, nv, bc, prec):
    D = len(n)
    cfg, f = wl.random_smooth(dim=D, n=n, nv=nv, seed=sum(n) + nv[0], amp=0.2, kn=3e-3, vmax=5.0)
    cfg = _bc(cfg, bc)
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(3)
    for t in range(cdugks.load().cdugks_tile_count(prec, D)):
        mode = cdugks.tile_shape(prec, D, t)[1]
        if not mode & 4 or mode & (3 | 8 | 16 | 32) or (mode & 128 and has_zero_node(cfg)):
            continue               # the fused and lean face-store shapes of the default scheme
        for groups in (1, 3, 64):
            s = cdugks.Solver(cfg, precision=prec, tile_id=t, velocity_groups=groups)
            s.init(f)
            s.step(3)
            check(s, o, prec, (t, groups))


@pytest.mark.parametrize("prec", [cdugks.FP32, cdugks.FP64])
@pytest.mark.parametrize("nv,acc", [((8, 8), (0.4, 0.0)), ((12, 6), (0.0, -0.3)), ((8, 9), (0.0, 0.5)),
                                    ((8, 8), (0.2, -0.3)), ((10, 6), (0.3, 0.0)), ((8, 4, 4), (0.0, 0.0, 0.4)),
                                    ((12, 4, 4), (0.0, 0.3, 0.0)), ((8, 4, 4), (0.5, 0.0, 0.0))])
def test_acceleration_along_each_axis_matches_oracle(oracle_mod, nv, acc, prec):
    D = len(nv)
    cfg, f = wl.random_smooth(dim=D, n=(33, 9, 5), nv=nv, seed=7, amp=0.2, kn=3e-3, vmax=5.0)
    cfg = _bc(cfg, [(P, P), (S, S), (P, P)][:D])
    cfg["accel"] = list(acc) + [0.0] * (3 - D)
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(3)
    for groups in (1, 4):
        s = cdugks.Solver(cfg, precision=prec, velocity_groups=groups)
        s.init(f)
        s.step(3)
        check(s, o, prec, groups)


def test_wait_hook_with_groups_of_uneven_chunks(oracle_mod):
    """The wait hook's staging sweep takes equal chunks a group (6 groups for the 7
    that the sweeps with upwind owners take of 16 chunks); the handle recovers."""
    cfg, f = wl.random_smooth(dim=2, n=(72, 28), nv=(8, 8), seed=1, amp=0.3, kn=3e-3)
    s = cdugks.Solver(cfg, precision=cdugks.FP32, tile_id=cdugks.find_tile(cdugks.FP32, 2, (32, 8), 4), velocity_groups=7)
    assert s.info().velocity_groups == 7
    lib = cdugks.load()
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
    check(s, o, cdugks.FP32, 7)


@pytest.mark.parametrize("prec", [cdugks.FP32, cdugks.FP64])
@pytest.mark.parametrize("n,nv,acc", [((64, 41), (32, 8), (0.4, 0.0)), ((64, 41), (32, 8), (0.0, -0.3)),
                                      ((64, 41), (32, 9), (0.0, 0.3)), ((13, 12, 9), (8, 8, 8), (0.0, 0.0, 0.4)),
                                      ((13, 12, 9), (8, 8, 8), (0.0, 0.3, 0.0)), ((13, 12, 9), (8, 8, 8), (0.5, 0.0, 0.0))])
def test_acceleration_prepass_along_lines_matches_oracle(oracle_mod, n, nv, acc, prec):
    """Enough lines for the pre-pass along the forced axis (152 blocks of cells x lines)."""
    D = len(n)
    cfg, f = wl.random_smooth(dim=D, n=n, nv=nv, seed=3, amp=0.2, kn=3e-3, vmax=5.0)
    cfg = _bc(cfg, [(P, P), (S, S), (P, P)][:D])
    cfg["accel"] = list(acc) + [0.0] * (3 - D)
    o = oracle_mod.Oracle(cfg)
    o.init(f)
    o.step(3)
    s = cdugks.Solver(cfg, precision=prec, velocity_groups=4)
    s.init(f)
    s.step(3)
    check(s, o, prec, acc)
