"""Routes of the face-store sweeps beside those of test_gpu_sweeps: against the FP64
oracle with the repository's targets (1e-5 FP32, 1e-12 FP64)."""
import numpy as np
import pytest

from paper_2208_09132_gb300 import cdugks, workloads as wl
from test_gpu_parity import _bc
from test_gpu_sweeps import check

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
