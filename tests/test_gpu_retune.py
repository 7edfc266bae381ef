"""Velocity groups and tile shapes changed on bound handles: a member of a batch
that is changed between batch steps (the batch keeps the plan that it was made
with), and handles that change after the binding."""
import numpy as np
import pytest

from paper_2208_09132_gb300 import cdugks, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [cdugks.FP32, cdugks.FP64])
@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("D,n,nv", [(1, (70,), (64,)), (1, (33,), (65,)), (2, (40, 9), (8, 6))])
def test_batch_keeps_its_plan_when_a_member_changes_groups_or_tile(prec, persistent, D, n, nv):
    """Bit for bit the batch whose members were left alone; the member then
    steps alone with its own groups."""
    cells, mode = {1: (64,), 2: (32, 8) if prec == cdugks.FP32 else (16, 8)}[D], 4
    if persistent and D == 2 and prec == cdugks.FP64:
        pytest.skip("no persistent shape")
    t = cdugks.find_tile(prec, D, cells, mode)
    assert t
    cfg, f = wl.random_smooth(dim=D, n=n, nv=nv, seed=5, amp=0.2, kn=3e-3, vmax=5.0)

    def run(change):
        out = []
        for first, later in ((1, 4), (4, 1), (3, 2)):
            s = [cdugks.Solver(cfg, precision=prec, tile_id=t, velocity_groups=first) for _ in range(2)]
            for x in s:
                x.init(f)
            b = cdugks.Batch(s, persistent=persistent)
            b.step(2)
            assert b.sync() == 0
            if change:
                s[0].set_velocity_groups(later)
                assert s[0].info().velocity_groups == later
                b.step(2)
                assert b.sync() == 0
                assert cdugks.load().cdugks_set_tile(s[1]._h, 0) == 0     # the recomputing sweeps
                b.step(2)
            else:
                b.step(4)
            assert b.sync() == 0
            out += [x.moments() for x in s] + [d for x in s for d in x.distributions()]
            if change:
                for x in s:
                    x.step(1)
                    assert x.sync_status() == 0
                assert np.isfinite(s[0].moments()).all()
                tol = 1e-5 if prec == cdugks.FP32 else 1e-12
                assert np.abs(s[0].moments() - s[1].moments()).max() <= tol * np.abs(s[1].moments()).max()
        return out

    for a, b in zip(run(True), run(False)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,n,nv", [(cdugks.FP64, 64, 12), (cdugks.FP32, 86, 45), (cdugks.FP32, 40, 16)])
def test_bound_handle_takes_four_waves_of_groups(prec, n, nv):
    """A workspace laid out for the automatic group count also has room for the
    groups that fill 152 SMs x 2 CTAs four times over."""
    from paper_2208_09132_gb300 import tune
    cfg, f = wl.kelvin_helmholtz(n=n, nv=nv)
    for t in {0, tune.default_choice(cfg, prec)[0]}:
        cells = cdugks.tile_shape(prec, 2, t)[0]
        tiles = -(-n // cells[0]) * -(-n // cells[1])
        most = min(-(-1216 // tiles), 64, -(-nv * nv // 4))
        s = cdugks.Solver(cfg, precision=prec, tile_id=t)
        s.init(f)
        s.step(2)
        auto = s.moments()
        s.set_velocity_groups(most)
        s.init(f)
        s.step(2)
        assert s.sync_status() == 0
        assert s.info().velocity_groups == most
        tol = 1e-5 if prec == cdugks.FP32 else 1e-12
        assert np.abs(s.moments() - auto).max() <= tol * np.abs(auto).max()


@pytest.mark.parametrize("nv", [(8, 8), (10, 9)])
def test_bound_handle_changes_between_the_face_store_shapes(oracle_mod, nv):
    """From the stored face store to the fused one (which has sweep A by upwind
    owners) and back, after the binding."""
    cfg, f = wl.random_smooth(dim=2, n=(70, 19), nv=nv, seed=4, amp=0.2, kn=3e-3, vmax=5.0)
    stored, fused = (cdugks.find_tile(cdugks.FP32, 2, (32, 8), m) for m in (6, 4))
    assert stored and fused
    s = cdugks.Solver(cfg, precision=cdugks.FP32, tile_id=stored)
    o = oracle_mod.Oracle(cfg)
    s.init(f)
    o.init(f)
    for t in (stored, fused, stored, fused):
        assert cdugks.load().cdugks_set_tile(s._h, t) == 0
        s.step(2)
        o.step(2)
        assert s.sync_status() == 0
        ref = o.moments()
        assert (np.abs(s.moments() - ref).max(axis=0) / np.abs(ref).max(axis=0)).max() <= 1e-5
