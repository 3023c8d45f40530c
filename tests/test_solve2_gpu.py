"""The solve with the whole grid resident on the chip (FP32, one launch a step
after the fused step): tiles and seams where it can go wrong, against the
launches of one round each (lbs_set_sor_persistent off), which run the same
iterates, and against the oracle.

The two forms agree to the rounding of FP32 (F32_IMPL_TOL of
test_parity_gpu) and stop after the same number of sweeps."""
import numpy as np
import pytest

import workloads as W
from oracle.ora import Oracle
from test_parity_gpu import F32_IMPL_TOL, F32_TOL, droplet, errors, within

pytestmark = pytest.mark.gpu


def run(cfg, f, steps, on, variant):
    from paper_2311_15242_gb300 import Solver
    s = Solver(cfg, storage="f32")
    s.set_sor_tile(variant)
    s.set_sor_persistent(on)
    s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
    s.step(steps)
    out, d = s.fields(), s.diagnostics()
    s.close()
    return out, d


@pytest.mark.parametrize("variant", [0, 5])
@pytest.mark.parametrize("nx,ny,wall", [
    (5, 9, (1, 1, 0)),      # one small tile, walls all round
    (48, 48, (0, 0, 0)),    # the largest periodic tile of the wide halo
    (64, 65, (1, 2, 0)),    # one full column of tiles, one cell over in y
    (49, 50, (0, 0, 0)),    # odd periodic x: a seam between tiles
    (63, 31, (0, 0, 0)),    # seams on both axes
    (130, 37, (1, 0, 0)),   # seam along y, three tiles along x
    (113, 97, (2, 1, 0)),   # odd walled axes
])
def test_resident_solve_equals_round_launches(nx, ny, wall, variant):
    cfg = droplet(nx=nx, ny=ny, R=min(nx, ny) / 4.0)
    cfg.update(wall=list(wall))
    f = W.initial_fields(cfg, seed=3, noise=0.02, u0=1e-4)
    a, da = run(cfg, f, 12, True, variant)
    b, db = run(cfg, f, 12, False, variant)
    err = errors(b, a)
    assert within(err, F32_IMPL_TOL), err
    assert da["sor_iters_psi"] == db["sor_iters_psi"]
    assert abs(da["surf_total"] / db["surf_total"] - 1.0) < 1e-7
    o = Oracle(cfg)
    o.init_fields(f["phi"], f["psi"], f["C"], f["u"])
    o.step(12)
    err = errors(o.fields(), a)
    assert within(err, F32_TOL), err


def test_one_round_between_barriers():
    """640 x 640: too large for the tiles of two rounds' halo, small enough
    for one round's."""
    cfg = W.bubble_array_2d(640, 2)
    cfg["wall"] = [0, 0, 0]
    f = W.initial_fields(cfg, seed=3, noise=0.02)
    a, da = run(cfg, f, 6, True, 0)
    b, db = run(cfg, f, 6, False, 0)
    err = errors(b, a)
    assert within(err, dict(F32_IMPL_TOL, psi=2e-5)), err
    assert da["sor_iters_psi"] == db["sor_iters_psi"]


def test_limit_of_rounds_and_restart():
    """A solve cut off by sor_max_iter (an odd number of rounds: the second
    round of a phase is dropped) reports it and keeps that round's result;
    stepping on after a restart from a saved state repeats bit for bit."""
    from paper_2311_15242_gb300 import Solver
    from paper_2311_15242_gb300.lbs import LBS_ENOCONV, LbsError
    cfg = droplet()
    cfg.update(sor_max_iter=2, sor_tol=1e-12)
    f = W.initial_fields(cfg, seed=3, noise=0.02)
    out = []
    for on in (True, False):
        s = Solver(cfg, storage="f32")
        s.set_sor_persistent(on)
        s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
        s.step(2)
        with pytest.raises(LbsError) as e:
            s.sync()
        assert e.value.code == LBS_ENOCONV
        assert s.diagnostics()["sor_iters_psi"] == 2
        out.append(s.fields())
        s.close()
    assert within(errors(out[1], out[0]), F32_IMPL_TOL)
    cfg = droplet(nx=63, ny=45)
    s = Solver(cfg, storage="f32")
    f = W.initial_fields(cfg, seed=4, noise=0.02)
    s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
    s.step(3)
    state = s.save_state()
    s.step(4)
    a = s.fields()
    s.load_state(state)
    s.step(4)
    b = s.fields()
    s.close()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def test_gangs_of_a_batch_equal_single_contexts():
    """Six instances whose tiles take two waves of the chip, one of odd height,
    one taken out of the work lists: each as its own context, the inactive one
    unchanged; and a batch with an odd periodic width, which the resident form
    does not take."""
    from paper_2311_15242_gb300 import Batch, Solver
    cfgs = [W.bubble_rise_2d(nx=200 + 8 * k, ny=400 + (k == 2), D_b=32.0, Eo=2.0 + k)
            for k in range(6)]
    odd = droplet(nx=45, ny=40)
    for group in (cfgs, [odd, cfgs[0]]):
        fs = [W.initial_fields(c, seed=k, noise=0.02) for k, c in enumerate(group)]
        b = Batch(group, storage="f32")
        for k, f in enumerate(fs):
            b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
        off = len(group) - 1
        b.step(3)
        kept = b.fields(off)
        b.set_active(off, False)
        b.step(9)
        assert b.status() == [0] * len(group)
        d = b.diagnostics()
        for k, (c, f) in enumerate(zip(group, fs)):
            got = b.fields(k)
            if k == off:
                assert all(np.array_equal(got[q], kept[q]) for q in got)
                continue
            s = Solver(c, storage="f32")
            s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
            s.step(12)
            err = errors(s.fields(), got)
            assert within(err, F32_IMPL_TOL), (k, err)
            assert s.diagnostics()["sor_iters_psi"] == d[k]["sor_iters_psi"]
            s.close()
        b.close()
