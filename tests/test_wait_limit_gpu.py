"""The wait of every one-launch solve runs out: the 2D solves (resident and
swept tile by tile), the 3D sweeps and a batch's gangs.  With a limit below the
time of one look at the arrivals only the block that arrives last goes on, so
every solve of more than one tile reports LBS_ETIMEOUT, each time; nothing hangs,
and once the limit is back and the fields are initialised again the run is a
fresh one's."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def fields(cfg, seed=5):
    return W.initial_fields(cfg, seed=seed, noise=0.02, u0=1e-3)


def init(s, f):
    s.init_fields(f["phi"], f["psi"], f["C"], f["u"])


@pytest.mark.parametrize("limit", [0, 1, 2])
@pytest.mark.parametrize("cfg,storage,variant", [
    (W.droplet_adsorption_2d(n=72, R=14.0), "f32", 0),      # resident, two rounds a barrier
    (W.droplet_adsorption_2d(n=72, R=14.0), "f16", 5),      # resident, one round
    (W.droplet_adsorption_2d(n=72, R=14.0), "f32", 8),      # tile by tile (8 sweeps a round)
    (W.droplet_adsorption_2d(n=128, R=25.0), "f64", 0),
    (W.shear_droplet_3d(nx=64, ny=48, nz=40, R=9.0), "bf16", 0),
], ids=["resident2", "resident4", "tiles", "f64", "sweeps3d"])
def test_wait_runs_out_every_time(cfg, storage, variant, limit):
    from paper_2311_15242_gb300 import Solver
    from paper_2311_15242_gb300.lbs import LBS_ETIMEOUT, LbsError
    f = fields(cfg)
    s = Solver(cfg, storage=storage)
    s.set_sor_tile(variant)
    s.set_sor_wait_limit(limit)
    init(s, f)
    for _ in range(4):
        s.step(1)
        with pytest.raises(LbsError) as e:
            s.sync()
        assert e.value.code == LBS_ETIMEOUT
    s.set_sor_wait_limit(1 << 24)
    fresh = Solver(cfg, storage=storage)
    fresh.set_sor_tile(variant)
    for q in (s, fresh):
        init(q, f)
        q.step(5)
        q.sync()
    a, b = s.fields(), fresh.fields()
    assert all(np.array_equal(a[k], b[k]) for k in a)
    s.close()
    fresh.close()


def test_wait_of_a_batch_runs_out():
    """An instance of one tile waits for nobody and goes on."""
    from paper_2311_15242_gb300 import Batch, Solver
    from paper_2311_15242_gb300.lbs import LBS_ETIMEOUT
    cfgs = [W.bubble_rise_2d(nx=96, ny=200 + 40 * k, D_b=32.0, Eo=3.0 + k) for k in range(12)]
    cfgs.append(W.droplet_adsorption_2d(n=40, R=9.0))
    fs = [fields(c, k) for k, c in enumerate(cfgs)]
    b = Batch(cfgs, storage="f32")
    b.set_sor_wait_limit(1)
    for k, f in enumerate(fs):
        b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
    for _ in range(3):
        b.step(1)
        assert b.status() == [LBS_ETIMEOUT] * 12 + [0]
    with pytest.raises(Exception, match="wait limit"):
        b.set_sor_wait_limit(-1)
    b.set_sor_wait_limit(1 << 24)
    for k, f in enumerate(fs[:12]):
        b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
    b.step(5)
    assert b.status() == [0] * 13
    for k, (c, f, n) in enumerate(zip(cfgs, fs, [5] * 12 + [8])):
        if k not in (0, 7, 12):
            continue
        s = Solver(c, storage="f32")
        init(s, f)
        s.step(n)
        a, g = s.fields(), b.fields(k)
        assert all(np.array_equal(a[q], g[q]) for q in a), k
        s.close()
    b.close()
