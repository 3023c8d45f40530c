"""3D: every sweep of a solve in one cooperative launch (k_sor_fs3, the default
in FP32 arithmetic) against the red and black half-sweeps as launches of their
own (lbs_set_sor_persistent off): the same operations on the same values, so
the fields agree to the rounding two compilations may differ by
(F32_IMPL_TOL) and the sweeps are as many.  Sizes at the edges of its tiles:
less than a tile, one cell over a tile's 60 columns or 28 rows, odd sides
between walls, chunks of z that end at an odd plane, more tiles than SMs."""
import pytest

import workloads as W
from test_parity_gpu import F32_IMPL_TOL, errors, within

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,wall,steps", [
    ((6, 4, 4), (0, 0, 0), 4),        # periodic images of cells inside the region
    ((5, 3, 3), (1, 2, 1), 4),
    ((64, 32, 10), (1, 1, 0), 4),     # the largest region without halo
    ((62, 30, 7), (0, 0, 2), 4),      # one pair over the periodic tile, odd z
    ((65, 33, 13), (2, 1, 1), 4),
    ((121, 57, 9), (1, 2, 2), 3),     # last tiles of odd width
    ((24, 20, 40), (0, 0, 1), 4),     # moving walls, several chunks
    ((720, 400, 4), (0, 0, 0), 2),    # more columns of tiles than SMs
])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_one_launch_equals_half_sweeps(shape, wall, steps, storage):
    from paper_2311_15242_gb300 import Solver
    nx, ny, nz = shape
    cfg = W.shear_droplet_3d(nx=nx, ny=ny, nz=nz, R=min(shape) / 3.0)
    cfg["wall"] = list(wall)
    if wall[2] != 1:  # (only bounce-back walls move)
        cfg["uw_lo"] = cfg["uw_hi"] = [[0.0] * 3] * 3
    f = W.initial_fields(cfg, seed=5, noise=0.02, u0=1e-3)
    out, d = {}, {}
    for on in (True, False):
        s = Solver(cfg, storage=storage)
        s.set_sor_persistent(on)
        s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
        s.step(steps)
        out[on], d[on] = s.fields(), s.diagnostics()
        s.close()
    err = errors(out[False], out[True])
    if storage == "f32":
        assert within(err, F32_IMPL_TOL), err
    else:  # (an FP32 rounding may send a 16-bit value to its other neighbour)
        assert max(err.values()) < 2e-2, err
    assert d[True]["sor_iters_psi"] == d[False]["sor_iters_psi"]
