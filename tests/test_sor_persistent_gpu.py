"""lbs_set_sor_persistent on FP64 grids of more tiles than SMs: a launch a round by
default (which is faster there), one launch when asked for, and back; the same
iterates, so FP64 fields agree to the rounding of the totals (1e-12)."""
import pytest

import workloads as W
from test_parity_gpu import errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,variant,default", [
    (400, 400, 0, False),  # 325 tiles of 32 x 16
    (400, 400, 5, False),  # 169 of 32 x 32
    (160, 160, 0, True),   # small tiles
])
def test_one_launch_when_asked_for(nx, ny, variant, default):
    from paper_2311_15242_gb300 import Solver
    cfg = W.droplet_adsorption_2d(n=nx, R=60.0)
    cfg.update(ny=ny)
    f = W.initial_fields(cfg, seed=3, noise=0.02, u0=1e-4)
    out = []
    for calls in ([], [True], [False], [False, True]):
        s = Solver(cfg, storage="f64")
        s.set_sor_tile(variant)
        for on in calls:
            s.set_sor_persistent(on)
        one = calls[-1] if calls else default
        assert (s.kernel_count() == 2) == one, calls
        s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
        s.step(3)
        out.append(s.fields())
        s.close()
    for o in out[1:]:
        assert max(errors(out[0], o).values()) < 1e-12
