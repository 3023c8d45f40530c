"""The fused 2D step with the small tile (16 x 8 cells) that grids of few
32 x 16 tiles get, at the edges of its tiles: sides one off a multiple of the
tile, walls and mirror planes inside the last tile, a grid smaller than a
tile, and the sizes on both sides of the choice (FP64 152 tiles, FP32 76),
against the oracle; FP64 differs by rounding order only (1e-9), FP32 by the
bounds of test_parity_gpu."""
import pytest

import workloads as W
from oracle.ora import Oracle
from test_parity_gpu import F32_TOL, droplet, errors, within

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,wall", [
    (7, 5, (1, 1, 0)), (17, 9, (1, 0, 0)), (33, 24, (2, 1, 0)), (31, 23, (0, 0, 0)),
    (65, 513, (1, 0, 0)), (64, 608, (0, 2, 0)),
])
def test_small_tile_matches_oracle(nx, ny, wall, storage):
    from paper_2311_15242_gb300 import Solver
    cfg = droplet(nx=nx, ny=ny, R=min(nx, ny) / 4.0)
    cfg.update(wall=list(wall))
    f = W.initial_fields(cfg, seed=5, noise=0.02, u0=1e-4)
    o = Oracle(cfg)
    o.init_fields(f["phi"], f["psi"], f["C"], f["u"])
    o.step(8)
    s = Solver(cfg, storage=storage)
    s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
    s.step(8)
    err = errors(o.fields(), s.fields())
    s.close()
    if storage == "f64":
        assert max(err.values()) < 1e-9, err
    else:
        assert within(err, F32_TOL), err
