"""The tiled 3D stencil kernels (gradient, force, collision: 16 x 8 cells on 4
planes, 2 in FP64) and the streaming kernel's plain pulls (warps none of whose
links cross a boundary) against the FP64 oracle, at sizes around the edges of a
tile: one cell less and more than a tile, grids smaller than its halo, rows
with a warp between the boundary ones; every kind of boundary on every axis.
Tolerances: those of the 3D parity tests (FP64 1e-9; FP32 F32_TOL, which is
relative to the flow between moving walls on z, so FP32 runs with those)."""
import pytest

import workloads as W
from test_parity_gpu import F32_TOL, errors, run_both, within

pytestmark = pytest.mark.gpu


def run(shape, wall, storage):
    nx, ny, nz = shape
    cfg = W.shear_droplet_3d(nx=nx, ny=ny, nz=nz, R=max(min(shape) / 3.0, 2.0))
    cfg["wall"] = list(wall)
    cfg["center"] = [(nx - 1) / 2 + 0.3, (ny - 1) / 2 - 0.2, (nz - 1) / 2 + 0.1]
    if wall[2] != 1:  # (only bounce-back walls move)
        cfg["uw_lo"] = cfg["uw_hi"] = [[0.0] * 3] * 3
    o, s = run_both(cfg, 8, storage, u0=1e-4)
    return errors(o.fields(), s.fields())


SHAPES = [((16, 8, 4), (0, 0, 0)), ((17, 9, 5), (1, 2, 1)), ((15, 7, 3), (2, 1, 2)),
          ((4, 4, 2), (0, 0, 0)), ((3, 3, 3), (1, 1, 1)), ((18, 10, 6), (0, 1, 0)),
          ((100, 10, 9), (0, 0, 1)), ((99, 9, 8), (2, 1, 0))]


@pytest.mark.parametrize("shape,wall", SHAPES)
def test_tiles_match_oracle_f64(shape, wall):
    err = run(shape, wall, "f64")
    assert max(err.values()) < 1e-9, err


@pytest.mark.parametrize("shape,wall", [k for k in SHAPES if k[0][2] > 2])
def test_tiles_match_oracle_f32(shape, wall):
    err = run(shape, (*wall[:2], 1), "f32")
    assert within(err, F32_TOL), err
