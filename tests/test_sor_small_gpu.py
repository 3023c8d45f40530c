"""FP64, variant 0 on a grid of few tiles: the 16 x 8 tile against variant 2
(16 x 16, the same sweeps a round) in both forms, one launch and one a round: the
same iterates, so as many sweeps and fields that differ by the order in which the
total is summed (1e-12 of a field's largest value).  Sizes around a tile, smaller
than its halo, an odd periodic axis (the list form), every kind of boundary; and
grids at which the rule's choices end: half as many 32 x 16 tiles as SMs, one more;
more tiles than SMs."""
import pytest

import workloads as W
from test_parity_gpu import errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,wall", [
    ((16, 8), (0, 0)), ((17, 9), (1, 2)), ((15, 7), (0, 1)), ((6, 4), (0, 0)), ((31, 33), (0, 0)),
    ((64, 40), (2, 1)), ((128, 304), (0, 1)), ((128, 305), (0, 1)), ((416, 384), (0, 0)),
])
def test_small_tile_equals_the_larger(shape, wall):
    from paper_2311_15242_gb300 import Solver
    nx, ny = shape
    cfg = W.droplet_adsorption_2d(n=nx, R=max(min(shape) / 3.0, 2.0), C0=0.5)
    cfg.update(ny=ny, wall=[*wall, 0], center=[(nx - 1) / 2 + 0.2, (ny - 1) / 2 - 0.1, 0.0], psi0=0.3)
    f = W.initial_fields(cfg, seed=4, noise=0.02, u0=1e-4)
    out, sweeps = [], []
    for tile, on in ((0, True), (0, False), (2, False)):
        s = Solver(cfg, storage="f64")
        s.set_sor_tile(tile)
        s.set_sor_persistent(on)
        s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
        s.step(5)
        out.append(s.fields())
        sweeps.append(s.diagnostics()["sor_iters_psi"])
        s.close()
    assert sweeps[0] == sweeps[1] == sweeps[2]
    for o in out[1:]:
        err = errors(out[0], o)
        assert max(err.values()) < 1e-12, err
