"""The fused step of a batch (one launch an instance, side by side on streams of
the batch) against a context of each instance's own: the same tile code, so the
fields agree to the rounding of two compilations (F32_IMPL_TOL; 16-bit storage
2e-2, where a rounding may send a population to its other neighbour) and the
sweeps are as many.  More instances than streams; few enough tiles for the small
ones; a change of the SOR tile at an odd step, where the populations are in the
second set, to a form with a launch a round and back; an instance taken out and
put back."""
import pytest

import workloads as W
from test_parity_gpu import F32_IMPL_TOL, errors, within

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("sizes", [
    [(34 + 6 * k, 90 + 13 * k) for k in range(11)],   # 190 tiles of 32 x 16
    [(33, 17), (16, 8), (31, 40)],                    # small tiles; walled odd widths
    [(64, 40)],
])
def test_fused_batch_equals_single_contexts(sizes, storage):
    from paper_2311_15242_gb300 import Batch, Solver
    cfgs = [W.bubble_rise_2d(nx=nx, ny=ny, D_b=min(nx, ny) / 2.5, Eo=2.0 + k)
            for k, (nx, ny) in enumerate(sizes)]
    fs = [W.initial_fields(c, seed=k, noise=0.02, u0=1e-4) for k, c in enumerate(cfgs)]
    b = Batch(cfgs, storage=storage)
    for k, f in enumerate(fs):
        b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
    plan = [(7, 0), (4, 7), (6, 0)]
    for i, (steps, tile) in enumerate(plan):
        b.set_tiles(32, 8, tile)
        if len(sizes) > 1:
            b.set_active(0, i != 1)
        b.step(steps)
    assert b.status() == [0] * len(cfgs)
    d = b.diagnostics()
    for k, (c, f) in enumerate(zip(cfgs, fs)):
        s = Solver(c, storage=storage)
        s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
        for i, (steps, tile) in enumerate(plan):
            if len(sizes) > 1 and k == 0 and i == 1:
                continue
            s.set_sor_tile(tile)
            s.step(steps)
        err = errors(s.fields(), b.fields(k))
        if storage == "f32":
            assert within(err, F32_IMPL_TOL), (k, err)
        else:
            assert max(err.values()) < 2e-2, (k, err)
        assert s.diagnostics()["sor_iters_psi"] == d[k]["sor_iters_psi"]
        s.close()
    b.close()
