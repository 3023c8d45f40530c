"""The resident solve (k_solve2; kb_solve2 of a batch) against the launches of
one round each: the same total, the same rescale, the same stop.

Both sum exact products in compensated FP32 strips and the strips in FP64.  The
strips' errors (2^-48 of a strip) average out over 10^3 and more of them, and an
FP64 sum of some 20 levels is off by 2^-53 times about their root: two ulps of
the total (2^-52 of it each) and one to spare.  Sums of FP32 pairs up to the grid
are off by 4 to 8."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOTAL_TOL = 3 * 2.0 ** -52


def solver(cfg, f, storage, on, variant=0):
    from paper_2311_15242_gb300 import Solver
    s = Solver(cfg, storage=storage)
    s.set_sor_tile(variant)
    s.set_sor_persistent(on)
    s.init_fields(f["phi"], f["psi"], f["C"], f["u"])
    return s


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n,variant", [(128, 0), (251, 0), (400, 0), (400, 5), (500, 0), (600, 0)])
def test_total_is_summed_in_double_precision(n, variant, storage):
    """One step: the solves' inputs are the same, and so are psi and C but for
    cells that hold less than 1e-14 of the largest value."""
    cfg = W.droplet_adsorption_2d(n=n, R=n * 0.2)
    f = W.initial_fields(cfg, seed=5, noise=0.02, u0=1e-3)
    pre = []
    for on in (True, False):
        s = solver(cfg, f, storage, on, variant)
        s.step(1)
        pre.append(s.step_result()[1])
        s.close()
    assert abs(pre[0] / pre[1] - 1.0) <= TOTAL_TOL, pre


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_totals_of_a_batch_of_several_waves(storage):
    """Nine instances (more than one wave of tiles) against their own contexts
    with a launch a round."""
    from paper_2311_15242_gb300 import Batch
    cfgs = [W.droplet_adsorption_2d(n=200 + 24 * k, R=40.0 + 4 * k) for k in range(9)]
    fs = [W.initial_fields(c, seed=k, noise=0.02, u0=1e-3) for k, c in enumerate(cfgs)]
    b = Batch(cfgs, storage=storage)
    for k, f in enumerate(fs):
        b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
    b.step(1)
    d = b.diagnostics()
    b.close()
    for k, (c, f) in enumerate(zip(cfgs, fs)):
        s = solver(c, f, storage, False)
        s.step(1)
        assert abs(d[k]["surf_pre_rescale"] / s.step_result()[1] - 1.0) <= TOTAL_TOL, k
        s.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("cfg,variant", [
    (W.bubble_rise_2d(nx=64, ny=517, D_b=32.0, Eo=5.0, Bi=0.3), 0),    # odd periodic y
    (W.bubble_rise_2d(nx=241, ny=300, D_b=64.0, Eo=10.0), 0),          # odd, walled x
    (W.bubble_rise_2d(nx=256, ny=1024, D_b=64.0, Eo=10.0), 0),
    (W.bubble_rise_2d(nx=128, ny=400, D_b=48.0, Eo=3.0), 3),           # 4 sweeps a round
    (W.droplet_adsorption_2d(n=400, R=75.0), 0),                       # tails down to 1e-37
    (W.droplet_adsorption_2d(n=63, R=15.0), 0),                        # odd: not resident
], ids=["64x517", "241x300", "256x1024", "128x400-4", "droplet400", "droplet63"])
def test_fields_equal_round_launches_to_the_bit(cfg, variant, storage):
    """The same roundings in the weights and in every sweep.  Density ratio 10
    (a factor 1 / rho^R0 whose product rounds) and FP16 populations, where
    one different bit would send others after it."""
    f = W.initial_fields(cfg, seed=5, noise=0.02, u0=1e-3)
    s = [solver(cfg, f, storage, on, variant) for on in (True, False)]
    for n in (1, 1, 10):
        for q in s:
            q.step(n)
        a, b = s[0].fields(), s[1].fields()
        assert {k: int((a[k] != b[k]).sum()) for k in a} == dict.fromkeys(a, 0)
        a, b = s[0].macro(), s[1].macro()
        assert {k: int((a[k] != b[k]).sum()) for k in a} == dict.fromkeys(a, 0)
    for q in s:
        q.close()


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_a_long_run_keeps_the_bits(storage):
    """1000 steps of the 40 x 72 bubble.  On a grid of so few warps a total that is
    a few times FP64's error off rounds the rescale step apart within some hundred
    steps, and the runs part."""
    from test_parity_gpu import bubble
    cfg = bubble()
    f = W.initial_fields(cfg, seed=7, noise=0.02)
    out = []
    for on in (True, False):
        s = solver(cfg, f, storage, on)
        s.step(1000)
        out.append(s.fields())
        s.close()
    assert {k: int((out[0][k] != out[1][k]).sum()) for k in out[0]} == dict.fromkeys(out[0], 0)
