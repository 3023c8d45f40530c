"""Batches of many small instances: the step up to the moments of t+1 is three
launches over all of them, not one an instance (which took 1.7 to 5.8 times as
long).  Both sides of the rule's lines (16 instances; 2^14 cells an instance).
Their solves in one launch and, where an odd periodic width keeps the batch from
it, a launch a round: the same bits; and both against the oracle (F32_TOL of
test_parity_gpu)."""
import numpy as np
import pytest

import workloads as W
from oracle.ora import Oracle
from test_parity_gpu import F32_TOL, droplet, errors, within

pytestmark = pytest.mark.gpu


def bubbles(sizes):
    return [W.bubble_rise_2d(nx=nx, ny=ny, D_b=min(nx, ny) / 2.5, Eo=2.0 + k % 7)
            for k, (nx, ny) in enumerate(sizes)]


def batch(cfgs, fs, storage):
    from paper_2311_15242_gb300 import Batch
    b = Batch(cfgs, storage=storage)
    for k, f in enumerate(fs):
        b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
    return b


def initial(cfgs):
    return [W.initial_fields(c, seed=k, noise=0.02, u0=1e-4) for k, c in enumerate(cfgs)]


RAGGED = [(33, 17), (16, 8), (31, 40)] * 6           # odd walled widths
WAVES = [(64, 100 + 3 * k) for k in range(40)]       # more tiles than SMs


@pytest.mark.parametrize("sizes,launches", [
    ([(32, 48)] * 64, 4),
    (RAGGED, 4),
    ([(24 + 3 * k, 40 + 7 * k) for k in range(17)], 4),
    ([(24 + 3 * k, 40 + 7 * k) for k in range(16)], 17),
    ([(128, 128)] * 17, 18),                         # the line itself
    ([(128, 128)] * 16 + [(128, 127)], 4),
], ids=["64", "ragged", "17", "16", "large", "below"])
def test_launches_of_a_step(sizes, launches):
    """The fused steps (one an instance) or three phases, and the solves."""
    cfgs = bubbles(sizes)
    from paper_2311_15242_gb300 import Batch
    b = Batch(cfgs, storage="f32")
    assert b.kernel_count() == launches
    b.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("sizes", [RAGGED, WAVES], ids=["ragged", "waves"])
def test_gangs_equal_round_launches_to_the_bit(sizes, storage):
    """Steps that end at odd ones, an instance taken out and put back."""
    cfgs = bubbles(sizes)
    fs = initial(cfgs)
    odd = droplet(nx=45, ny=40)
    got, its = [], []
    for extra in ([], [odd]):
        b = batch(cfgs + extra, fs + [W.initial_fields(odd, seed=99)] * len(extra), storage)
        for on, steps in ((True, 7), (False, 4), (True, 6)):
            b.set_active(1, on)
            b.step(steps)
        assert b.status() == [0] * (len(cfgs) + len(extra))
        got.append([b.fields(k) for k in range(len(cfgs))])
        its.append([d["sor_iters_psi"] for d in b.diagnostics()[:len(cfgs)]])
        b.close()
    assert its[0] == its[1]
    differ = {(k, q): int((x[q] != y[q]).sum()) for k, (x, y) in enumerate(zip(*got)) for q in x}
    assert not any(differ.values()), {k: v for k, v in differ.items() if v}


def test_small_instances_match_the_oracle():
    cfgs = bubbles(RAGGED)
    fs = initial(cfgs)
    b = batch(cfgs, fs, "f32")
    b.step(12)
    for k in (0, 1, 2, 17):
        o = Oracle(cfgs[k])
        f = fs[k]
        o.init_fields(f["phi"], f["psi"], f["C"], f["u"])
        o.step(12)
        err = errors(o.fields(), b.fields(k))
        assert within(err, F32_TOL), (k, err)
    b.close()


def test_small_instances_after_a_wait_that_ran_out():
    """Their solves' barriers start clear again."""
    from paper_2311_15242_gb300.lbs import LBS_ETIMEOUT
    cfgs = bubbles([(48, 130)] * 18)
    fs = initial(cfgs)
    got = []
    for limit in (1, 1 << 24):
        b = batch(cfgs, fs, "f32")
        b.set_sor_wait_limit(limit)
        b.step(3)
        assert b.status() == [LBS_ETIMEOUT if limit == 1 else 0] * 18
        b.set_sor_wait_limit(1 << 24)
        for k, f in enumerate(fs):
            b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
        b.step(5)
        assert b.status() == [0] * 18
        got.append([b.fields(k) for k in range(18)])
        b.close()
    assert all(np.array_equal(x[q], y[q]) for x, y in zip(*got) for q in x)
