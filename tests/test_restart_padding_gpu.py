"""A restart into a fresh context whose memory held other things before: rows of
odd length are padded, and what lies in the padding (here: NaN in every word of
the workspace) is nobody's value.  The steps after lbs_load_state are the
uninterrupted run's, bit for bit; psi and C's second buffers are written by no
one before the first solve."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("on", [True, False], ids=["one_launch", "launches"])
@pytest.mark.parametrize("cfg,storage", [
    (W.bubble_rise_3d(R=5, shape=(5, 5, 6)), "f32"),                 # 25 x 25 x 30, walls on x and y
    (W.bubble_rise_3d(R=5, shape=(5, 5, 6)), "bf16"),
    (W.adsorption_octant_3d(R=13), "f32"),                           # 65: two tiles along x
    (W.adsorption_octant_3d(R=7), "f64"),
    (W.bubble_rise_2d(nx=65, ny=91, D_b=24.0, Eo=3.0), "f32"),
    (W.bubble_rise_2d(nx=33, ny=57, D_b=12.0, Eo=3.0), "f64"),
], ids=lambda v: v if isinstance(v, str) else "%dx%dx%d" % (v["nx"], v["ny"], v["nz"]))
def test_restart_into_memory_full_of_nan(cfg, storage, on, monkeypatch):
    import torch

    from paper_2311_15242_gb300 import Solver
    f = W.initial_fields(cfg, seed=4, noise=0.02, u0=1e-3)
    a = Solver(cfg, storage=storage)
    a.set_sor_persistent(on)
    a.init_fields(f["phi"], f["psi"], f["C"], f["u"])
    a.step(3)
    state = a.save_state()
    a.step(5)

    plain = torch.empty

    def dirty(*args, **kw):
        t = plain(*args, **kw)
        if t.is_cuda:
            t.view(torch.uint8).fill_(255)
            torch.cuda.synchronize()
        return t

    with monkeypatch.context() as m:
        m.setattr(torch, "empty", dirty)
        b = Solver(cfg, storage=storage)
    assert int(b.ws[-1]) == 255
    b.set_sor_persistent(on)
    b.load_state(state)
    b.step(5)
    x, y = a.fields(), b.fields()
    assert {k: int((x[k] != y[k]).sum()) for k in x} == dict.fromkeys(x, 0)
    a.close()
    b.close()
