"""A batch whose CUDA calls fail: the failure is reported by the call that met it,
nothing is launched on lists that are not there, and the batch goes on once the
cause is gone.  The failures are made on the host: a preloaded stand-in for
cudaMalloc and the launch calls returns an error code for the n-th call it is armed
for (a child process, so that no other test sees it)."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STAND_IN = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
typedef struct { unsigned x, y, z; } dim3;
static int kind, left;
void fake_arm(int k, int n) { kind = k; left = n; }
int fake_left(void) { return left; }
static int hit(int k) { return kind == k && left > 0 && --left == 0; }
static void *real(const char *name) {
    static void *rt;
    if (!rt) rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    if (!rt) rt = dlopen("libcudart.so.13", RTLD_LAZY);
    return dlsym(rt, name);
}
int cudaMalloc(void **p, size_t n) {
    static int (*f)(void **, size_t);
    if (!f) f = real("cudaMalloc");
    if (hit(1)) { *p = 0; return 2; }  /* cudaErrorMemoryAllocation */
    return f(p, n);
}
#define LAUNCH(name)                                                                     \
    int name(const void *k, dim3 g, dim3 b, void **a, size_t m, void *s) {               \
        static int (*f)(const void *, dim3, dim3, void **, size_t, void *);              \
        if (!f) f = real(#name);                                                         \
        if (hit(2)) return 701; /* cudaErrorLaunchOutOfResources */                      \
        return f(k, g, b, a, m, s);                                                      \
    }
LAUNCH(cudaLaunchKernel)
LAUNCH(__cudaLaunchKernel)
"""

CHILD = r"""
import ctypes, json, os, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import workloads as W
from paper_2311_15242_gb300 import Batch
from paper_2311_15242_gb300.lbs import LBS_ECUDA, LbsError
fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
MALLOC, LAUNCH = 1, 2
cfgs = [W.bubble_rise_2d(nx=64 + 16 * k, ny=150 + 31 * k, D_b=24.0, Eo=2.0 + k) for k in range(4)]
fs = [W.initial_fields(c, seed=k, noise=0.02, u0=1e-3) for k, c in enumerate(cfgs)]

def make(graph=True):
    b = Batch(cfgs, storage="f32")
    b.set_graph(graph)
    for k, f in enumerate(fs):
        b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
    return b

def fails(call):
    try:
        call()
    except LbsError as e:
        return e.code == LBS_ECUDA
    return False

def same(b, steps):
    r = make()
    r.step(steps)
    ok = all(np.array_equal(x[q], y[q]) for x, y in ((b.fields(k), r.fields(k)) for k in range(4)) for q in x)
    r.close()
    return ok

out = {}
for n in (1, 4):  # the first and the last instance's launch
    b = make()
    fake.fake_arm(LAUNCH, n)
    out["capture %d" % n] = fails(lambda: b.step(1)) and fake.fake_left() == 0
    fake.fake_arm(0, 0)
    b.step(9)
    out["after capture %d" % n] = same(b, 9)
    b.close()
    b = make(graph=False)
    fake.fake_arm(LAUNCH, n)
    out["launch %d" % n] = fails(lambda: b.step(1)) and fake.fake_left() == 0
    fake.fake_arm(0, 0)
    for k, f in enumerate(fs):
        b.init_fields(k, f["phi"], f["psi"], f["C"], f["u"])
    b.step(3)
    out["after launch %d" % n] = same(b, 3)
    b.close()
if "lists" in sys.argv:
    for n in (1, 2, 3, 4):  # cells, SOR tiles, strips, gangs
        b = make()
        b.step(2)
        b.sync()
        fake.fake_arm(MALLOC, n)
        out["tiles %d" % n] = fails(lambda: b.set_tiles(32, 8, 0)) and fake.fake_left() == 0
        fake.fake_arm(0, 0)
        out["no step %d" % n] = fails(lambda: b.step(1))
        b.set_tiles(32, 8, 0)
        b.step(3)
        out["after tiles %d" % n] = same(b, 5)
        fake.fake_arm(MALLOC, n)
        out["active %d" % n] = fails(lambda: b.set_active(1, False))
        fake.fake_arm(0, 0)
        out["no step again %d" % n] = fails(lambda: b.step(1))
        b.set_active(1, False)
        b.set_active(1, True)
        b.step(2)
        out["after active %d" % n] = same(b, 7)
        b.close()
print(json.dumps(out))
"""


def test_failed_calls_of_a_batch(tmp_path):
    src, lib, child = tmp_path / "fake.c", tmp_path / "libfake.so", tmp_path / "child.py"
    src.write_text(STAND_IN)
    child.write_text(CHILD)
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", str(src), "-o", str(lib), "-ldl"])
    r = subprocess.run([sys.executable, str(child), ROOT, "lists"], capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=str(lib)), timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(out) == 32 and all(out.values()), {k: v for k, v in out.items() if not v}
