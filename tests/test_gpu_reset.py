"""Evaluators after a device reset: problems made on the new context solve as
those before it did, where N_max needs more shared memory than a kernel's
default limit.  A process of its own resets its own context, between calls,
with nothing in flight and every object of the old context destroyed."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes
import numpy as np
import paper_2609_21803_gb300 as P
import workloads as W

P.lib()
rt = ctypes.CDLL("libcudart.so.13")  # the runtime that the library has loaded


def ok(e):
    assert e == 0, e


class Dev:
    # a device array of the runtime
    def __init__(self, a):
        self.a, self.p = a, ctypes.c_void_p()
        ok(rt.cudaMalloc(ctypes.byref(self.p), ctypes.c_size_t(a.nbytes)))
        ok(rt.cudaMemcpy(self.p, ctypes.c_void_p(a.ctypes.data), ctypes.c_size_t(a.nbytes), 1))

    def back(self):
        ok(rt.cudaMemcpy(ctypes.c_void_p(self.a.ctypes.data), self.p, ctypes.c_size_t(self.a.nbytes), 2))
        ok(rt.cudaFree(self.p))
        return self.a.copy()


def solve(task):
    big = W.bimanual_instance(0) if task == "bimanual" else W.push_l4_instance(0)
    big = dict(big, knots_per_segment=30 if task == "bimanual" else 100, max_segments=6 if task == "bimanual" else 4)
    n, L = 3, big["max_segments"]
    seqs = np.random.default_rng(4).integers(0, 507 if task == "bimanual" else 12, (n, L))
    packed = P.pack_mode_seqs([tuple(int(m) for m in s) for s in seqs])
    d = Dev(packed.view(np.uint8).reshape(n, P.MODE_SEQ_BYTES).copy())
    cost, status = Dev(np.zeros(n, np.float32)), Dev(np.full(n, -1, np.int32))
    if task == "noalloc":
        P.comet_eval_modes_noalloc([big], None, None, d.p.value, n, None, cost.p.value, None, status.p.value)
    else:
        p = P.comet_problem_create([big])
        if task == "timed":
            P.comet_eval_modes_timed(p, dict(h_min=0.05, h_max=0.2, T_max=100.0), d.p.value, n, None, 4, cost.p.value,
                                     None, status.p.value)
        else:
            P.comet_eval_modes_budget(p, d.p.value, n, None, 4, cost.p.value, None, status.p.value)
        ok(rt.cudaDeviceSynchronize())
        P.comet_problem_destroy(p)
    ok(rt.cudaDeviceSynchronize())
    d.back()
    return cost.back(), status.back()


tasks = ("push", "timed", "bimanual", "noalloc")
before = [solve(t) for t in tasks]
ok(rt.cudaDeviceReset())
for t, (c, s) in zip(tasks, before):
    c2, s2 = solve(t)
    assert (c.view(np.int32) == c2.view(np.int32)).all() and (s == s2).all() and (s >= 0).all(), t
    print(t, c.tolist(), s.tolist())
"""


def test_problems_made_after_a_device_reset():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_21803_gb300 import build as B
    B.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
