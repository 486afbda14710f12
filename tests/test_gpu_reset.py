"""A device reset after pm_shutdown: the grouped model calls of every thread get
new page-locked memory, also where another thread shut down.  The reset ends the
context of a child process only."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes, threading
import numpy as np
import oracle as O
import paper_2605_04178_gb300 as pm
theta = O.prior_theta(152)
M = [100, 200, 300]
t_o, bm_o, bn_o, launch_o = O.grouped_autotune(np.array(M, np.int32), 1024, 512, 1, theta, 152)
out, first, reset = [], threading.Event(), threading.Event()

def work():
    out.append(pm.pm_grouped_autotune(M, 1024, 512, 1, theta, 152, stream=0))
    first.set()
    reset.wait()
    out.append(pm.pm_grouped_autotune(M, 1024, 512, 1, theta, 152, stream=0))
    out.append(pm.pm_grouped_predict(M, 1024, 512, *out[-1][1:3], *out[-1][3], 1, theta, 152, stream=0))

t = threading.Thread(target=work)
t.start()
assert first.wait(60)
pm.pm_shutdown()
assert ctypes.CDLL("libcuda.so.1").cuDevicePrimaryCtxReset_v2(0) == 0
reset.set()
t.join()
assert len(out) == 3 and out[0] == out[1] and out[2] == out[0][0]
assert abs(out[0][0] - t_o) <= 1e-5 * t_o
print("ok")
"""


def test_reset_after_another_threads_shutdown():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr
