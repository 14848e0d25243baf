"""Host calls from a thread with a small stack (64 KB, as a host application's
worker threads may have): the sort's layout is counted without its tables."""

import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CALL = """
import ctypes, threading
import synth
from paper_2602_23040_gb300 import api, _native as N
v = [synth.scenes.pinhole((0, 0, -3), 64, 48)] * {views}
p = api.Plan([(32, 32, 0, 0, 0)], (32, 32), 3, 1, "f32", v, 500)
lib, s, rc = N.load(), N.Sizes(), []
threading.stack_size(64 << 10)
t = threading.Thread(target=lambda: rc.append(lib.pk_plan_sizes(p.handle, ctypes.byref(s))))
t.start()
t.join()
assert rc == [0] and s.bin_kernels == p.sizes.bin_kernels > 0
"""


@pytest.mark.parametrize("views", [1, 3, 208])
def test_plan_sizes_on_a_small_stack(views):
    from paper_2602_23040_gb300 import build
    try:
        build.build()
    except RuntimeError as e:          # no nvcc on this machine
        pytest.skip(str(e))
    r = subprocess.run([sys.executable, "-c", CALL.format(views=views)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
