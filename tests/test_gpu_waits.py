"""A call that waits on the host gives up its core where the caller asked for
that (a primary context with blocking waits): behind 0.3 s of other work on
the stream, the waiting thread must have used little processor time."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import ctypes, time
cu = ctypes.CDLL("libcuda.so.1")
dev = ctypes.c_int()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(dev, 4) == 0                # CU_CTX_SCHED_BLOCKING_SYNC
import numpy as np, torch
import gen, oracle
import paper_2606_09318_gb300 as lr
for kind, n in (("random", (1 << 20) + 3), ("locality", 600_011)):       # the sums; the contracted nodes
    succ = gen.list_of_order_kind(kind, n, 630)
    s = torch.from_numpy(succ.view(np.int32)).cuda()
    want = oracle.rank(succ)
    np.testing.assert_array_equal(lr.rank(s).cpu().numpy(), want)
    torch.cuda.synchronize()
    torch.cuda._sleep(int(0.3 * 2.0e9))
    wall, cpu = time.perf_counter(), time.thread_time()
    out = lr.rank(s)
    wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
    np.testing.assert_array_equal(out.cpu().numpy(), want)
    print(kind, "waited %.3f s, used %.3f s" % (wall, cpu))
    assert wall > 0.1 and cpu < wall / 4, (kind, wall, cpu)
"""


def test_blocking_waits_are_honoured():
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
