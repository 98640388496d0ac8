"""A profiled call is the call that it would be without profiling: the same
kernel launches, the same ranks, and one level-0 chase among its phases."""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_09318_gb300 as lr  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32 if a.dtype == np.uint32 else a.dtype)).cuda()


def single(kind, n, seed, **kw):
    succ = gen.forest(n, seed, n_long=3, long_len=n // 8, mean_short=40)[0] if kind == "forest" else \
        gen.list_of_order_kind(kind, n, seed)
    s = dev(succ)
    return lambda: lr.rank(s, **kw), oracle.rank(succ)


def batch():
    offsets, succ, w = gen.batch_instances(40, 640, lo_exp=10.0, hi_exp=17.0)
    o, s, x = dev(offsets), dev(succ), dev(w)
    return lambda: lr.rank_batch(o, s, x), oracle.rank_batch(offsets, succ, w, np.int64)


CASES = {"list": lambda: single("random", (1 << 20) + 3, 641),
         "sampled list": lambda: single("random", (1 << 22) + 3, 642),
         "forest": lambda: single("forest", (1 << 20) + 3, 643),
         "validated": lambda: single("forest", (1 << 20) + 3, 644, validate=True),
         "contracted": lambda: single("locality", (1 << 22) + 3, 645),
         "batch": batch}


@pytest.mark.parametrize("name", list(CASES))
def test_profiled_route(name):
    call, want = CASES[name]()
    np.testing.assert_array_equal(call().cpu().numpy(), want)
    counts = []
    for on in (False, True):
        lr.profile_enable(on)
        lr.profile_read(reset=True)
        before = lr.kernel_launch_count()
        try:
            np.testing.assert_array_equal(call().cpu().numpy(), want)
        finally:
            lr.profile_enable(False)
        counts.append(lr.kernel_launch_count() - before)
    prof = lr.profile_read(reset=True)
    assert counts[0] == counts[1]
    assert prof["calls"] == 1 and prof["chase0_launches"] == 1
    assert prof["ms_prep"] > 0 and prof["ms_chase0"] > 0 and prof["ms_finalize"] > 0
