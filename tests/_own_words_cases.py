"""Cases of test_gpu_own_words.py, run in a process of its own with the debug
build, whose base case can be made to fail between its two launches
(LR_INJECT_LAUNCH_FAIL=1: on the host, nothing fails on the GPU).

The failed call has an out-of-range successor, whose error bit it leaves in
the words that the two launches share: no later call may report it."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import gen  # noqa: E402
import oracle  # noqa: E402
import torch  # noqa: E402
import paper_2606_09318_gb300 as lr  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def capture(side, s, out):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        lr.rank(s, out=out, max_lists=1, sync=False)
    return g


def case(n, later):
    good = gen.random_list(n, 620)
    want = oracle.rank(good)
    bad = good.copy()
    bad[5] = n
    s, b, out = dev(good), dev(bad), torch.empty(n, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(lr.rank(s, max_lists=1, stream=side).cpu().numpy(), want)
    g = capture(side, s, out)                          # the words are clean: the graph holds no clear
    os.environ["LR_INJECT_LAUNCH_FAIL"] = "1"
    try:
        lr.rank(b, max_lists=1, stream=side)
        raise AssertionError("the call did not fail")
    except lr.LRError as e:
        assert e.name == "LR_ERR_CUDA", e
    os.environ["LR_INJECT_LAUNCH_FAIL"] = "0"
    thrown = capture(side, s, out)                     # captured, never run
    if later == "replay":
        with torch.cuda.stream(side):
            g.replay()
        assert lr.device_status(side) == 0
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    for _ in range(2):
        np.testing.assert_array_equal(lr.rank(s, max_lists=1, stream=side).cpu().numpy(), want)
    del thrown


if __name__ == "__main__":
    assert lr.lib_path().endswith("liblr_debug.so"), lr.lib_path()
    case(int(sys.argv[1]), sys.argv[2])
    print("ok")
