"""The words that a base-case call shares between its two launches, when a
call fails between them (injected on the host with LR_INJECT_LAUNCH_FAIL=1:
nothing fails on the GPU) and when a capture is thrown away.

The failed call here has an out-of-range successor, whose error bit it leaves
in those words: no later call may report it."""
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
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def capture(side, s, out):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        lr.rank(s, out=out, max_lists=1, sync=False)
    return g


@pytest.mark.parametrize("n", [6000, 100_003])        # without and with marks of predecessors
@pytest.mark.parametrize("later", ["call", "replay"])
def test_after_a_call_that_failed_on_the_way(monkeypatch, n, later):
    good = gen.random_list(n, 620)
    want = oracle.rank(good)
    bad = good.copy()
    bad[5] = n
    s, b, out = dev(good), dev(bad), torch.empty(n, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(lr.rank(s, max_lists=1, stream=side).cpu().numpy(), want)
    g = capture(side, s, out)                          # the words are clean: the graph holds no clear
    monkeypatch.setenv("LR_INJECT_LAUNCH_FAIL", "1")
    with pytest.raises(lr.LRError) as e:
        lr.rank(b, max_lists=1, stream=side)
    assert e.value.name == "LR_ERR_CUDA"
    monkeypatch.delenv("LR_INJECT_LAUNCH_FAIL")
    thrown = capture(side, s, out)                     # captured, never run
    if later == "replay":
        with torch.cuda.stream(side):
            g.replay()
        assert lr.device_status(side) == 0
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    for _ in range(2):
        np.testing.assert_array_equal(lr.rank(s, max_lists=1, stream=side).cpu().numpy(), want)
    del thrown
