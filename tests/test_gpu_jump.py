"""The pointer-jumping base case (k_jump), reached through lr_rank with ruler
fractions that leave it levels of one element, of about one element per
thread, of several per thread and of more than one pass over the grid, against
the oracle; and invalid lists that only the base case can notice."""
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
    a = np.ascontiguousarray(a)
    return torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).cuda()


def status_of(succ, **kw):
    try:
        lr.rank(dev(succ), **kw)
        return "LR_OK"
    except lr.LRError as e:
        return e.name


@pytest.mark.parametrize("n,f0", [(1, 2), (2, 2), (257, 2), (12288, 2), (12289, 12289), (155_649, 2), (700_001, 2)])
@pytest.mark.parametrize("wt,rt", [(None, np.int32), (None, np.int64), (np.int32, np.int32), (np.int64, np.int64)])
def test_levels_equal_the_oracle(n, f0, wt, rt):
    succ = gen.random_list(n, 7000 + n)
    w = None
    if wt is not None:
        info = np.iinfo(wt)
        w = gen.rng(n).integers(info.min, info.max, size=n, dtype=wt, endpoint=True)
    got = lr.rank(dev(succ), None if w is None else dev(w), tuning=lr.Tuning(f0_inv=f0, contract=lr.CONTRACT_OFF),
                  rank_dtype=torch.int32 if rt == np.int32 else torch.int64)
    np.testing.assert_array_equal(got.cpu().numpy(), oracle.rank(succ, w, rt))


@pytest.mark.parametrize("mean_short", [1, 2, 5])
def test_last_level_of_many_lists(mean_short):
    # most elements are heads: the levels stop shrinking and the base case
    # takes more elements than the grid holds at once
    succ, _ = gen.forest((1 << 21) + 3, 7100 + mean_short, n_long=3, long_len=1 << 16, mean_short=mean_short)
    w = gen.weights_i64((1 << 21) + 3, 7101)
    np.testing.assert_array_equal(lr.rank(dev(succ)).cpu().numpy(), oracle.rank(succ))
    r, t, p = lr.rank_outputs(dev(succ), dev(w), term=True, prefix=True)
    want_r, want_t, want_p = oracle.rank_ext(succ, w, np.int64)
    np.testing.assert_array_equal(r.cpu().numpy(), want_r)
    np.testing.assert_array_equal(t.cpu().numpy().view(np.uint32), want_t)
    np.testing.assert_array_equal(p.cpu().numpy(), want_p)


@pytest.mark.parametrize("length", [2, 3, 4, 7, 64, 1023, 4096])
@pytest.mark.parametrize("n", [200, 5000, 300_001])
def test_cycles_beside_a_list(n, length):
    if length >= n:
        pytest.skip("longer than the list")
    lst = gen.random_list(n, 7200)
    cyc = n + np.roll(np.arange(length), -1)
    succ = np.concatenate([lst, cyc]).astype(np.uint32)
    assert oracle.rank_status(succ)[0] == oracle.CYCLE
    for f0 in (2, 8):
        assert status_of(succ, tuning=lr.Tuning(f0_inv=f0)) == "LR_ERR_CYCLE"
    assert status_of(lst) == "LR_OK"


@pytest.mark.parametrize("seed", range(6))
def test_two_lists_that_merge(seed):
    # the second list joins the first in its middle, at a ruler half of the
    # time: no cycle, and the chases alone see nothing when it is one
    n = 100_003
    a, b = gen.random_list(n, 7300 + seed), gen.random_list(n, 7400 + seed)
    succ = np.concatenate([a, b + n]).astype(np.uint32)
    tail = n + int(np.flatnonzero(b == np.arange(n))[0])
    succ[tail] = int(gen.rng(seed).integers(0, n))
    assert oracle.rank_status(succ)[0] == oracle.NOT_A_LIST
    for f0 in (2, 8):
        assert status_of(succ, tuning=lr.Tuning(f0_inv=f0)) == "LR_ERR_NOT_A_LIST"
        assert status_of(succ, tuning=lr.Tuning(f0_inv=f0), validate=True) == "LR_ERR_NOT_A_LIST"
