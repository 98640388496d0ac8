"""Weighted level 0 in 8-byte records, against the oracle: weights at the edges
of what the records hold and just beyond (16-byte records then), segments long
enough to be cut, int32 ranks with any weights, and the same where the device
decides (a bound on the lists, no wait)."""
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


RANGES = {
    "signed": (-(1 << 19), (1 << 19) - 1), "unsigned": (0, (1 << 20) - 1),
    "too low": (-(1 << 19) - 1, 5), "too high": (-1, 1 << 19), "too high unsigned": (0, 1 << 20),
    "int32": (-(1 << 31), (1 << 31) - 1), "int64": (-(1 << 63), (1 << 63) - 1),
}


def weights(n, name, seed):
    lo, hi = RANGES[name]
    w = gen.rng(seed).integers(lo, hi, size=n, dtype=np.int64, endpoint=True)
    w[n // 3], w[n // 2] = lo, hi                     # both ends occur
    return w


@pytest.mark.parametrize("name", list(RANGES))
@pytest.mark.parametrize("n", [600_011, (1 << 22) + 5])
def test_weight_ranges(n, name):
    succ, w = gen.random_list(n, 9000 + n), weights(n, name, 9001)
    want = oracle.rank(succ, w, np.int64)
    s, d = dev(succ), dev(w)
    off = lr.Tuning(contract=lr.CONTRACT_OFF)
    for kw in ({}, {"max_lists": 1}, {"validate": True}):      # waits; does not (from 2^22 on); bitmap heads
        np.testing.assert_array_equal(lr.rank(s, d, tuning=off, **kw).cpu().numpy(), want)
    np.testing.assert_array_equal(lr.rank(s, d, tuning=off, rank_dtype=torch.int32).cpu().numpy(),
                                  oracle.rank(succ, w, np.int32))


@pytest.mark.parametrize("name", ["signed", "unsigned"])
@pytest.mark.parametrize("f0", [1 << 14, 1 << 17])
def test_long_segments_are_cut(name, f0):
    n = (1 << 20) + 3
    lo, hi = RANGES[name]
    for fill in (lo or hi, hi):                       # every weight at one end: the largest offsets
        succ, w = gen.random_list(n, 9100), np.full(n, fill, dtype=np.int64)
        got = lr.rank(dev(succ), dev(w), tuning=lr.Tuning(f0_inv=f0, contract=lr.CONTRACT_OFF))
        np.testing.assert_array_equal(got.cpu().numpy(), oracle.rank(succ, w, np.int64))
    ident = gen.identity_list(n)
    w = weights(n, name, 9101)
    got = lr.rank(dev(ident), dev(w), tuning=lr.Tuning(f0_inv=f0, contract=lr.CONTRACT_OFF), max_lists=1)
    np.testing.assert_array_equal(got.cpu().numpy(), oracle.rank(ident, w, np.int64))


@pytest.mark.parametrize("name", ["signed", "unsigned", "too high", "int64"])
@pytest.mark.parametrize("hi_exp", [16.0, 19.0])
def test_batches_and_forests(name, hi_exp):
    k = 60
    lens = np.floor(2.0 ** gen.rng(9200).uniform(0, hi_exp, size=k)).astype(np.int64)
    lens[[3, 59]] = 0
    lens[5] = 1 << 19
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    lists = [gen.random_list(int(m), 9201 + j) if m else np.zeros(0, np.uint32) for j, m in enumerate(lens)]
    succ = np.concatenate(lists).astype(np.uint32)
    w = weights(succ.shape[0], name, 9202)
    want = oracle.rank_batch(offsets, succ, w, np.int64)
    for kw in ({}, {"max_lists": k}, {"validate": True}):
        got = lr.rank_batch(dev(offsets), dev(succ), dev(w), **kw)
        np.testing.assert_array_equal(got.cpu().numpy(), want)
        parts = lr.rank_batch_ptrs([dev(a) for a in lists], [dev(w[a:b]) for a, b in zip(offsets, offsets[1:])], **kw)
        np.testing.assert_array_equal(np.concatenate([q.cpu().numpy() for q in parts]), want)
    forest, nl = gen.forest(1 << 20, 9203, n_long=2, long_len=1 << 17, mean_short=3)      # singletons among them
    fw = weights(1 << 20, name, 9204)
    want = oracle.rank(forest, fw, np.int64)
    for kw in ({}, {"max_lists": nl}, {"validate": True}):
        np.testing.assert_array_equal(lr.rank(dev(forest), dev(fw), **kw).cpu().numpy(), want)


def test_order_and_errors():
    # a batch beyond L2 (element order), then a bad list among its instances
    rng = gen.rng(9300)
    lens = rng.integers(1 << 18, 1 << 20, size=32)
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    succ = np.concatenate([gen.random_list(int(m), 9301 + j) for j, m in enumerate(lens)]).astype(np.uint32)
    n = succ.shape[0]
    assert n * 8 > 128 << 20
    for name in ("unsigned", "int64"):
        w = weights(n, name, 9302)
        want = oracle.rank_batch(offsets, succ, w, np.int64)
        for kw in ({}, {"max_lists": 32}):
            np.testing.assert_array_equal(lr.rank_batch(dev(offsets), dev(succ), dev(w), **kw).cpu().numpy(), want)
    bad = succ.copy()
    a, m = int(offsets[7]), int(lens[7])
    tail = a + int(np.flatnonzero(bad[a:a + m] == np.arange(m))[0])
    bad[tail] = bad[a + 11]
    for kw in ({}, {"max_lists": 32}):
        with pytest.raises(lr.LRError):
            lr.rank_batch(dev(offsets), dev(bad), dev(w), **kw)
