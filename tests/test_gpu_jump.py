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


# ---- level 0 ranked by the base case itself (no ruling set), and its limits
@pytest.mark.parametrize("n", [12289, 40_001, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("kind", ["random", "locality", "identity", "forest"])
def test_level0_equals_the_oracle(n, kind):
    if kind == "forest":
        succ, nl = gen.forest(n, 7500 + n, n_long=2, long_len=n // 8, mean_short=9)
    else:
        succ, nl = gen.list_of_order_kind(kind, n, 7500 + n), 1
    w = gen.weights_i32(n, 7501)
    want, want_t, want_p = oracle.rank_ext(succ, w, np.int64)
    np.testing.assert_array_equal(lr.rank(dev(succ), validate=True).cpu().numpy(), oracle.rank(succ))
    np.testing.assert_array_equal(lr.rank(dev(succ), dev(w), max_lists=nl).cpu().numpy(), want)
    for weight in (None, dev(w)):                     # 8- and 16-byte records, the latter with terminals
        r, t, p = lr.rank_outputs(dev(succ), weight, term=True, prefix=weight is not None)
        np.testing.assert_array_equal(t.cpu().numpy().view(np.uint32), want_t)
    np.testing.assert_array_equal(r.cpu().numpy(), want)
    np.testing.assert_array_equal(p.cpu().numpy(), want_p)


@pytest.mark.parametrize("total_exp", [8.0, 13.0, 15.0])
@pytest.mark.parametrize("wt", [None, "i64"])
def test_batches_at_level0(total_exp, wt):
    k = 24
    lens = np.floor(2.0 ** gen.rng(int(total_exp)).uniform(0, total_exp, size=k)).astype(np.int64)
    lens[[0, 7, 23]] = 0
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    lists = [gen.random_list(int(m), 7600 + j) if m else np.zeros(0, np.uint32) for j, m in enumerate(lens)]
    succ = np.concatenate(lists).astype(np.uint32)
    w = gen.weights_i64(succ.shape[0], 7601) if wt else None
    rt = np.int64 if wt else np.int32
    want = oracle.rank_batch(offsets, succ, w, rt)
    for ml in (0, k):
        got = lr.rank_batch(dev(offsets), dev(succ), None if w is None else dev(w), max_lists=ml)
        np.testing.assert_array_equal(got.cpu().numpy(), want)
        parts = lr.rank_batch_ptrs([dev(a) for a in lists],
                                   None if w is None else [dev(w[a:b]) for a, b in zip(offsets, offsets[1:])],
                                   max_lists=ml)
        np.testing.assert_array_equal(np.concatenate([q.cpu().numpy() for q in parts]), want)


@pytest.mark.parametrize("n", [4097, 12288, 12289, 200_003])
def test_promised_lists_and_capture(n):
    succ, nl = gen.forest(n, 7700, n_long=1, long_len=n // 4, mean_short=16)
    want = oracle.rank(succ)
    np.testing.assert_array_equal(lr.rank(dev(succ), max_lists=nl).cpu().numpy(), want)
    if n <= 12288:                                    # the smallest sizes never counted lists
        np.testing.assert_array_equal(lr.rank(dev(succ), max_lists=1).cpu().numpy(), want)
    else:
        assert status_of(succ, max_lists=nl // 4) == "LR_ERR_CAPACITY"
    s, out, side = dev(succ), torch.empty(n, dtype=torch.int32, device="cuda"), torch.cuda.Stream()
    lr.rank(s, out=out, max_lists=nl, stream=side)
    out.zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        lr.rank(s, out=out, max_lists=nl, sync=False)
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), want)


# ---- the one-launch path of short lists (k_small) and the size above it
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 1023, 1024, 1025, 4095, 4096, 4097])
@pytest.mark.parametrize("wt,rt", [(None, np.int32), (None, np.int64), (np.int32, np.int64), (np.int64, np.int32)])
def test_short_lists(n, wt, rt):
    trt = torch.int32 if rt == np.int32 else torch.int64
    for succ in (gen.random_list(n, 7800 + n), gen.identity_list(n), np.arange(n, dtype=np.uint32)):
        w = None
        if wt is not None:
            info = np.iinfo(wt)
            w = gen.rng(n).integers(info.min, info.max, size=n, dtype=wt, endpoint=True)
        want = oracle.rank(succ, w, rt)
        dw = None if w is None else dev(w)
        np.testing.assert_array_equal(lr.rank(dev(succ), dw, rank_dtype=trt, validate=True).cpu().numpy(), want)
        assert lr.level_sizes() == [n]
        np.testing.assert_array_equal(lr.rank(dev(succ), dw, rank_dtype=trt, sync=False).cpu().numpy(), want)
        assert lr.device_status() == 0
    if n > 1:
        cyc = np.roll(np.arange(n, dtype=np.uint32), -1)          # one ring
        assert status_of(cyc) == "LR_ERR_CYCLE"
        out = gen.random_list(n, 7801)
        out[0] = n
        assert status_of(out) == "LR_ERR_OUT_OF_RANGE"
        star = np.zeros(n, dtype=np.uint32)                       # everybody before element 0
        assert status_of(star, validate=True) == ("LR_ERR_NOT_A_LIST" if n > 2 else "LR_OK")
        lr.rank(dev(cyc), sync=False)
        assert lr.status_string(lr.device_status()) == "LR_ERR_CYCLE"


def test_calls_leave_their_words_at_zero():
    # the error word, the list count and the predecessor marks of the two-launch
    # path are cleared by the call that used them: whatever came before on the
    # stream, the next call starts clean, in a captured graph as well
    st = torch.cuda.Stream()
    good = {n: gen.random_list(n, 9900 + n) for n in (5000, 20_000, 300_007, 1 << 19)}
    ring = np.roll(np.arange(20_000, dtype=np.uint32), -1)
    merged = good[300_007].copy()
    merged[int(np.flatnonzero(merged == np.arange(300_007))[0])] = merged[5]
    forest, nl = gen.forest(100_000, 9901, n_long=1, long_len=10, mean_short=5)
    want = {n: oracle.rank(s) for n, s in good.items()}
    # torch's streams come from a pool: graph and stream are the library's st
    s19, out = dev(good[1 << 19]), torch.empty(1 << 19, dtype=torch.int32, device="cuda")
    lr.rank(s19, out=out, max_lists=1, stream=st)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        lr.rank(s19, out=out, max_lists=1, sync=False)

    def status(succ, **kw):
        lr.rank(dev(succ), sync=False, stream=st, **kw)
        return lr.status_string(lr.device_status(st))

    bad = [(ring, {}, "LR_ERR_CYCLE"), (merged, {}, "LR_ERR_NOT_A_LIST"),
           (forest, {"max_lists": nl // 8}, "LR_ERR_CAPACITY")]
    for _ in range(2):
        for succ, kw, name in bad:
            torch.cuda.synchronize()
            assert status(succ, **kw) == name
            for n in good:
                got = lr.rank(dev(good[n]), validate=n == 5000, max_lists=1, stream=st)
                np.testing.assert_array_equal(got.cpu().numpy(), want[n])
            assert status(forest, max_lists=nl) == "LR_OK"
            out.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(st):
                g.replay()
            assert lr.device_status(st) == 0
            np.testing.assert_array_equal(out.cpu().numpy(), want[1 << 19])


@pytest.mark.parametrize("n", [(1 << 19) + 1, (1 << 22) + 9])
@pytest.mark.parametrize("wt", [None, "i32"])
def test_validation_by_counts(n, wt):
    # two predecessors are told from one by as many heads as terminals
    w = None if wt is None else dev(gen.weights_i32(n, 9950))
    host_w = None if wt is None else gen.weights_i32(n, 9950)
    rt = np.int32 if wt is None else np.int64
    one = gen.random_list(n, 9951)
    forest, _ = gen.forest(n, 9952, n_long=2, long_len=n // 8, mean_short=7)
    for succ in (one, forest):
        np.testing.assert_array_equal(lr.rank(dev(succ), w, validate=True).cpu().numpy(), oracle.rank(succ, host_w, rt))
        bad = succ.copy()
        inner = np.flatnonzero(bad != np.arange(n))
        a, b = int(inner[5]), int(inner[len(inner) // 2])
        bad[a] = bad[b]                                   # b's successor has two predecessors
        assert oracle.rank_status(bad)[0] != oracle.OK
        with pytest.raises(lr.LRError) as e:
            lr.rank(dev(bad), w, validate=True)
        assert e.value.name == "LR_ERR_NOT_A_LIST"
        lr.rank(dev(bad), w, validate=True, sync=False)
        assert lr.status_string(lr.device_status()) == "LR_ERR_NOT_A_LIST"
        bad[a] = n + 5
        with pytest.raises(lr.LRError) as e:
            lr.rank(dev(bad), w, validate=True)
        assert e.value.name == "LR_ERR_OUT_OF_RANGE"
    r, t, p = lr.rank_outputs(dev(one), w, term=True, prefix=True, validate=True)
    want_r, want_t, want_p = oracle.rank_ext(one, host_w, rt)
    np.testing.assert_array_equal(r.cpu().numpy(), want_r)
    np.testing.assert_array_equal(t.cpu().numpy().view(np.uint32), want_t)
    np.testing.assert_array_equal(p.cpu().numpy(), want_p)


def test_calls_back_to_back_on_two_streams():
    # a kernel may start before the one ahead of it has ended: many calls of
    # every kind, none waited for, each with its own inputs and outputs
    kinds = []
    for j, n in enumerate((20_000, 600_001, 1 << 20, 3_000_000)):
        succ = gen.random_list(n, 9900 + j) if j != 1 else gen.forest(n, 9900 + j, n_long=3, long_len=n // 8,
                                                                       mean_short=6)[0].astype(np.uint32)
        w = gen.weights_i32(n, 9910 + j) if j % 2 else None
        lists = int((succ == np.arange(n)).sum())
        want = oracle.rank(succ, w, np.int64 if j % 2 else np.int32)
        kinds.append((dev(succ), None if w is None else dev(w), lists, want))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    outs = []
    for rnd in range(12):
        for j, (succ, w, lists, want) in enumerate(kinds):
            st = streams[(rnd + j) % 2]
            with torch.cuda.stream(st):
                mine = succ.clone()
                out = lr.rank(mine, w, max_lists=lists if rnd % 3 else 0, sync=False, validate=rnd % 4 == 1)
                mine.fill_(0)                       # the call has read them by then
            outs.append((out, want))
    torch.cuda.synchronize()
    for out, want in outs:
        np.testing.assert_array_equal(out.cpu().numpy(), want)
