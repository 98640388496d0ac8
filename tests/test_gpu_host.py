"""lr_rank_host on pinned buffers, which the kernels read and write in place,
and on pageable and misaligned ones, which are copied: every form of level 0,
contracted lists, forests, weights too wide for 8-byte records, errors."""
import ctypes

import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_09318_gb300 as lr  # noqa: E402


def pinned(a, shift=0):
    a = a.view(np.int32) if a.dtype == np.uint32 else a
    t = torch.from_numpy(np.concatenate([a[:1]] * shift + [a])).pin_memory()
    return t[shift:]


def succ_of(kind, n, seed):
    if kind == "forest":
        return gen.forest(n, seed, n_long=2, long_len=n // 4, mean_short=5)[0].astype(np.uint32)
    return gen.list_of_order_kind(kind, n, seed)


@pytest.mark.parametrize("n", [1, 777, 4096, 4097, 70_001, (1 << 19) + 3, 1_500_001, (1 << 22) + 4099])
@pytest.mark.parametrize("kind", ["random", "locality", "forest"])
@pytest.mark.parametrize("wt", [None, "i32", "i64 wide"])
def test_pinned_buffers(n, kind, wt):
    if kind == "forest" and n < 1000:
        pytest.skip("too short for the generator")
    succ = succ_of(kind, n, 9990)
    w = None
    if wt == "i32":
        w = gen.weights_i32(n, 9991)
    elif wt:
        w = gen.weights_i64(n, 9992)
        w[n // 2] = 1 << 50
    rt = np.int32 if wt is None else np.int64
    want = oracle.rank(succ, w, rt)
    for shift in (0, 1):
        for validate in (False, True):
            out = torch.full((n + 1,), -7, dtype=torch.int32 if wt is None else torch.int64).pin_memory()[shift:n + shift]
            got = lr.rank_host(pinned(succ, shift), None if w is None else pinned(w, shift), out=out, validate=validate)
            np.testing.assert_array_equal(np.asarray(got), want)
    got = lr.rank_host(torch.from_numpy(succ.view(np.int32)), None if w is None else pinned(w))   # pageable successors
    np.testing.assert_array_equal(np.asarray(got), want)


@pytest.mark.parametrize("n", [1000, 100_000, 1_000_000])
def test_ranks_over_the_successors(n):
    succ = gen.random_list(n, 9993)
    s = pinned(succ)
    lr.rank_host(s, out=s)
    np.testing.assert_array_equal(s.numpy(), oracle.rank(succ))


def test_bytes_off_their_alignment():
    # a copy takes any address
    n = 600_001
    succ = gen.random_list(n, 9994)
    raw = torch.empty(4 * n + 16, dtype=torch.uint8).pin_memory()
    ctypes.memmove(raw.data_ptr() + 2, succ.ctypes.data, 4 * n)
    out = torch.empty(4 * n + 16, dtype=torch.uint8).pin_memory()
    code = lr.load().lr_rank_host(raw.data_ptr() + 2, None, n, out.data_ptr() + 6, None, None)
    assert code == 0
    got = np.empty(n, np.int32)
    ctypes.memmove(got.ctypes.data, out.data_ptr() + 6, 4 * n)
    np.testing.assert_array_equal(got, oracle.rank(succ))


@pytest.mark.parametrize("n", [1000, 100_000, 1_000_000])
def test_errors(n):
    succ = gen.random_list(n, 9995)
    bad = succ.copy()
    bad[n // 2] = n
    with pytest.raises(lr.LRError) as e:
        lr.rank_host(pinned(bad))
    assert e.value.name == "LR_ERR_OUT_OF_RANGE"
    np.testing.assert_array_equal(np.asarray(lr.rank_host(pinned(succ))), oracle.rank(succ))
