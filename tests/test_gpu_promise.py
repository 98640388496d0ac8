"""A broken promise of max_lists, at sizes that the base case ranks whole: it
is noticed exactly where the ruling set, which the level-0 form forces here,
runs out of room for the heads."""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_09318_gb300 as lr  # noqa: E402

RULING_SET = lr.Tuning(chase0=lr.CHASE0_EXCHANGE)


def status_of(s, **kw):
    try:
        return "LR_OK", lr.rank(s, **kw).cpu().numpy()
    except lr.LRError as e:
        return e.name, None


@pytest.mark.parametrize("n", [12289, 100_003, 1 << 19])
@pytest.mark.parametrize("kind", ["lists of one", "a long list and lists of one", "forest"])
def test_same_as_the_ruling_set(n, kind):
    if kind == "lists of one":
        succ = np.arange(n, dtype=np.uint32)
    elif kind == "forest":
        succ = gen.forest(n, 650, n_long=2, long_len=n // 8, mean_short=3)[0].astype(np.uint32)
    else:
        succ = np.arange(n, dtype=np.uint32)
        succ[: n // 2] = gen.random_list(n // 2, 651)
    want = oracle.rank(succ)
    s = torch.from_numpy(succ.view(np.int32)).cuda()
    lists = int((succ == np.arange(n)).sum())
    seen = set()
    for most in sorted({1, 3, lists // 8, lists // 4 - 1, lists // 4 + 1, lists // 2, lists - 1, lists, n} - {0}):
        got, ranks = status_of(s, max_lists=most)
        assert got == status_of(s, max_lists=most, tuning=RULING_SET)[0], most
        if got == "LR_OK":
            np.testing.assert_array_equal(ranks, want)
        if most >= lists:
            assert got == "LR_OK"
        seen.add(got)
    assert seen == {"LR_OK", "LR_ERR_CAPACITY"}
