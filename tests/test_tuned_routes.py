"""What the autotuner measures and what its table changes: the route of a
default call at sizes that the base case ranks, whole, at level 0."""
import json

import numpy as np
import pytest

import gen
import oracle
import paper_2606_09318_gb300 as lr

torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def clean_table(monkeypatch):
    monkeypatch.delenv("LR_TUNING", raising=False)
    lr.autotune_clear()
    yield
    lr.autotune_clear()


def load(tmp_path, log2n, f0, cutoff):
    entry = {"log2n": log2n, "weighted": 0, "batch": 0, "f0_inv": f0, "f_inv": 8, "cutoff": cutoff, "chase_block": 256,
             "chase_ctas": 0, "algorithm": 0, "ms": 1}
    src = tmp_path / "tune.json"
    src.write_text(json.dumps({"format": "lr_autotune 1", "entries": [entry]}))
    lr.autotune_load(str(src))


@pytest.mark.parametrize("n", [20_000, 131_072, 300_001, 1 << 19])
def test_plans_without_a_gpu(tmp_path, n):
    base = lr.workspace_size(n, max_lists=1)
    # the default spacing, named or not, is the default call; another one is the ruling set
    assert lr.workspace_size(n, max_lists=1, tuning=lr.Tuning(f0_inv=4, f_inv=8, cutoff=12288, chase_block=256)) == base
    assert lr.workspace_size(n, max_lists=1, tuning=lr.Tuning(f0_inv=5)) > base
    # an entry does not take the base case away, whatever bound was saved with it
    for cutoff in (4096, 8192, 12288):
        load(tmp_path, n.bit_length() - 1, 8, cutoff)
        assert lr.workspace_size(n, max_lists=1) == base


@pytest.mark.gpu
def test_tuned_calls_take_the_default_route(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    n = 100_000
    succ = gen.random_list(n, 610)
    want = oracle.rank(succ)
    s = torch.from_numpy(succ.view(np.int32)).cuda()

    def levels(**kw):
        np.testing.assert_array_equal(lr.rank(s, **kw).cpu().numpy(), want)
        return lr.level_sizes()

    assert levels() == [n]
    t = lr.autotune(n)
    assert levels() == [n] and levels(tuning=t) == [n]
    load(tmp_path, 16, 4, 4096)
    assert levels() == [n]
    assert len(levels(tuning=lr.Tuning(f0_inv=5))) > 1


@pytest.mark.gpu
def test_an_entry_without_a_search_leaves_its_octave_alone():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    before = lr.workspace_size(1_000_000, max_lists=1)
    lr.autotune(1 << 19)                             # ranked by the base case: nothing to search
    assert len(lr.autotune_entries()) == 1
    assert lr.workspace_size(1_000_000, max_lists=1) == before
