"""Workspace sizes rise with the number of elements (lr_workspace_size).

A workspace, or a pipeline, that is sized for n elements also serves every
shorter list.  The need itself falls where a rule on n takes fewer rulers, so
the sizes on both sides of every such rule are compared here, and a walk in
steps of a per cent.
"""
import itertools
import json

import numpy as np
import pytest

import gen
import oracle
import paper_2606_09318_gb300 as lr

JUMP = 393216                                    # rulers that the base case takes
SPACINGS = (4, 6, 8, 12, 16, 24, 32, 48, 64, 96)
STEPS = [3 << 18, 5 << 18, 5 << 19, 9 << 19, 1 << 23, 3 << 23, 5 << 23, 3 << 25, 1 << 27, 3 << 26, 1 << 29]
STEPS += [1 << b for b in range(10, 31)] + [f * (4 * JUMP + 1) for f in SPACINGS] + [0x7FFFFF01]
STEPS += [na << s << 14 for s in (3, 5, 8) for na in (136, 137, 186, 204, 227, 228)]     # the log form's buckets


def sizes():
    s = {int(1000 * 1.01 ** i) for i in range(1400)}
    s.update(b + d for b in STEPS for d in (-1, 0, 1))
    return sorted(n for n in s if n <= 1 << 31)


def check(**kw):
    before, at = 0, 0
    for n in sizes():
        need = lr.workspace_size(n, **kw)
        assert need >= before, (at, before, n, need)
        before, at = need, n


@pytest.mark.parametrize("weighted,rank64", [(False, False), (False, True), (True, False), (True, True)])
def test_size_rises_with_n(weighted, rank64, monkeypatch):
    monkeypatch.delenv("LR_TUNING", raising=False)
    for k, extra, most in itertools.product((0, 50), ({}, {"term": True}, {"prefix": True}), (1, 600_000)):
        check(k=k, weighted=weighted, rank64=rank64, max_lists=most, **extra)


def test_size_rises_with_n_tuned(tmp_path, monkeypatch):
    monkeypatch.delenv("LR_TUNING", raising=False)
    for tuning in (lr.Tuning(f0_inv=24), lr.Tuning(f_inv=16), lr.Tuning(spawn=1), lr.Tuning(cutoff=4096)):
        check(max_lists=1, tuning=tuning)
    entries = [{"log2n": b, "weighted": 0, "batch": 0, "f0_inv": f0, "f_inv": f, "cutoff": 12288, "chase_block": 256,
                "chase_ctas": 0, "algorithm": 0, "ms": 1} for b, f0, f in ((20, 4, 4), (21, 128, 16), (24, 8, 4), (27, 128, 16))]
    src = tmp_path / "tune.json"
    src.write_text(json.dumps({"format": "lr_autotune 1", "entries": entries}))
    lr.autotune_clear()
    try:
        lr.autotune_load(str(src))
        check(max_lists=1)
    finally:
        lr.autotune_clear()


@pytest.mark.gpu
@pytest.mark.parametrize("max_n,n", [(19_000_000, 18_874_379), (9_000_000, 8_388_607)])
def test_sized_for_more_serves_less(max_n, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    succ = gen.random_list(n, 95)
    want = oracle.rank(succ)
    host = torch.from_numpy(succ.view(np.int32)).pin_memory()
    pipe = lr.Pipeline(max_n, max_lists=1)
    out = pipe.submit(host)
    pipe.wait()
    np.testing.assert_array_equal(out.numpy(), want)
    pipe.close()
    ws = torch.empty(lr.workspace_size(max_n, max_lists=1), dtype=torch.uint8, device="cuda")
    got = lr.rank(host.cuda(), max_lists=1, workspace=ws)
    np.testing.assert_array_equal(got.cpu().numpy(), want)
