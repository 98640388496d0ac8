"""The words that a base-case call shares between its two launches, when a
call fails between them and when a capture is thrown away (GPU; the debug
build, in a process of its own: see _own_words_cases.py)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("n", [6000, 100_003])        # without and with marks of predecessors
@pytest.mark.parametrize("later", ["call", "replay"])
def test_after_a_call_that_failed_on_the_way(n, later):
    from paper_2606_09318_gb300 import build
    build.build(debug=True)
    env = dict(os.environ, LR_DEBUG_LIB="1")
    env.pop("LR_TUNING", None)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "_own_words_cases.py"), str(n), later], env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
