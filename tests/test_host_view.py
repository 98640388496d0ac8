"""Host buffers that kernels read and write in place: all of the buffer has to
be pinned, not only its ends.  The rule (csrc/lr_hostview.h) on the host,
against a map of pinned pieces; and registered memory on the GPU."""
import ctypes
import mmap
import os
import shutil
import subprocess

import numpy as np
import pytest

import gen
import oracle
import paper_2606_09318_gb300 as lr

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_09318_gb300", "csrc")
PROGRAM = """
#include <cstdint>
#include <cstdio>
#include <vector>
#include "lr_hostview.h"
struct Piece { size_t from, to; intptr_t shift; };          // pinned bytes; device address less host address
static char memory[4096];
static bool check(const std::vector<Piece> &pieces, size_t from, size_t to, bool want, intptr_t shift) {
  void *got = lr::pinned_view(memory + from, to - from, [&](const void *q, lr::PinnedPiece &p) {
    const size_t at = static_cast<const char *>(q) - memory;
    for (const Piece &x : pieces)
      if (at >= x.from && at < x.to) {
        p.device = reinterpret_cast<void *>(reinterpret_cast<intptr_t>(q) + x.shift);
        p.left = x.to - at;
        return true;
      }
    return false;
  });
  if (!want) return got == nullptr;
  return got == reinterpret_cast<void *>(reinterpret_cast<intptr_t>(memory + from) + shift);
}
int main() {
  const bool ok[] = {
      check({{0, 4096, 0}}, 0, 4096, true, 0),
      check({{64, 1064, 1 << 20}}, 64, 1064, true, 1 << 20),            // all of it, elsewhere on the device
      check({{64, 1064, 0}}, 100, 101, true, 0),
      check({{64, 1064, 0}}, 64, 1065, false, 0),                       // a byte beyond
      check({{64, 1064, 0}}, 63, 1064, false, 0),                       // a byte before
      check({{0, 1024, 0}, {2048, 4096, 0}}, 0, 4096, false, 0),        // both ends, not the middle
      check({{0, 1024, 0}, {1025, 4096, 0}}, 1000, 2000, false, 0),
      check({{0, 1024, 8}, {1024, 4096, 8}}, 1000, 2000, true, 8),      // one after the other
      check({{0, 1024, 8}, {1024, 4096, 16}}, 1000, 2000, false, 0),    // but not on the device
      check({{0, 16, 0}, {16, 32, 0}, {40, 64, 0}}, 0, 64, false, 0),
      check({}, 0, 8, false, 0)};
  int bad = 0, i = 0;
  for (bool b : ok) { if (!b) { printf("case %d\\n", i); ++bad; } ++i; }
  if (!bad) printf("ok\\n");
  return bad;
}
"""


def test_every_piece_is_asked_for(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    (tmp_path / "view.cc").write_text(PROGRAM)
    exe = str(tmp_path / "view")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "view.cc"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("n", [70_001, 700_001])
def test_registered_memory(n):
    """One registration, and three that follow each other: pinned throughout."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    succ = gen.random_list(n, 9996)
    want = oracle.rank(succ)
    torch.zeros(1).cuda()
    rt = torch.cuda.cudart()
    size = -(-(4 * n + 4096) // mmap.PAGESIZE) * mmap.PAGESIZE
    for cuts in ([0, size], [0, mmap.PAGESIZE, 2 * mmap.PAGESIZE, size]):
        buf = mmap.mmap(-1, size)
        base = np.frombuffer(buf, dtype=np.uint8).ctypes.data
        for a, b in zip(cuts, cuts[1:]):
            assert int(rt.cudaHostRegister(base + a, b - a, 0)) == 0
        ctypes.memmove(base + 100, succ.ctypes.data, 4 * n)
        out = torch.empty(n, dtype=torch.int32).pin_memory()
        assert lr.load().lr_rank_host(base + 100, None, n, out.data_ptr(), None, None) == 0
        np.testing.assert_array_equal(out.numpy(), want)
        assert lr.load().lr_rank_host(base + 100, None, n, base + 100, None, None) == 0      # over the successors
        got = np.empty(n, np.int32)
        ctypes.memmove(got.ctypes.data, base + 100, 4 * n)
        np.testing.assert_array_equal(got, want)
        for a in cuts[:-1]:
            assert int(rt.cudaHostUnregister(base + a)) == 0
