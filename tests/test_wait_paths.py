"""What a kernel has in flight when a bounded wait gives up: bulk copies must have landed before
the CTA ends, and MMAs and tensor-memory reads before tensor memory is released.  Those last
waits run with the abort flag already set, so they must not be cut short by it.

The drain helpers are compiled for the host and run over a model of a ring; the kernels' use of
them is read from their source (a timeout is not provoked on a GPU)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1508_02897_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "hd_tc.cuh"
using namespace hd;
// mbarriers of a ring: stage s has completed `done[s]` laps; its copy in flight, if any, lands after
// `delay` more polls of that stage.  A parity wait passes when the lap in progress has the other parity.
int main() {
  int bad = 0;
  for (int ns : {1, 2, 6, 16})
    for (long issued : {0L, 1L, 2L, 5L, 6L, 7L, 16L, 95L, 96L, 97L})
      for (int delay : {0, 1, 255, 256, 1000, 70000}) {
        std::vector<long> laps(ns, 0), done(ns, 0);
        std::vector<int> left(ns, delay);
        for (long k = 0; k < issued; ++k) laps[k % ns]++;
        for (int s = 0; s < ns; ++s) done[s] = laps[s] ? laps[s] - 1 : 0;   // the last lap of every used stage is in flight
        long polls = 0;
        tc::drain_ring(issued, ns, [&](int s, uint32_t parity) {
          ++polls;
          if (done[s] < laps[s] && left[s]-- <= 0) done[s]++;
          return (uint32_t)(done[s] & 1) != parity;
        });
        for (int s = 0; s < ns; ++s) bad += done[s] != laps[s];
        if (issued == 0) bad += polls != 0;
      }
  long polls = 0;   // a copy that never lands: the wait ends all the same
  bad += tc::drain([&]() { ++polls; return false; });
  bad += polls != (long)tc::kWaitLimit;
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


def _nvcc():
    return os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


@pytest.mark.skipif(not os.path.exists(_nvcc()), reason="needs nvcc")
def test_drains_outlast_the_copies_and_end(tmp_path):
    src = tmp_path / "drain.cu"
    src.write_text(HARNESS)
    exe = str(tmp_path / "drain")
    subprocess.run([_nvcc(), "-std=c++17", "-O1", "--extended-lambda", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


@pytest.mark.parametrize("name", ["hd_subst.cu", "hd_subst_sym.cu", "hd_subst_tc.cu", "hd_subst_x3.cu", "hd_gs.cu"])
def test_producers_drain_their_ring(name):
    """Every producer that leaves on a failed wait drains its copies without the abort flag."""
    s = _source(name)
    assert len(re.findall(r"tc::ring_drain\(", s)) == 1
    assert not re.search(r"wait\(&?[\w.]*\w+\[\w+ % \w+\]", s)   # no last round of waits that the flag ends


@pytest.mark.parametrize("name", ["hd_subst_tc.cu", "hd_subst_x3.cu"])
def test_tensor_memory_is_released_after_its_last_use(name):
    """Before the release: the MMAs issued so far (a commit of their own) and the epilogue's
    arrival, which it makes on a timeout too; neither wait looks at the abort flag."""
    s = _source(name)
    tail = s[s.index("mma_commit(fin)"):s.index("tcgen05.dealloc")]
    assert "tc::bar_drain(fin, 0);" in tail and "tc::bar_drain(edone, 0);" in tail and "abort_flag" not in tail
    assert len(re.findall(r"arrive\(edone\)", s)) == 1


def test_factorisation_releases_tensor_memory_after_its_last_mma():
    """After a timeout the last commit goes to a barrier that no other wait uses: the parity of a
    panel's barrier that never completed would pass at once."""
    s = _source("hd_factor_tc.cu")
    tail = s[s.index("release tensor memory"):s.index("tcgen05.dealloc")]
    bar = re.search(r"tc::mma_commit\((\w+)\)", tail).group(1)
    assert f"tc::bar_drain({bar}, 0)" in tail
    assert len(re.findall(rf"tc::mma_commit\({bar}\)", s)) == 1 and len(re.findall(rf"bar_init\({bar}, 1\)", s)) == 1
    assert not re.search(rf"(wait|spin)\({bar}\b", s)


def test_cluster_exchange_stops_after_a_timeout():
    """The CTAs of a cluster stay within two steps of each other only while every wait succeeds: a
    thread that gave up neither sends sums nor arms the barrier for more, and its CTA outlasts the
    sums that are still on their way to it."""
    s = _source("hd_subst_sym.cu")
    body = s[s.index("k_subst_sym("):s.index("static int sm_count()")]
    assert "if (K > 1) vec = false;" in body[body.index("auto fail"):]
    work = body[body.rindex("if (vec) {"):]   # the vector work of a step, which ends with the thread's first failed wait
    for op in ("cluster_send(", "mbarrier.arrive.expect_tx"):
        assert body.count(op) == work.count(op) > 0
    assert "if (*abort_flag) settle();" in body[body.rindex("cluster_sync_all();"):]
