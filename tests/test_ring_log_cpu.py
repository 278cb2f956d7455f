"""The X step's record of copies in flight (RingLog), driven on the host.

Stages refilled by neighbouring warps may be issued in either order, and after
an abort one of two neighbouring stages may not be issued at all.  Whatever the
order, an abort must wait for the last copies of every slot, in the phase that
those copies complete, and for nothing that was not issued."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1502_06894_gb300", "csrc")

PROGRAM = r"""
#include "corr_internal.cuh"
#include <cstdio>

// Stages [0, n) in a ring of `stages`, the first ring of them in order, then
// pairs (q, q + 1) in either order; the run ends after `ops` issues, or with
// stage `hole` left out although its successor was issued.
template <typename Check>
void run(int stages, int n, int swapped, int ops, int hole, Check check) {
  corr::RingLog<8> log;
  log.clear();
  int last[8];  // the definition: per slot the last stage issued
  for (int i = 0; i < 8; ++i) last[i] = -1;
  int done = 0;
  auto issue = [&](int q) {
    if (q >= n || q == hole || done >= ops) return;
    ++done;
    log.note(q % stages, q);
    last[q % stages] = q;
  };
  for (int q = 0; q < stages; ++q) issue(q);
  for (int q = stages; q < n; q += 2) {
    issue(swapped ? q + 1 : q);
    issue(swapped ? q : q + 1);
  }
  check(log, last);
}

int main() {
  int bad = 0, runs = 0;
  for (int stages = 2; stages <= 8; ++stages)
    for (int n = 1; n <= 4 * stages; ++n)
      for (int swapped = 0; swapped < 2; ++swapped)
        for (int ops = 0; ops <= n; ++ops)
          for (int hole = -1; hole < n; ++hole)
            run(stages, n, swapped, ops, hole, [&](const corr::RingLog<8>& log, const int* last) {
              ++runs;
              int seen[8] = {};
              log.for_each(stages, [&](int slot, unsigned parity) {
                seen[slot] = 1;
                // the barrier of a slot completes phase q / stages with stage q
                if (last[slot] < 0 || parity != (unsigned)((last[slot] / stages) & 1)) ++bad;
              });
              for (int i = 0; i < 8; ++i)
                if (seen[i] != (last[i] >= 0)) ++bad;
            });
  printf("%d %d\n", runs, bad);
  return bad != 0;
}
"""


def test_every_copy_in_flight_is_waited_for(tmp_path):
    from paper_1502_06894_gb300 import _build
    src = tmp_path / "t.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-I", CSRC, "-o", exe, str(src)], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    assert int(out.stdout.split()[0]) > 10000


def test_the_ring_keeps_that_record():
    """Both kernels note each issue in it, nothing is issued after an abort was
    seen, and the drain waits for what it holds."""
    text = open(os.path.join(CSRC, "k_xstage.cu")).read()
    assert text.count("s_log.note(slot, q);") == 2 and "issued = " not in text
    drain = text[text.index("void drain("):]
    assert "log->for_each(stages" in drain[:drain.index("atomicExch")]
    reclaim = text[text.index("int reclaim("):]
    assert "stop = *abort_flag" in reclaim[:reclaim.index("ring_wait(")] and "&& !stop)" in reclaim[:reclaim.index("return old;")]
