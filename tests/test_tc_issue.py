"""The issuing thread of the tensor-core kernel around the bounded wait for its constant operand (csrc/tc_issue.h), run on
the host with fakes: no MMA over an operand that has not landed, and no exit with its copy in flight."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2311_11348_gb300", "csrc")

# the block's life as in k_elem_tc: tiles until one fails, then the exit.  Arguments: the
# try on which the copy lands (0: never), ok at the start, tiles.  Prints waits mmas arrivals ok
HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "tc_issue.h"
int main(int, char** a) {
  const int lands = atoi(a[1]), tiles = atoi(a[3]);
  bool ok = atoi(a[2]) != 0, landed = false;
  int waits = 0, mmas = 0, arrivals = 0;
  auto wait = [&] { return ++waits == lands; };
  for (int t = 0; t < tiles && (ok || t == 0); ++t)
    ok = swedg::tc_issue(ok, landed, wait, [&] { ++mmas; }, [&] { ++arrivals; });
  swedg::tc_drain(landed, wait);
  printf("%d %d %d %d\n", waits, mmas, arrivals, (int)ok);
}
"""


def test_issue_and_drain(tmp_path):
    src, exe = tmp_path / "h.cpp", str(tmp_path / "h")
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)

    def run(*a):
        return tuple(int(x) for x in subprocess.run([exe, *map(str, a)], check=True, capture_output=True,
                                                    text=True).stdout.split())

    assert run(1, 1, 3) == (1, 3, 0, 1)  # lands at once: one wait for all tiles
    assert run(2, 1, 3) == (2, 0, 1, 0)  # the first wait runs out: no MMA, the barrier completed, the exit waits again
    assert run(0, 1, 3) == (2, 0, 1, 0)  # never lands: bounded all the same
    assert run(1, 0, 3) == (1, 0, 1, 0)  # an operand at a wrong address: no MMA
