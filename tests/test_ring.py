"""The producer of a shared-memory ring (csrc/ring.cuh), compiled for the host and
driven against barriers whose waits give up."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2409_01949_gb300", "csrc")

MODEL = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "ring.cuh"
struct Io {
  int stages, give_up;              // the wait_empty call that gives up (-1: none)
  int waits = 0, issued = 0;
  std::vector<int> landed;          // copies waited for
  std::vector<int> at;              // per stage: the last copy issued into it
  bool bad = false;
  bool wait_empty(int st, int ph) {
    const int b = waits++;
    bad |= st != b % stages || ph != (((b / stages) & 1) ^ 1);
    return b != give_up;
  }
  void issue(int b, int st) {
    bad |= b != issued || (give_up >= 0 && waits > give_up);
    ++issued;
    at[st] = b;
  }
  bool wait_full(int st, int ph) {
    bad |= at[st] < 0 || ph != ((at[st] / stages) & 1);
    landed.push_back(at[st]);
    return true;
  }
};
int main(int argc, char** argv) {
  for (int stages : {1, 3, 8})
    for (int n : {0, 1, 2, 7, 8, 9, 40})
      for (int give_up = -1; give_up < n; ++give_up) {
        Io io;
        io.stages = stages;
        io.give_up = give_up;
        io.at.assign(stages, -1);
        const bool ok = ring_produce(n, stages, io);
        const int want = give_up < 0 ? n : give_up;
        // every copy that may still be in flight is waited for
        std::vector<int> last;
        for (int b = want > stages ? want - stages : 0; b < want; ++b) last.push_back(b);
        if (io.bad || io.issued != want || ok != (give_up < 0) || io.landed != last) {
          printf("stages %d n %d give_up %d\n", stages, n, give_up);
          return 1;
        }
      }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_no_copy_after_a_wait_that_gave_up_and_none_left_in_flight(tmp_path):
    src = tmp_path / "r.cpp"
    src.write_text(MODEL)
    exe = str(tmp_path / "r")
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-I", CSRC, "-o", exe, str(src)], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
