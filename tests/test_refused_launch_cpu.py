"""Host logic of the whole-GPU iterations where the driver refuses a launch
(csrc/dpf_resident.h, compiled for the host with a launch that is told to fail)."""
import os
import subprocess

from paper_2603_28203_gb300.build import CSRC, INCLUDE, _cuda_home

SRC = """
#include <cstdio>
#include "dpf_resident.h"
using namespace dpf;
int main() {
  const int codes[] = {0, 720, 701, 801, 700, 719, 1};
  for (int e : codes) {
    GridShape g;
    g.ok = true;
    g.ctas = 7;
    int whole = 0, cleared = 0, streamed = 0, rc = 0;
    for (int span = 0; span < 2; ++span)
      rc = whole_or_streaming(g, [&] { ++whole; return e; }, [&] { ++cleared; }, [&] { ++streamed; return 0; });
    std::printf("%d %d %d %d %d %d\\n", e, rc, whole, cleared, streamed, (int)g.ok);
  }
}
"""


def test_a_refused_cooperative_launch_goes_on_streaming(tmp_path):
    """Refusals (720, 701, 801) run every interval with the streaming kernels
    and report success; success and other errors are passed on."""
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-I" + INCLUDE, "-I" + os.path.join(_cuda_home(), "include"),
                    str(tmp_path / "t.cpp"), "-o", exe, "-ldl"], check=True)
    rows = [tuple(int(v) for v in line.split()) for line in subprocess.check_output([exe], text=True).splitlines()]
    assert rows == [(0, 0, 2, 0, 0, 1), (720, 0, 1, 1, 2, 0), (701, 0, 1, 1, 2, 0), (801, 0, 1, 1, 2, 0),
                    (700, 700, 2, 0, 0, 1), (719, 719, 2, 0, 0, 1), (1, 1, 2, 0, 0, 1)]
