"""A batch's runs of chunks (rad_impl.h: chunk_run), compiled from the library's own header with the host compiler: an
item of several chunks never holds more than 1024 particles, however large the other jobs of the launch are, and a chunk
is never split."""
import os
import subprocess

import pytest

from test_tail_plan_cpu import CSRC, ROOT, _cuda_include

SRC = """
#include <cstdio>
#include "rad_impl.h"
int main() {
  long long per_item; int ck;
  while (std::scanf("%lld %d", &per_item, &ck) == 2) std::printf("%d\\n", radimpl::chunk_run(per_item, ck));
}
"""


def test_runs_are_short(tmp_path):
    import shutil
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("needs a host C++ compiler and the CUDA runtime headers")
    (tmp_path / "run.cpp").write_text(SRC)
    exe = str(tmp_path / "run")
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I", inc,
                    str(tmp_path / "run.cpp"), "-o", exe], check=True, capture_output=True)
    cases = [(p, ck) for p in (0, 1, 31, 500, 1023, 1024, 5000, 10 ** 6, 10 ** 13)
             for ck in (32, 64, 128, 256, 512, 768, 1024, 2048, 4096, 10752)]
    out = subprocess.run([exe], input="".join("%d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.split()
    for (per_item, ck), run in zip(cases, map(int, out)):
        assert run >= 1 and (run == 1 or run * ck <= min(per_item, 1024)), (per_item, ck, run)
        assert run == 1 or (run + 1) * ck > min(per_item, 1024)
