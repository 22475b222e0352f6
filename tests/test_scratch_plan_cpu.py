"""What a call allocates when memory is short (csrc/scratch_plan.h), compiled
for the host with allocations that fail above a limit."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_00193_gb300", "csrc")


def compiled_run(tmp_path, body):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text('#include <cassert>\n#include <cstdio>\n#include "scratch_plan.h"\nint main() {\n%s\n}\n' % body)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True, capture_output=True, text=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout


@pytest.mark.parametrize("room,held,expect", [
    (100, 0, "1 0"),      # fits at once
    (100, 40, "1 40"),    # fits beside what is held: that stays
    (59, 40, "1 0"),      # fits once it is given back
    (49, 0, "0 0"),       # nothing to give back
    (30, 20, "0 0"),      # not even then
])
def test_allocate_dropping(tmp_path, room, held, expect):
    out = compiled_run(tmp_path, """
  long room = %d, held = %d, want = 50;
  bool ok = mtp::allocate_dropping([&] { return held + want <= room; },
                                   [&] { if (!held) return false; held = 0; return true; });
  std::printf("%%d %%ld", (int)ok, held);""" % (room, held))
    assert out == expect
