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


@pytest.mark.parametrize("room,n,parts,graphs,expect", [
    # 295 components and 159 graphs in FP32: 1,180 B per atom and buffer, 1,272 B of graph values
    (10 ** 9, 4200, 4, 159, "1 4 1"),                       # everything fits
    (5 * 1180 * 4200 + 2 * 4 * 159 * 4224, 4200, 4, 159, "1 4 1"),       # to the byte
    (5 * 1180 * 4200 + 2 * 4 * 159 * 4224 - 1, 4200, 4, 159, "1 4 0"),   # not the graph values
    (5 * 1180 * 4200, 4200, 4, 159, "1 4 0"),
    (5 * 1180 * 4200 - 1, 4200, 4, 159, "1 1 0"),           # one share of the neighbours
    (2 * 1180 * 4200, 4200, 4, 159, "1 1 0"),
    (2 * 1180 * 4200 - 1, 4200, 4, 159, "0 0 0"),
    (2 * 1180 * 4200 - 1, 4200, 1, 0, "0 0 0"),
    (2 * 1180 * 8, 1, 1, 0, "1 1 0"),                       # one atom: a whole tile of 8
    (2 * 1180 * 8 - 1, 1, 1, 0, "0 0 0"),
])
def test_split_plan(tmp_path, room, n, parts, graphs, expect):
    out = compiled_run(tmp_path, """
  const auto p = mtp::plan_split_scratch(295, %d, %d, sizeof(float), %d, [](size_t b) { return b <= (size_t)%dll; });
  std::printf("%%d %%d %%d", (int)p.ok, p.parts, (int)p.graphs);""" % (n, parts, graphs, room))
    assert out == expect
