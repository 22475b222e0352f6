"""The straight-line contraction of levels 18 and 20 (groups of graphs, as the
mixed kernels of large systems run it) compiled for the host in double, against
the interpreter's records: energy, basis values and dE/dM."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

from tests.test_tile_program_cpu import PKG, basisgen, run_records

HARNESS = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <vector>
#include <utility>
#include "graphs.cuh"
using GR = mtp::%s;
int main() {
  const int comps = %d, m = %d, graphs = %d;
  const double nan = std::nan("");
  std::vector<double> M(comps, nan), D(comps, nan), xi(m), B(m, nan), G(graphs, nan), GB(graphs, nan);
  int n = 0;
  if (scanf("%%d", &n) != 1) return 1;
  std::vector<int> swept(n);
  for (int& c : swept) if (scanf("%%d", &c) != 1) return 1;
  for (int c : swept) if (scanf("%%lf", &M[c]) != 1) return 1;
  for (double& x : xi) if (scanf("%%lf", &x) != 1) return 1;
  [&]<int... K>(std::integer_sequence<int, K...>) { (GR::values<K>(M.data(), 1, G.data(), 1), ...); }
  (std::make_integer_sequence<int, GR::VALUE_GROUPS>());
  const double E = GR::products<true>(G.data(), 1, xi.data(), GB.data(), [&](int a, double v) { B[a] = v; });
  [&]<int... K>(std::integer_sequence<int, K...>) { (GR::adjoint<K>(M.data(), 1, GB.data(), 1, D.data()), ...); }
  (std::make_integer_sequence<int, GR::ADJOINT_GROUPS>());
  printf("%%.17g\n", E);
  for (double v : B) printf("%%.17g\n", v);
  for (int c : swept) printf("%%.17g\n", D[c]);
}
"""


@pytest.mark.parametrize("level", [18, 20])
def test_graph_code(tmp_path, level):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    lv = basisgen.Level(level)
    code = basisgen.emit_graph_groups(lv)
    code = code if isinstance(code, str) else "\n".join(code)
    code, n = re.subn(r"using R = float;", "using R = double;", code)
    assert n == 1
    (tmp_path / "graphs.cuh").write_text(code)
    name = re.search(r"struct (\w+)", code).group(1)
    (tmp_path / "t.cpp").write_text(HARNESS % (name, len(lv.comps), lv.m, len(lv.roots)))
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O0", "-std=c++20", "-I", str(tmp_path), "-I", os.path.join(PKG, "csrc"),
                    str(tmp_path / "t.cpp"), "-o", exe], check=True, capture_output=True, timeout=600)
    g = np.random.default_rng(level)
    u = g.normal(size=(9, 3))
    u /= np.linalg.norm(u, axis=-1, keepdims=True)
    f = g.normal(size=(9, lv.nmu)) * 0.3
    M = np.array([(f[:, mu] * u[:, 0] ** K[0] * u[:, 1] ** K[1] * u[:, 2] ** K[2]).sum()
                  for mu, K in (lv.comps[c] for c in lv.swept)])
    xi = g.normal(size=lv.m)
    text = "\n".join([str(len(lv.swept)), *map(str, lv.swept), *("%.17g" % v for v in M), *("%.17g" % v for v in xi)])
    res = subprocess.run([exe], input=text, check=True, capture_output=True, text=True, timeout=120)
    v = np.array([float(t) for t in res.stdout.split()])
    b, d = run_records(lv, M[:, None], xi)
    # sums of at most a few thousand FP64 products of the same values
    assert abs(v[0] - xi @ b[:, 0]) <= 1e-11 * np.abs(xi * b[:, 0]).sum()
    assert np.abs(v[1:1 + lv.m] - b[:, 0]).max() <= 1e-11 * np.abs(b).max()
    assert np.abs(v[1 + lv.m:] - d[:, 0]).max() <= 1e-11 * np.abs(d).max()
