"""Host-side sizing rules of the library, compiled from its headers (CPU)."""
import os
import subprocess

from paper_1205_6693_gb300 import _build


def run_rules(tmp_path, body):
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include "engine.h"\nusing namespace tr;\n'
                   "int main() {\n" + body + "\n}\n")
    subprocess.run([_build.nvcc(), "-std=c++17", *_build.ARCH, "-I" + _build.CSRC,
                    "-I" + os.path.join(_build.ROOT, "include"), str(src), "-o", str(exe)],
                   check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def test_vertex_ranges_fit_the_space_taken_for_any_triangle_count(tmp_path):
    # the space is taken from an upper bound of the triangles, the ranges from
    # their number: fewer triangles can mean more ranges
    out = run_rules(tmp_path, """
  int64_t bad = 0;
  for (int64_t m : {0, 1, 63, 64, 65, 4096, 77823, 77824, 77825, 2621440}) {
    int64_t most = 0;
    for (int64_t step = 1, t = 0; t < (int64_t)1 << 33; t += step) {
      const ListRanges r = list_ranges(t, m);
      if (r.n1 > most) most = r.n1;
      if (r.n2 > most) most = r.n2;
      if (list_ranges_most(t, m) < most) bad++;
      if (t > (int64_t)1 << 21) step = t / 4096;
    }
  }
  printf("%lld", (long long)bad);
""")
    assert out == "0"
