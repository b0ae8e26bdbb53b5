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


def test_a_peel_that_shares_the_device_is_limited_unless_it_is_wide(tmp_path):
    out = run_rules(tmp_path, """
  const int64_t wide = kWideWork;
  for (int64_t work : {(int64_t)0, wide / 2, wide - 1, wide, 40 * wide})
    printf("%d %d ", peel_sms(work, 152), peel_share(work, peel_sms(work, 152), 38));
  printf("| %d %d %d", peel_share(wide - 1, 24, 38), peel_share(wide - 1, 76, 0),
         peel_sms(0, 48));
""")
    assert out == "24 24 76 38 76 38 152 152 152 152 | 24 76 48"


def test_queued_small_requests_count_as_the_runs_they_make(tmp_path):
    out = run_rules(tmp_path, """
  struct R { int64_t rows; };
  auto runs = [](std::vector<int64_t> rows, int max_batch, int most) {
    std::vector<R> r;
    for (int64_t x : rows) r.push_back({x});
    std::vector<R *> q;
    for (R &x : r) q.push_back(&x);
    return queued_runs(q.begin(), q.end(), 100, max_batch, most);
  };
  printf("%d %d %d %d %d %d", runs({}, 4, 4), runs({1, 100, 7}, 4, 4), runs({1, 2, 3, 4, 5}, 4, 4),
         runs({1, 101, 2, 3, 102, 103}, 4, 8), runs({101, 101, 101}, 4, 2), runs({1, 1, 1}, 1, 8));
""")
    assert out == "0 1 2 5 2 3"
