"""Rules of the library that are plain host C++: compiled with the system compiler and run here."""

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2110_03607_gb300", "csrc")


def _run(tmp_path, headers, body):
    src = tmp_path / "rule.cpp"
    inc = "".join('#include "%s"\n' % os.path.join(CSRC, h) for h in headers)
    src.write_text("#include <cstdio>\n" + inc + "using namespace hotrg;\n"
                   "#define CHECK(x) do { if (!(x)) { std::printf(\"line %d: %s\\n\", __LINE__, #x); return 1; } } while (0)\n"
                   "int main() {\n" + body + "\nreturn 0;\n}\n")
    exe = tmp_path / "rule"
    subprocess.run(["g++", "-std=c++17", "-O1", "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_a_refused_product_moves_no_offset(tmp_path):
    """Two parity blocks share a buffer of partials: the second one's place follows from what the first
    wrote.  A refused first product (each status of the library) leaves the second at the start."""
    _run(tmp_path, ["partials.h"], """
      const long long mb = 128;
      for (int status = -7; status <= 0; ++status) {
        const int n = partials_written(status);
        CHECK(n == 0);
        CHECK((long long)n * mb * mb == 0);
      }
      CHECK(partials_written(1) == 1 && partials_written(256) == 256);
    """)


def test_a_class_is_lost_with_every_turn_that_mixes_it(tmp_path):
    """An even vector p turned against two odd ones q, r, in any order and with q against r: all three
    are mixtures afterwards.  Vectors of one class keep it, those of two components do not."""
    _run(tmp_path, ["eig_class.h"], """
      const int cls[3] = {+5, -5, -5};
      const int pairs[3][2] = {{0, 1}, {0, 2}, {1, 2}};
      const int order[4][3] = {{0, 1, -1}, {1, 0, -1}, {0, 2, -1}, {2, 1, 0}};
      for (auto& o : order) {
        bool lost[3] = {false, false, false};
        for (int step = 0; step < 3 && o[step] >= 0; ++step) {
          const int p = pairs[o[step]][0], q = pairs[o[step]][1];
          if (turn_ends_class(cls[p], lost[p], cls[q], lost[q])) lost[p] = lost[q] = true;
          CHECK(turn_ends_class(cls[p], lost[p], cls[q], lost[q]) == turn_ends_class(cls[q], lost[q], cls[p], lost[p]));
        }
        CHECK(lost[0] && lost[1] && lost[2]);
      }
      CHECK(!turn_ends_class(5, false, 5, false) && !turn_ends_class(0, false, 0, false));
      CHECK(turn_ends_class(5, false, 7, false) && turn_ends_class(5, false, -7, false) && turn_ends_class(5, false, 0, false));
    """)
