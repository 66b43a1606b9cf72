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


def test_classes_of_turned_vectors(tmp_path):
    """Even and odd vectors of a component are not turned against each other.  A vector without a class (0,
    or of another component) turned against an even one, that against an odd one, in any order that the
    rules allow: whatever took part in a mixture has no class left, and none is handed on by tiny angles."""
    _run(tmp_path, ["eig_class.h"], """
      CHECK(turn_forbidden(5, false, -5, false) && !turn_forbidden(0, false, 0, false));
      CHECK(!turn_forbidden(5, true, -5, false) && !turn_forbidden(5, false, -5, true));
      CHECK(!turn_forbidden(5, false, 5, false) && !turn_forbidden(5, false, -7, false));
      for (int other = -7; other <= 0; other += 7) {
        const int cls[4] = {+5, -5, -5, other};
        const int order[3][3][2] = {{{0, 3}, {0, 1}, {1, 2}}, {{3, 1}, {0, 1}, {0, 2}}, {{2, 3}, {0, 2}, {1, 0}}};
        for (auto& o : order) {
          bool lost[4] = {false, false, false, false}, mixed[4] = {false, false, false, false};
          for (auto& pq : o) {
            const int p = pq[0], q = pq[1];
            if (turn_forbidden(cls[p], lost[p], cls[q], lost[q])) continue;
            CHECK(!turn_ends_class(cls[p], lost[p], cls[q], lost[q], 1e-9));
            if (cls[p] != cls[q] || mixed[p] || mixed[q]) mixed[p] = mixed[q] = true;
            const bool ends = turn_ends_class(cls[p], lost[p], cls[q], lost[q], 0.7);
            CHECK(ends == turn_ends_class(cls[q], lost[q], cls[p], lost[p], -0.7));
            if (ends) lost[p] = lost[q] = true;
          }
          for (int i = 0; i < 4; ++i) CHECK(lost[i] == mixed[i]);
        }
      }
      CHECK(!turn_ends_class(5, false, 5, false, 1.0) && !turn_ends_class(0, false, 0, false, 1.0));
    """)


def test_grams_of_2d_steps_stay_on_the_fp64_pipe(tmp_path):
    """Up to the largest bonds (32 x 32 terms): the kept vectors of a degenerate cut follow their rounding."""
    _run(tmp_path, ["f64_rule.h"], """
      for (int c = 2; c <= 32; ++c)
        for (int j = 2; j <= 32; ++j) CHECK(!f64_gram_digits_pay(c * j, c * j, true));
      CHECK(f64_gram_digits_pay(256, 4096, true) && !f64_gram_digits_pay(24, 1 << 20, true));
      CHECK(!f64_digits_pay(256, 256, 255, false) && f64_digits_pay(256, 256, 256, false));
      CHECK(f64_digits_pay(256, 256, 512, true) && !f64_digits_pay(256, 256, 511, true));
    """)
