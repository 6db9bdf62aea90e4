"""Float64 value of an element's weight-class sums (csrc/class_sum.cuh), compiled for
the host: correctly rounded from the exact sum of the classes while all of them stay
below 2^30 in units of their last digit (sums around and beyond 2^53 for four and five
slices among them), with or without the checks of long contractions; beyond that within 2^-51 of the sum of their
magnitudes (S roundings of a float64 sum)."""
import os
import subprocess
import textwrap

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_class_sum_ranges(tmp_path):
    src = tmp_path / "cs.cpp"
    src.write_text(textwrap.dedent("""
        #include <cstdio>
        #include <random>
        #include "class_sum.cuh"
        static std::mt19937_64 rng(7);
        static int bad = 0;
        // classes of 24 significant bits below 2^top; exact sum in 128-bit integers
        template <int S, int BITS, bool INTS>
        void run(int top0, int top) {
          for (int it = 0; it < 20000; ++it) {
            float c[S];
            __int128 exact = 0, mag = 0;
            bool fits = true;
            for (int g = 0; g < S; ++g) {
              const int t = g == 0 ? top0 : top;
              double x = (double)(int64_t)(rng() >> (64 - t));
              if (it % 3 == 0) x = std::ldexp(1.0, t) - (double)(rng() & 3);
              float f = (float)x;
              if (it & 1 ? (rng() & 1) : g > 0 && (it & 2)) f = -f;
              exact = exact * ((__int128)1 << BITS) + (__int128)f;
              mag = mag * ((__int128)1 << BITS) + (__int128)fabsf(f);
              fits = fits && fabsf(f) < 1073741824.0f;
              c[g] = INTS ? f : std::ldexp(f, -BITS * g);
            }
            const int e = (int)(rng() % 1800) - 900;
            const double got = lno::class_sum<S, BITS, INTS, true>(c, e, false);
            const double want = std::ldexp((double)exact, e - BITS * (S - 1));
            const double tol = std::ldexp((double)mag, e - BITS * (S - 1) - 51);
            if (fits ? got != want : !(std::fabs(got - want) <= tol)) ++bad;
            if (top0 <= 28 && top <= 30 &&
                lno::class_sum<S, BITS, INTS, false>(c, e, false) != want) ++bad;
          }
        }
        int main() {
          for (int t0 : {1, 5, 19, 20, 21, 22, 24, 28, 29, 30, 31, 33})
            for (int t : {3, 16, 24, 29, 30, 32}) {
              run<2, 8, false>(t0, t);
              run<4, 8, false>(t0, t);
              run<5, 8, false>(t0, t);
              run<3, 11, true>(t0, t);
            }
          const float nan4[4] = {NAN, 1.f, 0.f, 0.f}, inf4[4] = {INFINITY, 0.f, 0.f, 0.f};
          if (!std::isnan(lno::class_sum<4, 8, false, true>(nan4, 0, false))) ++bad;
          if (!std::isnan(lno::class_sum<4, 8, false, false>(inf4, 0, true))) ++bad;
          const float flat[5] = {4194304.f, 0.f, 0.f, 0.f, 0.f};   // 2^22 2^32 = 2^54
          if (lno::class_sum<5, 8, false, false>(flat, -14, false) != 256.0) ++bad;
          std::printf("%d\\n", bad);
          return 0;
        }
    """))
    exe = tmp_path / "cs"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2311_10048_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True,
                          check=True).stdout.strip() == "0"
