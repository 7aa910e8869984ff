// Host harness for the high-word rounding of csrc/cast.cuh (cast_hi) against the general
// integer rounding (cast_terms_int) of the same header: random, sparse-significand, tie and
// range-edge values for each single-term format.  Prints "fmt taken declined bad": bad counts
// values that cast_hi takes and rounds differently, or declines although the general
// rounding takes them (zeros excepted: the general rounding serves them).
#include <cstdint>
#include <cstdio>

#include "cast.cuh"

static uint64_t state = 0x9E3779B97F4A7C15ull;
static uint64_t next() {   // SplitMix64
  uint64_t z = (state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

template <class F>
static void run(const char* name) {
  long taken = 0, declined = 0, bad = 0;
  for (int it = 0; it < 4000000; ++it) {
    const int k = (int)(next() % 2200) - 1100;
    uint64_t frac = next() & 0xFFFFFFFFFFFFFull;
    switch (next() % 6) {
      case 0: frac &= next() & next() & next(); break;                       // few bits set
      case 1: frac = (frac >> (52 - F::MB) << (52 - F::MB)) | (1ull << (51 - F::MB)); break;   // ties
      case 2: frac = ((frac >> (52 - F::MB) << (52 - F::MB)) | (1ull << (51 - F::MB))) + (next() % 3) - 1; break;
      case 3: frac = 0xFFFFFFFFFFFFFull - (next() % 4); break;               // carries
      default: break;
    }
    // exponents around the format's range at this k, and anywhere
    int E = (next() & 1) ? (int)(next() % 2048) : 1023 - k + F::EMIN - 3 + (int)(next() % (F::EMAX - F::EMIN + 7));
    if (E < 0 || E > 2047) E = (int)(next() % 2048);
    const uint64_t u = (next() << 63) | ((uint64_t)E << 52) | (frac & 0xFFFFFFFFFFFFFull);
    uint32_t t[3], v = 0;
    const bool g = lsq::cast_terms_int<F>(u, k, t);
    const bool h = lsq::cast_hi<F>(u, lsq::cast_range<F>(k), v);
    if (h) ++taken;
    else ++declined;
    if (h && (!g || v != t[0])) ++bad;
    if (!h && g && (u << 1) != 0 && E < 2046) ++bad;
  }
  std::printf("%s %ld %ld %ld\n", name, taken, declined, bad);
}

int main() {
  run<lsq::EncBF16>("bf16");
  run<lsq::EncF16>("f16");
  run<lsq::EncE4M3>("e4m3");
}
