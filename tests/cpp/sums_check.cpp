// Exact sums and range checks of the integer legs (mg_sums.h).
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>

#include "../../paper_2302_13903_gb300/csrc/mg_sums.h"

static int failures = 0;
#define CHECK(x)                                       \
  do {                                                 \
    if (!(x)) {                                        \
      std::printf("line %d: %s\n", __LINE__, #x);      \
      ++failures;                                      \
    }                                                  \
  } while (0)

// Pairs of values of one sign, up to the 4096 a thread of the sum pass adds: at
// 2^55 and more the plain 64-bit sum of 128 pairs wraps.
static void split_sum() {
  for (int bits : {0, 40, 54, 55, 57, 59})
    for (int sign : {1, -1})
      for (int planes : {4, 64, 128, 4096}) {
        const long long v = sign * ((1LL << bits) - 1);
        mg::SplitSum s;
        __int128 sum = 0;
        for (int p = 0; p < planes; ++p) {
          s.add(v + v + (p & 3));
          sum += v + v + (p & 3);
        }
        CHECK((__int128)s.hi() * ((__int128)1 << 32) + s.lo() == sum);
      }
}

// Against 64-bit pieces of the exact sum, for values up to the largest the legs
// form and as many of them as a thread of the source pass adds.
static void square_sum() {
  for (int bits : {0, 1, 24, 31, 32, 33, 48, 53, 58, 62, 63})
    for (int count : {1, 2, 128, 4096}) {
      mg::SquareSum s;
      unsigned __int128 low = 0;  // sums of the squares' lower and upper 64 bits
      unsigned __int128 high = 0;
      for (int q = 0; q < count; ++q) {
        const long long v = (long long)((1ull << bits) - 1 - (unsigned long long)(q % 3)) * (q % 2 ? 1 : -1);
        const long long r = bits < 2 ? (long long)((1ull << bits) - 1) : v;
        s.add(r);
        const unsigned __int128 a = r < 0 ? -(__int128)r : (__int128)r, sq = a * a;
        low += (unsigned long long)sq;
        high += (unsigned long long)(sq >> 64);
      }
      high += (unsigned long long)(low >> 64);
      CHECK(s.lo() == (unsigned long long)low);
      CHECK(s.hi() == (unsigned long long)high);
      CHECK(s.w4 == (unsigned)(high >> 64));
      const double want = (double)high * 0x1p64 + (double)(unsigned long long)low;
      CHECK(std::fabs(s.total() - want) <= 0x1p-52 * want);
    }
}

static void range() {
  const double limit = std::ldexp(1.0, 56);
  for (int sign : {1, -1}) {
    const double out[] = {limit, 1.5 * limit, 1e300, INFINITY, NAN};
    const double in[] = {0.0, 5e-324, 1.0, std::nextafter(limit, 0.0)};
    unsigned long long u;
    for (double x : out) {
      x = std::copysign(x, sign);
      std::memcpy(&u, &x, 8);
      CHECK(mg::past_range(u, 56));
    }
    for (double x : in) {
      x = std::copysign(x, sign);
      std::memcpy(&u, &x, 8);
      CHECK(!mg::past_range(u, 56));
    }
  }
}

int main() {
  split_sum();
  square_sum();
  range();
  std::printf(failures ? "FAILED\n" : "ok\n");
  return failures != 0;
}
