// Host check of row_exponent (the scale of an aligned row in the split form)
// and of the room that the leading digits leave in FP32 sums.  For largest
// entries over every binade (subnormals included), with high words around the
// threshold and at random: every entry up to the row's largest (the low word of
// the largest unknown) has |X| <= 2^(8S-1); in the default split its leading
// digit is at most 511 and the others in [-512, 511]; E is the binade's own or,
// only within 2^-9 below its end, one more.  Then the sums between two drains,
// with the rest of up to 4 that a drain leaves, stay within 2^24.  Prints
// "ok <cases>" and exits 0, or reports the first mismatch and exits 1.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#include "symctr_internal.h"

using namespace symctr;

namespace {

double from_bits(uint64_t b) {
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}

// round(x * 2^(38 - E)), exact: the scaled value has at most 53 bits
int64_t fixed39(double x, int e) { return (int64_t)std::floor(std::ldexp((long double)x, 38 - e) + 0.5L); }

bool digits_ok(int64_t X) {
  const int64_t B = 512ll * ((1ll << 30) + (1ll << 20) + (1ll << 10) + 1), Y = X + B;
  const int64_t a0 = (Y >> 30) - 512, a1 = ((Y >> 20) & 1023) - 512, a2 = ((Y >> 10) & 1023) - 512,
                a3 = (Y & 1023) - 512;
  if ((((a0 * 1024 + a1) * 1024 + a2) * 1024 + a3) != X) return false;
  return a0 >= -511 && a0 <= 511 && a1 >= -512 && a2 >= -512 && a3 >= -512;
}

}  // namespace

int main() {
  std::mt19937_64 rng(7);
  long cases = 0;
  auto check = [&](uint32_t hi, uint32_t lo) {
    const uint64_t known = hi != 0 ? (uint64_t)hi << 32 : (uint64_t)lo;
    if (known == 0) return true;
    const uint64_t most = hi != 0 ? known | 0xFFFFFFFFull : known;
    ++cases;
    int binade;
    std::frexp(from_bits(most), &binade);
    auto clamped = [&](int S) { return binade - 1 > 8 * S - 1076 ? binade - 1 : 8 * S - 1076; };
    const int own = clamped(5);
    const int e = row_exponent(known, 5);
    const double x = from_bits(most);
    const bool near = x >= std::ldexp(1.0 - std::ldexp(1.0, -9), own + 1);
    bool ok = e == own || (e == own + 1 && near);
    for (int S = 2; S <= 6; ++S)
      if (S != 5) ok = ok && row_exponent(known, S) == clamped(S);
    ok = ok && row_exponent(most, 5) == e;     // the low word does not count
    for (const double y : {x, -x, from_bits(known), -from_bits(known), x / 2, -x / 3})
      ok = ok && digits_ok(fixed39(y, e));
    if (!ok) std::printf("mismatch: high word %08x low %08x E %d, own %d\n", hi, lo, e, own);
    return ok;
  };
  for (uint32_t ef = 0; ef < 2047; ++ef)
    for (uint32_t f : {0u, 1u, 0x80000u, 0xFF000u, 0xFF7FAu, 0xFF7FBu, 0xFF7FCu, 0xFF7FDu, 0xFF7FEu, 0xFF7FFu,
                       0xFF800u, 0xFFBFFu, 0xFFFFEu, 0xFFFFFu})
      if (!check(ef << 20 | f, 0)) return 1;
  for (int nb = 1; nb <= 20; ++nb)             // subnormals: every length of the high word
    for (int i = 0; i < 4096; ++i) {
      const uint32_t top = i < 2048 ? 0xFFFFFFFFu - i : (uint32_t)rng() | 0x80000000u;
      if (!check(top >> (32 - nb), 0)) return 1;
    }
  for (int nb = 1; nb <= 32; ++nb)
    for (uint32_t top : {0x80000000u, 0xFFFFFFFFu, 0xFFBFF000u})
      if (!check(0, top >> (32 - nb))) return 1;
  for (int i = 0; i < 2000000; ++i)
    if (!check((uint32_t)(rng() % 0x7FF00000u), (uint32_t)rng())) return 1;
  for (int i = 0; i < 2000000; ++i)            // around the threshold
    if (!check((uint32_t)(rng() % 2046 + 1) << 20 | (uint32_t)(0xFF000 + rng() % 0x1000), 0)) return 1;
  const int64_t lead = 511, low = 512, rest = 4, limit = 1 << 24;
  if (64 * lead * lead + rest > limit || 32 * 2 * lead * low + rest > limit) {
    std::printf("the sums between two drains exceed 2^24\n");
    return 1;
  }
  std::printf("ok %ld\n", cases);
  return 0;
}
