// The integer split of an FP64 value into a float-float pair against the FP64 form: the same bits
// of both parts, on random values over the whole exponent range and on ties, carries, zeros,
// subnormals and non-finite values.  Prints "checked bad".
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "fmg_ff.cuh"

static unsigned long long state = 88172645463325252ull;
static unsigned long long rnd() {
  state ^= state << 13;
  state ^= state >> 7;
  state ^= state << 17;
  return state;
}
static unsigned bits(float f) {
  unsigned u;
  memcpy(&u, &f, 4);
  return u;
}
int main(int argc, char** argv) {
  const long n = argc > 1 ? atol(argv[1]) : 100000;
  long checked = 0, bad = 0;
  auto check = [&](unsigned long long b) {
    double x;
    memcpy(&x, &b, 8);
    const fmg::ff p = fmg::ff_from_double(x), q = fmg::ff_from_double_int(x);
    ++checked;
    const bool nan = p.hi != p.hi || p.lo != p.lo;
    if (nan ? (q.hi == q.hi && q.lo == q.lo) : (bits(p.hi) != bits(q.hi) || bits(p.lo) != bits(q.lo))) ++bad;
  };
  for (long i = 0; i < n; ++i) {
    const unsigned long long r = rnd();
    check(r);                                                                  // any exponent
    const unsigned long long e = 1023 - 80 + rnd() % 220, s = rnd() & 1;
    const unsigned long long f = r & 0xfffffffffffffull;
    check((s << 63) | (e << 52) | f);                                          // around the range's ends
    check((s << 63) | (e << 52) | (f & ~0x1fffffffull) | 0x10000000ull);       // ties
    check((s << 63) | (e << 52) | 0xfffffe0000000ull | (f & 0x1fffffffull));   // rounding over
    check((s << 63) | (e << 52) | (f & ~0x1fffffffull));                       // exact
  }
  for (unsigned long long s = 0; s < 2; ++s)
    for (unsigned long long v : {0ull, 1ull, 0xfffffffffffffull, 0x7ff0000000000000ull, 0x7ff8000000000000ull,
                                 0x7fefffffffffffffull, 0x0010000000000000ull})
      check((s << 63) | v);
  printf("%ld %ld\n", checked, bad);
  return bad != 0;
}
