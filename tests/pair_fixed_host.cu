// The fixed-point pair sequence of csrc/pair_fixed.cuh on the host: reads "k p dx dy" (hexadecimal
// floats), prints the four products of every order s = 0..2p as integers with 64 fractional bits.
#include <cstdio>
#include <vector>

#include "pair_fixed.cuh"

struct Entry {
  int64_t x, y;
};

int main() {
  const long double pi = 3.14159265358979323846264338327950288L;
  std::vector<Entry> tab(256);
  for (int i = 0; i < 256; ++i) {
    const long double a = 2 * pi * i / 256 - pi / 4;
    tab[i].x = (int64_t)rintl(cosl(a) * 0x1p62L);
    tab[i].y = (int64_t)rintl(sinl(a) * 0x1p62L);
  }
  double k, dx, dy;
  int p;
  while (scanf("%la %d %la %la", &k, &p, &dx, &dy) == 4) {
    const PairConsts q = pair_consts(k, pair_z_near(p));
    const double r2 = fma(dx, dx, dy * dy);
    if (pair_is_near(r2, q)) return 2;
    PairSeed o;
    pair_seed(dx, dy, r2, q, tab.data(), o);
    PairState a;
    PairStep t;
    pair_start(o, a, t);
    for (int s = 0; s <= 2 * p; s += 2) {
      int64_t v[8];
      pair_two_orders(a, t, 0, v);
      const long long sign = s & 2 ? -1 : 1;     // the sequence's signs + + - -
      for (int h = 0; h < 2 && s + h <= 2 * p; ++h)
        printf("%lld %lld %lld %lld\n", sign * (long long)v[4 * h], sign * (long long)v[4 * h + 1],
               sign * (long long)v[4 * h + 2], sign * (long long)v[4 * h + 3]);
    }
  }
  return 0;
}
