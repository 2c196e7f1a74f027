// Host-side check of the two-lane helpers (fx.cuh): each lane gives the
// scalar helper's bits, the fixed-point sum is within one unit of the exact
// increment over its whole range, and the lanes' fold keeps 44 bits.
#include "../paper_1006_0720_gb300/csrc/fx.cuh"
#include <cmath>
#include <cstdio>
#include <random>
using namespace fx;
static long bad = 0;
static void check(bool ok, const char* what) {
  if (!ok && ++bad < 10) printf("%s\n", what);
}
static bool same(df a, df b) { return f_bits(a.h) == f_bits(b.h) && f_bits(a.l) == f_bits(b.l); }
int main() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(-1, 1);
  auto rnd = [&](int span) { return from_double(U(g) * std::pow(2.0, -(int)(g() % span))); };
  for (int i = 0; i < 1000000; ++i) {
    const df a = rnd(40), b = rnd(40), c = rnd(40), d = rnd(40);
    const df2 p = mul_df2(pair(a, b), pair(c, d));
    check(same(p.lane0(), mul(a, c)) && same(p.lane1(), mul(b, d)), "mul_df2");
    const df2 q = mul_f2(pair(a, b), f2{c.h, d.h});
    check(same(q.lane0(), mul_f(a, c.h)) && same(q.lane1(), mul_f(b, d.h)), "mul_f2");
    acc x, y;
    x.init(a); x.add(c);
    y.init(b); y.add(d);
    acc2 z;
    z.init(pair(a, b)); z.add(pair(c, d));
    check(same(z.value().lane0(), x.value()) && same(z.value().lane1(), y.value()), "acc2");
    const df t = z.fold().value();
    const long double ex = (long double)a.h + a.l + b.h + b.l + c.h + c.l + d.h + d.l;
    const long double mag = fabsl(a.h) + fabsl(b.h) + fabsl(c.h) + fabsl(d.h);
    check(fabsl((long double)t.h + t.l - ex) <= mag * ldexpl(1.0L, -44), "fold");
    const int64_t X = (int64_t)(U(g) * std::pow(2.0, 62 - (int)(g() % 50)));
    const int64_t Y = (int64_t)(U(g) * std::pow(2.0, 62 - (int)(g() % 50)));
    const df2 o = fix2df2(X, Y, 56);
    check(same(o.lane0(), fix2df(X, 56)) && same(o.lane1(), fix2df(Y, 56)), "fix2df2");
    // increments: every magnitude up to the limits, the limits, zeros
    f2 h = {(float)(U(g) * std::pow(2.0, -(int)(g() % 70))), (float)(U(g) * std::pow(2.0, -(int)(g() % 70)))};
    f2 l = {(float)(U(g) * std::pow(2.0, -23 - (int)(g() % 60))), (float)(U(g) * std::pow(2.0, -23 - (int)(g() % 60)))};
    if (i % 100 == 0) h = f2{(g() & 1) ? 1.0f : -1.0f, (g() & 1) ? 0.0f : -0.0f};
    if (i % 100 < 2) l = f2{(g() & 1) ? kIncMax : -kIncMax, 0.0f};
    int64_t Xn = X, Yn = Y;
    add_inc2(Xn, Yn, h, l);
    const long double ix = ((long double)h.x + l.x) * ldexpl(1.0L, 56), iy = ((long double)h.y + l.y) * ldexpl(1.0L, 56);
    check(fabsl((long double)(Xn - X) - ix) <= 1.0L && fabsl((long double)(Yn - Y) - iy) <= 1.0L, "add_inc2");
  }
  printf("bad %ld\n", bad);
  return bad ? 1 : 0;
}
