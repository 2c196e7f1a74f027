// Host-side check of the range test in front of the fixed-point sum (fx.cuh):
// NaN or infinity in any single part is refused, the limits are where add_inc2
// has them, and a velocity with one NaN component gives a refused increment.
#include "../paper_1006_0720_gb300/csrc/fx.cuh"
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include <limits>
using namespace fx;
static int bad = 0;
static void check(bool ok, const char* what) {
  if (!ok) { ++bad; printf("%s\n", what); }
}
int main() {
  const float nan = std::numeric_limits<float>::quiet_NaN(), inf = std::numeric_limits<float>::infinity();
  const float wrong[] = {nan, -nan, inf, -inf};
  for (float w : wrong)
    for (int part = 0; part < 4; ++part) {
      float v[4] = {0.25f, -0.5f, 0x1p-30f, 0.0f};
      v[part] = w;
      check(!inc_fits(f2{v[0], v[1]}, f2{v[2], v[3]}), "a part that is not finite passes");
    }
  for (float h : {1.0f, -1.0f, 2.0f}) {
    check(!inc_fits(f2{h, 0.0f}, f2{0.0f, 0.0f}) && !inc_fits(f2{0.0f, h}, f2{0.0f, 0.0f}), "a whole unit passes");
  }
  const float below = std::nextafterf(1.0f, 0.0f), above = std::nextafterf(kIncMax, 1.0f);
  check(inc_fits(f2{below, -below}, f2{kIncMax, -kIncMax}), "the limits are refused");
  check(!inc_fits(f2{0.0f, 0.0f}, f2{above, 0.0f}) && !inc_fits(f2{0.0f, 0.0f}, f2{0.0f, -above}), "a low part above its limit passes");
  // the particle step's increment U dt + s dW
  for (int c = 0; c < 2; ++c) {
    const df one = from_double(0.7), dt = from_double(1e-3), s = from_double(1.4e-3), nn = df{nan, 0.0f};
    acc2 a;
    a.init(mul_df2(c == 0 ? pair(nn, one) : pair(one, nn), pair(dt, dt)));
    a.add(mul_f2(pair(s, s), f2{0.3f, -0.2f}));
    check(!inc_fits(a.h, a.l), "a NaN velocity component passes");
  }
  printf("bad %d\n", bad);
  return bad ? 1 : 0;
}
