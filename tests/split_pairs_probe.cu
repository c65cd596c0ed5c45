// Host probe of the pairs that a split step's stage sums and its new state are made
// of (step_split.cuh) against long double.  Prints one line per quantity: the
// largest error over its bound's unit.
#include <cmath>
#include <cstdio>
#include <random>

#include "step_split.cuh"

using namespace bhrt;
typedef long double LD;

static LD ld(F2 x) { return (LD)x.h + (LD)x.l; }
static LD ld(float a, float b, float c) { return (LD)a + (LD)b + (LD)c; }

int main() {
  std::mt19937_64 g(20260601);
  std::uniform_real_distribution<double> U(0, 1);
  const DPTab2 tab = make_tab2(kDP);
  auto draw = [&](double top) {
    return f2_of((U(g) - 0.5) * top * std::exp(-8.0 * U(g)));
  };
  // a product c k, and the sums of the tableau's rows over random stages
  LD ep = 0, es = 0;
  for (int t = 0; t < 100000; ++t) {
    F2 k[7][2];
    F2x2 kv[7];
    for (int j = 0; j < 7; ++j) {
      k[j][0] = draw(4.0);
      k[j][1] = draw(400.0);
      kv[j] = pair(k[j][0], k[j][1]);
    }
    for (int row = 0; row < 9; ++row) {
      const Coef* c = row < 7 ? tab.a[row] : (row == 7 ? tab.e : tab.d);
      const int n = row < 7 ? (row ? row : 1) : 7;
      F2x2 q = v_prod(c[0], kv[0]);
      for (int i = 0; i < 2; ++i) {
        const LD want = ((LD)c[0].h.x - (LD)c[0].nl.x) * ld(k[0][i]);
        const F2 p = i ? second(q) : first(q);
        if (want != 0) ep = fmaxl(ep, fabsl(((LD)p.h - (LD)p.l) / want - 1));
      }
      q.l = v_sub(0ull, q.l);
      for (int j = 1; j < n; ++j) q = v_acc(c[j], kv[j], q);
      for (int i = 0; i < 2; ++i) {
        LD want = 0, mag = 0;
        for (int j = 0; j < n; ++j) {
          const LD p = ((LD)c[j].h.x - (LD)c[j].nl.x) * ld(k[j][i]);
          want += p;
          mag += fabsl(p);
        }
        es = fmaxl(es, fabsl(ld(i ? second(q) : first(q)) - want) / mag);
      }
    }
  }
  // a state of 2,000 increments, each the h q of a step as d.h - d.l
  LD ea = 0;
  for (int t = 0; t < 200; ++t) {
    const F3 a = f3_of(1000.0 * U(g)), b = f3_of(3.0 * U(g));
    F3x2 y{pk(a.a, b.a), pk(a.b, b.b), pk(a.c, b.c)};
    LD sum[2] = {ld(a.a, a.b, a.c), ld(b.a, b.b, b.c)};
    for (int i = 0; i < 2000; ++i) {
      const F2 d0 = f2_of((U(g) - 0.5) * std::exp(8 * U(g) - 6)), d1 = f2_of((U(g) - 0.5) * 0.1);
      y = v_add3(y, pair(mk2(d0.h, -d0.l), mk2(d1.h, -d1.l)));
      sum[0] += ld(d0);
      sum[1] += ld(d1);
    }
    ea = fmaxl(ea, fabsl(ld(lo_of(y.a), lo_of(y.b), lo_of(y.c)) - sum[0]) / 2000);
    ea = fmaxl(ea, fabsl(ld(hi_of(y.a), hi_of(y.b), hi_of(y.c)) - sum[1]) / 2000);
  }
  std::printf("v_prod %.6Lg\nv_acc %.6Lg\nv_add3 %.6Lg\n", ep, es, ea);
  return 0;
}
