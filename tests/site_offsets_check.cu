// Host-side check of the index arithmetic of the fixed-link sweeps (compiled and
// run by test_site_offsets_host.py; no GPU needed): for every site of every
// parity and slice, SiteNb gives the coordinates of coords_in_slice, and index
// plus offset(mu, dir) is cb_shift's neighbour, with the reciprocals of
// index_inverse and with the plain divisions that replace them (inv = 0).  And
// index_div is the integer division over the whole range index_inverse admits.
#include <cstdio>
#include <cstdlib>

#include "lgt_device.cuh"

using namespace lgt;

static int check(int nt, int n3, int n2, int n1) {
  Geom g;
  g.n1 = n1, g.n2 = n2, g.n3 = n3, g.nt = nt;
  g.half1 = n1 / 2;
  g.vs_half = n1 * n2 * n3 / 2;
  g.vh = g.vs_half * nt;
  const unsigned i1 = index_inverse(g.vs_half, g.half1), i2 = index_inverse((long long)n2 * n3, n2);
  for (int use = 0; use < 2; use++)
    for (int p = 0; p < 2; p++)
      for (int t = 0; t < nt; t++)
        for (int j = 0; j < g.vs_half; j++) {
          const Coords c = coords_in_slice(g, p, t, j);
          const SiteNb s(g, use ? i1 : 0u, use ? i2 : 0u, p, t, j);
          const Coords d = s.coords(t);
          if (c.x1 != d.x1 || c.x2 != d.x2 || c.x3 != d.x3 || c.t != d.t) return 1;
          for (int mu = 0; mu < 4; mu++)
            for (int dir = -1; dir <= 1; dir += 2)
              if (t * g.vs_half + j + s.offset(g, mu, dir) != cb_shift(g, c, mu, dir)) return 2;
        }
  return 0;
}

int main() {
  const int L[][4] = {{2, 2, 2, 2}, {4, 6, 10, 14}, {6, 2, 4, 2}, {2, 4, 2, 6}, {8, 8, 8, 8}, {4, 2, 2, 30}, {2, 14, 22, 34}};
  for (auto &d : L)
    if (int r = check(d[0], d[1], d[2], d[3])) {
      printf("%d x %d x %d x %d: check %d failed\n", d[0], d[1], d[2], d[3], r);
      return 1;
    }
  for (int d = 1; d < 70000; d = d < 300 ? d + 1 : d * 3 / 2 + 1) {
    const long long top = (1ll << 32) / d;  // the largest limit with a reciprocal lies just below
    const long long limit = top < (1ll << 31) ? top - 1 : (1ll << 31) - 1;
    const unsigned inv = index_inverse(limit, d);
    if (d >= 2 && (limit * d < (1ll << 32)) != (inv != 0)) return printf("index_inverse(%lld, %d)\n", limit, d), 1;
    if (index_inverse(1ll << 32, d) != 0) return printf("index_inverse(2^32, %d)\n", d), 1;
    for (long long k = 0; k < 2000; k++)
      for (long long x : {k, limit - 1 - k, (limit / 2000) * k, (limit / d / 2) * d + k % (2 * d) - d})
        if (x >= 0 && x < limit && index_div((int)x, inv, d) != (int)(x / d)) return printf("%lld / %d\n", x, d), 1;
  }
  printf("ok\n");
  return 0;
}
