// Host-side check of the fixed-link sweeps' 32-bit byte offsets on lattices of up to
// 2^28 sites of a parity (compiled with the undefined-behaviour sanitiser and run by
// test_byte_offsets_host.py; no GPU and no field needed): offset of the site plus
// SiteNb::bytes is 16 times the neighbour's index, without an overflow of int.
#include <cstdio>

#include "lgt_device.cuh"

using namespace lgt;

static int check(int nt, int n3, int n2, int n1) {
  Geom g;
  g.n1 = n1, g.n2 = n2, g.n3 = n3, g.nt = nt;
  g.half1 = n1 / 2;
  g.vs_half = (int)((long long)n1 * n2 * n3 / 2);
  g.vh = g.vs_half * nt;
  const unsigned i1 = index_inverse(g.vs_half, g.half1), i2 = index_inverse((long long)n2 * n3, n2);
  const int ts[] = {0, 1, nt / 2, nt - 2, nt - 1};
  for (int p = 0; p < 2; p++)
    for (int t : ts)
      for (int k = 0; k < 4096; k++) {
        // the slice's first and last sites, its middle and a walk through it
        const int walk = (int)((long long)g.vs_half * k / 4096);
        for (int j : {k, g.vs_half - 1 - k, g.vs_half / 2 + k, walk}) {
          if (j < 0 || j >= g.vs_half) continue;
          const Coords c = coords_in_slice(g, p, t, j);
          const SiteNb s(g, i1, i2, p, t, j);
          const unsigned o = (unsigned)(t * g.vs_half + j) * 16u;
          for (int mu = 0; mu < 4; mu++)
            for (int dir = -1; dir <= 1; dir += 2)
              if ((unsigned long long)(unsigned)(o + s.bytes(g, mu, dir)) != 16ull * (unsigned)cb_shift(g, c, mu, dir))
                return printf("%d x %d x %d x %d: parity %d, slice %d, site %d, direction %d\n", nt, n3, n2, n1, p, t, j,
                              dir * (mu + 1));
        }
      }
  return 0;
}

int main() {
  const int L[][4] = {{2, 2, 2, 2}, {4, 6, 10, 14}, {256, 64, 128, 128},                        // 2^27 sites of a parity
                      {2, 512, 512, 512}, {512, 128, 64, 64}, {2, 2, 8192, 8192}, {8, 254, 510, 510},
                      {1022, 64, 64, 128}, {2, 510, 1022, 514}};                               // just below 2^28
  for (auto &d : L)
    if (check(d[0], d[1], d[2], d[3])) return 1;
  printf("ok\n");
  return 0;
}
