// Host-only check of the launch geometry of the stateless similarity calls (batch 0; no device needed, the SM
// count falls back to GB300's 152 without one), for every shape, window and similarity:
//   - the D chunks cover the depth exactly once and the CTAs are the tiles times the chunks;
//   - LNCC has the chunks of the engine's rule for one pair, SiLNCC at most 8 CTAs per SM unless one chunk
//     has more;
//   - a volume that the allocation-free call admits (128^3 voxels) has at most 2^17 CTAs, the partial
//     sums of its fixed scratch.
// Prints the number of cases checked and exits non-zero on the first violation.
#include <cstdio>

#include "kernels.h"

using namespace muster;

static int fail(const char* what, Dims n, int w, int kind) {
  std::printf("FAIL %s at D=%d H=%d W=%d window=%d kind=%d\n", what, n.n0, n.n1, n.n2, w, kind);
  return 1;
}

int main() {
  const int sizes[] = {3, 5, 8, 17, 31, 33, 40, 48, 64, 81, 96, 128, 160, 192, 256, 511, 1024, 4096};
  long checked = 0;
  for (int D : sizes)
    for (int H : sizes)
      for (int W : sizes)
        for (int w = 3; w <= 11; w += 2)
          for (int kind = 0; kind < 2; ++kind) {
            const Dims n{D, H, W};
            const SimGeom g = sim_geom(n, w, 0, kind);
            const long tiles = (long)((W + 31) / 32) * ((H + 15) / 16);
            if (g.tz < 1 || (long)g.nzc * g.tz < D || (long)(g.nzc - 1) * g.tz >= D) return fail("chunk cover", n, w, kind);
            if (g.ctas != tiles * g.nzc) return fail("CTA count", n, w, kind);
            if (kind == 1 && g.tz != sim_geom(n, w, 1, kind).tz) return fail("LNCC chunks", n, w, kind);
            if (kind == 0 && g.nzc > 1 && g.ctas > 8 * 152) return fail("SiLNCC chunks", n, w, kind);
            if ((double)D * H * W <= 2097152.0 && g.ctas > 1 << 17) return fail("partial sums", n, w, kind);
            ++checked;
          }
  std::printf("GEOMETRY-OK %ld\n", checked);
  return 0;
}
