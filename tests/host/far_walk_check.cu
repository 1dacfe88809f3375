// Host check of the far field's walk over an entry's window (Eq. tDxx): the lines
// outside the pair box, cut into pieces of `seg` points as the kernel takes them,
// against brute force.  Prints "ok" and exits 0, or the first mismatch and exits 1.
#include <cstdio>
#include <vector>

#include "../../paper_2208_06097_gb300/csrc/sea_internal.cuh"

static unsigned long long rng_state = 0x9E3779B97F4A7C15ULL;
static int rnd(int lo, int hi) {  // uniform in [lo, hi]
  rng_state = rng_state * 6364136223846793005ULL + 1442695040888963407ULL;
  return lo + (int)((rng_state >> 33) % (unsigned long long)(hi - lo + 1));
}

int main() {
  const int segs[] = {1, 2, 3, 8, 1024};
  for (int it = 0; it < 30000; ++it) {
    Entry e{};
    PairInfo P{};
    for (int a = 0; a < 3; ++a) {
      e.wl[a] = rnd(1, 13);
      e.ws[a] = rnd(-20, 20);
      P.ext[a] = rnd(1, 15);
      // pair box near, inside, around, across or away from the window
      P.lo[a] = e.ws[a] + rnd(-P.ext[a] - 2, e.wl[a] + 2);
    }
    const sea::WinSplit s = sea::window_split(e, P);
    const sea::WinLines nl = sea::window_lines(s, e.wl);
    const int wx = e.wl[0], wy = e.wl[1], wz = e.wl[2];
    const int seg = segs[it % 5], nseg = (wx + seg - 1) / seg;
    std::vector<int> seen((size_t)wx * wy * wz, 0);
    for (int item = 0; item < (nl.n_whole + nl.n_cut) * nseg; ++item) {
      const int i = item / nseg, x0 = (item - i * nseg) * seg, x1 = wx < x0 + seg ? wx : x0 + seg;
      int ty, tz;
      sea::window_outside_line(s, e.wl, i, &ty, &tz);
      const bool cut = i >= nl.n_whole;
      for (int tx = sea::window_piece_first(s, cut, x0); tx < x1;
           tx = sea::window_piece_next(s, cut, tx)) {
        if (tx < 0 || tx >= wx || ty < 0 || ty >= wy || tz < 0 || tz >= wz) {
          printf("it %d item %d: (%d, %d, %d) out of the window\n", it, item, tx, ty, tz);
          return 1;
        }
        ++seen[((size_t)tz * wy + ty) * wx + tx];
      }
    }
    for (int z = 0; z < wz; ++z)
      for (int y = 0; y < wy; ++y)
        for (int x = 0; x < wx; ++x) {
          const int l[3] = {e.ws[0] + x - P.lo[0], e.ws[1] + y - P.lo[1], e.ws[2] + z - P.lo[2]};
          bool in = true;
          for (int a = 0; a < 3; ++a) in = in && l[a] >= 0 && l[a] < P.ext[a];
          if (seen[((size_t)z * wy + y) * wx + x] != (in ? 0 : 1)) {
            printf("it %d: (%d, %d, %d) inside %d taken %d times\n", it, x, y, z, (int)in,
                   seen[((size_t)z * wy + y) * wx + x]);
            return 1;
          }
        }
  }
  printf("ok\n");
  return 0;
}
