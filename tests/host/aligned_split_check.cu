// Host-side check of the persistent loop's aligned split (tc_common.cuh), run on the CPU: over
// many cloud sizes and CTA counts, aligned_ctas() never exceeds the CTAs offered nor the
// contiguous split's busiest CTA, every CTA has a non-empty segment in one row block, and a row
// block's CTAs, in order, cover its tiles exactly once. Exit status 0 on success.
#include <cstdint>
#include <cstdio>

#include "../../paper_2406_05061_gb300/csrc/tc_common.cuh"

using namespace progot::tc;

static int check_side(int R, int T, int G, int64_t most) {
  int r = 0, t = 0;
  for (int c = 0; c < G; ++c) {
    const Seg sg = aligned_segment(R, T, G, c);
    if (t == 0 && aligned_begin(R, G, r) != c) return std::printf("R=%d T=%d G=%d: row block %d\n", R, T, G, r), 1;
    if (sg.r != r || sg.t0 != t || sg.t1 <= sg.t0 || sg.t1 > T || sg.t1 - sg.t0 > most)
      return std::printf("R=%d T=%d G=%d: CTA %d has (%d, %d..%d)\n", R, T, G, c, sg.r, sg.t0, sg.t1), 1;
    t = sg.t1;
    if (t == T) t = 0, ++r;
  }
  return r == R && t == 0 ? 0 : (std::printf("R=%d T=%d G=%d: ends in row block %d\n", R, T, G, r), 1);
}

int main() {
  int64_t found = 0;
  for (int sms : {1, 4, 7, 148, 152})
    for (int bn : {128, 256})
      for (int64_t n = 1; n <= 20000; n += n < 600 ? 37 : 211)
        for (int64_t m = 1; m <= 20000; m += m < 600 ? 41 : 193) {
          const int64_t Rx = (n + 127) / 128, Ry = (m + 127) / 128, Tx = (n + bn - 1) / bn, Ty = (m + bn - 1) / bn;
          int64_t g = Rx * Ty < Ry * Tx ? Rx * Ty : Ry * Tx;
          if (g > sms) g = sms;
          const int G = aligned_ctas(Rx, Ty, Ry, Tx, g);
          if (G == 0) continue;
          ++found;
          if (G > g || check_side((int)Rx, (int)Ty, G, (Rx * Ty + g - 1) / g) ||
              check_side((int)Ry, (int)Tx, G, (Ry * Tx + g - 1) / g))
            return 1;
        }
  std::printf("aligned split ok (%lld)\n", (long long)found);
  return found > 1000 ? 0 : 1;
}
