// Host check of the convolutions' plans, run by tests/test_conv_plans.py.
#include "../../paper_1104_1703_gb300/csrc/kernels_unet.cu"

#include <cstdio>

namespace gbmg {
void count_launch(unsigned long long) {}
int device_sms() { return 152; }
}  // namespace gbmg

using namespace gbmg;

static int fails = 0;

static void need(bool ok, const char* what, const ConvArgs& a) {
  if (ok) return;
  if (++fails <= 20) std::printf("%s: %d x %d x %d, %d -> %d, group %d\n", what, a.W, a.H, a.D, a.cin, a.cout, a.group);
}

static int tiles_of(const ConvArgs& a) {
  int bx, by, bz;
  conv_tile_box(a.W, a.H, a.D, kConvTileM, &bx, &by, &bz);
  return ((a.W + bx - 1) / bx) * ((a.H + by - 1) / by) * ((a.D + bz - 1) / bz);
}

static void check(int W, int H, int D, int cin, int cout) {
  ConvArgs a = {};
  a.W = W;
  a.H = H;
  a.D = D;
  a.cin = cin;
  a.cout = cout;
  conv_plan(a);
  need(a.bx * a.by * a.bz == kConvTileM * a.group, "box", a);
  need(a.ntx * a.bx >= W && a.nty * a.by >= H && a.ntz * a.bz >= D, "cover", a);
  need(a.bx <= 256 && a.by <= 256 && a.bz <= 256 && (!a.halo || (a.group + 2 <= 256 && a.bx == 128)), "copy box", a);
  need(a.stages >= 2 && a.stages <= kConvMaxStages && conv_smem_bytes(a) <= 227 * 1024, "shared memory", a);
  need(conv_tmem_cols(a.group, cout) <= 512, "TMEM columns", a);
  need(cin % a.span == 0 && (a.kc * 8) % a.span == 0 && (cin / 8) % a.kc == 0, "chunks", a);
  // tiles are put together only while about 100 groups are left for the SMs
  need(a.group == 1 || a.ntx * a.nty * a.ntz >= 100, "too few groups", a);
  need(a.group == 4 || tiles_of(a) < 8000 || 8 * cout > 512 || a.H < 4 || a.W < 2, "tiles apart", a);
}

int main() {
  const int sizes[] = {1, 2, 3, 4, 5, 7, 8, 16, 24, 31, 64, 100, 127, 128, 129, 136, 255, 256, 257, 511, 512, 513, 768, 1000, 1024};
  for (int W : sizes)
    for (int H : sizes)
      for (int D : sizes)
        for (int ch : {16, 32, 48, 64, 96, 128}) {
          check(W, H, D, 16, ch);
          check(W, H, D, ch, ch);
          check(W, H, D, 192, ch);
          check(W, H, D, ch, 192);
        }
  std::printf(fails ? "%d failures\n" : "ok\n", fails);
  return fails != 0;
}
