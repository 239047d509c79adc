// launch_pd_tma on two devices of one process (fake_cudart.c): each needs its
// own opt-in to the kernel's shared memory, and as many CTAs as it has SMs.
#include <cstdio>

#include "fs_kernels.h"

extern "C" int fake_device;
extern "C" unsigned fake_grid;

int main() {
  fs::LevelView L{};
  L.W = L.H = L.P = 2048;
  fs::PDState a{}, b{};
  fs::PDParams pp{50.f, 0.01f, 1.f};
  static fs::PdTmaMaps maps{};
  int bad = 0;
  for (int st : {fs::ST_F32, fs::ST_F16, fs::ST_BF16})
    for (int dev : {0, 1, 0}) {
      L.st = st;
      fake_device = dev;
      const cudaError_t e =
          fs::launch_pd_tma(L, a, b, pp, 7, 7, 0, maps, nullptr, 1000000, 0, nullptr);
      const unsigned want = dev == 0 ? 152 : 80;
      if (e != cudaSuccess || fake_grid != want) {
        std::printf("storage %d, device %d: error %d, %u CTAs for %u SMs\n", st, dev, (int)e,
                    fake_grid, want);
        bad = 1;
      }
    }
  return bad;
}
