// The half-row loads of the flow network's input extraction (net::half_row) on
// the host (test infrastructure): levels of random bytes between ASan-poisoned
// gaps, at every base offset and pitch remainder of a word, halves of rows
// inside, across and far beyond every edge, against plain byte reads.
#include "blockemu.h"
#include "initnet_dev.cuh"

#include <sanitizer/asan_interface.h>

#include <climits>
#include <random>
#include <vector>

using namespace vio;

int main() {
  std::mt19937 rng(3);
  long long n = 0, fails = 0;
  for (int w : {1, 3, 8, 17, 32, 67})
    for (int pad : {0, 1, 2, 5, (64 - w % 64) % 64})
      for (int base : {0, 1, 2, 3}) {
        const int h = 5, pitch = w + pad;
        std::vector<uint8_t> buf((size_t)(256 + pitch * h + 256));
        uint8_t* p = reinterpret_cast<uint8_t*>(((uintptr_t)buf.data() + 127) & ~(uintptr_t)63) + base;
        ASAN_POISON_MEMORY_REGION(buf.data(), buf.size());
        ASAN_UNPOISON_MEMORY_REGION(p, (size_t)pitch * h);
        for (int i = 0; i < pitch * h; ++i) p[i] = (uint8_t)rng();
        std::vector<int> xs = {INT_MIN, INT_MIN + 8, -1000000000, INT_MAX - 8, INT_MAX, 1000000000};
        for (int x = -20; x < w + 20; ++x) xs.push_back(x);
        for (int cy : {INT_MIN, -1, 0, 2, 4, 5, INT_MAX})
          for (int cx : xs) {
            unsigned b[2];
            net::half_row(p, w, h, pitch, cx, cy, b);
            for (int k = 0; k < 8; ++k, ++n) {
              const long long x = (long long)cx + k;
              const unsigned ref =
                  cy >= 0 && cy < h && x >= 0 && x < w ? p[(size_t)cy * pitch + x] : 0x80u;
              fails += ((b[k >> 2] >> (8 * (k & 3))) & 0xffu) != ref;
            }
          }
        ASAN_UNPOISON_MEMORY_REGION(buf.data(), buf.size());
      }
  printf("pixels %lld FAILS %lld\n", n, fails);
  return fails != 0;
}
