// The grouped tracker (track_group.cuh: 8 or 16 lanes per keypoint, staged
// windows, groups at levels of their own) run on the host against the
// per-warp tracker (track_dev.cuh), bit for bit (test infrastructure): two
// images whose levels sit between poisoned gaps, keypoints anywhere (near and
// outside the edges, far or non-finite starts), tracks of different depths,
// with and without the backward pass, and tracks that are run again as a
// plain track. Shared memory is a heap buffer of exactly the warp's size.
// argv[1]: lanes per keypoint; argv[2]: width; argv[3]: height; argv[4]:
// levels; argv[5]: level-0 pitch; argv[6]: seed.
#include "blockemu.h"
// asynchronous copies, done at once
inline void __pipeline_memcpy_async(void* d, const void* s, size_t n) { memcpy(d, s, n); }
inline void __pipeline_commit() {}
inline void __pipeline_wait_prior(int) {}
// packed FP32 instructions, lane by lane
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) {
  return float2{__fmaf_rn(a.x, b.x, c.x), __fmaf_rn(a.y, b.y, c.y)};
}
inline float2 __fadd2_rn(float2 a, float2 b) { return float2{a.x + b.x, a.y + b.y}; }
inline float2 __fmul2_rn(float2 a, float2 b) { return float2{a.x * b.x, a.y * b.y}; }
inline float2 __fadd2_rd(float2 a, float2 b) {
  return float2{__fadd_rd(a.x, b.x), __fadd_rd(a.y, b.y)};
}
#include "track_group.cuh"

#include <sanitizer/asan_interface.h>

#include <random>
#include <vector>

using namespace vio;

namespace {
constexpr long long kGap = 64;   // poisoned bytes around every level

struct Item {
  trk::Task task, again;
  bool empty, retry;
};
struct HostSource {
  const Geom& g;
  const Batch& b;
  const std::vector<Item>& items;
  std::vector<trk::TrackResult>& out;
  struct Ref {
    long long i;
    bool second;
  };
  long long total() const { return (long long)items.size(); }
  bool fetch(long long i, bool lead, Ref& ref, trk::Task& K) const {
    ref = Ref{i, false};
    if (items[i].empty) {
      if (lead) out[i].status = VIO_TRACK_EMPTY;
      return false;
    }
    K = items[i].task;
    return true;
  }
  void levels(const Ref&, bool back, int l, trk::Lv& S, trk::Lv& D) const {
    S = trk::get_lv(g, b, back ? 1 : 0, l);
    D = trk::get_lv(g, b, back ? 0 : 1, l);
  }
  bool finish(Ref& ref, bool lead, const trk::TrackResult& R, trk::Task& K) const {
    if (items[ref.i].retry && !ref.second) {
      ref.second = true;
      K = items[ref.i].again;
      return false;
    }
    if (lead) out[ref.i] = R;
    return true;
  }
};

template <int LPK>
void run(const HostSource& src) {
  std::vector<uint8_t> smem(trk::kWarpBytes<LPK> + 16, 0xA5);
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem.data() + 15) & ~(uintptr_t)15);
  for (int w = 0; w < 2; ++w)
    emu_run_block(32, [&] { trk::run_tracks<LPK>(src, w, 2, sm); }, EmuDim{0, 0, 0});
}
}  // namespace

int main(int argc, char** argv) {
  if (argc < 7) return 2;
  const int lpk = atoi(argv[1]), w = atoi(argv[2]), h = atoi(argv[3]), L = atoi(argv[4]);
  std::mt19937 rng(atoi(argv[6]));
  auto uni = [&](float a, float b) { return a + (b - a) * (float)(rng() % 100001) / 100000.f; };
  Geom g{};
  g.n_levels = L;
  long long up = kGap;
  for (int l = 0; l < L; ++l) {
    g.w[l] = w >> l;
    g.h[l] = h >> l;
    g.pitch[l] = l == 0 ? atoi(argv[5]) : l % 2 ? (g.w[l] + 127) & ~127 : g.w[l];
    if (l > 0) {
      g.off[l] = up;
      up = ((up + (long long)g.pitch[l] * g.h[l] + 15) & ~15LL) + kGap;
    }
  }
  const long long s0 = (((long long)g.pitch[0] * g.h[0]) + 15) & ~15LL;
  std::vector<uint8_t> l0((size_t)(kGap + 2 * (s0 + kGap))), ub((size_t)(2 * up + kGap));
  Batch b{l0.data() + kGap, s0 + kGap, ub.data(), up, 2};
  ASAN_POISON_MEMORY_REGION(l0.data(), l0.size());
  ASAN_POISON_MEMORY_REGION(ub.data(), ub.size());
  // a smooth texture, shifted and turned between the images
  const float ph[6] = {uni(0, 6), uni(0, 6), uni(0, 6), uni(0, 6), uni(0, 6), uni(0, 6)};
  const float sx = uni(-3, 3), sy = uni(-3, 3), th = uni(-0.03f, 0.03f);
  for (int img = 0; img < 2; ++img)
    for (int l = 0; l < L; ++l) {
      uint8_t* d = l == 0 ? const_cast<uint8_t*>(b.l0) + img * b.l0_stride
                          : b.upper + img * b.upper_stride + g.off[l];
      ASAN_UNPOISON_MEMORY_REGION(d, (size_t)g.pitch[l] * g.h[l]);
      const float sc = (float)(1 << l);
      for (int y = 0; y < g.h[l]; ++y)
        for (int x = 0; x < g.pitch[l]; ++x) {
          float X = x * sc, Y = y * sc;
          if (img) {
            const float xx = X - sx, yy = Y - sy;
            X = xx + th * yy;
            Y = yy - th * xx;
          }
          float v = 0;
          for (int k = 0; k < 6; ++k)
            v += std::sin((0.05f + 0.06f * k) * ((k & 1) ? X : 0.7f * X + Y) + 0.09f * k * Y + ph[k]);
          d[(size_t)y * g.pitch[l] + x] =
              x < g.w[l] ? (uint8_t)std::min(255.f, std::max(0.f, 128 + 30 * v)) : 0x5A;
        }
    }
  const float nan = std::nanf("");
  std::vector<Item> items(45);
  for (size_t i = 0; i < items.size(); ++i) {
    Item& I = items[i];
    I.empty = rng() % 9 == 0;
    I.retry = rng() % 4 == 0;
    trk::Task& K = I.task;
    K = trk::Task{};
    K.px = uni(-4.f, (float)w + 4);
    K.py = uni(-4.f, (float)h + 4);
    if (i % 5 == 0) K.px = uni(7.5f, 12.f);
    if (i % 7 == 0) K.py = (float)h - uni(8.f, 12.f);
    K.has_init = rng() % 2;
    K.ix = K.px + uni(-4, 4);
    K.iy = K.py + uni(-4, 4);
    K.ith = uni(-0.1f, 0.1f);
    if (i == 11) { K.has_init = true; K.ix = 1e30f; }
    if (i == 12) { K.has_init = true; K.iy = nan; }
    if (i == 13) { K.has_init = true; K.ix = -3e9f; K.ith = 2.f; }
    if (i == 14) K.px = nan;
    if (i == 15) { K.has_init = true; K.ith = 2.9f; }
    K.top = (int)(rng() % L);
    K.iters = i % 11 == 0 ? 0 : 3 + (int)(rng() % 3);
    K.fb = rng() % 4 != 0;
    K.fb_max = 0.2f;
    I.again = K;
    I.again.has_init = false;
    I.again.top = L - 1;
  }
  std::vector<trk::TrackResult> got(items.size()), ref(items.size());
  for (auto& r : got) r = trk::TrackResult{-1, false, 0, 0, 0, 0, 0};
  const HostSource src{g, b, items, got};
  if (lpk == 4) run<4>(src);
  else if (lpk == 8) run<8>(src);
  else run<16>(src);
  for (size_t i = 0; i < items.size(); ++i) {
    if (items[i].empty) continue;
    const trk::Task& K = items[i].retry ? items[i].again : items[i].task;
    emu_run_block(32, [&] {
      trk::Pos tf{};
      float thf = 0, dist = 0, last = 0;
      bool have = false;
      const TrackCfg cfg{K.iters, K.fb, K.fb_max, -1};
      const int st = trk::track_fb(g, b, 0, b, 1, K.px, K.py, K.has_init, K.ix, K.iy, K.ith, cfg,
                                   K.top, threadIdx.x & 31, tf, thf, have, dist, last);
      if ((threadIdx.x & 31) == 0)
        ref[i] = trk::TrackResult{st, have, have ? (float)tf.ax + tf.dx : nan,
                                  have ? (float)tf.ay + tf.dy : nan, have ? thf : nan, dist,
                                  have ? last : nan};
    }, EmuDim{0, 0, 0});
  }
  int fails = 0, ok = 0, n_status[16] = {0};
  for (size_t i = 0; i < items.size(); ++i) {
    const auto &a = got[i], &c = ref[i];
    if (items[i].empty) {
      fails += a.status != VIO_TRACK_EMPTY;
      continue;
    }
    auto same = [](float x, float y) { return memcmp(&x, &y, 4) == 0 || (x != x && y != y); };
    const bool eq = a.status == c.status && a.have == c.have && same(a.x, c.x) && same(a.y, c.y) &&
                    same(a.th, c.th) && same(a.dist, c.dist) && same(a.last, c.last);
    if (!eq) {
      printf("item %zu: status %d / %d, x %.9g / %.9g, y %.9g / %.9g, th %.9g / %.9g, fb %.9g / %.9g, last %.9g / %.9g\n",
             i, a.status, c.status, a.x, c.x, a.y, c.y, a.th, c.th, a.dist, c.dist, a.last, c.last);
      ++fails;
    }
    ok += c.status == VIO_TRACK_OK;
    ++n_status[c.status & 15];
  }
  printf("items %zu ok %d oob-template %d oob-warp %d fb %d FAILS %d\n", items.size(), ok, n_status[1],
         n_status[2], n_status[5], fails);
  return fails != 0;
}
