// The patch tracker by groups of lanes: a warp tracks 32 / LPK keypoints at a
// time, LPK lanes (4, 8 or 16) each; the kernels use 4 (kGroupLanes), the host
// check 16 too. Same arithmetic as the per-warp form of
// track_dev.cuh, bit for bit: a lane that owns the pattern points i, i + LPK,
// i + 2 LPK, ... adds locally what the per-warp form's first reduction rounds
// add across lanes, in the same order, so only the last rounds remain as
// shuffles.
//
// What bounds it, and why this split. With one keypoint per warp a
// Gauss-Newton step is about 140 instructions, half of them the reduction and
// the scalar update that every lane repeats, and its eight byte loads take
// 2.7 L1 wavefronts each (32 lanes touch five rows): a launch that fills the
// GPU ran at 82% of the L1's wavefront rate. Here the update is shared by eight
// keypoints, two samples of a lane go through each packed FP32 instruction,
// and the texels come from shared memory: per level the template's 18-row
// region and a 24-row window of the target are copied asynchronously. The
// window has 2 to 5 pixels of play; a step whose samples might leave it copies
// it again around the current position. 58 instructions a keypoint and step.
// What is left are dependent instructions at three warps per scheduler (162
// registers a thread) and the instruction cache.
//
// Measured (640 x 480, five levels, five steps, forward and backward, us;
// keypoints: one per warp / 4 lanes / 8 lanes each):
//   2400: 38 / 57 / 43    4200: 57 / 57    4800: 68 / 57 / 51
//   9600: 112 / 70 / 78   14400: 158 / 96 / 129    24000: 246 / 185 / 234
// (one per warp: 2400 and 4200 with the packed step of track_dev.cuh, the
// others before it). A group of four lanes takes about 55 us however few
// keypoints there are, so a launch of fewer than 28 keypoints per SM keeps a
// warp each.
// Level-0 rows that start at any byte (641 x 479; one per warp / 4 lanes, and in
// brackets 4 lanes copying such rows byte by byte, as they first did):
//   9280: 108 / 79 (102)    23200: 236 / 216 (288)
//   level 0 alone: 9280: 34 / 27 (52)    23200: 70 / 62 (105)
//   753 x 481, 6216: 78 / 76 (106)    level 0 alone: 22.9 / 24.0 (49.6)
// so such launches keep a warp each below 48 keypoints per SM.
//
// A group is a small state machine (keypoint, direction, level) that advances
// by one level per turn of the warp's loop, independently of the warp's other
// groups; a group whose keypoint is done takes the next one of its warp's.
// Failed tracks, skipped levels and tracks from a learned start (which cover
// fewer levels) therefore leave few lanes idle.
#pragma once
#ifdef __CUDACC__
#include <cuda_pipeline_primitives.h>
#endif

#include "track_dev.cuh"

namespace vio {
namespace trk {

constexpr unsigned kFull = 0xffffffffu;
// copied regions of one keypoint: rows of 32 bytes from a multiple of 8, 40 bytes
// apart (a row's samples, and the groups', fall on different banks)
constexpr int kPitch = 40;
constexpr int kTplRows = 18, kTplCols = 24;   // columns from a multiple of 4 on
constexpr int kWinRows = 24, kWinCols = 28;
constexpr int kTplBytes = kTplRows * kPitch;
constexpr int kGroupBytes = kTplBytes + kWinRows * kPitch;
static_assert(kWinCols + 4 <= 32 && kTplCols + 4 <= 32 && kPitch >= 32 && kGroupBytes % 16 == 0 &&
                  kGroupBytes / 4 % 32 == 4,
              "a region's columns fit its rows, groups start four banks apart");
// > radius of the pattern (7.616), with room for rounding: 1000 steps lengthen (cs,
// sn) by 3e-4 at most, from below sqrt(kMaxNorm2) at a level's start
constexpr float kReach = 7.63f;
constexpr float kMaxNorm2 = 1.003f;

// Lane gl of a group owns the pattern points gl + LPK s, slot s < 2 NP, in
// pairs of slots (2 j, 2 j + 1). A slot without a point has weight 0 (and
// K = 0) and stands at the pattern's centre; only the last pair has any.
template <int LPK>
struct GroupPts {
  static constexpr int NP = (kNP + 2 * LPK - 1) / (2 * LPK);   // 7, 4, 2 pairs
  float2 u[NP], v[NP];
  float2 wl;
  // the pattern's 12 hull points (+-3, +-7), (+-5, +-5), (+-7, +-3), shared out
  // over the lanes: a sample position is monotone in u and in v (each rounding
  // is), so every sample lies inside the level iff these do
  static constexpr int NHULL = (12 + LPK - 1) / LPK;
  __device__ __forceinline__ explicit GroupPts(int gl) {
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      float c[2][2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int i = gl + LPK * (2 * j + e);
        int iu = 0, iv = 0;
        if (i < kNP) point_of(i, iu, iv);
        c[e][0] = (float)iu;
        c[e][1] = (float)iv;
      }
      u[j] = make_float2(c[0][0], c[1][0]);
      v[j] = make_float2(c[0][1], c[1][1]);
    }
    wl = make_float2(gl + LPK * (2 * NP - 2) < kNP ? 1.f : 0.f,
                     gl + LPK * (2 * NP - 1) < kNP ? 1.f : 0.f);
  }
};

// Shared memory of a warp: its groups' regions.
template <int LPK>
constexpr int kWarpBytes = 32 / LPK * kGroupBytes;

// Sums over a lane's slots: get(j) is pair j's value, add(j, t) = pair j's value
// added to t (the per-warp form's second point of a lane). The first
// reduction rounds of the per-warp form follow, in its order: with 16 lanes a
// pair's two halves; with 8, pairs (0, 2) + (1, 3), then the halves; with 4,
// (0, 4) + (2, 6) and (1, 5) + (3), these two, then the halves.
template <int LPK, class Get, class Add>
__device__ __forceinline__ float fold(Get get, Add add) {
  float2 t;
  if (LPK == 16) {
    t = add(1, get(0));
  } else if (LPK == 8) {
    t = add2(add(2, get(0)), add(3, get(1)));
  } else {
    const float2 a = add2(add(4, get(0)), add(6, get(2)));
    t = add2(a, add2(add(5, get(1)), get(3)));
  }
  return t.x + t.y;
}

// The remaining rounds across the group's lanes (every lane gets the total).
template <int LPK, int N>
__device__ __forceinline__ void group_sum(float (&v)[N]) {
  static_assert(N % 2 == 0, "pairs of values");
#pragma unroll
  for (int o = LPK / 2; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const float a = __shfl_xor_sync(kFull, v[i], o), b = __shfl_xor_sync(kFull, v[i + 1], o);
      const float2 t = add2(make_float2(v[i], v[i + 1]), make_float2(a, b));
      v[i] = t.x;
      v[i + 1] = t.y;
    }
}

// Copies pixels [x0, x0 + COLS) (x0 a multiple of 4) of rows y0 .. y0 + ROWS -
// 1 of a level into shared memory, row r's pixel x at dst + 40 r + x - (x0 &
// ~7), by the LPK lanes of a group. Rows outside the level repeat its edge;
// pixels outside it are left as they are (no sample that counts uses them).
// Completed by __pipeline_wait_prior(0) of the lanes that called it and a
// __syncwarp. Rows that start on 8-byte boundaries (upper levels always do) go
// in 8-byte copies.
template <int LPK, int ROWS, int COLS>
__device__ __forceinline__ void copy_region(uint8_t* dst, const Lv& L, int x0, int y0, int gl) {
  const unsigned al = (unsigned)(reinterpret_cast<uintptr_t>(L.p) | (uintptr_t)L.pitch);
  if ((al & 7) == 0) {
    // a chunk that starts inside the level ends inside the row's pitch
    constexpr int RPI = LPK / 4;
    const int c = gl & 3, x = (x0 & ~7) + 8 * c;
    if (x >= 0 && x < L.w && x < x0 + COLS) {
      dst += 8 * c;
      const uint8_t* src = L.p + x;
#pragma unroll 6
      for (int r = gl >> 2; r < ROWS; r += RPI) {
        const int y = min(max(y0 + r, 0), L.h - 1);
        __pipeline_memcpy_async(dst + r * kPitch, src + (unsigned)y * (unsigned)L.pitch, 8);
      }
    }
    return;
  }
  if ((al & 3) == 0) {
    // a word at a time
#pragma unroll 1
    for (int s = gl; s < COLS / 4; s += LPK) {
      const int x = x0 + 4 * s;
      if (x < 0 || x >= L.w) continue;
      uint8_t* d = dst + (x0 & 7) + 4 * s;
#pragma unroll 6
      for (int r = 0; r < ROWS; ++r) {
        const int y = min(max(y0 + r, 0), L.h - 1);
        __pipeline_memcpy_async(d + r * kPitch,
                                L.p + ((unsigned)y * (unsigned)L.pitch + (unsigned)x), 4);
      }
    }
    return;
  }
  // rows that start at any byte: a row per lane, aligned words shifted into
  // place; bytes where such a word might lie outside the image
  constexpr int NW = COLS / 4;
  const uintptr_t begin = reinterpret_cast<uintptr_t>(L.p);
  const uintptr_t end = begin + (unsigned)(L.h - 1) * (unsigned)L.pitch + (unsigned)L.w;
#pragma unroll 3
  for (int r = gl; r < ROWS; r += LPK) {
    const int y = min(max(y0 + r, 0), L.h - 1);
    const uint8_t* row = L.p + (unsigned)y * (unsigned)L.pitch;
    uint8_t* d = dst + (r * kPitch + (x0 & 7));
    const uintptr_t p = reinterpret_cast<uintptr_t>(row) + (intptr_t)x0, a = p & ~(uintptr_t)3;
    if (a >= begin && a + 4 * (NW + 1) <= end) {
      const unsigned* q = reinterpret_cast<const unsigned*>(a);
      const int sh = 8 * (int)(p & 3);
      unsigned w[NW + 1];
#pragma unroll
      for (int k = 0; k <= NW; ++k) w[k] = __ldg(q + k);
#pragma unroll
      for (int k = 0; k < NW; ++k)
        *reinterpret_cast<unsigned*>(d + 4 * k) = __funnelshift_r(w[k], w[k + 1], sh);
    } else {
#pragma unroll 1
      for (int x = max(x0, 0); x < min(x0 + COLS, L.w); ++x) d[x - x0] = __ldg(row + x);
    }
  }
}

template <int LPK>
struct GroupTpl {
  float2 K[GroupPts<LPK>::NP][3];
  float c0, c1, c2, S;
};

// build_template of track_dev.cuh from the copied region `st` (columns from
// (Qx - 8) & ~3, rows from Qy - 8). Returns a VIO_TRACK_* status, uniform in
// the group. Every lane of the warp calls it.
template <int LPK>
__device__ __forceinline__ int group_template(const uint8_t* st, int Qx, float fx, float fy,
                                              const GroupPts<LPK>& P, GroupTpl<LPK>& T) {
  constexpr int NP = GroupPts<LPK>::NP;
  const float2 w00 = both(__fmul_rn(1.f - fx, 1.f - fy)), w10 = both(__fmul_rn(fx, 1.f - fy));
  const float2 w01 = both(__fmul_rn(1.f - fx, fy)), w11 = both(__fmul_rn(fx, fy));
  // pixel Q - 1 + (u, v): v + 7 rows down, u + 7 columns right of Qx - 8
  const uint8_t* base = st + (7 * kPitch + 7 + ((Qx - 8) & 7));
  float2 I[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    float t[2][4][4];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float u = e ? P.u[j].y : P.u[j].x, v = e ? P.v[j].y : P.v[j].x;
      const uint8_t* a =
          base + (__float_as_int(__fmaf_rn(v, (float)kPitch, u + kFloorBias)) - kFloorBiasBits);
      const bool some = LPK * (2 * j + e) < kNP;   // a slot that no lane has needs no pixels
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          t[e][r][c] = !some || ((r == 0 || r == 3) && (c == 0 || c == 3))
                           ? 0.f
                           : (float)a[r * kPitch + c];
    }
    auto bl = [&](int r, int c) {   // the interpolant with (r, c) its first pixel
      auto px = [&](int y, int x) { return make_float2(t[0][y][x], t[1][y][x]); };
      return fma2(w11, px(r + 1, c + 1),
                  fma2(w01, px(r + 1, c), fma2(w10, px(r, c + 1), mul2(w00, px(r, c)))));
    };
    float2 s = bl(1, 1);
    float2 gx = mul2(both(0.5f), sub2(bl(1, 2), bl(1, 0)));
    float2 gy = mul2(both(0.5f), sub2(bl(2, 1), bl(0, 1)));
    if (j == NP - 1) {   // slots without a point add nothing
      const bool o0 = P.wl.x != 0.f, o1 = P.wl.y != 0.f;
      s = make_float2(o0 ? s.x : 0.f, o1 ? s.y : 0.f);
      gx = make_float2(o0 ? gx.x : 0.f, o1 ? gx.y : 0.f);
      gy = make_float2(o0 ? gy.x : 0.f, o1 ? gy.y : 0.f);
    }
    I[j] = s;
    T.K[j][0] = gx;
    T.K[j][1] = gy;
    T.K[j][2] = fma2(make_float2(-gx.x, -gx.y), P.v[j], mul2(gy, P.u[j]));
  }
  float acc[10];
  acc[0] = fold<LPK>([&](int j) { return I[j]; },
                     [&](int j, float2 t) { return add2(t, I[j]); });
  auto products = [&](int i, int k) {   // k = 3: the intensities
    auto b = [&](int j) { return k < 3 ? T.K[j][k < 3 ? k : 0] : I[j]; };
    return fold<LPK>([&](int j) { return fma2(T.K[j][i], b(j), both(0.f)); },
                     [&](int j, float2 t) { return fma2(T.K[j][i], b(j), t); });
  };
  acc[1] = products(0, 0);
  acc[2] = products(0, 1);
  acc[3] = products(0, 2);
  acc[4] = products(1, 1);
  acc[5] = products(1, 2);
  acc[6] = products(2, 2);
  acc[7] = products(0, 3);
  acc[8] = products(1, 3);
  acc[9] = products(2, 3);
  group_sum<LPK>(acc);
  T.S = acc[0];
  if (!(acc[0] > 0.f)) return VIO_TRACK_ZERO_MEAN;
  const float eps = __fmul_rn(1e-9f, acc[1] + acc[4] + acc[6]);
  Chol C;
  if (!(acc[1] > eps)) return VIO_TRACK_DEGENERATE_H;
  C.i00 = rsqrtf(acc[1]);
  C.l10 = __fmul_rn(acc[2], C.i00);
  C.l20 = __fmul_rn(acc[3], C.i00);
  const float d1 = __fmaf_rn(-C.l10, C.l10, acc[4]);
  if (!(d1 > eps)) return VIO_TRACK_DEGENERATE_H;
  C.i11 = rsqrtf(d1);
  C.l21 = __fmul_rn(__fmaf_rn(-C.l20, C.l10, acc[5]), C.i11);
  const float d2 = __fmaf_rn(-C.l21, C.l21, __fmaf_rn(-C.l20, C.l20, acc[6]));
  if (!(d2 > eps)) return VIO_TRACK_DEGENERATE_H;
  C.i22 = rsqrtf(d2);
  C.solve(acc[7], acc[8], acc[9], T.c0, T.c1, T.c2);
  // K = the solves of Chol::solve, two points at a time
  const float2 i00 = both(C.i00), i11 = both(C.i11), i22 = both(C.i22);
  const float2 l10 = both(-C.l10), l20 = both(-C.l20), l21 = both(-C.l21);
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const float2 y0 = mul2(T.K[j][0], i00);
    const float2 y1 = mul2(fma2(l10, y0, T.K[j][1]), i11);
    const float2 y2 = mul2(fma2(l21, y1, fma2(l20, y0, T.K[j][2])), i22);
    T.K[j][2] = mul2(y2, i22);
    T.K[j][1] = mul2(fma2(l21, T.K[j][2], y1), i11);
    T.K[j][0] = mul2(fma2(l20, T.K[j][2], fma2(l10, T.K[j][1], y0)), i00);
  }
  return VIO_TRACK_OK;
}

// The copied window of the target: pixels [x0, x0 + kWinCols) x [y0, y0 +
// kWinRows), and the range of the warp's offset for which every sample lies
// inside it and inside the level.
struct Win {
  int x0, y0;
  float lx, hx, ly, hy;
  __device__ __forceinline__ void place(const Pos& t) {
    x0 = (t.ax + (int)floorf(t.dx) - 10) & ~3;
    y0 = t.ay + (int)floorf(t.dy) - 11;
  }
  // a window that touches the level (a start may lie anywhere)
  __device__ __forceinline__ bool near(const Lv& D) const {
    return x0 > -64 && x0 < D.w && y0 > -64 && y0 < D.h;
  }
  // samples take pixels floor and floor + 1
  __device__ __forceinline__ bool holds(const Pos& t) const {
    const float x = (float)(x0 - t.ax), y = (float)(y0 - t.ay);
    return t.dx >= x + kReach && t.dx <= x + ((float)(kWinCols - 1) - kReach) &&
           t.dy >= y + kReach && t.dy <= y + ((float)(kWinRows - 1) - kReach);
  }
  __device__ __forceinline__ void range(const Pos& t, const Lv& D) {
    if (!near(D)) {
      lx = ly = 3.0e38f;
      hx = hy = -3.0e38f;
      return;
    }
    lx = (float)(max(x0, 0) - t.ax) + kReach;
    hx = (float)(min(x0 + kWinCols, D.w) - 1 - t.ax) - kReach;
    ly = (float)(max(y0, 0) - t.ay) + kReach;
    hy = (float)(min(y0 + kWinRows, D.h) - 1 - t.ay) - kReach;
  }
  __device__ __forceinline__ bool clear(const Pos& t) const {
    return t.dx >= lx && t.dx <= hx && t.dy >= ly && t.dy <= hy;
  }
};

// The four sums of a Gauss-Newton step over the lane's samples (r[0] the
// intensities, r[1..3] the products with K), folded. Every sample lies in the
// window.
template <int LPK>
__device__ __forceinline__ void group_samples(const uint8_t* win, const Win& N,
                                              const GroupTpl<LPK>& T, const GroupPts<LPK>& P,
                                              const Warp& W, float (&r)[4]) {
  constexpr int NP = GroupPts<LPK>::NP;
  // offset of the pixel (floor x, floor y): the floors sit in the low bits of
  // the biased floats (gn_step), the biases cancel modulo 2^32
  const unsigned wbase = (unsigned)(W.t.ax - (N.x0 & ~7)) +
                         (unsigned)(W.t.ay - N.y0) * (unsigned)kPitch -
                         (unsigned)kFloorBiasBits * (unsigned)(kPitch + 1);
  const float2 cs = both(W.cs), sn = both(W.sn), ns = both(-W.sn);
  const float2 dx = both(W.t.dx), dy = both(W.t.dy), bias = both(kFloorBias);
  const float2 nbias = both(-kFloorBias);
  float2 I[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const float2 vx = fma2(cs, P.u[j], fma2(ns, P.v[j], dx));
    const float2 vy = fma2(sn, P.u[j], fma2(cs, P.v[j], dy));
    const float2 tx = add2_rd(vx, bias), ty = add2_rd(vy, bias);
    const float2 fx = sub2(vx, add2(tx, nbias)), fy = sub2(vy, add2(ty, nbias));
    const uint8_t* p = win + (__float_as_uint(ty.x) * (unsigned)kPitch +
                              (__float_as_uint(tx.x) + wbase));
    const uint8_t* q = win + (__float_as_uint(ty.y) * (unsigned)kPitch +
                              (__float_as_uint(tx.y) + wbase));
    // a pair's second slot that no lane has needs no pixels (weight 0)
    const bool two = LPK * (2 * j + 1) < kNP;
    const float2 a = make_float2((float)p[0], two ? (float)q[0] : 0.f);
    const float2 b = make_float2((float)p[1], two ? (float)q[1] : 0.f);
    const float2 c = make_float2((float)p[kPitch], two ? (float)q[kPitch] : 0.f);
    const float2 d = make_float2((float)p[kPitch + 1], two ? (float)q[kPitch + 1] : 0.f);
    const float2 top = fma2(fx, sub2(b, a), a), bot = fma2(fx, sub2(d, c), c);
    I[j] = fma2(fy, sub2(bot, top), top);
  }
  r[0] = fold<LPK>([&](int j) { return I[j]; },
                   [&](int j, float2 t) {
                     return j == NP - 1 ? fma2(P.wl, I[j], t) : add2(t, I[j]);
                   });
#pragma unroll
  for (int k = 0; k < 3; ++k)
    r[k + 1] = fold<LPK>([&](int j) { return fma2(T.K[j][k], I[j], both(0.f)); },
                         [&](int j, float2 t) { return fma2(T.K[j][k], I[j], t); });
}

// Whether the lane's hull points' samples lie inside the level.
template <int LPK>
__device__ __forceinline__ bool hull_inside(const Lv& D, int gl, const Warp& W) {
  const unsigned xmax = (unsigned)(D.w - 2), ymax = (unsigned)(D.h - 2);
  bool ok = true;
#pragma unroll
  for (int j = 0; j < GroupPts<LPK>::NHULL; ++j) {
    const int i = gl + LPK * j, m = i < 12 ? i >> 2 : 0;
    const float hu = 3.f + 2.f * m, hv = 7.f - 2.f * m;
    const float u = (i & 1) ? -hu : hu, v = (i & 2) ? -hv : hv;
    const float vx = __fmaf_rn(W.cs, u, __fmaf_rn(-W.sn, v, W.t.dx));
    const float vy = __fmaf_rn(W.sn, u, __fmaf_rn(W.cs, v, W.t.dy));
    const int ix = W.t.ax + (__float_as_int(__fadd_rd(vx, kFloorBias)) - kFloorBiasBits);
    const int iy = W.t.ay + (__float_as_int(__fadd_rd(vy, kFloorBias)) - kFloorBiasBits);
    ok = ok && (unsigned)ix <= xmax && (unsigned)iy <= ymax;
  }
  return ok;
}

// The update of a Gauss-Newton step from its four totals (gn_step of
// track_dev.cuh after its reduction).
template <int LPK>
__device__ __forceinline__ int group_update(const GroupTpl<LPK>& T, const float (&r)[4], Warp& W,
                                            float& moved) {
  const float q = __fdividef(T.S, r[0]);
  const float d0 = __fmaf_rn(-q, r[1], T.c0);
  const float d1 = __fmaf_rn(-q, r[2], T.c1);
  const float d2 = __fmaf_rn(-q, r[3], T.c2);
  const float s01 = fabsf(d0) + fabsf(d1);
  if (!(r[0] < 1e29f && r[0] > 0.f && s01 + fabsf(d2) < 3.0e38f))
    return r[0] >= 1e29f ? VIO_TRACK_OOB_WARP
                         : !(r[0] > 0.f) ? VIO_TRACK_ZERO_MEAN : VIO_TRACK_NAN;
  moved = __fmaf_rn(kPatRadius, fabsf(d2), s01);
  float cd, sd, a, b;
  small_rot(d2, cd, sd, a, b);
  const float vx = __fmaf_rn(-b, d1, __fmul_rn(a, d0));
  const float vy = __fmaf_rn(a, d1, __fmul_rn(b, d0));
  W.t.dx = __fmaf_rn(W.cs, vx, __fmaf_rn(-W.sn, vy, W.t.dx));
  W.t.dy = __fmaf_rn(W.sn, vx, __fmaf_rn(W.cs, vy, W.t.dy));
  const float cs = __fmaf_rn(-W.sn, sd, __fmul_rn(W.cs, cd));
  const float sn = __fmaf_rn(W.cs, sd, __fmul_rn(W.sn, cd));
  W.cs = cs;
  W.sn = sn;
  W.th += d2;
  return VIO_TRACK_OK;
}

// A keypoint's track as handed over by a source: position, start, levels and
// checks; and its result.
struct Task {
  float px, py, ix, iy, ith;   // keypoint; start (used when has_init)
  bool has_init;
  int top, iters, fb;
  float fb_max;
};
struct TrackResult {
  int status;
  bool have;        // a forward result exists
  float x, y, th, dist, last;
};

// Runs the tracks of a source on this warp: items first, first + stride, ...
// below src.total(). smem: the warp's kWarpBytes<LPK>, 16-byte aligned. Src:
//   Ref                            what a group keeps of its item
//   fetch(item, lead, ref, task)   false: nothing to track (outputs written by
//                                  the group's lane with `lead`)
//   levels(ref, back, l, S, D)     level l of the template's and the target's
//                                  image (forward or backward pass)
//   finish(ref, lead, res, task)   false: track the keypoint again as `task`
template <int LPK, class Src>
__device__ __forceinline__ void run_tracks(const Src& src, long long first, long long stride,
                                           uint8_t* smem) {
  constexpr int NG = 32 / LPK;
  const int lane = threadIdx.x & 31, gl = lane & (LPK - 1), gi = lane / LPK;
  const bool lead = gl == 0;
  uint8_t* tpl = smem + gi * kGroupBytes;
  uint8_t* win = tpl + kTplBytes;
  const GroupPts<LPK> P(gl);
  const long long total = src.total();
  long long next = first;
  typename Src::Ref ref;
  Task K{};
  Pos p{}, tf{};
  Warp W{};
  float thf = 0.f, last = 0.f;
  int l = 0;
  bool active = false, back = false;

  bool fresh = false;    // a direction starts at the next turn, from (t0, th0)
  Pos t0{};
  float th0 = 0.f;
  auto begin = [&] {     // the forward pass of the task
    p = split(K.px, K.py);
    back = false;
    last = 0.f;
    t0 = K.has_init ? split(K.ix, K.iy) : p;
    th0 = K.has_init ? K.ith : 0.f;
    fresh = true;
  };

  for (;;) {
    // idle groups take the warp's next items
    unsigned idle = __ballot_sync(kFull, lead && !active);
    while (idle != 0u && next < total) {
      if (!active) {
        const long long item = next + stride * __popc(idle & ((1u << (gi * LPK)) - 1u));
        if (item < total && src.fetch(item, lead, ref, K)) {
          active = true;
          begin();
        }
      }
      next += stride * __popc(idle);
      idle = __ballot_sync(kFull, lead && !active);
    }
    if (__popc(idle) == NG) break;

    // one level of every active group
    Lv S{}, D{};
    Win N{};
    int Qx = 0, Qy = 0, st = VIO_TRACK_OOB_TEMPLATE;
    float fx = 0.f, fy = 0.f, moved = 0.f;
    bool ok = false;        // the template's region lies inside the level
    __syncwarp();           // the previous level's reads are done
    if (fresh) {
      fresh = false;
      l = K.top;
      to_level1(t0.ax, t0.dx, l, W.t.ax, W.t.dx);
      to_level1(t0.ay, t0.dy, l, W.t.ay, W.t.dy);
      W.th = th0;
      float a, b;
      small_rot(th0, W.cs, W.sn, a, b);
    }
    if (active) {
      src.levels(ref, back, l, S, D);
      const Pos& q = back ? tf : p;
      to_level1(q.ax, q.dx, l, Qx, fx);
      to_level1(q.ay, q.dy, l, Qy, fy);
      ok = Qx - 7 >= 1 && Qx + 7 <= S.w - 3 && Qy - 7 >= 1 && Qy + 7 <= S.h - 3;
      if (ok) {
        N.place(W.t);
        N.range(W.t, D);
        copy_region<LPK, kTplRows, kTplCols>(tpl, S, (Qx - 8) & ~3, Qy - 8, gl);
        if (N.near(D)) copy_region<LPK, kWinRows, kWinCols>(win, D, N.x0, N.y0, gl);
      }
    }
    __pipeline_commit();
    __pipeline_wait_prior(0);
    __syncwarp();
    GroupTpl<LPK> T;
    const int ts = group_template<LPK>(tpl, Qx, fx, fy, P, T);
    if (ok) st = ts;
    bool run = ok && ts == VIO_TRACK_OK;   // steps are being taken
    const bool built = run;
    // the samples stay in the window because the pattern, turned by (cs, sn),
    // stays inside kReach: not with a start angle that is not finite, which has
    // no samples and no mean (as in gn_step). 24,000 keypoints take 0.4% longer
    // with this test.
    if (run && K.iters > 0 && !(__fmaf_rn(W.cs, W.cs, __fmul_rn(W.sn, W.sn)) < kMaxNorm2)) {
      st = VIO_TRACK_ZERO_MEAN;
      run = false;
    }
    const int iters = (int)__reduce_max_sync(kFull, run ? (unsigned)K.iters : 0u);
    for (int it = 0; it < iters; ++it) {
      bool step = run && it < K.iters;
      bool inside = true;
      if (__any_sync(kFull, step && !N.clear(W.t))) {
        // near the window's or the level's edge: copy the window again around
        // the position if it has left it, and test the hull points
        if (step && !N.holds(W.t)) {
          N.place(W.t);
          N.range(W.t, D);
          if (N.near(D) && N.holds(W.t)) {
            copy_region<LPK, kWinRows, kWinCols>(win, D, N.x0, N.y0, gl);
          } else {
            // every sample lies outside the level (a non-finite position has
            // no samples, and no mean)
            st = fabsf(W.t.dx) + fabsf(W.t.dy) < 3.0e38f ? VIO_TRACK_OOB_WARP
                                                         : VIO_TRACK_ZERO_MEAN;
            step = run = false;
          }
        }
        __pipeline_commit();
        __pipeline_wait_prior(0);
        __syncwarp();
        inside = hull_inside<LPK>(D, gl, W);
      }
      float r[4] = {0.f, 0.f, 0.f, 0.f};
      if (step) {
        group_samples<LPK>(win, N, T, P, W, r);
        if (!inside) r[0] += 1e30f;   // as in gn_step
      }
      __syncwarp();
      group_sum<LPK>(r);
      if (step) {
        st = group_update<LPK>(T, r, W, moved);
        run = st == VIO_TRACK_OK;
      }
    }
    if (active) {
      bool done = false;        // this direction has ended
      if (built && !run) {
        done = true;            // a step failed
      } else {
        if (built) {
          rebase(W.t);
          st = VIO_TRACK_OK;
        }
        if (l == 0) {
          done = true;          // st: OK, or the level-0 template's failure
        } else {
          W.t.ax *= 2;
          W.t.ay *= 2;
          W.t.dx *= 2.f;
          W.t.dy *= 2.f;
          rebase(W.t);
          --l;
        }
      }
      if (done) {
        TrackResult R;
        R.dist = __int_as_float(0x7fc00000);
        bool end = true;
        if (!back) {
          R.have = st == VIO_TRACK_OK;
          if (R.have) {
            tf = W.t;
            thf = W.th;
            last = moved;
            if (K.fb) {
              // backward: from the forward estimate's inverse
              back = true;
              t0 = p;
              th0 = -thf;
              fresh = true;
              end = false;
            }
          }
        } else {
          R.have = true;
          if (st == VIO_TRACK_OK) {
            const float ex = (float)(W.t.ax - p.ax) + (W.t.dx - p.dx);
            const float ey = (float)(W.t.ay - p.ay) + (W.t.dy - p.dy);
            R.dist = sqrtf(__fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
            if (R.dist > K.fb_max) st = VIO_TRACK_FB_FAIL;
          }
        }
        if (end) {
          const float qnan = __int_as_float(0x7fc00000);
          R.status = st;
          R.x = R.have ? (float)tf.ax + tf.dx : qnan;
          R.y = R.have ? (float)tf.ay + tf.dy : qnan;
          R.th = R.have ? thf : qnan;
          R.last = R.have ? last : qnan;
          active = !src.finish(ref, lead, R, K);
          if (active) begin();
        }
      }
    }
  }
}

// Lanes per keypoint of the launches, and the warps of a launch over `total`
// items: at most what the GPU holds at 162 registers a thread, then few enough
// that every group gets about as many.
constexpr int kGroupLanes = 4;
constexpr int kGroupThreads = 64;   // CTA size
constexpr int kGroupCtasPerSm = 6;
inline long long group_ctas(long long total) {
  constexpr int NG = kGroupThreads / kGroupLanes;
  const long long most = (long long)kGroupCtasPerSm * sm_count() * NG;
  const long long rounds = (total + most - 1) / most;
  return (total + rounds * NG - 1) / (rounds * NG);
}

}  // namespace trk
}  // namespace vio
