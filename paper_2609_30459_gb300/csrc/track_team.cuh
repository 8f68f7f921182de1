// The patch tracker by pairs of warps: a CTA of two warps per keypoint, for
// launches that leave much of the GPU idle. Same arithmetic as track_dev.cuh,
// bit for bit.
//
// What bounds it, and why this split. Such a launch takes as long as one
// keypoint's chain of dependent steps. Per level a single warp needs 0.31 us
// for a Gauss-Newton step and 1.3 us before the first one for the template:
// its loads (from L2 on first touch), the ten-value reduction, the factor and
// the solves. A direction's templates depend on the keypoint alone, so the
// second warp builds those of the lower levels while the first builds the top
// one and iterates there; the first then finds each next template in shared
// memory. The second also touches the target's rows around the start, which
// the first step of each level then finds in the L1. One copy of the
// template's code (second warp) and one of the step's (first warp) keep both
// in the instruction cache; the levels' geometry goes through shared memory
// rather than the arguments' constant bank at every level.
//
// Measured (752 x 480, four levels, five steps, forward and backward, us a
// launch; keypoints: a warp each / a pair of warps each):
//   300: 21.7 / 16.6    600: 21.7 / 18.1    900: 24.0 / 20.2
//   1200: 24.0 / 23.0   1500: 27.1 / 26.4   1800 (two waves): 27.2 / 37.7
// So the pair is used for launches of one wave. From about six keypoints per
// SM on a launch grows with their number although neither unit is full (1,500
// slots of a step: issue slots 36% busy, L1 wavefronts 30%).
#pragma once
#include "track_group.cuh"

namespace vio {
namespace trk {

constexpr int kTeamThreads = 64;
constexpr int kTeamCtasPerSm = 10;   // 102 registers a thread at most
// The CTAs of one wave.
inline long long team_ctas() { return (long long)kTeamCtasPerSm * sm_count(); }

struct TeamSmem {
  Lv lv[2][VIO_MAX_LEVELS];         // source and target of the forward pass
  float k[VIO_MAX_LEVELS][6][32];   // Tpl::K of every lane
  float c[VIO_MAX_LEVELS][4];       // c0, c1, c2, S
  int status[VIO_MAX_LEVELS];
  int op, top;                      // the next direction: forward, backward or none
  Pos p;                            // its template's position
  Pos t;                            // its start
};
enum { kTeamDone, kTeamForward, kTeamBackward };

// Reads level `l` of the target where the keypoint's pattern starts from t
// (level 0), for the L1 only.
__device__ __forceinline__ void touch_target(const Lv& D, const Pos& t, int l, const LanePts& P) {
#ifdef __CUDACC__
  int qx, qy;
  float f;
  to_level1(t.ax, t.dx, l, qx, f);
  to_level1(t.ay, t.dy, l, qy, f);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int x = min(max(qx + P.iu[j], 0), D.w - 1), y = min(max(qy + P.iv[j], 0), D.h - 1);
    unsigned v = 0;
    asm volatile("ld.global.nc.u8 %0, [%1];" : "+r"(v) : "l"(D.p + (long long)y * D.pitch + x));
  }
#endif
}

// Tracks item w of the source (track_group.cuh's run_tracks) by this CTA.
template <class Src>
__device__ __forceinline__ void team_track(const Src& src, long long w, TeamSmem& sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (w >= src.total()) return;
  typename Src::Ref ref;
  Task K{};
  if (!src.fetch(w, threadIdx.x == 0, ref, K)) return;
  const LanePts P = lane_points(lane);

  if (warp > 0) {
    // the levels' geometry once, a lane each, rather than through the
    // arguments' constant bank at every level
    if (lane < VIO_MAX_LEVELS) src.levels(ref, false, lane, sm.lv[0][lane], sm.lv[1][lane]);
    for (;;) {
      __syncthreads();                    // the direction is set
      const int op = sm.op, top = sm.top;
      if (op == kTeamDone) return;
      const Pos p = sm.p, t = sm.t;
      for (int l = top; l >= 0; --l) {
        Tpl T;
        const int st = build_template(sm.lv[op == kTeamBackward][l], p, l, lane, P, T);
        if (st == VIO_TRACK_OK) {
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) sm.k[l][3 * j + i][lane] = T.K[j][i];
          if (lane == 0) {
            sm.c[l][0] = T.c0;
            sm.c[l][1] = T.c1;
            sm.c[l][2] = T.c2;
            sm.c[l][3] = T.S;
          }
        }
        if (lane == 0) sm.status[l] = st;
        if (op == kTeamForward) touch_target(sm.lv[1][l], t, l, P);
        __syncthreads();                  // level l is there
      }
    }
  }

  // one direction per turn: forward from the task's start, then backward
  // from the forward result. The loop holds the only copy of the steps' code.
  const float qnan = __int_as_float(0x7fc00000);
  TrackResult R{};
  Pos p{}, tpl{}, t0{};
  float th0 = 0.f;
  bool back = false, fresh = true;
  for (;;) {
    if (fresh) {
      fresh = back = false;
      p = tpl = t0 = split(K.px, K.py);
      th0 = 0.f;
      if (K.has_init) {
        t0 = split(K.ix, K.iy);
        th0 = K.ith;
      }
    }
    if (lane == 0) {
      sm.op = back ? kTeamBackward : kTeamForward;
      sm.top = K.top;
      sm.p = tpl;
      sm.t = t0;
    }
    __syncthreads();
    Warp W;
    to_level1(t0.ax, t0.dx, K.top, W.t.ax, W.t.dx);
    to_level1(t0.ay, t0.dy, K.top, W.t.ay, W.t.dy);
    W.th = th0;
    {
      float a, b;
      small_rot(th0, W.cs, W.sn, a, b);
    }
    int st = VIO_TRACK_OK;
    float last = 0.f;
    int l = K.top;
    for (;; --l) {
      __syncthreads();                    // level l's template is there
      const Lv D = sm.lv[back ? 0 : 1][l];
      const int ts = sm.status[l];
      if (ts == VIO_TRACK_OK) {
        Tpl T;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int i = 0; i < 3; ++i) T.K[j][i] = sm.k[l][3 * j + i][lane];
        T.c0 = sm.c[l][0];
        T.c1 = sm.c[l][1];
        T.c2 = sm.c[l][2];
        T.S = sm.c[l][3];
        float moved = 0.f;
        for (int it = 0; it < K.iters; ++it) {
          st = gn_step(D, T, lane, P, W, moved);
          if (st != VIO_TRACK_OK) break;
        }
        if (st != VIO_TRACK_OK) break;
        if (l == 0) last = moved;
        rebase(W.t);
      } else if (l == 0) {
        st = ts;
      }
      if (l == 0) break;
      W.t.ax *= 2;
      W.t.ay *= 2;
      W.t.dx *= 2.f;
      W.t.dy *= 2.f;
      rebase(W.t);
    }
    for (; l > 0; --l) __syncthreads();   // the levels left after a failure

    if (!back) {
      R.have = st == VIO_TRACK_OK;
      R.x = R.have ? (float)W.t.ax + W.t.dx : qnan;
      R.y = R.have ? (float)W.t.ay + W.t.dy : qnan;
      R.th = R.have ? W.th : qnan;
      R.last = R.have ? last : qnan;
      R.dist = qnan;
      if (R.have && K.fb) {
        // template on the target at the forward result, unrotated; start at
        // the forward estimate's inverse
        back = true;
        tpl = W.t;
        t0 = p;
        th0 = -W.th;
        continue;
      }
    } else if (st == VIO_TRACK_OK) {
      const float ex = (float)(W.t.ax - p.ax) + (W.t.dx - p.dx);
      const float ey = (float)(W.t.ay - p.ay) + (W.t.dy - p.dy);
      R.dist = sqrtf(__fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
      if (R.dist > K.fb_max) st = VIO_TRACK_FB_FAIL;
    }
    R.status = st;
    if (src.finish(ref, lane == 0, R, K)) break;
    fresh = true;
  }
  if (lane == 0) sm.op = kTeamDone;
  __syncthreads();
}

}  // namespace trk
}  // namespace vio
