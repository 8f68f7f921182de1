// Pyramidal inverse-compositional KLT (Sec. III-E, Eq. 4-5) for the stage
// entry points vio_track_patches / vio_stereo_match, and the
// forward-backward distance check. The tracker itself is in track_dev.cuh (a
// warp per keypoint), track_team.cuh (small launches) and track_group.cuh
// (large ones).
#include "track_team.cuh"

namespace vio {
namespace {

struct TrackArgs {
  Geom g;
  Batch src, dst;
  const float* pts;    // float2 per slot
  const float* init;   // float3 per slot or null
  const int32_t* count;
  int capacity, n_images;
  TrackCfg cfg;
  float* out3;         // float3 per slot or null
  float* out2;         // float2 per slot or null
  uint8_t* status;
  float* fb_dist;
  float* last_step;    // per slot or null
  int shared_pts;      // 1: every image tracks the same keypoints (pts, count of image 0)
};

constexpr int TRK_THREADS = 128;

__global__ void __launch_bounds__(TRK_THREADS) track_kernel(const __grid_constant__ TrackArgs a) {
  const long long wid = ((long long)blockIdx.x * TRK_THREADS + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const long long total = (long long)a.capacity * a.n_images;
  if (wid >= total) return;
  const int img = (int)(wid / a.capacity);
  const int k = (int)(wid - (long long)img * a.capacity);
  const int n = a.count ? min(a.count[a.shared_pts ? 0 : img], a.capacity) : a.capacity;
  const long long pk = a.shared_pts ? k : wid;   // keypoint slot of the source list
  const float nanf_ = __int_as_float(0x7fc00000);
  if (k >= n) {
    if (lane == 0) {
      a.status[wid] = VIO_TRACK_EMPTY;
      if (a.out3) a.out3[3 * wid] = a.out3[3 * wid + 1] = a.out3[3 * wid + 2] = nanf_;
      if (a.out2) a.out2[2 * wid] = a.out2[2 * wid + 1] = nanf_;
      if (a.fb_dist) a.fb_dist[wid] = nanf_;
      if (a.last_step) a.last_step[wid] = nanf_;
    }
    return;
  }
  trk::Pos tf;
  float thf = 0.f, dist, last = 0.f;
  bool have;
  const bool hi = a.init != nullptr;
  const int st = trk::track_fb(a.g, a.src, img, a.dst, img, a.pts[2 * pk], a.pts[2 * pk + 1],
                               hi, hi ? a.init[3 * wid] : 0.f, hi ? a.init[3 * wid + 1] : 0.f,
                               hi ? a.init[3 * wid + 2] : 0.f, a.cfg, top_level(a.cfg, a.g),
                               lane, tf, thf, have, dist, last);
  if (lane == 0) {
    a.status[wid] = (uint8_t)st;
    const float ox = have ? (float)tf.ax + tf.dx : nanf_;
    const float oy = have ? (float)tf.ay + tf.dy : nanf_;
    if (a.out3) {
      a.out3[3 * wid] = ox;
      a.out3[3 * wid + 1] = oy;
      a.out3[3 * wid + 2] = have ? thf : nanf_;
    }
    if (a.out2) {
      a.out2[2 * wid] = ox;
      a.out2[2 * wid + 1] = oy;
    }
    if (a.fb_dist) a.fb_dist[wid] = dist;
    if (a.last_step) a.last_step[wid] = have ? last : nanf_;
  }
}

// Keypoint wid = image * capacity + slot.
struct StageSource {
  const TrackArgs& a;
  struct Ref {
    long long wid;
    int img;
  };
  __device__ __forceinline__ long long total() const {
    return (long long)a.capacity * a.n_images;
  }
  __device__ __forceinline__ bool fetch(long long wid, bool lead, Ref& ref, trk::Task& K) const {
    const int img = (int)(wid / a.capacity);
    const int k = (int)(wid - (long long)img * a.capacity);
    const int n = a.count ? min(a.count[a.shared_pts ? 0 : img], a.capacity) : a.capacity;
    ref.wid = wid;
    ref.img = img;
    if (k >= n) {
      const float nanf_ = __int_as_float(0x7fc00000);
      if (lead) write(wid, trk::TrackResult{VIO_TRACK_EMPTY, false, nanf_, nanf_, nanf_, nanf_,
                                            nanf_});
      return false;
    }
    const long long pk = a.shared_pts ? k : wid;   // keypoint slot of the source list
    K.px = a.pts[2 * pk];
    K.py = a.pts[2 * pk + 1];
    K.has_init = a.init != nullptr;
    if (K.has_init) {
      K.ix = a.init[3 * wid];
      K.iy = a.init[3 * wid + 1];
      K.ith = a.init[3 * wid + 2];
    }
    K.top = top_level(a.cfg, a.g);
    K.iters = a.cfg.gn_iters;
    K.fb = a.cfg.fb;
    K.fb_max = a.cfg.fb_max_dist;
    return true;
  }
  __device__ __forceinline__ void levels(const Ref& ref, bool back, int l, trk::Lv& S,
                                         trk::Lv& D) const {
    S = trk::get_lv(a.g, back ? a.dst : a.src, ref.img, l);
    D = trk::get_lv(a.g, back ? a.src : a.dst, ref.img, l);
  }
  __device__ __forceinline__ bool finish(const Ref& ref, bool lead, const trk::TrackResult& R,
                                         trk::Task&) const {
    if (lead) write(ref.wid, R);
    return true;
  }
  __device__ __forceinline__ void write(long long wid, const trk::TrackResult& R) const {
    a.status[wid] = (uint8_t)R.status;
    if (a.out3) {
      a.out3[3 * wid] = R.x;
      a.out3[3 * wid + 1] = R.y;
      a.out3[3 * wid + 2] = R.th;
    }
    if (a.out2) {
      a.out2[2 * wid] = R.x;
      a.out2[2 * wid + 1] = R.y;
    }
    if (a.fb_dist) a.fb_dist[wid] = R.dist;
    if (a.last_step) a.last_step[wid] = R.last;
  }
};

__global__ void __launch_bounds__(trk::kGroupThreads, trk::kGroupCtasPerSm)
    track_groups_kernel(const __grid_constant__ TrackArgs a) {
  constexpr int WPB = trk::kGroupThreads / 32;
  __shared__ __align__(16) uint8_t smem[WPB * trk::kWarpBytes<trk::kGroupLanes>];
  const int warp = threadIdx.x >> 5;
  trk::run_tracks<trk::kGroupLanes>(StageSource{a}, (long long)blockIdx.x * WPB + warp,
                                    (long long)gridDim.x * WPB,
                                    smem + warp * trk::kWarpBytes<trk::kGroupLanes>);
}

// A CTA per keypoint.
__global__ void __launch_bounds__(trk::kTeamThreads, trk::kTeamCtasPerSm)
    track_team_kernel(const __grid_constant__ TrackArgs a) {
  __shared__ trk::TeamSmem sm;
  trk::team_track(StageSource{a}, blockIdx.x, sm);
}

__global__ void fb_check_kernel(const float* __restrict__ orig, const float* __restrict__ back,
                                const int32_t* __restrict__ count, int capacity,
                                long long total, float max_dist, uint8_t* __restrict__ status,
                                float* __restrict__ dist) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int img = (int)(i / capacity);
  const int k = (int)(i - (long long)img * capacity);
  const int n = count ? min(count[img], capacity) : capacity;
  if (k >= n || status[i] != VIO_TRACK_OK) return;
  const float ex = back[3 * i] - orig[2 * i];
  const float ey = back[3 * i + 1] - orig[2 * i + 1];
  const float d = sqrtf(ex * ex + ey * ey);
  if (dist) dist[i] = d;
  if (!(d <= max_dist)) status[i] = VIO_TRACK_FB_FAIL;
}

}  // namespace

cudaError_t launch_track(const Geom& g, const Batch& src, const Batch& dst, const float* pts,
                         const float* init, const int32_t* count, int capacity,
                         const TrackCfg& cfg, float* out3, float* out2, uint8_t* status,
                         float* fb_dist, cudaStream_t s, bool shared_pts, float* last_step) {
  TrackArgs a{g,    src,  dst,    pts,     init,      count,
              capacity, src.n, cfg, out3, out2, status, fb_dist, last_step,
              shared_pts ? 1 : 0};
  const long long warps = (long long)capacity * src.n;
  if (warps == 0) return cudaSuccess;
  // groups of lanes where the keypoints fill the GPU, a warp each where they
  // are fewer; rows that start at any byte cost a group more (track_group.cuh
  // has both sides measured for either)
  const bool words =
      ((reinterpret_cast<uintptr_t>(src.l0) | reinterpret_cast<uintptr_t>(dst.l0) |
        (uintptr_t)src.l0_stride | (uintptr_t)dst.l0_stride | (uintptr_t)g.pitch[0]) & 3) == 0;
  if (warps >= (words ? 28LL : 48LL) * sm_count()) {
    track_groups_kernel<<<(unsigned)trk::group_ctas(warps), trk::kGroupThreads, 0, s>>>(a);
    return cudaGetLastError();
  }
  // one wave of CTAs of two warps each (track_team.cuh)
  if (warps <= trk::team_ctas()) {
    track_team_kernel<<<(unsigned)warps, trk::kTeamThreads, 0, s>>>(a);
    return cudaGetLastError();
  }
  const long long blocks = (warps * 32 + TRK_THREADS - 1) / TRK_THREADS;
  track_kernel<<<(unsigned)blocks, TRK_THREADS, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_fb_check(const float* orig, const float* back, const int32_t* count,
                            int capacity, int n_images, float max_dist, uint8_t* status,
                            float* dist, cudaStream_t s) {
  const long long total = (long long)capacity * n_images;
  if (total == 0) return cudaSuccess;
  fb_check_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(orig, back, count, capacity,
                                                                  total, max_dist, status, dist);
  return cudaGetLastError();
}

}  // namespace vio
