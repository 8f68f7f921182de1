// Model-based start of a track (Sec. III-E): the warp starts where the
// camera model, the predicted pose and the keypoint's inverse depth put the
// sample pattern in the target image. One thread per keypoint (eight in a
// small launch): the keypoint and its 52 pattern points (a fronto-parallel
// patch at the keypoint's inverse depth) are back-projected through the source
// pinhole, moved by the relative pose and projected through the target
// pinhole; the start translation is the keypoint's projection and the start
// angle the least-squares rotation from the pattern offsets to the projected
// offsets.
#include "common.cuh"
#include "track_dev.cuh"

namespace vio {
namespace {

struct PredictArgs {
  vio_pinhole ks, kd;
  const vio_pose* pose;   // per image
  const float* pts;       // [img][cap] float2
  const float* rho;       // [img][cap]
  const int32_t* count;   // per image, or null
  int cap, n_images;
  float* init;            // [img][cap] float3
  uint8_t* valid;         // [img][cap], or null
};

// Every product that meets a sum is an explicit FMA or an unfused product, so
// that the two kernels below round alike and a keypoint's start does not depend
// on the size of its launch. Left to the compiler, the unrolled points of a
// thread were contracted another way than a lane's: same positions, other last
// bits of the angle (error against 64 bits over 6000 keypoints, mean 6.9e-7
// rad, 6.3e-7 so).

// Projection of the source pixel (x, y) at depth z into the target; false if
// it is not in front of the target camera.
__device__ __forceinline__ bool project(const PredictArgs& a, const vio_pose& T, float x, float y,
                                        float z, float& u, float& v) {
  const float X = __fmul_rn(x - a.ks.cx, z / a.ks.fx), Y = __fmul_rn(y - a.ks.cy, z / a.ks.fy);
  auto row = [&](int i) {
    return __fadd_rn(__fadd_rn(__fmaf_rn(T.R[3 * i], X, __fmul_rn(T.R[3 * i + 1], Y)),
                               __fmul_rn(T.R[3 * i + 2], z)),
                     T.t[i]);
  };
  const float qx = row(0), qy = row(1), qz = row(2);
  if (!(qz > 0.f)) return false;
  const float iz = 1.f / qz;
  u = __fmaf_rn(__fmul_rn(a.kd.fx, qx), iz, a.kd.cx);
  v = __fmaf_rn(__fmul_rn(a.kd.fy, qy), iz, a.kd.cy);
  return true;
}

// A point's terms of the two sums: pattern offset (u, v), projected offset
// (dx, dy).
__device__ __forceinline__ float dot_term(float u, float v, float dx, float dy) {
  return __fmaf_rn(u, dx, __fmul_rn(v, dy));
}
__device__ __forceinline__ float cross_term(float u, float v, float dx, float dy) {
  return __fmaf_rn(u, dy, -__fmul_rn(v, dx));
}

__global__ void predict_kernel(const __grid_constant__ PredictArgs a) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)a.n_images * a.cap) return;
  const int img = (int)(i / a.cap), k = (int)(i - (long long)img * a.cap);
  const int n = a.count ? min(max(a.count[img], 0), a.cap) : a.cap;
  if (k >= n) {
    if (a.valid) a.valid[i] = 0;
    return;
  }
  const vio_pose T = a.pose[img];
  const float px = a.pts[2 * i], py = a.pts[2 * i + 1];
  const float rho = a.rho[i];
  float tx = px, ty = py, th = 0.f;
  bool ok = rho > 0.f;
  if (ok) {
    const float z = 1.f / rho;
    ok = project(a, T, px, py, z, tx, ty);
    float dot = 0.f, cross = 0.f;
    constexpr trk::Pattern P = trk::make_pattern();
#pragma unroll
    for (int j = 0; j < trk::kNP; ++j) {
      const float u = P.u[j], v = P.v[j];
      float yx = tx, yy = ty;
      ok = project(a, T, px + u, py + v, z, yx, yy) && ok;
      const float dx = yx - tx, dy = yy - ty;
      dot = __fadd_rn(dot, dot_term(u, v, dx, dy));
      cross = __fadd_rn(cross, cross_term(u, v, dx, dy));
    }
    if (ok) th = atan2f(cross, dot);
  }
  if (!ok) {
    tx = px;
    ty = py;
    th = 0.f;
  }
  a.init[3 * i] = tx;
  a.init[3 * i + 1] = ty;
  a.init[3 * i + 2] = th;
  if (a.valid) a.valid[i] = ok ? 1 : 0;
}

// The same by eight lanes per keypoint, for launches of few keypoints: one
// thread's 52 projections, each with a division, are a chain of 4 us however
// few there are. A lane projects seven of the points; the two sums take the
// lanes' terms in the order of the points, as one thread does: the same results
// bit for bit. us a launch, keypoints: a thread each / eight lanes each:
//   900: 6.5 / 3.4    3000: 6.7 / 3.7    9000: 6.7 / 4.5    15000: 6.7 / 5.8
//   30000: 7.1 / 9.0    150000: 14.0 / 35.8 (the sums' exchanges)
constexpr int kLanes = 8;
constexpr long long kLanesPerSm = 96;   // keypoints per SM up to which it is the faster form
__global__ void predict_lanes_kernel(const __grid_constant__ PredictArgs a) {
  const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kLanes;
  if (i >= (long long)a.n_images * a.cap) return;
  const int g = threadIdx.x & (kLanes - 1);
  const unsigned mask = ((1u << kLanes) - 1u) << (threadIdx.x & 31 & ~(kLanes - 1));
  const int img = (int)(i / a.cap), k = (int)(i - (long long)img * a.cap);
  const int n = a.count ? min(max(a.count[img], 0), a.cap) : a.cap;
  if (k >= n) {
    if (a.valid && g == 0) a.valid[i] = 0;
    return;
  }
  const vio_pose T = a.pose[img];
  const float px = a.pts[2 * i], py = a.pts[2 * i + 1];
  const float rho = a.rho[i];
  float tx = px, ty = py, th = 0.f;
  bool ok = rho > 0.f;
  if (ok) {
    const float z = 1.f / rho;
    ok = project(a, T, px, py, z, tx, ty);
    constexpr int kPer = (trk::kNP + kLanes - 1) / kLanes;
    float d[kPer], c[kPer];
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int j = r * kLanes + g;
      d[r] = c[r] = 0.f;
      if (j < trk::kNP) {
        int iu = 0, iv = 0;
        trk::point_of(j, iu, iv);
        const float u = (float)iu, v = (float)iv;
        float yx = tx, yy = ty;
        ok = project(a, T, px + u, py + v, z, yx, yy) && ok;
        const float dx = yx - tx, dy = yy - ty;
        d[r] = dot_term(u, v, dx, dy);
        c[r] = cross_term(u, v, dx, dy);
      }
    }
    ok = __all_sync(mask, ok);
    float dot = 0.f, cross = 0.f;
#pragma unroll
    for (int j = 0; j < trk::kNP; ++j) {
      dot = __fadd_rn(dot, __shfl_sync(mask, d[j / kLanes], j % kLanes, kLanes));
      cross = __fadd_rn(cross, __shfl_sync(mask, c[j / kLanes], j % kLanes, kLanes));
    }
    if (ok) th = atan2f(cross, dot);
  }
  if (!ok) {
    tx = px;
    ty = py;
    th = 0.f;
  }
  if (g == 0) {
    a.init[3 * i] = tx;
    a.init[3 * i + 1] = ty;
    a.init[3 * i + 2] = th;
    if (a.valid) a.valid[i] = ok ? 1 : 0;
  }
}

bool pinhole_ok(const vio_pinhole* k) {
  return k && k->fx > 0.f && k->fy > 0.f && k->cx == k->cx && k->cy == k->cy;
}

}  // namespace
}  // namespace vio

extern "C" vio_status vio_predict_warp(const vio_pinhole* k_src, const vio_pinhole* k_dst,
                                       const vio_pose* d_pose, const float* d_pts,
                                       const float* d_inv_depth, const int32_t* d_count,
                                       int32_t capacity, int32_t n_images, float* d_init,
                                       uint8_t* d_valid, void* stream) {
  if (!vio::pinhole_ok(k_src) || !vio::pinhole_ok(k_dst) || !d_pose || !d_pts ||
      !d_inv_depth || !d_init || capacity < 0 || n_images < 0)
    return VIO_ERR_INVALID_ARG;
  const long long total = (long long)capacity * n_images;
  if (total == 0) return VIO_OK;
  vio::PredictArgs a{*k_src, *k_dst, d_pose, d_pts, d_inv_depth, d_count, capacity, n_images,
                     d_init, d_valid};
  const int threads = 128;
  const long long blocks = (total + threads - 1) / threads;
  if (blocks > 0x7fffffffLL) return VIO_ERR_UNSUPPORTED;
  if (total <= vio::kLanesPerSm * vio::sm_count()) {
    vio::predict_lanes_kernel<<<(unsigned)((total * vio::kLanes + threads - 1) / threads), threads,
                                0, (cudaStream_t)stream>>>(a);
    return cudaGetLastError() == cudaSuccess ? VIO_OK : VIO_ERR_CUDA;
  }
  vio::predict_kernel<<<(unsigned)blocks, threads, 0, (cudaStream_t)stream>>>(a);
  return cudaGetLastError() == cudaSuccess ? VIO_OK : VIO_ERR_CUDA;
}
