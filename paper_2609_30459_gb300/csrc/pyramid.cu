// Image pyramid entry point (Sec. III-C, Eq. 1-3): one launch per level, each
// straight from the level below (level_strip of pyramid_dev.cuh).
//
// What bounds it: the latency of its loads (a thread has all of its rows in
// flight, 21 loads), for a few images the launches, which are programmatic
// dependents of one another. A thread makes eight columns of two rows, so that
// an input row is loaded and unpacked twice and no shared memory or barrier is
// needed; the inner columns' threads share warps of their own and never test
// for an edge. 185 images of 752 x 480 to four levels, caches cold: 53 us;
// passes of two levels through shared-memory tiles of 128 x 128 pixels took 91
// us, bound by the shared-memory wavefronts of every output's 5 x 24 source
// bytes.
#include <algorithm>

#include "pyramid_dev.cuh"

namespace vio {
namespace {

constexpr int LEVEL_THREADS = 128;

template <int R>
__global__ void __launch_bounds__(LEVEL_THREADS)
    pyr_level_kernel(const __grid_constant__ Geom g, const __grid_constant__ Batch b, int s,
                     pyr::Strips p, int round_mode) {
  // a programmatic dependent of the level below's launch (no-ops otherwise)
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  pyr::make_strip<R>(g, b, s, p, blockIdx.x * LEVEL_THREADS + threadIdx.x, b.n, round_mode,
                     [](int i) { return i; });
}

// Two levels per launch through shared-memory tiles: the deeper levels of a
// frame step, where a launch costs more than the levels do.
__global__ void __launch_bounds__(pyr::kThreads) pyr_pass_kernel(Geom g, Batch b, int s, int m,
                                                                 int T, int ntx, int nty,
                                                                 int round_mode) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int tiles = ntx * nty;
  const int img = blockIdx.x / tiles;
  const int t = blockIdx.x - img * tiles;
  const int ty = t / ntx, tx = t - ty * ntx;
  pyr::pyramid_pass(g, b, img, s, m, T, tx, ty, ntx, nty, round_mode, smem);
}

}  // namespace

cudaError_t launch_pyramid_rest(const Geom& g, const Batch& b, int s0, int round_mode,
                                cudaStream_t st) {
  int s = s0;
  for (; s + 2 < g.n_levels; s += 2) {
    const int m = 2, T = pyr::top_tile(m, pyr::kRestShift);
    int ntx, nty;
    pyr::pass_tiles(g.w, g.h, s, m, T, ntx, nty);
    const int smem = pyr::pass_smem_max(g.w, g.h, s, m, T);
    if (smem > 40 * 1024) {   // 48 KiB less the static part
      const cudaError_t e = cudaFuncSetAttribute(
          pyr_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
    }
    const long long blocks = (long long)ntx * nty * b.n;
    pyr_pass_kernel<<<(unsigned)blocks, pyr::kThreads, smem, st>>>(g, b, s, m, T, ntx, nty,
                                                                   round_mode);
  }
  return s + 1 < g.n_levels ? launch_pyramid_from(g, b, s, round_mode, st) : cudaGetLastError();
}

cudaError_t launch_pyramid_from(const Geom& g, const Batch& b, int s0, int round_mode,
                                cudaStream_t st, bool* small_out) {
  bool small = false;   // the previous level's launch left most of the GPU idle
  for (int s = s0; s + 1 < g.n_levels; ++s) {
    // output rows per thread: 2 (7 input rows for 4 of their own, all loaded
    // ahead: 28 us for level 1 of 185 images; 4 rows, 36 us, hold too many
    // registers to cover the loads), 1 where 2 leave less than two warps per
    // scheduler
    const int rows =
        pyr::strip_threads(pyr::strips(g, s, 2), b.n) < 256LL * sm_count() ? 1 : 2;
    const pyr::Strips p = pyr::strips(g, s, rows);
    // 32-bit thread numbers: more images in further launches
    const int most = (int)std::min<long long>(
        b.n, std::max<long long>(1, (1LL << 30) / pyr::strip_threads(p, 1)));
    for (int i0 = 0; i0 < b.n; i0 += most) {
      Batch bc = b;
      bc.l0 += (long long)i0 * b.l0_stride;
      bc.upper += (long long)i0 * b.upper_stride;
      bc.n = std::min(most, b.n - i0);
      const long long threads = pyr::strip_threads(p, bc.n);
      const cudaError_t e = launch_dependent(
          rows == 2 ? pyr_level_kernel<2> : pyr_level_kernel<1>,
          dim3((unsigned)((threads + LEVEL_THREADS - 1) / LEVEL_THREADS)), LEVEL_THREADS, 0, st,
          small && s > s0, g, bc, s, p, round_mode);
      if (e != cudaSuccess) return e;
      small = threads <= 32LL * kDependentMaxWarpsPerSm * sm_count();
    }
  }
  if (small_out) *small_out = small;
  return cudaGetLastError();
}

cudaError_t launch_pyramid(const Geom& g, const Batch& b, int round_mode, cudaStream_t s,
                           bool* small) {
  return launch_pyramid_from(g, b, 0, round_mode, s, small);
}

}  // namespace vio
