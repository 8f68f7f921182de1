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

// A strip is a group of eight columns x a block of R output rows of an image. Threads first take the inner groups of every image's blocks, columns
// fastest, then the first and last groups, so that the warps of the former
// never meet the edge.
template <int R>
__global__ void __launch_bounds__(LEVEL_THREADS)
    pyr_level_kernel(const __grid_constant__ Geom g, const __grid_constant__ Batch b, int s,
                     int inner, int edge, int blocks, int round_mode) {
  // a programmatic dependent of the level below's launch (no-ops otherwise)
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const unsigned add2 = round_mode == 0 ? 0x00800080u : 0u;
  unsigned t = blockIdx.x * LEVEL_THREADS + threadIdx.x;
  const unsigned n_inner = (unsigned)(inner * blocks) * (unsigned)b.n;
  const unsigned n_inner_up = (n_inner + 31u) & ~31u;   // edges start a warp of their own
  const bool at_edge = t >= n_inner_up;
  if (!at_edge && t >= n_inner) return;
  if (at_edge) t -= n_inner_up;
  const unsigned cols = (unsigned)(at_edge ? edge : inner), per = cols * (unsigned)blocks;
  const int img = (int)(t / per);
  if (img >= b.n) return;
  const unsigned q = t - (unsigned)img * per;
  const int by = (int)(q / cols), c = (int)(q - (unsigned)by * cols);
  const int gx = at_edge ? (c == 0 ? 0 : inner + c) : c + 1;
  const int y0 = by * R;
  const uint8_t* src = level_ptr(g, b, img, s);
  if (!at_edge && ((reinterpret_cast<uintptr_t>(src) | (uintptr_t)g.pitch[s]) & 15) == 0)
    pyr::level_strip<R, true>(g, b, img, s, 8 * gx, y0, add2);
  else
    pyr::level_strip<R, false>(g, b, img, s, 8 * gx, y0, add2);
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
    // inner groups: the words beside their 16 input columns lie in the level
    const int groups = (g.w[s + 1] + 7) / 8, h = g.h[s + 1];
    const int inner = std::max(0, std::min(groups - 1, (g.w[s] - 20) / 16 + 1) - 1);
    const int edge = groups - inner;
    // output rows per thread: 2 (7 input rows for 4 of their own, all loaded
    // ahead: 28 us for level 1 of 185 images; 4 rows, 36 us, hold too many
    // registers to cover the loads), 1 where 2 leave less than two warps per
    // scheduler
    const int rows = (long long)groups * ((h + 1) / 2) * b.n < 256LL * sm_count() ? 1 : 2;
    const int blocks = (h + rows - 1) / rows;
    const long long per = (long long)groups * blocks;
    // 32-bit thread numbers: more images in further launches
    const int most = (int)std::min<long long>(b.n, std::max<long long>(1, (1LL << 30) / per));
    for (int i0 = 0; i0 < b.n; i0 += most) {
      Batch bc = b;
      bc.l0 += (long long)i0 * b.l0_stride;
      bc.upper += (long long)i0 * b.upper_stride;
      bc.n = std::min(most, b.n - i0);
      const long long threads = ((long long)inner * blocks * bc.n + 31) / 32 * 32 +
                                (long long)edge * blocks * bc.n;
      const cudaError_t e = launch_dependent(
          rows == 2 ? pyr_level_kernel<2> : pyr_level_kernel<1>,
          dim3((unsigned)((threads + LEVEL_THREADS - 1) / LEVEL_THREADS)), LEVEL_THREADS, 0, st,
          small && s > s0, g, bc, s, inner, edge, blocks, round_mode);
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
