// The per-frame frontend as three dependent launches (Sec. III-B's stage
// order, with its data dependencies kept and its serialisation removed), for
// up to kMaxGroups groups of same-size stereo streams merged into each launch:
//
//  K1 frame_front_kernel    pyramid levels 1-4 of both cameras of every stream
//                           (one pyramid pass per tile) and, in the same
//                           launch, the per-cell FAST/NMS top-k candidates of
//                           camera 0. Levels beyond 4 follow as a further pass.
//                           A large step runs frame_level_kernel per level and
//                           K1 for the detection alone (split_front).
//  KN frame_initnet_kernel  (only with the learned initializer) persistent
//                           CTAs over rounds of 32 live tracks of one
//                           camera: network input from the previous and
//                           current pyramids, forward pass on the tcgen05
//                           tensor cores -> flow proposal + confidence.
//  K2 frame_track_kernel    one warp per keypoint (two in a small step,
//                           frame_track_team_kernel; four lanes in a large
//                           one, frame_track_groups_kernel): temporal
//                           tracking of every live track of both cameras
//                           (previous -> current pyramid; from the proposal
//                           over the lower levels when it is confident, the
//                           plain track otherwise or when that fails) AND
//                           stereo matching (camera 0 -> 1) of every cell's
//                           top-k candidates.
//  K3 frame_finalize_kernel one CTA per stream: keep the tracks that passed,
//                           count them per cell, select per cell the first
//                           k - count candidates (the detection of Sec. III-D
//                           with the cell buffer), append them to camera 0 and
//                           their successful matches to camera 1.
//
// Matching every candidate, rather than only the selected ones, lets stereo
// matching run beside temporal tracking instead of after it. A keypoint's
// match depends only on its position and the two current pyramids, so the
// result for every selected keypoint is the one the sequential order gives;
// the candidates that the occupancy rejects are simply not used. That costs
// a match per cell per frame where only a few cells take new keypoints, so
// the other order is a tunable (stereo_after): K2 tracks temporally only,
// K3 selects and appends to camera 0, then
//  K4 frame_stereo_kernel   one warp per selected keypoint: stereo matching;
//  K5 frame_append_kernel   one CTA per stream: the successful matches, in
//                           order, appended to camera 1.
// Both orders give the same lists bit for bit.
//
// Streams are either stepped together with host-side parity (unslotted), or
// each keeps its own parity, first-frame flag and activity in device memory
// (slotted): inactive streams are skipped and keep their state, so one
// captured launch sequence serves any subset of streams.
#include "detect_dev.cuh"
#include "finalize_dev.cuh"
#include "frame.cuh"
#include "initnet_dev.cuh"
#include "initnet_tc.cuh"
#include "pyramid_dev.cuh"
#include "track_team.cuh"

namespace vio {
namespace {


struct K1Args {
  Geom g;
  Batch all;           // images of the launch
  int m, T;            // levels and deepest-level tile of the first pyramid pass (m = 0: none)
  int ntx, nty;        // tiles of the first pass
  int det_step;        // 1: every image is a unit; 2: stream units (camera 0 detects)
  int blocks_per_unit; // det_step * tiles + detection blocks
  det::CellGeom cg;
  int n_cells, gy;
  const uint8_t* mask; // per detected image, or null
  long long mask_stride;
  unsigned long long* cand;
  int32_t* cand_count;
  int round_mode;
  // stream units (det_step == 2)
  int slotted, n_streams;
  const int32_t* parity;
  const int32_t* active;
  int32_t* step_ctr;   // incremented by block 0 (nullable)
  int32_t* ctr_copy;   // nullable: the new count is also stored here
};

struct MultiK1 {
  int n;
  long long block_end[kMaxGroups];
  K1Args a[kMaxGroups];
};

template <typename M>
__device__ __forceinline__ int group_of(const M& mm, long long i, long long& start) {
  int g = 0;
  while (g + 1 < mm.n && i >= mm.block_end[g]) ++g;
  start = g ? mm.block_end[g - 1] : 0;
  return g;
}

// Block layout per group: units, each unit = the pyramid tiles of its images
// followed by the detection cells of its first image, so that the blocks
// reading one image run together and its level 0 is read from DRAM about once.
// NT threads per CTA: 256 for a single frame's latency, 128 for throughput
// over many streams (a tunable of the batch).
template <int NT, bool MASKED>
__global__ void __launch_bounds__(NT, 768 / NT) frame_front_kernel(const __grid_constant__ MultiK1 mm) {
  extern __shared__ __align__(16) uint8_t smem[];
  long long start;
  const int gi = group_of(mm, blockIdx.x, start);
  const K1Args& a = mm.a[gi];
  const long long b = blockIdx.x - start;
  if (b == 0 && threadIdx.x == 0 && a.step_ctr) {
    const int c = *a.step_ctr + 1;
    *a.step_ctr = c;
    if (a.ctr_copy) *a.ctr_copy = c;
  }
  const int unit = (int)(b / a.blocks_per_unit);
  const int rem = (int)(b - (long long)unit * a.blocks_per_unit);
  int base = unit * a.det_step;
  if (a.det_step == 2 && a.slotted) {
    if (a.active && a.active[unit] == 0) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      return;
    }
    base = 2 * (a.parity[unit] * a.n_streams + unit);
  }
  const int tiles = a.ntx * a.nty;
  const int n_pyr = a.m > 0 ? a.det_step * tiles : 0;
  if (rem < n_pyr) {
    const int img = base + rem / tiles;
    const int t = rem % tiles;
    const int ty = t / a.ntx, tx = t - ty * a.ntx;
    if (a.det_step == 2 || img < a.all.n)
      pyr::pyramid_pass(a.g, a.all, img, 0, a.m, a.T, tx, ty, a.ntx, a.nty, a.round_mode, smem);
    return;
  }
  if (a.n_cells > 0)
    det::detect_block<MASKED>(level_ptr(a.g, a.all, base, 0), a.g.w[0], a.g.h[0], a.g.pitch[0],
                              a.cg, a.gy, rem - n_pyr,
                              MASKED ? a.mask + (long long)unit * a.mask_stride : nullptr,
                              a.cand + (long long)unit * a.n_cells * a.cg.k,
                              a.cand_count + (long long)unit * a.n_cells, smem);
  // after the level launches of a split front (a no-op otherwise): they read
  // the same frames and write nothing this launch reads, so it ran beside them
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// One pyramid level of both cameras of every active stream of every group (the
// front of a large step, see split_front): level s + 1 from level s, two
// output rows per thread (level_strip of pyramid_dev.cuh).
struct LevelGroup {
  Geom g;
  Batch all;
  int slotted, n_streams, round_mode;
  const int32_t* parity;
  const int32_t* active;
  pyr::Strips p;
};
struct MultiLevel {
  int n, s;
  long long block_end[kMaxGroups];
  LevelGroup a[kMaxGroups];
};
constexpr int LEVEL_THREADS = 128;
__global__ void __launch_bounds__(LEVEL_THREADS)
    frame_level_kernel(const __grid_constant__ MultiLevel mm) {
  // a programmatic dependent of the level below's launch (no-ops otherwise)
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  long long start;
  const int gi = group_of(mm, blockIdx.x, start);
  const LevelGroup& a = mm.a[gi];
  pyr::make_strip<2>(a.g, a.all, mm.s, a.p,
                     (unsigned)(blockIdx.x - start) * LEVEL_THREADS + threadIdx.x,
                     2 * a.n_streams, a.round_mode, [&](int i) {
                       const int unit = i >> 1;
                       if (!a.slotted) return i;
                       if (a.active && a.active[unit] == 0) return -1;
                       return 2 * (a.parity[unit] * a.n_streams + unit) + (i & 1);
                     });
}

struct MultiK2 {
  int n;
  long long block_end[kMaxGroups];   // in warps here
  FrameLaunch f[kMaxGroups];
};

// Flow proposals of every live track: persistent CTAs over tiles of
// ntc::ROUND consecutive slots of one keypoint list (the temporal numbering of
// frame_track_kernel: list (2 stream + camera), slot); tiles past a list's
// count are skipped whole.
struct MultiKN {
  int n;
  long long block_end[kMaxGroups];   // in keypoint lists (2 per stream)
  int32_t* fault;                    // VIO_ERR_TIMEOUT when a completion wait gave up
  FrameLaunch f[kMaxGroups];
};

// Tile of the launch: a list's slots s0 .. s0 + nv - 1.
struct NetTile {
  int gi, list, s0, nv;
  StreamRef r;
  long long in_list;
};

static_assert(KN_MAX_LISTS * 4 + 64 + ntc::SMEM <= 227 * 1024,
              "shared memory of the proposal kernel");

// Per-list tile counts, prefix-summed in shared memory (every CTA), so that
// the tiles that hold keypoints are dealt out evenly over the CTAs.
struct NetLists {
  int n;                              // lists
  int* end;                           // inclusive prefix of tiles per list
};

__device__ __forceinline__ int list_tiles(const MultiKN& mm, int li, int& gi, int& list,
                                          long long& in_list, StreamRef& r) {
  long long start;
  gi = group_of(mm, li, start);       // block_end counts lists here
  const FrameLaunch& f = mm.f[gi];
  list = (int)(li - start);
  const int s = list >> 1, c = list & 1;
  r = stream_ref(f, s);
  if (!r.active || !r.have_prev) return 0;
  in_list = ((long long)r.li * f.n_streams + s) * 2 + c;
  const int count = min(f.list_count[in_list], f.cap);
  return (count + ntc::ROUND - 1) / ntc::ROUND;
}

__device__ __forceinline__ NetTile net_tile(const MultiKN& mm, const NetLists& L, int v) {
  // the list holding valid tile v: first prefix end above v
  int lo = 0, hi = L.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (L.end[mid] > v) hi = mid; else lo = mid + 1;
  }
  NetTile T{};
  const int n_tiles = list_tiles(mm, lo, T.gi, T.list, T.in_list, T.r);
  const int j = v - (L.end[lo] - n_tiles);
  const FrameLaunch& f = mm.f[T.gi];
  const int count = min(f.list_count[T.in_list], f.cap);
  T.s0 = j * ntc::ROUND;
  T.nv = min(ntc::ROUND, count - T.s0);
  return T;
}

// Network inputs of a launch's tiles for ntc::run: the thread's row of a
// group, four channels (source / target at levels a and b) prefetched as
// aligned words.
struct KNSource {
  const MultiKN* mm;
  NetLists L;
  int n_valid;
  using Tile = NetTile;
  struct Regs {
    net::RowWords R[4];
    bool live;
  };
  __device__ int n_tiles() const { return n_valid; }
  __device__ Tile tile(int v) const { return net_tile(*mm, L, v); }
  __device__ void load(const Tile& T, int g, Regs& R) const {
    const FrameLaunch& f = mm->f[T.gi];
    const int i = g * ntc::GROUP + ntc::item_sample(), r = ntc::item_row(), c = T.list & 1;
    R.live = i < T.nv;
    if (!R.live) return;
    const float* xy = f.list_xy + 2 * (T.in_list * f.cap + T.s0 + i);
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
      net::row_prefetch(R.R[ch], f.g, (ch & 1) ? f.cur : f.prev,
                        ((ch & 1) ? T.r.cur_img : T.r.prev_img) + c,
                        ch < 2 ? f.net_la : f.net_lb, xy[0], xy[1], r);
  }
  __device__ void store(uint8_t* sm, const Regs& R) const {
    uint32_t px[4][4];
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
      if (R.live) {
        ntc::row_bytes(R.R[ch], px[ch]);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) px[ch][k] = 0x80808080u;
      }
    }
    if (ntc::NH == 1 || (threadIdx.x >> 7))
      ntc::store_row_bytes<1>(sm, ntc::item_sample(), ntc::item_row(), px);
    if (ntc::NH == 1 || !(threadIdx.x >> 7))
      ntc::store_row_bytes<0>(sm, ntc::item_sample(), ntc::item_row(), px);
  }
  __device__ void write(const Tile& T, int s, float dx, float dy, float conf) const {
    const FrameLaunch& f = mm->f[T.gi];
    float* o = f.net_out + 3 * ((long long)T.list * f.cap + T.s0 + s);
    o[0] = dx;
    o[1] = dy;
    o[2] = conf;
  }
};

// Persistent CTAs over the tiles that hold keypoints (valid tile v goes to
// CTA v mod gridDim.x). Needs level_a, level_b >= 1 (aligned level rows).
__global__ void __launch_bounds__(ntc::THREADS, 1) frame_initnet_kernel(
    const __grid_constant__ MultiKN mm) {
  extern __shared__ __align__(16) uint8_t sm[];
  __shared__ int ends[KN_MAX_LISTS];
  __shared__ int warp_tot[ntc::THREADS / 32];
  const int n_lists = (int)mm.block_end[mm.n - 1];
  // per-list tile counts and their inclusive prefix (chunks of blockDim.x)
  int carry = 0;
  for (int base = 0; base < n_lists; base += blockDim.x) {
    const int li = base + threadIdx.x;
    int nt = 0;
    if (li < n_lists) {
      int gi, list;
      long long in_list;
      StreamRef r;
      nt = list_tiles(mm, li, gi, list, in_list, r);
    }
    int incl = nt;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    int before = carry;
    for (int w = 0; w < warp; ++w) before += warp_tot[w];
    if (li < n_lists) ends[li] = before + incl;
    int tot = 0;
    for (int w = 0; w < ntc::THREADS / 32; ++w) tot += warp_tot[w];
    carry += tot;
    __syncthreads();
  }
  const KNSource src{&mm, NetLists{n_lists, ends}, carry};
  ntc::run(src, mm.f[0].net, sm, mm.fault);
}

// Occupancy hint of the tracking launch (blocks of up to 512 threads, this
// many per SM: 2 caps registers at 64 per thread); unset = compiler's choice.
#ifdef VIO_TRACK_MIN_BLOCKS
#define VIO_TRACK_BOUNDS __launch_bounds__(512, VIO_TRACK_MIN_BLOCKS)
#else
#define VIO_TRACK_BOUNDS
#endif

__global__ void VIO_TRACK_BOUNDS frame_track_kernel(const __grid_constant__ MultiK2 mm) {
  // the finalisation (launched as this launch's programmatic dependent) may
  // take its SM now and wait there for this launch's completion
  asm volatile("griddepcontrol.launch_dependents;");
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= mm.block_end[mm.n - 1]) return;
  long long start;
  const int gi = group_of(mm, w, start);
  const FrameLaunch& f = mm.f[gi];
  const long long wl = w - start;
  const float qnan = __int_as_float(0x7fc00000);
  const TrackCfg cfg{f.p.gn_iters, 1, f.p.fb_max_dist, -1};
  const int top = f.g.n_levels - 1;
  const long long n_temporal = 2LL * f.n_streams * f.cap;
  trk::Pos tf;
  float thf, dist;
  bool have;
  if (wl < n_temporal) {
    const int list = (int)(wl / f.cap);       // 2s + c
    const int slot = (int)(wl - (long long)list * f.cap);
    const int s = list >> 1, c = list & 1;
    const StreamRef r = stream_ref(f, s);
    if (!r.active) return;
    const long long in_list = ((long long)r.li * f.n_streams + s) * 2 + c;
    if (!r.have_prev || slot >= f.list_count[in_list]) {
      if (lane == 0) f.trk_status[wl] = VIO_TRACK_EMPTY;
      return;
    }
    const long long src = in_list * f.cap + slot;
    const float px = f.list_xy[2 * src], py = f.list_xy[2 * src + 1];
    int st = VIO_TRACK_EMPTY;
    bool learned = false;
    if (f.net) {
      const float* q = f.net_out + 3 * wl;
      if (q[2] >= f.net_tau) {
        float last;
        st = trk::track_fb(f.g, f.prev, r.prev_img + c, f.cur, r.cur_img + c, px, py,
                                      true, px + q[0], py + q[1], 0.f, cfg, f.net_top, lane, tf,
                                      thf, have, dist, last);
        learned = st == VIO_TRACK_OK && !(f.net_max_step > 0.f && last > f.net_max_step);
      }
    }
    if (!learned) {
      float last;
      st = trk::track_fb(f.g, f.prev, r.prev_img + c, f.cur, r.cur_img + c, px, py,
                                    false, 0.f, 0.f, 0.f, cfg, top, lane, tf, thf, have, dist,
                                    last);
    }
    if (lane == 0) {
      if (f.net) f.trk_learned[wl] = learned ? 1 : 0;
      f.trk_status[wl] = (uint8_t)st;
      f.trk_xy[2 * wl] = have ? (float)tf.ax + tf.dx : qnan;
      f.trk_xy[2 * wl + 1] = have ? (float)tf.ay + tf.dy : qnan;
    }
    return;
  }
  const long long w2 = wl - n_temporal;
  const int k = f.p.k_per_cell;
  const int n_cells = (f.g.w[0] / f.p.cell_w) * (f.g.h[0] / f.p.cell_h);
  const int per = n_cells * k;
  const int s = (int)(w2 / per);
  const int rem = (int)(w2 - (long long)s * per);
  const int cell = rem / k, rr = rem - cell * k;
  const StreamRef r = stream_ref(f, s);
  if (!r.active) return;
  if (rr >= f.cand_count[(long long)s * n_cells + cell]) {
    if (lane == 0) f.spec_status[w2] = VIO_TRACK_EMPTY;
    return;
  }
  const unsigned long long key = f.cand[w2];
  const unsigned idx = ~(unsigned)(key & 0xffffffffu);
  const float x = (float)(idx % (unsigned)f.g.w[0]), y = (float)(idx / (unsigned)f.g.w[0]);
  float last;
  const int st = trk::track_fb(f.g, f.cur, r.cur_img, f.cur, r.cur_img + 1, x, y,
                                          false, 0.f, 0.f, 0.f, cfg, top, lane, tf, thf, have,
                                          dist, last);
  if (lane == 0) {
    f.spec_status[w2] = (uint8_t)st;
    f.spec_xy[2 * w2] = have ? (float)tf.ax + tf.dx : qnan;
    f.spec_xy[2 * w2 + 1] = have ? (float)tf.ay + tf.dy : qnan;
  }
}

// The items of frame_track_kernel (temporal tracks and stereo candidates of
// every group, in its numbering) for the grouped tracker.
struct FrameTracks {
  const MultiK2& mm;
  struct Ref {
    long long out;        // temporal or stereo slot of the group
    int gi, s_img, d_img; // group, source and target image
    bool temporal, learned;
  };
  __device__ __forceinline__ long long total() const { return mm.block_end[mm.n - 1]; }
  __device__ __forceinline__ bool fetch(long long w, bool lead, Ref& ref, trk::Task& K) const {
    long long start;
    ref.gi = group_of(mm, w, start);
    const FrameLaunch& f = mm.f[ref.gi];
    const long long wl = w - start;
    const long long n_temporal = 2LL * f.n_streams * f.cap;
    ref.temporal = wl < n_temporal;
    ref.learned = false;
    K.has_init = false;
    K.top = f.g.n_levels - 1;
    K.iters = f.p.gn_iters;
    K.fb = 1;
    K.fb_max = f.p.fb_max_dist;
    if (ref.temporal) {
      const int list = (int)(wl / f.cap);       // 2s + c
      const int slot = (int)(wl - (long long)list * f.cap);
      const int s = list >> 1, c = list & 1;
      const StreamRef r = stream_ref(f, s);
      if (!r.active) return false;
      ref.out = wl;
      const long long in_list = ((long long)r.li * f.n_streams + s) * 2 + c;
      if (!r.have_prev || slot >= f.list_count[in_list]) {
        if (lead) f.trk_status[wl] = VIO_TRACK_EMPTY;
        return false;
      }
      const long long src = in_list * f.cap + slot;
      K.px = f.list_xy[2 * src];
      K.py = f.list_xy[2 * src + 1];
      ref.s_img = r.prev_img + c;
      ref.d_img = r.cur_img + c;
      if (f.net) {
        const float* q = f.net_out + 3 * wl;
        if (q[2] >= f.net_tau) {
          ref.learned = true;
          K.has_init = true;
          K.ix = K.px + q[0];
          K.iy = K.py + q[1];
          K.ith = 0.f;
          K.top = f.net_top;
        }
      }
      return true;
    }
    const long long w2 = wl - n_temporal;
    const int k = f.p.k_per_cell;
    const int n_cells = (f.g.w[0] / f.p.cell_w) * (f.g.h[0] / f.p.cell_h);
    const int per = n_cells * k;
    const int s = (int)(w2 / per);
    const int rem = (int)(w2 - (long long)s * per);
    const int cell = rem / k, rr = rem - cell * k;
    const StreamRef r = stream_ref(f, s);
    if (!r.active) return false;
    ref.out = w2;
    if (rr >= f.cand_count[(long long)s * n_cells + cell]) {
      if (lead) f.spec_status[w2] = VIO_TRACK_EMPTY;
      return false;
    }
    const unsigned idx = ~(unsigned)(f.cand[w2] & 0xffffffffu);
    K.px = (float)(idx % (unsigned)f.g.w[0]);
    K.py = (float)(idx / (unsigned)f.g.w[0]);
    ref.s_img = r.cur_img;
    ref.d_img = r.cur_img + 1;
    return true;
  }
  __device__ __forceinline__ void levels(const Ref& ref, bool back, int l, trk::Lv& S,
                                         trk::Lv& D) const {
    const FrameLaunch& f = mm.f[ref.gi];
    const Batch& from = ref.temporal ? f.prev : f.cur;
    S = trk::get_lv(f.g, back ? f.cur : from, back ? ref.d_img : ref.s_img, l);
    D = trk::get_lv(f.g, back ? from : f.cur, back ? ref.s_img : ref.d_img, l);
  }
  __device__ __forceinline__ bool finish(Ref& ref, bool lead, const trk::TrackResult& R,
                                         trk::Task& K) const {
    const FrameLaunch& f = mm.f[ref.gi];
    bool learned = ref.learned;
    if (learned) {
      learned = R.status == VIO_TRACK_OK && !(f.net_max_step > 0.f && R.last > f.net_max_step);
      if (!learned) {   // the plain track
        ref.learned = false;
        K.has_init = false;
        K.top = f.g.n_levels - 1;
        return false;
      }
    }
    if (lead) {
      if (ref.temporal) {
        if (f.net) f.trk_learned[ref.out] = learned ? 1 : 0;
        f.trk_status[ref.out] = (uint8_t)R.status;
        f.trk_xy[2 * ref.out] = R.x;
        f.trk_xy[2 * ref.out + 1] = R.y;
      } else {
        f.spec_status[ref.out] = (uint8_t)R.status;
        f.spec_xy[2 * ref.out] = R.x;
        f.spec_xy[2 * ref.out + 1] = R.y;
      }
    }
    return true;
  }
};

__global__ void __launch_bounds__(trk::kGroupThreads, trk::kGroupCtasPerSm)
    frame_track_groups_kernel(const __grid_constant__ MultiK2 mm) {
  constexpr int WPB = trk::kGroupThreads / 32;
  __shared__ __align__(16) uint8_t smem[WPB * trk::kWarpBytes<trk::kGroupLanes>];
  const int warp = threadIdx.x >> 5;
  trk::run_tracks<trk::kGroupLanes>(FrameTracks{mm}, (long long)blockIdx.x * WPB + warp,
                                    (long long)gridDim.x * WPB,
                                    smem + warp * trk::kWarpBytes<trk::kGroupLanes>);
}

// A CTA per slot.
__global__ void __launch_bounds__(trk::kTeamThreads, trk::kTeamCtasPerSm)
    frame_track_team_kernel(const __grid_constant__ MultiK2 mm) {
  asm volatile("griddepcontrol.launch_dependents;");   // as in frame_track_kernel
  __shared__ trk::TeamSmem sm;
  trk::team_track(FrameTracks{mm}, blockIdx.x, sm);
}

struct MultiK3 {
  int n;
  long long block_end[kMaxGroups];   // in blocks (= streams)
  FrameLaunch f[kMaxGroups];
};

// One CTA per stream. Each thread owns a contiguous run of list slots (then
// of cells), so each phase is one block-wide scan of packed counts.
__global__ void __launch_bounds__(K3_THREADS)
    frame_finalize_kernel(const __grid_constant__ MultiK3 mm) {
  // launched as the tracking launch's programmatic dependent: wait for its
  // completion and memory (a no-op after an ordinary launch); the stereo
  // launch that may follow can be scheduled now
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  extern __shared__ int occ_s[];
  __shared__ int ws32[K3_THREADS / 32];
  __shared__ unsigned long long ws64[K3_THREADS / 32];
  long long start;
  const int gi = group_of(mm, blockIdx.x, start);
  const FrameLaunch& f = mm.f[gi];
  const int s = (int)(blockIdx.x - start);
  finalize_stream(f, s, occ_s, ws32, ws64);
}

// ---- the after-selection order: stereo matching of the selected keypoints

// Selected keypoints a stream can have: every cell's k, at most the capacity.
__host__ __device__ inline int max_new(const FrameLaunch& f) {
  const int n = (f.g.w[0] / f.p.cell_w) * (f.g.h[0] / f.p.cell_h) * f.p.k_per_cell;
  return n < f.cap ? n : f.cap;
}

__global__ void frame_stereo_kernel(const __grid_constant__ MultiK2 mm) {
  // a programmatic dependent of the finalisation; the append may be
  // scheduled now
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= mm.block_end[mm.n - 1]) return;
  long long start;
  const int gi = group_of(mm, w, start);
  const FrameLaunch& f = mm.f[gi];
  const int mn = max_new(f);
  const long long wl = w - start;
  const int s = (int)(wl / mn), slot = (int)(wl - (long long)s * mn);
  const StreamRef r = stream_ref(f, s);
  if (!r.active || slot >= f.new_count[s]) return;
  const long long q = (long long)s * f.cap + slot;
  const TrackCfg cfg{f.p.gn_iters, 1, f.p.fb_max_dist, -1};
  trk::Pos tf;
  float thf, dist, last;
  bool have;
  const int st = trk::track_fb(f.g, f.cur, r.cur_img, f.cur, r.cur_img + 1, f.new_xy[2 * q],
                               f.new_xy[2 * q + 1], false, 0.f, 0.f, 0.f, cfg,
                               f.g.n_levels - 1, lane, tf, thf, have, dist, last);
  if (lane == 0) {
    const long long o = (long long)s * mn + slot;
    f.spec_status[o] = (uint8_t)st;
    f.spec_xy[2 * o] = have ? (float)tf.ax + tf.dx : __int_as_float(0x7fc00000);
    f.spec_xy[2 * o + 1] = have ? (float)tf.ay + tf.dy : __int_as_float(0x7fc00000);
  }
}

// Appends the successful matches of a stream's selected keypoints, in their
// order, to camera 1 after its surviving tracks, and ends the stream's step.
__global__ void __launch_bounds__(K3_THREADS)
    frame_append_kernel(const __grid_constant__ MultiK3 mm) {
  asm volatile("griddepcontrol.wait;" ::: "memory");   // after the stereo matching
  __shared__ int ws32[K3_THREADS / 32];
  long long start;
  const int gi = group_of(mm, blockIdx.x, start);
  const FrameLaunch& f = mm.f[gi];
  const int s = (int)(blockIdx.x - start);
  const StreamRef sr = stream_ref(f, s);
  if (!sr.active) return;
  const int t = threadIdx.x;
  const long long cap = f.cap;
  const int mn = max_new(f);
  const long long cnt_out = ((long long)sr.lo * f.n_streams + s) * 2;
  const long long out1 = (cnt_out + 1) * cap;
  const int surv1 = f.list_count[cnt_out + 1];           // K3 left the survivors' count
  const int ctr = *(f.ctr_copy ? f.ctr_copy : f.step_ctr);
  int32_t* st = f.stats + ((long long)((ctr - 1) % VIO_STATS_RING) * f.n_streams + s) * VIO_N_STATS;
  const int n_new = f.new_count[s];
  const int id0 = f.next_id[s] - st[VIO_STAT_NEW];
  const int run = (n_new + K3_THREADS - 1) / K3_THREADS;
  int m_tot = 0;
  for (int r0 = 0; r0 < run; r0 += kRunMax) {
    const int rl = min(kRunMax, run - r0);
    const int first = t * run + r0;
    unsigned keep = 0;
    for (int j = 0; j < rl; ++j) {
      const int i = first + j;
      if (i < n_new && f.spec_status[(long long)s * mn + i] == VIO_TRACK_OK) keep |= 1u << j;
    }
    int tot;
    int o = m_tot + block_scan<int>(__popc(keep), ws32, tot);
    for (int j = 0; j < rl; ++j) {
      if (!(keep & (1u << j))) continue;
      const int i = first + j;
      const int o1 = surv1 + o++;
      if (o1 < f.cap) {
        const long long q = (long long)s * mn + i;
        f.list_xy[2 * (out1 + o1)] = f.spec_xy[2 * q];
        f.list_xy[2 * (out1 + o1) + 1] = f.spec_xy[2 * q + 1];
        f.list_id[out1 + o1] = id0 + i;
        f.list_status[out1 + o1] = VIO_TRACK_OK;
      }
    }
    m_tot += tot;
    __syncthreads();
  }
  if (t == 0) {
    f.list_count[cnt_out + 1] = min(surv1 + m_tot, f.cap);
    st[VIO_STAT_MATCHED] = m_tot;
    if (f.slotted) {
      f.parity[s] = sr.lo;
      f.have_prev[s] = 1;
    }
  }
}

// The front of a large step: a launch per pyramid level and then the detection
// alone, in place of one launch of tiles that compute up to four levels each
// beside the detection blocks. The fused launch saves launches where they
// are the time (one 752 x 480 frame: 15 us against 28 us in four launches),
// but recomputes halos and runs both parts at the larger one's shared memory
// and registers. us a whole step, split / fused with 256 threads / with 128:
//   0.7 Mi pixels (one 752 x 480 stream): 61 / 57 / 57
//   1.4 (two): 73 / 74 / 72    2.1 (three): 97 / 96 / 91
//   2.8 (four): 112 / 111 / 109    3.4 (five): 120 / 123 / 119
//   3.5 (two of 1280 x 720): 146 / 148 / 151
//   4.0 (one of 1480 x 1420): 135 / 148 / 154
//   4.1 (six of 752 x 480): 145 / 148 / 146
//   4.1 (28 of 320 x 240): 136 / 143 / 135
//   5.3 (three of 1280 x 720): 183 / 202 / 199
//   7.9 (two of 1920 x 1080): 203 / 234 / 233
//   27.9 (16 of four sizes): 492 / 698 / 631
// Only when the levels of the fused pass are left to this rule (pyr_first 0).
constexpr long long kSplitPixels = 4LL << 20;
bool split_front(const Geom* g, const int* n_streams, int n_groups, int pyr_first) {
  long long px = 0;
  for (int i = 0; i < n_groups; ++i) px += 2LL * n_streams[i] * g[i].w[0] * g[i].h[0];
  return pyr_first == 0 && px >= kSplitPixels;
}

// Slots of a step's tracking launch per SM from which it runs by groups of lanes
// (track_group.cuh) instead of a warp per keypoint. Counted as used are, of a
// list's slots, at most two per keypoint that a frame can add: a stream keeps
// about one, and raising a capacity alone does not change the kernel (counted
// in full, a step of two 752 x 480 streams of 300 cells took 116 us with room
// for 8000 keypoints, by groups, and 86 with a warp each).
//
// Many slots of a step are empty and many tracks end early, which costs a warp
// of its own little and a group its turn. us a step with 2 slots a cell, groups
// / warps; all cells textured, half of them, 15%:
//   slots per SM
//    66 (two 1920 x 1080):  149 / 161, 139 / 119, 117 / 90
//   118 (12 of 752 x 480):  182 / 192, 138 / 143, 117 / 97
//   118, learned start:     222 / 228, 192 / 184, 171 / 135
//   132 (four 1920 x 1080): 257 / 266, 160 / 183, 134 / 113
//   197 (20 of 752 x 480):  300 / 283, 215 / 193, 136 / 115
//   197 (the same, 753 x 481): 322 / 278, 234 / 201, 150 / 126
//   197, learned start:     310 / 319, 243 / 237, 196 / 148
//   276 (7 of 640 x 480, 16 x 16 cells): 303 / 387, 221 / 246, 135 / 121
//   280 (16 of four odd sizes): 469 / 499, 342 / 334, 219 / 191
//   289 (16 of four sizes): 414 / 498, 296 / 323, 185 / 171
//   289, learned start:     501 / 566, 364 / 385, 251 / 212
// Below 200 the groups lose with half of the lists filled about what they gain
// with all of them.
constexpr long long kGroupSlotsPerSm = 200;

// Levels the fused pass of K1 computes (the rest follow in further passes);
// pyr_first < 0: none.
int first_levels(const Geom& g, int pyr_first) {
  if (pyr_first < 0) return 0;
  const int m = g.n_levels > 1 ? pyr::pass_levels(g.n_levels, 0) : 0;
  return (pyr_first > 0 && pyr_first < m) ? pyr_first : m;
}

K1Args front_args(const vio_params& p, const Geom& g, const Batch& all, int det_step,
                  const uint8_t* mask, long long mask_stride, unsigned long long* cand,
                  int32_t* cand_count, int tile_shift, int pyr_first, int threads,
                  int det_warps) {
  const int gx = g.w[0] / p.cell_w, gy = g.h[0] / p.cell_h;
  K1Args a{};
  a.g = g;
  a.all = all;
  a.m = first_levels(g, pyr_first);
  a.T = a.m > 0 ? pyr::top_tile(a.m, tile_shift) : 1;
  a.ntx = a.nty = 1;
  if (a.m > 0) pyr::pass_tiles(g.w, g.h, 0, a.m, a.T, a.ntx, a.nty);
  a.det_step = det_step;
  a.n_cells = gx * gy;
  a.gy = gy;
  a.cg = det::CellGeom{p.cell_w, p.cell_h, gx, p.k_per_cell, p.thresholds[p.n_thresholds - 1],
                       p.detect_border, 1, 1, 1, p.select_mode};
  det::detect_setup(a.cg, threads, det_warps);
  // at least one block: the group's first one counts its steps
  a.blocks_per_unit = std::max(1, (a.m > 0 ? det_step * a.ntx * a.nty : 0) +
                                      (a.n_cells > 0 ? det::detect_blocks(gx, gy, a.cg.bcx, a.cg.bcy)
                                                     : 0));
  a.mask = mask;
  a.mask_stride = mask_stride;
  a.cand = cand;
  a.cand_count = cand_count;
  a.round_mode = p.round_mode;
  return a;
}

template <int NT, bool MASKED>
cudaError_t launch_k1_nt(const MultiK1& mm, int smem, cudaStream_t s, bool beside) {
  if (smem > 40 * 1024) {   // 48 KiB less the static part
    const cudaError_t e = cudaFuncSetAttribute(
        frame_front_kernel<NT, MASKED>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  const long long blocks = mm.block_end[mm.n - 1];
  if (blocks <= 0) return cudaSuccess;
  return launch_dependent(frame_front_kernel<NT, MASKED>, dim3((unsigned)blocks), NT, (size_t)smem,
                          s, beside, mm);
}

// MASKED when any group of the launch has a per-pixel detection mask. beside:
// as a programmatic dependent of the level launches.
cudaError_t launch_k1(const MultiK1& mm, int smem, int threads, cudaStream_t s, bool beside) {
  bool masked = false;
  for (int i = 0; i < mm.n; ++i) masked = masked || mm.a[i].mask != nullptr;
  if (masked)
    return threads == 128 ? launch_k1_nt<128, true>(mm, smem, s, beside)
                          : launch_k1_nt<256, true>(mm, smem, s, beside);
  return threads == 128 ? launch_k1_nt<128, false>(mm, smem, s, beside)
                        : launch_k1_nt<256, false>(mm, smem, s, beside);
}

}  // namespace

int frame_front_smem(const Geom& g, const vio_params& p, int tile_shift, int pyr_first,
                     int threads, int det_warps) {
  det::CellGeom cg{p.cell_w, p.cell_h, g.w[0] / p.cell_w, p.k_per_cell, 0, 0, 1, 1, 1};
  int smem = det::detect_setup(cg, threads, det_warps);
  const int m = first_levels(g, pyr_first);
  if (m > 0) {
    const int ps = pyr::pass_smem_max(g.w, g.h, 0, m, pyr::top_tile(m, tile_shift));
    smem = ps > smem ? ps : smem;
  }
  return smem;
}

cudaError_t launch_frames(const FrameLaunch* fl, int n_groups, const FrameTune& tune,
                          cudaStream_t s, cudaEvent_t* marks, int part) {
  if (n_groups < 1 || n_groups > kMaxGroups) return cudaErrorInvalidValue;
  auto mark = [&](int i) {
    if (marks && marks[i]) cudaEventRecord(marks[i], s);
  };

  cudaError_t e = cudaSuccess;
  long long acc = 0;
  if (part != 2) {
    // K1: pyramid levels 1-4 + detection candidates (camera 0 of each stream)
    mark(0);
    Geom geoms[kMaxGroups];
    int ns[kMaxGroups];
    for (int i = 0; i < n_groups; ++i) {
      geoms[i] = fl[i].g;
      ns[i] = fl[i].n_streams;
    }
    const bool split = split_front(geoms, ns, n_groups, tune.pyr_first);
    const int pyr_first = split ? -1 : tune.pyr_first;
    const int k1_threads = split ? 128 : tune.k1_threads;
    MultiK1 m1{};
    m1.n = n_groups;
    int smem1 = 0;
    long long cells = 0;
    for (int i = 0; i < n_groups; ++i)
      cells += (long long)fl[i].n_streams * (fl[i].g.w[0] / fl[i].p.cell_w) *
               (fl[i].g.h[0] / fl[i].p.cell_h);
    const int gw = tune.det_warps > 0
                       ? tune.det_warps
                       : det::warps_per_cell(cells, sm_count(), det::kFrontWarpsPerSm);
    for (int i = 0; i < n_groups; ++i) {
      const FrameLaunch& f = fl[i];
      K1Args a = front_args(f.p, f.g, f.cur, 2, nullptr, 0, f.cand, f.cand_count,
                            tune.pyr_tile_shift, pyr_first, k1_threads, gw);
      a.slotted = f.slotted;
      a.n_streams = f.n_streams;
      a.parity = f.parity;
      a.active = f.active;
      a.step_ctr = f.step_ctr;
      a.ctr_copy = f.ctr_copy;
      m1.a[i] = a;
      acc += (long long)f.n_streams * a.blocks_per_unit;
      m1.block_end[i] = acc;
      const int sm = frame_front_smem(f.g, f.p, tune.pyr_tile_shift, pyr_first, k1_threads, gw);
      smem1 = sm > smem1 ? sm : smem1;
    }
    // beside one another as programmatic dependents, while the detection is
    // eight CTAs per SM at most (six are resident at once; two 1920 x 1080 pairs, pipelined over four frames:
    // 734 to 715 us; the batch's 2240 CTAs: 675 us so, 699 us beside)
    bool beside = split && acc <= 8LL * sm_count();
    for (int lv = 0; split; ++lv) {
      MultiLevel ml{};
      ml.n = n_groups;
      ml.s = lv;
      acc = 0;
      for (int i = 0; i < n_groups; ++i) {
        const FrameLaunch& f = fl[i];
        if (lv + 1 < f.g.n_levels) {
          ml.a[i] = LevelGroup{f.g, f.cur, f.slotted, f.n_streams, f.p.round_mode, f.parity,
                               f.active, pyr::strips(f.g, lv, 2)};
          acc += (pyr::strip_threads(ml.a[i].p, 2 * f.n_streams) + LEVEL_THREADS - 1) /
                 LEVEL_THREADS;
        }
        ml.block_end[i] = acc;
      }
      if (acc == 0) {
        beside = beside && lv > 0;
        break;
      }
      e = launch_dependent(frame_level_kernel, dim3((unsigned)acc), LEVEL_THREADS, 0, s,
                           beside && lv > 0, ml);
      if (e != cudaSuccess) return e;
    }
    e = launch_k1(m1, smem1, k1_threads, s, beside);
    if (e != cudaSuccess) return e;
    // levels beyond the first pass
    mark(1);
    for (int i = 0; i < n_groups && !split; ++i) {
      const FrameLaunch& f = fl[i];
      const int m1 = first_levels(f.g, tune.pyr_first);
      if (f.g.n_levels > 1 + m1) {
        e = launch_pyramid_rest(f.g, f.cur, m1, f.p.round_mode, s);
        if (e != cudaSuccess) return e;
      }
    }
  }
  if (part == 1) return cudaGetLastError();

  // KN: flow proposals (every group has the initializer on, or none)
  mark(2);
  if (fl[0].net) {
    MultiKN mn{};
    mn.n = n_groups;
    acc = 0;                                    // keypoint lists
    long long tiles = 0;                        // tiles if every list were full
    for (int i = 0; i < n_groups; ++i) {
      mn.f[i] = fl[i];
      acc += 2LL * fl[i].n_streams;
      tiles += 2LL * fl[i].n_streams * ((fl[i].cap + ntc::ROUND - 1) / ntc::ROUND);
      mn.block_end[i] = acc;
    }
    if (acc > KN_MAX_LISTS) return cudaErrorInvalidValue;
    static PerDeviceOnce kn_attr;
    e = once_per_device(kn_attr, [] {
      return cudaFuncSetAttribute(frame_initnet_kernel,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, ntc::SMEM);
    });
    if (e != cudaSuccess) return e;
    mn.fault = net_fault_word();
    const int sms = sm_count();
    const long long blocks = tiles < sms ? tiles : sms;
    if (blocks > 0)
      frame_initnet_kernel<<<(unsigned)blocks, ntc::THREADS, ntc::SMEM, s>>>(mn);
  }

  // K2: temporal tracking + stereo matching of all candidates
  mark(3);
  MultiK2 m2{};
  m2.n = n_groups;
  acc = 0;
  long long used = 0;   // slots, as kGroupSlotsPerSm counts them
  for (int i = 0; i < n_groups; ++i) {
    const FrameLaunch& f = fl[i];
    m2.f[i] = f;
    m2.f[i].stereo_after = tune.stereo_after;
    const int n_cells = (f.g.w[0] / f.p.cell_w) * (f.g.h[0] / f.p.cell_h);
    acc += 2LL * f.n_streams * f.cap +
           (tune.stereo_after ? 0LL : (long long)f.n_streams * n_cells * f.p.k_per_cell);
    m2.block_end[i] = acc;
    const long long fresh = (long long)n_cells * f.p.k_per_cell;
    used += f.n_streams * (2 * std::min<long long>(f.cap, 2 * fresh) +
                           (tune.stereo_after ? 0 : fresh));
  }
  const int k2t = tune.k2_threads;
  const bool k2_small = acc <= (long long)kDependentMaxWarpsPerSm * sm_count();
  if (acc > 0) {
    const long long blocks2 = (acc * 32 + k2t - 1) / k2t;
    if (used >= kGroupSlotsPerSm * sm_count())
      frame_track_groups_kernel<<<(unsigned)trk::group_ctas(acc), trk::kGroupThreads, 0, s>>>(m2);
    else if (acc <= trk::team_ctas())   // one wave (track_team.cuh)
      frame_track_team_kernel<<<(unsigned)acc, trk::kTeamThreads, 0, s>>>(m2);
    else
      frame_track_kernel<<<(unsigned)blocks2, k2t, 0, s>>>(m2);
  }

  // K3: finalize
  mark(4);
  MultiK3 m3{};
  m3.n = n_groups;
  acc = 0;
  int smem3 = 0;
  for (int i = 0; i < n_groups; ++i) {
    const FrameLaunch& f = fl[i];
    m3.f[i] = f;
    m3.f[i].stereo_after = tune.stereo_after;
    acc += f.n_streams;
    m3.block_end[i] = acc;
    const int sm = (f.g.w[0] / f.p.cell_w) * (f.g.h[0] / f.p.cell_h) * (int)sizeof(int);
    smem3 = sm > smem3 ? sm : smem3;
  }
  if (smem3 > 40 * 1024) {   // 48 KiB less the static part
    e = cudaFuncSetAttribute(frame_finalize_kernel,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem3);
    if (e != cudaSuccess) return e;
  }
  // a programmatic dependent of a small tracking launch (a single frame): its
  // CTA is resident and waiting when the tracking ends
  e = launch_dependent(frame_finalize_kernel, dim3((unsigned)acc), K3_THREADS, (size_t)smem3, s,
                       k2_small, m3);
  if (e != cudaSuccess) return e;
  if (tune.stereo_after) {
    // K4: stereo matching of the selected keypoints; K5: append to camera 1
    MultiK2 m4{};
    m4.n = n_groups;
    long long w4 = 0;
    for (int i = 0; i < n_groups; ++i) {
      m4.f[i] = m3.f[i];
      w4 += (long long)fl[i].n_streams * max_new(fl[i]);
      m4.block_end[i] = w4;
    }
    if (w4 > 0) {
      const long long blocks4 = (w4 * 32 + k2t - 1) / k2t;
      e = launch_dependent(frame_stereo_kernel, dim3((unsigned)blocks4), (unsigned)k2t, 0, s, true,
                           m4);
      if (e != cudaSuccess) return e;
    }
    e = launch_dependent(frame_append_kernel, dim3((unsigned)acc), K3_THREADS, 0, s,
                         w4 <= (long long)kDependentMaxWarpsPerSm * sm_count(), m3);
    if (e != cudaSuccess) return e;
  }
  mark(5);
  return cudaGetLastError();
}

int frame_launches(const Geom* g, const int* n_streams, int n_groups, bool with_net,
                   bool stereo_after, int pyr_first) {
  int n = (with_net ? 4 : 3) + (stereo_after ? 2 : 0);   // K1, (KN), K2, K3, (K4, K5)
  if (split_front(g, n_streams, n_groups, pyr_first)) {
    int levels = 0;
    for (int i = 0; i < n_groups; ++i) levels = levels > g[i].n_levels ? levels : g[i].n_levels;
    return n + levels - 1;
  }
  for (int i = 0; i < n_groups; ++i) {
    const int rest = g[i].n_levels - 1 - first_levels(g[i], pyr_first);
    if (rest > 0) n += pyr::rest_passes(rest);
  }
  return n;
}

}  // namespace vio
