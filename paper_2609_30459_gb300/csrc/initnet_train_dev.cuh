// Device code of the flow network's training pass (the train kernel of
// initnet.cu): forward pass with BF16 activations on mma.sync tiles, the loss
// of the flow and confidence outputs, and the backward pass in FP32.
//
// A CTA of eight warps takes two samples at a time through all layers and keeps
// its share of every weight gradient in registers from its first sample to its
// last (36 sums of each 3x3 layer, 32 of fc1 a thread), so that a sample adds
// to no memory: each layer's gradient is a small matrix product in which a
// thread owns four output channels x one input channel x nine taps and reads
// its operands as 16-byte words (FP32 copies of the activations; the gradients
// of a layer's outputs as [position][channel]). What bounds it: about 0.5 M
// FP32 multiply-adds a sample, at 36 of them per 8 shared-memory loads, and
// the barriers between the layers. The CTA's sums go once, by whole rows
// staged in shared memory, to the global gradient. A minibatch of 1024: 88 us,
// against 660 us with a sample per warp that added every product to sums in
// shared memory by atomics (28 thousand a sample) from scalar loads.
//
// The forward pass gives a warp a 16-position tile of conv1 or an 8-channel
// tile of the later layers of one sample: the products and the order of the
// sums are those of one warp running the whole sample.
#pragma once
#include <math.h>

#include "initnet_dev.cuh"

namespace vio {
namespace net {

constexpr int TRAIN_WARPS = 8;
constexpr int TRAIN_S = 2;   // samples at a time
static_assert(TRAIN_WARPS == 4 * TRAIN_S, "four warps a sample");

// FP32 copies of the bordered activations: row pitches and channel strides in
// floats (rows 16-byte aligned, channels on different banks)
constexpr int XF_P = 20, XF_C = 18 * XF_P;      // x  [4][18][20]
constexpr int H1F_P = 12, H1F_C = 10 * H1F_P;   // h1 [32][10][12]
constexpr int H2F_P = 8, H2F_C = 6 * H2F_P + 4; // h2 [32][6][8] + 4
// byte offsets in a sample's piece
constexpr int TS_X = 0;                            // BF16 [4][18][18]
constexpr int TS_H1 = TS_X + 4 * XP * XP * 2;      // BF16 [32][10][10]
constexpr int TS_H2 = TS_H1 + 32 * H1P * H1P * 2;  // BF16 [32][6][6]
constexpr int TS_H3 = TS_H2 + 32 * H2P * H2P * 2;  // BF16 [128]
constexpr int TS_H4 = TS_H3 + 128 * 2;             // BF16 [64]
constexpr int TS_XF = (TS_H4 + 64 * 2 + 15) & ~15;
constexpr int TS_H1F = TS_XF + 4 * XF_C * 4;
constexpr int TS_H2F = TS_H1F + 32 * H1F_C * 4;
constexpr int TS_H3F = TS_H2F + 32 * H2F_C * 4;
constexpr int TS_H4F = TS_H3F + 128 * 4;
constexpr int TS_DA1 = TS_H4F + 64 * 4;            // [64 positions][32 channels]
constexpr int TS_DA2 = TS_DA1 + 64 * 32 * 4;       // [16][32]
constexpr int TS_DA3 = TS_DA2 + 16 * 32 * 4;       // [4][32]
constexpr int TS_DA4 = TS_DA3 + 4 * 32 * 4;        // [64]
constexpr int TS_DO = TS_DA4 + 64 * 4;             // [4] (3 used)
constexpr int TS_BYTES = TS_DO + 16;
static_assert(TS_BYTES % 16 == 0 && TS_XF % 16 == 0 && TS_H1F % 16 == 0 && TS_H2F % 16 == 0 &&
                  TS_DA1 % 16 == 0,
              "16-byte rows");
// byte offsets in the CTA's shared memory: transposed weights as BF16 pairs
// (output channels 2p, 2p + 1 in the low and high half), tap offsets, samples
constexpr int TB_W2 = 0;                        // [16 pairs][9 taps][32 input channels]
constexpr int TB_W3 = TB_W2 + 16 * 288 * 4;
constexpr int TB_W4 = TB_W3 + 16 * 288 * 4;     // [32 pairs][128 inputs]
constexpr int TB_T1 = TB_W4 + 32 * 128 * 4;     // tap offsets of conv1..3 (uint16)
constexpr int TB_T2 = TB_T1 + K1 * 2;
constexpr int TB_T3 = TB_T2 + K2 * 2;
constexpr int TB_S = (TB_T3 + K3 * 2 + 15) & ~15;
constexpr int TB_USED = TB_S + TRAIN_S * TS_BYTES;
constexpr int TB_GRAD = N_MASTER * 4;           // the gradient's staging, at the end
constexpr int train_smem_bytes() { return ((TB_USED > TB_GRAD ? TB_USED : TB_GRAD) + 127) & ~127; }

// CTAs of a launch on n_sms SMs (one per SM: its registers)
inline int train_blocks(int n, int n_sms) {
  if (n <= n_sms) return n;
  const int pairs = (n + TRAIN_S - 1) / TRAIN_S;
  return pairs < n_sms ? pairs : n_sms;
}

__device__ __forceinline__ float bf_lo(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf_hi(uint32_t p) { return __uint_as_float(p & 0xffff0000u); }

// NT 8-channel tiles nt0 .. of 16-position tile mt of a 3x3 stride-2
// convolution of a bordered BF16 map [CIN][HIN+2][HIN+2]: accumulators acc.
// tab[k] = the offset of tap k (0xffff: a padding tap, zero).
template <int CIN, int HIN, int KPAD, int NT>
__device__ __forceinline__ void conv_tile(const uint16_t* in, const uint16_t* tab,
                                          const uint16_t* W, int mt, int nt0, int lane,
                                          float (&acc)[NT][4]) {
  constexpr int HOUT = HIN / 2, P = HIN + 2, M = HOUT * HOUT;
  const int g = lane >> 2, t = lane & 3;
  int base[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = mt * 16 + g + 8 * h, q = r < M ? r : 0;   // a row past M is not used
    base[h] = 2 * (q / HOUT) * P + 2 * (q % HOUT);
  }
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[nt][e] = 0.f;
#pragma unroll 3
  for (int ks = 0; ks < KPAD / 16; ++ks) {
    uint32_t a[4];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const uint32_t o2 =
          *reinterpret_cast<const uint32_t*>(tab + ks * 16 + 8 * half + 2 * t);
      const int o0 = (int)(o2 & 0xffffu), o1 = (int)(o2 >> 16);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t lo, hi;
        if (KPAD == CIN * 9) {
          lo = in[base[h] + o0];
          hi = in[base[h] + o1];
        } else {
          lo = o0 != 0xffff ? in[base[h] + o0] : (uint16_t)0;
          hi = o1 != 0xffff ? in[base[h] + o1] : (uint16_t)0;
        }
        a[h + 2 * half] = lo | (hi << 16);
      }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const uint16_t* wr = W + ((nt0 + nt) * 8 + g) * KPAD + ks * 16 + 2 * t;
      const uint32_t b0 = __ldg(reinterpret_cast<const uint32_t*>(wr));
      const uint32_t b1 = __ldg(reinterpret_cast<const uint32_t*>(wr + 8));
      mma16816(acc[nt], a, b0, b1);
    }
  }
}

// Bias, ReLU and BF16 of conv_tile's accumulators: f(channel, position, bits).
template <int NT, class F>
__device__ __forceinline__ void tile_out(const float (&acc)[NT][4], const float* bias, int M,
                                         int mt, int nt0, int lane, F f) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = mt * 16 + g + 8 * (e >> 1), n = (nt0 + nt) * 8 + 2 * t + (e & 1);
      if (r < M) f(n, r, f2bf(fmaxf(acc[nt][e] + bias[n], 0.f)));
    }
}

// The training pass of one CTA over pairs of samples, pair blockIdx.x, +
// gridDim.x, ...; dsm: the CTA's shared memory (train_smem_bytes(), 16-byte
// aligned).
__device__ __forceinline__ void train_block(const void* __restrict__ packed_w,
                                            const uint16_t* __restrict__ x,
                                            const float* __restrict__ flow,
                                            const int32_t* __restrict__ index, int n,
                                            float grad_scale, float radius,
                                            float* __restrict__ grad,
                                            float* __restrict__ loss_sum, uint8_t* dsm) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ws = warp >> 2, wq = warp & 3;       // the warp's sample and quarter
  const Packed P = packed(packed_w);
  uint32_t* w2t = reinterpret_cast<uint32_t*>(dsm + TB_W2);
  uint32_t* w3t = reinterpret_cast<uint32_t*>(dsm + TB_W3);
  uint32_t* w4t = reinterpret_cast<uint32_t*>(dsm + TB_W4);
  uint16_t* tab1 = reinterpret_cast<uint16_t*>(dsm + TB_T1);
  uint16_t* tab2 = reinterpret_cast<uint16_t*>(dsm + TB_T2);
  uint16_t* tab3 = reinterpret_cast<uint16_t*>(dsm + TB_T3);
  uint8_t* smp = dsm + TB_S;
  auto at = [&](int s, int off) { return smp + s * TS_BYTES + off; };
  auto u16 = [&](int s, int off) { return reinterpret_cast<uint16_t*>(at(s, off)); };
  auto f32 = [&](int s, int off) { return reinterpret_cast<float*>(at(s, off)); };

  // transposed weights, tap offsets, zero borders (never written again)
  for (int e = tid; e < 16 * 288; e += blockDim.x) {
    const int p = e / 288, r = e - p * 288, tap = r >> 5, c = r & 31, k = c * 9 + tap;
    w2t[e] = (uint32_t)P.w[OFF_W2 + 2 * p * K2 + k] |
             ((uint32_t)P.w[OFF_W2 + (2 * p + 1) * K2 + k] << 16);
    w3t[e] = (uint32_t)P.w[OFF_W3 + 2 * p * K3 + k] |
             ((uint32_t)P.w[OFF_W3 + (2 * p + 1) * K3 + k] << 16);
  }
  for (int e = tid; e < 32 * 128; e += blockDim.x) {
    const int p = e >> 7, k = e & 127;
    w4t[e] = (uint32_t)P.w[OFF_W4 + 2 * p * K4 + k] |
             ((uint32_t)P.w[OFF_W4 + (2 * p + 1) * K4 + k] << 16);
  }
  for (int k = tid; k < K2; k += blockDim.x) {
    const int o1 = tap_off(k, 36, XP);
    if (k < K1) tab1[k] = o1 < 0 ? (uint16_t)0xffff : (uint16_t)o1;
    tab2[k] = (uint16_t)tap_off(k, K2, H1P);
    tab3[k] = (uint16_t)tap_off(k, K3, H2P);
  }
  for (int e = tid; e < TRAIN_S * TS_BYTES / 4; e += blockDim.x)
    reinterpret_cast<uint32_t*>(smp)[e] = 0u;
  __syncthreads();

  // this thread's gradient sums. 3x3 layers: output channels 4 og .. 4 og + 3,
  // one input channel, nine taps (conv1: over the positions of output row
  // `warp` only); fc1: outputs n4 .., inputs k8 ..; fc2: one weight
  const int og = lane & 7, ci = lane >> 3, c2 = warp * 4 + ci;
  const int n4 = 4 * (tid >> 4), k8 = 8 * (tid & 15);
  float g1[4][9], g2[4][9], g3[4][9], g4[4][8], b1[4], b2[4], b3[4], b4[4];
  float g5 = 0.f, b5 = 0.f, lsum = 0.f;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
#pragma unroll
    for (int k = 0; k < 9; ++k) g1[a][k] = g2[a][k] = g3[a][k] = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) g4[a][k] = 0.f;
    b1[a] = b2[a] = b3[a] = b4[a] = 0.f;
  }

  // with no more samples than CTAs, one at a time (train_blocks)
  const int per = n <= (int)gridDim.x ? 1 : TRAIN_S;
  const int pairs = (n + per - 1) / per;
  for (int pr = blockIdx.x; pr < pairs; pr += gridDim.x) {
    const int ns = min(per, n - pr * per);    // samples of this pair
    const bool live = ws < ns;
    long long sample = 0;
    if (live) {
      const long long i = (long long)pr * per + ws;
      sample = index ? index[i] : i;
      const uint16_t* src = x + sample * 1024;
      uint16_t* xb = u16(ws, TS_X);
      float* xf = f32(ws, TS_XF);
      for (int e = tid & 127; e < 1024; e += 128) {
        const int ch = e >> 8, r = (e >> 4) & 15, c = e & 15;
        const uint16_t v = src[e];
        xb[ch * XP * XP + (r + 1) * XP + (c + 1)] = v;
        xf[ch * XF_C + (r + 1) * XF_P + (c + 1)] = bf2f(v);
      }
    }
    __syncthreads();
    if (live) {   // conv1: position tile wq, all channels
      float acc[4][4];
      conv_tile<4, 16, K1, 4>(u16(ws, TS_X), tab1, P.w + OFF_W1, wq, 0, lane, acc);
      uint16_t* hb = u16(ws, TS_H1);
      float* hf = f32(ws, TS_H1F);
      tile_out<4>(acc, P.b + OFF_B1, 64, wq, 0, lane, [&](int c, int r, uint16_t v) {
        const int i = (r >> 3) + 1, j = (r & 7) + 1;
        hb[c * H1P * H1P + i * H1P + j] = v;
        hf[c * H1F_C + i * H1F_P + j] = bf2f(v);
      });
    }
    __syncthreads();
    if (live) {   // conv2: channel tile wq
      float acc[1][4];
      conv_tile<32, 8, K2, 1>(u16(ws, TS_H1), tab2, P.w + OFF_W2, 0, wq, lane, acc);
      uint16_t* hb = u16(ws, TS_H2);
      float* hf = f32(ws, TS_H2F);
      tile_out<1>(acc, P.b + OFF_B2, 16, 0, wq, lane, [&](int c, int r, uint16_t v) {
        const int i = (r >> 2) + 1, j = (r & 3) + 1;
        hb[c * H2P * H2P + i * H2P + j] = v;
        hf[c * H2F_C + i * H2F_P + j] = bf2f(v);
      });
    }
    __syncthreads();
    if (live) {   // conv3
      float acc[1][4];
      conv_tile<32, 4, K3, 1>(u16(ws, TS_H2), tab3, P.w + OFF_W3, 0, wq, lane, acc);
      tile_out<1>(acc, P.b + OFF_B3, 4, 0, wq, lane, [&](int c, int r, uint16_t v) {
        u16(ws, TS_H3)[c * 4 + r] = v;
        f32(ws, TS_H3F)[c * 4 + r] = bf2f(v);
      });
    }
    __syncthreads();
    if (live) {   // fc1: 16 outputs
      float acc[2][4];
      fc_layer<K4, 2>(u16(ws, TS_H3), P.w + OFF_W4 + 16 * wq * K4, lane, acc);
      if ((lane >> 2) == 0)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int k = 16 * wq + nt * 8 + 2 * (lane & 3) + e;
            const uint16_t v = f2bf(fmaxf(acc[nt][e] + P.b[OFF_B4 + k], 0.f));
            u16(ws, TS_H4)[k] = v;
            f32(ws, TS_H4F)[k] = bf2f(v);
          }
    }
    __syncthreads();
    if (live && wq == 0) {   // fc2, the loss and the gradient down to fc1's outputs
      float acc[1][4];
      fc_layer<K5, 1>(u16(ws, TS_H4), P.w + OFF_W5, lane, acc);
      const float o0 = __shfl_sync(0xffffffffu, acc[0][0], 0) + P.b[OFF_B5 + 0];
      const float o1 = __shfl_sync(0xffffffffu, acc[0][1], 0) + P.b[OFF_B5 + 1];
      const float o2 = __shfl_sync(0xffffffffu, acc[0][0], 1) + P.b[OFF_B5 + 2];
      // loss and dL/do (the label carries no gradient)
      const float fx = flow[2 * sample], fy = flow[2 * sample + 1];
      const float t0 = fx / kScale, t1 = fy / kScale;
      const float y = hypotf(o0 * kScale - fx, o1 * kScale - fy) < radius ? 1.f : 0.f;
      const float sg = 1.f / (1.f + expf(-o2));
      lsum += (o0 - t0) * (o0 - t0) + (o1 - t1) * (o1 - t1) -
              (y * logf(sg + 1e-12f) + (1.f - y) * logf(1.f - sg + 1e-12f));
      const float d[3] = {grad_scale * 2.f * (o0 - t0), grad_scale * 2.f * (o1 - t1),
                          grad_scale * (sg - y)};
      if (lane < 3) f32(ws, TS_DO)[lane] = lane == 0 ? d[0] : lane == 1 ? d[1] : d[2];
      for (int k = lane; k < 64; k += 32) {
        const float dh = bf2f(P.w[OFF_W5 + k]) * d[0] + bf2f(P.w[OFF_W5 + K5 + k]) * d[1] +
                         bf2f(P.w[OFF_W5 + 2 * K5 + k]) * d[2];
        f32(ws, TS_DA4)[k] = f32(ws, TS_H4F)[k] > 0.f ? dh : 0.f;
      }
    }
    __syncthreads();
    // fc2 and fc1 gradients
    for (int s = 0; s < ns; ++s) {
      if (tid < 192) g5 += f32(s, TS_DO)[tid >> 6] * f32(s, TS_H4F)[tid & 63];
      if (tid < 3) b5 += f32(s, TS_DO)[tid];
      const float4 d = *reinterpret_cast<const float4*>(f32(s, TS_DA4) + n4);
      const float4 h0 = *reinterpret_cast<const float4*>(f32(s, TS_H3F) + k8);
      const float4 h1 = *reinterpret_cast<const float4*>(f32(s, TS_H3F) + k8 + 4);
      const float dv[4] = {d.x, d.y, d.z, d.w};
      const float hv[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        b4[a] += dv[a];
#pragma unroll
        for (int k = 0; k < 8; ++k) g4[a][k] += dv[a] * hv[k];
      }
    }
    if (live) {   // da3: input k of fc1, flattened (channel, position)
      const int k = tid & 127;
      const float* da4 = f32(ws, TS_DA4);
      float s0 = 0.f, s1 = 0.f;
#pragma unroll 4
      for (int p = 0; p < 32; p += 2) {
        const float4 d = *reinterpret_cast<const float4*>(da4 + 2 * p);
        const uint32_t w0 = w4t[p * 128 + k], w1 = w4t[(p + 1) * 128 + k];
        s0 += bf_lo(w0) * d.x;
        s1 += bf_hi(w0) * d.y;
        s0 += bf_lo(w1) * d.z;
        s1 += bf_hi(w1) * d.w;
      }
      f32(ws, TS_DA3)[(k & 3) * 32 + (k >> 2)] = f32(ws, TS_H3F)[k] > 0.f ? s0 + s1 : 0.f;
    }
    __syncthreads();
    // conv3's gradient
    for (int s = 0; s < ns; ++s) {
      const float* hc = f32(s, TS_H2F) + c2 * H2F_C;
      float h[5][5];
#pragma unroll
      for (int r = 0; r < 5; ++r) {
        const float4 q = *reinterpret_cast<const float4*>(hc + r * H2F_P);
        h[r][0] = q.x;
        h[r][1] = q.y;
        h[r][2] = q.z;
        h[r][3] = q.w;
        h[r][4] = hc[r * H2F_P + 4];
      }
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const float4 d =
            *reinterpret_cast<const float4*>(f32(s, TS_DA3) + p * 32 + 4 * og);
        const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          b3[a] += dv[a];
#pragma unroll
          for (int k = 0; k < 9; ++k)
            g3[a][k] += dv[a] * h[2 * (p >> 1) + k / 3][2 * (p & 1) + k % 3];
        }
      }
    }
    // da2: lane = input channel, the 2x2 pixels of block (i, j) = wq
    if (live) {
      const int i = wq >> 1, j = wq & 1;
      const float* d3 = f32(ws, TS_DA3);
      float o00 = 0.f, o01 = 0.f, o10 = 0.f, o11 = 0.f;
#pragma unroll 2
      for (int o = 0; o < 32; o += 4) {
        auto da = [&](int ii, int jj) {
          return ii < 2 && jj < 2
                     ? *reinterpret_cast<const float4*>(d3 + (2 * ii + jj) * 32 + o)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        const float4 A = da(i, j), B = da(i, j + 1), C = da(i + 1, j), D = da(i + 1, j + 1);
        const float av[4] = {A.x, A.y, A.z, A.w}, bv[4] = {B.x, B.y, B.z, B.w};
        const float cv[4] = {C.x, C.y, C.z, C.w}, dv[4] = {D.x, D.y, D.z, D.w};
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          uint32_t w[9];
#pragma unroll
          for (int k = 0; k < 9; ++k) w[k] = w3t[(o / 2 + q) * 288 + k * 32 + lane];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int z = 2 * q + e;
            auto wt = [&](int u, int v) { return e ? bf_hi(w[3 * u + v]) : bf_lo(w[3 * u + v]); };
            o00 += wt(1, 1) * av[z];
            o01 += wt(1, 2) * av[z] + wt(1, 0) * bv[z];
            o10 += wt(2, 1) * av[z] + wt(0, 1) * cv[z];
            o11 += wt(2, 2) * av[z] + wt(2, 0) * bv[z] + wt(0, 2) * cv[z] + wt(0, 0) * dv[z];
          }
        }
      }
      const uint16_t* hb = u16(ws, TS_H2) + lane * H2P * H2P;
      float* d2 = f32(ws, TS_DA2) + lane;
      auto put = [&](int yy, int xx, float v) {
        d2[(4 * yy + xx) * 32] = bf2f(hb[(yy + 1) * H2P + xx + 1]) > 0.f ? v : 0.f;
      };
      put(2 * i, 2 * j, o00);
      put(2 * i, 2 * j + 1, o01);
      put(2 * i + 1, 2 * j, o10);
      put(2 * i + 1, 2 * j + 1, o11);
    }
    __syncthreads();
    // conv2's gradient, by output rows
    for (int si = 0; si < 4 * ns; ++si) {
      const int s = si >> 2, i = si & 3;
      const float* hc = f32(s, TS_H1F) + c2 * H1F_C + 2 * i * H1F_P;
      float dv[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 d =
            *reinterpret_cast<const float4*>(f32(s, TS_DA2) + (4 * i + j) * 32 + 4 * og);
        dv[j][0] = d.x;
        dv[j][1] = d.y;
        dv[j][2] = d.z;
        dv[j][3] = d.w;
#pragma unroll
        for (int a = 0; a < 4; ++a) b2[a] += dv[j][a];
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const float4 q0 = *reinterpret_cast<const float4*>(hc + u * H1F_P);
        const float4 q1 = *reinterpret_cast<const float4*>(hc + u * H1F_P + 4);
        const float h[9] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, hc[u * H1F_P + 8]};
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int v = 0; v < 3; ++v)
#pragma unroll
            for (int a = 0; a < 4; ++a) g2[a][3 * u + v] += dv[j][a] * h[2 * j + v];
      }
    }
    // da1: lane = input channel, pixel rows 2 i, 2 i + 1 of row i = wq
    if (live) {
      const int i = wq;
      const float* d2 = f32(ws, TS_DA2);
      float o[2][8];
#pragma unroll
      for (int k = 0; k < 8; ++k) o[0][k] = o[1][k] = 0.f;
#pragma unroll 1
      for (int oc = 0; oc < 32; oc += 4) {
        float dv[2][5][4];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int j = 0; j < 5; ++j) {
            const float4 d = j < 4 && i + r < 4
                                 ? *reinterpret_cast<const float4*>(d2 + (4 * (i + r) + j) * 32 + oc)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
            dv[r][j][0] = d.x;
            dv[r][j][1] = d.y;
            dv[r][j][2] = d.z;
            dv[r][j][3] = d.w;
          }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          uint32_t w[9];
#pragma unroll
          for (int k = 0; k < 9; ++k) w[k] = w2t[(oc / 2 + q) * 288 + k * 32 + lane];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int z = 2 * q + e;
            float wt[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) wt[k] = e ? bf_hi(w[k]) : bf_lo(w[k]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float A = dv[0][j][z], B = dv[0][j + 1][z];
              const float C = dv[1][j][z], D = dv[1][j + 1][z];
              o[0][2 * j] += wt[4] * A;
              o[0][2 * j + 1] += wt[5] * A + wt[3] * B;
              o[1][2 * j] += wt[7] * A + wt[1] * C;
              o[1][2 * j + 1] += wt[8] * A + wt[6] * B + wt[2] * C + wt[0] * D;
            }
          }
        }
      }
      const uint16_t* hb = u16(ws, TS_H1) + lane * H1P * H1P;
      float* d1 = f32(ws, TS_DA1) + lane;
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k = 0; k < 8; ++k)
          d1[(8 * (2 * i + r) + k) * 32] =
              bf2f(hb[(2 * i + r + 1) * H1P + k + 1]) > 0.f ? o[r][k] : 0.f;
    }
    __syncthreads();
    // conv1's gradient: output row `warp`
    for (int s = 0; s < ns; ++s) {
      const float* hc = f32(s, TS_XF) + ci * XF_C + 2 * warp * XF_P;
      float dv[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 d =
            *reinterpret_cast<const float4*>(f32(s, TS_DA1) + (8 * warp + j) * 32 + 4 * og);
        dv[j][0] = d.x;
        dv[j][1] = d.y;
        dv[j][2] = d.z;
        dv[j][3] = d.w;
#pragma unroll
        for (int a = 0; a < 4; ++a) b1[a] += dv[j][a];
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        float h[17];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 q = *reinterpret_cast<const float4*>(hc + u * XF_P + 4 * k);
          h[4 * k] = q.x;
          h[4 * k + 1] = q.y;
          h[4 * k + 2] = q.z;
          h[4 * k + 3] = q.w;
        }
        h[16] = hc[u * XF_P + 16];
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int v = 0; v < 3; ++v)
#pragma unroll
            for (int a = 0; a < 4; ++a) g1[a][3 * u + v] += dv[j][a] * h[2 * j + v];
      }
    }
    __syncthreads();
  }

  // the CTA's gradient in the master layout, then one add per parameter
  float* G = reinterpret_cast<float*>(dsm);
  for (int i = tid; i < M_W2; i += blockDim.x) G[i] = 0.f;   // conv1: eight warps' sums
  __syncthreads();
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int o = 4 * og + a;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      atomicAdd(&G[M_W1 + o * 36 + ci * 9 + k], g1[a][k]);
      G[M_W2 + o * 288 + c2 * 9 + k] = g2[a][k];
      G[M_W3 + o * 288 + c2 * 9 + k] = g3[a][k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) G[M_W4 + (n4 + a) * 128 + k8 + k] = g4[a][k];
    if (ci == 0) atomicAdd(&G[M_B1 + o], b1[a]);
    if (c2 == 0) {
      G[M_B2 + o] = b2[a];
      G[M_B3 + o] = b3[a];
    }
    if (k8 == 0) G[M_B4 + n4 + a] = b4[a];
  }
  if (tid < 192) G[M_W5 + tid] = g5;
  if (tid < 3) G[M_B5 + tid] = b5;
  if (lane == 0 && wq == 0) atomicAdd(loss_sum, lsum);
  __syncthreads();
  // CTAs start at different parameters, so that few meet at one address
  const int rot = (int)((long long)blockIdx.x * N_MASTER / gridDim.x);
  for (int i = tid; i < N_MASTER; i += blockDim.x) {
    int e = i + rot;
    if (e >= N_MASTER) e -= N_MASTER;
    if (G[e] != 0.f) atomicAdd(&grad[e], G[e]);
  }
}

}  // namespace net
}  // namespace vio
