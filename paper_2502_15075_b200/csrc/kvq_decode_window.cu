// Decode attention over the residual window (Sec. 4.1's buffer of recent full-precision tokens): the newest
// seq_len % R tokens of a stream are 16-bit rows in a ring, not pages.  One CTA per (batch, kv-head) stream computes
// softmax-attention partials (m, l, o) of all (row, head) pairs over those at most R - 1 tokens in fp32 and leaves
// them in the stream's last partial slot, where the main kernel's merge picks them up; a stream without pages gets
// its output written here.
// Runs in front of the tcgen05 kernel only; the warp-level kernel takes the window itself (window_partial in kvq_decode_mma_kernel.cuh).
//
// At most 64 KB per stream, so latency is all there is: every thread loads its share of the keys and of the values (16-byte
// pieces) before it computes anything.  Logits: four lanes per token, a quarter of the channels each, four heads at once.  Values:
// D / 8 lanes per row, 8 channels x four heads in registers, summed over the token groups through shared memory.  A decode call over
// 32 sequences x 8 KV heads of 63 window tokens and no pages, 4 query heads each, replayed: 73 us with a thread per (head, token)
// and per (head, channel) and 2-byte loads, 14 us now (the launch of the page kernel, which finds nothing to do, included).
#include "kvq_internal.h"

namespace kvq {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxR = 128;

template <int D, int DTYPE>
__global__ void __launch_bounds__(kThreads)
decode_window_kernel(Geom g, CachePtrs c, const uint16_t* __restrict__ q, float c1, float* __restrict__ ws, int s_cap,
                     void* __restrict__ out, int out_dtype) {
  constexpr int Q = D / 4, QP = Q + 4;                     // channels per lane of a token; padded: the quarters on different banks
  constexpr int KP = kMaxR / (kThreads / 4), KV = Q / 8;   // token passes of the logits, 16-byte pieces per lane and token
  constexpr int LPR = D / 8, NG = kThreads / LPR;          // lanes per value row, token groups
  constexpr int VH = kMaxGroupHeads;                       // (row, head) pairs per KV head, taken four at a time
  constexpr int VP = kMaxR / NG, NRED = kThreads / 32;     // value rows per thread; one sum per warp
  __shared__ __align__(16) float sq[VH][4][QP];            // queries, prescaled (softmax scale * log2 e)
  __shared__ __align__(16) float sp[kMaxR][VH];            // logits, then weights
  __shared__ __align__(16) float so[NRED][VH][D];
  __shared__ float sm[VH], sl[VH];
  const int stream = blockIdx.x, b = stream / g.Hkv, h = stream % g.Hkv;
  const int R = g.R, Gq = g.G, nvh = g.G * g.rows;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  begin_after_predecessor();
  const int n = clamped_len(c.seq_len, b, g.capacity);
  const int f = (n / R) * R, nw = n - f;     // tokens f .. n-1 are in the window, in the ring's slots 0 .. nw-1
  auto out_index = [&](int vh, int d) {
    return (((size_t)b * g.rows + vh / Gq) * g.Hq + (size_t)h * Gq + vh % Gq) * D + d;
  };
  auto store_out = [&](size_t oi, float r) {
    if (out_dtype == KVQ_FP32) static_cast<float*>(out)[oi] = r;
    else static_cast<uint16_t*>(out)[oi] = f32_to_bits16(r, out_dtype);
  };
  if (nw == 0) {
    if (n == 0) {                            // an empty sequence: zeros
      for (int idx = tid; idx < nvh * D; idx += kThreads) store_out(out_index(idx / D, idx % D), 0.f);
    }
    return;
  }
  auto unpack = [](const uint4& r, float (&x)[8]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[2 * i] = bits16_to_f32((uint16_t)(w[i] & 0xFFFF), DTYPE);
      x[2 * i + 1] = bits16_to_f32((uint16_t)(w[i] >> 16), DTYPE);
    }
  };
  // ---- all loads of the window (key row, value row of slot i side by side)
  const uint16_t* win = c.kv_win + (size_t)stream * R * 2 * D;
  const int kt = tid >> 2, kq = tid & 3, vg = tid / LPR, vl = tid % LPR;
  uint4 kraw[KP][KV], vraw[VP];
#pragma unroll
  for (int p = 0; p < KP; ++p) {
    const int i = kt + p * (kThreads / 4);
#pragma unroll
    for (int j = 0; j < KV; ++j)
      kraw[p][j] = i < nw ? *reinterpret_cast<const uint4*>(win + (size_t)i * 2 * D + kq * Q + 8 * j) : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int p = 0; p < VP; ++p) {
    const int i = vg + p * NG;
    vraw[p] = i < nw ? *reinterpret_cast<const uint4*>(win + (size_t)i * 2 * D + D + 8 * vl) : make_uint4(0u, 0u, 0u, 0u);
  }
  for (int idx = tid; idx < VH * D; idx += kThreads) {
    const int vh = idx / D, d = idx % D;
    float x = 0.f;
    if (vh < nvh) x = bits16_to_f32(q[out_index(vh, d)], g.in_dtype) * c1;
    sq[vh][d / Q][d % Q] = x;
  }
  __syncthreads();
  // ---- logits
#pragma unroll
  for (int p = 0; p < KP; ++p) {
    const int i = kt + p * (kThreads / 4);
    if (p * (kThreads / 4) >= nw) break;     // (whole CTA)
#pragma unroll 1
    for (int v0 = 0; v0 < nvh; v0 += 4) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < KV; ++j) {
        float x[8];
        unpack(kraw[p][j], x);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4 a = *reinterpret_cast<const float4*>(&sq[v0 + e][kq][8 * j]);
          const float4 z = *reinterpret_cast<const float4*>(&sq[v0 + e][kq][8 * j + 4]);
          acc[e] = fmaf(a.x, x[0], fmaf(a.y, x[1], fmaf(a.z, x[2], fmaf(a.w, x[3], acc[e]))));
          acc[e] = fmaf(z.x, x[4], fmaf(z.y, x[5], fmaf(z.z, x[6], fmaf(z.w, x[7], acc[e]))));
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 1);
        acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 2);
        // causal limit of the pair's query row; the token's four lanes store a pair each
        const int limit = n - (g.rows - 1 - min((v0 + e) / Gq, g.rows - 1));
        if (e == kq && i < nw) sp[i][v0 + e] = f + i < limit ? acc[e] : -INFINITY;
      }
    }
  }
  __syncthreads();
  // ---- softmax of one pair per warp
  if (warp < nvh) {
    float x[kMaxR / 32], m = -INFINITY, sum = 0.f;
#pragma unroll
    for (int u = 0; u < kMaxR / 32; ++u) {
      const int i = lane + 32 * u;
      x[u] = i < nw ? sp[i][warp] : -INFINITY;
      m = fmaxf(m, x[u]);
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
#pragma unroll
    for (int u = 0; u < kMaxR / 32; ++u) {
      const int i = lane + 32 * u;
      const float p = (m == -INFINITY || i >= nw) ? 0.f : exp2f(x[u] - m);
      if (i < nw) sp[i][warp] = p;
      sum += p;
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (lane == 0) { sm[warp] = m; sl[warp] = sum; }
  }
  __syncthreads();
  // ---- weighted values: this thread's rows, then the groups of its warp, then the warps
#pragma unroll 1
  for (int v0 = 0; v0 < nvh; v0 += 4) {
    float o[4][8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
#pragma unroll
      for (int j = 0; j < 8; ++j) o[e][j] = 0.f;
    }
#pragma unroll
    for (int p = 0; p < VP; ++p) {
      const int i = vg + p * NG;
      if (i < nw) {
        float x[8];
        unpack(vraw[p], x);
        const float4 w4 = *reinterpret_cast<const float4*>(&sp[i][v0]);      // (pairs beyond nvh: never stored)
        const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
          for (int j = 0; j < 8; ++j) o[e][j] = fmaf(w[e], x[j], o[e][j]);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
#pragma unroll
        for (int off = LPR; off < 32; off <<= 1) o[e][j] += __shfl_xor_sync(0xffffffffu, o[e][j], off);
      }
      if (lane < LPR) {
        *reinterpret_cast<float4*>(&so[warp][v0 + e][8 * vl]) = make_float4(o[e][0], o[e][1], o[e][2], o[e][3]);
        *reinterpret_cast<float4*>(&so[warp][v0 + e][8 * vl + 4]) = make_float4(o[e][4], o[e][5], o[e][6], o[e][7]);
      }
    }
  }
  __syncthreads();
  for (int idx = tid; idx < nvh * D; idx += kThreads) {
    const int vh = idx / D, d = idx % D;
    float r = 0.f;
#pragma unroll
    for (int w = 0; w < NRED; ++w) r += so[w][vh][d];
    if (f == 0) {                            // no pages at all: this is the whole attention
      store_out(out_index(vh, d), sl[vh] > 0.f ? r / sl[vh] : 0.f);
    } else {
      float* dst = ws + (((size_t)stream * s_cap + (s_cap - 1)) * nvh + vh) * (D + 2);
      if (d == 0) { dst[0] = sm[vh]; dst[1] = sl[vh]; }
      dst[2 + d] = r;
    }
  }
}

}  // namespace

int launch_decode_window(const Geom& g, const CachePtrs& c, const void* q, void* out, int out_dtype, float c1,
                         float* ws, int s_cap, cudaStream_t stream) {
  const uint16_t* qq = static_cast<const uint16_t*>(q);
  const dim3 grid(g.B * g.Hkv);
  auto launch = [&](auto kern) { return launch_dependent(kern, grid, kThreads, 0, stream, 1, g, c, qq, c1, ws, s_cap, out, out_dtype); };
  const bool bf = g.in_dtype == KVQ_BF16;
  const cudaError_t e = g.D == 128 ? launch(bf ? decode_window_kernel<128, KVQ_BF16> : decode_window_kernel<128, KVQ_FP16>)
                                   : launch(bf ? decode_window_kernel<64, KVQ_BF16> : decode_window_kernel<64, KVQ_FP16>);
  return e == cudaSuccess ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
}

}  // namespace kvq
