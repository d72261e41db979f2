// kvq_quant_error: the reconstruction-error analysis of the cache quantizer in one pass over new K and V
// (Sec. 4.1 experiment (i); MSE(A, A^) = ||A - A^||_F^2 / entries, App. B.4).  Every token row is quantized in
// registers exactly as kvq_quantize_append would (same group parameters, same codes), reconstructed as
// x^ = fmaf(code, scale, zero) and compared with the input; nothing packed is written.  Per (batch, kv-head)
// the kernel adds sum x^2 and sum (x - x^)^2 of keys and of values to four doubles.
#include <math.h>

#include <type_traits>

#include "kvq_quantize.cuh"

namespace kvq {

namespace {

__device__ __forceinline__ __half2 as_half2(uint32_t u) { return *reinterpret_cast<const __half2*>(&u); }

constexpr int kThreads = 128;
constexpr int kPerSm = 12;

// One side (keys: blockIdx.z = 0, values: 1).  A row of D channels is spread over D/8 lanes, 8 channels each, and a lane
// takes the same channels of four rows at a time.  Minimum and negated maximum of a group travel as one pair of the 16-bit
// input type (exact), reduced so that every lane of a group ends up with one of the four rows: the parameters (two
// divisions) are made once per lane and row and fetched from there.  Where all groups of a warp are plain (see plain_group) codes need
// no clamp; the magic number is added by a fused multiply-add (see code_word4); two neighbouring channels share every fp32 operation
// that has a packed form, and a row's squares are added as two chains of four.  20 M elements a call (80 streams x 1000 tokens x 128, K
// and V), twelve calls in a row: 191 us without packed operations, 174 with clamps, 169 now; 64-bit comparison of the sums 1.2e-8 at
// first, 1.0e-8 now.  Bound by the fp32 pipes and issue (72 % of the slots; twelve CTAs per SM, each three turns of rows).  Not faster: 256
// threads a CTA 186, eight CTAs per SM 179, eight rows per lane 196, longer fp32 sums, compensated fp32 sums in place of doubles, the
// next turn's rows in flight at eight CTAs per SM.  162 us without the rounding of x^, which is part of the error, however.
template <int D, int DTYPE>
__global__ void __launch_bounds__(kThreads, kPerSm)
quant_error_kernel(Geom g, const uint16_t* __restrict__ k, const uint16_t* __restrict__ v, int64_t sb, int64_t sh,
                   int64_t st, int n_tokens, double* __restrict__ sums) {
  using H2 = typename Pair16<DTYPE>::type;
  constexpr int LPR = D / 8, RPW = 32 / LPR, ROWS = 4;   // lanes per row, rows per warp and load, rows per lane
  constexpr int kStep = (kThreads / 32) * RPW * ROWS;    // rows per CTA and turn
  __shared__ double part[2][kThreads / 32];
  const int side = blockIdx.z;
  const int bh = blockIdx.y, b = bh / g.Hkv, h = bh % g.Hkv;
  const int bits = side ? g.vb : g.kb, gsz = side ? g.gv : g.gk;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l = lane % LPR, r0 = warp * RPW + lane / LPR;
  const uint16_t* in = (side ? v : k) + (int64_t)b * sb + (int64_t)h * sh + 8 * l;
  const int lpg = gsz >> 3;                              // lanes per group: 4, 8 or 16
  const int b0 = lane & 1, b1 = (lane >> 1) & 1, gbase = lane & ~(lpg - 1);
  const float qmax = (float)((1 << (bits & 15)) - 1), up = (float)(1 << (bits & 15)), down = 1.0f / up, rtop = kRoundMagic + qmax;
  double acc2 = 0.0, acce = 0.0;
  begin_after_predecessor();
  for (int base = blockIdx.x * kStep; base < n_tokens; base += gridDim.x * kStep) {
    uint4 raw[ROWS];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const int t = base + i * (kStep / ROWS) + r0;      // rows beyond the end are zeros and add nothing
      raw[i] = t < n_tokens ? *reinterpret_cast<const uint4*>(in + (int64_t)t * st) : make_uint4(0u, 0u, 0u, 0u);
    }
    uint32_t meta = 0u;                                  // of the lane's row: scale and zero, 2^-bits / scale
    float inv = 0.f;
    auto parameters = [&](auto nans_tag) {               // whether the group is plain (nans: see minmax8)
      constexpr bool nans = decltype(nans_tag)::value;
      H2 m[ROWS];                                        // (minimum, - maximum) of the lane's channels
#pragma unroll
      for (int i = 0; i < ROWS; ++i) m[i] = minmax8<DTYPE, nans>(raw[i]);
      auto swap = [](H2 x, int off) {
        const uint32_t o = __shfl_xor_sync(FULL, *reinterpret_cast<uint32_t*>(&x), off);
        return *reinterpret_cast<const H2*>(&o);
      };
      // the first two steps hand half of the rows to the lane opposite: the lane keeps row 2 b0 + b1
      const H2 a0 = min_pair(b0 ? m[2] : m[0], swap(b0 ? m[0] : m[2], 1), nans);
      const H2 a1 = min_pair(b0 ? m[3] : m[1], swap(b0 ? m[1] : m[3], 1), nans);
      H2 a = min_pair(b1 ? a1 : a0, swap(b1 ? a0 : a1, 2), nans);
      const H2 a4 = swap(a, 4);
      if (lpg >= 8) a = min_pair(a, a4, nans);
      const H2 a8 = swap(a, 8);
      if (lpg >= 16) a = min_pair(a, a8, nans);
      const float2 f = pair_to_f32(a);
      const GroupParams p = group_params(f.x, -f.y, qmax);
      meta = p.meta; inv = p.inv * down;
      return plain_group(f.x, -f.y, p, qmax);
    };
    f32x2 s2[ROWS], se[ROWS];                            // sums over the even and the odd channels of a row
    auto add_rows = [&](auto plain_tag) {
      constexpr bool plain = decltype(plain_tag)::value;
#pragma unroll
      for (int i = 0; i < ROWS; ++i) {
        const int src = gbase + (i >> 1) + 2 * (i & 1);  // the lane of the group that holds row i
        const float2 sz = __half22float2(as_half2(__shfl_sync(FULL, meta, src)));
        const float ii = __shfl_sync(FULL, inv, src);
        const f32x2 si = pack2(sz.x, sz.x), zi = pack2(sz.y, sz.y), nz = pack2(-sz.y, -sz.y);
        const H2* p = reinterpret_cast<const H2*>(&raw[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 f = pair_to_f32(p[j]);
          const f32x2 x = pack2(f.x, f.y);
          s2[i] = j ? fma2(x, x, s2[i]) : mul2(x, x);
          const f32x2 t = add2(x, nz);
          f32x2 r;
          if constexpr (plain) {
            r = fma2(mul2(t, pack2(ii, ii)), pack2(up, up), pack2(kRoundMagic, kRoundMagic));
          } else {
            const float2 tf = unpack2(t);
            const float2 rf = unpack2(fma2(pack2(__saturatef(__fmul_rn(tf.x, ii)), __saturatef(__fmul_rn(tf.y, ii))), pack2(up, up), pack2(kRoundMagic, kRoundMagic)));
            r = pack2(fminf(rf.x, rtop), fminf(rf.y, rtop));
          }
          const f32x2 code = add2(r, pack2(-kRoundMagic, -kRoundMagic));
          const f32x2 d = fma2(fma2(code, si, zi), pack2(-1.0f, -1.0f), x);      // (the rounding of x^ belongs to the error)
          se[i] = j ? fma2(d, d, se[i]) : mul2(d, d);
        }
      }
    };
    if (bits == 16 || __all_sync(FULL, parameters(std::true_type{}))) {
      add_rows(std::true_type{});
    } else {
      parameters(std::false_type{});
      add_rows(std::false_type{});
    }
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const float2 ts = unpack2(s2[i]), te = unpack2(se[i]);
      acc2 += (double)__fadd_rn(ts.x, ts.y);
      acce += (double)__fadd_rn(te.x, te.y);
    }
  }
  if (bits == 16) acce = 0.0;                            // passed through: no error
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    acc2 += __shfl_xor_sync(FULL, acc2, off);
    acce += __shfl_xor_sync(FULL, acce, off);
  }
  if (lane == 0) { part[0][warp] = acc2; part[1][warp] = acce; }
  __syncthreads();
  if (threadIdx.x < 2) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) t += part[threadIdx.x][w];
    atomicAdd(sums + (size_t)bh * 4 + 2 * side + threadIdx.x, t);
  }
}

}  // namespace

int launch_quant_error(const Geom& g, const void* k, const void* v, int64_t sb, int64_t sh, int64_t st, int n_tokens,
                       double* sums, cudaStream_t stream) {
  const int streams = g.B * g.Hkv;
  const uint16_t* kk = static_cast<const uint16_t*>(k);
  const uint16_t* vv = static_cast<const uint16_t*>(v);
  // one wave of CTAs, no more of them than turns of rows (twelve calls when this was chosen: 12 CTAs of 128 threads per SM
  // 188 us, 8: 198 us)
  const int step = (kThreads / 32) * (32 / (g.D / 8)) * 4;
  int gx = (n_tokens + step - 1) / step, want = 148 * kPerSm / (2 * streams);
  if (want < 1) want = 1;
  if (gx > want) gx = want;
  auto launch = [&](auto kern) {
    return launch_dependent(kern, dim3(gx, streams, 2), kThreads, 0, stream, 1, g, kk, vv, sb, sh, st, n_tokens, sums);
  };
  const bool bf = g.in_dtype == KVQ_BF16;
  const cudaError_t e = g.D == 128 ? launch(bf ? quant_error_kernel<128, KVQ_BF16> : quant_error_kernel<128, KVQ_FP16>)
                                   : launch(bf ? quant_error_kernel<64, KVQ_BF16> : quant_error_kernel<64, KVQ_FP16>);
  return e == cudaSuccess ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
}

}  // namespace kvq
