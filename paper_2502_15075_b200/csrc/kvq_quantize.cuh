// Device functions that the quantize-append kernels and the error analysis share: minima and maxima of 16-bit pairs, rounding
// and packing of codes, and a complete 128-token block of channel-wise keys.
#pragma once

#include "kvq_internal.h"

namespace kvq {

constexpr uint32_t FULL = 0xffffffffu;
constexpr float kRoundMagic = 12582912.0f;   // 1.5 * 2^23: adding it rounds to nearest-even at integer precision

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// Two 16-bit inputs as a packed pair of their own type, for exact minima and maxima.
template <int DTYPE> struct Pair16 { using type = __half2; };
template <> struct Pair16<KVQ_BF16> { using type = __nv_bfloat162; };
__device__ __forceinline__ float2 pair_to_f32(__half2 h) { return __half22float2(h); }
__device__ __forceinline__ float2 pair_to_f32(__nv_bfloat162 h) { return __bfloat1622float2(h); }
__device__ __forceinline__ __half2 lows(__half2 a, __half2 b) { return __lows2half2(a, b); }
__device__ __forceinline__ __half2 highs(__half2 a, __half2 b) { return __highs2half2(a, b); }
__device__ __forceinline__ __nv_bfloat162 lows(__nv_bfloat162 a, __nv_bfloat162 b) { return __lows2bfloat162(a, b); }
__device__ __forceinline__ __nv_bfloat162 highs(__nv_bfloat162 a, __nv_bfloat162 b) { return __highs2bfloat162(a, b); }

// (minimum, - maximum) of the eight values of a 16-byte piece.  NANS: a NaN among them makes both NaN, else it is passed over.
__device__ __forceinline__ __half2 min_pair(__half2 a, __half2 b, bool nans) { return nans ? __hmin2_nan(a, b) : __hmin2(a, b); }
__device__ __forceinline__ __half2 max_pair(__half2 a, __half2 b, bool nans) { return nans ? __hmax2_nan(a, b) : __hmax2(a, b); }
__device__ __forceinline__ __nv_bfloat162 min_pair(__nv_bfloat162 a, __nv_bfloat162 b, bool nans) { return nans ? __hmin2_nan(a, b) : __hmin2(a, b); }
__device__ __forceinline__ __nv_bfloat162 max_pair(__nv_bfloat162 a, __nv_bfloat162 b, bool nans) { return nans ? __hmax2_nan(a, b) : __hmax2(a, b); }
template <int DTYPE, bool NANS = false>
__device__ __forceinline__ typename Pair16<DTYPE>::type minmax8(const uint4& r) {
  using H2 = typename Pair16<DTYPE>::type;
  const H2* h = reinterpret_cast<const H2*>(&r);
  const H2 lo = min_pair(min_pair(h[0], h[1], NANS), min_pair(h[2], h[3], NANS), NANS);
  const H2 hi = __hneg2(max_pair(max_pair(h[0], h[1], NANS), max_pair(h[2], h[3], NANS), NANS));
  return min_pair(lows(lo, hi), highs(lo, hi), NANS);
}

// An append of t_new tokens at position t0 fits the cache; written without a sum that could overflow.
__host__ __device__ __forceinline__ bool append_fits(int t0, int t_new, int capacity) {
  return t0 >= 0 && t0 <= capacity - t_new;
}

// The 16-byte pieces (eight channels 8 v .. 8 v + 7, v = tid % 16) of new key rows as saturated fp16, rotated if asked.
// The 16 lanes of a row take part together (the rotation shuffles between them).
template <int DTYPE, bool ROT>
__device__ __forceinline__ uint4 key_row_fp16(uint4 val, const int8_t* __restrict__ signs, int v) {
  if constexpr (DTYPE == KVQ_BF16 || ROT) {
    uint32_t w[4] = {val.x, val.y, val.z, val.w};
    float x[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (DTYPE == KVQ_BF16) {
        x[2 * i] = __uint_as_float(w[i] << 16);
        x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
      } else {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
        x[2 * i] = f.x;
        x[2 * i + 1] = f.y;
      }
    }
    if constexpr (ROT) rotate_row8<128>(x, signs, v);
    // saturating: the conversion rounds to nearest (infinity from 65520 on), the packed clamp brings infinities to 65504
    const __half2 top = __half2half2(__ushort_as_half(0x7BFF)), bottom = __half2half2(__ushort_as_half(0xFBFF));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __half2 h = __hmin2(__hmax2(__floats2half2_rn(x[2 * i], x[2 * i + 1]), bottom), top);
      w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  } else {
    return val;
  }
}

// Codes of four values as the four bytes of a word: rint(clamp((x - z) * inv, 0, qmax)), the fixed formula.  `inv_q` is
// inv * 2^-BITS (exact), so that the saturation of a multiplication to [0, 1] is the clamp to [0, 2^BITS] (a NaN becomes
// 0); the fused multiply-add by 2^BITS onto 1.5 * 2^23 rounds to nearest-even, and the upper clamp follows on two codes at a time.
template <int BITS>
__device__ __forceinline__ uint32_t code_word4(const float (&x)[4], const float (&z)[4], const float (&inv_q)[4]) {
  uint32_t n[4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    n[j] = __float_as_uint(__fmaf_rn(__saturatef(__fmul_rn(__fsub_rn(x[j], z[j]), inv_q[j])), (float)(1 << BITS), kRoundMagic));
  constexpr uint32_t TOP = ((1u << BITS) - 1u) * 0x00010001u;
  const uint32_t even = __vminu2(prmt(n[0], n[2], 0x5410), TOP), odd = __vminu2(prmt(n[1], n[3], 0x5410), TOP);
  return even + odd * 256u;
}

// Whether no value of a group needs a clamp: the values of its codes before rounding grow with x, so they all round to 0 .. qmax when
// those of its minimum and maximum do.  True for every group of 16-bit values whose minimum and scale are normal fp16 numbers (the
// zero-point is then the minimum itself, and a scale rounded down takes the maximum to qmax (1 + 2^-11) at most); false for a NaN.
__device__ __forceinline__ bool plain_group(float mn, float mx, const GroupParams& p, float qmax) {
  return __fmul_rn(__fsub_rn(mn, p.z), p.inv) >= -0.5f && __fmul_rn(__fsub_rn(mx, p.z), p.inv) < qmax + 0.5f;
}

// Codes of four values of plain groups as the four bytes of a word, two values per operation: rint((x - z) * inv) in the low bits of
// the sum with 1.5 * 2^23.  nz: minus the zero-points; inv_q: inv * 2^-BITS, as above (a product by inv itself and the sum behind it
// would be contracted to one operation with one rounding, although both ask for their own).
template <int BITS>
__device__ __forceinline__ uint32_t code_word4_plain(f32x2 x01, f32x2 x23, f32x2 nz01, f32x2 nz23, f32x2 inv01, f32x2 inv23) {
  const f32x2 magic = pack2(kRoundMagic, kRoundMagic), up = pack2((float)(1 << BITS), (float)(1 << BITS));
  const float2 a = unpack2(fma2(mul2(add2(x01, nz01), inv01), up, magic)), b = unpack2(fma2(mul2(add2(x23, nz23), inv23), up, magic));
  return prmt(prmt(__float_as_uint(a.x), __float_as_uint(a.y), 0x0040), prmt(__float_as_uint(b.x), __float_as_uint(b.y), 0x0040), 0x5410);
}

// Clamped codes as in code_word4, two values per operation and of one group: for rotated keys, whose groups are not looked at for plain ones.
template <int BITS>
__device__ __forceinline__ uint32_t code_word4_packed(const float (&x)[4], float z, float inv_q) {
  uint32_t n[4];
  constexpr float UP = (float)(1 << BITS);
#pragma unroll
  for (int j = 0; j < 4; j += 2) {
    const float2 t = unpack2(add2(pack2(x[j], x[j + 1]), pack2(-z, -z)));
    const f32x2 u = pack2(__saturatef(__fmul_rn(t.x, inv_q)), __saturatef(__fmul_rn(t.y, inv_q)));
    const float2 r = unpack2(fma2(u, pack2(UP, UP), pack2(kRoundMagic, kRoundMagic)));
    n[j] = __float_as_uint(r.x);
    n[j + 1] = __float_as_uint(r.y);
  }
  constexpr uint32_t TOP = ((1u << BITS) - 1u) * 0x00010001u;
  const uint32_t even = __vminu2(prmt(n[0], n[2], 0x5410), TOP), odd = __vminu2(prmt(n[1], n[3], 0x5410), TOP);
  return even + odd * 256u;
}

// Channel-wise quantization of one complete 128-token block, head_dim 128, 4- or 8-bit codes, held in the registers of
// 256 threads: thread (tr = tid / 16, v = tid % 16) has channels 8 v .. 8 v + 7 of tokens tr + 16 i as fp16.  Minimum and
// maximum are taken two channels at a time in fp16 (exact), first in the thread, then over the warps through 4 KB of
// shared memory; the parameters are made once per channel.  At 4 bits the lanes whose codes share bytes (v and v ^ 2) swap one word
// per token, and each stores one word of the row: the 16 lanes of a row write its 64 (8 bits: 128) bytes whole.
struct KchanShared {
  uint4 mn[8][16], mx[8][16];       // per warp: the eight channels of each v
  __align__(16) float2 par[128];    // (zero, 2^-KB / scale) per channel, or both for two channels at a time
};
template <int KB>
__device__ __forceinline__ void kchan_block(const uint4 (&val)[8], KchanShared& sh, uint8_t* __restrict__ pg, const Geom& g, int tid) {
  constexpr int ROW = 128 * KB / 8;
  const int tr = tid >> 4, v = tid & 15, warp = tid >> 5, lane = tid & 31;
  __half2 mn[4], mx[4];
  auto h2 = [](uint32_t u) { return *reinterpret_cast<const __half2*>(&u); };
  auto u32 = [](__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); };
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t w[4] = {val[i].x, val[i].y, val[i].z, val[i].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      mn[j] = i ? __hmin2(mn[j], h2(w[j])) : h2(w[j]);
      mx[j] = i ? __hmax2(mx[j], h2(w[j])) : h2(w[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    mn[j] = __hmin2(mn[j], h2(__shfl_xor_sync(FULL, u32(mn[j]), 16)));
    mx[j] = __hmax2(mx[j], h2(__shfl_xor_sync(FULL, u32(mx[j]), 16)));
  }
  if (lane < 16) {
    sh.mn[warp][v] = make_uint4(u32(mn[0]), u32(mn[1]), u32(mn[2]), u32(mn[3]));
    sh.mx[warp][v] = make_uint4(u32(mx[0]), u32(mx[1]), u32(mx[2]), u32(mx[3]));
  }
  __syncthreads();
  if (tid < 128) {
    const __half* a = reinterpret_cast<const __half*>(sh.mn) + tid;       // channel tid of warp 0
    const __half* b = reinterpret_cast<const __half*>(sh.mx) + tid;
    __half lo = a[0], hi = b[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) { lo = __hmin(lo, a[128 * w]); hi = __hmax(hi, b[128 * w]); }
    const GroupParams p = group_params(__half2float(lo), __half2float(hi), (float)((1 << KB) - 1));
    reinterpret_cast<uint32_t*>(pg + g.k_meta_off)[tid] = p.meta;
    sh.par[tid] = make_float2(p.z, p.inv * (1.0f / (float)(1 << KB)));
  }
  __syncthreads();
  float z[8], inv_q[8];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 p = *reinterpret_cast<const float4*>(&sh.par[8 * v + 2 * j]);
    z[2 * j] = p.x; inv_q[2 * j] = p.y; z[2 * j + 1] = p.z; inv_q[2 * j + 1] = p.w;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t w[4] = {val[i].x, val[i].y, val[i].z, val[i].w};
    uint32_t word[2];
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const float2 f0 = __half22float2(h2(w[2 * hh])), f1 = __half22float2(h2(w[2 * hh + 1]));
      const float x[4] = {f0.x, f0.y, f1.x, f1.y};
      const float zz[4] = {z[4 * hh], z[4 * hh + 1], z[4 * hh + 2], z[4 * hh + 3]};
      const float ii[4] = {inv_q[4 * hh], inv_q[4 * hh + 1], inv_q[4 * hh + 2], inv_q[4 * hh + 3]};
      word[hh] = code_word4<KB>(x, zz, ii);
    }
    uint8_t* row = pg + (tr + 16 * i) * ROW;
    if constexpr (KB == 4) {
      const int rh = v & 1, f = (v >> 1) & 1, mw = v >> 2;
      const uint32_t other = __shfl_xor_sync(FULL, f ? word[0] : word[1], 2);       // the partner's half of the word this lane stores
      *reinterpret_cast<uint32_t*>(row + (2 * rh + f) * 16 + mw * 4) = f ? (other | (word[1] << 4)) : (word[0] | (other << 4));
    } else {
      const int rh = v & 1, mw = v >> 1;
#pragma unroll
      for (int hh = 0; hh < 2; ++hh)
        *reinterpret_cast<uint32_t*>(row + (mw >> 2) * 64 + (2 * rh + hh) * 16 + (mw & 3) * 4) = word[hh];
    }
  }
  __syncthreads();                       // the scratch may be used for another block
}

// The same from the input rows as they are, without conversions, clamps or scalar operations: true, or false with nothing settled where
// a channel of the block is not plain (see plain_group; here also: beyond the fp16 range).  The quantizer sees the keys as fp16 values.
// fp16 inputs are those; a bf16 value within the range is one too unless it lies below the normal fp16 numbers, where it has to be
// rounded to a multiple of 2^-24: the sum with 0.75 does that (its last place is 2^-24 there, and above it holds all of a bf16 value),
// and 0.75 leaves again with the zero-point, whose sum with it is exact as well.  `next` is called when `val` has been read.
template <int DTYPE, int KB, typename Next>
__device__ __forceinline__ bool kchan_block_plain(const uint4 (&val)[8], KchanShared& sh, uint8_t* __restrict__ pg, const Geom& g, int tid, Next&& next) {
  using H2 = typename Pair16<DTYPE>::type;
  constexpr int ROW = 128 * KB / 8;
  constexpr float SHIFT = DTYPE == KVQ_BF16 ? 0.75f : 0.0f, UP = (float)(1 << KB);
  const int tr = tid >> 4, v = tid & 15, warp = tid >> 5, lane = tid & 31;
  auto h2 = [](uint32_t u) { return *reinterpret_cast<const H2*>(&u); };
  auto u32 = [](H2 h) { return *reinterpret_cast<const uint32_t*>(&h); };
  {
    H2 mn[4], mx[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t w[4] = {val[i].x, val[i].y, val[i].z, val[i].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        mn[j] = i ? min_pair(mn[j], h2(w[j]), true) : h2(w[j]);
        mx[j] = i ? max_pair(mx[j], h2(w[j]), true) : h2(w[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      mn[j] = min_pair(mn[j], h2(__shfl_xor_sync(FULL, u32(mn[j]), 16)), true);
      mx[j] = max_pair(mx[j], h2(__shfl_xor_sync(FULL, u32(mx[j]), 16)), true);
    }
    if (lane < 16) {
      sh.mn[warp][v] = make_uint4(u32(mn[0]), u32(mn[1]), u32(mn[2]), u32(mn[3]));
      sh.mx[warp][v] = make_uint4(u32(mx[0]), u32(mx[1]), u32(mx[2]), u32(mx[3]));
    }
  }
  __syncthreads();
  next();
  bool plain = true;
  if (tid < 64) {                        // two channels a thread
    const uint32_t* a = reinterpret_cast<const uint32_t*>(sh.mn) + tid;
    const uint32_t* b = reinterpret_cast<const uint32_t*>(sh.mx) + tid;
    H2 lo = h2(a[0]), hi = h2(b[0]);
#pragma unroll
    for (int w = 1; w < 8; ++w) { lo = min_pair(lo, h2(a[64 * w]), true); hi = max_pair(hi, h2(b[64 * w]), true); }
    const float2 l2 = pair_to_f32(lo), u2 = pair_to_f32(hi);
    const float qmax = (float)((1 << KB) - 1);
    uint2 meta;
    float4 par;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float l = e ? l2.y : l2.x, u = e ? u2.y : u2.x;
      plain &= l >= -65504.0f && u <= 65504.0f;
      const float l16 = __half2float(__ushort_as_half(f32_to_fp16_sat_bits(l))), u16 = __half2float(__ushort_as_half(f32_to_fp16_sat_bits(u)));
      const GroupParams p = group_params(l16, u16, qmax);
      plain &= plain_group(l16, u16, p, qmax);
      (e ? meta.y : meta.x) = p.meta;
      (e ? par.z : par.x) = -(p.z + SHIFT);
      (e ? par.w : par.y) = p.inv * (1.0f / UP);
    }
    reinterpret_cast<uint2*>(pg + g.k_meta_off)[tid] = meta;
    reinterpret_cast<float4*>(sh.par)[tid] = make_float4(par.x, par.z, par.y, par.w);      // (- zero, - zero, 2^-KB / scale, 2^-KB / scale)
  }
  if (!__syncthreads_and(plain)) return false;
  f32x2 nz[4], inv_q[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 p = reinterpret_cast<const float4*>(sh.par)[4 * v + j];
    nz[j] = pack2(p.x, p.y); inv_q[j] = pack2(p.z, p.w);
  }
  const f32x2 up = pack2(UP, UP), magic = pack2(kRoundMagic, kRoundMagic), shift = pack2(SHIFT, SHIFT);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t w[4] = {val[i].x, val[i].y, val[i].z, val[i].w};
    uint32_t pair[4];                    // two codes each, bytes 0 and 1
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = pair_to_f32(h2(w[j]));
      f32x2 x = pack2(f.x, f.y);
      if constexpr (DTYPE == KVQ_BF16) x = add2(x, shift);
      const float2 r = unpack2(fma2(mul2(add2(x, nz[j]), inv_q[j]), up, magic));
      pair[j] = prmt(__float_as_uint(r.x), __float_as_uint(r.y), 0x0040);
    }
    const uint32_t word[2] = {prmt(pair[0], pair[1], 0x5410), prmt(pair[2], pair[3], 0x5410)};
    uint8_t* row = pg + (tr + 16 * i) * ROW;
    if constexpr (KB == 4) {
      const int rh = v & 1, f = (v >> 1) & 1, mw = v >> 2;
      const uint32_t other = __shfl_xor_sync(FULL, f ? word[0] : word[1], 2);       // the partner's half of the word this lane stores
      *reinterpret_cast<uint32_t*>(row + (2 * rh + f) * 16 + mw * 4) = f ? (other | (word[1] << 4)) : (word[0] | (other << 4));
    } else {
      const int rh = v & 1, mw = v >> 1;
#pragma unroll
      for (int hh = 0; hh < 2; ++hh)
        *reinterpret_cast<uint32_t*>(row + (mw >> 2) * 64 + (2 * rh + hh) * 16 + (mw & 3) * 4) = word[hh];
    }
  }
  __syncthreads();                       // the scratch may be used for another block
  return true;
}

// Block `page` of a stream, complete after this append: slots [0, t0 - 128 page) from the tail, the rest from the input.
// in: the thread's channel piece of token 0 of the sequence.  All 256 threads take part.
template <int DTYPE, int KB, bool ROT>
__device__ __forceinline__ void kchan_complete_block(const Geom& g, const CachePtrs& c, int bh, int page, int t0,
                                                     const uint16_t* __restrict__ in, int64_t st, KchanShared& scratch, int tid) {
  const int tr = tid >> 4, v = tid & 15, tb = page << 7, lo = max(t0 - tb, 0);
  const uint16_t* tail = c.k_tail + (size_t)bh * kPageTokens * 128;
  uint4 val[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int slot = tr + 16 * i;
    if (slot < lo) val[i] = *reinterpret_cast<const uint4*>(tail + (size_t)slot * 128 + v * 8);
    else val[i] = __ldcs(reinterpret_cast<const uint4*>(in + (int64_t)(tb + slot) * st));
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint4 conv = key_row_fp16<DTYPE, ROT>(val[i], c.k_signs, v);
    if (tr + 16 * i >= lo) val[i] = conv;
  }
  kchan_block<KB>(val, scratch, c.pages + ((size_t)bh * g.n_pages + page) * g.page_bytes, g, tid);
}

// New rows of the block that stays incomplete go to the tail.
template <int DTYPE, bool ROT>
__device__ __forceinline__ void kchan_tail_rows(const CachePtrs& c, int bh, int page, int t0, int end,
                                                const uint16_t* __restrict__ in, int64_t st, int tid) {
  const int tr = tid >> 4, v = tid & 15, tb = page << 7, hi = end - tb;
  uint16_t* tail = c.k_tail + (size_t)bh * kPageTokens * 128;
  for (int s0 = max(t0 - tb, 0); s0 < hi; s0 += 16) {
    const int slot = s0 + tr;
    uint4 val = make_uint4(0u, 0u, 0u, 0u);
    if (slot < hi) val = __ldcs(reinterpret_cast<const uint4*>(in + (int64_t)(tb + slot) * st));
    val = key_row_fp16<DTYPE, ROT>(val, c.k_signs, v);
    if (slot < hi) *reinterpret_cast<uint4*>(tail + (size_t)slot * 128 + v * 8) = val;
  }
}

}  // namespace kvq
