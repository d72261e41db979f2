// kvq_dequantize kernel: x^ = fmaf(code, scale, zero) rounded to the 16-bit
// input type (App. B.1: A^ = scale * Q, here with the group minimum as offset).
//
// One CTA per (page, stream, side).  Fast path (2 / 4 / 8 bits): keys go straight from global to global memory (a
// thread owns a chunk of a token row, whose bytes are four consecutive channels of every 16-channel slice), values
// through a padded [128][D + 8] shared tile that stmatrix fills transposed; code bytes become floats by a byte
// permute and an exact subtraction.  Bit planes and 16-bit passthrough: the packed page is copied to shared memory
// and expanded element by element into the tile.  Bound by the 16-bit stores (they write 4-8x what they read).
#include "kvq_internal.h"

namespace kvq {

namespace {

constexpr int kThreads = 256;
constexpr int kTilePad = 8;     // the shared [128][D + 8] tile: a row stride of D + 8 elements spreads the token rows
                                // over the banks (a stride of D would put every row on the same banks)

// All sizes that index arithmetic divides by are powers of two: use shifts.
__device__ __forceinline__ int ilog2(int x) { return 31 - __clz(x); }

__device__ __forceinline__ float meta_scale(uint32_t m) { return __half2float(__ushort_as_half((uint16_t)(m & 0xFFFF))); }
__device__ __forceinline__ float meta_zero(uint32_t m) { return __half2float(__ushort_as_half((uint16_t)(m >> 16))); }

// Expand a code region of a bit-plane width (1, 3, 6 bits) into tile[t][d], element by element.
__device__ __forceinline__ void expand_planes(const uint8_t* spage, const Geom& g, bool is_v, uint16_t* tile, int tid) {
  const int D = g.D, b = is_v ? g.vb : g.kb, gs = is_v ? g.gv : g.gk;
  const uint8_t* region = spage + (is_v ? g.v_codes_off : 0);
  const uint32_t* meta = reinterpret_cast<const uint32_t*>(spage + (is_v ? g.v_meta_off : g.k_meta_off));
  const int lD = ilog2(D), lgs = ilog2(gs), ng = D >> lgs;
  for (int idx = tid; idx < kPageTokens * D; idx += kThreads) {
    const int t = idx >> lD, d = idx & (D - 1);
    const uint32_t m = meta[t * ng + (d >> lgs)];
    const float code = (float)load_code_any(region, is_v, t, d, D, b);
    tile[t * (D + kTilePad) + d] = f32_to_bits16(fmaf(code, meta_scale(m), meta_zero(m)), g.in_dtype);
  }
}

// Copy token rows [lo, hi) of a tile with row stride `ts` elements to out rows (16-byte vectors).
__device__ __forceinline__ void store_rows(const uint16_t* tile, int ts, uint16_t* out, int D, int lo, int hi, int tid) {
  const int vpr = D / 8, lv = ilog2(vpr);
  for (int idx = tid; idx < (hi - lo) * vpr; idx += kThreads) {
    const int t = lo + (idx >> lv), v = idx & (vpr - 1);
    __stcs(reinterpret_cast<uint4*>(out + (size_t)t * D) + v, reinterpret_cast<const uint4*>(tile + t * ts)[v]);   // written once, not re-read here
  }
}

// ---------------------------------------------------------------------------------------------------------
// Fast path: widths 2 / 4 / 8.  Everything a thread indexes is a compile-time offset from its own base; the four
// code bytes of a word become floats without a conversion instruction (byte -> 0x4B0000bb = 2^23 + code, minus 2^23: exact), and
// two elements share the subtraction, the fused multiply-add of the fixed formula and the rounding to 16 bits.
// ---------------------------------------------------------------------------------------------------------
// Bytes i and j of `bytes` as exact floats.
__device__ __forceinline__ f32x2 code_pair(uint32_t bytes, int i, int j) {
  const float a = __uint_as_float(__byte_perm(bytes, 0x4B000000u, 0x7540u + (uint32_t)i));
  const float b = __uint_as_float(__byte_perm(bytes, 0x4B000000u, 0x7540u + (uint32_t)j));
  return add2(pack2(a, b), pack2(-8388608.0f, -8388608.0f));
}
template <int DTYPE>
__device__ __forceinline__ uint32_t pack16(f32x2 v) {
  const float2 f = unpack2(v);
  if constexpr (DTYPE == KVQ_FP16) {
    const __half2 h = __floats2half2_rn(f.x, f.y);
    return *reinterpret_cast<const uint32_t*>(&h);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(f.x, f.y);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
}

// Keys of one page, straight from global memory to global memory: thread item = (token, chunk of its row); the chunk's bytes are
// four consecutive channels of every 16-channel slice, so each slice gives one 8-byte store and the four threads of a token write 32
// contiguous bytes.  AXIS 1: (scale, zero) per channel; an incomplete last page (tail != nullptr) has its keys as fp16 rows.
template <int B, int D, int AXIS, int DTYPE>
__device__ __forceinline__ void fast_keys(const Geom& g, const uint8_t* __restrict__ pg, const uint16_t* __restrict__ tail,
                                          uint16_t* __restrict__ out, int lo, int hi, int tid) {
  constexpr int FPB = 8 / B, ROW = D * B / 8;
  constexpr int WPC = D * B / 128;                       // words per chunk: 1, 2, 4 (one load), 8 (two quads)
  constexpr uint32_t MASK = ((1u << B) - 1u) * 0x01010101u;
  if constexpr (AXIS == 1) {
    if (tail != nullptr) {
      for (int idx = tid; idx < (hi - lo) * (D / 8); idx += kThreads) {
        const int t = lo + idx / (D / 8), v = idx % (D / 8);
        uint4 r = *reinterpret_cast<const uint4*>(tail + (size_t)t * D + 8 * v);
        if constexpr (DTYPE == KVQ_BF16) {
          uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
            w[i] = pack16<DTYPE>(pack2(f.x, f.y));
          }
          r = make_uint4(w[0], w[1], w[2], w[3]);
        }
        __stcs(reinterpret_cast<uint4*>(out + (size_t)t * D + 8 * v), r);
      }
      return;
    }
  }
  const uint32_t* meta = reinterpret_cast<const uint32_t*>(pg + g.k_meta_off);
  const int lgk = ilog2(g.gk), ngk = D >> lgk;
  for (int item = tid; item < kPageTokens * 4; item += kThreads) {
    const int t = item >> 2, chunk = item & 3;
    if (t < lo || t >= hi) continue;
    uint32_t w[WPC];
    const uint8_t* row = pg + t * ROW;
    if constexpr (WPC == 1) {
      w[0] = __ldcs(reinterpret_cast<const uint32_t*>(row + chunk * 4));
    } else if constexpr (WPC == 2) {
      const uint2 v = __ldcs(reinterpret_cast<const uint2*>(row + chunk * 8));
      w[0] = v.x; w[1] = v.y;
    } else {
#pragma unroll
      for (int qd = 0; qd < WPC / 4; ++qd) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4*>(row + qd * 64 + chunk * 16));
        w[4 * qd + 0] = v.x; w[4 * qd + 1] = v.y; w[4 * qd + 2] = v.z; w[4 * qd + 3] = v.w;
      }
    }
    uint16_t* orow = out + (size_t)t * D + 4 * chunk;
    f32x2 sc[2], ze[2];
#pragma unroll
    for (int r = 0; r < D / 16; ++r) {                   // slice r: channels 16 r + 4 chunk + {0..3}
      const uint32_t bytes = (w[r / FPB] >> (B * (r % FPB))) & MASK;
      if constexpr (AXIS == 1) {
        const uint4 m = __ldg(reinterpret_cast<const uint4*>(meta + 16 * r + 4 * chunk));
        sc[0] = pack2(meta_scale(m.x), meta_scale(m.y)); ze[0] = pack2(meta_zero(m.x), meta_zero(m.y));
        sc[1] = pack2(meta_scale(m.z), meta_scale(m.w)); ze[1] = pack2(meta_zero(m.z), meta_zero(m.w));
      } else if (r == 0 || ((16 * r) & (g.gk - 1)) == 0) {     // a new group (the same for all threads)
        const uint32_t m = __ldg(meta + t * ngk + ((16 * r) >> lgk));
        sc[0] = sc[1] = pack2(meta_scale(m), meta_scale(m));
        ze[0] = ze[1] = pack2(meta_zero(m), meta_zero(m));
      }
      const uint32_t a = pack16<DTYPE>(fma2(code_pair(bytes, 0, 1), sc[0], ze[0]));
      const uint32_t b = pack16<DTYPE>(fma2(code_pair(bytes, 2, 3), sc[1], ze[1]));
      __stcs(reinterpret_cast<uint2*>(orow + 16 * r), make_uint2(a, b));
    }
  }
}

// Rotated keys of one page: as fast_keys, rotated back (x = signs * H y / sqrt(D)) before they are rounded.  A thread has channels
// 16 r + 4 chunk + j of its token, so of the butterfly stages h = 1, 2, 4, ..., in this order, only h = 4 and 8 cross lanes (two shuffles
// per element instead of the four of eight consecutive channels a lane).  32 streams x 30,000 tokens K4V2, both sides: 213 us with
// the page staged in shared memory and element-wise expansion, 135 now.  The signs may lie at any address: they are read byte by byte,
// once per CTA, and a row takes them as words of shared memory (four bytes a word from global memory for every row: 142.)
template <int B, int D, int AXIS, int DTYPE>
__device__ __forceinline__ void fast_keys_rotated(const Geom& g, const uint8_t* __restrict__ pg, const uint16_t* __restrict__ tail,
                                                  const int8_t* __restrict__ signs, uint16_t* __restrict__ out, int lo, int hi, int tid) {
  constexpr int FPB = 8 / B, ROW = D * B / 8, WPC = D * B / 128, NR = D / 16;
  constexpr uint32_t MASK = ((1u << B) - 1u) * 0x01010101u, FULL = 0xffffffffu;
  const uint32_t* meta = reinterpret_cast<const uint32_t*>(pg + g.k_meta_off);
  const int lgk = ilog2(g.gk), ngk = D >> lgk, chunk = tid & 3;
  const float s4 = (chunk & 1) ? -1.0f : 1.0f, s8 = (chunk & 2) ? -1.0f : 1.0f;      // a butterfly between lanes: o + s x (exact product)
  __shared__ char4 sign[D / 4];
  if (tid < D) reinterpret_cast<int8_t*>(sign)[tid] = __ldg(signs + tid);
  __syncthreads();
  for (int item = tid; item < kPageTokens * 4; item += kThreads) {
    const int t = item >> 2;
    const bool active = t >= lo && t < hi;
    if (!__any_sync(FULL, active)) continue;
    f32x2 x[NR][2];
    if (AXIS == 1 && tail != nullptr) {
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        uint2 v = make_uint2(0u, 0u);
        if (active) v = *reinterpret_cast<const uint2*>(tail + (size_t)t * D + 16 * r + 4 * chunk);
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&v.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
        x[r][0] = pack2(a.x, a.y);
        x[r][1] = pack2(b.x, b.y);
      }
    } else {
      uint32_t w[WPC];                                     // (of any token of the page: inactive lanes take part in the shuffles)
      const uint8_t* row = pg + t * ROW;
      if constexpr (WPC == 1) {
        w[0] = __ldcs(reinterpret_cast<const uint32_t*>(row + chunk * 4));
      } else if constexpr (WPC == 2) {
        const uint2 v = __ldcs(reinterpret_cast<const uint2*>(row + chunk * 8));
        w[0] = v.x; w[1] = v.y;
      } else {
#pragma unroll
        for (int qd = 0; qd < WPC / 4; ++qd) {
          const uint4 v = __ldcs(reinterpret_cast<const uint4*>(row + qd * 64 + chunk * 16));
          w[4 * qd + 0] = v.x; w[4 * qd + 1] = v.y; w[4 * qd + 2] = v.z; w[4 * qd + 3] = v.w;
        }
      }
      f32x2 sc[2], ze[2];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const uint32_t bytes = (w[r / FPB] >> (B * (r % FPB))) & MASK;
        if constexpr (AXIS == 1) {
          const uint4 m = __ldg(reinterpret_cast<const uint4*>(meta + 16 * r + 4 * chunk));
          sc[0] = pack2(meta_scale(m.x), meta_scale(m.y)); ze[0] = pack2(meta_zero(m.x), meta_zero(m.y));
          sc[1] = pack2(meta_scale(m.z), meta_scale(m.w)); ze[1] = pack2(meta_zero(m.z), meta_zero(m.w));
        } else if (r == 0 || ((16 * r) & (g.gk - 1)) == 0) {
          const uint32_t m = __ldg(meta + t * ngk + ((16 * r) >> lgk));
          sc[0] = sc[1] = pack2(meta_scale(m), meta_scale(m));
          ze[0] = ze[1] = pack2(meta_zero(m), meta_zero(m));
        }
        x[r][0] = fma2(code_pair(bytes, 0, 1), sc[0], ze[0]);
        x[r][1] = fma2(code_pair(bytes, 2, 3), sc[1], ze[1]);
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const float2 a = unpack2(x[r][0]), b = unpack2(x[r][1]);                             // h = 1
      const f32x2 p = pack2(__fadd_rn(a.x, a.y), __fsub_rn(a.x, a.y)), q = pack2(__fadd_rn(b.x, b.y), __fsub_rn(b.x, b.y));
      x[r][0] = add2(p, q);                                                                // h = 2
      x[r][1] = fma2(q, pack2(-1.0f, -1.0f), p);
#pragma unroll
      for (int e = 0; e < 2; ++e) {                                                        // h = 4, 8
        float2 o = unpack2(x[r][e]);
        o.x = __shfl_xor_sync(FULL, o.x, 1); o.y = __shfl_xor_sync(FULL, o.y, 1);
        x[r][e] = fma2(pack2(s4, s4), x[r][e], pack2(o.x, o.y));
        o = unpack2(x[r][e]);
        o.x = __shfl_xor_sync(FULL, o.x, 2); o.y = __shfl_xor_sync(FULL, o.y, 2);
        x[r][e] = fma2(pack2(s8, s8), x[r][e], pack2(o.x, o.y));
      }
    }
#pragma unroll
    for (int h = 1; h < NR; h <<= 1) {                                                     // h = 16, 32, 64
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if ((r & h) == 0) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const f32x2 a = x[r][e], b = x[r + h][e];
            x[r][e] = add2(a, b);
            x[r + h][e] = fma2(b, pack2(-1.0f, -1.0f), a);
          }
        }
      }
    }
    if (!active) continue;
    uint16_t* orow = out + (size_t)t * D + 4 * chunk;
    constexpr float NORM = inv_sqrt_dim<D>();
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const char4 s = sign[4 * r + chunk];
      const uint32_t a = pack16<DTYPE>(mul2(mul2(x[r][0], pack2(NORM, NORM)), pack2((float)s.x, (float)s.y)));
      const uint32_t b = pack16<DTYPE>(mul2(mul2(x[r][1], pack2(NORM, NORM)), pack2((float)s.z, (float)s.w)));
      __stcs(reinterpret_cast<uint2*>(orow + 16 * r), make_uint2(a, b));
    }
  }
}

// Values of one page.  A warp takes the 32 16-byte quads of one word column of a 32-token block: lane (gq, tq) has the codes of
// channels 16 m + 8 rh + gq for eight tokens, and the pairs (2 tq, 2 tq + 1) of a word are what stmatrix transposes: one instruction
// puts two channel octets of 16 tokens into the padded [128][D + 8] tile as whole 16-byte pieces, whose rows leave with 16-byte stores.
// Keys and values of 64 streams x 32,768 tokens (K4V2, 1.29 GB): 254 us with one 2-byte shared store per element, 201 to 210 now, which
// is the rate of a plain copy (200 us).
template <int B, int D, int DTYPE>
__device__ __forceinline__ void fast_values(const Geom& g, const uint8_t* __restrict__ pg, uint16_t* tile,
                                            uint16_t* __restrict__ out, int lo, int hi, int tid) {
  constexpr int FPB = 8 / B, TS = D + kTilePad, NMW = D * B / 128;      // word columns per block
  constexpr uint32_t MASK = ((1u << B) - 1u) * 0x01010101u;
  const uint4* codes = reinterpret_cast<const uint4*>(pg + g.v_codes_off);
  const uint32_t* meta = reinterpret_cast<const uint32_t*>(pg + g.v_meta_off);
  const int lgv = ilog2(g.gv), ngv = D >> lgv;
  const int lane = tid & 31, tq = lane & 3;
  // the 16-byte row of the tile that this lane's address names: matrix (half, rh) = lane / 8, token lane % 8 of the half
  const uint32_t row0 = (uint32_t)__cvta_generic_to_shared(tile + (8 * (lane >> 4) + (lane & 7)) * TS + 8 * ((lane >> 3) & 1));
  for (int item = tid >> 5; item < 4 * NMW; item += kThreads / 32) {
    const int blk = item / NMW, mw = item % NMW;
    const uint4 v = __ldcs(codes + item * 32 + lane);
    const uint32_t ww[4] = {v.x, v.y, v.z, v.w};           // sub = 2 rh + kh
    const uint32_t* mt = meta + (blk * 32 + 2 * tq) * ngv + ((16 * FPB * mw) >> lgv);
    f32x2 sc[2][2], ze[2][2];                              // [kh][half]: tokens 16 kh + 8 half + 2 tq + {0, 1}
    auto load_meta = [&](const uint32_t* m) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t a = __ldg(m + 8 * i * ngv), b = __ldg(m + (8 * i + 1) * ngv);
        sc[i >> 1][i & 1] = pack2(meta_scale(a), meta_scale(b));
        ze[i >> 1][i & 1] = pack2(meta_zero(a), meta_zero(b));
      }
    };
    load_meta(mt);
    const uint32_t dst = row0 + 2 * (blk * 32 * TS + 16 * FPB * mw);
#pragma unroll
    for (int f = 0; f < FPB; ++f) {
      if (FPB == 4 && f == 2 && g.gv == 32) load_meta(mt + 1);       // four fields of 16 channels span two groups of 32
#pragma unroll
      for (int kh = 0; kh < 2; ++kh) {
        uint32_t r[2][2];                                  // [half][rh]
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
          const uint32_t bytes = (ww[2 * rh + kh] >> (B * f)) & MASK;       // tokens 2 tq, 2 tq + 8, 2 tq + 1, 2 tq + 9
          r[0][rh] = pack16<DTYPE>(fma2(code_pair(bytes, 0, 2), sc[kh][0], ze[kh][0]));
          r[1][rh] = pack16<DTYPE>(fma2(code_pair(bytes, 1, 3), sc[kh][1], ze[kh][1]));
        }
        asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                     ::"r"(dst + 2 * (16 * kh * TS + 16 * f)), "r"(r[0][0]), "r"(r[0][1]), "r"(r[1][0]), "r"(r[1][1]) : "memory");
      }
    }
  }
  __syncthreads();
  store_rows(tile, TS, out, D, lo, hi, tid);
}

// Five CTAs per SM (64 streams x 32,768 tokens K4V2, both sides: four 214 us, five 201, six 202).
constexpr int kFastPerSm = 5;
template <int B> struct Width { static constexpr int value = B; };

// grid (pages, streams, sides); blockIdx.z + side0: 0 values, 1 keys.  KB / VB: the side's width, 0 = this launch has no such
// side, -1 = read from the geometry (a launch of both sides).
template <int D, int KB, int VB, int AXIS, bool ROT, int DTYPE>
__global__ void __launch_bounds__(kThreads, ROT ? 3 : kFastPerSm)
dequant_fast_kernel(Geom g, CachePtrs c, uint16_t* k_out, uint16_t* v_out, int t_begin, int t_end, int page0, int side0) {
  extern __shared__ __align__(16) uint8_t smem[];
  begin_after_predecessor();
  const int tid = threadIdx.x;
  const int bh = blockIdx.y, b = bh / g.Hkv;
  const int n = paged_len(c.seq_len, b, g.capacity, g.R);
  const int hi = min(t_end, n);
  const int page = page0 + blockIdx.x;
  const int lo_t = max(t_begin, page * kPageTokens), hi_t = min(hi, page * kPageTokens + kPageTokens);
  if (lo_t >= hi_t) return;
  const uint8_t* pg = c.pages + ((size_t)bh * g.n_pages + page) * g.page_bytes;
  const int lo = lo_t - page * kPageTokens, hi_l = hi_t - page * kPageTokens;
  const size_t out_base = ((size_t)bh * g.capacity + (size_t)page * kPageTokens) * D;
  if (blockIdx.z + side0 == 0) {
    uint16_t* tile = reinterpret_cast<uint16_t*>(smem);
    uint16_t* out = v_out + out_base;
    if constexpr (VB > 0) fast_values<VB, D, DTYPE>(g, pg, tile, out, lo, hi_l, tid);
    if constexpr (VB < 0) {
      if (g.vb == 2) fast_values<2, D, DTYPE>(g, pg, tile, out, lo, hi_l, tid);
      else if (g.vb == 4) fast_values<4, D, DTYPE>(g, pg, tile, out, lo, hi_l, tid);
      else fast_values<8, D, DTYPE>(g, pg, tile, out, lo, hi_l, tid);
    }
  } else {
    const uint16_t* tail = (AXIS == 1 && n < (page + 1) * kPageTokens) ? c.k_tail + (size_t)bh * kPageTokens * D : nullptr;
    uint16_t* out = k_out + out_base;
    auto keys = [&](auto width) {
      constexpr int B = decltype(width)::value;
      if constexpr (ROT) fast_keys_rotated<B, D, AXIS, DTYPE>(g, pg, tail, c.k_signs, out, lo, hi_l, tid);
      else fast_keys<B, D, AXIS, DTYPE>(g, pg, tail, out, lo, hi_l, tid);
    };
    if constexpr (KB > 0) keys(Width<KB>{});
    if constexpr (KB < 0) {
      if (g.kb == 2) keys(Width<2>{});
      else if (g.kb == 4) keys(Width<4>{});
      else keys(Width<8>{});
    }
  }
}

// KB, VB as above.
template <int KB, int VB>
int launch_fast(const Geom& g, const CachePtrs& c, uint16_t* k_out, uint16_t* v_out, int t_begin, int t_end, int page0,
                int n_pages, cudaStream_t stream) {
  const dim3 grid(n_pages, g.B * g.Hkv, KB != 0 && VB != 0 ? 2 : 1);
  const size_t smem = VB != 0 ? (size_t)kPageTokens * (g.D + kTilePad) * 2 : 0;      // the value side's tile
  auto run = [&](auto kern) {
    const cudaError_t e = launch_dependent(kern, grid, kThreads, smem, stream, 1, g, c, k_out, v_out, t_begin, t_end, page0, VB != 0 ? 0 : 1);
    return e == cudaSuccess ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
  };
  const bool h = g.in_dtype == KVQ_FP16, rot = KB != 0 && c.k_signs != nullptr, chan = KB != 0 && g.k_axis == 1;
#define KVQ_DQ(D_, A_, R_) \
  if (g.D == D_ && chan == (A_ == 1) && rot == R_) \
    return run(h ? dequant_fast_kernel<D_, KB, VB, A_, R_, KVQ_FP16> : dequant_fast_kernel<D_, KB, VB, A_, R_, KVQ_BF16>);
  KVQ_DQ(128, 0, false) KVQ_DQ(64, 0, false)
  if constexpr (KB != 0) { KVQ_DQ(128, 1, false) KVQ_DQ(64, 1, false) KVQ_DQ(128, 0, true) KVQ_DQ(64, 0, true) KVQ_DQ(128, 1, true) KVQ_DQ(64, 1, true) }
#undef KVQ_DQ
  return KVQ_ERR_UNSUPPORTED;
}

// 16-bit passthrough and bit planes.
__global__ void __launch_bounds__(kThreads)
dequant_kernel(Geom g, CachePtrs c, uint16_t* k_out, uint16_t* v_out,
               int t_begin, int t_end, int page0, int side0) {
  extern __shared__ __align__(16) uint8_t smem[];
  begin_after_predecessor();
  const int D = g.D, tid = threadIdx.x;
  uint8_t* spage = smem;
  uint16_t* tile = reinterpret_cast<uint16_t*>(smem + ((g.page_bytes + 15) & ~15));   // [128][D]
  const int bh = blockIdx.y;
  const int b = bh / g.Hkv;
  const int n = paged_len(c.seq_len, b, g.capacity, g.R);      // tokens behind a residual window are in the pages
  const int hi = min(t_end, n);
  const int page = page0 + blockIdx.x;
  const int lo_t = max(t_begin, page * kPageTokens), hi_t = min(hi, page * kPageTokens + kPageTokens);
  if (lo_t >= hi_t) return;
  const uint8_t* pg = c.pages + ((size_t)bh * g.n_pages + page) * g.page_bytes;
  // only this CTA's side of the page: keys [0, v_codes_off), values [v_codes_off, page_bytes)
  const int side = blockIdx.z + side0;
  const int v16_lo = (side == 0 ? g.v_codes_off : 0) / 16;
  const int v16_hi = (side == 0 ? g.page_bytes : g.v_codes_off) / 16;
  for (int i = v16_lo + tid; i < v16_hi; i += kThreads)
    reinterpret_cast<uint4*>(spage)[i] = __ldcs(reinterpret_cast<const uint4*>(pg) + i);
  __syncthreads();
  const int lo = lo_t - page * kPageTokens, hi_l = hi_t - page * kPageTokens;
  const size_t out_base = ((size_t)bh * g.capacity + (size_t)page * kPageTokens) * D;

  // the side: 0 values, 1 keys (two CTAs share a page so that short ranges still fill the GPU)
  const bool is_v = side == 0;
  uint16_t* out = (is_v ? v_out : k_out) + out_base;
  if ((is_v ? g.vb : g.kb) == 16) {
    store_rows(reinterpret_cast<const uint16_t*>(spage + (is_v ? g.v_codes_off : 0)), D, out, D, lo, hi_l, tid);
  } else {
    expand_planes(spage, g, is_v, tile, tid);
    __syncthreads();
    store_rows(tile, D + kTilePad, out, D, lo, hi_l, tid);
  }
}

// Tokens still in the residual window are the 16-bit inputs themselves: copy their rows out.
__global__ void __launch_bounds__(kThreads)
window_dequant_kernel(Geom g, CachePtrs c, uint16_t* k_out, uint16_t* v_out, int t_begin, int t_end) {
  begin_after_predecessor();
  const int bh = blockIdx.x, b = bh / g.Hkv;
  const int D = g.D, R = g.R, vpr = D / 8;
  const int n = clamped_len(c.seq_len, b, g.capacity);
  const int lo = max(t_begin, (n / R) * R), hi = min(t_end, n);
  for (int idx = threadIdx.x; idx < (hi - lo) * 2 * vpr; idx += kThreads) {
    const int t = lo + idx / (2 * vpr), side = (idx / vpr) & 1, v = idx % vpr;
    uint16_t* dst = side ? v_out : k_out;
    if (!dst) continue;
    reinterpret_cast<uint4*>(dst + ((size_t)bh * g.capacity + t) * D)[v] =
        reinterpret_cast<const uint4*>(c.kv_win + (((size_t)bh * R + (t % R)) * 2 + side) * D)[v];
  }
}

}  // namespace

int launch_dequantize(const Geom& g, const CachePtrs& c, void* k_out, void* v_out, int t_begin, int t_end,
                      cudaStream_t stream) {
  if (t_end <= t_begin) return KVQ_OK;
  const int page0 = t_begin / kPageTokens;
  const int page1 = (t_end + kPageTokens - 1) / kPageTokens;
  const size_t smem = (size_t)((g.page_bytes + 15) & ~15) + (size_t)kPageTokens * (g.D + kTilePad) * 2;
  cudaFuncSetAttribute(dequant_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       128 * 128 * 4 + 128 * (128 + kTilePad) * 2);
  uint16_t* ko = static_cast<uint16_t*>(k_out);
  uint16_t* vo = static_cast<uint16_t*>(v_out);
  const int np = page1 - page0;
  // sides the fast kernel serves (2 / 4 / 8 bits)
  auto fast_bits = [](int b) { return b == 2 || b == 4 || b == 8; };
  const bool fast_v = vo && fast_bits(g.vb);
  const bool fast_k = ko && fast_bits(g.kb);
  int rc = KVQ_OK;
  auto window_rows = [&]() {      // tokens that are still in the residual window
    return g.R == 0 || launch_dependent(window_dequant_kernel, dim3(g.B * g.Hkv), kThreads, 0, stream, 1, g, c, ko, vo, t_begin, t_end) == cudaSuccess
               ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
  };
  // A short range (the newest page of every stream in a decode step) is one launch for both sides; a long one
  // keeps a launch per side, where the key CTAs run without the value side's shared-memory tile.
  if (fast_v && fast_k && (long long)np * g.B * g.Hkv <= 148 * 8) {
    rc = launch_fast<-1, -1>(g, c, ko, vo, t_begin, t_end, page0, np, stream);
    return rc != KVQ_OK ? rc : window_rows();
  }
  if (fast_v) {
    if (g.vb == 2) rc = launch_fast<0, 2>(g, c, ko, vo, t_begin, t_end, page0, np, stream);
    else if (g.vb == 4) rc = launch_fast<0, 4>(g, c, ko, vo, t_begin, t_end, page0, np, stream);
    else rc = launch_fast<0, 8>(g, c, ko, vo, t_begin, t_end, page0, np, stream);
    if (rc != KVQ_OK) return rc;
  }
  if (fast_k) {
    if (g.kb == 2) rc = launch_fast<2, 0>(g, c, ko, vo, t_begin, t_end, page0, np, stream);
    else if (g.kb == 4) rc = launch_fast<4, 0>(g, c, ko, vo, t_begin, t_end, page0, np, stream);
    else rc = launch_fast<8, 0>(g, c, ko, vo, t_begin, t_end, page0, np, stream);
    if (rc != KVQ_OK) return rc;
  }
  // whatever is left goes through the general kernel
  const bool gen_v = vo && !fast_v, gen_k = ko && !fast_k;
  if (gen_v || gen_k) {
    dim3 grid(np, g.B * g.Hkv, (gen_v && gen_k) ? 2 : 1);
    if (launch_dependent(dequant_kernel, grid, kThreads, smem, stream, 1, g, c, ko, vo, t_begin, t_end, page0, gen_v ? 0 : 1) != cudaSuccess)
      return KVQ_ERR_CUDA_LAUNCH;
  }
  return window_rows();
}

}  // namespace kvq
