// The templated fast decode kernel (see kvq_decode_mma.cuh for the design).
#pragma once

#include <type_traits>

#include "kvq_decode_mma.cuh"

namespace kvq {
namespace mma {

// Shared-memory carve-up (dynamic): ring | barriers | prefix | misc | weights | reductions | channel-wise scratch
struct SmemLayout {
  int page_stride, ring_bytes, bar_off, pref_off, misc_off, w_off, red_off, chan_off, total;
};
// weights: the PV operands of a page as the owners of its four 32-token blocks leave them, per value group and block
// (16 NH bytes per lane), for two pages in turn.
// chan: channel-wise keys keep, per ring stage, the page's q operands made by the producer warp
// (NH x 2 x D/16 x 32 words) followed by 8 zero-point sums and 8 fixed-point scales (one per head).
__host__ __device__ constexpr int weight_block_bytes(int nh) { return 512 * nh; }
__host__ __device__ constexpr int reduction_bytes(int ngv) { return 4 * (8 * ngv * 8 + (8 + 4 + 8) * 4); }   // per warp: p z sums (64 bits), maxima, scale limit, l
__host__ __device__ inline int chan_stage_bytes(int D, int nh) { return nh * 2 * (D / 16) * 32 * 4 + 64; }
__host__ __device__ inline SmemLayout smem_layout(int page_bytes, int stages, int batch, int D, int nh, int ngv, bool chan) {
  SmemLayout s;
  s.page_stride = (page_bytes + 127) & ~127;
  s.ring_bytes = s.page_stride * stages;
  s.bar_off = s.ring_bytes;
  s.pref_off = s.bar_off + 16 * 8 * 2;                      // up to 32 barriers: (full, empty[, ready]) per stage
  s.misc_off = (s.pref_off + 2 * (batch + 1) * 4 + 15) & ~15;      // two prefixes: pages, and pages + stream gaps
  s.w_off = s.misc_off + 64;
  s.red_off = s.w_off + 2 * ngv * 4 * weight_block_bytes(nh);
  s.chan_off = s.red_off + reduction_bytes(ngv);
  s.total = s.chan_off + (chan ? stages * chan_stage_bytes(D, nh) : 0);
  return s;
}

// Stages of the ring for `minb` resident CTAs per SM, or fewer than two where a configuration does not fit.
// Deeper rings do not help, and more bytes in flight cost DRAM efficiency: at most four stages and 54 KB (K4V4, 17 KB pages, 8B
// shape: four stages 97.9 us, three 89.8 us; K4V2, 13 KB pages: four 76.8 us, three 77.3 us).
inline int ring_stages(const Geom& g, int nh, int ngv, bool chan, int minb) {
  const int budget = (227 * 1024) / minb - 1024;            // shared memory per CTA
  int stages = (budget - smem_layout(0, 0, g.B, g.D, nh, ngv, chan).total) /
               (((g.page_bytes + 127) & ~127) + (chan ? chan_stage_bytes(g.D, nh) : 0));
  if (stages > 4) stages = 4;
  if (stages > 2 && stages * ((g.page_bytes + 127) & ~127) > 54 * 1024) stages = 3;
  return stages;
}
// Whether a residual window of nw tokens may be read from the ring: its logits read whole tiles of 16 rows (key row, value row), the
// last one beyond the rows that were copied.
__host__ __device__ inline bool window_fits_ring(const SmemLayout& sl, int nw, int D) { return ((nw + 15) & ~15) * 4 * D <= sl.ring_bytes; }

// prmt.b32 with the full selector semantics (a selector nibble with bit 3 set replicates the sign of the byte).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
// D += A(16x32, row, unsigned bytes) * B(32x8, col, unsigned bytes), int32 accumulate.
__device__ __forceinline__ void mma16832_u8u8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                              uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The same with a zero accumulator: D = A B.
__device__ __forceinline__ void mma16832_u8u8_zero(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                   uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(0));
}
__device__ __forceinline__ void mma16832_u8s8_zero(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                   uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(0));
}
__device__ __forceinline__ void mbar_arrive_if(uint32_t bar, bool p) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar), "r"((uint32_t)p) : "memory");
}
// Barrier of `nthreads` threads that also says whether any of them came with p.
__device__ __forceinline__ bool named_bar_any(int id, int nthreads, bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r) : "r"((uint32_t)p), "r"(id), "r"(nthreads) : "memory");
  return r != 0;
}

// Four values times `scale` rounded to integers |Q| <= 32512 and split into two balanced signed bytes, Q = hi * 256 + lo: the four hi
// bytes or the four lo bytes as one word.  The sum with 1.5 * 2^23 (+ 128 for the hi bytes: hi = (Q + 128) >> 8) leaves Q as the low bits
// of n; the caller gets them all added up.  scale_q: scale * 2^-8 (the product is rounded before it is rounded to an integer, by a fused
// operation that takes the 2^8 back).  sel: bytes 1 (hi) or 0 (lo) of two words.
__device__ __forceinline__ uint32_t fixed_point_limb(const float (&t)[4], f32x2 scale_q, f32x2 magic, uint32_t sel, uint32_t& nsum) {
  const f32x2 up = pack2(256.0f, 256.0f);
  const float2 a = unpack2(fma2(mul2(pack2(t[0], t[1]), scale_q), up, magic)), b = unpack2(fma2(mul2(pack2(t[2], t[3]), scale_q), up, magic));
  const uint32_t n0 = __float_as_uint(a.x), n1 = __float_as_uint(a.y), n2 = __float_as_uint(b.x), n3 = __float_as_uint(b.y);
  nsum += n0 + n1 + n2 + n3;
  return prmt(prmt(n0, n1, sel), prmt(n2, n3, sel), 0x5410);
}

// The split balances time, not pages.  Ending one stream and starting the next costs a CTA about as much as several pages
// (load and convert the next queries, publish a partial, perhaps merge), so every stream is given a gap of virtual pages in front
// of its real ones and the split is taken on that virtual axis; with many CTAs per stream the gap also keeps shares from
// crossing into the next stream for a page or two.  Eight pages at head_dim 128 (70B shape at 128k tokens 237 us, gap 6 239.5, 4 242; 64
// windowed streams of 16,000 tokens 63.6, 65.3, 68.0; two layers of 128 x 32,767 174.7, 174.6, 175.6; short ragged ones of one head a lane
// gain: 80 streams of 4,000 tokens 73.2, 70.6, 70.0).  Channel-wise keys, whose pages take longer: 2 (two ragged 14B-shaped layers 226
// us; 5: 228, 8: 233).  At head_dim 64 a page is half the work: 12 (1B shape, append 128 and decode, 16 layers: 18 301.6 us, 15 297.0, 12 296.4;
// eight layers of 64 streams of 1,000 tokens 103.5, 102.9, 99.6, 64 ragged ones of 4,000 122.2, 120.3, 118.9), but only up to 64 streams: with
// more of them a share is not much longer than such a gap, and some are left with nothing else (steps of four 1B-shaped layers, gap 8 / 12: 72 x
// 1,200 51.2 / 54.3, 96 x 1,200 54.7 / 57.0, 128 x 4,000 76.9 / 80.2, 256 x 4,000 106.6 / 111.7, 512 x 4,000 166 / 167).  Up to 64 streams the two
// lie close since a stream's count word is started early: eight streams of 512 tokens 45.0 / 40.4, of 4,000
// 50.6 / 49.2, but 48 x 2,000 50.4 / 53.1, 64 ragged ones of 4,000 57.2 / 59.4 and the 1B shape with append 128, 16 layers, 280 / 284.
// Of the CTAs that share an SM the hardware favours the older ones (0.85 / 0.91 / 0.99 us per page at three per SM, 0.96 / 1.01 at two),
// so the launch waves are weighted (8B shape K4V2 when the weights were chosen: 1040 76.1 us, 1080 77.3, equal 80.4).
constexpr int kGapPages = 8, kGapPages64 = 12, kGapStreams64 = 64, kGapPagesChan = 2;
constexpr float kQFix = 32512.0f;          // largest |Q| of the 16-bit fixed-point q (hi limb stays within +-127)
constexpr float kQFix3 = 8300000.0f;       // ... of the 24-bit fixed-point q * s of channel-wise keys (three limbs)

// Four values |t| <= kQFix3 rounded to integers Q and taken apart as two's-complement bytes,
// Q = b2 * 65536 + b1 * 256 + b0 with b2 signed and b1, b0 unsigned; byte j of w[k] is b_k of t[j].  The even operand
// columns carry b2 in n-tile 0 (signed bytes) and b1 in n-tile 1 (unsigned bytes), the odd ones nothing in n-tile 0 and b0 in n-tile 1.
__device__ __forceinline__ void fixed_point_bytes3(const float (&t)[4], uint32_t (&w)[3]) {
  const uint32_t q0 = (uint32_t)__float2int_rn(t[0]), q1 = (uint32_t)__float2int_rn(t[1]);
  const uint32_t q2 = (uint32_t)__float2int_rn(t[2]), q3 = (uint32_t)__float2int_rn(t[3]);
  const uint32_t lo01 = prmt(q0, q1, 0x5140u), lo23 = prmt(q2, q3, 0x5140u);      // bytes (0, 0), (1, 1) of a pair
  w[0] = prmt(lo01, lo23, 0x5410u);
  w[1] = prmt(lo01, lo23, 0x7632u);
  w[2] = prmt(prmt(q0, q1, 0x0062u), prmt(q2, q3, 0x0062u), 0x5410u);
}
// The softmax weights enter PV as fixed point P = rint(p * s_V * 2^PBITS / s_lim), p = 2^(logit - reference) with the
// reference kHeadroom bits above the largest logit seen so far, so that a larger logit rarely forces a rescale.
// Tokens whose P falls below one unit vanish, so the width matters over long contexts: four byte limbs, all 32 bits of them.  The
// reference is common to the CTA's four warps, so headroom is kept to four bits: a unit is 2^-28 of the largest weight (heavy-tailed
// channel-wise keys, 64-bit comparison: 31 bits and 6 of headroom 2.1e-5, against 6.7e-6 with a reference per warp).
constexpr int kPBits = 32;
constexpr float kHeadroom = 4.0f;
constexpr int kFlushPages = 128;           // fold the int32 value accumulators at least this often: 128 x 128 tokens x 255 x 255 < 2^31

// The query values a lane needs as MMA operand: head hb (a (row, head) pair when several rows are served), channels
// 16 r + 4 tid + {0..3} for every slot r; heads >= G are zero.  First as they are in memory, so that they can be on their way ...
template <int D>
__device__ __forceinline__ void load_q_raw(const Geom& g, const uint16_t* __restrict__ q, int b, int h, int hb, int tid, uint2 (&raw)[D / 16]) {
  const int Gq = g.G, G = g.G * g.rows;
  const uint16_t* qrow = q + (((size_t)b * g.rows + hb / Gq) * g.Hq + (size_t)h * Gq + hb % Gq) * D;
#pragma unroll
  for (int r = 0; r < D / 16; ++r) {
    raw[r] = make_uint2(0u, 0u);
    if (hb < G) raw[r] = *reinterpret_cast<const uint2*>(qrow + 16 * r + 4 * tid);
  }
}
// ... then in fp32, rotated like the keys if the cache rotates them.  Returns max |q| over the lane's values (the caller reduces over the quad).
template <int D>
__device__ __forceinline__ float convert_q_lane(const Geom& g, const CachePtrs& c, const uint2 (&raw)[D / 16], int tid, float (&qv)[D / 16][4]) {
  constexpr int NR = D / 16;
  constexpr uint32_t FULL = 0xffffffffu;
  if (g.in_dtype == KVQ_FP16) {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const float2 x = __half22float2(as_h2(raw[r].x)), y = __half22float2(as_h2(raw[r].y));
      qv[r][0] = x.x; qv[r][1] = x.y; qv[r][2] = y.x; qv[r][3] = y.y;
    }
  } else {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      qv[r][0] = __uint_as_float(raw[r].x << 16); qv[r][1] = __uint_as_float(raw[r].x & 0xFFFF0000u);
      qv[r][2] = __uint_as_float(raw[r].y << 16); qv[r][3] = __uint_as_float(raw[r].y & 0xFFFF0000u);
    }
  }
        if (c.k_signs != nullptr) {
          // rotated keys: give q the same rotation, q' = H (signs * q) / sqrt(D); channel 16 r + 4 tid + j,
          // so the butterflies run over j inside the lane, over tid across lanes, over r inside the lane
#pragma unroll
          for (int r = 0; r < NR; ++r) {
#pragma unroll
            for (int j = 0; j < 4; ++j) qv[r][j] *= (float)c.k_signs[16 * r + 4 * tid + j];
            float a = qv[r][0], bq = qv[r][1], cq = qv[r][2], dq = qv[r][3];
            qv[r][0] = (a + bq) + (cq + dq); qv[r][1] = (a - bq) + (cq - dq);
            qv[r][2] = (a + bq) - (cq + dq); qv[r][3] = (a - bq) - (cq - dq);
#pragma unroll
            for (int m = 1; m < 4; m <<= 1) {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float o = __shfl_xor_sync(FULL, qv[r][j], m);
                qv[r][j] = (tid & m) ? o - qv[r][j] : qv[r][j] + o;
              }
            }
          }
#pragma unroll
          for (int hh = 1; hh < NR; hh <<= 1) {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              if ((r & hh) == 0) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float a = qv[r][j], bq = qv[r + hh][j];
                  qv[r][j] = a + bq;
                  qv[r + hh][j] = a - bq;
                }
              }
            }
          }
#pragma unroll
          for (int r = 0; r < NR; ++r) {
#pragma unroll
            for (int j = 0; j < 4; ++j) qv[r][j] *= inv_sqrt_dim<D>();
          }
        }
        float amax = 0.f;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
#pragma unroll
          for (int j = 0; j < 4; ++j) amax = fmaxf(amax, fabsf(qv[r][j]));
        }
  return amax;
}

// Weighted position of a CTA on the virtual axis in units of 1 / (148 * 1000 * waves) of the whole: two or three launch
// waves of 148 CTAs (one per CTA that an SM holds) with weights W0, [1000,] 2000 - W0.
template <int WAVES> struct WaveWeights;
template <> struct WaveWeights<3> { static constexpr int w[3] = {1040, 1000, 960}; };
template <> struct WaveWeights<2> { static constexpr int w[3] = {1010, 990, 0}; };
template <int WAVES>
__host__ __device__ __forceinline__ long long wave_prefix(int cta) {
  constexpr int W0 = WaveWeights<WAVES>::w[0], W1 = WaveWeights<WAVES>::w[1], W2 = WaveWeights<WAVES>::w[2];
  const int k = cta / 148, r = cta % 148;
  return (k == 0 ? 0 : k == 1 ? W0 : k == 2 ? W0 + W1 : W0 + W1 + W2) * 148ll + (long long)r * (k == 0 ? W0 : k == 1 ? W1 : W2);
}
// First virtual page of a CTA's share: equal shares, or shares weighted by launch wave.
template <int WAVES>
static __host__ __device__ __forceinline__ long long share_start_virtual(const FlatPlan& plan, bool waves, int cta) {
  if (!waves) return plan.lo(cta);
  return plan.N * wave_prefix<WAVES>(cta) / (148ll * 1000 * WAVES);
}
// The CTA whose share holds virtual page v: the largest c with N prefix(c) < (v + 1) U, found wave by wave (the
// prefix is linear inside a wave), one division.
template <int WAVES>
static __host__ __device__ __forceinline__ int cta_of_virtual(const FlatPlan& plan, bool waves, long long v) {
  if (!waves) return plan.cta_of(v);
  constexpr int W0 = WaveWeights<WAVES>::w[0], W1 = WaveWeights<WAVES>::w[1], W2 = WaveWeights<WAVES>::w[2];
  const long long a = (v + 1) * (148ll * 1000 * WAVES) - 1;      // N prefix(c) <= a
  const long long b1 = plan.N * (148ll * W0), b2 = plan.N * (148ll * (W0 + W1));
  const int k = (WAVES == 3 && a >= b2) ? 2 : a >= b1 ? 1 : 0;
  const long long base = k == 2 ? b2 : k == 1 ? b1 : 0;
  const long long r = divide(a - base, plan.N * (k == 2 ? W2 : k == 1 ? W1 : W0));
  return 148 * k + (int)(r < 147 ? r : 147);
}
// Where a CTA's share starts: its first real page, flat and as (sequence, KV head, page).  sPref, sVPref: pages per sequence over all KV
// heads, and pages with gaps, as prefixes over the batch.  The CTA behind the last one that takes part starts where the pages end.
struct ShareStart { long long x; int b, h, page; };
template <int WAVES>
static __host__ __device__ __forceinline__ ShareStart share_start(const FlatPlan& plan, bool waves, int cta, const int* sPref,
                                                     const int* sVPref, int B, int Hkv, int gap) {
  const long long v = share_start_virtual<WAVES>(plan, waves, cta);
  if (v >= plan.N) return {sPref[B], 0, 0, 0};
  int lo_ = 0, hi_ = B - 1;                        // last batch entry with sVPref <= v
  while (lo_ < hi_) {
    const int mid = (lo_ + hi_ + 1) >> 1;
    if (sVPref[mid] <= v) lo_ = mid; else hi_ = mid - 1;
  }
  const int len = (sVPref[lo_ + 1] - sVPref[lo_]) / Hkv, pb = len - gap;
  const int vs = (int)v - sVPref[lo_], hh = vs / len, off = vs - hh * len, pg = off > gap ? off - gap : 0;
  return {(long long)sPref[lo_] + (long long)hh * pb + pg, lo_, hh, pg};
}
// The CTA that holds a virtual page of a stream whose first page is xs: which = 0 its first page, 1 its last one, 2 the page before the gap
// in front of it (-1 where there is none).
template <int WAVES>
static __host__ __device__ __forceinline__ int stream_cta(const FlatPlan& plan, bool waves, long long xs, int pages, int gap, int which) {
  const long long v = which == 0 ? xs : which == 1 ? xs + pages - 1 : xs - gap - 1;
  return v < 0 ? -1 : cta_of_virtual<WAVES>(plan, waves, v);
}
// The CTAs of a stream, from those three: its partials are those of first .. last.  window: the one that takes its residual window - the
// first whose share lies in the gap in front of the stream (short contexts), else the one with the first page.
struct StreamCtas {
  int first, last, window;
  __host__ __device__ __forceinline__ StreamCtas(int first_, int last_, int before_gap)
      : first(first_), last(last_), window(before_gap + 1 < first_ ? before_gap + 1 : first_) {}
  __host__ __device__ __forceinline__ int partials() const { return last - first + 1; }
  // CTAs that count themselves in when they are through with the stream
  __host__ __device__ __forceinline__ int counted(bool has_window) const { return partials() + (has_window && window < first ? 1 : 0); }
};
// The time-balanced split (stream gaps) pays where the arithmetic per page limits the kernel (token-wise and
// channel-wise keys alike); pages of 10 bits per element pair and more lose with it and keep the plain split by pages.
__host__ __device__ constexpr int gap_pages(int D, int kb, int vb, int k_axis, int streams) {
  return kb + vb <= 8 ? (k_axis == 1 ? kGapPagesChan : D == 64 && streams <= kGapStreams64 ? kGapPages64 : kGapPages) : 0;
}
// Whether the shares of a full grid are weighted by launch wave: only where every stream's partials fit its slots all the
// same.  A stream of P pages touches fewer than 2 + (P - 1) / s CTAs when no share is smaller than s virtual pages (the shares
// between its first and its last one lie within its pages), so P - 1 <= (slots - 1) s keeps it within its slots; make_plan
// bounds equal shares the same way, which are larger than the lightest weighted one.
template <int WAVES>
static __host__ __device__ __forceinline__ bool weighted_shares(const FlatPlan& plan, int gap, int grid, int pages_max, int slots) {
  constexpr int WMIN = WaveWeights<WAVES>::w[WAVES - 1];      // lightest wave; s = N WMIN / (1000 grid)
  return gap != 0 && grid == WAVES * 148 && plan.c_eff == grid && plan.N >= 8ll * grid &&
         (pages_max - 1) * 1000ll * grid <= (slots - 1) * plan.N * WMIN;
}

// D += A(16x16, row) * B(16x8, col), bf16 operands, fp32 accumulate.
__device__ __forceinline__ void mma16816_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Attention over the residual window (Sec. 4.1's buffer of recent full-precision tokens) of one stream, by the four consumer warps: the
// newest nw <= 127 tokens are 16-bit rows in a ring (key row, value row of slot i side by side), positions f .. f + nw - 1.  Leaves the
// partial (m, l, o) at `part`, or the output of a stream that has no pages (part = nullptr).  Run once per stream, it is bound by
// fetching its instructions and by latency, so it is kept short: a thread sums two channels over every 128 / (D / 2)-th token.  Logits are
// exact products of the 16-bit keys and queries, summed in fp32 by the tensor cores, 16 tokens a warp and step, a column per (row,
// head) pair; weights and the sums of weighted values are fp32.  scratch: 128 x 4 NH floats; red_max, red_sum: 4 x 8 each; win: the rows,
// in global or shared memory.  As a kernel of its own in front of this one (32 CTAs on 148 SMs, then a launch that waits for it) the window
// cost 7 us a layer: eight layers of 4 x 8 streams of 2,000 tokens with two drafted rows 192 us, 154 here; always by the CTA with the
// stream's first page 182.
template <int D, int NH>
__device__ __forceinline__ void window_partial(const Geom& g, const uint16_t* win, const uint16_t* __restrict__ q, float c1, int n, int f, int nw,
                                               float* scratch, float* red_max, float* red_sum, float* __restrict__ part, void* __restrict__ out,
                                               size_t out0, int out_dtype) {
  constexpr int NC = 128, NR = D / 16, VH = 4 * NH, TG = NC / (D / 2);       // token groups of the weighted values
  constexpr uint32_t FULL = 0xffffffffu;
  const int tid_ = threadIdx.x, lane = tid_ & 31, warp = tid_ >> 5, gid = lane >> 2, tid = lane & 3;
  const int Gq = g.G, nvh = g.G * g.rows;
  const bool bf = g.in_dtype == KVQ_BF16;
  const int cp = tid_ % (D / 2), tg = tid_ / (D / 2);
  // ---- logits: warp w takes tokens 16 w .. 16 w + 15 and, of a window of 128, those 64 behind
  uint2 qf[NR];
  {
    const uint16_t* qrow = q + (size_t)(gid / Gq) * g.Hq * D + (size_t)(gid % Gq) * D;
#pragma unroll
    for (int r = 0; r < NR; ++r) qf[r] = gid < nvh ? *reinterpret_cast<const uint2*>(qrow + 16 * r + 4 * tid) : make_uint2(0u, 0u);
  }
  float m0 = -INFINITY, m1 = -INFINITY;          // of (row, head) pairs 2 tid, 2 tid + 1
  const int lim0 = n - f - (g.rows - 1 - min(2 * tid / Gq, g.rows - 1)), lim1 = n - f - (g.rows - 1 - min((2 * tid + 1) / Gq, g.rows - 1));
#pragma unroll 1
  for (int t0 = 16 * warp; t0 < nw; t0 += 64) {
    const uint16_t* ka = win + (size_t)(t0 + gid) * 2 * D + 4 * tid;       // (rows beyond nw are there, in the window or in the ring, see window_fits_ring; their logits are dropped)
    float S[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const uint2 a = *reinterpret_cast<const uint2*>(ka + 16 * r), b = *reinterpret_cast<const uint2*>(ka + 16 * D + 16 * r);
      if (bf) mma16816_bf16(S, a.x, b.x, a.y, b.y, qf[r].x, qf[r].y);
      else mma16816(S, a.x, b.x, a.y, b.y, qf[r].x, qf[r].y);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int t = t0 + gid + 8 * e;
      const float x = t < min(nw, lim0) ? c1 * S[2 * e] : -INFINITY, y = t < min(nw, lim1) ? c1 * S[2 * e + 1] : -INFINITY;
      m0 = fmaxf(m0, x); m1 = fmaxf(m1, y);
      if (2 * tid < VH) *reinterpret_cast<float2*>(scratch + t * VH + 2 * tid) = make_float2(x, y);
    }
  }
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) {
    m0 = fmaxf(m0, __shfl_xor_sync(FULL, m0, off));
    m1 = fmaxf(m1, __shfl_xor_sync(FULL, m1, off));
  }
  if (gid == 0) { red_max[warp * 8 + 2 * tid] = m0; red_max[warp * 8 + 2 * tid + 1] = m1; }
  named_bar_sync(1, NC);
  // ---- weights: thread (token, pair) by pairs; sums per warp
  {
    const int vh = tid_ % VH;
    const float m = fmaxf(fmaxf(red_max[vh], red_max[8 + vh]), fmaxf(red_max[16 + vh], red_max[24 + vh]));
    float sum = 0.f;
    for (int t = tid_ / VH; t < nw; t += NC / VH) {
      const float p = m == -INFINITY ? 0.f : exp2f(scratch[t * VH + vh] - m);
      scratch[t * VH + vh] = p;
      sum += p;
    }
    __syncwarp();
#pragma unroll
    for (int off = VH; off < 32; off <<= 1) sum += __shfl_xor_sync(FULL, sum, off);
    if (lane < VH) red_sum[warp * 8 + lane] = sum;
  }
  named_bar_sync(1, NC);
  // ---- weighted values
  float o[VH][2];
#pragma unroll
  for (int e = 0; e < VH; ++e) o[e][0] = o[e][1] = 0.f;
#pragma unroll 8
  for (int t = tg; t < nw; t += TG) {
    const uint32_t raw = *reinterpret_cast<const uint32_t*>(win + ((size_t)t * 2 + 1) * D + 2 * cp);
    const float2 v = bf ? make_float2(__uint_as_float(raw << 16), __uint_as_float(raw & 0xFFFF0000u)) : __half22float2(as_h2(raw));
#pragma unroll
    for (int e = 0; e < VH; e += 4) {
      const float4 w = *reinterpret_cast<const float4*>(scratch + t * VH + e);
      o[e][0] = fmaf(w.x, v.x, o[e][0]); o[e][1] = fmaf(w.x, v.y, o[e][1]);
      o[e + 1][0] = fmaf(w.y, v.x, o[e + 1][0]); o[e + 1][1] = fmaf(w.y, v.y, o[e + 1][1]);
      o[e + 2][0] = fmaf(w.z, v.x, o[e + 2][0]); o[e + 2][1] = fmaf(w.z, v.y, o[e + 2][1]);
      o[e + 3][0] = fmaf(w.w, v.x, o[e + 3][0]); o[e + 3][1] = fmaf(w.w, v.y, o[e + 3][1]);
    }
  }
  named_bar_sync(1, NC);                         // the weights have been read: their place takes the other groups' sums
  if (tg > 0) {
#pragma unroll
    for (int e = 0; e < VH; ++e) *reinterpret_cast<float2*>(scratch + ((tg - 1) * VH + e) * D + 2 * cp) = make_float2(o[e][0], o[e][1]);
  }
  named_bar_sync(1, NC);
  if (tg == 0) {
#pragma unroll
    for (int e = 0; e < VH; ++e) {
#pragma unroll
      for (int k = 0; k < TG - 1; ++k) {
        const float2 x = *reinterpret_cast<const float2*>(scratch + (k * VH + e) * D + 2 * cp);
        o[e][0] += x.x; o[e][1] += x.y;
      }
      if (e < nvh) {
        const float l = (red_sum[e] + red_sum[8 + e]) + (red_sum[16 + e] + red_sum[24 + e]);
        if (part != nullptr) {
          float* dst = part + e * (D + 2);
          if (cp == 0) {
            dst[0] = fmaxf(fmaxf(red_max[e], red_max[8 + e]), fmaxf(red_max[16 + e], red_max[24 + e]));
            dst[1] = l;
          }
          *reinterpret_cast<float2*>(dst + 2 + 2 * cp) = make_float2(o[e][0], o[e][1]);
        } else {
          const size_t oi = out0 + ((size_t)(e / Gq) * g.Hq + e % Gq) * D + 2 * cp;
          const float x = l > 0.f ? o[e][0] / l : 0.f, y = l > 0.f ? o[e][1] / l : 0.f;
          if (out_dtype == KVQ_FP32) *reinterpret_cast<float2*>(static_cast<float*>(out) + oi) = make_float2(x, y);
          else *reinterpret_cast<uint32_t*>(static_cast<uint16_t*>(out) + oi) = (uint32_t)f32_to_bits16(x, out_dtype) | ((uint32_t)f32_to_bits16(y, out_dtype) << 16);
        }
      }
    }
  }
  named_bar_sync(1, NC);                         // the scratch may be used again
}

// Template parameters: head_dim, key bits, value bits, key axis (0 token-wise, 1 channel-wise), key / value groups
// per row, NH = query heads per lane (1: up to 4 heads per KV head, 2: up to 8), resident CTAs per SM.
//
// Both contractions run on integer tensor-core MMAs over the raw code bytes (m16n8k32, int32 accumulate).
// The 8 columns of an MMA carry (head, limb) pairs: q as 16-bit fixed point in two signed bytes for QK^T, the
// softmax weight times the value scale as 32-bit fixed point in four unsigned bytes for PV.  Lane (g, t) of a
// warp (g = lane / 4, t = lane % 4) owns query heads t (and t + 4 when NH = 2): its accumulator columns 2t, 2t+1
// are the limbs of that head, so logits, softmax and the fixed-point weights need no exchange between lanes.
//
// The four consumer warps share a page twice: for logits and weights each takes 32 of its tokens, for PV each takes a quarter of the
// channels of all 128.  In between the weights pass through shared memory as ready MMA operands, behind the page's one
// barrier, which also says whether any warp saw a logit above the common reference (or a value scale above the common
// limit; then all move it and make their weights again).  A warp's accumulators are a quarter of what whole rows per warp take
// (32 registers for 8 heads, where 24-bit weights alone took 96 and spilled): 8 heads have 32-bit weights and four bits of
// headroom too, channel-wise keys three CTAs per SM instead of two, and a stream's end needs no sum over the warps but two scalars per head.
// Bound by the length of the instruction stream: a warp issues every 6 to 7 cycles, so what counts is instructions per page.  A page
// without masks (all but a stream's last) runs code without a condition.  Against whole rows per warp, one layer, 24 calls in a
// replayed graph: 8B shape 32k K4V2 80.0 -> 78.5 us (16k: 48.7 -> 45.4, K2V4 49.6 -> 45.8, K4V4 54.8 -> 51.5, K8V4 75.2 -> 70.7, groups of
// 32 / 64 57.9 / 59.4 -> 52.4 / 52.7); 8 heads per KV head 16 x 16,384 tokens 84 -> 68; channel-wise 16 x 32,768 tokens K4V2 183 -> 154,
// 16,384 tokens K8V2 101.6 -> 88.4; 4 x 8 streams of 4,000 tokens 22.5 -> 18.0.
// The two token rows of a lane share every fp32 operation on logits and weights that has a packed form: two 70B-shaped layers at 128k
// tokens, step 256 -> 251 us, 8B shape 181 -> 179.
constexpr int kConsumerWarps = 4;
template <int D, int KB, int VB, int KAXIS, int NGK, int NGV, int NH, int MINB, bool WIN>
__global__ void __launch_bounds__((kConsumerWarps + 1) * 32, MINB)
decode_mma_kernel(Geom g, CachePtrs c, const uint16_t* __restrict__ q, float c1, float* __restrict__ ws,
                  int s_cap, int stages, void* __restrict__ out, int out_dtype, unsigned long long call_id,
                  unsigned long long wait_ns, long long skip_x) {
  constexpr int NW = kConsumerWarps;
  constexpr int NR = D / 16;                // 16-channel register slots per key row
  constexpr int KS32 = D / 32;              // k-steps of an 8-bit MMA over the channels
  constexpr int MT = D / 16;                // m-tiles of PV (16 channels each)
  constexpr int MTW = MT / NW;              // ... of one warp
  constexpr int KW = D * KB / 128;          // key words per lane per token row
  constexpr int FPBV = 8 / VB;              // value codes per byte (channels 16 apart)
  constexpr int QPW = MTW > FPBV ? MTW / FPBV : 1;   // quads of value words per lane, warp and 32-token block
  constexpr int TPQ = MTW / QPW;            // m-tiles of the warp in a quad
  constexpr int NTV = 2 * NH;               // n-tiles of PV: (head, limb) columns, four limbs
  constexpr int NTK = KAXIS == 1 ? 2 : 1;   // n-tiles of QK^T per head set: two byte limbs of q, or three of q * s
  constexpr int K_ROW_BYTES = D * KB / 8;
  constexpr int V_BLOCK_BYTES = 4 * D * VB;
  // page geometry (the same numbers the host put into Geom)
  constexpr int K_META_OFF = kPageTokens * K_ROW_BYTES;
  constexpr int V_CODES_OFF = K_META_OFF + (KAXIS == 1 ? 4 * D : kPageTokens * NGK * 4);
  constexpr int V_META_OFF = V_CODES_OFF + 4 * V_BLOCK_BYTES;
  constexpr int NCONS = NW * 32;
  constexpr uint32_t FULL = 0xffffffffu;
  const int GAP = gap_pages(D, KB, VB, KAXIS, g.B * g.Hkv);      // (known at compile time at head_dim 128)
  constexpr int WAVES = MINB;               // CTAs per SM = launch waves (the weights apply to a grid of 148 * WAVES)
  static_assert(MT % NW == 0 && (MT / NGV) % MTW == 0, "a warp's channels are whole m-tiles of one value group");
  static_assert(KAXIS == 0 || KB != 2, "channel-wise 2-bit keys are not instantiated");
  constexpr bool NIBBLES = KB == 4 && KAXIS == 0 && NH == 1 && NR / NGK >= 4;      // key codes by nibble (see the logits)
  static_assert(MT % FPBV == 0, "value m-tiles come in groups that share a byte");

  extern __shared__ __align__(128) uint8_t smem[];
  const SmemLayout sl = smem_layout(g.page_bytes, stages, g.B, D, NH, NGV, KAXIS == 1);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + sl.bar_off);   // full[0..stages), empty[0..stages)
  int* sPref = reinterpret_cast<int*>(smem + sl.pref_off);
  int* sVPref = sPref + (g.B + 1);                                   // the same prefix with GAP more per stream
  // [0] CTA that takes the segment's window, [1] abort flag, [2] published count, [3] CTAs that count themselves, [4..7] share ends, [8..9] segment
  // slot / partials, [10] CTAs taking part, [11..13] cursor, [14] weighted shares, [15] free.  A word has one meaning and one place that sets it
  // (besides the abort flag's start): whoever reads it is a barrier away from that place on both sides.
  int* sMisc = reinterpret_cast<int*>(smem + sl.misc_off);
  double* sZ = reinterpret_cast<double*>(smem + sl.red_off);         // [NW][8][NGV] sums of weight x zero-point
  float* sMax = reinterpret_cast<float*>(sZ + NW * 8 * NGV);         // [NW][8] block maxima
  float* sLim = sMax + NW * 8;                                       // [NW][4] value scales (one used)
  float* sSum = sLim + NW * 4;                                       // [NW][8] sums of weights

  const int tid_ = threadIdx.x, lane = tid_ & 31, warp = __shfl_sync(FULL, tid_ >> 5, 0);     // (known to be the same in a warp)
  const int gid = lane >> 2, tid = lane & 3;
  // Several query rows per head (g.rows > 1) are served as virtual heads: row r of head j is virtual head
  // r * Gq + j, with its own causal limit on the tokens it may see.
  const int B = g.B, Hkv = g.Hkv, Gq = g.G, G = g.G * g.rows;

  // ---- plan, all of it on warp 0 (the others wait at one barrier): pages per sequence, prefix over the batch,
  // this CTA's share of the pages and the stream its first page lies in
  const int s_plan = s_cap - (g.R ? 1 : 0);       // the last partial slot of a stream belongs to its residual window
  if (warp == 0) {
    if (lane == 0) {
      sPref[0] = 0; sVPref[0] = 0; sMisc[1] = 0;
      for (int s = 0; s < stages; ++s) {
        mbar_init(smem_u32(&bars[s]), 1);
        mbar_init(smem_u32(&bars[stages + s]), 4);
        if constexpr (KAXIS == 1) mbar_init(smem_u32(&bars[2 * stages + s]), 1);     // ready: operands of the page made
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
  }
  begin_after_predecessor();
  // the queries, which a stream's start waits for, come to L2 while the split is worked out
  for (long long i = ((long long)blockIdx.x * blockDim.x + tid_) * 64; i < (long long)B * g.rows * g.Hq * D; i += (long long)gridDim.x * blockDim.x * 64)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(q + i));
  if (warp == 0) {
    int carry = 0, vcarry = 0, pmax = 0;
    for (int base = 0; base < B; base += 32) {
      const int i = base + lane;
      const int pages = (i < B) ? (paged_len(c.seq_len, i, g.capacity, g.R) + kPageTokens - 1) >> 7 : 0;
      pmax = max(pmax, pages);
      int v = pages * Hkv;
      int vv = v > 0 ? v + GAP * Hkv : 0;
      for (int off = 1; off < 32; off <<= 1) {
        int u = __shfl_up_sync(FULL, v, off), uu = __shfl_up_sync(FULL, vv, off);
        if (lane >= off) { v += u; vv += uu; }
      }
      if (i < B) { sPref[i + 1] = v + carry; sVPref[i + 1] = vv + vcarry; }
      carry += __shfl_sync(FULL, v, 31);
      vcarry += __shfl_sync(FULL, vv, 31);
    }
    for (int off = 16; off; off >>= 1) pmax = max(pmax, __shfl_xor_sync(FULL, pmax, off));
    __syncwarp();
    if (lane < 2) {
      // lane 0: the share's first page, the CTAs that take part and the cursor; lane 1: the share's end
      const FlatPlan p0 = make_plan(vcarry, pmax + GAP, gridDim.x, s_plan);
      const bool w0 = weighted_shares<WAVES>(p0, GAP, gridDim.x, pmax, s_plan);
      ShareStart at{0, 0, 0, 0};
      if (p0.N != 0 && (int)blockIdx.x < p0.c_eff) at = share_start<WAVES>(p0, w0, (int)blockIdx.x + lane, sPref, sVPref, B, Hkv, GAP);
      *reinterpret_cast<long long*>(sMisc + 4 + 2 * lane) = at.x;
      if (lane == 0) { sMisc[10] = p0.c_eff; sMisc[11] = at.b; sMisc[12] = at.h; sMisc[13] = at.page; sMisc[14] = w0; }
    }
  }
  __syncthreads();
  // a sequence without pages has no CTA of its own: its output rows are zero, or the attention over its residual window
  for (int bb = blockIdx.x; bb < B; bb += gridDim.x) {
    if (sPref[bb + 1] == sPref[bb] && (!WIN || clamped_len(c.seq_len, bb, g.capacity) == 0)) {
      for (int i = tid_; i < g.rows * g.Hq * D; i += blockDim.x) {
        const size_t oi = (size_t)bb * g.rows * g.Hq * D + i;
        if (out_dtype == KVQ_FP32) static_cast<float*>(out)[oi] = 0.f;
        else static_cast<uint16_t*>(out)[oi] = 0;
      }
    }
  }
  [[maybe_unused]] auto window_of = [&](int bb, int hh, int n, const uint16_t* rows, float* part) {
    const int f = n / g.R * g.R;
    const size_t first = ((size_t)bb * g.rows * g.Hq + (size_t)hh * Gq) * D;
    window_partial<D, NH>(g, rows, q + first, c1, n, f, n - f, reinterpret_cast<float*>(smem + sl.w_off), sMax, sSum,
                          part, out, first, out_dtype);
  };
  if constexpr (WIN) {
    if (warp < NW) {
#pragma unroll 1
      for (int st = blockIdx.x; st < B * Hkv; st += gridDim.x) {
        const int bb = st / Hkv, n = clamped_len(c.seq_len, bb, g.capacity);
        if (sPref[bb + 1] == sPref[bb] && n > 0) window_of(bb, st - bb * Hkv, n, c.kv_win + (size_t)st * g.R * (2 * D), nullptr);
      }
    }
  }
  if (sVPref[B] == 0 || (int)blockIdx.x >= sMisc[10]) return;
  const int x_lo = (int)*reinterpret_cast<const long long*>(sMisc + 4), x_hi = (int)*reinterpret_cast<const long long*>(sMisc + 6);
  // The CTAs of a stream.  A warp works them out together, a lane each: one thread after the other's divisions held up the first page (16
  // layers of the 1B shape 312 -> 309 us, eight ragged K4V4 layers 147.8 -> 146, window of drafts, with three such lookups, 153.5 -> 145.5; 16
  // windowed sequences of 30,000 tokens 139 -> 135).
  auto stream_ctas = [&](int bb, int hh, int pages) {
    FlatPlan plan;                         // on the virtual axis (pages + a gap in front of every stream); kept in shared memory
    plan.N = sVPref[B];
    plan.c_eff = sMisc[10];
    const long long xs = (long long)sVPref[bb] + (long long)hh * (pages + GAP) + GAP;   // the stream's first real page, virtual axis
    int cta = -1;
    if (lane < (WIN ? 3 : 2)) cta = stream_cta<WAVES>(plan, GAP != 0 && sMisc[14] != 0, xs, pages, GAP, lane);
    return StreamCtas(__shfl_sync(FULL, cta, 0), __shfl_sync(FULL, cta, 1), __shfl_sync(FULL, cta, 2));
  };
  [[maybe_unused]] bool win_only = false;
  if (x_lo >= x_hi) {                                // a share that lies inside a gap
    if constexpr (!WIN) return;
    bool takes = false;
    if (warp == 0) {
      const int bb = sMisc[11], hh = sMisc[12], n = clamped_len(c.seq_len, bb, g.capacity);
      takes = n % g.R != 0 && stream_ctas(bb, hh, (sPref[bb + 1] - sPref[bb]) / Hkv).window == (int)blockIdx.x;
    }
    if (!__syncthreads_or(takes)) return;            // (all warps leave or none: the answer comes with the barrier, not through a word)
    win_only = true;
  }

  // ---- cursor: first page of this CTA -> (b, h, page)
  int b = sMisc[11], h = sMisc[12], page = sMisc[13];
  int pages_b = (sPref[b + 1] - sPref[b]) / Hkv;
  const uint32_t ring = smem_u32(smem);
  const uint32_t bar0 = smem_u32(bars);
  volatile int* abort_flag = sMisc + 1;
  volatile int* n_published = sMisc + 2;      // count returned for the partial just published
  const unsigned long long id40 = (call_id & 0xFFFFFFFFFFull) ? (call_id & 0xFFFFFFFFFFull) : 1ull;

  // =========================================================== producer warp
  if (KAXIS == 0 && warp == NW) {
    if (lane == 0) {
      int it = 0, stage = 0;
      uint32_t phase = 1;                // parity of the previous round of `empty`
      bool ok = true;
      const uint64_t policy = l2_evict_first_policy();
      for (int x = x_lo; x < x_hi; ++x, ++it) {
        if (it >= stages) {
          ok = mbar_wait(bar0 + 8 * (stages + stage), phase, wait_ns);
          if (!ok || *abort_flag) { ok = false; break; }
        }
        const uint8_t* src = c.pages + ((size_t)(b * Hkv + h) * g.n_pages + page) * (size_t)g.page_bytes;
        const uint32_t fb = bar0 + 8 * stage;
        if (x != skip_x) {          // (skip_x: test hook - a page that never arrives makes the consumers' bounded wait expire)
          mbar_expect_tx(fb, (uint32_t)g.page_bytes);
          bulk_load(ring + stage * sl.page_stride, src, (uint32_t)g.page_bytes, fb, policy);
        }
        if (++stage == stages) { stage = 0; phase ^= 1; }
        if (++page == pages_b) {
          page = 0;
          if (++h == Hkv) {
            h = 0;
            do { ++b; } while (b < B && sPref[b + 1] == sPref[b]);
            if (b < B) pages_b = (sPref[b + 1] - sPref[b]) / Hkv;
          }
        }
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(c.status, KVQ_STATUS_DEVICE_TIMEOUT);
      }
      // Never leave while a copy may still be writing this CTA's shared memory: wait (bounded) for the
      // last copies issued, whether or not a consumer is still going to.
      for (int k = 1; k <= stages && k <= it; ++k) {
        const int j = it - k;
        mbar_wait(bar0 + 8 * (j % stages), (j / stages) & 1, wait_ns);
      }
    }
    return;
  }

  // =========================================================== producer and preparation warp (channel-wise keys)
  // Per page, the operand of the integer QK^T MMAs is q_d * s_d in 24-bit fixed point (scale from max|q| of the head
  // times the page's largest channel scale), and sum_d q_d z_d is one fp32 scalar per head.  The warp that issues the copies makes
  // both for every page that has landed, in the lane arrangement the consumers' B fragments have, leaves them in the stage's operand
  // buffer and signals the stage's `ready` barrier; for the incomplete last block it leaves q split into fp16 high and low parts
  // instead (operands of the fp16 MMAs on the tail keys).  Copies come first: it issues into every stage that is free before it takes
  // the next page.  Its time per page bounds the kernel, so the two lanes that share a head split the channel slots (147 instructions a
  // page instead of 270): two ragged 14B-shaped layers 265 -> 231 us, 240 with a sixth warp for the operands, which leaves 96 registers
  // per thread at three CTAs per SM instead of 128, so that the page code spills (270 us without the split work).
  if constexpr (KAXIS == 1) {
    if (warp == NW) {
      constexpr int CSB = NH * 2 * NR * 32 * 4 + 64;
      const uint64_t policy = l2_evict_first_policy();
      int istage = 0, ib = b, ih = h, ipage = page, ipages = pages_b, ix = x_lo;       // the next page to copy
      uint32_t iphase = 1;               // parity of the previous round of `empty`
      int stage = 0, x = x_lo;           // the next page to prepare
      uint32_t phase = 0;
      // the lanes of an even and of the odd operand column share a head: each takes half of the channel slots for both columns
      constexpr int HR = NR / 2;
      const int r0 = HR * (gid & 1), even = lane & ~4;
      float qv[NH][HR][4];
      float amaxB[NH];
      int cur_b = -1, cur_h = -1;
      bool ok = true;
      unsigned long long t_idle = 0;
      auto next_of = [&](int& bb, int& hh, int& pg, int& np) {
        if (++pg == np) {
          pg = 0;
          if (++hh == Hkv) {
            hh = 0;
            do { ++bb; } while (bb < B && sPref[bb + 1] == sPref[bb]);
            if (bb < B) np = (sPref[bb + 1] - sPref[bb]) / Hkv;
          }
        }
      };
      while (x < x_hi) {
        if (ix < x_hi && (ix - x_lo < stages || __all_sync(FULL, mbar_test_wait(bar0 + 8 * (stages + istage), iphase)))) {
          if (lane == 0 && ix != skip_x) {          // (skip_x: test hook - a page that never arrives makes the consumers' bounded wait expire)
            const uint8_t* src = c.pages + ((size_t)(ib * Hkv + ih) * g.n_pages + ipage) * (size_t)g.page_bytes;
            mbar_expect_tx(bar0 + 8 * istage, (uint32_t)g.page_bytes);
            bulk_load(ring + istage * sl.page_stride, src, (uint32_t)g.page_bytes, bar0 + 8 * istage, policy);
          }
          __syncwarp();
          if (++istage == stages) { istage = 0; iphase ^= 1; }
          next_of(ib, ih, ipage, ipages);
          ++ix;
          t_idle = 0;
          continue;
        }
        if (x == ix || !__all_sync(FULL, mbar_test_wait(bar0 + 8 * stage, phase))) {
          // neither a free stage nor a page that has landed: look again, for a bounded time
          const unsigned long long now = __shfl_sync(FULL, globaltimer_ns(), 0);
          if (t_idle == 0) t_idle = now;
          if (now - t_idle > wait_ns || __any_sync(FULL, *abort_flag != 0)) { ok = false; break; }
          continue;
        }
        t_idle = 0;
        if (b != cur_b || h != cur_h) {          // a new stream: its queries
          cur_b = b; cur_h = h;
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
            float q_all[NR][4];
            uint2 q_raw[NR];
            load_q_raw<D>(g, q, b, h, (gid >> 1) + 4 * nh, tid, q_raw);
            float am = convert_q_lane<D>(g, c, q_raw, tid, q_all);
#pragma unroll
            for (int r = 0; r < HR; ++r) {
#pragma unroll
              for (int j = 0; j < 4; ++j) qv[nh][r][j] = (gid & 1) ? q_all[HR + r][j] : q_all[r][j];
            }
            am = fmaxf(am, __shfl_xor_sync(FULL, am, 1));
            amaxB[nh] = fmaxf(am, __shfl_xor_sync(FULL, am, 2));
          }
        }
        const int n_tok = paged_len(c.seq_len, b, g.capacity, g.R);
        const bool tail_pg = n_tok - page * kPageTokens < kPageTokens;
        const uint8_t* sp = smem + stage * sl.page_stride;
        uint32_t* ops = reinterpret_cast<uint32_t*>(smem + sl.chan_off + stage * CSB);     // [NH][2][NR][32]
        float* opf = reinterpret_cast<float*>(ops + NH * 2 * NR * 32);                      // zq[8], hs[8]
        if (tail_pg) {
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
#pragma unroll
            for (int r = 0; r < HR; ++r) {
              uint32_t h0, l0_, h1, l1_;
              split_h2(qv[nh][r][0], qv[nh][r][2], h0, l0_);
              split_h2(qv[nh][r][1], qv[nh][r][3], h1, l1_);
              uint32_t* o = ops + (nh * 2 * NR + r0 + r) * 32 + even;
              o[0] = h0; o[4] = l0_;
              o[NR * 32] = h1; o[NR * 32 + 4] = l1_;
            }
          }
        } else {
          const uint32_t* km = reinterpret_cast<const uint32_t*>(sp + K_META_OFF);
          uint32_t top = 0u;               // (scales are not negative: their bits are in the order of their values)
          if (4 * lane < D) {
            const uint4 mm = *reinterpret_cast<const uint4*>(km + 4 * lane);
            top = max(max(mm.x & 0xFFFFu, mm.y & 0xFFFFu), max(mm.z & 0xFFFFu, mm.w & 0xFFFFu));
          }
          const float smax = meta_s(__reduce_max_sync(FULL, top));
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
            const int hb = (gid >> 1) + 4 * nh;
            const float am = amaxB[nh] * smax;
            const float scale = am > 0.f ? kQFix3 / am : 0.f;
            f32x2 zsum2 = pack2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < HR; ++r) {
              const uint4 mm = *reinterpret_cast<const uint4*>(km + 16 * (r0 + r) + 4 * tid);     // (s, z) of 4 channels
              const uint32_t mw[4] = {mm.x, mm.y, mm.z, mm.w};
              float t[4];
#pragma unroll
              for (int j = 0; j < 4; j += 2) {
                const float2 a = __half22float2(as_h2(mw[j])), d = __half22float2(as_h2(mw[j + 1]));
                const f32x2 q2 = pack2(qv[nh][r][j], qv[nh][r][j + 1]);
                zsum2 = fma2(q2, pack2(a.y, d.y), zsum2);
                const float2 x = unpack2(mul2(mul2(q2, pack2(a.x, d.x)), pack2(scale, scale)));
                t[j] = x.x; t[j + 1] = x.y;
              }
              uint32_t w[3];
              fixed_point_bytes3(t, w);
              uint32_t* o = ops + (nh * 2 * NR + r0 + r) * 32 + even;
              o[0] = w[2]; o[4] = 0u;
              o[NR * 32] = w[1]; o[NR * 32 + 4] = w[0];
            }
            float zsum = unpack2(zsum2).x + unpack2(zsum2).y;
            zsum += __shfl_xor_sync(FULL, zsum, 4);
            zsum += __shfl_xor_sync(FULL, zsum, 1);
            zsum += __shfl_xor_sync(FULL, zsum, 2);
            if (tid == 0 && (gid & 1) == 0) {
              opf[hb] = c1 * zsum;
              opf[8 + hb] = am > 0.f ? c1 / scale : 0.f;
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar0 + 8 * (2 * stages + stage));
        if (++stage == stages) { stage = 0; phase ^= 1; }
        next_of(b, h, page, pages_b);
        ++x;
      }
      if (!ok) {
        *abort_flag = 1;
        if (lane == 0) atomicOr(c.status, KVQ_STATUS_DEVICE_TIMEOUT);
        // never leave while a copy may still be writing this CTA's shared memory: wait (bounded) for those not seen yet
        for (; x < ix; ++x) {
          mbar_wait(bar0 + 8 * stage, phase, wait_ns);
          if (++stage == stages) { stage = 0; phase ^= 1; }
        }
      }
      return;
    }
  }

  // =========================================================== consumer warps
  uint32_t qB[NH][NTK][NR];    // QK^T B operands: column gid = (head gid/2 + 4 nh, limb gid%2), channels 16 r + 4 tid + {0..3};
                               // channel-wise keys: n-tile 0 carries (byte 2 signed, none), n-tile 1 (byte 1, byte 0) unsigned
  float hs[NH];                // c1 / fixed-point scale of q, own heads (tid + 4 nh)
  float qsum[NH][NGK];         // c1 * sum of q over each key group, own heads
  float zq[NH];                // channel-wise keys: c1 * sum_d q_d z_d of the current page, own heads
  float m_ref[NH], l[NH], zacc[NH][NGV];     // reference: the same in all warps; sums: over this warp's tokens
  int Oi[NTV][MTW][4];         // PV accumulators: n-tiles 2 nh, 2 nh + 1 hold limbs (3, 2) and (1, 0) of head tid + 4 nh
  double acc[NH][MTW][2];      // what has been folded out of them: channel 16 (MTW warp + i) + 8 r + gid
  constexpr float PONE = (float)(1u << (kPBits - 1)) * 2.0f;     // 2^PBITS
  // sscale = 2^PBITS / s_lim, s_lim a power of two above every value scale of the stream folded into the weights so far (2^-40 at first)
  constexpr float SSCALE0 = PONE / 9.094947e-13f;
  float sscale = SSCALE0;
  int page_no = 0, stage = 0;
  uint32_t phase = 0;
  bool aborted = false;
  constexpr int KCB = (KW < 4 ? KW : 4) * 4;     // bytes of a lane chunk's first quad of key words
  const int lane_k = (warp * 32 + gid) * K_ROW_BYTES + tid * KCB;
  const int lane_km = K_META_OFF + (warp * 32 + gid) * 4 * NGK;
  const int lane_vm = V_META_OFF + (warp * 32 + gid) * 4 * NGV;
  const int mt0 = MTW * warp;                    // first m-tile of this warp, its field of a value byte, its value group
  const int f0 = mt0 % FPBV, jw = mt0 / (MT / NGV);
  const int lane_v = V_CODES_OFF + (mt0 / FPBV) * 512 + lane * 16;
  constexpr int WB = weight_block_bytes(NH);

  // A page that is not there yet (the whole warp comes here): wait for it, bounded; on expiry set the status and go on without waiting (the barriers keep their
  // protocol, what is computed no longer matters and reads nothing out of range).
  auto wait_slowly = [&](uint32_t bar) {
    if (aborted) return;
    const bool got = mbar_wait_slow(bar, phase, wait_ns);
    if (!__all_sync(FULL, got)) {
      aborted = true;
      *abort_flag = 1;
      if (lane == 0) atomicOr(c.status, KVQ_STATUS_DEVICE_TIMEOUT);
      __syncwarp();
    }
  };
  // Fold the int32 accumulators into 64-bit sums and clear them (the sum of code terms and the sum of zero-points that meets it at
  // the segment's end are each up to a few hundred times their difference).
  auto flush_acc = [&]() {
#pragma unroll
    for (int i = 0; i < MTW; ++i) {
      const double fw = (double)((1.0f / sscale) / (float)(1 << (VB * ((f0 + i) % FPBV))));      // sscale is a power of two
#pragma unroll
      for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) {
          const long long v = (((long long)Oi[2 * nh][i][2 * r] << 24) + ((long long)Oi[2 * nh][i][2 * r + 1] << 16)) +
                              (((long long)Oi[2 * nh + 1][i][2 * r] << 8) + Oi[2 * nh + 1][i][2 * r + 1]);
          acc[nh][i][r] += (double)v * fw;
        }
      }
#pragma unroll
      for (int nt = 0; nt < NTV; ++nt) { Oi[nt][i][0] = Oi[nt][i][1] = Oi[nt][i][2] = Oi[nt][i][3] = 0; }
    }
  };

  for (int x = x_lo; x < x_hi || (WIN && win_only);) {
    const int seg_pages = WIN && win_only ? 0 : min(pages_b - page, x_hi - x);
    const int n_all = clamped_len(c.seq_len, b, g.capacity);
    const int n_tok = g.R ? (n_all / g.R) * g.R : n_all;          // tokens of the sequence that are in the pages
    // a block is unmasked when all of its 32 tokens exist and every query row may see them (several causal rows:
    // row r sees the first n - (rows - 1 - r) tokens of the n the sequence holds, window included)
    const int n_unmasked = min(n_tok, n_all - (g.rows - 1));
    const int stream = b * Hkv + h;
    // the queries are on their way while one warp works out
    [[maybe_unused]] uint2 q_raw[NH][NR];
    if constexpr (KAXIS == 0) {
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) load_q_raw<D>(g, q, b, h, (gid >> 1) + 4 * nh, tid, q_raw[nh]);
    }
    // which of the stream's partials this CTA writes, and how many there are: one warp works it out now, everybody
    // reads it after the barrier at the segment's end (the barrier that closed the last segment keeps its readers apart)
    if (warp == 0) {
      const StreamCtas ctas = stream_ctas(b, h, pages_b);
      if (lane == 0) {
        sMisc[8] = (int)blockIdx.x - ctas.first;
        sMisc[9] = ctas.partials();
        if constexpr (WIN) {
          sMisc[0] = ctas.window;
          sMisc[3] = ctas.counted(n_all > n_tok);
        }
      }
    }

    // the stream's residual window: one more partial, in the slot behind the page partials', by a CTA whose share lies in the gap in
    // front of the stream (its ring is free for the rows), else by the one that has its first page, counted with that one's own
    if constexpr (WIN) {
      if (page == 0 && n_all > n_tok) {
        named_bar_sync(1, NCONS);
        if (sMisc[0] == (int)blockIdx.x) {
          const uint16_t* rows = c.kv_win + (size_t)stream * g.R * (2 * D);
          const int bytes = (n_all - n_tok) * 4 * D;
          if (win_only && window_fits_ring(sl, n_all - n_tok, D)) {
            if (tid_ == 0 && skip_x != -2 - (long long)x_lo) {          // (test hook, as for pages)
              mbar_expect_tx(bar0, (uint32_t)bytes);
              bulk_load(ring, rows, (uint32_t)bytes, bar0, l2_evict_first_policy());
            }
            if (!__all_sync(FULL, mbar_try_wait(bar0, 0))) wait_slowly(bar0);
            rows = reinterpret_cast<const uint16_t*>(smem);
          }
          window_of(b, h, n_all, rows, ws + ((size_t)stream * s_cap + (s_cap - 1)) * G * (D + 2));
        }
      }
    }

    // ---- segment start: q operands, group sums and a clean state for this stream's heads (the scale limit too: under one
    // of another stream with larger values this stream's weights would vanish)
    sscale = SSCALE0;
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) {
      hs[nh] = 0.f;
      if constexpr (KAXIS == 0) {       // (channel-wise keys: the producer warp makes the operands, per page)
        float qv[NR][4];
        float amax = convert_q_lane<D>(g, c, q_raw[nh], tid, qv);
        amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, 1));
        amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, 2));
        // 16-bit fixed point relative to the head's largest entry: Q = rint(q * scale), |Q| <= 32512
        const float scale = amax > 0.f ? kQFix / amax : 0.f;
        const float hsb = amax > 0.f ? c1 / scale : 0.f;
        const f32x2 scale_q = pack2(scale * 0.00390625f, scale * 0.00390625f);
        const float magicf = 12582912.0f + ((gid & 1) ? 0.0f : 128.0f);
        const f32x2 magic = pack2(magicf, magicf);
        const uint32_t sel = (gid & 1) ? 0x0040u : 0x0051u;
        uint32_t qs[NGK];
#pragma unroll
        for (int j = 0; j < NGK; ++j) qs[j] = 0u - (uint32_t)(4 * (NR / NGK)) * __float_as_uint(magicf);      // (what the words carry besides Q)
#pragma unroll
        for (int r = 0; r < NR; ++r) qB[nh][0][r] = fixed_point_limb(qv[r], scale_q, magic, sel, qs[r / (NR / NGK)]);
        hs[nh] = __shfl_sync(FULL, hsb, 8 * tid);
        // the zero-point term uses the sum of the same fixed-point q the MMAs see: the two large terms
        // s (q . c) and z sum(q) of a logit then cancel exactly as they do for the exact q
#pragma unroll
        for (int j = 0; j < NGK; ++j) {
          int v = (int)qs[j];
          v += __shfl_xor_sync(FULL, v, 1);
          v += __shfl_xor_sync(FULL, v, 2);
          qsum[nh][j] = hs[nh] * (float)__shfl_sync(FULL, v, 8 * tid);
        }
        if constexpr (NIBBLES) hs[nh] *= 0.0625f;
      }
      m_ref[nh] = -INFINITY;
      l[nh] = 0.f;
      zq[nh] = 0.f;
#pragma unroll
      for (int j = 0; j < NGV; ++j) zacc[nh][j] = 0.f;
#pragma unroll
      for (int i = 0; i < MTW; ++i) acc[nh][i][0] = acc[nh][i][1] = 0.0;
    }
#pragma unroll
    for (int i = 0; i < MTW; ++i) {
#pragma unroll
      for (int nt = 0; nt < NTV; ++nt) { Oi[nt][i][0] = Oi[nt][i][1] = Oi[nt][i][2] = Oi[nt][i][3] = 0; }
    }

    // Start the stream's count word for this launch, unless another CTA has: the last merge cleared it, so that counting a partial takes
    // one addition at the segment's end.  Started there, by whoever came first, the CTAs of a stream that finished together swapped
    // against one another: one sequence of 30,000 tokens (8B shape, four layers) 162 -> 85 us, 16 layers of the 1B shape that take in 128
    // tokens 328 -> 313, eight ragged K4V4 layers 166 -> 150, 70B-shaped 247 -> 239.  (By another thread than the bookkeeping's and
    // behind the queries: 1 to 2 % of a short step.  A word with other contents is started when it is counted in, see tagged_count.)
    if (tid_ == 32 && (seg_pages < pages_b || n_all > n_tok))
      atomicCAS(reinterpret_cast<unsigned long long*>(ws + tag_offset_floats(B * Hkv, s_cap, G, D)) + stream, 0ull, id40 << 24);

    auto process = [&](auto full_tag, int pp) {
      constexpr bool FULL_PAGE = decltype(full_tag)::value;
      const int nv = FULL_PAGE ? kPageTokens : min(kPageTokens, n_tok - (page + pp) * kPageTokens);
      const bool tail_k = (KAXIS == 1) && (nv < kPageTokens);
      const uint8_t* sp = smem + stage * sl.page_stride;
      uint8_t* wbuf = smem + sl.w_off + (page_no & 1) * (NGV * 4 * WB);
      // ---- logits of the warp's 32 tokens, two tiles of 16; (scale, zero) of their values
      f32x2 L[2][NH];                    // [tile][head], of rows gid and gid + 8
      f32x2 sv[2][NGV], zv[2][NGV];
      const bool active = FULL_PAGE || warp * 32 < nv;
      const bool masked = !FULL_PAGE && (page + pp) * kPageTokens + warp * 32 + 32 > n_unmasked;
      bool trig = false;
      float bmax[NH], smax = 0.f;
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) bmax[nh] = -INFINITY;
      if (active) {
        [[maybe_unused]] const uint32_t* ops = nullptr;      // channel-wise keys: the page's operands
        if constexpr (KAXIS == 1) {
          ops = reinterpret_cast<const uint32_t*>(smem + sl.chan_off + stage * (NH * 2 * NR * 32 * 4 + 64));
          const float* opf = reinterpret_cast<const float*>(ops + NH * 2 * NR * 32);
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
#pragma unroll
            for (int nt = 0; nt < NTK; ++nt) {
#pragma unroll
              for (int r = 0; r < NR; ++r) qB[nh][nt][r] = ops[((nh * 2 + nt) * NR + r) * 32 + lane];
            }
            zq[nh] = opf[tid + 4 * nh];
            hs[nh] = opf[8 + tid + 4 * nh];
          }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int tok0 = warp * 32 + 16 * u + gid;        // page-local tokens of this lane's two rows: tok0, tok0 + 8
          if (KAXIS == 1 && tail_k) {
            // tokens of the incomplete block: fp16 keys from the tail against q as fp16 high + low parts (operand
            // column gid = (head gid/2 + 4 nh, part gid%2), so lane columns 2 tid, 2 tid + 1 are the two parts of
            // head tid + 4 nh)
            const uint16_t* tl = c.k_tail + ((size_t)stream * kPageTokens + tok0) * D;
            const bool v0 = tok0 < nv, v1 = tok0 + 8 < nv;
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              float S[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
              for (int r = 0; r < NR; ++r) {
                uint2 ra = make_uint2(0u, 0u), rb = make_uint2(0u, 0u);
                if (v0) ra = *reinterpret_cast<const uint2*>(tl + 16 * r + 4 * tid);
                if (v1) rb = *reinterpret_cast<const uint2*>(tl + 8 * D + 16 * r + 4 * tid);
                const uint32_t a0 = __byte_perm(ra.x, ra.y, 0x5410), a1 = __byte_perm(rb.x, rb.y, 0x5410);
                const uint32_t a2 = __byte_perm(ra.x, ra.y, 0x7632), a3 = __byte_perm(rb.x, rb.y, 0x7632);
                mma16816(S, a0, a1, a2, a3, qB[nh][0][r], qB[nh][NTK - 1][r]);    // q's fp16 parts, made by the producer warp
              }
              L[u][nh] = pack2(c1 * (S[0] + S[1]), c1 * (S[2] + S[3]));
            }
          } else {
            uint32_t ka[KW], kb2[KW];
            const uint8_t* krow = sp + lane_k + u * (16 * K_ROW_BYTES);           // this lane's chunk of row tok0
            load_words<KW>(krow, 64, ka);
            load_words<KW>(krow + 8 * K_ROW_BYTES, 64, kb2);
            int S[NGK][NH][NTK][4];
            if constexpr (NIBBLES) {
              // 4-bit codes where four slots share a group: the low nibbles of two words are one MMA's operands, their high nibbles
              // (masked where they stand, codes times 16) another one's with an accumulator of its own; 16 low + high = 16 sum, and
              // the factor is taken out with the query's scale.  No shifts, and chains half as long: two 8B-shaped layers at 32k tokens,
              // step 179 -> 174 us (with two heads a lane the second accumulator costs what the shifts cost)
#pragma unroll
              for (int j = 0; j < NGK; ++j) {
                int hi[4];
#pragma unroll
                for (int i = 0; i < KW / NGK / 2; ++i) {
                  const int w0 = j * (KW / NGK) + 2 * i, w1 = w0 + 1;
                  constexpr uint32_t M = 0x0F0F0F0Fu;
                  const uint32_t l0 = ka[w0] & M, l1 = kb2[w0] & M, l2 = ka[w1] & M, l3 = kb2[w1] & M;
                  const uint32_t h0 = ka[w0] & ~M, h1 = kb2[w0] & ~M, h2 = ka[w1] & ~M, h3 = kb2[w1] & ~M;
                  const uint32_t bl0 = qB[0][0][2 * w0], bl1 = qB[0][0][2 * w1], bh0 = qB[0][0][2 * w0 + 1], bh1 = qB[0][0][2 * w1 + 1];
                  if (i == 0) { mma16832_u8s8_zero(S[j][0][0], l0, l1, l2, l3, bl0, bl1); mma16832_u8s8_zero(hi, h0, h1, h2, h3, bh0, bh1); }
                  else { mma16832_u8s8(S[j][0][0], l0, l1, l2, l3, bl0, bl1); mma16832_u8s8(hi, h0, h1, h2, h3, bh0, bh1); }
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) S[j][0][0][e] = S[j][0][0][e] * 16 + hi[e];
              }
            } else {
#pragma unroll
              for (int s = 0; s < KS32; ++s) {
                const int j = s / (KS32 / NGK);
                const bool first = s % (KS32 / NGK) == 0;
                const uint32_t a0 = key_slot<KB, KW>(ka, 2 * s), a1 = key_slot<KB, KW>(kb2, 2 * s);
                const uint32_t a2 = key_slot<KB, KW>(ka, 2 * s + 1), a3 = key_slot<KB, KW>(kb2, 2 * s + 1);
#pragma unroll
                for (int nh = 0; nh < NH; ++nh) {
#pragma unroll
                  for (int nt = 0; nt < NTK; ++nt) {
                    const uint32_t b0 = qB[nh][nt][2 * s], b1 = qB[nh][nt][2 * s + 1];
                    if (nt == 0) { if (first) mma16832_u8s8_zero(S[j][nh][nt], a0, a1, a2, a3, b0, b1); else mma16832_u8s8(S[j][nh][nt], a0, a1, a2, a3, b0, b1); }
                    else { if (first) mma16832_u8u8_zero(S[j][nh][nt], a0, a1, a2, a3, b0, b1); else mma16832_u8u8(S[j][nh][nt], a0, a1, a2, a3, b0, b1); }
                  }
                }
              }
            }
            // accumulator columns 2 tid, 2 tid + 1 = (hi, lo) limbs of head tid + 4 nh: sum_d code_d Q_d = 256 hi + lo
            // (channel-wise keys: the signed top byte in n-tile 0, the two unsigned lower bytes in n-tile 1; these two meet as integers,
            // the top byte joins them in fp32)
            if constexpr (KAXIS == 1) {
#pragma unroll
              for (int nh = 0; nh < NH; ++nh) {
                // (the two lower bytes' sums fit 32 bits together: 128 x 255 x 255 x 257 < 2^31)
                const f32x2 lo = pack2((float)(S[0][nh][NTK - 1][0] * 256 + S[0][nh][NTK - 1][1]), (float)(S[0][nh][NTK - 1][2] * 256 + S[0][nh][NTK - 1][3]));
                const f32x2 t = fma2(pack2((float)S[0][nh][0][0], (float)S[0][nh][0][2]), pack2(65536.f, 65536.f), lo);
                L[u][nh] = fma2(t, pack2(hs[nh], hs[nh]), pack2(zq[nh], zq[nh]));
              }
            } else {
              const uint32_t* km = reinterpret_cast<const uint32_t*>(sp + lane_km + u * (16 * 4 * NGK));   // row tok0
#pragma unroll
              for (int j = 0; j < NGK; ++j) {
                const float2 ma = __half22float2(as_h2(km[j]));                       // (scale, zero) of row tok0
                const float2 mb = __half22float2(as_h2(km[8 * NGK + j]));             // ... of row tok0 + 8
                const f32x2 s2 = pack2(ma.x, mb.x), z2 = pack2(ma.y, mb.y);
#pragma unroll
                for (int nh = 0; nh < NH; ++nh) {
                  const f32x2 t = pack2((float)(S[j][nh][0][0] * 256 + S[j][nh][0][1]), (float)(S[j][nh][0][2] * 256 + S[j][nh][0][3]));
                  const f32x2 x = fma2(mul2(s2, pack2(hs[nh], hs[nh])), t, mul2(z2, pack2(qsum[nh][j], qsum[nh][j])));
                  L[u][nh] = j == 0 ? x : add2(L[u][nh], x);
                }
              }
            }
          }
          const uint32_t* vm = reinterpret_cast<const uint32_t*>(sp + lane_vm + u * (16 * 4 * NGV));
#pragma unroll
          for (int j = 0; j < NGV; ++j) {
            const float2 fa = __half22float2(as_h2(vm[j])), fb = __half22float2(as_h2(vm[8 * NGV + j]));
            sv[u][j] = pack2(fa.x, fb.x);
            zv[u][j] = pack2(fa.y, fb.y);
          }
          if (masked) {
            const int tokg = (page + pp) * kPageTokens + tok0;        // position of row tok0 in the sequence
            const bool there0 = tok0 < nv, there1 = tok0 + 8 < nv;
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              // tokens the lane's head may attend to: the causal limit of its query row
              const int lim = n_all - (g.rows - 1 - min((tid + 4 * nh) / Gq, g.rows - 1));
              float2 x = unpack2(L[u][nh]);
              if (!there0 || tokg >= lim) x.x = -INFINITY;
              if (!there1 || tokg + 8 >= lim) x.y = -INFINITY;
              L[u][nh] = pack2(x.x, x.y);
            }
#pragma unroll
            for (int j = 0; j < NGV; ++j) {
              const float2 x = unpack2(sv[u][j]), y = unpack2(zv[u][j]);
              sv[u][j] = pack2(there0 ? x.x : 0.f, there1 ? x.y : 0.f);
              zv[u][j] = pack2(there0 ? y.x : 0.f, there1 ? y.y : 0.f);
            }
          }
#pragma unroll
          for (int j = 0; j < NGV; ++j) smax = fmaxf(smax, fmaxf(unpack2(sv[u][j]).x, unpack2(sv[u][j]).y));
        }
        // ---- softmax reference / scale check (rarely true)
        trig = smax * sscale >= PONE;
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) {
          const float2 x = unpack2(L[0][nh]), y = unpack2(L[1][nh]);
          bmax[nh] = fmaxf(fmaxf(x.x, x.y), fmaxf(y.x, y.y));
          trig |= bmax[nh] > m_ref[nh];
        }
      }

      // ---- weights: p = 2^(logit - reference) <= 2^-headroom, P = rint(p * s_V * sscale) < 2^PBITS, left for all warps as
      // the B operands of the block; the sums over the warp's own tokens are kept apart until the reference holds
      float psum[NH], zsum[NH][NGV];
      auto make_weights = [&]() {
        // One head a lane: sums in one chain, token tok0 + 8 before tok0, tile after tile (neighbouring tokens that cancel do so
        // exactly; the last bits of every output follow this order).  Two heads: two chains, over tok0 and over tok0 + 8, in packed
        // operations; one chain costs two 70B-shaped layers at 128k tokens 4.5 us (246.5 -> 251), one-head shapes nothing.
        constexpr bool CHAINS = NH == 2;
        [[maybe_unused]] f32x2 psum2[NH], zsum2[NH][NGV];
        uint32_t bV[NGV][NTV][2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          f32x2 p[NH];
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
            const float2 x = unpack2(add2(L[u][nh], pack2(-m_ref[nh], -m_ref[nh])));
            float2 e = make_float2(ex2(x.x), ex2(x.y));
            if (masked) {       // a head that has seen no token yet has no reference: its weights are zero
              const float2 y = unpack2(L[u][nh]);
              if (y.x == -INFINITY) e.x = 0.f;
              if (y.y == -INFINITY) e.y = 0.f;
            }
            p[nh] = pack2(e.x, e.y);
            if constexpr (CHAINS) psum2[nh] = u == 0 ? p[nh] : add2(psum2[nh], p[nh]);
            else psum[nh] = u == 0 ? e.x + e.y : psum[nh] + (e.x + e.y);
          }
#pragma unroll
          for (int j = 0; j < NGV; ++j) {
            const f32x2 ss = mul2(sv[u][j], pack2(sscale, sscale));
            uint32_t Pa[NH], Pb[NH];
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              if constexpr (CHAINS) {
                zsum2[nh][j] = u == 0 ? mul2(p[nh], zv[u][j]) : fma2(p[nh], zv[u][j], zsum2[nh][j]);
              } else {
                const float2 e = unpack2(p[nh]), z = unpack2(zv[u][j]);
                zsum[nh][j] = fmaf(e.x, z.x, u == 0 ? e.y * z.y : fmaf(e.y, z.y, zsum[nh][j]));
              }
              const float2 x = unpack2(mul2(p[nh], ss));
              Pa[nh] = __float2uint_rn(x.x);      // token tok0
              Pb[nh] = __float2uint_rn(x.y);      // token tok0 + 8
            }
            // one 16-bit element per (column, lane row) = that column's limb of tokens (tok0, tok0 + 8); the 8x8
            // transpose turns lane columns into the B operand (column = lane/4, tokens 2t, 2t+8, 2t+1, 2t+9)
#pragma unroll
            for (int nh = 0; nh < NH; ++nh) {
              bV[j][2 * nh][u] = movmatrix_trans(prmt(Pa[nh], Pb[nh], 0x6273));         // limbs (3, 2): bytes a3 b3 a2 b2
              bV[j][2 * nh + 1][u] = movmatrix_trans(prmt(Pa[nh], Pb[nh], 0x4051));     // limbs (1, 0): bytes a1 b1 a0 b0
            }
          }
        }
        if constexpr (CHAINS) {
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
            psum[nh] = unpack2(psum2[nh]).x + unpack2(psum2[nh]).y;
#pragma unroll
            for (int j = 0; j < NGV; ++j) zsum[nh][j] = unpack2(zsum2[nh][j]).x + unpack2(zsum2[nh][j]).y;
          }
        }
#pragma unroll
        for (int j = 0; j < NGV; ++j) {
          uint8_t* w = wbuf + (j * 4 + warp) * WB;
#pragma unroll
          for (int nh = 0; nh < NH; ++nh)
            *reinterpret_cast<uint4*>(w + 512 * nh + lane * 16) = make_uint4(bV[j][2 * nh][0], bV[j][2 * nh][1], bV[j][2 * nh + 1][0], bV[j][2 * nh + 1][1]);
        }
      };
      if (active) make_weights();
      if (named_bar_any(1, NCONS, trig)) {
        // somebody saw a larger logit or value scale: all warps move to the new reference and limit together
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) smax = fmaxf(smax, __shfl_xor_sync(FULL, smax, off));
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) {
#pragma unroll
          for (int off = 4; off < 32; off <<= 1) bmax[nh] = fmaxf(bmax[nh], __shfl_xor_sync(FULL, bmax[nh], off));
          if (gid == 0) sMax[warp * 8 + tid + 4 * nh] = bmax[nh];
        }
        if (lane == 0) sLim[warp * 4] = smax;
        named_bar_sync(1, NCONS);
        flush_acc();                                   // with the scale the accumulated weights were made with
        smax = fmaxf(fmaxf(sLim[0], sLim[4]), fmaxf(sLim[8], sLim[12]));
        if (smax * sscale >= PONE) {
          // next power of two above the largest value scale: p * s * sscale < 2^PBITS for every p <= 1
          sscale = PONE / __uint_as_float((__float_as_uint(smax) & 0x7F800000u) + 0x00800000u);
        }
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) {
          const float* mx = sMax + tid + 4 * nh;
          const float bm = fmaxf(fmaxf(mx[0], mx[8]), fmaxf(mx[16], mx[24]));
          if (bm > m_ref[nh]) {
            const float nref = bm + kHeadroom;
            const float a = (m_ref[nh] == -INFINITY) ? 0.f : ex2(m_ref[nh] - nref);
            m_ref[nh] = nref;
            l[nh] *= a;
#pragma unroll
            for (int j = 0; j < NGV; ++j) zacc[nh][j] *= a;
#pragma unroll
            for (int i = 0; i < MTW; ++i) { acc[nh][i][0] *= (double)a; acc[nh][i][1] *= (double)a; }
          }
        }
        if (active) make_weights();
        named_bar_sync(1, NCONS);
      }
      if (active) {
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) {
          l[nh] += psum[nh];
#pragma unroll
          for (int j = 0; j < NGV; ++j) zacc[nh][j] += zsum[nh][j];
        }
      }

      // ---- PV of the warp's channels over the page's blocks, on the raw code bytes: one mask per register.  Field f of every
      // byte belongs to m-tile FPBV q + f, whose accumulators carry the factor 2^(VB f).
#pragma unroll
      for (int blk = 0; blk < 4; ++blk) {
        if (FULL_PAGE || blk * 32 < nv) {
          const uint8_t* w = wbuf + (jw * 4 + blk) * WB;
          uint32_t bw[NTV][2];
#pragma unroll
          for (int nh = 0; nh < NH; ++nh) {
            const uint4 w4 = *reinterpret_cast<const uint4*>(w + 512 * nh + lane * 16);
            bw[2 * nh][0] = w4.x; bw[2 * nh][1] = w4.y; bw[2 * nh + 1][0] = w4.z; bw[2 * nh + 1][1] = w4.w;
          }
#pragma unroll
          for (int qd = 0; qd < QPW; ++qd) {
            const uint4 vw = *reinterpret_cast<const uint4*>(sp + lane_v + blk * V_BLOCK_BYTES + qd * 512);
#pragma unroll
            for (int t = 0; t < TPQ; ++t) {
              const int i = qd * TPQ + t;
              uint32_t a0 = vw.x, a2 = vw.y, a1 = vw.z, a3 = vw.w;     // words (rh, kh) = (0,0), (0,1), (1,0), (1,1)
              if constexpr (VB != 8) {
                constexpr uint32_t M0 = ((1u << VB) - 1u) * 0x01010101u;
                const uint32_t mask = M0 << (VB * (TPQ == FPBV ? t : f0 + t));
                a0 &= mask; a1 &= mask; a2 &= mask; a3 &= mask;
              }
#pragma unroll
              for (int nt = 0; nt < NTV; ++nt) mma16832_u8u8(Oi[nt][i], a0, a1, a2, a3, bw[nt][0], bw[nt][1]);
            }
          }
        }
      }
    };

#pragma unroll 1
    for (int pp = 0; pp < seg_pages; ++pp) {
      if (!__all_sync(FULL, mbar_try_wait(bar0 + 8 * stage, phase))) wait_slowly(bar0 + 8 * stage);
      if constexpr (KAXIS == 1) {         // the operands of the page
        if (!__all_sync(FULL, mbar_try_wait(bar0 + 8 * (2 * stages + stage), phase))) wait_slowly(bar0 + 8 * (2 * stages + stage));
      }
      // a page whose tokens all exist and may be seen by every query row needs no masks
      if ((page + pp + 1) * kPageTokens <= n_unmasked) process(std::true_type{}, pp);
      else process(std::false_type{}, pp);
      __syncwarp();
      mbar_arrive_if(bar0 + 8 * (stages + stage), lane == 0);
      if (++stage == stages) { stage = 0; phase ^= 1; }
      if ((++page_no & (kFlushPages - 1)) == 0) flush_acc();      // long before the int32 accumulators can overflow
    }

    // ---- segment end: sum over the warps' tokens, write this warp's channels of the partial
    {
      flush_acc();
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        double z[NGV];
#pragma unroll
        for (int j = 0; j < NGV; ++j) z[j] = (double)zacc[nh][j];
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
          l[nh] += __shfl_xor_sync(FULL, l[nh], off);
#pragma unroll
          for (int j = 0; j < NGV; ++j) z[j] += __shfl_xor_sync(FULL, z[j], off);
        }
        if (gid == 0) {
          sSum[warp * 8 + tid + 4 * nh] = l[nh];
#pragma unroll
          for (int j = 0; j < NGV; ++j) sZ[(warp * 8 + tid + 4 * nh) * NGV + j] = z[j];
        }
      }
      named_bar_sync(1, NCONS);
      // The flat split gives a stream to a run of consecutive CTAs, one partial slot each.  A CTA that holds the
      // whole stream writes the output at once; otherwise it stores its partial, counts itself in, and the CTA
      // that completes the count merges all partials of the stream by log-sum-exp and stores the output.
      const int slot = sMisc[8], n_part = sMisc[9];
      const bool has_win = WIN && n_all > n_tok;                 // its partial is in slot s_cap - 1
      if ((slot >= 0 && slot < s_plan) || (WIN && win_only)) {
        const bool direct = n_part == 1 && !has_win;
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) {
          const int head = tid + 4 * nh;
          if (head < G && !(WIN && win_only)) {
            float lsum = 0.f;
            double zsum = 0.0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
              lsum += sSum[w * 8 + head];
              zsum += sZ[(w * 8 + head) * NGV + jw];
            }
            const size_t oi = (((size_t)b * g.rows + head / Gq) * g.Hq + (size_t)h * Gq + head % Gq) * D;
            float* dst = ws + (((size_t)stream * s_cap + slot) * G + head) * (D + 2);
            if (!direct && warp == 0 && gid == 0) { dst[0] = m_ref[nh]; dst[1] = lsum; }
#pragma unroll
            for (int i = 0; i < MTW; ++i) {
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                const int d = 16 * (mt0 + i) + 8 * r + gid;
                const float o = (float)(acc[nh][i][r] + zsum);
                if (direct) {
                  const float v = lsum > 0.f ? o / lsum : 0.f;
                  if (out_dtype == KVQ_FP32) static_cast<float*>(out)[oi + d] = v;
                  else static_cast<uint16_t*>(out)[oi + d] = f32_to_bits16(v, out_dtype);
                } else {
                  dst[2 + d] = o;
                }
              }
            }
          }
        }
        if (!direct) {
          __threadfence();
          named_bar_sync(1, NCONS);
          unsigned long long* counts = reinterpret_cast<unsigned long long*>(ws + tag_offset_floats(B * Hkv, s_cap, G, D));
          if (tid_ == 0) *n_published = (int)tagged_count(counts + stream, id40);
          named_bar_sync(1, NCONS);
          if (*n_published == (WIN ? sMisc[3] : n_part)) {
            __threadfence();
            // a warp per head, two or four channels per lane; eight partials' loads are in flight at a time
            constexpr int C2 = D / 64;
#pragma unroll 1
            for (int head = warp; head < G; head += NW) {
              const float* base = ws + (((size_t)stream * s_cap) * G + head) * (D + 2);
              const size_t slot_stride = (size_t)G * (D + 2);
              float mstar = -INFINITY, den = 0.f;
              float2 num[C2];
#pragma unroll
              for (int e = 0; e < C2; ++e) num[e] = make_float2(0.f, 0.f);
              const int n_merge = n_part + (has_win ? 1 : 0);
#pragma unroll 1
              for (int j0 = 0; j0 < n_merge; j0 += 8) {
                float2 ml[8], oj[8][C2];
#pragma unroll
                for (int u = 0; u < 8; ++u) {                   // issue the loads of a batch before using any
                  const bool on = j0 + u < n_merge;
                  const int sj = (j0 + u < n_part) ? j0 + u : s_cap - 1;      // the window's partial comes last
                  const float2* pj = reinterpret_cast<const float2*>(base + (size_t)(on ? sj : 0) * slot_stride);
                  ml[u] = on ? __ldcg(pj) : make_float2(-INFINITY, 0.f);
#pragma unroll
                  for (int e = 0; e < C2; ++e) oj[u][e] = on ? __ldcg(pj + 1 + lane + 32 * e) : make_float2(0.f, 0.f);
                }
                float mb = mstar;
#pragma unroll
                for (int u = 0; u < 8; ++u) mb = fmaxf(mb, ml[u].x);
                if (mb == -INFINITY) continue;
                const float keep = (mstar == -INFINITY) ? 0.f : ex2(mstar - mb);
                den *= keep;
#pragma unroll
                for (int e = 0; e < C2; ++e) { num[e].x *= keep; num[e].y *= keep; }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const float wgt = (ml[u].x == -INFINITY) ? 0.f : ex2(ml[u].x - mb);
                  den = fmaf(wgt, ml[u].y, den);
#pragma unroll
                  for (int e = 0; e < C2; ++e) { num[e].x = fmaf(wgt, oj[u][e].x, num[e].x); num[e].y = fmaf(wgt, oj[u][e].y, num[e].y); }
                }
                mstar = mb;
              }
              const size_t oi = (((size_t)b * g.rows + head / Gq) * g.Hq + (size_t)h * Gq + head % Gq) * D;
#pragma unroll
              for (int e = 0; e < C2; ++e) {
                const float rx = den > 0.f ? num[e].x / den : 0.f, ry = den > 0.f ? num[e].y / den : 0.f;
                const int d = 2 * (lane + 32 * e);
                if (out_dtype == KVQ_FP32) *reinterpret_cast<float2*>(static_cast<float*>(out) + oi + d) = make_float2(rx, ry);
                else *reinterpret_cast<uint32_t*>(static_cast<uint16_t*>(out) + oi + d) =
                         (uint32_t)f32_to_bits16(rx, out_dtype) | ((uint32_t)f32_to_bits16(ry, out_dtype) << 16);
              }
            }
            if (tid_ == 0) counts[stream] = 0ull;
          }
        }
      }
      named_bar_sync(1, NCONS);
    }

    if (WIN && win_only) {
      if (aborted) mbar_wait(bar0, 0, wait_ns);      // never leave while the copy may still be writing this CTA's shared memory (bounded)
      return;
    }
    // ---- advance the cursor past this segment
    x += seg_pages;
    page += seg_pages;
    if (page == pages_b) {
      page = 0;
      if (++h == Hkv) {
        h = 0;
        do { ++b; } while (b < B && sPref[b + 1] == sPref[b]);
        if (b < B) pages_b = (sPref[b + 1] - sPref[b]) / Hkv;
      }
    }
  }
}

// Launches one instantiation; defined per instantiation unit.
template <int D, int KB, int VB, int KAXIS, int NGK, int NGV, int NH, int MINB>
int launch_mma_inst(const Geom& g, const CachePtrs& c, const void* q, float c1, float* ws, int s_cap,
                    void* out, int out_dtype, unsigned long long call_id, unsigned long long wait_ns, long long skip_x,
                    cudaStream_t stream) {
  const int stages = ring_stages(g, NH, NGV, KAXIS == 1, MINB);
  if (stages < 2) return KVQ_ERR_UNSUPPORTED;
  const SmemLayout sl = smem_layout(g.page_bytes, stages, g.B, D, NH, NGV, KAXIS == 1);
  auto kern = decode_mma_kernel<D, KB, VB, KAXIS, NGK, NGV, NH, MINB, false>;
  if constexpr (KAXIS == 0) {
    if (g.R) kern = decode_mma_kernel<D, KB, VB, KAXIS, NGK, NGV, NH, MINB, true>;
  }
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sl.total) != cudaSuccess)
    return KVQ_ERR_CUDA_LAUNCH;
  const cudaError_t e = launch_dependent(kern, dim3(148 * MINB), (kConsumerWarps + 1) * 32, sl.total, stream, 1, g, c,
                                         static_cast<const uint16_t*>(q), c1, ws, s_cap, stages, out, out_dtype, call_id, wait_ns, skip_x);
  return e == cudaSuccess ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
}

}  // namespace mma
}  // namespace kvq
