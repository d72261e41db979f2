// kvq_quantize_append for a few tokens per sequence (a decoding step, drafted tokens, a short chunk): the whole call in one
// launch - token-wise quantization, channel-wise keys with their tail, the residual window and the new sequence lengths.
//
// A cluster of up to eight CTAs serves one sequence and the CTAs share out its KV heads; when all have read the old length
// (cluster barrier) one thread stores the new one.  A token row is spread over D / 8 lanes, eight consecutive channels each; lanes whose
// codes share bytes merge them with shuffles.  The call is bound by latency, not by bytes: the code is kept short and is
// the same for every width, because in a step the instructions come from L2 each time.  The task kernels of
// kvq_quantize.cu (32 tokens a warp, several thousand instructions) and a launch for the lengths take 4.2 us at the least and 6 to 7 for a
// few tokens, this kernel 2.9 at the least and 4.5.
#include "kvq_quantize.cuh"

namespace kvq {

namespace {

constexpr int kMaxThreads = 1024;
inline int heads_per_cta(int n_kv_heads) { return (n_kv_heads + 7) / 8; }
constexpr int kChanThreads = 256;       // channel-wise keys: what a block's registers are laid out for

__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();                         // (.aligned takes whole warps; loops before it end lane by lane)
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// CHAN: channel-wise keys (head_dim 128, 4 or 8 bits), else keys are token-wise.  ROT: keys are rotated.
template <int D, int DTYPE, bool ROT, bool CHAN>
__global__ void __launch_bounds__(CHAN ? kChanThreads : kMaxThreads)
append_rows_kernel(Geom g, CachePtrs c, const uint16_t* __restrict__ k_new, const uint16_t* __restrict__ v_new, int64_t sb,
                   int64_t sh, int64_t st, int t_new) {
  constexpr int LPR = D / 8, RPW = 32 / LPR;             // lanes per row, rows per warp
  const int b = blockIdx.y, rank = blockIdx.x, ranks = gridDim.x;
  const int tid = threadIdx.x, lane = tid & 31, l = lane % LPR;
  begin_after_predecessor();
  const int t0 = c.seq_len[b];
  const bool fits = append_fits(t0, t_new, g.capacity);
  if (fits) {
    const int nh = (g.Hkv - rank + ranks - 1) / ranks;   // this CTA's heads: rank, rank + ranks, ...
    const int R = g.R, end = t0 + t_new;
    const int qa = R ? (t0 / R) * R : t0, qb = R ? (end / R) * R : end;      // tokens to quantize now
    const int nq = qb - qa, total = nh * (CHAN ? 1 : 2) * nq;
    // the next row's loads are in flight while this one is quantized (16 layers of the 1B shape that take in 128 tokens, four turns of
    // rows a warp, and decode: 351 -> 338 us)
    struct Row { uint4 raw; int hs, t; };
    auto fetch = [&](int base) {
      const int idx = base + lane / LPR < total ? base + lane / LPR : base;
      Row r;
      r.hs = idx / nq;
      r.t = qa + idx - r.hs * nq;
      const bool is_v = CHAN || (r.hs & 1) == 0;
      const int h = rank + ranks * (CHAN ? r.hs : r.hs >> 1);
      const uint16_t* src = (is_v ? v_new : k_new) + (int64_t)b * sb + (int64_t)h * sh + (int64_t)(r.t - t0) * st;
      if (r.t < t0) src = c.kv_win + (((size_t)b * g.Hkv + h) * R + r.t % R) * (2 * D) + (is_v ? D : 0);       // still in the residual window
      r.raw = *reinterpret_cast<const uint4*>(src + 8 * l);
      return r;
    };
    const int first = (tid >> 5) * RPW, step = (blockDim.x >> 5) * RPW;
    Row next{};
    if (first < total) next = fetch(first);
    for (int base = first; base < total; base += step) {
      const bool active = base + lane / LPR < total;
      const int hs = next.hs, t = next.t;
      const bool is_v = CHAN || (hs & 1) == 0;
      const int h = rank + ranks * (CHAN ? hs : hs >> 1), bh = b * g.Hkv + h;
      const uint4 raw = next.raw;
      if (base + step < total) next = fetch(base + step);
      const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
      float x[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        x[2 * i] = bits16_to_f32((uint16_t)(rw[i] & 0xFFFF), DTYPE);
        x[2 * i + 1] = bits16_to_f32((uint16_t)(rw[i] >> 16), DTYPE);
      }
      if constexpr (ROT && !CHAN) {
        float y[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = x[i];
        rotate_row8<D>(y, c.k_signs, l);
        if (!is_v) {
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = y[i];
        }
      }
      const int bits = is_v ? g.vb : g.kb, gsz = is_v ? g.gv : g.gk, lpg = gsz >> 3;       // lanes per group
      const float qmax = (float)((1 << bits) - 1);
      float mn = fminf(fminf(fminf(x[0], x[1]), fminf(x[2], x[3])), fminf(fminf(x[4], x[5]), fminf(x[6], x[7])));
      float mx = fmaxf(fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])), fmaxf(fmaxf(x[4], x[5]), fmaxf(x[6], x[7])));
#pragma unroll
      for (int off = 1; off < LPR; off <<= 1) {
        const float a = __shfl_xor_sync(FULL, mn, off), z = __shfl_xor_sync(FULL, mx, off);
        if (off < lpg) { mn = fminf(mn, a); mx = fmaxf(mx, z); }
      }
      const GroupParams p = group_params(mn, mx, qmax);
      uint32_t n[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) n[i] = code_of_fast(x[i], p, qmax);
      // fields of a byte: channels 16 apart, that is lanes 2 (and 4) apart; every lane of a byte ends up with all its fields
      const int lf = bits == 8 ? 0 : bits == 4 ? 1 : 2;      // log2 of the fields per byte
      const int rh = l & 1, f = (l >> 1) & ((1 << lf) - 1), mw = l >> (1 + lf);
      uint32_t w[2];
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        w[hh] = (n[4 * hh] | (n[4 * hh + 1] << 8) | (n[4 * hh + 2] << 16) | (n[4 * hh + 3] << 24)) << (bits * f);
        const uint32_t o2 = __shfl_xor_sync(FULL, w[hh], 2);
        if (lf >= 1) w[hh] |= o2;
        const uint32_t o4 = __shfl_xor_sync(FULL, w[hh], 4);
        if (lf == 2) w[hh] |= o4;
      }
      if (!active) continue;
      uint8_t* pg = c.pages + ((size_t)bh * g.n_pages + (t >> 7)) * g.page_bytes;
      const int tp = t & 127, ng = D / gsz;
      if ((l & (lpg - 1)) == 0)
        reinterpret_cast<uint32_t*>(pg + (is_v ? g.v_meta_off : g.k_meta_off))[tp * ng + (8 * l) / gsz] = p.meta;
      if (!is_v) {
        const int wpc = D * bits / 128;
        uint8_t* row = pg + tp * (D * bits / 8);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh)
          if (lf == 0 || f == hh) *reinterpret_cast<uint32_t*>(row + chunk_word_byte(2 * rh + hh, mw, wpc, 4)) = w[hh];
      } else {
        const int tau = tp & 31, kh = tau >> 4, u = tau & 15;
        uint8_t* vb = pg + g.v_codes_off + (tp >> 5) * (4 * D * bits) + mw * 512 + ((u & 7) >> 1) * 16 +
                      4 * (2 * rh + kh) + 2 * (u & 1) + (u >> 3);
        const uint64_t bytes = (uint64_t)w[0] | ((uint64_t)w[1] << 32);
        for (int i = (8 >> lf) * f; i < (8 >> lf) * (f + 1); ++i) vb[64 * i] = (uint8_t)(bytes >> (8 * i));
      }
    }
    if constexpr (CHAN) {
      __shared__ KchanShared scratch;
      for (int h = rank; h < g.Hkv; h += ranks) {
        const int bh = b * g.Hkv + h;
        const uint16_t* in = k_new + (int64_t)b * sb + (int64_t)h * sh - (int64_t)t0 * st + (tid & 15) * 8;
        if ((end >> 7) > (t0 >> 7)) {
          if (g.kb == 4) kchan_complete_block<DTYPE, 4, ROT>(g, c, bh, t0 >> 7, t0, in, st, scratch, tid);
          else kchan_complete_block<DTYPE, 8, ROT>(g, c, bh, t0 >> 7, t0, in, st, scratch, tid);
        }
        kchan_tail_rows<DTYPE, ROT>(c, bh, end >> 7, t0, end, in, st, tid);       // (no rows when the append ends with the block)
      }
    }
    if (R) {
      // tokens that stay in the residual window; its older rows have been read by this CTA above
      __syncthreads();
      const int first = max(t0, qb), vpr = D / 8, nw = (end - first) * 2 * vpr;
      for (int idx = tid; idx < nh * nw; idx += blockDim.x) {
        const int h = rank + ranks * (idx / nw), r = idx % nw, t = first + r / (2 * vpr), side = (r / vpr) & 1, v = r % vpr;
        const uint16_t* src = (side ? v_new : k_new) + (int64_t)b * sb + (int64_t)h * sh + (int64_t)(t - t0) * st + 8 * v;
        *reinterpret_cast<uint4*>(c.kv_win + ((((size_t)b * g.Hkv + h) * R + t % R) * 2 + side) * D + 8 * v) =
            *reinterpret_cast<const uint4*>(src);
      }
    }
  }
  cluster_barrier();                                     // every CTA of the sequence has read its length
  if (rank == 0 && tid == 0) {
    if (fits) c.seq_len[b] = t0 + t_new;
    else atomicOr(c.status, KVQ_STATUS_CAPACITY);
  }
}

}  // namespace

// A sequence has at most eight CTAs, so the time goes with the rows of one of them: its KV heads x new tokens.  Up to 120 CTAs (fifteen
// sequences of eight heads) every cluster finds SMs of its own; beyond, two clusters share them and a row costs more.
inline bool own_sms(const Geom& g) {
  const int per_cta = heads_per_cta(g.Hkv);
  return (long long)g.B * ((g.Hkv + per_cta - 1) / per_cta) <= 120;
}

// Both sides measured as a layer's append and decode behind 1,000 tokens, replayed graph, us of four layers, this launch / tasks + lengths
// (K4V2; in eager steps the second costs another 3 to 5 us):
//    8 KV heads, head_dim 128:   48 tokens: 8 sequences 62.5 / 68.7, 14 72.5 / 81.4, 15 74.5 / 84.2;   64 tokens: 65.1 / 68.4, 75.4 / 81.6, 77.6 / 84.2
//                                40 tokens: 16 sequences 80.0 / 78.9, 18 87.3 / 87.5, 20 83.1 / 83.5, 28 90.0 / 90.4;   56 tokens: 88.0 / 82.6, 95.9 / 91.8
//    8 KV heads, head_dim 64:    128 tokens: 8 sequences 61.9 / 66.6, 15 70.4 / 76.7;   80 tokens: 16 73.3 / 72.0, 18 78.4 / 78.1, 24 81.9 / 81.9
//    8 KV heads, rotated:        48 tokens: 14 sequences 80.3 / 91.0, 15 83.3 / 95.5;   40 tokens: 16 92.6 / 93.9, 20 96.0 / 99.1;   64 tokens: 16 107 / 95
//    8 KV heads, window of 64:   48 tokens: 14 sequences 66.7 / 85.0, 16 72.6 / 91.3;   64 tokens, a block for sure: 8 76.6 / 89.3, 16 107 / 107, 32 141 / 149
//   10 channel-wise heads:       24 tokens: 8 sequences 75.7 / 82.3, 16 94.3 / 101;   36 tokens: 85.2 / 84.3, 104 / 104;   48 tokens: 90.2 / 85.5, 108 / 104
// (a layer of 16 heads: 20 tokens, 16 sequences 23.2 / 23.3, 32 30.9 / 33.9; 32 tokens, 15 sequences 22.5 / 23.6, 16 25.9 / 23.5; with a window 32
// tokens, 8 sequences 18.5 / 21.5, 16 26.3 / 27.9.)  So 64 rows a CTA at head_dim 128 and 128 at head_dim 64 while clusters have their own SMs
// or with a residual window, else 40 and 80.  Rotated keys cost more a row: 40 rows beyond eight heads (one call of sixteen in a row: 16 heads
// rotated, 20 tokens 6.4 / 6.7, 32 tokens 8.3 / 8.5).  Channel-wise keys also pay for a block a head: 36 tokens at ten heads.
// An append of at most 64 tokens of channel-wise keys completes at most one block.
bool append_rows_serves(const Geom& g, bool rotated, int t_new) {
  auto width = [](int b) { return b == 2 || b == 4 || b == 8; };
  if (t_new > 64 * 128 / g.D || !width(g.kb) || !width(g.vb)) return false;
  const long long heads = heads_per_cta(g.Hkv);
  if (g.k_axis == 1) return g.D == 128 && g.kb != 2 && heads * (t_new + 12) <= 96;
  const int limit = g.R ? 64 : !own_sms(g) || (heads > 1 && rotated) ? 40 : 64;
  return heads * t_new * g.D <= limit * 128;
}

int launch_append_rows(const Geom& g, const CachePtrs& c, const void* k_new, const void* v_new, int64_t sb, int64_t sh,
                       int64_t st, int t_new, cudaStream_t stream) {
  const int per_cta = heads_per_cta(g.Hkv), ranks = (g.Hkv + per_cta - 1) / per_cta;        // at most 8 CTAs, evenly loaded
  const bool chan = g.k_axis == 1, rot = c.k_signs != nullptr;
  int threads = per_cta * 2 * (t_new + g.R) * (g.D / 8);
  // 1,024 threads where every cluster finds SMs of its own (64 tokens as above, 512 / 1,024 threads: 8 sequences 67.1 / 65.1, 12 76.6 / 74.5, 15
  // 79.6 / 77.6; 16 sequences, whose CTAs then no longer share SMs, 90.9 / 97.1), and no window (a block's rows only when one is completed)
  const int most = g.R || !own_sms(g) ? kMaxThreads / 2 : kMaxThreads;
  threads = chan ? kChanThreads : threads > most ? most : (threads + 31) / 32 * 32;
  const uint16_t* k = static_cast<const uint16_t*>(k_new);
  const uint16_t* v = static_cast<const uint16_t*>(v_new);
  cudaError_t e;
#define KVQ_ROWS(D_, T_, C_)                                                                                             \
  launch_dependent(rot ? append_rows_kernel<D_, T_, true, C_> : append_rows_kernel<D_, T_, false, C_>, dim3(ranks, g.B), \
                   threads, 0, stream, ranks, g, c, k, v, sb, sh, st, t_new)
  const bool bf = g.in_dtype == KVQ_BF16;
  if (chan) e = bf ? KVQ_ROWS(128, KVQ_BF16, true) : KVQ_ROWS(128, KVQ_FP16, true);
  else if (g.D == 128) e = bf ? KVQ_ROWS(128, KVQ_BF16, false) : KVQ_ROWS(128, KVQ_FP16, false);
  else e = bf ? KVQ_ROWS(64, KVQ_BF16, false) : KVQ_ROWS(64, KVQ_FP16, false);
#undef KVQ_ROWS
  return e == cudaSuccess ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
}

}  // namespace kvq
