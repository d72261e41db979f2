// kvq_quantize_append kernels: group-wise asymmetric round-to-nearest
// quantization (App. B.1 quantizer per group; Sec. 4.1 grouping: token-wise
// groups along head_dim, or channel-wise groups over a 128-token block with an
// fp16 residual tail) and packing into the page layout.
//
// Token-wise kernel: a warp takes passes of two or four tokens a lane over blocks of 32 tokens (64 for head_dim 64 at 2
// bits) of one stream and one side (keys or values).  A byte of the packed page holds codes of channels that
// lie 16 apart, so a lane loads, for each of its tokens, the 8/b 16-byte pieces whose codes share
// bytes: every output byte, and with four tokens (values) or four channels (keys) every output
// word, is then assembled in that lane's registers and stored directly - codes need no shared memory, no
// atomics, no read-modify-write; a token that is not new is simply not stored (byte stores for
// values).  Group minima and maxima are reduced with a few shuffles between the lanes of a row.
// Long calls are bound by the memory system and the length of a warp's chain, short ones by fetching instructions.
#include <algorithm>

#include "kvq_quantize.cuh"

namespace kvq {

namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;

// Where the 16-bit row of a task-local token comes from: the call's input, or - for the first n_win tokens of a task
// when a residual window is kept - the window's ring of rows (token t in slot t % R; a task never wraps the ring).
struct RowSrc {
  const uint16_t* in;     // row of task-local token 0 in the input (never dereferenced before the first new token)
  int64_t st;             // input row stride in elements
  const uint16_t* win;    // window row of task-local token 0 (this side), or nullptr
  int n_win;              // task-local tokens [0, n_win) are read from the window
  int wst;                // window row stride in elements (2 D: key row, value row)
  __device__ __forceinline__ const uint16_t* row(int tau) const {
    return (tau < n_win) ? win + (size_t)tau * wst : in + (int64_t)tau * st;
  }
};

// Tokens handled by one warp task: 32, or 64 where 32 tokens would leave a lane fewer than the four tokens
// that make up a word of value codes.
__host__ __device__ constexpr int task_tokens(int D, int bits) { return (D == 64 && bits == 2) ? 64 : 32; }

// Value e (0..7) of a 16-byte piece in fp32.
template <int DTYPE>
__device__ __forceinline__ float piece_value(const uint4& r, int e) {
  const uint32_t w = e < 2 ? r.x : e < 4 ? r.y : e < 6 ? r.z : r.w;
  if constexpr (DTYPE == KVQ_BF16) return __uint_as_float((e & 1) ? (w & 0xFFFF0000u) : (w << 16));
  else { const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w)); return (e & 1) ? f.y : f.x; }
}

// Task-local token of token slot k: of the four of a value word (slots 4 i .. 4 i + 3), or of a key row.
template <bool IS_V, int RS>
__device__ __forceinline__ int token_slot(int k, int rs) {
  if constexpr (IS_V) {
    const int cmb = (k >> 2) * RS + rs, j = k & 3;         // cmb = (block, half, t) of the word; j = byte
    return 32 * (cmb >> 3) + 16 * ((cmb >> 2) & 1) + 2 * (cmb & 3) + (j >> 1) + 8 * (j & 1);
  } else {
    return k * RS + rs;
  }
}

// Tokens of a lane per pass: four make up a word of value codes.  Keys at 2 bits, whose pieces of four tokens would take 64 registers
// beside those of the arithmetic, go by two and in passes of 4 KB, as most sides do: four layers of 40 streams x 3,000 tokens K2V4 92 us by
// four, 87.5 by two; two of 64 x 4,000 81.7 and 78.8.
__host__ __device__ constexpr int pass_tokens(int bits, bool is_v) { return bits == 2 && !is_v ? 2 : 4; }

// One pass over pass_tokens tokens of every lane, one side of a task of TT tokens; tokens [lo, hi) of the task are new.  load(kk, f): the
// lane's piece f of its token kk.  next is called when the pieces have been read.  codes: keys - the page's key row of the task's first
// token; values - the page's value block of the task's first token.  meta_out: metadata row of the task's first token.
//
// Lane = (row slot rs, word column mw, row half rh): it owns, for each of its tokens, the FPB pieces of 8 channels
// 16 (FPB mw + f) + 8 rh + {0..7}, f < FPB, whose codes share bytes.  The minima / maxima of its tokens are reduced
// with a shuffle reduce-scatter, so that the group parameters (two divisions) are computed once per group rather than once
// per lane, and are then broadcast to the lanes of the group.  Minimum and negated maximum travel as one pair of the 16-bit type.
// PLAIN: if all groups of the warp are plain (see plain_group; all but those with values beyond the fp16 range or scales and minima
// below its normal numbers are), codes need no clamp and two values share every operation: 8.7 instructions per element instead of
// 10.6; else nothing is stored and the answer is false.  A value word's two ways of leaving, whole or byte by byte, are one branch behind
// all eight words (a branch per word: 8 streams x 500 tokens K4V2 11.8 us against 8.7).
template <int BITS, bool IS_V, int D, int DTYPE, bool PLAIN, typename Load, typename Next>
__device__ __forceinline__ bool quantize_pass(Load&& load, Next&& next, int gsz, int lo, int hi, uint8_t* __restrict__ codes,
                                              uint32_t* __restrict__ meta_out, int lane, int pass) {
  using H2 = typename Pair16<DTYPE>::type;
  constexpr int FPB = 8 / BITS, TK = pass_tokens(BITS, IS_V);
  constexpr int NMW = (D / 16) / FPB;        // word columns per row half
  constexpr int LR = 2 * NMW;                // lanes per token row
  constexpr int RS = 32 / LR;                // token rows per load instruction
  constexpr int K_ROW_BYTES = D * BITS / 8;
  constexpr int NSET = FPB == 4 ? 2 : 1;      // a lane's fields may belong to two groups (groups of 32 at 2 bits)
  constexpr float DOWN = 1.0f / (float)(1 << BITS);
  const int rs = lane / LR, cs = lane % LR, mw = cs >> 1, rh = cs & 1;
  const float qmax = (float)((1 << BITS) - 1);
  const int spg = gsz >> 4;                                  // 16-channel slices per group
  const bool split = FPB > spg;
  const int lpg = split ? 2 : 2 * spg / FPB;                 // lanes per group: 2, 4, 8 or 16
  const int ng = D / gsz;
  const int b0 = cs & 1, b1 = (cs >> 1) & 1;
  const int gbase = lane & ~(lpg - 1);                       // first lane of this lane's group

  auto token_of = [&](int k) { return token_slot<IS_V, RS>(k, rs); };
  auto swap = [](H2 x, int off) {
    const uint32_t o = __shfl_xor_sync(FULL, *reinterpret_cast<uint32_t*>(&x), off);
    return *reinterpret_cast<const H2*>(&o);
  };

  uint4 raw[TK][FPB];
  bool valid[TK];
#pragma unroll
  for (int kk = 0; kk < TK; ++kk) {
    const int tau = token_of(TK * pass + kk);
    valid[kk] = tau >= lo && tau < hi;
#pragma unroll
    for (int f = 0; f < FPB; ++f) raw[kk][f] = load(kk, f);
  }
  // ---- minima / maxima of the lane's fields, per token and per set
  H2 m[NSET][TK];
#pragma unroll
  for (int kk = 0; kk < TK; ++kk) {
    m[0][kk] = minmax8<DTYPE, PLAIN>(raw[kk][0]);
    if constexpr (FPB == 2) m[0][kk] = min_pair(m[0][kk], minmax8<DTYPE, PLAIN>(raw[kk][1]), PLAIN);
    if constexpr (FPB == 4) {
      m[0][kk] = min_pair(m[0][kk], minmax8<DTYPE, PLAIN>(raw[kk][1]), PLAIN);
      m[1][kk] = min_pair(minmax8<DTYPE, PLAIN>(raw[kk][2]), minmax8<DTYPE, PLAIN>(raw[kk][3]), PLAIN);
      if (!split) m[0][kk] = min_pair(m[0][kk], m[1][kk], PLAIN);
    }
  }
  // ---- reduce-scatter over the lanes of the group: after lane bit 0 a lane holds tokens 2 b0 + {0, 1}, after
  // bit 1 (groups of 4 lanes or more) token 2 b0 + b1; of two tokens it holds token b0; higher bits are plain butterflies
  float pz[NSET][2], pinv[NSET][2];
  uint32_t pmeta[NSET][2];
  bool plain = true;
#pragma unroll
  for (int e = 0; e < NSET; ++e) {
    if (e == 1 && !split) break;
    H2 a0, a1;
    if constexpr (TK == 4) {
      a0 = min_pair(b0 ? m[e][2] : m[e][0], swap(b0 ? m[e][0] : m[e][2], 1), PLAIN);
      a1 = min_pair(b0 ? m[e][3] : m[e][1], swap(b0 ? m[e][1] : m[e][3], 1), PLAIN);
      if (lpg >= 4) a0 = min_pair(b1 ? a1 : a0, swap(b1 ? a0 : a1, 2), PLAIN);
    } else {
      a0 = a1 = min_pair(b0 ? m[e][1] : m[e][0], swap(b0 ? m[e][0] : m[e][1], 1), PLAIN);
      if (lpg >= 4) a0 = min_pair(a0, swap(a0, 2), PLAIN);
    }
    if (lpg >= 8) a0 = min_pair(a0, swap(a0, 4), PLAIN);
    if (lpg >= 16) a0 = min_pair(a0, swap(a0, 8), PLAIN);
    const float2 f0 = pair_to_f32(a0);
    const GroupParams p0 = group_params(f0.x, -f0.y, qmax);
    if constexpr (PLAIN) plain &= plain_group(f0.x, -f0.y, p0, qmax);
    pz[e][0] = p0.z; pinv[e][0] = p0.inv * DOWN; pmeta[e][0] = p0.meta;
    pz[e][1] = 0.f; pinv[e][1] = 0.f; pmeta[e][1] = 0u;
    if (TK == 4 && lpg == 2) {
      const float2 f1 = pair_to_f32(a1);
      const GroupParams p1 = group_params(f1.x, -f1.y, qmax);
      if constexpr (PLAIN) plain &= plain_group(f1.x, -f1.y, p1, qmax);
      pz[e][1] = p1.z; pinv[e][1] = p1.inv * DOWN; pmeta[e][1] = p1.meta;
    }
  }
  next();                                   // (the shuffles above have seen all of `raw`: its place may be filled again)
  if constexpr (PLAIN) {
    if (!__all_sync(FULL, plain)) return false;
  }
  // the lane (one per group) that holds a token's parameters stores its metadata word
  if ((cs & (lpg - 1) & -TK) == 0) {
#pragma unroll
    for (int e = 0; e < NSET; ++e) {
      if (e == 1 && !split) break;
      const int gi = (16 * FPB * mw) / gsz + e;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (i == 1 && (TK == 2 || lpg != 2)) break;
        const int kk = TK == 2 ? b0 : 2 * b0 + (lpg >= 4 ? b1 : i);
        const int tau = token_of(TK * pass + kk);
        if (tau >= lo && tau < hi) meta_out[tau * ng + gi] = pmeta[e][i];
      }
    }
  }
  // ---- the group's parameters, fetched from the lane that made them
  float z[NSET][TK], inv[NSET][TK];
#pragma unroll
  for (int kk = 0; kk < TK; ++kk) {
    const int srcl = gbase + (TK == 2 ? kk : lpg >= 4 ? (kk >> 1) + 2 * (kk & 1) : (kk >> 1));
    const int el = TK == 2 || lpg >= 4 ? 0 : kk & 1;
    z[0][kk] = __shfl_sync(FULL, el ? pz[0][1] : pz[0][0], srcl);
    inv[0][kk] = __shfl_sync(FULL, el ? pinv[0][1] : pinv[0][0], srcl);
    if constexpr (NSET == 2) {
      z[1][kk] = z[0][kk]; inv[1][kk] = inv[0][kk];
      if (split) {
        z[1][kk] = __shfl_sync(FULL, el ? pz[1][1] : pz[1][0], srcl);
        inv[1][kk] = __shfl_sync(FULL, el ? pinv[1][1] : pinv[1][0], srcl);
      }
    }
  }
  if constexpr (!IS_V) {
    // ---- keys: the four bytes of a word are channels 4 hh + {0..3} of this lane's 8, chunk 2 rh + hh, word mw of the row
    constexpr int wpc = D * BITS / 128;
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      const int tau = token_of(TK * pass + kk);
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        uint32_t w = 0;
#pragma unroll
        for (int f = FPB - 1; f >= 0; --f) {
          const int e = NSET == 2 ? f >> 1 : 0;
          float x[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = piece_value<DTYPE>(raw[kk][f], 4 * hh + j);
          if constexpr (PLAIN) {
            const f32x2 nz = pack2(-z[e][kk], -z[e][kk]), ii = pack2(inv[e][kk], inv[e][kk]);
            w = w * (1u << BITS) + code_word4_plain<BITS>(pack2(x[0], x[1]), pack2(x[2], x[3]), nz, nz, ii, ii);
          } else {
            const float zz[4] = {z[e][kk], z[e][kk], z[e][kk], z[e][kk]}, ii[4] = {inv[e][kk], inv[e][kk], inv[e][kk], inv[e][kk]};
            w = w * (1u << BITS) + code_word4<BITS>(x, zz, ii);
          }
        }
        if (valid[kk])
          *reinterpret_cast<uint32_t*>(codes + (size_t)tau * K_ROW_BYTES + chunk_word_byte(2 * rh + hh, mw, wpc, 4)) = w;
      }
    }
  } else {
    // ---- values: the four bytes of a word are this lane's four tokens; word of channel slot i at lane chunk 4 i + t
    const int cmb = pass * RS + rs;
    uint8_t* wbase = codes + (size_t)(cmb >> 3) * (4 * D * BITS) + mw * 512 + (cmb & 3) * 16 +
                     4 * (2 * rh + ((cmb >> 2) & 1));
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      w[i] = 0;
#pragma unroll
      for (int f = FPB - 1; f >= 0; --f) {
        const int e = NSET == 2 ? f >> 1 : 0;
        float x[4];
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) x[kk] = piece_value<DTYPE>(raw[kk][f], i);
        if constexpr (PLAIN)
          w[i] = w[i] * (1u << BITS) + code_word4_plain<BITS>(pack2(x[0], x[1]), pack2(x[2], x[3]), pack2(-z[e][0], -z[e][1]), pack2(-z[e][2], -z[e][3]),
                                                        pack2(inv[e][0], inv[e][1]), pack2(inv[e][2], inv[e][3]));
        else
          w[i] = w[i] * (1u << BITS) + code_word4<BITS>(x, z[e], inv[e]);
      }
    }
    if (valid[0] && valid[1] && valid[2] && valid[3]) {
#pragma unroll
      for (int i = 0; i < 8; ++i) *reinterpret_cast<uint32_t*>(wbase + 64 * i) = w[i];
    } else {
#pragma unroll
      for (int kk = 0; kk < TK; ++kk) {
        if (valid[kk]) {
#pragma unroll
          for (int i = 0; i < 8; ++i) wbase[64 * i + kk] = (uint8_t)(w[i] >> (8 * kk));
        }
      }
    }
  }
  return true;
}

// The same with clamped codes, out of line: few passes need it.
template <int BITS, bool IS_V, int D, int DTYPE>
__device__ __noinline__ void quantize_pass_clamped(RowSrc rsrc, int gsz, int lo, int hi, uint8_t* __restrict__ codes,
                                                   uint32_t* __restrict__ meta_out, int lane, int pass) {
  constexpr int FPB = 8 / BITS, LR = 2 * (D / 16) / FPB, RS = 32 / LR;
  const int rs = lane / LR, cs = lane % LR;
  auto load = [&](int kk, int f) {
    const int tau = token_slot<IS_V, RS>(pass_tokens(BITS, IS_V) * pass + kk, rs);
    return *reinterpret_cast<const uint4*>(rsrc.row(min(max(tau, lo), hi - 1)) + 16 * (FPB * (cs >> 1) + f) + 8 * (cs & 1));
  };
  quantize_pass<BITS, IS_V, D, DTYPE, false>(load, [] {}, gsz, lo, hi, codes, meta_out, lane, pass);
}

// The rows of a long append are read once: they leave the L2 first, as with a streaming load, and what else is there stays (the rows that
// a residual window takes behind the same call, the pages just written, other tensors).  Four layers of 32 streams x 2,000 tokens K4V2,
// default / evict-first: with a window of 128 118 / 96 us, without one 57 / 55; one of 64 x 8,000 70 / 68.5, 64 x 16,000 132 / 132.  A call of
// more than four times the L2 has nothing there to keep, and the hint costs it: 64 x 32,767 255 / 259.  (policy: 0 = no hint.)
__device__ __forceinline__ uint64_t read_once_policy(int t_new, int D) {
  if ((long long)gridDim.y * t_new * D * 4 > (512ll << 20)) return 0;
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  return policy;
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint64_t policy) {
  if (policy != 0)
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(policy) : "memory");
  else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// The passes of one side of a stream that fall to a warp: first, first + step, ... of all passes over the 32- or 64-token blocks that
// hold tokens [qa, qb).  slot: 16 bytes per lane and piece of a pass in shared memory.  Every lane copies the pieces that it will read
// itself and needs no barrier; those of the next pass are on their way while this one is quantized.  K and V of 64 streams x 32,767
// tokens (K4V2, 1.29 GB), loads into registers and clamped codes before / now: 262 / 252 us on one GPU, 250 / 243 on another (four CTAs
// per SM; three 248, five 248; two passes ahead at three CTAs per SM 256; pieces read twice instead of held, for more warps: 252 to 325).
// The same loads and stores without the arithmetic between them take 220 us; one grid that goes through all streams pass by pass 299.
template <int BITS, bool IS_V, int D, int DTYPE>
__device__ __forceinline__ void quantize_passes(const Geom& g, const CachePtrs& c, const uint16_t* __restrict__ in, int64_t st, int bh, int t0, int qa,
                                                int qb, int t_new, int first, int step, uint4* slot, int lane) {
  constexpr int FPB = 8 / BITS, LR = 2 * (D / 16) / FPB, RS = 32 / LR, TT = task_tokens(D, BITS);
  constexpr int TK = pass_tokens(BITS, IS_V), NP = TT / RS / TK;
  static_assert(TT % (TK * RS) == 0, "a lane's tokens of a task make up whole passes");
  const int rs = lane / LR, cs = lane % LR;
  const int gsz = IS_V ? g.gv : g.gk, R = g.R;
  const int first_task = qa / TT, n = ((qb + TT - 1) / TT - first_task) * NP;
  const uint16_t* win = R ? c.kv_win + (size_t)bh * R * (2 * D) + (IS_V ? D : 0) : nullptr;
  in += 16 * FPB * (cs >> 1) + 8 * (cs & 1) - (int64_t)t0 * st;
  slot += lane;
  const uint32_t slot_s = (uint32_t)__cvta_generic_to_shared(slot);
  const uint64_t policy = read_once_policy(t_new, D);
  auto issue = [&](int u) {
    const int tk0 = (first_task + u / NP) * TT;
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      const int t = min(max(tk0 + token_slot<IS_V, RS>(TK * (u % NP) + kk, rs), qa), qb - 1);     // (tokens that are not new: any that is)
      const uint16_t* p = in + (int64_t)t * st;
      if (R && t < t0) p = win + (size_t)(t % R) * (2 * D) + 16 * FPB * (cs >> 1) + 8 * (cs & 1);
#pragma unroll
      for (int f = 0; f < FPB; ++f) cp_async16(slot_s + 512 * (kk * FPB + f), p + 16 * f, policy);
    }
  };
  auto load = [&](int kk, int f) { return slot[32 * (kk * FPB + f)]; };
  if (first < n) issue(first);
#pragma unroll 1
  for (int u = first; u < n; u += step) {
    const int tk0 = (first_task + u / NP) * TT, tp0 = tk0 & 127;
    const int lo = max(qa, tk0) - tk0, hi = min(qb, tk0 + TT) - tk0;
    uint8_t* pg = c.pages + ((size_t)bh * g.n_pages + (tk0 >> 7)) * g.page_bytes;
    uint8_t* codes = IS_V ? pg + g.v_codes_off + (size_t)(tp0 >> 5) * (4 * D * BITS) : pg + tp0 * (D * BITS / 8);
    uint32_t* meta = reinterpret_cast<uint32_t*>(pg + (IS_V ? g.v_meta_off : g.k_meta_off)) + tp0 * (D / gsz);
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!quantize_pass<BITS, IS_V, D, DTYPE, true>(load, [&] { if (u + step < n) issue(u + step); }, gsz, lo, hi, codes, meta, lane, u % NP)) {
      RowSrc rsrc;
      rsrc.in = in - (16 * FPB * (cs >> 1) + 8 * (cs & 1)) + (int64_t)tk0 * st;
      rsrc.st = st;
      rsrc.n_win = R ? max(0, min(TT, t0 - tk0)) : 0;
      rsrc.wst = 2 * D;
      rsrc.win = R ? win + (size_t)(tk0 % R) * (2 * D) : nullptr;
      quantize_pass_clamped<BITS, IS_V, D, DTYPE>(rsrc, gsz, lo, hi, codes, meta, lane, u % NP);
    }
  }
}

// Rotated keys (y = H (signs * x) / sqrt(D), then token-wise groups): tokens [lo, hi) of a task, one token of a lane at a time with
// the next one's loads in flight (bound by fetching instructions beside the value side's code; two tokens at a time were slower, 32
// streams x 2,047 tokens 24.8 us against 24; with the signs converted for every token and lanes' own divisions 36 us).  The transform and
// the codes take two neighbouring channels per operation: four such chunks 90.9 -> 86.2 us.
// Lanes and fields as in quantize_pass; butterfly stages in the order h = 1, 2, 4, ...: bits of i in the lane, rh across
// lanes, bits of f in the lane, bits of mw across lanes.
template <int BITS, int D, int DTYPE>
__device__ __forceinline__ void quantize_task_rotated(const RowSrc& rsrc, int gsz, int lo, int hi, uint8_t* __restrict__ codes,
                                                      uint32_t* __restrict__ meta_out, int lane, const int8_t* __restrict__ signs) {
  constexpr int FPB = 8 / BITS, NMW = (D / 16) / FPB, LR = 2 * NMW, RS = 32 / LR;
  constexpr int K_ROW_BYTES = D * BITS / 8, NSET = FPB == 4 ? 2 : 1, wpc = D * BITS / 128;
  constexpr float DOWN = 1.0f / (float)(1 << BITS);
  const int rs = lane / LR, cs = lane % LR, mw = cs >> 1, rh = cs & 1;
  const float qmax = (float)((1 << BITS) - 1);
  const int spg = gsz >> 4, lpg = FPB > spg ? 2 : 2 * spg / FPB, ng = D / gsz;
  const bool split = FPB > spg;
  float sg[FPB][8];
#pragma unroll
  for (int f = 0; f < FPB; ++f) {
#pragma unroll
    for (int i = 0; i < 8; ++i) sg[f][i] = (float)signs[16 * (FPB * mw + f) + 8 * rh + i];
  }
  const float srh = rh ? -1.0f : 1.0f;             // a butterfly between lanes: o + s x (the product with +-1 is exact)
  uint4 next[FPB];
  auto fetch = [&](int tau) {
#pragma unroll
    for (int f = 0; f < FPB; ++f) {
      next[f] = make_uint4(0u, 0u, 0u, 0u);
      if (tau < hi) next[f] = __ldcs(reinterpret_cast<const uint4*>(rsrc.row(tau) + 16 * (FPB * mw + f) + 8 * rh));
    }
  };
  fetch(lo + rs);
#pragma unroll 1
  for (int base = lo; base < hi; base += RS) {
    const int tau = base + rs;
    // (two neighbouring channels share an operation; differences as sums with a product by -1, which is exact)
    const f32x2 minus = pack2(-1.0f, -1.0f);
    f32x2 y[FPB][4];
#pragma unroll
    for (int f = 0; f < FPB; ++f) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        y[f][i] = mul2(pack2(piece_value<DTYPE>(next[f], 2 * i), piece_value<DTYPE>(next[f], 2 * i + 1)), pack2(sg[f][2 * i], sg[f][2 * i + 1]));
    }
    fetch(tau + RS);
#pragma unroll
    for (int f = 0; f < FPB; ++f) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 a = unpack2(y[f][i]);
        y[f][i] = pack2(__fadd_rn(a.x, a.y), __fsub_rn(a.x, a.y));
      }
#pragma unroll
      for (int h = 1; h < 4; h <<= 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if ((i & h) == 0) {
            const f32x2 a = y[f][i], c = y[f][i + h];
            y[f][i] = add2(a, c);
            y[f][i + h] = fma2(c, minus, a);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float2 o = unpack2(y[f][i]);
        o.x = __shfl_xor_sync(FULL, o.x, 1); o.y = __shfl_xor_sync(FULL, o.y, 1);
        y[f][i] = fma2(pack2(srh, srh), y[f][i], pack2(o.x, o.y));
      }
    }
#pragma unroll
    for (int hf = 1; hf < FPB; hf <<= 1) {
#pragma unroll
      for (int f = 0; f < FPB; ++f) {
        if ((f & hf) == 0) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const f32x2 a = y[f][i], c = y[f + hf][i];
            y[f][i] = add2(a, c);
            y[f + hf][i] = fma2(c, minus, a);
          }
        }
      }
    }
#pragma unroll
    for (int hm = 1; hm < NMW; hm <<= 1) {
      const float sm = (mw & hm) ? -1.0f : 1.0f;
#pragma unroll
      for (int f = 0; f < FPB; ++f) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float2 o = unpack2(y[f][i]);
          o.x = __shfl_xor_sync(FULL, o.x, 2 * hm); o.y = __shfl_xor_sync(FULL, o.y, 2 * hm);
          y[f][i] = fma2(pack2(sm, sm), y[f][i], pack2(o.x, o.y));
        }
      }
    }
    float x[FPB][8];
#pragma unroll
    for (int f = 0; f < FPB; ++f) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 a = unpack2(mul2(y[f][i], pack2(inv_sqrt_dim<D>(), inv_sqrt_dim<D>())));
        x[f][2 * i] = a.x; x[f][2 * i + 1] = a.y;
      }
    }
    // (from the first value on, as everywhere: a row of NaN has the same parameters in every kernel)
    float mn[NSET], mx[NSET];
#pragma unroll
    for (int f = 0; f < FPB; ++f) {
      const int e = NSET == 2 ? f >> 1 : 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const bool first = i == 0 && f == (FPB / NSET) * e;
        mn[e] = first ? x[f][i] : fminf(mn[e], x[f][i]);
        mx[e] = first ? x[f][i] : fmaxf(mx[e], x[f][i]);
      }
    }
    if constexpr (NSET == 2) {
      if (!split) {
        mn[0] = mn[1] = fminf(mn[0], mn[1]);
        mx[0] = mx[1] = fmaxf(mx[0], mx[1]);
      }
    }
    float z[NSET], inv[NSET];
#pragma unroll
    for (int e = 0; e < NSET; ++e) {
#pragma unroll
      for (int off = 1; off < LR; off <<= 1) {
        const float oa = __shfl_xor_sync(FULL, mn[e], off), oc = __shfl_xor_sync(FULL, mx[e], off);
        if (off < lpg) { mn[e] = fminf(mn[e], oa); mx[e] = fmaxf(mx[e], oc); }
      }
      const GroupParams p = group_params(mn[e], mx[e], qmax);
      z[e] = p.z;
      inv[e] = p.inv * DOWN;
      if (tau < hi && (cs & (lpg - 1)) == 0 && (e == 0 || split)) meta_out[tau * ng + (16 * FPB * mw) / gsz + e] = p.meta;
    }
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      uint32_t w = 0;
#pragma unroll
      for (int f = FPB - 1; f >= 0; --f) {
        const int e = NSET == 2 ? f >> 1 : 0;
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = x[f][4 * hh + j];
        w = w * (1u << BITS) + code_word4_packed<BITS>(v, z[e], inv[e]);
      }
      if (tau < hi)
        *reinterpret_cast<uint32_t*>(codes + (size_t)tau * K_ROW_BYTES + chunk_word_byte(2 * rh + hh, mw, wpc, 4)) = w;
    }
  }
}

// Bit-plane widths (1, 3, 6 bits): a plain variant, one token row per warp step.  A lane holds 8 consecutive
// channels of a row, groups reduce by butterflies, and every code's plane fields are cleared and set with atomic
// AND / OR on the 32-bit words of the page (several lanes share a word).  Not tuned: these widths are served for
// the paper's 1-, 3- and 6-bit settings, the 2/4/8-bit path above is the fast one.
template <int D, int DTYPE>
__device__ __forceinline__ void quantize_task_planes(const RowSrc& rsrc, int gsz, int bits,
                                                     bool is_v, int lo, int hi, int tp0, uint8_t* __restrict__ region,
                                                     uint32_t* __restrict__ meta_out, int lane) {
  constexpr int LPR = D / 8, RPW = 32 / LPR;           // lanes per row, rows per warp step
  const int l = lane % LPR, r0 = lane / LPR;
  const int lpg = gsz >> 3, ng = D / gsz;
  const float qmax = (float)((1 << bits) - 1);
  for (int base = lo; base < hi; base += RPW) {
    const int tau = base + r0;                         // task-local token
    const bool valid = tau < hi;
    uint4 raw = make_uint4(0u, 0u, 0u, 0u);
    if (valid) raw = *reinterpret_cast<const uint4*>(rsrc.row(tau) + 8 * l);
    const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
    float x[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[2 * i] = bits16_to_f32((uint16_t)(rw[i] & 0xFFFF), DTYPE);
      x[2 * i + 1] = bits16_to_f32((uint16_t)(rw[i] >> 16), DTYPE);
    }
    float mn = x[0], mx = x[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) { mn = fminf(mn, x[i]); mx = fmaxf(mx, x[i]); }
#pragma unroll
    for (int off = 1; off < 16; off <<= 1) {
      if (off < lpg) {
        mn = fminf(mn, __shfl_xor_sync(FULL, mn, off));
        mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, off));
      }
    }
    const GroupParams p = group_params(mn, mx, qmax);
    if (!valid) continue;
    const int t = tp0 + tau;                           // page-local token
    if ((l & (lpg - 1)) == 0) meta_out[tau * ng + (8 * l) / gsz] = p.meta;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t code = code_of(x[i], p, qmax);
      int hb, lb;
      planes_of(bits, hb, lb);
#pragma unroll
      for (int plane = 0; plane < 2; ++plane) {
        if (plane == 1 && lb == 0) break;
        int wb, bit, pb;
        plane_pos(is_v, t, 8 * l + i, D, bits, plane, wb, bit, pb);
        const uint32_t field = (plane == 0 ? (code >> lb) : code) & ((1u << pb) - 1u);
        uint32_t* w = reinterpret_cast<uint32_t*>(region + wb);
        atomicAnd(w, ~(((1u << pb) - 1u) << bit));
        atomicOr(w, field << bit);
      }
    }
  }
}

// 16-bit passthrough of one side of a task: rows [lo, hi) copied to the page as they are.
__device__ __forceinline__ void copy_task_side(const RowSrc& rsrc, int D, int lo, int hi,
                                               uint16_t* __restrict__ dst_rows, int lane) {
  const int lpr = D >> 3, rps = 32 / lpr, l = lane & (lpr - 1);
  for (int row = lo + lane / lpr; row < hi; row += rps)
    *reinterpret_cast<uint4*>(dst_rows + (size_t)row * D + l * 8) =
        *reinterpret_cast<const uint4*>(rsrc.row(row) + l * 8);
}

// Token-wise quantization of V and of K, a side per blockIdx.z.  grid.y = stream, grid.x strides over the passes (or, for 16-bit
// rows, bit planes and rotated keys, over the warp tasks) touched by this append.  Rotated keys take longer than the values beside them
// and come first: four chunks of 32 streams x 2,047 tokens 80 us with the values first, 75 now (87 before the passes were pipelined).
__host__ __device__ constexpr int slot_bytes(int bits, bool is_v) { return 32 * 16 * pass_tokens(bits, is_v) * (8 / bits); }        // a warp's pieces of a pass
template <int D, int DTYPE, bool ROT>
__global__ void __launch_bounds__(kThreads, D == 64 && !ROT ? 5 : 4)
quant_token_kernel(Geom g, CachePtrs c, const uint16_t* __restrict__ k_new, const uint16_t* __restrict__ v_new,
                   int64_t sb, int64_t sh, int64_t st, int t_new) {
  extern __shared__ __align__(16) uint8_t smem[];
  begin_after_predecessor();
  const bool is_v = blockIdx.z == (ROT ? 1 : 0);           // rotated keys take longer and come first
  const int bh = blockIdx.y;
  const int b = bh / g.Hkv, h = bh % g.Hkv;
  const int t0 = c.seq_len[b];
  if (!append_fits(t0, t_new, g.capacity)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bits = is_v ? g.vb : g.kb;
  // tokens to quantize: the new ones, or - with a residual window of R tokens - the blocks of R that this append
  // completes (their first tokens may come from the window, the rest from the input)
  const int R = g.R;
  const int qa = R ? (t0 / R) * R : t0, qb = R ? ((t0 + t_new) / R) * R : t0 + t_new;
  if (qb <= qa) return;
  const uint16_t* in = (is_v ? v_new : k_new) + (int64_t)b * sb + (int64_t)h * sh;
  const int gsz = is_v ? g.gv : g.gk;
  const int first = blockIdx.x * kWarps + warp, step = gridDim.x * kWarps;

  if ((bits == 2 || bits == 4 || bits == 8) && (is_v || !ROT)) {
    uint4* slot = reinterpret_cast<uint4*>(smem + warp * slot_bytes(bits, is_v));
#define KVQ_PASSES(BITS_, V_) quantize_passes<BITS_, V_, D, DTYPE>(g, c, in, st, bh, t0, qa, qb, t_new, first, step, slot, lane)
    if (is_v) {
      if (bits == 2) KVQ_PASSES(2, true);
      else if (bits == 4) KVQ_PASSES(4, true);
      else KVQ_PASSES(8, true);
    } else if constexpr (!ROT) {
      if (bits == 2) KVQ_PASSES(2, false);
      else if (bits == 4) KVQ_PASSES(4, false);
      else KVQ_PASSES(8, false);
    }
#undef KVQ_PASSES
    return;
  }
  // 16-bit rows, bit planes, rotated keys: a warp per task
  const int TT = (bits == 16 || is_plane_width(bits)) ? 32 : task_tokens(D, bits);
  const int first_task = qa / TT;
  const int n_tasks = (qb + TT - 1) / TT - first_task;
  for (int j = first; j < n_tasks; j += step) {
    const int tk0 = (first_task + j) * TT;                     // first token of the task
    const int lo = max(qa, tk0) - tk0, hi = min(qb, tk0 + TT) - tk0;
    const int page = tk0 >> 7, tp0 = tk0 & 127;                // page-local token of the task's first row
    uint8_t* pg = c.pages + ((size_t)bh * g.n_pages + page) * g.page_bytes;
    // row 0 of the task in the input (may lie before the first new token; never dereferenced there)
    RowSrc rs;
    rs.in = in + (int64_t)(tk0 - t0) * st;
    rs.st = st;
    rs.n_win = R ? max(0, min(TT, t0 - tk0)) : 0;
    rs.wst = 2 * D;
    rs.win = R ? c.kv_win + ((size_t)bh * R + (tk0 % R)) * (2 * D) + (is_v ? D : 0) : nullptr;
    uint8_t* region = pg + (is_v ? g.v_codes_off : 0);
    uint32_t* meta = reinterpret_cast<uint32_t*>(pg + (is_v ? g.v_meta_off : g.k_meta_off)) + (bits == 16 ? 0 : tp0 * (D / gsz));
    if (bits == 16) {
      copy_task_side(rs, D, lo, hi, reinterpret_cast<uint16_t*>(region) + (size_t)tp0 * D, lane);
    } else if (is_plane_width(bits)) {
      quantize_task_planes<D, DTYPE>(rs, gsz, bits, is_v, lo, hi, tp0, region, meta, lane);
    } else if constexpr (ROT) {
      uint8_t* kr = pg + (size_t)tp0 * (D * bits / 8);
      if (bits == 2) quantize_task_rotated<2, D, DTYPE>(rs, gsz, lo, hi, kr, meta, lane, c.k_signs);
      else if (bits == 4) quantize_task_rotated<4, D, DTYPE>(rs, gsz, lo, hi, kr, meta, lane, c.k_signs);
      else quantize_task_rotated<8, D, DTYPE>(rs, gsz, lo, hi, kr, meta, lane, c.k_signs);
    }
  }
}

// Pack K rows: `codes` holds bytes [ntok rows][D]; row r goes to page-local token slot0 + r.
__device__ __forceinline__ void pack_k_rows(const uint8_t* codes, int code_stride, int ntok, int slot0,
                                            uint8_t* kregion, int D, int b, int tid) {
  const int wpr = D * b / 32;    // words per row
  const int wpc = wpr / 4;       // words per chunk
  const int nf = 32 / b;
  for (int idx = tid; idx < ntok * wpr; idx += kThreads) {
    int r = idx / wpr, wi = idx % wpr;
    int chunk = wi / wpc, word = wi % wpc;
    uint32_t w = 0;
    for (int f = 0; f < nf; ++f) {
      int d = k_field_channel(chunk, word, f, b);
      w |= (uint32_t)codes[r * code_stride + d] << (f * b);
    }
    *reinterpret_cast<uint32_t*>(kregion + (size_t)(slot0 + r) * (D * b / 8) + chunk_word_byte(chunk, word, wpc, 4)) = w;
  }
}

// Channel-wise quantization of K, head_dim 128, 4- or 8-bit codes: CTA j of a stream takes every grid.x-th of the 128-token blocks that
// this append completes; CTA 0, which alone reads the tail (for the first block), also writes the rows of the block that stays
// incomplete to it.  A block stays in the registers of 256 threads; the next one is on its way to shared memory meanwhile, each
// thread's own pieces, so that no barrier is needed for them.  K and V of 120 streams x 16,383 tokens (values by the kernel above): 286 us
// with one block per CTA, converted to fp16, clamped and packed value by value (15 instructions per element, issue 68 %), 251 now (four
// CTAs per SM 250, but 171 us against 147 for rotated keys of 130 streams x 330 tokens; CTAs for 6, 12 or 24 blocks per SM at a time 255, 251, 251).
template <int DTYPE, int KB, bool ROT>
__global__ void __launch_bounds__(256, 3)
quant_kchan_fast_kernel(Geom g, CachePtrs c, const uint16_t* __restrict__ k_new, int64_t sb, int64_t sh, int64_t st, int t_new) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ KchanShared scratch;
  begin_after_predecessor();
  const int bh = blockIdx.y, b = bh / g.Hkv, h = bh % g.Hkv;
  const int t0 = c.seq_len[b];
  if (!append_fits(t0, t_new, g.capacity)) return;
  const int end = t0 + t_new, first_page = t0 >> 7, complete = (end >> 7) - first_page;      // blocks that are complete after this append
  const int tid = threadIdx.x;
  const uint16_t* in = k_new + (int64_t)b * sb + (int64_t)h * sh - (int64_t)t0 * st + (tid & 15) * 8;
  int j = blockIdx.x;
  if (j < complete && (ROT || (j == 0 && (t0 & 127) != 0))) {        // rows from the tail, or to be rotated
    kchan_complete_block<DTYPE, KB, ROT>(g, c, bh, first_page + j, t0, in, st, scratch, tid);
    j += gridDim.x;
  }
  if constexpr (ROT) {
    for (; j < complete; j += gridDim.x) kchan_complete_block<DTYPE, KB, ROT>(g, c, bh, first_page + j, t0, in, st, scratch, tid);
  } else {
    // a thread copies the pieces that it will read itself; those of the next block are on their way while this one is quantized
    uint4* slot = reinterpret_cast<uint4*>(smem) + tid;
    const uint32_t slot_s = (uint32_t)__cvta_generic_to_shared(slot);
    const uint64_t policy = read_once_policy(t_new, 128);
    auto issue = [&](int block) {
      const uint16_t* p = in + (int64_t)(((first_page + block) << 7) + (tid >> 4)) * st;
#pragma unroll
      for (int i = 0; i < 8; ++i, p += 16 * st) cp_async16(slot_s + 4096 * i, p, policy);
    };
    if (j < complete) issue(j);
#pragma unroll 1
    for (; j < complete; j += gridDim.x) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      uint4 val[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) val[i] = slot[256 * i];
      uint8_t* pg = c.pages + ((size_t)bh * g.n_pages + first_page + j) * g.page_bytes;
      if (!kchan_block_plain<DTYPE, KB>(val, scratch, pg, g, tid, [&] { if (j + (int)gridDim.x < complete) issue(j + gridDim.x); })) {
#pragma unroll
        for (int i = 0; i < 8; ++i) val[i] = key_row_fp16<DTYPE, false>(val[i], nullptr, tid & 15);
        kchan_block<KB>(val, scratch, pg, g, tid);
      }
    }
  }
  if (blockIdx.x == 0 && (end & 127) != 0) kchan_tail_rows<DTYPE, ROT>(c, bh, end >> 7, t0, end, in, st, tid);
}

// Channel-wise quantization of K over 128-token blocks with the fp16 tail, the shapes that the kernel above does not
// serve (head_dim 64, 2-bit codes).  CTA j of a stream handles the j-th block touched by this append.  CTA 0 also
// handles the final block when that one is incomplete (it writes the tail, which
// CTA 0 must have finished reading first).
__global__ void __launch_bounds__(kThreads)
quant_kchan_kernel(Geom g, CachePtrs c, const uint16_t* __restrict__ k_new,
                   int64_t sb, int64_t sh, int64_t st, int t_new) {
  extern __shared__ __align__(16) uint8_t smem[];
  begin_after_predecessor();
  const int D = g.D;
  uint16_t* sX = reinterpret_cast<uint16_t*>(smem);          // [128][D] fp16 bits
  uint8_t* sC = smem + (size_t)kPageTokens * D * 2;           // [128][D] codes
  const int bh = blockIdx.y;
  const int b = bh / g.Hkv, h = bh % g.Hkv;
  const int t0 = c.seq_len[b];
  if (!append_fits(t0, t_new, g.capacity)) return;
  const int end = t0 + t_new;
  const int first_page = t0 >> 7;
  const int nblk = ((end + 127) >> 7) - first_page;
  const bool last_partial = (end & 127) != 0;
  const int tid = threadIdx.x;
  uint16_t* tail = c.k_tail + (size_t)bh * kPageTokens * D;
  const float qmax = (float)((1 << g.kb) - 1);

  for (int pass = 0; pass < 2; ++pass) {
    int j;
    if (pass == 0) {
      j = blockIdx.x;
      if (j >= nblk) return;
      if (j == nblk - 1 && last_partial && j != 0) return;   // done by CTA 0 in its second pass
    } else {
      if (blockIdx.x != 0 || nblk <= 1 || !last_partial) return;
      j = nblk - 1;
      __syncthreads();
    }
    const int page = first_page + j;
    const int tb = page << 7;
    const int lo = max(t0, tb) - tb, hi = min(end, tb + 128) - tb;   // new tokens occupy slots [lo, hi)
    const bool complete = (hi == 128);
    // gather the block: slots [0, lo) from the tail, [lo, hi) from the input (as saturated fp16)
    // (a row is handled by D/8 consecutive lanes, which is what the rotation's shuffles expect; every lane of a
    // warp runs the loop body, rows past the end are inactive)
    const int vec_per_row = D / 8;   // 16-byte vectors
    for (int base = 0; base < hi * vec_per_row; base += kThreads) {
      const int idx = base + tid;
      const bool active = idx < hi * vec_per_row;
      const int slot = idx / vec_per_row, v = idx % vec_per_row;
      uint4 val = make_uint4(0u, 0u, 0u, 0u);
      const bool is_new = active && slot >= lo;
      if (active && !is_new) val = *reinterpret_cast<const uint4*>(tail + (size_t)slot * D + v * 8);
      if (is_new)
        val = *reinterpret_cast<const uint4*>(k_new + (int64_t)b * sb + (int64_t)h * sh +
                                              (int64_t)(tb + slot - t0) * st + v * 8);
      if (c.k_signs != nullptr || g.in_dtype == KVQ_BF16) {
        // new tokens: to fp32, rotate if asked, store as saturated fp16
        uint32_t* w = reinterpret_cast<uint32_t*>(&val);
        float x[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          x[2 * i] = bits16_to_f32((uint16_t)(w[i] & 0xFFFF), g.in_dtype);
          x[2 * i + 1] = bits16_to_f32((uint16_t)(w[i] >> 16), g.in_dtype);
        }
        if (c.k_signs != nullptr) {
          if (D == 128) rotate_row8<128>(x, c.k_signs, v); else rotate_row8<64>(x, c.k_signs, v);
        }
        if (is_new) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            w[i] = (uint32_t)f32_to_fp16_sat_bits(x[2 * i]) | ((uint32_t)f32_to_fp16_sat_bits(x[2 * i + 1]) << 16);
        }
      }
      if (is_new && !complete) *reinterpret_cast<uint4*>(tail + (size_t)slot * D + v * 8) = val;
      if (active) *reinterpret_cast<uint4*>(sX + (size_t)slot * D + v * 8) = val;
    }
    if (!complete) continue;
    __syncthreads();
    uint8_t* pg = c.pages + ((size_t)bh * g.n_pages + page) * g.page_bytes;
    for (int d = tid; d < D; d += kThreads) {
      float mn = INFINITY, mx = -INFINITY;
      for (int t = 0; t < kPageTokens; ++t) {
        float x = bits16_to_f32(sX[t * D + d], KVQ_FP16);
        mn = fminf(mn, x);
        mx = fmaxf(mx, x);
      }
      GroupParams p = group_params(mn, mx, qmax);
      reinterpret_cast<uint32_t*>(pg + g.k_meta_off)[d] = p.meta;
      for (int t = 0; t < kPageTokens; ++t)
        sC[t * D + d] = (uint8_t)code_of(bits16_to_f32(sX[t * D + d], KVQ_FP16), p, qmax);
    }
    __syncthreads();
    pack_k_rows(sC, D, kPageTokens, 0, pg, D, g.kb, tid);
  }
}

// Residual window: the new tokens that stay unquantized (positions >= the last complete block of R) are copied to
// the ring, key row and value row of token t in slot t % R.  Runs after the quantize kernel, which may still read
// the slots being replaced.
__global__ void __launch_bounds__(kThreads)
window_store_kernel(Geom g, CachePtrs c, const uint16_t* __restrict__ k_new, const uint16_t* __restrict__ v_new,
                    int64_t sb, int64_t sh, int64_t st, int t_new) {
  begin_after_predecessor();
  const int bh = blockIdx.y, b = bh / g.Hkv, h = bh % g.Hkv;
  const int t0 = c.seq_len[b];
  if (!append_fits(t0, t_new, g.capacity)) return;
  const int R = g.R, D = g.D, vpr = D / 8;
  const int first = max(t0, ((t0 + t_new) / R) * R), n = t0 + t_new - first;     // tokens first .. first + n - 1 stay
  for (int idx = blockIdx.x * kThreads + threadIdx.x; idx < n * 2 * vpr; idx += gridDim.x * kThreads) {
    const int t = first + idx / (2 * vpr), side = (idx / vpr) & 1, vcol = idx % vpr;
    const uint16_t* src = (side ? v_new : k_new) + (int64_t)b * sb + (int64_t)h * sh + (int64_t)(t - t0) * st + 8 * vcol;
    uint16_t* dst = c.kv_win + (((size_t)bh * R + (t % R)) * 2 + side) * D + 8 * vcol;
    *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
  }
}

__global__ void bump_seq_len_kernel(Geom g, CachePtrs c, int t_new) {
  begin_after_predecessor();
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= g.B) return;
  int t0 = c.seq_len[b];
  if (!append_fits(t0, t_new, g.capacity)) {
    atomicOr(c.status, KVQ_STATUS_CAPACITY);
  } else {
    c.seq_len[b] = t0 + t_new;
  }
}

}  // namespace

int launch_quantize_append(const Geom& g, const CachePtrs& c, const void* k_new, const void* v_new,
                           int64_t sb, int64_t sh, int64_t st, int t_new, cudaStream_t stream) {
  if (append_rows_serves(g, c.k_signs != nullptr, t_new)) return launch_append_rows(g, c, k_new, v_new, sb, sh, st, t_new, stream);
  const uint16_t* k = static_cast<const uint16_t*>(k_new);
  const uint16_t* v = static_cast<const uint16_t*>(v_new);
  // 32-token tasks touched per stream: at most ceil(t_new / 32) + 1; a CTA for every four of them, up to eight waves of CTAs, whose warps stride
  // over the passes (16-bit rows, bit planes, rotated keys: over the tasks)
  const int max_tasks = (t_new + 31) / 32 + 1;
  // (head_dim 64: a CTA for eight, and five CTAs per SM; when that was chosen four layers of 64 streams x 4,096 tokens 99 us, a CTA for four
  // 102, at four CTAs 106)
  const bool rot = c.k_signs != nullptr && g.k_axis == 0;
  const int per_cta = g.D == 64 && !rot ? 2 * kWarps : kWarps;
  int gx = (max_tasks + per_cta - 1) / per_cta;
  const int streams = g.B * g.Hkv;
  const int want = (148 * 16 + streams - 1) / streams;       // enough CTAs to fill the GPU, not one per task
  if (gx > want) gx = want;
  // Both sides token-wise and by passes, head_dim 128: whole waves of the four CTAs that an SM holds, so that no last wave is nearly empty and a
  // warp has passes to load ahead.  One wave where a warp then has at most eight pieces of 4 KB and both sides take about as long (values of 4
  // bits, keys of 2 or 4), two up to sixty with keys of 4 and values of 2 or 4 bits, else up to thirty, beyond that a warp per task up to eight waves.
  // As many CTAs as tasks / two waves / one, us, before the rows left the L2 first (streams x tokens, layers):
  //            40 x 3,000, 4          16 x 8,000, 4          64 x 4,000, 2          64 x 8,000, 1          64 x 16,000, 1
  //   K4V4     88.6 / 84.0 / 79.9     91.7 / 88.6 / 80.8     81.3 / 76.4 / 80.0     73.1 / 72.6 / 76.0     138.5 / 140.3 / 146.3
  //   K2V4     89.6 / 87.2 / 82.8     93.3 / 91.4 / 84.1     81.7 / 78.2 / 84.0     75.0 / 72.8 / 78.5     140.5 / 139.1 / 151.6
  //   K4V2     88.8 / 85.3 / 87.3     92.0 / 89.2 / 89.7     79.7 / 75.7 / 84.7     73.1 / 71.5 / 78.1     135.5 / 133.7 / 147.5
  //   K8V4    102.7 / 96.6 / 102.1   106.2 / 100.3 / 103.7   94.6 / 88.7 / 104.7    86.9 / 83.1 / 99.3     164.9 / 158.7 / 189.8
  // (pieces of one wave: 6, 7, 14, 27, 54; since the rows leave the L2 first 48 x 16,000 K4V2 104.0 / 99.6 and K4V4 108.1 / 104.3 with as many
  // CTAs as tasks / two waves, K2V4 106.4 / 108.4, 64 x 16,000 K8V8 184 / 193).
  // Fewer than four CTAs of a wave for each stream and side: no rule, the waves would not be whole.  At head_dim 64 whole waves lose (64
  // streams x 4,096 tokens, 4 layers, 96.5 / 95.0 / 105.4; 40 x 2,500 52.6 / 52.4 / 58.7).
  const int per_x = 2 * streams, resident = 4 * 148;
  auto by_passes = [](int bits) { return bits == 2 || bits == 4 || bits == 8; };
  if (g.D == 128 && g.k_axis == 0 && !rot && by_passes(g.kb) && by_passes(g.vb) && 4 * per_x <= resident) {
    const long long pieces = 2ll * max_tasks * per_x / (kWarps * resident);        // per warp of a single wave
    const int waves = pieces <= 8 && g.kb <= 4 && g.vb == 4 ? 1 : pieces <= (g.kb == 4 && g.vb <= 4 ? 60 : 30) ? 2 : 0;
    if (waves != 0) gx = std::min(gx, waves * resident / per_x);
  }
  dim3 grid1(gx, streams, g.k_axis == 0 ? 2 : 1);            // which side comes first: see the kernel
  auto side_slots = [](int bits, bool is_v) { return bits == 2 || bits == 4 || bits == 8 ? kWarps * slot_bytes(bits, is_v) : 0; };
  const size_t smem1 = std::max(side_slots(g.vb, true), g.k_axis == 0 && !rot ? side_slots(g.kb, false) : 0);
  cudaError_t e = cudaSuccess;
  auto run = [&](auto kern, dim3 grid, unsigned threads, size_t smem, auto... args) {      // (the first failure ends the call)
    if (e == cudaSuccess) e = launch_dependent(kern, grid, threads, smem, stream, 1, args...);
  };
#define KVQ_QLAUNCH(D_, T_) \
  run(rot ? quant_token_kernel<D_, T_, true> : quant_token_kernel<D_, T_, false>, grid1, kThreads, smem1, g, c, k, v, sb, sh, st, t_new)
  if (g.D == 128 && g.in_dtype == KVQ_BF16) KVQ_QLAUNCH(128, KVQ_BF16);
  else if (g.D == 128) KVQ_QLAUNCH(128, KVQ_FP16);
  else if (g.in_dtype == KVQ_BF16) KVQ_QLAUNCH(64, KVQ_BF16);
  else KVQ_QLAUNCH(64, KVQ_FP16);
#undef KVQ_QLAUNCH
  dim3 grid2((t_new + 127) / 128 + 1, streams);
  if (g.k_axis == 1 && g.D == 128 && (g.kb == 4 || g.kb == 8)) {
    grid2.x = std::min<unsigned>(grid2.x, (148 * 12 + streams - 1) / streams);
#define KVQ_KCHAN(T_, KB_)                                                                                           \
  run(c.k_signs ? quant_kchan_fast_kernel<T_, KB_, true> : quant_kchan_fast_kernel<T_, KB_, false>, grid2, 256, c.k_signs ? 0 : 32768, g, c, k, \
      sb, sh, st, t_new)
    if (g.in_dtype == KVQ_BF16) { if (g.kb == 4) KVQ_KCHAN(KVQ_BF16, 4); else KVQ_KCHAN(KVQ_BF16, 8); }
    else { if (g.kb == 4) KVQ_KCHAN(KVQ_FP16, 4); else KVQ_KCHAN(KVQ_FP16, 8); }
#undef KVQ_KCHAN
  } else if (g.k_axis == 1) {
    size_t smem = (size_t)kPageTokens * g.D * 3;
    cudaFuncSetAttribute(quant_kchan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 128 * 3);
    run(quant_kchan_kernel, grid2, kThreads, smem, g, c, k, sb, sh, st, t_new);
  }
  if (g.R) run(window_store_kernel, dim3(1, streams), kThreads, 0, g, c, k, v, sb, sh, st, t_new);
  run(bump_seq_len_kernel, dim3((g.B + 127) / 128), 128, 0, g, c, t_new);
  return e == cudaSuccess ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
}

}  // namespace kvq
