// Dispatch of the fast decode path (the merge of the split partials is part of the kernel).
#include <atomic>
#include <chrono>

#include "kvq_decode_mma_kernel.cuh"

namespace kvq {
namespace mma {

// Instantiation units (kvq_decode_mma_inst_*.cu).
#define KVQ_MMA_DECL(D, KB, VB, KAXIS, NGK, NGV, NH, MINB)                                                  \
  extern template int launch_mma_inst<D, KB, VB, KAXIS, NGK, NGV, NH, MINB>(                                   \
      const Geom&, const CachePtrs&, const void*, float, float*, int, void*, int, unsigned long long,              \
      unsigned long long, long long, cudaStream_t);
#include "kvq_decode_mma_list.inc"
#undef KVQ_MMA_DECL

}  // namespace mma

constexpr int kFlatGrid = 2 * 148;   // slot capacity is sized for grids up to twice this

int flat_slot_cap(const Geom& g) {
  const int streams = g.B * g.Hkv;
  int s = (2 * kFlatGrid + streams - 1) / streams + 2;
  if (s > g.n_pages + 1) s = g.n_pages + 1;
  if (g.R) s += 1;                           // one more slot per stream: the partial of the residual window
  return s;
}

// Partials [streams][slots][G][D + 2] floats, then one 64-bit count word per stream.
size_t flat_workspace_bytes(const Geom& g) {
  const int s_cap = flat_slot_cap(g);
  return mma::tag_offset_floats(g.B * g.Hkv, s_cap, g.G * g.rows, g.D) * sizeof(float) + (size_t)g.B * g.Hkv * 8;
}

// Id of a launch: the words that count a stream's finished partials carry it, so that neither stale workspace
// contents nor an earlier call's counts are ever taken for this call's.  Starts at a clock value, never 0.
static unsigned long long next_call_id() {
  static std::atomic<unsigned long long> counter{
      ((unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count() << 20) | 1ull};
  unsigned long long v = counter.fetch_add(1, std::memory_order_relaxed);
  return v ? v : counter.fetch_add(1, std::memory_order_relaxed);
}

// Finds the instantiation for this geometry; launches it unless `probe`.  *grid = CTAs of the launch, *ring (may be null) = its ring.
static int pick(const Geom& g, const CachePtrs& c, const void* q, float c1, float* ws, int s_cap, void* out,
                int out_dtype, const DecodeDebug& dbg, cudaStream_t stream, bool probe, int* grid,
                mma::SmemLayout* ring = nullptr) {
  const int ngk = (g.k_axis == 1 || g.kb == 16) ? 1 : g.D / g.gk;
  const int ngv = (g.vb == 16) ? 1 : g.D / g.gv;
  const int nh = g.G * g.rows <= 4 ? 1 : 2;                                // (virtual) query heads per lane
#define KVQ_MMA_DECL(D_, KB_, VB_, KAXIS_, NGK_, NGV_, NH_, MINB_)                                      \
  if (g.D == D_ && g.kb == KB_ && g.vb == VB_ && g.k_axis == KAXIS_ && ngk == NGK_ && ngv == NGV_ &&          \
      NH_ == nh) {                                                                                            \
    *grid = 148 * MINB_;                                                                                      \
    if (ring) *ring = mma::smem_layout(g.page_bytes, mma::ring_stages(g, NH_, NGV_, KAXIS_ == 1, MINB_), g.B, D_, NH_, NGV_, KAXIS_ == 1); \
    if (probe) return KVQ_OK;                                                                                 \
    return mma::launch_mma_inst<D_, KB_, VB_, KAXIS_, NGK_, NGV_, NH_, MINB_>(                          \
        g, c, q, c1, ws, s_cap, out, out_dtype, next_call_id(),                                               \
        dbg.wait_us ? 1000ull * dbg.wait_us : mma::kWaitTimeoutNs, dbg.skip_page, stream);                    \
  }
#include "kvq_decode_mma_list.inc"
#undef KVQ_MMA_DECL
  return KVQ_ERR_UNSUPPORTED;
}

bool decode_mma_supported(const Geom& g) {
  if (g.B > mma::kMaxBatchFlat) return false;
  CachePtrs none{};
  int grid = 0;
  return pick(g, none, nullptr, 0.f, nullptr, 0, nullptr, 0, DecodeDebug{}, nullptr, true, &grid) == KVQ_OK;
}

namespace {
// The kernel's plan for given lengths, worked out on the host by the same functions.  Each stream's CTAs go to `each`(stream, CTAs, whether it
// has a residual window), null for a stream without pages.
template <int WAVES, typename Each>
void host_plan(const Geom& g, int gap, const int32_t* seq_len, int64_t* starts, int32_t* cursors, int32_t* info, Each&& each) {
  auto len = [&](int b) { return seq_len[b] < 0 ? 0 : seq_len[b] > g.capacity ? g.capacity : seq_len[b]; };
  int pref[mma::kMaxBatchFlat + 1] = {}, vpref[mma::kMaxBatchFlat + 1] = {};
  int pmax = 0;
  for (int b = 0; b < g.B; ++b) {
    const int n = len(b), pages = ((g.R ? n / g.R * g.R : n) + kPageTokens - 1) / kPageTokens;
    pmax = pages > pmax ? pages : pmax;
    pref[b + 1] = pref[b] + pages * g.Hkv;
    vpref[b + 1] = vpref[b] + (pages ? (pages + gap) * g.Hkv : 0);
  }
  const int slots = flat_slot_cap(g) - (g.R ? 1 : 0);
  const mma::FlatPlan plan = mma::make_plan(vpref[g.B], pmax + gap, WAVES * 148, slots);
  const bool waves = mma::weighted_shares<WAVES>(plan, gap, WAVES * 148, pmax, slots);
  info[0] = slots; info[1] = plan.c_eff; info[2] = waves;
  for (int c = 0; c <= plan.c_eff && plan.N; ++c) {
    const mma::ShareStart at = mma::share_start<WAVES>(plan, waves, c, pref, vpref, g.B, g.Hkv, gap);
    starts[c] = at.x;
    if (c < plan.c_eff) { cursors[3 * c] = at.b; cursors[3 * c + 1] = at.h; cursors[3 * c + 2] = at.page; }
  }
  for (int b = 0; b < g.B; ++b) {
    const int pages = (pref[b + 1] - pref[b]) / g.Hkv;
    for (int h = 0; h < g.Hkv; ++h) {
      const long long xs = (long long)vpref[b] + (long long)h * (pages + gap) + gap;
      auto cta = [&](int which) { return pages ? mma::stream_cta<WAVES>(plan, waves, xs, pages, gap, which) : -1; };
      const mma::StreamCtas ctas(cta(0), cta(1), cta(2));
      each(b * g.Hkv + h, pages ? &ctas : nullptr, len(b) % (g.R ? g.R : 1) != 0);
    }
  }
}
}  // namespace

int decode_mma_plan(const Geom& g, const int32_t* seq_len, int32_t* parts, int32_t* windows, int64_t* starts, int32_t* cursors, int32_t* info) {
  CachePtrs none{};
  int grid = 0;
  if (g.B > mma::kMaxBatchFlat) return KVQ_ERR_UNSUPPORTED;
  const int rc = pick(g, none, nullptr, 0.f, nullptr, 0, nullptr, 0, DecodeDebug{}, nullptr, true, &grid);
  if (rc != KVQ_OK) return rc;
  const int gap = mma::gap_pages(g.D, g.kb, g.vb, g.k_axis, g.B * g.Hkv);
  auto each = [&](int stream, const mma::StreamCtas* ctas, bool has_window) {
    if (parts) {
      parts[2 * stream] = ctas ? ctas->first : 0;
      parts[2 * stream + 1] = ctas ? ctas->partials() : 0;
    }
    if (windows) {
      windows[2 * stream] = ctas && has_window ? ctas->window : -1;
      windows[2 * stream + 1] = ctas ? ctas->counted(has_window) : 0;
    }
  };
  if (grid == 3 * 148) host_plan<3>(g, gap, seq_len, starts, cursors, info, each);
  else host_plan<2>(g, gap, seq_len, starts, cursors, info, each);
  return KVQ_OK;
}

namespace {
__global__ void divide_kernel(const long long* n, const long long* d, long long* q, int count) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) q[i] = mma::divide(n[i], d[i]);
}
}  // namespace

int debug_divide(const int64_t* n, const int64_t* d, int64_t* q, int count, cudaStream_t stream) {
  divide_kernel<<<(count + 255) / 256, 256, 0, stream>>>(reinterpret_cast<const long long*>(n), reinterpret_cast<const long long*>(d),
                                                        reinterpret_cast<long long*>(q), count);
  return cudaGetLastError() == cudaSuccess ? KVQ_OK : KVQ_ERR_CUDA_LAUNCH;
}

int decode_mma_ring(const Geom& g, int32_t* info) {
  CachePtrs none{};
  int grid = 0;
  mma::SmemLayout ring{};
  if (g.B > mma::kMaxBatchFlat) return KVQ_ERR_UNSUPPORTED;
  const int rc = pick(g, none, nullptr, 0.f, nullptr, 0, nullptr, 0, DecodeDebug{}, nullptr, true, &grid, &ring);
  if (rc != KVQ_OK) return rc;
  info[0] = ring.ring_bytes;
  for (info[1] = g.R ? g.R - 1 : 0; info[1] > 0 && !mma::window_fits_ring(ring, info[1], g.D);) --info[1];
  return KVQ_OK;
}

int launch_decode_mma(const Geom& g, const CachePtrs& c, const void* q, void* out, int out_dtype, float c1,
                      float* ws, const DecodeDebug& dbg, cudaStream_t stream) {
  const int s_cap = flat_slot_cap(g);
  int grid = 0;
  if (dbg.fast_impl == 2) {
    if (!decode_tc_supported(g, c)) return KVQ_ERR_UNSUPPORTED;
    if (g.R) {      // the residual window first: its partial (or, for sequences without pages, the output) is ready when the last partial is merged
      const int rc = launch_decode_window(g, c, q, out, out_dtype, c1, ws, s_cap, stream);
      if (rc != KVQ_OK) return rc;
    }
    return launch_decode_tc(g, c, q, c1, ws, s_cap, out, out_dtype, next_call_id(),
                            dbg.wait_us ? 1000ull * dbg.wait_us : mma::kWaitTimeoutNs, dbg.skip_page, stream);
  }
  return pick(g, c, q, c1, ws, s_cap, out, out_dtype, dbg, stream, false, &grid);
}

}  // namespace kvq
