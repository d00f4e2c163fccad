// sampler.cu -- curvature-guided subgraph samplers (§3.2, Eq. 7 and Eq. 8: the experiments'
// ERC-LG-sub(node) and ERC-LG-sub(edge), GraphSAINT-style) and GraphSAINT's count normalisation.
//
// A draw is exact integer inverse-CDF sampling: the float32 probabilities become fixed-point
// weights W_i = round(p_i 2^40) (from the float's bits, no float arithmetic), an exclusive scan
// gives E_i = W_0 + .. + W_{i-1} and T, a 64-bit Philox word x gives r = floor(x T / 2^64), and
// the draw is the largest i with E_i <= r (that i has W_i > 0).  Everything is integer, so the
// drawn indices do not depend on summation order.  The drawn nodes (or the drawn edges'
// endpoints) are marked and compacted in id order; the subgraph's edges are the canonical edges
// with both endpoints marked (induced), or the drawn edges themselves, compacted in id order.
//
// A subgraph is drawn for every training step, so passes and round trips count: the weights are
// formed inside the scan, a draw marks at once, and a compaction is one pass that reads the marks
// (or tests the endpoints), finds its place by look-back and writes the ids.  169k nodes, 16,934
// draws and the subgraph's counts: 164 us, 232 us before; 64.3M edges, 6.4M draws: 1.44 ms, 3.95 ms
// before, with separate passes for weights, draws, marks, induced flags, scans and compactions and
// two round trips.
#include <algorithm>

#include "erc_internal.cuh"

namespace erc {
namespace {

constexpr int ST = 256;
constexpr int SWARPS = ST / 32;
// Entries per thread of a scan or compaction tile: 32 from SLARGE entries on, so that the look-back
// over the tiles in flight stays short, 8 below, so that a small graph's passes spread over SMs.
constexpr int SIPT_LARGE = 32, SIPT_SMALL = 8;
constexpr int64_t SLARGE = 1 << 20;
constexpr int SMID = 64;
constexpr uint32_t SAMPLER_TAG = 0x53414D50u;

struct SamplePlan {
  int64_t *E, *Emid, *totals;  // Emid: every SMID-th entry of E; totals: [0] T [1] nodes [2] edges
  uint8_t *nmark, *emark;
  uint32_t* nbits;             // the node marks as bits
  // look-back words of the passes over the weights, the nodes and the edges, side by side
  unsigned long long *status, *status_n, *status_m;
  size_t words;
  unsigned* err;  // [0] the abort word; [1..3] the passes' tickets
};
// Bits of the abort word.  Once one is set the passes that follow write nothing: a call that
// reports an error leaves its outputs alone.  (A word of its own for each reason, read by every
// block of the compactions, took 3% to 12% of a call.)
constexpr unsigned WAIT_RAN_OUT = 1, BAD_PROB = 2, NO_WEIGHT = 4;  // tile_prefix sets the first

inline int64_t stile(int64_t count) { return ST * (count < SLARGE ? SIPT_SMALL : SIPT_LARGE); }
inline int64_t stiles(int64_t count) { return (count + stile(count) - 1) / stile(count); }
// The most tiles of a pass over `count` entries or fewer: just below SLARGE entries there are four
// times as many as from SLARGE on (512 against 128).
inline int64_t stiles_max(int64_t count) {
  return std::max(stiles(count), stiles(std::min(count, SLARGE - 1)));
}

// copies of the node marks: at most 16, and 64 MB of them
constexpr int64_t MARK_COPIES = 16, MARK_BYTES = int64_t(64) << 20;
inline int mark_copies(int32_t n) {
  return (int)std::max<int64_t>(1, std::min(MARK_COPIES, MARK_BYTES / n));
}
// the most bytes of marks of a graph of n nodes or fewer
inline int64_t mark_bytes_max(int64_t n) {
  return std::max(n, std::min(MARK_COPIES * n, MARK_BYTES));
}

// The plan of every call on a graph of n nodes and m edges, drawn by node or by edge.  No array
// shrinks as n or m grows, so a workspace serves every graph up to the sizes it was reported for.
void plan_sample(Arena& a, SamplePlan& p, int32_t n, int64_t m) {
  const int64_t count = std::max<int64_t>(n, m);  // entries drawn from, at most
  p.E = a.take<int64_t>(count);
  p.Emid = a.take<int64_t>(count / SMID + 1);
  p.nmark = a.take<uint8_t>(mark_bytes_max(n));
  p.nbits = a.take<uint32_t>((size_t)n / 32 + 1);
  p.emark = a.take<uint8_t>(m > 0 ? m : 1);
  p.totals = a.take<int64_t>(4);
  p.err = a.take<unsigned>(8);
  const int64_t w = stiles_max(count), wn = stiles_max(n), wm = stiles_max(m);
  p.words = (size_t)(w + wn + wm);
  p.status = a.take<unsigned long long>(p.words);
  p.status_n = p.status + w;
  p.status_m = p.status_n + wn;
}

// W = round(p 2^40) (half up) from the bits of p; p must lie in [0, 1]
__device__ __forceinline__ uint64_t fixed_weight(float p, bool& bad) {
  if (!(p >= 0.f && p <= 1.f)) {
    bad = true;
    return 0;
  }
  if (p == 0.f) return 0;
  const uint32_t bits = __float_as_uint(p);
  const int e = (int)(bits >> 23);
  const uint64_t mant = e ? ((bits & 0x7fffffu) | 0x800000u) : (bits & 0x7fffffu);
  const int shift = (e ? e - 150 : -149) + 40;  // p 2^40 = mant 2^shift
  if (shift >= 0) return mant << shift;
  return shift > -40 ? (mant + (1ull << (-shift - 1))) >> (-shift) : 0;
}

// the block's tile of a pass, or -1 once the call has failed
__device__ __forceinline__ int64_t claim_tile(unsigned* ticket, const unsigned* abort) {
  __shared__ unsigned s_tile;
  if (threadIdx.x == 0) s_tile = aborted(abort) ? 0xffffffffu : atomicAdd(ticket, 1u);
  __syncthreads();
  return s_tile == 0xffffffffu ? -1 : (int64_t)s_tile;
}

// E, Emid and T of the weights.  A warp takes 32 SIPT consecutive entries, a lane four neighbouring
// ones of each 128, so that a scan over the lanes serves 128 entries; `vec`: prob is 16-byte
// aligned.
template <int SIPT>
__global__ void __launch_bounds__(ST)
    k_weight_scan(const float* __restrict__ prob, int64_t count, bool vec, int64_t* __restrict__ E,
                  int64_t* __restrict__ Emid, int64_t* __restrict__ total,
                  unsigned long long* status, unsigned* ticket, unsigned* abort,
                  unsigned spin_limit) {
  constexpr int64_t STILE = ST * SIPT;
  __shared__ unsigned long long s_warp[SWARPS], s_prefix, s_total;
  const int64_t t = claim_tile(ticket, abort);
  if (t < 0) return;
  constexpr int ROUNDS = SIPT / 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t base = t * STILE + (int64_t)warp * 32 * SIPT + 4 * lane;
  float4 p[ROUNDS];
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    const int64_t i = base + 128 * j;
    if (vec && i + 4 <= count) {
      p[j] = __ldg(reinterpret_cast<const float4*>(prob + i));
    } else {
      p[j].x = i + 0 < count ? prob[i + 0] : 0.f;
      p[j].y = i + 1 < count ? prob[i + 1] : 0.f;
      p[j].z = i + 2 < count ? prob[i + 2] : 0.f;
      p[j].w = i + 3 < count ? prob[i + 3] : 0.f;
    }
  }
  bool bad = false;
  unsigned long long sum = 0;
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j)
    sum += fixed_weight(p[j].x, bad) + fixed_weight(p[j].y, bad) + fixed_weight(p[j].z, bad) +
           fixed_weight(p[j].w, bad);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s_warp[warp] = sum;
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(abort, BAD_PROB);
  if (warp == 0) {
    const unsigned long long w = lane < SWARPS ? s_warp[lane] : 0;
    unsigned long long inc = w;
#pragma unroll
    for (int o = 1; o < SWARPS; o <<= 1) {
      const unsigned long long x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane < SWARPS) s_warp[lane] = inc - w;
    const unsigned long long tot = __shfl_sync(0xffffffffu, inc, SWARPS - 1);
    const unsigned long long prefix = tile_prefix(status, t, tot, spin_limit, abort);
    if (lane == 0) {
      s_prefix = prefix;
      s_total = prefix + tot;
    }
  }
  __syncthreads();
  unsigned long long run = s_prefix + s_warp[warp];
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    const int64_t i = base + 128 * j;
    const unsigned long long w0 = fixed_weight(p[j].x, bad), w1 = fixed_weight(p[j].y, bad),
                             w2 = fixed_weight(p[j].z, bad), w3 = fixed_weight(p[j].w, bad);
    const unsigned long long w = w0 + w1 + w2 + w3;
    unsigned long long inc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    const unsigned long long e0 = run + inc - w, e1 = e0 + w0, e2 = e1 + w1, e3 = e2 + w2;
    if (i + 4 <= count) {
      *reinterpret_cast<ulonglong2*>(E + i) = make_ulonglong2(e0, e1);
      *reinterpret_cast<ulonglong2*>(E + i + 2) = make_ulonglong2(e2, e3);
    } else {
      if (i + 0 < count) E[i + 0] = (int64_t)e0;
      if (i + 1 < count) E[i + 1] = (int64_t)e1;
      if (i + 2 < count) E[i + 2] = (int64_t)e2;
    }
    if (lane % (SMID / 4) == 0 && i < count) Emid[i / SMID] = (int64_t)e0;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  if ((t + 1) * STILE >= count && threadIdx.x == 0) {
    *total = (int64_t)s_total;
    if (s_total == 0) atomicOr(abort, NO_WEIGHT);
  }
}

// draw k: the largest i with E_i <= floor(x_k T / 2^64), found in the scan's tiles (their final
// status words hold the sums with each tile: 8 bytes a tile, 63 KB for 64M entries), then in Emid
// (L2), then among the SMID entries of E it leads to: a plain binary search over E misses L2 about
// eight times a draw on 64M entries.  Marks node i, or edge i's endpoints and, where emark is not
// null, the edge.  Stores to one line queue up in L2, and a power-law graph's draws keep hitting
// the lines of its hubs: the blocks spread them over `copies` arrays of marks, which the compaction
// joins.  (Testing a mark before storing it queues the test behind the stores: 276 us against 31
// for 129k draws over 6,821 nodes.)
__global__ void __launch_bounds__(ST)
    k_draw(const int64_t* __restrict__ E, const int64_t* __restrict__ Emid, int64_t count,
           int64_t tile, const unsigned long long* __restrict__ status,
           const int64_t* __restrict__ tot,
           int64_t budget, uint2 key, int64_t first, uint32_t stream,
           const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
           uint8_t* __restrict__ nmark, int32_t n, int copies, uint8_t* __restrict__ emark,
           const unsigned* abort) {
  if (aborted(abort)) return;
  nmark += (size_t)(blockIdx.x % copies) * n;
  const uint64_t T = (uint64_t)tot[0];
  const int64_t tiles = (count + tile - 1) / tile;
  for (int64_t k = (int64_t)blockIdx.x * ST + threadIdx.x; k < budget;
       k += (int64_t)gridDim.x * ST) {
    const uint64_t d = (uint64_t)(first + k);
    const uint4 w =
        philox4x32_10(make_uint4((uint32_t)d, (uint32_t)(d >> 32), SAMPLER_TAG, stream), key);
    const uint64_t x = ((uint64_t)w.x << 32) | w.y;
    const int64_t r = (int64_t)__umul64hi(x, T);
    int64_t lo = 0, hi = tiles - 1;  // first tile whose sum with it exceeds r
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if ((int64_t)(__ldg(status + mid) >> 2) > r) hi = mid; else lo = mid + 1;
    }
    // the last of Emid, then of E, with E <= r (the first of each range always is)
    const int64_t tile_end = min(count, (lo + 1) * tile);
    lo = lo * (tile / SMID);
    hi = (tile_end - 1) / SMID;
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (Emid[mid] <= r) lo = mid; else hi = mid - 1;
    }
    lo = lo * SMID;
    hi = min(tile_end, lo + SMID) - 1;
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (E[mid] <= r) lo = mid; else hi = mid - 1;
    }
    const int64_t i = lo;
    if (stream) {
      if (emark) emark[i] = 1;
      const int32_t u = eu[i], v = ev[i];
      nmark[u] = 1;
      nmark[v] = 1;
    } else {
      nmark[i] = 1;
    }
  }
}

struct MarkedFlag {
  const uint8_t* mark;
  __device__ bool operator()(int64_t i) const { return mark[i] != 0; }
};
struct CopiesFlag {  // marked in any of the copies, `n` apart
  const uint8_t* mark;
  int64_t n;
  int copies;
  __device__ bool operator()(int64_t i) const {
    unsigned any = 0;
    for (int c = 0; c < copies; ++c) any |= mark[c * n + i];
    return any != 0;
  }
};
struct InducedFlag {  // both endpoints of edge i are marked
  const int32_t *eu, *ev;
  const uint32_t* nbits;
  __device__ bool operator()(int64_t i) const {
    const int32_t u = __ldg(eu + i), v = __ldg(ev + i);
    return (__ldg(nbits + (u >> 5)) >> (u & 31)) & (__ldg(nbits + (v >> 5)) >> (v & 31)) & 1u;
  }
};

// the ids i < count with flag(i), ascending, and the flags as bits where `bits` is not null (an
// eighth of the marks' bytes: 2.4M nodes' bits mostly stay in L1 while the edges test them)
template <int SIPT, class Flag>
__global__ void __launch_bounds__(ST)
    k_compact(Flag flag, int64_t count, int32_t* __restrict__ out, uint32_t* __restrict__ bits,
              int64_t* __restrict__ total,
              unsigned long long* status, unsigned* ticket, unsigned* abort, unsigned spin_limit) {
  constexpr int64_t STILE = ST * SIPT;
  __shared__ unsigned s_warp[SWARPS];
  __shared__ unsigned long long s_prefix, s_total;
  const int64_t t = claim_tile(ticket, abort);
  if (t < 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t base = t * STILE + (int64_t)warp * 32 * SIPT;
  unsigned mine = 0;  // the flags of entries base + 32 lane .. + 31
  unsigned cnt = 0;
#pragma unroll
  for (int j = 0; j < SIPT; ++j) {
    const int64_t i = base + 32 * j + lane;
    const unsigned bal = __ballot_sync(0xffffffffu, i < count && flag(i));
    if (lane == j) mine = bal;
    cnt += __popc(bal);
  }
  if (bits && lane < SIPT && base + 32 * lane < count) bits[(base >> 5) + lane] = mine;
  static_assert(SIPT <= 32, "a lane holds one ballot");
  if (lane == 0) s_warp[warp] = cnt;
  __syncthreads();
  if (warp == 0) {
    const unsigned w = lane < SWARPS ? s_warp[lane] : 0;
    unsigned inc = w;
#pragma unroll
    for (int o = 1; o < SWARPS; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane < SWARPS) s_warp[lane] = inc - w;
    const unsigned tot = __shfl_sync(0xffffffffu, inc, SWARPS - 1);
    const unsigned long long prefix = tile_prefix(status, t, tot, spin_limit, abort);
    if (lane == 0) {
      s_prefix = prefix;
      s_total = prefix + tot;
    }
  }
  __syncthreads();
  int64_t at = (int64_t)s_prefix + s_warp[warp];
#pragma unroll
  for (int j = 0; j < SIPT; ++j) {
    const unsigned bal = __shfl_sync(0xffffffffu, mine, j);
    if ((bal >> lane) & 1u)
      out[at + __popc(bal & ((1u << lane) - 1u))] = (int32_t)(base + 32 * j + lane);
    at += __popc(bal);
  }
  if ((t + 1) * STILE >= count && threadIdx.x == 0) *total = (int64_t)s_total;
}

__global__ void k_saint_counts(const int32_t* __restrict__ nodes, int64_t n_s,
                               const int32_t* __restrict__ edges, int64_t m_s,
                               int32_t* __restrict__ node_count, int32_t* __restrict__ edge_count) {
  // ids are distinct within a subgraph, so each counter is touched once per call
  for (int64_t i = (int64_t)blockIdx.x * ST + threadIdx.x; i < n_s + m_s;
       i += (int64_t)gridDim.x * ST) {
    if (i < n_s)
      node_count[nodes[i]] += 1;
    else
      edge_count[edges[i - n_s]] += 1;
  }
}

__global__ void k_saint_norm(const int64_t* __restrict__ row_ptr,
                             const int32_t* __restrict__ csr_eid, int32_t n,
                             const int32_t* __restrict__ node_count,
                             const int32_t* __restrict__ edge_count, int32_t N,
                             float* __restrict__ lam, float* __restrict__ alpha) {
  for (int64_t v = (int64_t)blockIdx.x * ST + threadIdx.x; v < n; v += (int64_t)gridDim.x * ST) {
    const int32_t cv = node_count[v];
    lam[v] = __fdiv_rn((float)cv, (float)N);
    for (int64_t j = row_ptr[v]; j < row_ptr[v + 1]; ++j)
      alpha[j] = cv > 0 ? __fdiv_rn((float)edge_count[csr_eid[j]], (float)cv) : 0.f;
  }
}

template <class Flag>
erc_status compact(Flag flag, int64_t count, int32_t* out, uint32_t* bits, int64_t* total,
                   unsigned long long* status, unsigned* ticket, unsigned* abort, unsigned limit,
                   cudaStream_t s) {
  const unsigned grid = (unsigned)stiles(count);
  if (count < SLARGE)
    k_compact<SIPT_SMALL><<<grid, ST, 0, s>>>(flag, count, out, bits, total, status, ticket, abort,
                                              limit);
  else
    k_compact<SIPT_LARGE><<<grid, ST, 0, s>>>(flag, count, out, bits, total, status, ticket, abort,
                                              limit);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  return ERC_OK;
}

}  // namespace
}  // namespace erc

using namespace erc;

extern "C" size_t erc_sample_workspace_size(int32_t n, int64_t m, int64_t budget) {
  if (n < 1 || m < 0 || budget < 0) return 0;
  Arena a(nullptr);
  SamplePlan p;
  plan_sample(a, p, n, m);
  return a.used + 256;
}

extern "C" erc_status erc_sample_subgraph(const erc_graph* g, int32_t kind, const float* prob,
                                          int64_t budget, uint64_t seed, int64_t first_draw,
                                          int32_t induced, int32_t* nodes, int32_t* n_out,
                                          int32_t* edges, int64_t* m_out, void* ws,
                                          size_t ws_bytes, erc_stream stream) {
  clear_error();
  ERC_TRY(check_graph(g));
  ERC_REQUIRE(kind == ERC_SAMPLE_NODES || kind == ERC_SAMPLE_EDGES, "bad sampler kind %d", kind);
  ERC_REQUIRE(budget >= 0 && first_draw >= 0, "budget and first_draw must be >= 0");
  ERC_REQUIRE(n_out && m_out, "n_out and m_out are required");
  ERC_REQUIRE(g->eu && g->ev, "graph edge list required");
  const bool by_edge = kind == ERC_SAMPLE_EDGES;
  const int64_t count = by_edge ? g->m : g->n;
  ERC_REQUIRE(prob || count == 0, "prob is required");
  ERC_REQUIRE(nodes && (edges || g->m == 0), "nodes and edges are required");
  if (ws_bytes < erc_sample_workspace_size(g->n, g->m, budget))
    return set_error(ERC_ERR_CAPACITY, "workspace too small");
  cudaStream_t s = as_stream(stream);
  Arena ar(reinterpret_cast<void*>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255)));
  SamplePlan p;
  plan_sample(ar, p, g->n, g->m);
  *n_out = 0;
  *m_out = 0;
  if (count == 0 || budget == 0) return ERC_OK;
  const bool drawn_edges = by_edge && !induced;  // the subgraph keeps the drawn edges alone
  unsigned* abort = p.err;
  ERC_CUDA(cudaMemsetAsync(p.err, 0, 8 * sizeof(unsigned), s));
  ERC_CUDA(cudaMemsetAsync(p.status, 0, p.words * sizeof(*p.status), s));
  const int copies = mark_copies(g->n);
  ERC_CUDA(cudaMemsetAsync(p.nmark, 0, (size_t)g->n * copies, s));
  if (drawn_edges) ERC_CUDA(cudaMemsetAsync(p.emark, 0, (size_t)g->m, s));
  // Nothing is read back before the end.  A wait that gives up within a compaction leaves its
  // output incomplete; the prefixes are then below their true values, so every index stays in
  // range.
  const unsigned limit = wait_limit(LOOKBACK_SPINS);
  const bool vec = (reinterpret_cast<uintptr_t>(prob) & 15) == 0;
  if (count < SLARGE)
    k_weight_scan<SIPT_SMALL><<<(unsigned)stiles(count), ST, 0, s>>>(
        prob, count, vec, p.E, p.Emid, &p.totals[0], p.status, p.err + 1, abort, limit);
  else
    k_weight_scan<SIPT_LARGE><<<(unsigned)stiles(count), ST, 0, s>>>(
        prob, count, vec, p.E, p.Emid, &p.totals[0], p.status, p.err + 1, abort, limit);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  const uint2 key = make_uint2((uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
  k_draw<<<grid_for(budget, ST), ST, 0, s>>>(
      p.E, p.Emid, count, stile(count), p.status, p.totals, budget, key, first_draw,
      by_edge ? 1u : 0u, g->eu, g->ev, p.nmark, g->n, copies, drawn_edges ? p.emark : nullptr,
      abort);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  ERC_TRY(compact(CopiesFlag{p.nmark, g->n, copies}, (int64_t)g->n, nodes, p.nbits, &p.totals[1],
                  p.status_n, p.err + 2, abort, limit, s));
  if (g->m > 0) {
    if (drawn_edges)
      ERC_TRY(compact(MarkedFlag{p.emark}, g->m, edges, (uint32_t*)nullptr, &p.totals[2],
                      p.status_m, p.err + 3, abort, limit, s));
    else
      ERC_TRY(compact(InducedFlag{g->eu, g->ev, p.nbits}, g->m, edges, (uint32_t*)nullptr,
                      &p.totals[2], p.status_m, p.err + 3, abort, limit, s));
  }
  int64_t h_tot[3] = {0, 0, 0};
  unsigned h_err = 0;
  ERC_CUDA(cudaMemcpyAsync(h_tot, p.totals, 3 * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  ERC_CUDA(cudaMemcpyAsync(&h_err, abort, sizeof h_err, cudaMemcpyDeviceToHost, s));
  ERC_CUDA(cudaStreamSynchronize(s));
  // a probability out of range stops other tiles' waits, and a scan that gave up may total zero
  if (h_err & BAD_PROB)
    return set_error(ERC_ERR_INVALID_ARG, "probabilities must lie in [0, 1]");
  if (h_err & WAIT_RAN_OUT)
    return set_error(ERC_ERR_TIMEOUT, "a bounded wait in the sampler's scans ran out");
  if (h_err & NO_WEIGHT)
    return set_error(ERC_ERR_INVALID_ARG, "every probability rounds to zero");
  *n_out = (int32_t)h_tot[1];
  *m_out = g->m > 0 ? h_tot[2] : 0;
  return ERC_OK;
}

extern "C" erc_status erc_saint_counts(const erc_graph* g, const int32_t* nodes, int32_t n_s,
                                       const int32_t* edges, int64_t m_s, int32_t* node_count,
                                       int32_t* edge_count, erc_stream stream) {
  clear_error();
  ERC_TRY(check_graph(g));
  ERC_REQUIRE(n_s >= 0 && n_s <= g->n && m_s >= 0 && m_s <= g->m, "bad subgraph sizes");
  ERC_REQUIRE((nodes && node_count) || n_s == 0, "nodes and node_count are required");
  ERC_REQUIRE((edges && edge_count) || m_s == 0, "edges and edge_count are required");
  if (n_s + m_s == 0) return ERC_OK;
  k_saint_counts<<<grid_for(n_s + m_s, ST), ST, 0, as_stream(stream)>>>(nodes, n_s, edges, m_s,
                                                                        node_count, edge_count);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  return ERC_OK;
}

extern "C" erc_status erc_saint_norm(const erc_graph* g, const int32_t* node_count,
                                     const int32_t* edge_count, int32_t N, float* lambda,
                                     float* alpha, erc_stream stream) {
  clear_error();
  ERC_TRY(check_graph(g));
  ERC_REQUIRE(N >= 1 && N < (1 << 24), "N must be in [1, 2^24)");
  ERC_REQUIRE(node_count && lambda && (g->m == 0 || (edge_count && alpha && g->csr_eid)),
              "counts and outputs are required");
  k_saint_norm<<<grid_for(g->n, ST), ST, 0, as_stream(stream)>>>(
      g->row_ptr, g->csr_eid, g->n, node_count, edge_count, N, lambda, alpha);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  return ERC_OK;
}
