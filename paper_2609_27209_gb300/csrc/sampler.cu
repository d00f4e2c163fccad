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
// draws and the subgraph's counts: 182 us, 233 us before; 64.3M edges, 6.4M draws: 2.24 ms, 3.96 ms
// before, with separate passes for weights, draws, marks, induced flags, scans and compactions and
// two round trips.
#include "erc_internal.cuh"

namespace erc {
namespace {

constexpr int ST = 256;
constexpr int SWARPS = ST / 32;
constexpr int SIPT = 32;               // entries per thread of a scan or compaction tile: few tiles, so
constexpr int STILE = ST * SIPT;       // that the look-back over those in flight stays short
constexpr uint32_t SAMPLER_TAG = 0x53414D50u;

struct SamplePlan {
  int64_t *E, *totals;  // totals: [0] T [1] nodes [2] edges
  uint8_t *nmark, *emark;
  unsigned long long* status;  // look-back words of the three passes
  unsigned* err;  // [0] a probability outside [0, 1]; [1] the abort word; [2..4] the passes' tickets
};

inline int64_t stiles(int64_t count) { return (count + STILE - 1) / STILE; }

void plan_sample(Arena& a, SamplePlan& p, int64_t count, int32_t n, int64_t m) {
  p.E = a.take<int64_t>(count);
  p.nmark = a.take<uint8_t>(n);
  p.emark = a.take<uint8_t>(m > 0 ? m : 1);
  p.totals = a.take<int64_t>(4);
  p.err = a.take<unsigned>(8);
  p.status = a.take<unsigned long long>(stiles(count) + stiles(n) + stiles(m) + 1);
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

// the block's tile of a pass, or -1 once a wait of the call has given up
__device__ __forceinline__ int64_t claim_tile(unsigned* ticket, const unsigned* abort) {
  __shared__ unsigned s_tile;
  if (threadIdx.x == 0) s_tile = aborted(abort) ? 0xffffffffu : atomicAdd(ticket, 1u);
  __syncthreads();
  return s_tile == 0xffffffffu ? -1 : (int64_t)s_tile;
}

// E and T of the weights.  A warp takes 32 SIPT consecutive entries, 32 at a time.
__global__ void __launch_bounds__(ST)
    k_weight_scan(const float* __restrict__ prob, int64_t count, int64_t* __restrict__ E,
                  int64_t* __restrict__ total, unsigned long long* status, unsigned* err,
                  unsigned spin_limit) {
  __shared__ unsigned long long s_warp[SWARPS], s_prefix, s_total;
  const int64_t t = claim_tile(err + 2, err + 1);
  if (t < 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t base = t * STILE + (int64_t)warp * 32 * SIPT + lane;
  float p[SIPT];
#pragma unroll
  for (int j = 0; j < SIPT; ++j) p[j] = base + 32 * j < count ? prob[base + 32 * j] : 0.f;
  bool bad = false;
  unsigned long long sum = 0;
#pragma unroll
  for (int j = 0; j < SIPT; ++j) sum += fixed_weight(p[j], bad);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s_warp[warp] = sum;
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, 1u);
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
    const unsigned long long prefix = tile_prefix(status, t, tot, spin_limit, err + 1);
    if (lane == 0) {
      s_prefix = prefix;
      s_total = prefix + tot;
    }
  }
  __syncthreads();
  unsigned long long run = s_prefix + s_warp[warp];
#pragma unroll
  for (int j = 0; j < SIPT; ++j) {
    const unsigned long long w = fixed_weight(p[j], bad);
    unsigned long long inc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (base + 32 * j < count) E[base + 32 * j] = (int64_t)(run + inc - w);
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  if ((t + 1) * STILE >= count && threadIdx.x == 0) *total = (int64_t)s_total;
}

// draw k: the largest i with E_i <= floor(x_k T / 2^64); marks node i, or edge i's endpoints and,
// where emark is not null, the edge.  A mark is tested first: most draws of a power-law graph's
// endpoints find theirs set, and a cached read is cheaper than a byte store.
__global__ void __launch_bounds__(ST)
    k_draw(const int64_t* __restrict__ E, int64_t count, const int64_t* __restrict__ tot,
           int64_t budget, uint2 key, int64_t first, uint32_t stream,
           const int32_t* __restrict__ eu, const int32_t* __restrict__ ev, uint8_t* nmark,
           uint8_t* emark, const unsigned* abort) {
  if (aborted(abort)) return;
  const uint64_t T = (uint64_t)tot[0];
  for (int64_t k = (int64_t)blockIdx.x * ST + threadIdx.x; k < budget;
       k += (int64_t)gridDim.x * ST) {
    const uint64_t d = (uint64_t)(first + k);
    const uint4 w =
        philox4x32_10(make_uint4((uint32_t)d, (uint32_t)(d >> 32), SAMPLER_TAG, stream), key);
    const uint64_t x = ((uint64_t)w.x << 32) | w.y;
    const int64_t r = (int64_t)__umul64hi(x, T);
    int64_t lo = 0, hi = count;  // first index with E > r, minus one
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (E[mid] <= r) lo = mid + 1; else hi = mid;
    }
    const int64_t i = lo - 1;
    if (stream) {
      if (emark) emark[i] = 1;
      const int32_t u = eu[i], v = ev[i];
      if (!__ldcg(nmark + u)) nmark[u] = 1;
      if (!__ldcg(nmark + v)) nmark[v] = 1;
    } else {
      if (!__ldcg(nmark + i)) nmark[i] = 1;
    }
  }
}

struct MarkedFlag {
  const uint8_t* mark;
  __device__ bool operator()(int64_t i) const { return mark[i] != 0; }
};
struct InducedFlag {  // both endpoints of edge i are marked
  const int32_t *eu, *ev;
  const uint8_t* nmark;
  __device__ bool operator()(int64_t i) const {
    return __ldg(nmark + eu[i]) & __ldg(nmark + ev[i]);
  }
};

// the ids i < count with flag(i), ascending
template <class Flag>
__global__ void __launch_bounds__(ST)
    k_compact(Flag flag, int64_t count, int32_t* __restrict__ out, int64_t* __restrict__ total,
              unsigned long long* status, unsigned* ticket, unsigned* abort, unsigned spin_limit) {
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
  static_assert(SIPT == 32, "a lane holds one ballot");
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

}  // namespace
}  // namespace erc

using namespace erc;

extern "C" size_t erc_sample_workspace_size(int32_t n, int64_t m, int64_t budget) {
  if (n < 1 || m < 0 || budget < 0) return 0;
  Arena a(nullptr);
  SamplePlan p;
  plan_sample(a, p, n > m ? n : m, n, m);
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
  plan_sample(ar, p, g->n > g->m ? g->n : g->m, g->n, g->m);
  *n_out = 0;
  *m_out = 0;
  if (count == 0 || budget == 0) return ERC_OK;
  const bool drawn_edges = by_edge && !induced;  // the subgraph keeps the drawn edges alone
  unsigned* abort = p.err + 1;
  unsigned long long* st_n = p.status + stiles(count);
  unsigned long long* st_m = st_n + stiles(g->n);
  ERC_CUDA(cudaMemsetAsync(p.err, 0, 8 * sizeof(unsigned), s));
  ERC_CUDA(cudaMemsetAsync(p.status, 0,
                           (size_t)(stiles(count) + stiles(g->n) + stiles(g->m)) *
                               sizeof(unsigned long long), s));
  ERC_CUDA(cudaMemsetAsync(p.nmark, 0, (size_t)g->n, s));
  if (drawn_edges) ERC_CUDA(cudaMemsetAsync(p.emark, 0, (size_t)g->m, s));
  // Nothing is read back before the end: a probability outside [0, 1] counts as zero, with a total of
  // zero every draw is the last index, and the prefixes are only ever below their true values when
  // a bounded wait gives up, so every index stays in range; the host then reports the error.
  const unsigned limit = wait_limit(LOOKBACK_SPINS);
  k_weight_scan<<<(unsigned)stiles(count), ST, 0, s>>>(prob, count, p.E, &p.totals[0], p.status,
                                                       p.err, limit);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  const uint2 key = make_uint2((uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
  k_draw<<<grid_for(budget, ST), ST, 0, s>>>(p.E, count, p.totals, budget, key, first_draw,
                                             by_edge ? 1u : 0u, g->eu, g->ev, p.nmark,
                                             drawn_edges ? p.emark : nullptr, abort);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  k_compact<<<(unsigned)stiles(g->n), ST, 0, s>>>(MarkedFlag{p.nmark}, (int64_t)g->n, nodes,
                                                  &p.totals[1], st_n, p.err + 3, abort, limit);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  if (g->m > 0) {
    if (drawn_edges)
      k_compact<<<(unsigned)stiles(g->m), ST, 0, s>>>(MarkedFlag{p.emark}, g->m, edges,
                                                      &p.totals[2], st_m, p.err + 4, abort, limit);
    else
      k_compact<<<(unsigned)stiles(g->m), ST, 0, s>>>(InducedFlag{g->eu, g->ev, p.nmark}, g->m,
                                                      edges, &p.totals[2], st_m, p.err + 4, abort,
                                                      limit);
    count_launches(1);
    ERC_CUDA(cudaGetLastError());
  }
  int64_t h_tot[3] = {0, 0, 0};
  unsigned h_err[2] = {0, 0};
  ERC_CUDA(cudaMemcpyAsync(h_tot, p.totals, 3 * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  ERC_CUDA(cudaMemcpyAsync(h_err, p.err, 2 * sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  ERC_CUDA(cudaStreamSynchronize(s));
  if (h_err[0]) return set_error(ERC_ERR_INVALID_ARG, "probabilities must lie in [0, 1]");
  if (h_err[1]) return set_error(ERC_ERR_TIMEOUT, "a bounded wait in the sampler's scans ran out");
  if (h_tot[0] == 0) return set_error(ERC_ERR_INVALID_ARG, "every probability rounds to zero");
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
