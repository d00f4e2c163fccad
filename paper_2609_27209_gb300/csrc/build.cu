// build.cu -- erc_build_laplacian: the simple undirected graph behind L = D - A = B^T W B (§3.1.1).
//
// Every input edge u != v becomes one key (min << B | max) carrying its weight; a stable radix sort
// lays the canonical pairs out in lexicographic order with duplicates adjacent and in input order,
// and one pass merges them into the numbered edge list (eu, ev, ew).  In the symmetric CSR a row's
// smaller neighbours come first: the upper slots (row u, column v > u) are the edge list itself,
// and the lower slots (row v, column u < v) are the edges in the order of (v, u), which a stable
// sort of the edge list by v gives.  With U[r] and L[r] the numbers of upper and lower slots in the
// rows before r, row_ptr[r] = U[r] + L[r]; the i-th lower slot of the whole matrix sits at U[v] + i
// and edge e's upper slot at e + L[u + 1].
//
// Sorting one key an edge (and then the edges by half a key) moves less than half the bytes of
// sorting both directions by whole keys, and every edge id is known where its slot is written: no
// search in the partner row.  What bounds each kernel is HBM, except where noted.  65.6M input
// edges, 2.45M nodes: 9.1 ms, of 43.5 ms before (both directions sorted, binary searches).
#include <algorithm>

#include "erc_internal.cuh"

namespace erc {
namespace {

constexpr int BT = 256;
constexpr int RADIX = 1 << RS_BITS;

struct BuildPlan {
  uint64_t *keys, *keys_alt;
  uint32_t *vals, *vals_alt;
  float *w, *val;                // merged weights by edge; by CSR slot when the caller wants none
  uint32_t *upper, *lower;       // [n + 1] U and L, cleared together (NO_START)
  // the next four are cleared together
  int64_t* m;                    // the number of edges
  unsigned* err;                 // [0] bit 0: node id out of range, bit 1: bad weight; [1] a merged
                                 // weight differs from 1; [2] the abort word (a wait gave up);
                                 // [3] the merge's ticket
  unsigned long long* counts;    // [RS_MAX_PASSES][RADIX] digit counts of every sort pass
  unsigned long long* status;    // look-back words of the merge, one a tile
  void* sort_tmp;
};
constexpr uint32_t NO_START = ~0u;  // a row without slots whose start is not known yet

constexpr int MERGE_IPT = 8;
constexpr int MERGE_BLOCKS = 4;  // per SM
constexpr int MERGE_TILE = BT * MERGE_IPT;

inline int bit_length(uint32_t x) { return x ? 32 - __builtin_clz(x) : 0; }
// sort passes over a whole key (two ids) and over one id
inline int key_passes(int32_t n) { return (2 * bit_length((uint32_t)n) + RS_BITS - 1) / RS_BITS; }
inline int id_passes(int32_t n) { return (bit_length((uint32_t)n) + RS_BITS - 1) / RS_BITS; }

void plan_build(Arena& a, BuildPlan& p, int32_t n, int64_t m_in) {
  p.keys = a.take<uint64_t>(m_in);
  p.keys_alt = a.take<uint64_t>(m_in);
  p.vals = a.take<uint32_t>(m_in);
  p.vals_alt = a.take<uint32_t>(m_in);
  p.w = a.take<float>(m_in);
  p.val = a.take<float>(2 * m_in);
  p.upper = a.take<uint32_t>((size_t)n + 1);
  p.lower = a.take<uint32_t>((size_t)n + 1);
  p.m = a.take<int64_t>(1);
  p.err = a.take<unsigned>(4);
  p.counts = a.take<unsigned long long>(RS_MAX_PASSES * RADIX);
  p.status = a.take<unsigned long long>((m_in + MERGE_TILE - 1) / MERGE_TILE + 1);
  p.sort_tmp = a.take<char>(radix_sort_temp_bytes(m_in));
}

__device__ __forceinline__ int64_t gtid() { return (int64_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return (int64_t)gridDim.x * blockDim.x; }

// Digit counts of the keys a block writes, for `passes` digits from bit `shift` up: four copies in
// shared memory, chosen by the lane, because the high digits of a power-law graph's ids are mostly
// equal and atomics on one word queue up.
struct DigitCounts {
  unsigned c[4][RS_MAX_PASSES / 2][RADIX];
};
__device__ __forceinline__ void counts_clear(DigitCounts& h) {
  for (int i = threadIdx.x; i < (int)(sizeof(h.c) / 4); i += blockDim.x) (&h.c[0][0][0])[i] = 0;
  __syncthreads();
}
__device__ __forceinline__ void counts_add(DigitCounts& h, uint64_t key, int shift, int passes) {
  for (int p = 0; p < passes; ++p)
    atomicAdd(&h.c[threadIdx.x & 3][p][(unsigned)(key >> (shift + p * RS_BITS)) & (RADIX - 1)], 1u);
}
__device__ __forceinline__ void counts_flush(DigitCounts& h, unsigned long long* out, int passes) {
  __syncthreads();
  for (int i = threadIdx.x; i < passes * RADIX; i += blockDim.x) {
    unsigned s = 0;
    for (int k = 0; k < 4; ++k) s += h.c[k][i / RADIX][i % RADIX];
    if (s) atomicAdd(out + i, (unsigned long long)s);
  }
}

// keys (self-loops: the sentinel, which sorts last) with their weights' bits, and the digit counts
__global__ void __launch_bounds__(BT)
    k_emit(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
           const float* __restrict__ w, int64_t m_in, int32_t n, int B, uint64_t sent, int passes,
           uint64_t* __restrict__ keys, uint32_t* __restrict__ vals,
           unsigned long long* __restrict__ counts, unsigned* __restrict__ err) {
  __shared__ DigitCounts h;
  counts_clear(h);
  unsigned bad = 0;
  for (int64_t i = gtid(); i < m_in; i += gstride()) {
    const int32_t a = src[i], b = dst[i];
    const bool range_ok = a >= 0 && a < n && b >= 0 && b < n;
    if (!range_ok) bad |= 1u;
    if (w) {
      const float x = w[i];
      if (!(x > 0.f) || !isfinite(x)) bad |= 2u;
      vals[i] = __float_as_uint(x);
    }
    uint64_t k = sent;
    if (range_ok && a != b) k = ((uint64_t)min(a, b) << B) | (uint64_t)max(a, b);
    keys[i] = k;
    counts_add(h, k, 0, passes);
  }
  if (bad) atomicOr(err, bad);
  counts_flush(h, counts, passes);
}

// The sorted keys to the edge list: a key that differs from the one before it heads a run of
// duplicates and becomes the next edge, in one pass with decoupled look-back over the tiles' head
// counts (as in the scan; a word is count << 2 | flag).  The head's thread merges its run: the
// float64 sum of the duplicates' weights in input order (the sort is stable), rounded once.  Also
// written: U of the rows that have upper slots, the edges as keys (v << B | u) for the sort by v,
// and that sort's digit counts.
__global__ void __launch_bounds__(BT, MERGE_BLOCKS)
    k_merge(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ wbits, int64_t m_in,
            int32_t n, int B, uint64_t sent, int dup_first, int vpasses, int32_t* __restrict__ eu,
            int32_t* __restrict__ ev, float* __restrict__ ew, float* __restrict__ wout,
            uint64_t* __restrict__ vkeys, uint32_t* __restrict__ vvals,
            uint32_t* __restrict__ upper, unsigned long long* __restrict__ counts,
            unsigned long long* status, int64_t* __restrict__ m_out, unsigned* __restrict__ err,
            unsigned spin_limit) {
  __shared__ DigitCounts h;
  __shared__ unsigned s_off[MERGE_IPT][BT / 32];  // heads of each 32 keys, then their prefix
  __shared__ unsigned s_tile, s_total;
  __shared__ unsigned long long s_prefix;
  unsigned* abort = err + 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  counts_clear(h);
  for (;;) {
    if (threadIdx.x == 0) s_tile = aborted(abort) ? 0xffffffffu : atomicAdd(err + 3, 1u);
    __syncthreads();
    const int64_t t = s_tile, base = t * MERGE_TILE;
    if (s_tile == 0xffffffffu || base >= m_in) break;
    uint64_t k[MERGE_IPT], before[MERGE_IPT];
    unsigned heads[MERGE_IPT];
#pragma unroll
    for (int j = 0; j < MERGE_IPT; ++j) {
      const int64_t i = base + j * BT + threadIdx.x;
      k[j] = i < m_in ? keys[i] : sent;
      before[j] = i > 0 && i < m_in ? keys[i - 1] : sent;  // no key before the first
    }
#pragma unroll
    for (int j = 0; j < MERGE_IPT; ++j) {
      heads[j] = __ballot_sync(0xffffffffu, k[j] != sent && k[j] != before[j]);
      if (lane == 0) s_off[j][warp] = __popc(heads[j]);
    }
    __syncthreads();
    if (warp == 0) {
      // 64 counts in key order (j, warp): two a lane
      static_assert(MERGE_IPT * (BT / 32) == 64, "two counts a lane");
      unsigned* c = &s_off[0][0];
      const unsigned a = c[2 * lane], b = c[2 * lane + 1];
      unsigned inc = a + b;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
      }
      c[2 * lane] = inc - a - b;
      c[2 * lane + 1] = inc - b;
      const unsigned total = __shfl_sync(0xffffffffu, inc, 31);
      const unsigned long long prefix = tile_prefix(status, t, total, spin_limit, abort);
      if (lane == 0) {
        s_total = total;
        s_prefix = prefix;
      }
    }
    __syncthreads();
    const uint64_t mask = (1ull << B) - 1ull;
    bool other = false;
#pragma unroll
    for (int j = 0; j < MERGE_IPT; ++j) {
      if (!((heads[j] >> lane) & 1u)) continue;
      const int64_t i = base + j * BT + threadIdx.x;
      const uint32_t e =
          (uint32_t)s_prefix + s_off[j][warp] + __popc(heads[j] & ((1u << lane) - 1u));
      float merged = wbits ? __uint_as_float(wbits[i]) : 1.f;
      if (!dup_first && i + 1 < m_in && keys[i + 1] == k[j]) {  // float64 only where a run is
        double acc = (double)merged;
        for (int64_t d = i + 1; d < m_in && keys[d] == k[j]; ++d)
          acc += wbits ? (double)__uint_as_float(wbits[d]) : 1.0;
        merged = (float)acc;
      }
      const int32_t u = (int32_t)(k[j] >> B), v = (int32_t)(k[j] & mask);
      eu[e] = u;
      ev[e] = v;
      wout[e] = merged;
      if (ew) ew[e] = merged;
      other |= merged != 1.f;
      const uint64_t vk = ((uint64_t)v << B) | (uint64_t)u;
      vkeys[e] = vk;
      vvals[e] = e;
      counts_add(h, vk, B, vpasses);
      // row u starts here unless the key before lies in it
      if (before[j] == sent || (int32_t)(before[j] >> B) != u) upper[u] = e;
    }
    if (!wbits && __any_sync(0xffffffffu, other) && lane == 0) atomicOr(err + 1, 1u);
    if (base + MERGE_TILE >= m_in && threadIdx.x == 0) *m_out = (int64_t)(s_prefix + s_total);
    __syncthreads();
  }
  counts_flush(h, counts, vpasses);
}

// The starts of the rows without slots in a list of m slots sorted by row: the first slot of a
// later row, by binary search, a thread a row.  The searches of neighbouring rows take the same
// steps, so a warp's loads are one line each and mostly in L1; a serial fill by the thread of the
// next slot's row lasts as long as the longest run of such rows.  1M users with the smaller ids,
// 0.1M items, 3M edges: a build of 0.73 ms (4.06 with the serial fill, 3.3 of them in one thread);
// 10M nodes, 0.1M edges: 1.11 ms (1.93); 2.45M nodes, 64.3M edges, few such rows: 9.1 ms either
// way.
struct RowOfEdge {
  const int32_t* eu;
  __device__ int32_t operator()(uint32_t i) const { return __ldg(eu + i); }
};
struct RowOfKey {
  const uint64_t* key;
  int B;
  __device__ int32_t operator()(uint32_t i) const { return (int32_t)(__ldg(key + i) >> B); }
};
template <class RowOf>
__global__ void __launch_bounds__(BT)
    k_fill_starts(RowOf row_of, const int64_t* __restrict__ m_ptr, int32_t n,
                  uint32_t* __restrict__ start, const unsigned* abort) {
  if (aborted(abort)) return;
  const uint32_t m = (uint32_t)*m_ptr;
  for (int64_t r = gtid(); r <= n; r += gstride()) {
    if (start[r] != NO_START) continue;
    uint32_t lo = 0, hi = m;  // m <= 2^30: their sum fits
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (row_of(mid) < r) lo = mid + 1; else hi = mid;
    }
    start[r] = lo;
  }
}

// lower slots, in the order of (v, u): slot i sits at U[v] + i.  Also L of the rows that have some.
__global__ void __launch_bounds__(BT)
    k_lower(const uint64_t* __restrict__ vkeys, const uint32_t* __restrict__ vvals,
            const float* __restrict__ w, const uint32_t* __restrict__ upper,
            const int64_t* __restrict__ m_ptr, int B, int32_t* __restrict__ col,
            int32_t* __restrict__ csr_eid, float* __restrict__ val, uint32_t* __restrict__ lower,
            const unsigned* abort) {
  if (aborted(abort)) return;
  const int64_t m = *m_ptr;
  const uint64_t mask = (1ull << B) - 1ull;
  for (int64_t i = gtid(); i < m; i += gstride()) {
    const uint64_t k = vkeys[i];
    const uint32_t e = vvals[i];
    const int32_t v = (int32_t)(k >> B);
    const int64_t at = (int64_t)upper[v] + i;
    col[at] = (int32_t)(k & mask);
    csr_eid[at] = (int32_t)e;
    val[at] = w[e];
    if (i == 0 || (int32_t)(vkeys[i - 1] >> B) != v) lower[v] = (uint32_t)i;
  }
}

// upper slots: edge e sits at e + L[u + 1].  Also row_ptr.
__global__ void __launch_bounds__(BT)
    k_upper(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
            const float* __restrict__ w, const uint32_t* __restrict__ upper,
            const uint32_t* __restrict__ lower, const int64_t* __restrict__ m_ptr, int32_t n,
            int32_t* __restrict__ col, int32_t* __restrict__ csr_eid, float* __restrict__ val,
            int64_t* __restrict__ row_ptr, const unsigned* abort) {
  if (aborted(abort)) return;
  const int64_t m = *m_ptr;
  for (int64_t e = gtid(); e < m; e += gstride()) {
    const int64_t at = e + (int64_t)lower[eu[e] + 1];
    col[at] = ev[e];
    csr_eid[at] = (int32_t)e;
    val[at] = w[e];
  }
  for (int64_t r = gtid(); r <= n; r += gstride())
    row_ptr[r] = (int64_t)upper[r] + (int64_t)lower[r];
}

// A running sum in three float32 words, each addition's error carried to the next word exactly: at
// least 70 bits, where float64 has 53.  GB300 adds float64 at a sixty-fourth of the float32 rate,
// and the conversions run there too; three words take 13 float32 operations an addend.  The addends
// are positive: once the sum passes the largest float the first word stays infinite, and so is the
// sum (the other words then hold differences of infinities).
struct Sum3 {
  float a = 0.f, b = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float2 s = df_two_sum(a, x);
    const float2 t = df_two_sum(b, s.y);
    a = s.x;
    b = t.x;
    c = __fadd_rn(c, t.y);
  }
  __device__ __forceinline__ double value() const {
    return isinf(a) ? (double)a : (double)a + ((double)b + (double)c);
  }
};

// A row's weights summed to at least float64's precision, rounded once.  Eight lanes a row; a
// warp's rows of more than 256 neighbours are taken by the whole warp, one after another, so that a
// hub does not hold up its warp at eight lanes.  2.45M nodes, 64.3M edges: 367 us; 862 us with
// float64 sums, 5.4 ms with one thread a row.
constexpr int DL = 8;
__global__ void __launch_bounds__(BT)
    k_degree(const int64_t* __restrict__ row_ptr, const float* __restrict__ val, int32_t n,
             float* __restrict__ deg, const unsigned* abort) {
  if (aborted(abort)) return;
  const int lane = threadIdx.x & 31, gl = lane & (DL - 1);
  const int64_t r = gtid() / DL;
  const int64_t j0 = r < n ? row_ptr[r] : 0, j1 = r < n ? row_ptr[r + 1] : 0;
  const bool is_long = j1 - j0 > 256;
  Sum3 sum;
  if (!is_long)
#pragma unroll 4
    for (int64_t j = j0 + gl; j < j1; j += DL) sum.add(__ldg(val + j));
  double acc = sum.value();
#pragma unroll
  for (int o = DL / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  for (unsigned todo = __ballot_sync(0xffffffffu, is_long && gl == 0); todo; todo &= todo - 1) {
    const int owner = __ffs(todo) - 1;
    const int64_t a = __shfl_sync(0xffffffffu, j0, owner), b = __shfl_sync(0xffffffffu, j1, owner);
    Sum3 part;
#pragma unroll 4
    for (int64_t j = a + lane; j < b; j += 32) part.add(__ldg(val + j));
    double all = part.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
    if (lane == owner) acc = all;
  }
  if (gl == 0 && r < n) deg[r] = (float)acc;
}

}  // namespace
}  // namespace erc

using namespace erc;

extern "C" size_t erc_build_laplacian_workspace_size(int32_t n, int64_t m_in) {
  if (m_in < 0 || n < 0) return 0;
  Arena a(nullptr);
  BuildPlan p;
  plan_build(a, p, n, m_in);
  return a.used + 256;
}

erc_status erc::build_laplacian_impl(int32_t n, const int32_t* src, const int32_t* dst,
                                     const float* w, int64_t m_in, int32_t dup_policy,
                                     int64_t* row_ptr, int32_t* col, float* val, float* deg,
                                     int32_t* csr_eid, int32_t* eu, int32_t* ev, float* ew,
                                     int64_t* m_out, void* ws, size_t ws_bytes, cudaStream_t s,
                                     int* nonunit) {
  ERC_REQUIRE(n >= 1, "n must be >= 1 (got %d)", n);
  ERC_REQUIRE(m_in >= 0 && m_in <= (int64_t(1) << 30), "m_in out of range (%lld)",
              (long long)m_in);
  ERC_REQUIRE(dup_policy == ERC_DUP_SUM || dup_policy == ERC_DUP_FIRST, "bad dup_policy %d",
              dup_policy);
  ERC_REQUIRE(row_ptr && deg && m_out, "row_ptr, deg and m_out are required");
  ERC_REQUIRE(m_in == 0 || (src && dst && col && csr_eid && eu && ev),
              "src, dst, col, csr_eid, eu, ev are required");
  ERC_REQUIRE(!(w && !val && m_in > 0), "val is required for a weighted graph");
  if (ws_bytes < erc_build_laplacian_workspace_size(n, m_in))
    return set_error(ERC_ERR_CAPACITY, "workspace too small: %zu < %zu", ws_bytes,
                     erc_build_laplacian_workspace_size(n, m_in));
  Arena a(reinterpret_cast<void*>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255)));
  BuildPlan p;
  plan_build(a, p, n, m_in);

  // the launch sequence is replayed from a cached CUDA graph: a dozen or so kernels whose launch
  // overhead would otherwise exceed the run time of the small ones
  const int B = bit_length((uint32_t)n);  // 2^B > n - 1: every id fits, and the sentinel sorts last
  const uint64_t sent = (2 * B >= 64) ? ~0ull : ((1ull << (2 * B)) - 1ull);
  const int passes = key_passes(n), vpasses = id_passes(n);
  unsigned* abort = p.err + 2;
  float* cval = val ? val : p.val;
  const int64_t tiles = (m_in + MERGE_TILE - 1) / MERGE_TILE;
  auto bytes_between = [](const void* from, const void* to) {
    return (size_t)(static_cast<const char*>(to) - static_cast<const char*>(from));
  };
  auto enqueue = [&](cudaStream_t cs) -> erc_status {
    ERC_CUDA(cudaMemsetAsync(p.m, 0, bytes_between(p.m, p.status + tiles), cs));
    if (m_in > 0) {
      ERC_CUDA(cudaMemsetAsync(p.upper, 0xff, bytes_between(p.upper, p.lower + n + 1), cs));
      ERC_TRY(radix_sort_begin(m_in, p.sort_tmp, cs));
      // blocks that count digits: few enough that their flushes do not queue at the 256 counters
      k_emit<<<grid_for(m_in, BT, 4), BT, 0, cs>>>(src, dst, w, m_in, n, B, sent, passes, p.keys,
                                                   p.vals, p.counts, p.err);
      count_launches(1);
      ERC_CUDA(cudaGetLastError());
      uint64_t *ka = p.keys, *kb = p.keys_alt;
      uint32_t *va = w ? p.vals : nullptr, *vb = w ? p.vals_alt : nullptr;
      int pass = 0;
      for (int i = 0; i < passes; ++i, ++pass) {
        ERC_TRY(radix_sort_pass(ka, va, kb, vb, m_in, nullptr, i * RS_BITS, pass,
                                p.counts + pass * RADIX, p.sort_tmp, cs, abort));
        std::swap(ka, kb);
        std::swap(va, vb);
      }
      unsigned long long* vcounts = p.counts + pass * RADIX;
      // blocks that take tiles until none is left, so that their digit counts are flushed once
      k_merge<<<(unsigned)std::min<int64_t>(tiles, MERGE_BLOCKS * sm_count()), BT, 0, cs>>>(
          ka, va, m_in, n, B, sent, dup_policy == ERC_DUP_FIRST, vpasses, eu, ev, ew, p.w, kb,
          vb ? vb : p.vals_alt, p.upper, vcounts, p.status, p.m, p.err, wait_limit(LOOKBACK_SPINS));
      count_launches(1);
      ERC_CUDA(cudaGetLastError());
      k_fill_starts<<<grid_for(n + 1LL, BT), BT, 0, cs>>>(RowOfEdge{eu}, p.m, n, p.upper, abort);
      count_launches(1);
      ERC_CUDA(cudaGetLastError());
      uint64_t *sa = kb, *sb = ka;
      uint32_t *ta = vb ? vb : p.vals_alt, *tb = va ? va : p.vals;
      for (int i = 0; i < vpasses; ++i, ++pass) {
        ERC_TRY(radix_sort_pass(sa, ta, sb, tb, m_in, p.m, B + i * RS_BITS, pass,
                                p.counts + pass * RADIX, p.sort_tmp, cs, abort));
        std::swap(sa, sb);
        std::swap(ta, tb);
      }
      k_lower<<<grid_for(m_in, BT), BT, 0, cs>>>(sa, ta, p.w, p.upper, p.m, B, col, csr_eid, cval,
                                                 p.lower, abort);
      count_launches(1);
      ERC_CUDA(cudaGetLastError());
      k_fill_starts<<<grid_for(n + 1LL, BT), BT, 0, cs>>>(RowOfKey{sa, B}, p.m, n, p.lower, abort);
      count_launches(1);
      ERC_CUDA(cudaGetLastError());
      k_upper<<<grid_for(std::max<int64_t>(m_in, n + 1LL), BT), BT, 0, cs>>>(
          eu, ev, p.w, p.upper, p.lower, p.m, n, col, csr_eid, cval, row_ptr, abort);
      count_launches(1);
      ERC_CUDA(cudaGetLastError());
    } else {
      ERC_CUDA(cudaMemsetAsync(row_ptr, 0, (size_t)(n + 1) * sizeof(int64_t), cs));
    }
    k_degree<<<(unsigned)(((int64_t)n * DL + BT - 1) / BT), BT, 0, cs>>>(row_ptr, cval, n, deg,
                                                                         abort);
    count_launches(1);
    ERC_CUDA(cudaGetLastError());
    return ERC_OK;
  };
  GraphKey key;
  key.add((uint64_t)n).add((uint64_t)m_in).add((uint64_t)dup_policy).add(src).add(dst).add(w);
  key.add(row_ptr).add(col).add(val).add(deg).add(csr_eid).add(eu).add(ev).add(ew).add(a.base);
  key.add((uint64_t)wait_limit(0));
  ERC_TRY(graph_launch(key, enqueue, s));
  int64_t h_m = 0;
  unsigned h_err[3] = {0, 0, 0};
  ERC_CUDA(cudaMemcpyAsync(&h_m, p.m, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  ERC_CUDA(cudaMemcpyAsync(h_err, p.err, 3 * sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  ERC_CUDA(cudaStreamSynchronize(s));
  if (h_err[2])
    return set_error(ERC_ERR_TIMEOUT, "a bounded wait in the Laplacian build's scans ran out; "
                                      "the outputs are undefined");
  if (h_err[0] & 1u) return set_error(ERC_ERR_INVALID_ARG, "node id outside [0, %d)", n);
  if (h_err[0] & 2u) return set_error(ERC_ERR_INVALID_ARG, "edge weight not finite and positive");
  *m_out = h_m;
  if (nonunit) *nonunit = w ? 1 : (int)h_err[1];
  return ERC_OK;
}
extern "C" erc_status erc_build_laplacian(int32_t n, const int32_t* src, const int32_t* dst,
                                          const float* w, int64_t m_in, int32_t dup_policy,
                                          int64_t* row_ptr, int32_t* col, float* val, float* deg,
                                          int32_t* csr_eid, int32_t* eu, int32_t* ev, float* ew,
                                          int64_t* m_out, void* ws, size_t ws_bytes,
                                          erc_stream stream) {
  clear_error();
  return build_laplacian_impl(n, src, dst, w, m_in, dup_policy, row_ptr, col, val, deg, csr_eid,
                              eu, ev, ew, m_out, ws, ws_bytes, as_stream(stream), nullptr);
}

extern "C" erc_status erc_build_laplacian_ex(int32_t n, const int32_t* src, const int32_t* dst,
                                             const float* w, int64_t m_in, int32_t dup_policy,
                                             int64_t* row_ptr, int32_t* col, float* val,
                                             float* deg, int32_t* csr_eid, int32_t* eu,
                                             int32_t* ev, float* ew, int64_t* m_out,
                                             int32_t* unit_weights, void* ws, size_t ws_bytes,
                                             erc_stream stream) {
  clear_error();
  ERC_REQUIRE(unit_weights, "unit_weights is required");
  int nonunit = 1;
  ERC_TRY(build_laplacian_impl(n, src, dst, w, m_in, dup_policy, row_ptr, col, val, deg, csr_eid,
                               eu, ev, ew, m_out, ws, ws_bytes, as_stream(stream), &nonunit));
  *unit_weights = nonunit ? 0 : 1;
  return ERC_OK;
}
