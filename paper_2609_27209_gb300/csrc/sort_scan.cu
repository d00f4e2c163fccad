// sort_scan.cu -- device-wide exclusive scan (int64) for the samplers (§3.2) and the passes of a
// stable LSD radix sort of (u64 key, u32 value) pairs for the Laplacian build (§3.1.1); both are
// deterministic.
#include "erc_internal.cuh"

namespace erc {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_IPT = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_IPT;

struct LoadI64 {
  const int64_t* p;
  __device__ int64_t operator()(int64_t i) const { return p[i]; }
};
struct LoadFlag {
  const uint8_t* p;
  __device__ int64_t operator()(int64_t i) const { return (int64_t)p[i]; }
};

// block-wide exclusive scan of one value per thread; returns the exclusive prefix, *block_total
// receives the block's sum
__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* block_total) {
  __shared__ int64_t warp_tot[SCAN_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int64_t t = lane < SCAN_THREADS / 32 ? warp_tot[lane] : 0;
    int64_t ti = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t u = __shfl_up_sync(0xffffffffu, ti, o);
      if (lane >= o) ti += u;
    }
    if (lane < SCAN_THREADS / 32) warp_tot[lane] = ti - t;  // exclusive warp offsets
    if (lane == SCAN_THREADS / 32 - 1) *block_total = ti;
  }
  __syncthreads();
  int64_t r = warp_tot[warp] + inc - v;
  __syncthreads();
  return r;
}

// Single-pass exclusive scan with decoupled look-back (D. Merrill, M. Garland, "Single-pass
// Parallel Prefix Scan with Decoupled Look-back", 2016).  Tiles are claimed in order through an
// atomic ticket, so a tile only waits on tiles that have already started.  Each tile publishes
// its aggregate, then its inclusive prefix, in one 64-bit status word (value << 2 | flag, flag 1
// = aggregate, 2 = inclusive prefix); the tile's first warp walks back over its predecessors,
// 32 at a time, until it meets an inclusive prefix.  Integer sums: the result does not depend on
// the order in which tiles finish.  Inputs are non-negative and their total below 2^62.
// Every poll of a predecessor's status is bounded: after `spin_limit` polls (or once another tile
// has given up) the tile sets the call's abort word and takes the predecessor as an inclusive
// prefix of zero, so its output stays within [0, the true prefix].  A block that starts after the
// abort word is set takes no ticket and does nothing: no tile ever waits on a tile that no block
// has claimed.
template <class Load>
__global__ void __launch_bounds__(SCAN_THREADS)
    k_scan_onepass(Load in, int64_t n, unsigned long long* status, unsigned* ticket, int64_t* out,
                   int64_t* total, unsigned* abort, unsigned spin_limit) {
  __shared__ int64_t tile[SCAN_TILE];
  __shared__ unsigned s_tile;
  __shared__ int64_t s_prefix;
  if (threadIdx.x == 0) s_tile = aborted(abort) ? 0xffffffffu : atomicAdd(ticket, 1u);
  __syncthreads();
  if (s_tile == 0xffffffffu) return;
  const int64_t t = s_tile;
  const int64_t base = t * SCAN_TILE;
#pragma unroll
  for (int j = 0; j < SCAN_IPT; ++j) {
    const int j2 = j * SCAN_THREADS + threadIdx.x;
    const int64_t i = base + j2;
    tile[j2] = i < n ? in(i) : 0;
  }
  __syncthreads();
  int64_t v[SCAN_IPT];
  int64_t sum = 0;
#pragma unroll
  for (int j = 0; j < SCAN_IPT; ++j) {
    v[j] = tile[threadIdx.x * SCAN_IPT + j];
    sum += v[j];
  }
  __shared__ int64_t agg;
  const int64_t excl = block_exclusive_scan(sum, &agg);
  volatile unsigned long long* st = status;
  if (threadIdx.x < 32) {  // the first warp publishes and looks back
    const int lane = threadIdx.x;
    if (t == 0) {
      if (lane == 0) {
        st[0] = ((unsigned long long)agg << 2) | 2ull;
        s_prefix = 0;
      }
    } else {
      if (lane == 0) st[t] = ((unsigned long long)agg << 2) | 1ull;
      int64_t prefix = 0;
      int64_t j = t - 1;
      bool done = false;
      while (!done) {
        // lanes read predecessors j, j-1, ..., j-31 (those that exist)
        const int64_t q = j - lane;
        unsigned long long w = 0;
        if (q >= 0) {
          unsigned spins = 0;
          while (((w = st[q]) & 3ull) == 0ull) {
            if (++spins > spin_limit || aborted(abort)) {  // bounded: record it and take zero
              atomicOr(abort, 1u);
              w = 2ull;
              break;
            }
          }
        } else {
          w = 2ull;  // before tile 0: an inclusive prefix of 0
        }
        const unsigned incl = __ballot_sync(0xffffffffu, (w & 3ull) == 2ull);
        const int stop = incl ? __ffs(incl) - 1 : 32;  // nearest inclusive prefix
        int64_t part = lane <= stop ? (int64_t)(w >> 2) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        prefix += part;
        done = incl != 0;
        j -= 32;
      }
      if (lane == 0) {
        st[t] = ((unsigned long long)(prefix + agg) << 2) | 2ull;
        s_prefix = prefix;
      }
    }
  }
  __syncthreads();
  int64_t run = excl + s_prefix;
#pragma unroll
  for (int j = 0; j < SCAN_IPT; ++j) {
    tile[threadIdx.x * SCAN_IPT + j] = run;
    run += v[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < SCAN_IPT; ++j) {
    const int j2 = j * SCAN_THREADS + threadIdx.x;
    const int64_t i = base + j2;
    if (i < n) out[i] = tile[j2];
  }
  if (total && base + SCAN_TILE >= n && threadIdx.x == 0) *total = s_prefix + agg;
}

inline int64_t scan_blocks(int64_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE; }

// tmp: [status: ntiles u64][ticket]
template <class Load>
erc_status scan_impl(Load in, int64_t n, int64_t* out, int64_t* total, int64_t* tmp,
                     cudaStream_t s, unsigned* abort) {
  if (!abort) return set_error(ERC_ERR_INVALID_ARG, "internal: scan without an abort word");
  if (n <= 0) {
    if (total) ERC_CUDA(cudaMemsetAsync(total, 0, sizeof(int64_t), s));
    return ERC_OK;
  }
  const int64_t nb = scan_blocks(n);
  unsigned long long* status = reinterpret_cast<unsigned long long*>(tmp);
  unsigned* ticket = reinterpret_cast<unsigned*>(status + nb);
  ERC_CUDA(cudaMemsetAsync(status, 0, (size_t)nb * sizeof(unsigned long long) + 8, s));
  k_scan_onepass<<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, status, ticket, out, total, abort,
                                                       wait_limit(LOOKBACK_SPINS));
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  return ERC_OK;
}

// ------------------------------------------------------------------------------------------------
// Stable LSD radix sort of (u64 key, u32 value) pairs, one kernel per 8-bit digit (the digit counts
// of every pass come from the kernel that wrote the keys): a tile ranks its keys, publishes its
// digit counts, learns the counts of the tiles before it by decoupled look-back (as in the scan
// above, one digit per thread) and writes its keys.  What bounds a pass is HBM: 12 bytes read and
// written per pair.  The tile is therefore brought into digit order in shared memory first, so
// that a digit's keys leave as one run (16 keys, 128 bytes on average) instead of one 8-byte and
// one 4-byte store each (the three kernels per pass it replaces -- count, scan, scatter straight
// from registers -- took 3.8 ms for 131M pairs).
// A block's tile is split into warp sub-tiles in warp-striped order so that (warp, step, lane)
// order equals key order, which makes the ranks stable.
// A status word holds value << 16 | pass << 2 | flag: no pass needs its status cleared.
// ------------------------------------------------------------------------------------------------
constexpr int RS_THREADS = 256;  // one digit per thread
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_IPT = 16;
constexpr int RS_TILE = RS_THREADS * RS_IPT;
constexpr int RS_RADIX = 1 << RS_BITS;
static_assert(RS_RADIX == RS_THREADS, "one digit per thread");

struct SortShared {
  uint64_t key[RS_TILE];
  uint32_t val[RS_TILE];
  unsigned whist[RS_WARPS][RS_RADIX];
  unsigned local[RS_RADIX];  // first slot of a digit's keys in the tile
  int64_t dest[RS_RADIX];    // where the digit's keys go, less `local`
  unsigned wsum[RS_WARPS];
  unsigned tile;
};

template <bool VALS>
__global__ void __launch_bounds__(RS_THREADS)
    k_radix_pass(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                 uint64_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out, int64_t n_max,
                 const int64_t* __restrict__ n_ptr, int shift, int pass,
                 const unsigned long long* __restrict__ counts, unsigned long long* status,
                 unsigned* ticket, unsigned* abort, unsigned spin_limit) {
  extern __shared__ __align__(16) unsigned char sort_smem[];
  SortShared& sh = *reinterpret_cast<SortShared*>(sort_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) sh.tile = aborted(abort) ? 0xffffffffu : atomicAdd(ticket, 1u);
  for (int d = lane; d < RS_RADIX; d += 32) sh.whist[warp][d] = 0;
  __syncthreads();
  if (sh.tile == 0xffffffffu) return;
  const int64_t n = n_ptr ? min(n_max, *n_ptr) : n_max;
  const int64_t t = sh.tile, tile0 = t * RS_TILE;
  if (tile0 >= n) return;  // nobody waits on a tile past the end
  const int count = (int)min((int64_t)RS_TILE, n - tile0);

  // ---- keys in warp-striped order, ranked among the warp's equal digits
  const int sub = warp * 32 * RS_IPT;
  const unsigned lt_mask = (1u << lane) - 1u;
  uint64_t k[RS_IPT];
  uint32_t v[VALS ? RS_IPT : 1];
  unsigned short rank[RS_IPT];
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j) {
    const int i = sub + j * 32 + lane;
    k[j] = i < count ? keys[tile0 + i] : 0;
    if (VALS) v[j] = i < count ? vals[tile0 + i] : 0;
  }
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j) {
    const bool ok = sub + j * 32 + lane < count;
    const unsigned d = ok ? (unsigned)(k[j] >> shift) & (RS_RADIX - 1) : RS_RADIX;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const unsigned before = ok ? sh.whist[warp][d] : 0;
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) sh.whist[warp][d] = before + __popc(peers);
    __syncwarp();
    rank[j] = (unsigned short)(before + __popc(peers & lt_mask));
  }
  __syncthreads();

  // ---- digit tid: its keys in this tile, published; its first slot in the tile
  unsigned mine = 0;
#pragma unroll
  for (int w = 0; w < RS_WARPS; ++w) {
    const unsigned c = sh.whist[w][tid];
    sh.whist[w][tid] = mine;
    mine += c;
  }
  const unsigned long long tag = (unsigned long long)(pass + 1) << 2;
  volatile unsigned long long* st = status;
  st[t * RS_RADIX + tid] = (unsigned long long)mine << 16 | tag | (t == 0 ? 2ull : 1ull);
  unsigned inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  // the digit's first key over all tiles: the counts of the smaller digits
  unsigned long long base = counts[tid], binc = base;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long x = __shfl_up_sync(0xffffffffu, binc, o);
    if (lane >= o) binc += x;
  }
  __shared__ unsigned long long wbase[RS_WARPS];
  if (lane == 31) {
    sh.wsum[warp] = inc;
    wbase[warp] = binc;
  }
  __syncthreads();
  unsigned local = inc - mine;
  unsigned long long dest = binc - base;
  for (int w = 0; w < warp; ++w) {
    local += sh.wsum[w];
    dest += wbase[w];
  }
  sh.local[tid] = local;

  // ---- the keys into digit order (overlaps the wait for the tiles before)
  __syncthreads();
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j) {
    if (sub + j * 32 + lane >= count) continue;
    const unsigned d = (unsigned)(k[j] >> shift) & (RS_RADIX - 1);
    const unsigned at = sh.local[d] + sh.whist[warp][d] + rank[j];
    sh.key[at] = k[j];
    if (VALS) sh.val[at] = v[j];
  }

  // ---- digit tid in the tiles before this one, eight status words a trip
  if (t > 0) {
    unsigned long long before = 0;
    bool done = false;
    for (int64_t q = t - 1; !done; q -= 8) {
      unsigned long long w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = q - i >= 0 ? st[(q - i) * RS_RADIX + tid] : 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (done) break;
        unsigned spins = 0;
        while ((w[i] & 0xfffcull) != tag) {  // not published yet
          if (++spins > spin_limit || aborted(abort)) {  // bounded: record it and take zero
            atomicOr(abort, 1u);
            w[i] = tag | 2ull;
            break;
          }
          w[i] = st[(q - i) * RS_RADIX + tid];
        }
        before += w[i] >> 16;
        done = (w[i] & 3ull) == 2ull;  // tile 0 always is
      }
    }
    st[t * RS_RADIX + tid] = (before + mine) << 16 | tag | 2ull;
    dest += before;
  }
  sh.dest[tid] = (int64_t)dest - local;
  __syncthreads();
  for (int i = tid; i < count; i += RS_THREADS) {
    const uint64_t key = sh.key[i];
    const int64_t at = sh.dest[(unsigned)(key >> shift) & (RS_RADIX - 1)] + i;
    keys_out[at] = key;
    if (VALS) vals_out[at] = sh.val[i];
  }
}

}  // namespace

size_t scan_temp_bytes(int64_t n) {
  return (size_t)(scan_blocks(n > 0 ? n : 1) + 1) * sizeof(unsigned long long) + 256;
}

erc_status exclusive_scan_i64(const int64_t* in, const uint8_t* flags, int64_t* out, int64_t n,
                              int64_t* total, void* tmp, cudaStream_t s, unsigned* abort) {
  if (in) return scan_impl(LoadI64{in}, n, out, total, static_cast<int64_t*>(tmp), s, abort);
  return scan_impl(LoadFlag{flags}, n, out, total, static_cast<int64_t*>(tmp), s, abort);
}

inline int64_t sort_tiles(int64_t n) { return (n + RS_TILE - 1) / RS_TILE; }

// tmp: [status: tiles x RS_RADIX][tickets: RS_MAX_PASSES]
size_t radix_sort_temp_bytes(int64_t n) {
  return (size_t)sort_tiles(n > 0 ? n : 1) * RS_RADIX * sizeof(unsigned long long) +
         RS_MAX_PASSES * sizeof(unsigned);
}

erc_status radix_sort_begin(int64_t n, void* tmp, cudaStream_t s) {
  ERC_CUDA(cudaMemsetAsync(tmp, 0, radix_sort_temp_bytes(n), s));
  return ERC_OK;
}

erc_status radix_sort_open() {
  const int bytes = (int)sizeof(SortShared);
  ERC_CUDA(cudaFuncSetAttribute((const void*)k_radix_pass<true>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  ERC_CUDA(cudaFuncSetAttribute((const void*)k_radix_pass<false>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  return ERC_OK;
}

erc_status radix_sort_pass(const uint64_t* keys, const uint32_t* vals, uint64_t* keys_out,
                           uint32_t* vals_out, int64_t n_max, const int64_t* n, int shift, int pass,
                           const unsigned long long* counts, void* tmp, cudaStream_t s,
                           unsigned* abort) {
  if (n_max <= 0) return ERC_OK;
  unsigned long long* status = static_cast<unsigned long long*>(tmp);
  unsigned* tickets = reinterpret_cast<unsigned*>(status + sort_tiles(n_max) * RS_RADIX);
  const unsigned grid = (unsigned)sort_tiles(n_max);
  const unsigned limit = wait_limit(LOOKBACK_SPINS);
  if (vals)
    k_radix_pass<true><<<grid, RS_THREADS, sizeof(SortShared), s>>>(
        keys, vals, keys_out, vals_out, n_max, n, shift, pass, counts, status, tickets + pass,
        abort, limit);
  else
    k_radix_pass<false><<<grid, RS_THREADS, sizeof(SortShared), s>>>(
        keys, nullptr, keys_out, nullptr, n_max, n, shift, pass, counts, status, tickets + pass,
        abort, limit);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  return ERC_OK;
}

}  // namespace erc
