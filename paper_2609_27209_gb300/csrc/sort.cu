// sort.cu -- the passes of a stable, deterministic LSD radix sort of (u64 key, u32 value) pairs for
// the Laplacian build (§3.1.1).
#include <algorithm>

#include "erc_internal.cuh"

namespace erc {

namespace {

// ------------------------------------------------------------------------------------------------
// Stable LSD radix sort of (u64 key, u32 value) pairs, one kernel per 8-bit digit, the method of
// A. Adinets, D. Merrill, "Onesweep: A Faster Least Significant Digit Radix Sort for GPUs", 2022
// (the digit counts of every pass come from the kernel that wrote the keys): a tile ranks its keys,
// publishes its digit counts, learns the counts of the tiles before it by decoupled look-back (as
// tile_prefix, one digit per thread) and writes its keys.  HBM would bound a pass at 0.23 ms for
// 65.6M pairs (12 bytes read and written each); the chain of a tile's phases makes it 0.62 ms, so
// as many tiles as fit overlap on an SM.  The tile is brought into digit order in shared memory
// first, so that a digit's keys leave as one run (10 keys, 80 bytes on average) instead of one
// 8-byte and one 4-byte store each (the three kernels per pass it replaces -- count, scan, scatter
// straight from registers -- took 3.8 ms for 131M pairs).  A block's tile is split into warp
// sub-tiles in warp-striped order so that (warp, step, lane) order equals key order, which makes
// the ranks stable.  A status word holds count << 16 | pass << 2 | flag (1 the tile's count, 2 with
// all tiles before): no pass needs its status cleared.  Keys and values take turns in the shared
// buffer.
constexpr int RS_THREADS = 256;  // one digit per thread
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_RADIX = 1 << RS_BITS;
static_assert(RS_RADIX == RS_THREADS, "one digit per thread");
constexpr int LB = 8;
// Tiles of 256 x 10 keys, which leave four blocks an SM their registers (65.6M edges: 9.1 ms a
// build; 12 keys a thread 10.1 with spills or 10.6 with three blocks, 16 keys 10.6); below RS_SMALL
// keys 256 x 8, so that a small graph's passes spread over more SMs (2,000-node run: 22 us less
// than with 16).
constexpr int64_t RS_SMALL = 2 << 20;

template <int IPT>
struct SortShared {
  uint64_t key[RS_THREADS * IPT];  // the tile's keys in digit order, then its values
  unsigned whist[RS_WARPS][RS_RADIX];
  unsigned local[RS_RADIX];  // first slot of a digit's keys in the tile
  uint32_t dest[RS_RADIX];   // where the digit's keys go, less `local` (modulo 2^32)
  unsigned wsum[RS_WARPS], wbase[RS_WARPS];
  unsigned tile;
};

template <int RS_IPT, bool VALS>
__global__ void __launch_bounds__(RS_THREADS, 4)
    k_radix_pass(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                 uint64_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out, int64_t n_max,
                 const int64_t* __restrict__ n_ptr, int shift, int pass,
                 const unsigned long long* __restrict__ counts, unsigned long long* status,
                 unsigned* ticket, unsigned* abort, unsigned spin_limit) {
  constexpr int RS_TILE = RS_THREADS * RS_IPT;
  __shared__ SortShared<RS_IPT> sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) sh.tile = aborted(abort) ? 0xffffffffu : atomicAdd(ticket, 1u);
  for (int d = lane; d < RS_RADIX; d += 32) sh.whist[warp][d] = 0;
  __syncthreads();
  if (sh.tile == 0xffffffffu) return;
  const int64_t n = n_ptr ? min(n_max, *n_ptr) : n_max;
  const int64_t t = sh.tile, tile0 = t * RS_TILE;
  if (tile0 >= n) return;  // nobody waits on a tile past the end
  const int count = (int)min((int64_t)RS_TILE, n - tile0);

  // ---- keys in warp-striped order, ranked among the warp's equal digits: the first lane of each
  // group of peers counts the group in; the counts come back in a second loop, so that the steps'
  // latencies overlap
  const int sub = warp * 32 * RS_IPT;
  const unsigned lt_mask = (1u << lane) - 1u;
  uint64_t k[RS_IPT];
  unsigned rank[RS_IPT];  // leading lane << 16 | peers before this lane
  unsigned before[RS_IPT];
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j) {
    const int i = sub + j * 32 + lane;
    k[j] = i < count ? keys[tile0 + i] : 0;
  }
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j) {
    const bool ok = sub + j * 32 + lane < count;
    const unsigned d = ok ? (unsigned)(k[j] >> shift) & (RS_RADIX - 1) : RS_RADIX;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int lead = __ffs(peers) - 1;
    before[j] = ok && lane == lead ? atomicAdd(&sh.whist[warp][d], (unsigned)__popc(peers)) : 0u;
    rank[j] = (unsigned)lead << 16 | (unsigned)__popc(peers & lt_mask);
    __syncwarp();  // the next step's counts come after this one's
  }
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j)
    rank[j] = __shfl_sync(0xffffffffu, before[j], (int)(rank[j] >> 16)) + (rank[j] & 0xffffu);
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
  // the digit's first key over all tiles: the counts of the smaller digits
  const unsigned base = (unsigned)counts[tid];
  unsigned inc = mine, binc = base;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
    const unsigned y = __shfl_up_sync(0xffffffffu, binc, o);
    if (lane >= o) {
      inc += x;
      binc += y;
    }
  }
  if (lane == 31) {
    sh.wsum[warp] = inc;
    sh.wbase[warp] = binc;
  }
  __syncthreads();
  unsigned local = inc - mine, dest = binc - base;
  for (int w = 0; w < warp; ++w) {
    local += sh.wsum[w];
    dest += sh.wbase[w];
  }
  sh.local[tid] = local;

  // ---- the keys into digit order (overlaps the wait for the tiles before)
  __syncthreads();
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j) {
    if (sub + j * 32 + lane >= count) continue;
    const unsigned d = (unsigned)(k[j] >> shift) & (RS_RADIX - 1);
    rank[j] += sh.local[d] + sh.whist[warp][d];  // the key's slot
    sh.key[rank[j]] = k[j];
  }
  uint32_t v[VALS ? RS_IPT : 1];
  if (VALS)
#pragma unroll
    for (int j = 0; j < RS_IPT; ++j) {
      const int i = sub + j * 32 + lane;
      v[j] = i < count ? vals[tile0 + i] : 0;
    }

  // ---- digit tid in the tiles before this one, LB status words a trip
  if (t > 0) {
    unsigned long long sum = 0;
    bool done = false;
    for (int64_t q = t - 1; !done; q -= LB) {
      unsigned long long w[LB];
#pragma unroll
      for (int i = 0; i < LB; ++i) w[i] = q - i >= 0 ? st[(q - i) * RS_RADIX + tid] : 0;
#pragma unroll
      for (int i = 0; i < LB; ++i) {
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
        sum += w[i] >> 16;
        done = (w[i] & 3ull) == 2ull;  // tile 0 always is
      }
    }
    st[t * RS_RADIX + tid] = (sum + mine) << 16 | tag | 2ull;
    dest += (unsigned)sum;
  }
  sh.dest[tid] = dest - local;
  __syncthreads();
  uint32_t at[RS_IPT];
#pragma unroll
  for (int j = 0; j < RS_IPT; ++j) {
    const int i = j * RS_THREADS + tid;
    if (i >= count) continue;
    const uint64_t key = sh.key[i];
    at[j] = sh.dest[(unsigned)(key >> shift) & (RS_RADIX - 1)] + (uint32_t)i;
    keys_out[at[j]] = key;
  }
  if (VALS) {
    uint32_t* val = reinterpret_cast<uint32_t*>(sh.key);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_IPT; ++j)
      if (sub + j * 32 + lane < count) val[rank[j]] = v[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_IPT; ++j) {
      const int i = j * RS_THREADS + tid;
      if (i < count) vals_out[at[j]] = val[i];
    }
  }
}

}  // namespace

namespace {
inline bool sort_small(int64_t n) { return n < RS_SMALL; }
inline int64_t sort_tiles(int64_t n) {
  const int64_t tile = RS_THREADS * (sort_small(n) ? 8 : 10);
  return n > 0 ? (n + tile - 1) / tile : 1;
}

template <int IPT>
void launch_pass(const uint64_t* keys, const uint32_t* vals, uint64_t* keys_out,
                 uint32_t* vals_out, int64_t n_max, const int64_t* n, int shift, int pass,
                 const unsigned long long* counts, unsigned long long* status, unsigned* ticket,
                 cudaStream_t s, unsigned* abort) {
  const unsigned grid = (unsigned)sort_tiles(n_max), limit = wait_limit(LOOKBACK_SPINS);
  if (vals)
    k_radix_pass<IPT, true><<<grid, RS_THREADS, 0, s>>>(keys, vals, keys_out, vals_out, n_max, n,
                                                        shift, pass, counts, status, ticket, abort,
                                                        limit);
  else
    k_radix_pass<IPT, false><<<grid, RS_THREADS, 0, s>>>(keys, vals, keys_out, vals_out, n_max, n,
                                                         shift, pass, counts, status, ticket, abort,
                                                         limit);
}
}  // namespace

// tmp: [tickets][status: tiles x RS_RADIX].  Just below RS_SMALL keys there are more tiles than
// from there on (1,024 against 820); the size covers the most tiles of n keys or fewer, so that
// storage sized for a larger input serves a smaller one.  A tile's status words start on a line.
constexpr size_t RS_TICKETS = 256;  // bytes
static_assert(RS_MAX_PASSES * sizeof(unsigned) <= RS_TICKETS, "a ticket a pass");
inline size_t sort_tmp_bytes(int64_t tiles) {
  return RS_TICKETS + (size_t)tiles * RS_RADIX * sizeof(unsigned long long);
}
size_t radix_sort_temp_bytes(int64_t n) {
  return sort_tmp_bytes(std::max(sort_tiles(n), sort_tiles(std::min(n, RS_SMALL - 1))));
}

erc_status radix_sort_begin(int64_t n, void* tmp, cudaStream_t s) {
  ERC_CUDA(cudaMemsetAsync(tmp, 0, sort_tmp_bytes(sort_tiles(n)), s));
  return ERC_OK;
}

erc_status radix_sort_pass(const uint64_t* keys, const uint32_t* vals, uint64_t* keys_out,
                           uint32_t* vals_out, int64_t n_max, const int64_t* n, int shift, int pass,
                           const unsigned long long* counts, void* tmp, cudaStream_t s,
                           unsigned* abort) {
  if (n_max <= 0) return ERC_OK;
  unsigned* ticket = static_cast<unsigned*>(tmp) + pass;
  unsigned long long* status =
      reinterpret_cast<unsigned long long*>(static_cast<char*>(tmp) + RS_TICKETS);
  if (sort_small(n_max))
    launch_pass<8>(keys, vals, keys_out, vals_out, n_max, n, shift, pass, counts, status, ticket, s,
                   abort);
  else
    launch_pass<10>(keys, vals, keys_out, vals_out, n_max, n, shift, pass, counts, status, ticket,
                    s, abort);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  return ERC_OK;
}

}  // namespace erc
