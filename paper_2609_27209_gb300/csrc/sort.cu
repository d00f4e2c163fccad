// sort.cu -- the passes of a stable, deterministic LSD radix sort of (u64 key, u32 value) pairs for
// the Laplacian build (§3.1.1).
#include "erc_internal.cuh"

namespace erc {

namespace {

// ------------------------------------------------------------------------------------------------
// Stable LSD radix sort of (u64 key, u32 value) pairs, one kernel per 8-bit digit (the digit counts
// of every pass come from the kernel that wrote the keys): a tile ranks its keys, publishes its
// digit counts, learns the counts of the tiles before it by decoupled look-back (as tile_prefix, one
// digit per thread) and writes its keys.  What bounds a pass is HBM: 12 bytes read and
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
constexpr int LB = 16;
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

  // ---- digit tid in the tiles before this one, LB status words a trip: the walk back over the
  // hundreds of tiles in flight takes an L2 latency a trip
  if (t > 0) {
    unsigned long long before = 0;
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
