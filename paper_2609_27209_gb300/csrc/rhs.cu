// rhs.cu -- erc_jl_rhs: Y = B^T W^{1/2} Q for a batch of projection columns (§3.1.2), with the
// signs of Q generated in registers by Philox4x32-10 and never stored.
//
// Row u of Y gathers over u's CSR slots: the canonical edge e = (eu, ev) contributes
// sigma * sqrt(w_e) * Q[e, c] with sigma = +1 when u = eu (the smaller id) and -1 otherwise.
// Summing in CSR order makes Y deterministic without atomics.
#include "erc_internal.cuh"

namespace erc {
namespace {

// Row u of Y: the LPR lanes of a group walk u's CSR slots LPR at a time.  Lane l generates the
// Philox words of slot jb + l (one block of four words per 128 columns that the group covers) and
// leaves them in shared memory with the slot's coefficient; the slots are then applied in CSR
// order, each lane reading the one word that holds its four columns' signs.  The orientation sigma
// goes into the words (all signs of a slot flipped), and a sign is applied by moving its bit to the
// coefficient's sign bit.
//
// What bounds it is instruction issue: each of the 2m slots costs a lane two shared loads and a
// dozen operations (passing the words by shuffles, four a slot and the selection of one of them,
// took about 28).  2.45M nodes, 64.3M edges, 128 columns: 2.77 ms, 6.71 ms with the shuffles.
template <int LPR, int VPL, bool WEIGHTED>
__global__ void __launch_bounds__(256)
    k_jl_rhs(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
             const float* __restrict__ val, const int32_t* __restrict__ csr_eid, int32_t n,
             uint2 key, float inv_sqrt_k, int32_t c0, int32_t kc, int32_t ld,
             float* __restrict__ Y) {
  constexpr int NB = (4 * LPR * VPL + 127) / 128 + 1;  // 128-column Philox blocks a group can span
  constexpr int GPB = 256 / LPR;
  // a slot's words; groups are padded apart so that they meet in different banks
  __shared__ __align__(16) uint32_t s_word[GPB][LPR * 4 * NB + 4];
  __shared__ float s_coef[WEIGHTED ? GPB : 1][WEIGHTED ? LPR : 1];
  const int gl = threadIdx.x & (LPR - 1), gi = threadIdx.x / LPR;
  const unsigned gm = group_mask<LPR>();
  const int64_t ngroups = (int64_t)gridDim.x * GPB;
  const int nvec = ld >> 2;
  const int g0 = c0 >> 7;
  const int nb = ((c0 + 4 * (nvec - 1)) >> 7) - g0 + 1;
  int at[VPL], sh[VPL];  // the lane's word among a slot's 4 NB, and the shift of its columns' bits
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int q = min(gl + LPR * v, nvec - 1);
    const int c = c0 + 4 * q;  // c0 % 4 == 0: the four columns share one word
    at[v] = (c >> 5) - 4 * g0;
    sh[v] = 28 - (c & 31);  // the column's bit 0 to bit 28, and so on to bit 31
  }
  for (int64_t u = (int64_t)blockIdx.x * GPB + gi; u < n; u += ngroups) {
    float4 acc[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t j0 = row_ptr[u], j1 = row_ptr[u + 1];
    // the next slots' ids are loaded before the present ones are applied
    uint32_t e = 0;
    int32_t other = 0;
    float w = 0.f;
    auto fetch = [&](int64_t j) {
      if (j >= j1) return;
      e = (uint32_t)__ldg(csr_eid + j);
      other = __ldg(col + j);
      if (WEIGHTED) w = __ldg(val + j);
    };
    fetch(j0 + gl);
    for (int64_t jb = j0; jb < j1; jb += LPR) {
      if (jb + gl < j1) {
        // u is the larger endpoint: row e is e_nb - e_u
        const uint32_t flip = other < u ? ~0u : 0u;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          if (b >= nb) break;
          const uint4 x = philox4x32_10(make_uint4((uint32_t)(g0 + b), 0u, e, 0u), key);
          *reinterpret_cast<uint4*>(s_word[gi] + gl * 4 * NB + 4 * b) =
              make_uint4(x.x ^ flip, x.y ^ flip, x.z ^ flip, x.w ^ flip);
        }
        if (WEIGHTED) s_coef[gi][gl] = sqrtf(w) * inv_sqrt_k;
      }
      fetch(jb + LPR + gl);
      __syncwarp(gm);
      const int cnt = (int)min((int64_t)LPR, j1 - jb);
#pragma unroll 4
      for (int k = 0; k < cnt; ++k) {
        const uint32_t cf = __float_as_uint(WEIGHTED ? s_coef[WEIGHTED ? gi : 0][WEIGHTED ? k : 0]
                                                     : inv_sqrt_k);
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const uint32_t bits = s_word[gi][k * 4 * NB + at[v]];
          const uint32_t top = bits << sh[v];
          acc[v].x += __uint_as_float(cf ^ ((top << 3) & 0x80000000u));
          acc[v].y += __uint_as_float(cf ^ ((top << 2) & 0x80000000u));
          acc[v].z += __uint_as_float(cf ^ ((top << 1) & 0x80000000u));
          acc[v].w += __uint_as_float(cf ^ (top & 0x80000000u));
        }
      }
      __syncwarp(gm);
    }
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int q = gl + LPR * v;
      if (q < nvec) {
        float4 o = acc[v];
        const int cb = 4 * q;
        if (cb + 0 >= kc) o.x = 0.f;
        if (cb + 1 >= kc) o.y = 0.f;
        if (cb + 2 >= kc) o.z = 0.f;
        if (cb + 3 >= kc) o.w = 0.f;
        reinterpret_cast<float4*>(Y + (size_t)u * ld)[q] = o;
      }
    }
  }
}

__global__ void k_philox_signs(uint2 key, int64_t e0, int64_t e1, int32_t c0, int32_t c1,
                               uint32_t* __restrict__ out) {
  const int64_t ncol = c1 - c0;
  const int64_t total = (e1 - e0) * ncol;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = e0 + t / ncol;
    const int c = c0 + (int)(t % ncol);
    const uint4 w = philox4x32_10(
        make_uint4((uint32_t)(c >> 7), 0u, (uint32_t)(e & 0xffffffff), (uint32_t)(e >> 32)), key);
    const int wi = (c >> 5) & 3;
    const uint32_t word = wi == 0 ? w.x : wi == 1 ? w.y : wi == 2 ? w.z : w.w;
    out[t] = (word >> (c & 31)) & 1u;
  }
}

}  // namespace
}  // namespace erc

using namespace erc;

extern "C" erc_status erc_jl_rhs(const erc_graph* g, uint64_t seed, int32_t K, int32_t c0,
                                 int32_t kc, float* Y, int32_t ld, erc_stream stream) {
  clear_error();
  ERC_TRY(check_graph(g));
  ERC_REQUIRE(K >= 1 && kc >= 1 && c0 >= 0 && (int64_t)c0 + kc <= K,
              "need 0 <= c0, 1 <= kc, c0 + kc <= K (c0=%d kc=%d K=%d)", c0, kc, K);
  ERC_REQUIRE(c0 % 4 == 0, "c0 must be a multiple of 4 (got %d)", c0);
  ERC_REQUIRE(ld >= kc && ld % 4 == 0 && ld <= MAX_LD, "bad ld %d for kc %d", ld, kc);
  ERC_REQUIRE(Y && (reinterpret_cast<uintptr_t>(Y) & 15) == 0, "Y must be 16-byte aligned");
  ERC_REQUIRE(g->m < (int64_t(1) << 31), "m must be < 2^31");
  cudaStream_t s = as_stream(stream);
  const uint2 key = make_uint2((uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
  const float inv_sqrt_k = (float)(1.0 / sqrt((double)K));
  return dispatch_shape(ld / 4, [&](auto lpr, auto vpl) -> erc_status {
    constexpr int LPR = decltype(lpr)::value, VPL = decltype(vpl)::value;
    const int grid = grid_for(g->n, 256 / LPR);
    if (g->val)
      k_jl_rhs<LPR, VPL, true><<<grid, 256, 0, s>>>(g->row_ptr, g->col, g->val, g->csr_eid, g->n,
                                                    key, inv_sqrt_k, c0, kc, ld, Y);
    else
      k_jl_rhs<LPR, VPL, false><<<grid, 256, 0, s>>>(g->row_ptr, g->col, g->val, g->csr_eid, g->n,
                                                     key, inv_sqrt_k, c0, kc, ld, Y);
    count_launches(1);
    ERC_CUDA(cudaGetLastError());
    return ERC_OK;
  });
}

extern "C" erc_status erc_philox_signs(uint64_t seed, int64_t e0, int64_t e1, int32_t c0,
                                       int32_t c1, uint32_t* out_bits, erc_stream stream) {
  clear_error();
  ERC_REQUIRE(e0 >= 0 && e1 >= e0 && c0 >= 0 && c1 >= c0, "bad ranges");
  ERC_REQUIRE(out_bits || e1 == e0 || c1 == c0, "out_bits is required");
  const int64_t total = (e1 - e0) * (int64_t)(c1 - c0);
  if (total == 0) return ERC_OK;
  const uint2 key = make_uint2((uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
  k_philox_signs<<<grid_for(total, 256), 256, 0, as_stream(stream)>>>(key, e0, e1, c0, c1,
                                                                      out_bits);
  count_launches(1);
  ERC_CUDA(cudaGetLastError());
  return ERC_OK;
}
