// cg_device.cuh -- device code shared by the CG translation units: the operator's argument
// block and row gather (L_eps p_u = eps p_u + sum_v w_uv (p_u - p_v), Eq. 5), the per-column
// dot-product combination, and the resident CG kernel (Algorithm 1, §3.1.3), whose plain and
// Jacobi-preconditioned instantiations are compiled in separate units.
#pragma once

#include "erc_internal.cuh"

namespace erc {
namespace {

constexpr int T = 256;
constexpr int WARPS = T / 32;
// default poll limits of the bounded waits: the vector update's grid barrier (which sleeps 64 ns
// between polls) and the resident solver's synchronisations (one L2 round trip per poll); either
// is seconds, far beyond any legitimate wait
constexpr unsigned SPIN_LIMIT = 1u << 24;
constexpr unsigned RES_SPIN_LIMIT = 1u << 22;
enum { MODE_STEP = 0, MODE_APPLY = 1, MODE_RESID = 2 };

struct SpmmArgs {
  const int64_t* row_ptr;
  const int32_t* col;
  const float* val;
  int32_t n, ld, kc;
  float eps;
  int32_t H;               // rows with more than H neighbours are split over a block
  const int32_t* heavy;    // their ids, ascending
  const int64_t* nheavy;   // their number (device)
  const float* P;  // operand: P (step/apply) or X (residual)
  float* AP;       // output of step/apply
  const float* Y;  // residual mode
  ColReduce cr;
  float* alpha;
  const double* rr;
  int* active;
  int* flags;
  double* pap_out;  // apply mode, may be null
  const double* yy;
  const int* iters;
  const int* conv;
  float* relres_out;
  int32_t* iters_out;
};

__device__ __forceinline__ float4 ld_f4(const float* p) {
  return __ldg(reinterpret_cast<const float4*>(p));
}
__device__ __forceinline__ float4 f4_zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// per-warp then per-block combination of per-thread column partials of a row-group kernel with
// NW warps; the cross-warp step runs over chunks of CH columns (scratch holds NW x CH)
template <int LPR, int VPL, int NW, int CH>
__device__ __forceinline__ void block_partials_groups(float2 (&d)[VPL][4], float2* sbuf,
                                                      float2* scratch, int ld) {
#pragma unroll
  for (int off = LPR; off < 32; off <<= 1) {
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float2 o;
        o.x = __shfl_xor_sync(0xffffffffu, d[v][t].x, off);
        o.y = __shfl_xor_sync(0xffffffffu, d[v][t].y, off);
        d[v][t] = df_add(d[v][t], o);
      }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int cb = 0; cb < ld; cb += CH) {
    if (lane < LPR) {
#pragma unroll
      for (int v = 0; v < VPL; ++v)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int c = 4 * (lane + LPR * v) + t;
          if (c >= cb && c < cb + CH && c < ld) scratch[warp * CH + (c - cb)] = d[v][t];
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < CH && cb + c < ld; c += blockDim.x) {
      float2 acc = make_float2(0.f, 0.f);
      for (int w = 0; w < NW; ++w) acc = df_add(acc, scratch[w * CH + c]);
      sbuf[cb + c] = acc;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------- the row walk
// Two float32 values in a 64-bit register, and the packed operations on them: each half is rounded
// as the scalar operation rounds it, at half the issue slots.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// a - b: the product with -1 is exact, so the one rounding is the difference's
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, pack2(-1.f, -1.f), a); }

// df_fma on two columns at once: (hi, lo) += a b
__device__ __forceinline__ void df_fma2(f32x2& hi, f32x2& lo, f32x2 a, f32x2 b) {
  const f32x2 p = mul2(a, b), pe = fma2(a, b, mul2(p, pack2(-1.f, -1.f)));
  const f32x2 s = add2(hi, p), bb = sub2(s, hi);
  f32x2 e = add2(sub2(hi, sub2(s, bb)), sub2(p, bb));
  e = add2(e, add2(lo, pe));
  hi = add2(s, e);
  lo = sub2(e, sub2(hi, s));
}

// four consecutive columns of a row
struct Quad {
  f32x2 a, b;
};
__device__ __forceinline__ Quad quad(float4 v) { return Quad{pack2(v.x, v.y), pack2(v.z, v.w)}; }
__device__ __forceinline__ float4 unquad(Quad q) {
  const float2 x = unpack2(q.a), y = unpack2(q.b);
  return make_float4(x.x, x.y, y.x, y.y);
}
template <bool L2ONLY>
__device__ __forceinline__ Quad ld_quad(const float* p) {
  return quad(L2ONLY ? __ldcg(reinterpret_cast<const float4*>(p)) : ld_f4(p));
}

// Four columns at p, past L1, where `on`, else v.  A predicated load: a branch would make the lanes
// of its two sides wait one after the other.
__device__ __forceinline__ Quad ldcg_quad_if(bool on, const float* p, Quad v) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t"
      "@q ld.global.cg.v2.u64 {%0, %1}, [%2];\n\t}"
      : "+l"(v.a), "+l"(v.b)
      : "l"(p), "r"((unsigned)on));
  return v;
}
__device__ __forceinline__ float4 ldcg_f4_if(bool on, const float* p, float4 v) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t"
      "@q ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w)
      : "l"(p), "r"((unsigned)on));
  return v;
}

// The neighbour ids (and weights) of a group's step, in shared memory: the step reads four at a
// time, where lanes that passed each other the ids would take a shuffle for every slot.  With
// NB = 2 the next step's are put beside this step's; with one set, in the resident solver, whose
// rows compete for the memory, they wait until the group is done with them.
template <int U, bool WEIGHTED, int NB>
struct alignas(16) Slots {
  uint32_t id[NB][U];
  float w[NB][U];
};
template <int U, int NB>
struct alignas(16) Slots<U, false, NB> {
  uint32_t id[NB][U];
};

// A group of LPR lanes walks a list of `nrows` rows, four columns a lane: row k's sum over its
// neighbours, acc = sum_j w_j (p_u - p_{col_j}) in CSR order, goes to emit(k, u, p_u, acc).
// bounds(k, start, len, u) names row k: its id and the CSR slots [start, start + len) to sum, len
// < 0 for a row that is not this walk's to emit.  own(u) is this lane's quad of p_u; srcq is
// column-quad address of row 0.  L2ONLY loads p through L2 only: required where p is rewritten
// within the same launch.  A lane with `on` false loads no neighbour (own must give it zero).
//
// The gathers are random row reads that L2 serves at up to 20 TB/s (64 bytes a clock and SM), if
// enough of them are in flight: what bounds a walk is the latency of the chain row bounds ->
// neighbour ids -> neighbour rows.  So the chain is taken apart: a step gathers up to U rows at
// once, and while they are on their way the next step's ids are loaded, which at a row's end are
// the next row's first, and the bounds of the row after that.  The short last step of a row takes
// 4, 8 or U slots; those past the end hold the row itself.  Through L1 they are loaded, from a
// cached line, and add exactly zero (128 columns, 150k nodes, 1.5M edges: 130 us, 139 with the
// loads predicated off).  Past L1 each would be a request to L2, so they are predicated off, and
// p_u stands for them (20,000 nodes, 160,000 edges, 32 columns: 477 us a solve, 544 with them).
//
// The groups of a warp take their steps together, with the longest one's count: left to themselves
// they drift apart, and a warp then issues, and waits for, each group's gathers in turn (1M nodes,
// 8M edges of a power law, 32 columns: 383 us an application, 508 before; 1M nodes, 3M edges:
// 178 us, 237 before).
template <int LPR, int U, bool WEIGHTED, bool L2ONLY, class Bounds, class Own, class Emit>
__device__ __forceinline__ void walk_rows(const SpmmArgs& a, const float* __restrict__ srcq,
                                          int gl, unsigned gm,
                                          Slots<U, WEIGHTED, L2ONLY ? 1 : 2>& slots, int nrows,
                                          bool on, Bounds&& bounds, Own&& own, Emit&& emit) {
  constexpr int E = (U + LPR - 1) / LPR;  // ids a lane fetches
  constexpr bool TOGETHER = LPR < 32;
  constexpr int NB = L2ONLY ? 1 : 2;
  const uint32_t ld = (uint32_t)a.ld;
  auto put = [&](int b, const uint32_t(&c)[E], const float(&w)[E]) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int k = gl + e * LPR;
      if (U % LPR != 0 && k >= U) continue;
      slots.id[b][k] = c[e];
      if constexpr (WEIGHTED) slots.w[b][k] = w[e];
    }
  };
  auto fetch = [&](uint32_t u, uint32_t j, int rem, uint32_t(&c)[E], float(&w)[E]) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int k = gl + e * LPR;
      c[e] = u;
      w[e] = 0.f;
      if (k < U && k < rem) {
        c[e] = (uint32_t)__ldg(a.col + (size_t)(j + (uint32_t)k));
        if (WEIGHTED) w[e] = __ldg(a.val + (size_t)(j + (uint32_t)k));
      }
    }
  };
  uint32_t u = 0, nu = 0, j = 0, nj = 0;  // slots are below 2^32: m < 2^31
  int rem = -1, nrem = -1;
  if (nrows > 0) bounds(0, j, rem, u);
  if (nrows > 1) bounds(1, nj, nrem, nu);
  uint32_t c[E];
  float w[E];
  int b = 0;  // the set that holds this step's slots
  fetch(u, j, rem, c, w);
  __syncwarp(gm);  // the group is done with the slots of an earlier walk
  put(0, c, w);
  __syncwarp(gm);
  Quad pu = {0, 0}, acc = {0, 0};
  bool fresh = true;
  for (int k = 0; TOGETHER ? __any_sync(0xffffffffu, k < nrows) : k < nrows;) {
    const bool last = rem <= U;
    fetch(last ? nu : u, last ? nj : j + U, last ? nrem : rem - U, c, w);
    uint32_t bj = 0, bu = 0;
    int brem = -1;
    if (last && k + 2 < nrows) bounds(k + 2, bj, brem, bu);
    if (fresh && (!TOGETHER || k < nrows)) pu = own(u);
    auto step = [&](auto count) {
      constexpr int N = decltype(count)::value;
      Quad v[N];
#pragma unroll
      for (int t = 0; t < N; t += 4) {
        const uint4 id = *reinterpret_cast<const uint4*>(&slots.id[b][t]);
        const uint32_t ids[4] = {id.x, id.y, id.z, id.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if constexpr (L2ONLY)
            v[t + r] = ldcg_quad_if(on && t + r < rem, srcq + (size_t)ids[r] * ld, pu);
          else
            v[t + r] = on ? quad(ld_f4(srcq + (size_t)ids[r] * ld)) : Quad{0, 0};
      }
#pragma unroll
      for (int t = 0; t < N; t += 4) {
        float4 wq = make_float4(1.f, 1.f, 1.f, 1.f);
        if constexpr (WEIGHTED) wq = *reinterpret_cast<const float4*>(&slots.w[b][t]);
        const float ws[4] = {wq.x, wq.y, wq.z, wq.w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const f32x2 da = sub2(pu.a, v[t + r].a), db = sub2(pu.b, v[t + r].b);
          if (WEIGHTED) {
            const f32x2 w2 = pack2(ws[r], ws[r]);
            acc.a = fma2(w2, da, acc.a);
            acc.b = fma2(w2, db, acc.b);
          } else {
            acc.a = add2(acc.a, da);
            acc.b = add2(acc.b, db);
          }
        }
      }
    };
    const int most = TOGETHER ? __reduce_max_sync(0xffffffffu, rem) : rem;
    if (most > 0) {
      if (most <= 4) step(ic<4>{});
      else if (U > 8 && most <= 8) step(ic<8>{});
      else step(ic<U>{});
    }
    if constexpr (NB == 1) __syncwarp(TOGETHER ? 0xffffffffu : gm);
    b = NB - 1 - b;
    put(b, c, w);  // with two sets: last read one step ago, before that step's barrier
    if (last) {
      if (rem >= 0) emit(k, u, pu, TOGETHER && rem == 0 ? Quad{0, 0} : acc);
      acc = Quad{0, 0};
      ++k;
      u = nu;
      j = nj;
      rem = nrem;
      nu = bu;
      nj = bj;
      nrem = brem;
    } else {
      j += U;
      rem -= U;
    }
    fresh = last;
    __syncwarp(TOGETHER ? 0xffffffffu : gm);
  }
}

// the CSR slots of row u
__device__ __forceinline__ void row_slots(const int64_t* row_ptr, int64_t u, uint32_t& j,
                                          uint32_t& len) {
  j = (uint32_t)__ldg(row_ptr + u);
  len = (uint32_t)__ldg(row_ptr + u + 1) - j;
}
// slice s of `parts` equal ones of a heavy row's slots
__device__ __forceinline__ void heavy_slice(const int64_t* row_ptr, int64_t u, int s, int parts,
                                            uint32_t& j, int& len) {
  uint32_t j0, n;
  row_slots(row_ptr, u, j0, n);
  const uint32_t per = (n + parts - 1) / parts;
  const uint32_t s0 = min(n, s * per), s1 = min(n, s0 + per);
  j = j0 + s0;
  len = (int)(s1 - s0);
}
// eps p_u + acc
__device__ __forceinline__ Quad apply_quad(float eps, Quad pu, Quad acc) {
  const f32x2 e = pack2(eps, eps);
  return Quad{fma2(e, pu.a, acc.a), fma2(e, pu.b, acc.b)};
}

// acc[v] += w (p_u - p_v) over the CSR slots [j, j + len) of row u, for the lane's VPL quads of
// every neighbour at once: rows of more than 128 columns.  The ids pass by shuffles, and 8 / VPL
// neighbours are in flight.  A walk for each quad passes over the row bounds and ids twice and
// waits twice (10,000 nodes, 256 columns: 60,000 edges 976 us a solve, 881 with both quads at once,
// 875 before the walk; 120,000 edges 1,130, 901 and 890).
template <int LPR, int VPL, bool WEIGHTED, bool L2ONLY>
__device__ __forceinline__ void gather_wide(const SpmmArgs& a, const float* __restrict__ src,
                                            int gl, unsigned gm, int nvec, unsigned on,
                                            uint32_t j, int len,
                                            const float4 (&pu)[VPL], float4 (&acc)[VPL]) {
  constexpr int U = 8 / VPL;
  for (int jb = 0; jb < len; jb += LPR) {
    int32_t cidx = 0;
    float wv = 1.f;
    if (jb + gl < len) {
      cidx = __ldg(a.col + (size_t)(j + (uint32_t)(jb + gl)));
      if (WEIGHTED) wv = __ldg(a.val + (size_t)(j + (uint32_t)(jb + gl)));
    }
    const int cnt = min(LPR, len - jb);
    for (int t = 0; t < cnt; t += U) {
      int cj[U];
      float wj[U];
      float4 pv[U][VPL];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        cj[k] = __shfl_sync(gm, cidx, (t + k) & (LPR - 1), LPR);
        wj[k] = WEIGHTED ? __shfl_sync(gm, wv, (t + k) & (LPR - 1), LPR) : 1.f;
        if (t + k >= cnt) wj[k] = 0.f;
      }
#pragma unroll
      for (int k = 0; k < U; ++k)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int q = gl + LPR * v;
          const bool take = q < nvec && t + k < cnt && ((on >> v) & 1u);
          const float* at = src + (size_t)cj[k] * a.ld + 4 * q;
          if constexpr (L2ONLY)
            pv[k][v] = ldcg_f4_if(take, at, pu[v]);
          else
            pv[k][v] = take ? ld_f4(at) : pu[v];
        }
#pragma unroll
      for (int k = 0; k < U; ++k)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          acc[v].x = fmaf(wj[k], pu[v].x - pv[k][v].x, acc[v].x);
          acc[v].y = fmaf(wj[k], pu[v].y - pv[k][v].y, acc[v].y);
          acc[v].z = fmaf(wj[k], pu[v].z - pv[k][v].z, acc[v].z);
          acc[v].w = fmaf(wj[k], pu[v].w - pv[k][v].w, acc[v].w);
        }
    }
  }
}

// the vectors and per-column state of one batched solve
struct VecArgs {
  int32_t n, ld, kc;
  double tol2;
  int32_t max_iter;
  const float* Y;
  float *X, *R, *P, *AP;
  float *alpha, *beta;
  double *rr, *yy;  // rr: r.r, or r.z with the Jacobi preconditioner; yy: y.y
  int *active, *conv, *iters, *flags;
  unsigned* gen;
  ColReduce cr;
  // Jacobi preconditioner M = diag(L_eps) = deg + eps (z = r / M): the weighted degrees, or
  // null for plain CG
  const float* deg;
  float eps;
  unsigned spin_limit;  // polls of a bounded wait before it gives up (sets flags[3])
};

// 1 / (deg_u + eps), the inverse diagonal of L_eps at row u
__device__ __forceinline__ float jacobi_inv(const float* deg, int64_t u, float eps) {
  return 1.f / (__ldg(deg + u) + eps);
}

__device__ __forceinline__ float4 f4_scale(float4 v, float s) {
  return make_float4(v.x * s, v.y * s, v.z * s, v.w * s);
}

// ---------------------------------------------------------------------------- resident CG
// When r and Ap of every row fit in the SMs' shared memory, one cooperative launch runs the whole
// solve.  Block b owns rows [b rb, b rb + rb): their r and Ap live in its shared memory, x and p
// in global memory (p is gathered by other blocks); where room is left (PS), the block's own rows
// of p are kept in shared memory too, and global p is only written and gathered.  Per iteration:
//   A  Ap = L_eps p on own rows (heavy rows by the whole block), p.Ap    -> reduce: alpha
//   B  x += alpha p, r -= alpha Ap, r.r                                  -> reduce: beta, stop
//   C  p = r + beta p                                                    -> barrier
// Where node ids follow the degree (power-law graphs often come so), contiguous ranges give the
// first block the hubs and every other block waits for it in A.  Such a solve runs A on dealt
// rows instead (block b takes rows b, b + G, ...) and hands Ap to the owners through global
// memory: the reduction of p.Ap between A and B orders the hand-over, so it costs no further
// synchronisation.  B, C and their sums keep their blocks.  A 60,013-node power-law graph (411k
// edges, 36 columns, Jacobi) took 14.2 ms a solve on its contiguous ranges and takes 1.7 ms; the
// even 20,000-node graph of 128 columns keeps its ranges (1.49 ms then, 1.41 ms with the walk).
// A grid synchronisation is an arrival (a release-add on a counter after the block's partials
// are written) and a bounded wait until all blocks have arrived.  There is no finishing block:
// after a reduction every block sums all blocks' partials itself, in the same fixed order, so
// every block derives the same alpha, beta and stop decisions into its own shared memory.  The
// counter only grows, so the s-th synchronisation waits for s * gridDim arrivals and needs no
// reset.  Data written by other blocks inside the launch (p, the partials) is read through L2
// (ld.global.cg), never through L1.  The vector phases B and C issue the loads of several rows
// before using any of them.
// With the Jacobi preconditioner (PC; an option, not the paper's method) z = r / (deg + eps):
// the start is p = z0, B also sums r.z (alpha and beta then use r.z in place of r.r, the stop
// test keeps r.r), and C forms p = z + beta p.
constexpr int PT = 512;
constexpr int PWARPS = PT / 32;
constexpr int PCH = 64;
constexpr int RMAXLD = 256;  // widest row block the resident kernel takes (64 float4)
constexpr int HROWS_MAX = 8;
constexpr int RU = 2;  // float4 loads per lane in flight in phases B and C
// neighbour rows in flight per row group in the gathers (fewer for the narrowest rows, so that no
// shape's slots take more than 8 KB: the memory left bounds the rows that the solver can take)
template <int LPR>
constexpr int RUB = LPR == 4 ? 8 : 16;

struct ResArgs {
  SpmmArgs s;
  VecArgs v;
  int32_t rb;     // rows per block
  int32_t hrows;  // heavy rows whose slices the shared memory holds at once
};

__device__ __forceinline__ float4 ldcg_f4(const float* p) {
  return __ldcg(reinterpret_cast<const float4*>(p));
}

// count this block in at the next synchronisation; the __syncthreads before thread 0's release
// orders the whole block's writes (and its reads of earlier partials) before it
__device__ __forceinline__ void res_arrive(unsigned* arr) {
  __syncthreads();
  if (threadIdx.x == 0) red_release_add(arr, 1u);
}
// bounded wait until `target` arrivals: after `limit` polls it sets flags[3] and returns
__device__ __forceinline__ void res_wait(const unsigned* arr, unsigned target, int* flags,
                                         unsigned limit) {
  if (threadIdx.x == 0) {
    unsigned spins = 0;
    while ((int)(ld_acquire(arr) - target) < 0) {  // one L2 round trip per poll
      if (++spins > limit) {
        atomicOr(&flags[3], 1);
        break;
      }
    }
  }
  __syncthreads();
}

// floats of the region that the resident kernel uses for the heavy-row slices, `hrows` rows of vpl
// quads per thread, and, after the operator, as the reduction scratch [2 * PT float pairs]
__host__ __device__ constexpr size_t resident_shared_floats(int hrows, int vpl) {
  return 4 * (size_t)PT * (size_t)(hrows * vpl);
}

// o = L_eps s on the rows r0 + i rstep, i < nrows, of s = src (n x ld): o_u = eps s_u +
// sum_v w_uv (s_u - s_v).  own(u, v) is float4 slot v of the lane of s_u.  The rows heavier than
// a.H (the ascending list hv[0..nh) of their i) are split over all groups of the block, hrows of
// them between two barriers, and their slices are added in group order; the others take one group
// each.  emit(i, u, v, s_u, o_u) runs once per row and valid slot.  Slots whose bit in `on` is
// clear are neither loaded nor gathered (s_u = 0 there).
template <int LPR, int VPL, bool WEIGHTED, class Own, class Emit>
__device__ __forceinline__ void block_apply(const SpmmArgs& a, const float* src, int64_t r0,
                                            int64_t rstep, int nrows, const int* hv, int nh,
                                            int hrows, float* comb,
                                            Slots<RUB<LPR>, WEIGHTED, 1>& slots, int gl, int gi,
                                            unsigned gm, unsigned on, Own&& own, Emit&& emit) {
  constexpr int GPB = PT / LPR;
  const int nvec = a.ld >> 2;
  float4* part = reinterpret_cast<float4*>(comb);  // [hrows][VPL][PT]
  if constexpr (VPL > 1) {
    auto load = [&](int64_t u, float4(&pu)[VPL], float4(&acc)[VPL]) {
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        pu[v] = gl + LPR * v < nvec && ((on >> v) & 1u) ? own(u, v) : f4_zero();
        acc[v] = f4_zero();
      }
    };
    auto give = [&](int i, int64_t u, const float4(&pu)[VPL], const float4(&acc)[VPL]) {
#pragma unroll
      for (int v = 0; v < VPL; ++v)
        if (gl + LPR * v < nvec)
          emit(i, u, v, pu[v], unquad(apply_quad(a.eps, quad(pu[v]), quad(acc[v]))));
    };
    float4 pu[VPL], acc[VPL];
    for (int hb = 0; hb < nh; hb += hrows) {
      const int cnt = min(hrows, nh - hb);
      for (int k = 0; k < cnt; ++k) {
        const int64_t u = r0 + hv[hb + k] * rstep;
        uint32_t j;
        int len;
        heavy_slice(a.row_ptr, u, gi, GPB, j, len);
        load(u, pu, acc);
        gather_wide<LPR, VPL, WEIGHTED, true>(a, src, gl, gm, nvec, on, j, len, pu, acc);
#pragma unroll
        for (int v = 0; v < VPL; ++v) part[(k * VPL + v) * PT + threadIdx.x] = acc[v];
      }
      __syncthreads();
      for (int k = gi; k < cnt; k += GPB) {
        const int i = hv[hb + k];
        load(r0 + i * rstep, pu, acc);
#pragma unroll
        for (int v = 0; v < VPL; ++v)
#pragma unroll 4
          for (int g = 0; g < GPB; ++g) {
            const float4 x = part[(k * VPL + v) * PT + g * LPR + gl];
            acc[v].x += x.x;
            acc[v].y += x.y;
            acc[v].z += x.z;
            acc[v].w += x.w;
          }
        give(i, r0 + i * rstep, pu, acc);
      }
      __syncthreads();
    }
    for (int i = gi; i < nrows; i += GPB) {
      const int64_t u = r0 + i * rstep;
      uint32_t j, len;
      row_slots(a.row_ptr, u, j, len);
      if (len > (uint32_t)a.H) continue;
      load(u, pu, acc);
      gather_wide<LPR, VPL, WEIGHTED, true>(a, src, gl, gm, nvec, on, j, (int)len, pu, acc);
      give(i, u, pu, acc);
    }
    return;
  }
  const bool valid = gl < nvec, lane_on = valid && (on & 1u);
  const float* srcq = src + 4 * (valid ? gl : 0);
  auto own_quad = [&](uint32_t u) { return lane_on ? quad(own((int64_t)u, 0)) : Quad{0, 0}; };
  for (int hb = 0; hb < nh; hb += hrows) {
    const int cnt = min(hrows, nh - hb);
    walk_rows<LPR, RUB<LPR>, WEIGHTED, true>(
        a, srcq, gl, gm, slots, cnt, lane_on,
        [&](int k, uint32_t& j, int& len, uint32_t& u) {
          u = (uint32_t)(r0 + hv[hb + k] * rstep);
          heavy_slice(a.row_ptr, u, gi, GPB, j, len);
        },
        own_quad,
        [&](int k, uint32_t, Quad, Quad acc) { part[k * PT + threadIdx.x] = unquad(acc); });
    // a group adds the slices of at most one row; its p is on the way meanwhile
    static_assert(GPB >= HROWS_MAX, "a group a heavy row");
    const int i = gi < cnt ? hv[hb + gi] : 0;
    const int64_t u = r0 + i * rstep;
    const Quad pu = gi < cnt ? own_quad((uint32_t)u) : Quad{0, 0};
    __syncthreads();
    if (gi < cnt) {
      Quad sum = {0, 0};
#pragma unroll 8
      for (int g = 0; g < GPB; ++g) {
        const Quad x = quad(part[gi * PT + g * LPR + gl]);
        sum.a = add2(sum.a, x.a);
        sum.b = add2(sum.b, x.b);
      }
      if (valid) emit(i, u, 0, unquad(pu), unquad(apply_quad(a.eps, pu, sum)));
    }
    __syncthreads();
  }
  const int mine = nrows > gi ? (nrows - gi + GPB - 1) / GPB : 0;
  walk_rows<LPR, RUB<LPR>, WEIGHTED, true>(
      a, srcq, gl, gm, slots, mine, lane_on,
      [&](int k, uint32_t& j, int& len, uint32_t& u) {
        u = (uint32_t)(r0 + (gi + k * GPB) * rstep);
        uint32_t n;
        row_slots(a.row_ptr, u, j, n);
        len = n > (uint32_t)a.H ? -1 : (int)n;
      },
      own_quad,
      [&](int k, uint32_t u, Quad pu, Quad acc) {
        if (valid)
          emit(gi + k * GPB, (int64_t)u, 0, unquad(pu), unquad(apply_quad(a.eps, pu, acc)));
      });
}

// the block's part of a grid-wide column sum: publish the block's partials (row blockIdx.x of
// part), count in, wait for every block, then sum all blocks' rows in a fixed order into sbuf
__device__ __forceinline__ void res_reduce(float2* part, int ld, const float2* bpart,
                                           float2* sbuf, float2* scratch, unsigned* arrivals,
                                           unsigned& nsync, int* flags, unsigned limit) {
  for (int c = threadIdx.x; c < ld; c += PT) part[(size_t)blockIdx.x * ld + c] = bpart[c];
  res_arrive(arrivals);
  res_wait(arrivals, ++nsync * gridDim.x, flags, limit);
  colsum_rows(part, gridDim.x, ld, sbuf, scratch);
}

template <int LPR, int VPL, bool WEIGHTED, bool PS, bool PC>
__global__ void __launch_bounds__(PT, 1) k_cg_resident(ResArgs ra) {
  extern __shared__ __align__(16) float dsm[];
  const SpmmArgs& a = ra.s;
  const VecArgs& va = ra.v;
  constexpr int GPB = PT / LPR;
  constexpr int NU = RU > VPL ? RU / VPL : 1;  // rows whose loads are in flight together
  const int gl = threadIdx.x & (LPR - 1);
  const int gi = threadIdx.x / LPR;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ld = a.ld, nvec = ld >> 2;
  const int G = gridDim.x;
  const unsigned gm = group_mask<LPR>();
  const int64_t r0 = (int64_t)blockIdx.x * ra.rb;
  const int nrows = (int)max((int64_t)0, min((int64_t)a.n, r0 + ra.rb) - r0);
  float* rs = dsm;                                     // [rb][ld]  r of own rows
  float* aps = rs + (size_t)ra.rb * ld;                // [rb][ld]  Ap of own rows
  float* ps = aps + (size_t)ra.rb * ld;                // [rb][ld]  p of own rows (PS only)
  float2* sbuf = reinterpret_cast<float2*>(PS ? ps + (size_t)ra.rb * ld : ps);  // [ld]
  // one region, used as the heavy-row slices [hrows][PT] in the operator and as the reduction
  // scratch [PWARPS][PCH] = 2 * PT float pairs after it; then the heavy-row list [rb] of the rows
  // the block gathers
  float* comb = reinterpret_cast<float*>(sbuf + ld);
  float2* scratch = sbuf + ld;
  int* hv = reinterpret_cast<int*>(comb + resident_shared_floats(ra.hrows, VPL));
  // block partials, one region per reduction kind so that no block overwrites partials another
  // block may still be summing: [G][ld] each
  float2* part_pap = a.cr.part1;
  // r.r rounded to float: sums of squares lose at most 2^-24 of their total that way, and every
  // block reads half the bytes
  float* part_rr = reinterpret_cast<float*>(a.cr.part1 + (size_t)G * ld);
  float* part_rz = part_rr + (size_t)G * ld;  // r.z (PC), also a sum of non-negative terms
  float2* part_init = a.cr.part1 + 2 * (size_t)G * ld;
  float2* part_yz = a.cr.part1 + 3 * (size_t)G * ld;  // y.z at the start (PC)
  float2* part_res = a.cr.part1 + 4 * (size_t)G * ld;
  unsigned* arrivals = va.gen;
  // per-column CG state, the same in every block
  constexpr int MAXC = 4 * LPR * VPL;
  __shared__ float2 s_rr[MAXC], s_yy[MAXC];  // float pairs; s_rr holds r.z with PC
  __shared__ float2 s_rz[PC ? MAXC : 1];        // the new r.z of phase B (PC)
  __shared__ __align__(16) float s_alpha[MAXC], s_beta[MAXC];
  __shared__ __align__(16) int s_active[MAXC];
  __shared__ int s_iters[MAXC], s_conv[MAXC];
  __shared__ int s_nh, s_wcnt[PWARPS];
  __shared__ unsigned s_most;
  __shared__ Slots<RUB<LPR>, WEIGHTED, 1> slots[VPL == 1 ? GPB : 1];  // the wide rows have none

  // ---- which rows the block gathers in A: its own, or dealt ones where the own ranges are so
  // uneven that the largest would cost more than 4 us an iteration over the mean.  A gathered
  // 128-byte line costs about 1 ns of an SM where L2 bounds the gathers (13 to 20 TB/s over 152
  // SMs): 4,000 lines, where handing Ap over through L2 costs under a microsecond.  Every block
  // finds the same.
  if (threadIdx.x == 0) {
    s_nh = 0;
    s_most = 0;
  }
  __syncthreads();
  for (int b = threadIdx.x; b < G; b += PT) {
    const int64_t lo = min((int64_t)a.n, (int64_t)b * ra.rb), hi = min((int64_t)a.n, lo + ra.rb);
    atomicMax(&s_most, (unsigned)(a.row_ptr[hi] - a.row_ptr[lo]));
  }
  __syncthreads();
  const int64_t excess = (int64_t)s_most - a.row_ptr[a.n] / G;
  const bool deal = excess * ((ld + 31) / 32) > 4000;
  const int64_t g0 = deal ? blockIdx.x : r0, gstep = deal ? G : 1;  // rows g0 + i gstep, i < grows
  const int grows = !deal ? nrows : a.n > g0 ? (int)((a.n - g0 + G - 1) / G) : 0;

  // ---- those of them heavier than a.H, ascending
  for (int base = 0; base < grows; base += PT) {
    const int i = base + threadIdx.x;
    const bool heavy =
        i < grows && a.row_ptr[g0 + i * gstep + 1] - a.row_ptr[g0 + i * gstep] > a.H;
    const unsigned bal = __ballot_sync(0xffffffffu, heavy);
    if (lane == 0) s_wcnt[warp] = __popc(bal);
    __syncthreads();
    int off = s_nh, tot = 0;
    for (int w = 0; w < PWARPS; ++w) {
      if (w < warp) off += s_wcnt[w];
      tot += s_wcnt[w];
    }
    if (heavy) hv[off + __popc(bal & ((1u << lane) - 1u))] = i;
    __syncthreads();
    if (threadIdx.x == 0) s_nh += tot;
    __syncthreads();
  }
  const int nh = s_nh;

  // ---- r = p = y (columns kc.. zero; with PC p = z = y / (deg + eps)), x = 0; y.y (and y.z)
  // -> the per-column state
  float2 dot[VPL][4];
  float2 dz[PC ? VPL : 1][4];  // r.z partials (PC)
#pragma unroll
  for (int v = 0; v < VPL; ++v)
#pragma unroll
    for (int t = 0; t < 4; ++t) dot[v][t] = make_float2(0.f, 0.f);
#pragma unroll
  for (int v = 0; v < (PC ? VPL : 1); ++v)
#pragma unroll
    for (int t = 0; t < 4; ++t) dz[v][t] = make_float2(0.f, 0.f);
  for (int i = gi; i < nrows; i += GPB) {
    const float di = PC ? jacobi_inv(va.deg, r0 + i, a.eps) : 1.f;
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int q = gl + LPR * v;
      if (q >= nvec) continue;
      const size_t o = (size_t)(r0 + i) * ld + 4 * q;
      float4 y = ld_f4(a.Y + o);
      const int cb = 4 * q;
      if (cb + 0 >= a.kc) y.x = 0.f;
      if (cb + 1 >= a.kc) y.y = 0.f;
      if (cb + 2 >= a.kc) y.z = 0.f;
      if (cb + 3 >= a.kc) y.w = 0.f;
      const float4 p0 = PC ? f4_scale(y, di) : y;
      reinterpret_cast<float4*>(rs + (size_t)i * ld)[q] = y;
      if (PS) reinterpret_cast<float4*>(ps + (size_t)i * ld)[q] = p0;
      *reinterpret_cast<float4*>(const_cast<float*>(a.P) + o) = p0;
      *reinterpret_cast<float4*>(va.X + o) = f4_zero();
      dot[v][0] = df_fma(dot[v][0], y.x, y.x);
      dot[v][1] = df_fma(dot[v][1], y.y, y.y);
      dot[v][2] = df_fma(dot[v][2], y.z, y.z);
      dot[v][3] = df_fma(dot[v][3], y.w, y.w);
      if constexpr (PC) {
        dz[v][0] = df_fma(dz[v][0], y.x, p0.x);
        dz[v][1] = df_fma(dz[v][1], y.y, p0.y);
        dz[v][2] = df_fma(dz[v][2], y.z, p0.z);
        dz[v][3] = df_fma(dz[v][3], y.w, p0.w);
      }
    }
  }
  unsigned nsync = 0;
  block_partials_groups<LPR, VPL, PWARPS, PCH>(dot, sbuf, scratch, ld);
  if constexpr (PC) {
    // y.y and y.z of the block published together, one synchronisation (which also publishes
    // p), then both sums: y.z to s_rr, y.y left in sbuf
    for (int c = threadIdx.x; c < ld; c += PT) part_init[(size_t)blockIdx.x * ld + c] = sbuf[c];
    block_partials_groups<LPR, VPL, PWARPS, PCH>(dz, sbuf, scratch, ld);
    for (int c = threadIdx.x; c < ld; c += PT) part_yz[(size_t)blockIdx.x * ld + c] = sbuf[c];
    res_arrive(arrivals);
    res_wait(arrivals, ++nsync * G, va.flags, va.spin_limit);
    colsum_rows(part_yz, G, ld, sbuf, scratch);
    for (int c = threadIdx.x; c < ld; c += PT) s_rr[c] = sbuf[c];
    colsum_rows(part_init, G, ld, sbuf, scratch);
  } else {
    res_reduce(part_init, ld, sbuf, sbuf, scratch, arrivals, nsync, va.flags,
               va.spin_limit);  // also publishes p
  }
  int any = 0;
  for (int c = threadIdx.x; c < ld; c += PT) {
    const float2 v = sbuf[c];
    const double vd = df_value(v);
    int act = 0, cv = 1;
    if (c < a.kc) {
      if (!isfinite(vd) || (PC && !isfinite(s_rr[c].x))) {
        cv = 0;
        if (blockIdx.x == 0) atomicOr(&va.flags[1], 1);
      } else if (vd > 0.0 && !(vd <= va.tol2 * vd)) {
        act = 1;
        cv = 0;
      }
    }
    s_yy[c] = v;
    if (!PC) s_rr[c] = v;
    s_alpha[c] = 0.f;
    s_beta[c] = 0.f;
    s_active[c] = act;
    s_iters[c] = 0;
    s_conv[c] = cv;
    any |= act;
  }
  any = __syncthreads_or(any);

  while (any) {
    if (*(volatile int*)&va.flags[3] != 0) break;
    // ---------------- A: Ap = L_eps p on own rows, p.Ap
    if (nsync > 1) res_wait(arrivals, nsync * G, va.flags, va.spin_limit);  // every p written
    // this lane's float4 slots with an active column: converged columns are neither gathered
    // nor updated (their alpha is 0)
    unsigned on = 0;
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int q = gl + LPR * v;
      if (q < nvec) {
        const int4 act = reinterpret_cast<const int4*>(s_active)[q];
        if (act.x | act.y | act.z | act.w) on |= 1u << v;
      }
    }
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
      for (int t = 0; t < 4; ++t) dot[v][t] = make_float2(0.f, 0.f);
    block_apply<LPR, VPL, WEIGHTED>(
        a, a.P, g0, gstep, grows, hv, nh, ra.hrows, comb, slots[VPL == 1 ? gi : 0], gl, gi, gm, on,
        [&](int64_t u, int v) {
          const int q = gl + LPR * v;
          return PS && !deal ? reinterpret_cast<const float4*>(ps + (size_t)(u - r0) * ld)[q]
                             : ldcg_f4(a.P + (size_t)u * ld + 4 * q);
        },
        [&](int i, int64_t u, int v, float4 pu, float4 o) {
          const int q = gl + LPR * v;
          if (deal)
            *reinterpret_cast<float4*>(a.AP + (size_t)u * ld + 4 * q) = o;
          else
            reinterpret_cast<float4*>(aps + (size_t)i * ld)[q] = o;
          dot[v][0] = df_fma(dot[v][0], pu.x, o.x);
          dot[v][1] = df_fma(dot[v][1], pu.y, o.y);
          dot[v][2] = df_fma(dot[v][2], pu.z, o.z);
          dot[v][3] = df_fma(dot[v][3], pu.w, o.w);
        });
    block_partials_groups<LPR, VPL, PWARPS, PCH>(dot, sbuf, scratch, ld);
    res_reduce(part_pap, ld, sbuf, sbuf, scratch, arrivals, nsync, va.flags, va.spin_limit);
    for (int c = threadIdx.x; c < ld; c += PT) {
      const float2 v = sbuf[c];
      float al = 0.f;
      if (s_active[c]) {
        const float q = df_div(s_rr[c], v);
        if (!(v.x > 0.f) || !isfinite(q)) {
          s_active[c] = 0;
          if (blockIdx.x == 0) atomicOr(&va.flags[1], 1);
        } else {
          al = q;
        }
      }
      s_alpha[c] = al;
    }
    __syncthreads();

    // ---------------- B: x += alpha p, r -= alpha Ap, r.r (and r.z)
    float4 al[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int q = gl + LPR * v;
      al[v] = q < nvec ? reinterpret_cast<const float4*>(s_alpha)[q] : f4_zero();
      for (int t = 0; t < 4; ++t) dot[v][t] = make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int v = 0; v < (PC ? VPL : 1); ++v)
#pragma unroll
      for (int t = 0; t < 4; ++t) dz[v][t] = make_float2(0.f, 0.f);
    for (int i0 = gi; i0 < nrows; i0 += NU * GPB) {
      float4 p[NU][VPL], x[NU][VPL], ap[NU][VPL];
      float di[NU];
#pragma unroll
      for (int k = 0; k < NU; ++k)
        di[k] = PC && i0 + k * GPB < nrows ? jacobi_inv(va.deg, r0 + i0 + k * GPB, a.eps) : 1.f;
#pragma unroll
      for (int k = 0; k < NU; ++k)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int i = i0 + k * GPB, q = gl + LPR * v;
          if (i < nrows && q < nvec && ((on >> v) & 1u)) {
            const size_t o = (size_t)(r0 + i) * ld + 4 * q;
            p[k][v] = PS ? reinterpret_cast<const float4*>(ps + (size_t)i * ld)[q] : ldcg_f4(a.P + o);
            x[k][v] = *reinterpret_cast<const float4*>(va.X + o);
            ap[k][v] = deal ? ldcg_f4(a.AP + o)
                            : reinterpret_cast<const float4*>(aps + (size_t)i * ld)[q];
          }
        }
#pragma unroll
      for (int k = 0; k < NU; ++k)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int i = i0 + k * GPB, q = gl + LPR * v;
          if (i >= nrows || q >= nvec || !((on >> v) & 1u)) continue;
          float4 xx = x[k][v], r = reinterpret_cast<const float4*>(rs + (size_t)i * ld)[q];
          const float4 pp = p[k][v];
          xx.x = fmaf(al[v].x, pp.x, xx.x);
          xx.y = fmaf(al[v].y, pp.y, xx.y);
          xx.z = fmaf(al[v].z, pp.z, xx.z);
          xx.w = fmaf(al[v].w, pp.w, xx.w);
          r.x = fmaf(-al[v].x, ap[k][v].x, r.x);
          r.y = fmaf(-al[v].y, ap[k][v].y, r.y);
          r.z = fmaf(-al[v].z, ap[k][v].z, r.z);
          r.w = fmaf(-al[v].w, ap[k][v].w, r.w);
          *reinterpret_cast<float4*>(va.X + (size_t)(r0 + i) * ld + 4 * q) = xx;
          reinterpret_cast<float4*>(rs + (size_t)i * ld)[q] = r;
          dot[v][0] = df_fma(dot[v][0], r.x, r.x);
          dot[v][1] = df_fma(dot[v][1], r.y, r.y);
          dot[v][2] = df_fma(dot[v][2], r.z, r.z);
          dot[v][3] = df_fma(dot[v][3], r.w, r.w);
          if constexpr (PC) {
            const float4 z = f4_scale(r, di[k]);
            dz[v][0] = df_fma(dz[v][0], r.x, z.x);
            dz[v][1] = df_fma(dz[v][1], r.y, z.y);
            dz[v][2] = df_fma(dz[v][2], r.z, z.z);
            dz[v][3] = df_fma(dz[v][3], r.w, z.w);
          }
        }
    }
    block_partials_groups<LPR, VPL, PWARPS, PCH>(dot, sbuf, scratch, ld);
    for (int c = threadIdx.x; c < ld; c += PT)
      part_rr[(size_t)blockIdx.x * ld + c] = __fadd_rn(sbuf[c].x, sbuf[c].y);
    if constexpr (PC) {
      block_partials_groups<LPR, VPL, PWARPS, PCH>(dz, sbuf, scratch, ld);
      for (int c = threadIdx.x; c < ld; c += PT)
        part_rz[(size_t)blockIdx.x * ld + c] = __fadd_rn(sbuf[c].x, sbuf[c].y);
    }
    res_arrive(arrivals);
    res_wait(arrivals, ++nsync * G, va.flags, va.spin_limit);
    if constexpr (PC) {
      colsum_rows_f(part_rz, G, ld, sbuf, scratch);
      for (int c = threadIdx.x; c < ld; c += PT) s_rz[c] = sbuf[c];
    }
    colsum_rows_f(part_rr, G, ld, sbuf, scratch);
    any = 0;
    for (int c = threadIdx.x; c < ld; c += PT) {
      float be = 0.f;
      int act = s_active[c];
      if (act) {
        const float2 rn = sbuf[c];
        const float2 rho = PC ? s_rz[c] : rn;  // the numerator of beta
        const int it = s_iters[c] + 1;
        s_iters[c] = it;
        if (!isfinite(rn.x) || !isfinite(rho.x)) {
          act = 0;
          if (blockIdx.x == 0) atomicOr(&va.flags[1], 1);
        } else {
          be = df_div(rho, s_rr[c]);
          s_rr[c] = rho;
          if (df_value(rn) <= va.tol2 * df_value(s_yy[c])) {
            s_conv[c] = 1;
            act = 0;
          } else if (it >= va.max_iter) {
            act = 0;
          }
        }
        s_active[c] = act;
      }
      s_beta[c] = be;
      any |= act;
    }
    any = __syncthreads_or(any);  // the same in every block
    if (!any) break;

    // ---------------- C: p = r + beta p (PC: p = z + beta p) on active columns
    int4 act[VPL];
    float4 be[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int q = gl + LPR * v;
      act[v] = q < nvec ? reinterpret_cast<const int4*>(s_active)[q] : make_int4(0, 0, 0, 0);
      be[v] = q < nvec ? reinterpret_cast<const float4*>(s_beta)[q] : f4_zero();
    }
    for (int i0 = gi; i0 < nrows; i0 += NU * GPB) {
      float4 p[NU][VPL];
      float di[NU];
#pragma unroll
      for (int k = 0; k < NU; ++k)
        di[k] = PC && i0 + k * GPB < nrows ? jacobi_inv(va.deg, r0 + i0 + k * GPB, a.eps) : 1.f;
#pragma unroll
      for (int k = 0; k < NU; ++k)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int i = i0 + k * GPB, q = gl + LPR * v;
          if (i < nrows && (act[v].x | act[v].y | act[v].z | act[v].w))
            p[k][v] = PS ? reinterpret_cast<const float4*>(ps + (size_t)i * ld)[q]
                         : ldcg_f4(a.P + (size_t)(r0 + i) * ld + 4 * q);
        }
#pragma unroll
      for (int k = 0; k < NU; ++k)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int i = i0 + k * GPB, q = gl + LPR * v;
          if (i >= nrows || !(act[v].x | act[v].y | act[v].z | act[v].w)) continue;
          float4 r = reinterpret_cast<const float4*>(rs + (size_t)i * ld)[q];
          if (PC) r = f4_scale(r, di[k]);  // z
          float4 pp = p[k][v];
          if (act[v].x) pp.x = fmaf(be[v].x, pp.x, r.x);
          if (act[v].y) pp.y = fmaf(be[v].y, pp.y, r.y);
          if (act[v].z) pp.z = fmaf(be[v].z, pp.z, r.z);
          if (act[v].w) pp.w = fmaf(be[v].w, pp.w, r.w);
          *reinterpret_cast<float4*>(const_cast<float*>(a.P) + (size_t)(r0 + i) * ld + 4 * q) = pp;
          if (PS) reinterpret_cast<float4*>(ps + (size_t)i * ld)[q] = pp;
        }
    }
    res_arrive(arrivals);
    ++nsync;
  }

  // ---- true residual y - L_eps x of the returned iterate (every block's x is final: the last
  // reduction ordered its writes), relative to ||y||; iterations and the unconverged count
#pragma unroll
  for (int v = 0; v < VPL; ++v)
#pragma unroll
    for (int t = 0; t < 4; ++t) dot[v][t] = make_float2(0.f, 0.f);
  block_apply<LPR, VPL, WEIGHTED>(
      a, va.X, g0, gstep, grows, hv, nh, ra.hrows, comb, slots[VPL == 1 ? gi : 0], gl, gi, gm, ~0u,
      [&](int64_t u, int v) { return ldcg_f4(va.X + (size_t)u * ld + 4 * (gl + LPR * v)); },
      [&](int, int64_t u, int v, float4, float4 o) {
        const int q = gl + LPR * v, cb = 4 * q;
        const float4 y = ld_f4(a.Y + (size_t)u * ld + 4 * q);
        const float rx = cb + 0 < a.kc ? y.x - o.x : 0.f;
        const float ry = cb + 1 < a.kc ? y.y - o.y : 0.f;
        const float rz = cb + 2 < a.kc ? y.z - o.z : 0.f;
        const float rw = cb + 3 < a.kc ? y.w - o.w : 0.f;
        dot[v][0] = df_fma(dot[v][0], rx, rx);
        dot[v][1] = df_fma(dot[v][1], ry, ry);
        dot[v][2] = df_fma(dot[v][2], rz, rz);
        dot[v][3] = df_fma(dot[v][3], rw, rw);
      });
  block_partials_groups<LPR, VPL, PWARPS, PCH>(dot, sbuf, scratch, ld);
  res_reduce(part_res, ld, sbuf, sbuf, scratch, arrivals, nsync, va.flags, va.spin_limit);
  if (blockIdx.x == 0)
    for (int c = threadIdx.x; c < a.kc; c += PT) {
      const float q = s_yy[c].x > 0.f ? df_div(sbuf[c], s_yy[c]) : 0.f;
      a.relres_out[c] = sqrtf(fmaxf(q, 0.f));
      a.iters_out[c] = s_iters[c];
      if (!s_conv[c]) atomicAdd(&va.flags[2], 1);
    }
}

// the resident kernel of a row-block shape: nvec float4 per row, weighted or not, p of the own
// rows in shared memory (ps) or not; null for rows wider than 256 floats
template <bool PC>
const void* resident_kernel_for(int nvec, bool weighted, bool ps) {
  const void* k = nullptr;
  auto pick = [&](auto lpr, auto vpl) {
    constexpr int LPR = decltype(lpr)::value, VPL = decltype(vpl)::value;
    if (ps)
      k = weighted ? (const void*)k_cg_resident<LPR, VPL, true, true, PC>
                   : (const void*)k_cg_resident<LPR, VPL, false, true, PC>;
    else
      k = weighted ? (const void*)k_cg_resident<LPR, VPL, true, false, PC>
                   : (const void*)k_cg_resident<LPR, VPL, false, false, PC>;
  };
  if (nvec <= 4) pick(ic<4>{}, ic<1>{});
  else if (nvec <= 8) pick(ic<8>{}, ic<1>{});
  else if (nvec <= 16) pick(ic<16>{}, ic<1>{});
  else if (nvec <= 32) pick(ic<32>{}, ic<1>{});
  else if (nvec <= 64) pick(ic<32>{}, ic<2>{});
  return k;  // wider rows use the multi-kernel path
}

}  // namespace

// the preconditioned (Jacobi) resident kernels, compiled in cg_pcg.cu
const void* resident_kernel_pc(int nvec, bool weighted, bool ps);

}  // namespace erc
