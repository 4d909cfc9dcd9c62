// Router: logits z = W_r x (+ bias), top-k by (z desc, id asc), softmax over the chosen.
//
// MoE routing selects a subset of experts per token (Background section of the paper).
// Logits are computed with a compensated dot product (Ogita, Rump & Oishi, "Accurate sum and
// dot product", SIAM J. Sci. Comput. 2005, algorithm Dot2): every product is split exactly
// into value + error with an FMA, the running sum is kept as an unevaluated pair, and the pair
// is rounded to fp32 once.  The result is the fp32 rounding of the exact dot product except
// where the exact value lies within ~n*2^-48 relative of a rounding boundary, so selection does
// not depend on the summation order.
//
// One thread-block cluster of 16 blocks per token (8 where the GPU does not schedule clusters of
// 16): block r computes the logits of experts [r*ceil(E/nc), (r+1)*ceil(E/nc)), with
// 16 / ceil(E/nc) warps per expert
// when the block has fewer experts than warps (each warp a lane-interleaved share of the row,
// its loads issued together; the warps' compensated pairs are then added with the same
// error-free steps), and stores them straight into block 0's shared memory.  After
// a cluster barrier, block 0 gathers all logits through distributed shared memory, ranks each
// expert by counting the experts ahead of it, and keeps the k first.  With one token per call,
// block 0 then runs the layer's slot resolve (lru_warp) on cache state it prefetched into
// registers while the logits were being computed.  No global atomics or fences on the path.
//
// Calls with many tokens (T >= kTiledMinT) read W_r once per 64 tokens in a plain fp32 product that
// singles out the experts that can be chosen, and compute those exactly: see k_logits_fp32.
#include <cooperative_groups.h>

#include <algorithm>

#include "mf_lru.cuh"

namespace cg = cooperative_groups;

namespace mf {
namespace {

constexpr int kThreadsR = 512;
constexpr int kWarpsR = kThreadsR / 32;
constexpr int kChunk = 8;  // float4 loads of W (and of x) a lane issues before using them
constexpr int kPre = kMaxExperts / kThreadsR;  // prefetched cache-state entries per thread

struct F2 {
  float hi, lo;
};

__device__ __forceinline__ F2 two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}

// (s, c) += a * b, error-free product split plus compensated running sum
__device__ __forceinline__ void dot2(float& s, float& c, float a, float b) {
  float p = __fmul_rn(a, b);
  float pe = __fmaf_rn(a, b, -p);
  F2 t = two_sum(s, p);
  s = t.hi;
  c = __fadd_rn(c, __fadd_rn(t.lo, pe));
}

// (s, c) += (s2, c2) for compensated pairs
__device__ __forceinline__ void pair_add(float& s, float& c, float s2, float c2) {
  const F2 t = two_sum(s, s2);
  s = t.hi;
  c = __fadd_rn(__fadd_rn(c, c2), t.lo);
}

// The first chunk of logit_part's W loads, issued before x is in shared memory.
__device__ __forceinline__ void w_preload(const float* __restrict__ w, int n4, int first, int step, float4* a) {
  const float4* w4 = reinterpret_cast<const float4*>(w);
  const uint64_t pol = l2_evict_last();  // W_r is read again by the layer's next call
#pragma unroll
  for (int u = 0; u < kChunk; ++u) {
    const int q = first + u * step;
    if (q < n4) a[u] = ld_hint(w4 + q, pol);
  }
}

// Compensated partial dot product of one expert row with x (in shared memory) over the float4
// indices q = first, first + step, ... (< H / 4), summed over the warp; returns the pair in (s, c).
// `pre` holds the first chunk's W values (w_preload).
__device__ __forceinline__ void logit_part(const float* __restrict__ w, const float* xs, int n4, int first, int step,
                                           const float4* pre, float& s, float& c) {
  s = 0.f;
  c = 0.f;
  const float4* w4 = reinterpret_cast<const float4*>(w);
  const float4* x4 = reinterpret_cast<const float4*>(xs);
  for (int q0 = first; q0 < n4; q0 += kChunk * step) {
    float4 a[kChunk], b[kChunk];
#pragma unroll
    for (int u = 0; u < kChunk; ++u) {  // all loads of the chunk first
      const int q = q0 + u * step;
      if (q < n4) {
        a[u] = q0 == first ? pre[u] : ld_hint(w4 + q, l2_evict_last());
        b[u] = x4[q];
      }
    }
#pragma unroll
    for (int u = 0; u < kChunk; ++u) {
      if (q0 + u * step < n4) {
        dot2(s, c, a[u].x, b[u].x);
        dot2(s, c, a[u].y, b[u].y);
        dot2(s, c, a[u].z, b[u].z);
        dot2(s, c, a[u].w, b[u].w);
      }
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float so = __shfl_xor_sync(0xffffffffu, s, off);
    const float co = __shfl_xor_sync(0xffffffffu, c, off);
    pair_add(s, c, so, co);
  }
}

__device__ __forceinline__ bool cluster_rank_zero() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r == 0;
}

// The logit by which an expert is ranked: one that is not a number counts as the lowest, so that the order
// is total and the k first places name k distinct experts whatever the inputs are.
__device__ __forceinline__ float rank_key(float z) { return fmaxf(z, -INFINITY); }

// Rank by counting: position of expert e = experts with a larger logit, or equal and lower id; the k
// first to s_sel / s_zsel.  tpe consecutive lanes share an expert, each counting over every tpe-th other
// expert.  The block's z are written before (with a barrier); ends with a barrier.
template <int kThreads>
__device__ __forceinline__ void rank_topk(const float* s_z, int E, int k, int* s_sel, float* s_zsel) {
  const int tid = threadIdx.x;
  int tpe = 1;
  while (tpe < 32 && tpe * 2 * E <= kThreads) tpe *= 2;
  const int per_pass = kThreads / tpe, part = tid % tpe;
  for (int e0 = 0; e0 < E; e0 += per_pass) {  // block-uniform
    const int e = e0 + tid / tpe;
    const bool valid = e < E;
    const float z = valid ? rank_key(s_z[e]) : 0.f;
    int r = 0;
    if (valid)
      for (int e2 = part; e2 < E; e2 += tpe) {
        const float z2 = rank_key(s_z[e2]);
        r += (z2 > z) || (z2 == z && e2 < e);
      }
    for (int off = tpe >> 1; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
    if (valid && part == 0 && r < k) {
      s_sel[r] = e;
      s_zsel[r] = s_z[e];
    }
  }
  __syncthreads();
}

// softmax over the chosen, by one warp: lane j < k holds exp(z_j - z_0); fixed shuffle-tree sum
__device__ __forceinline__ void softmax_topk(const Dev& d, int t, int k, const int* s_sel, const float* s_zsel) {
  const int lane = threadIdx.x & 31;
  const float ex = lane < k ? expf(s_zsel[lane] - s_zsel[0]) : 0.f;
  float den = ex;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
  if (lane < k) {
    const size_t at = (size_t)t * k + lane;
    d.idx[at] = s_sel[lane];
    d.g[at] = ex / den;
    if (d.idx_out) d.idx_out[at] = s_sel[lane];
    if (d.w_out) d.w_out[at] = ex / den;
  }
}

__global__ void __launch_bounds__(kThreadsR)
    k_router(Dev d, const float* __restrict__ x, const float* __restrict__ wr, const float* __restrict__ bias, int T,
             int layer, int fuse_resolve, float* __restrict__ x_copy, int nc) {
  extern __shared__ __align__(16) float s_x[];  // the token's x, read once per block
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int t = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = d.H, E = d.E, k = d.k, S = d.S_active;
  const int epc = (E + nc - 1) / nc;
  // this warp's first expert and its first W chunk, requested before x is staged
  const int e0 = rank * epc, e1 = min(E, e0 + epc);
  const int wpe = epc >= kWarpsR ? 1 : kWarpsR / epc;  // warps per expert
  const int ew = kWarpsR / wpe;                         // experts per pass
  const int part = warp % wpe, n4 = H / 4;
  // a programmatic launch may begin during the previous kernel: nothing above touched global memory
  pdl_wait();
  float4 pre[kChunk];
  if (e0 + warp / wpe < e1 && warp / wpe < ew) w_preload(wr + (size_t)(e0 + warp / wpe) * H, n4, part * 32 + lane, wpe * 32, pre);
  {  // x may be pinned host memory read over the CPU-GPU link: once per block
    const float4* x4 = reinterpret_cast<const float4*>(x + (size_t)t * H);
    float4* sx4 = reinterpret_cast<float4*>(s_x);
    for (int i = threadIdx.x; i < H / 4; i += kThreadsR) {
      const float4 v = x4[i];
      sx4[i] = v;
      if (x_copy && cluster_rank_zero()) reinterpret_cast<float4*>(x_copy + (size_t)t * H)[i] = v;  // for the FFN
    }
  }
  __syncthreads();

  __shared__ __align__(16) float s_z[kMaxExperts];  // block 0: every logit (the blocks store theirs)
  __shared__ float s_ps[kWarpsR], s_pc[kWarpsR];  // each warp's compensated partial
  __shared__ int s_sel[kMaxTopK];
  __shared__ float s_zsel[kMaxTopK];
  __shared__ int s_slot_of[kMaxExperts];
  __shared__ int s_expert_of[kMaxExperts];
  __shared__ uint64_t s_lastuse[kMaxExperts];
  __shared__ int s_uslot[kMaxTopK];

  // block 0 of a one-token call: start loading the layer's cache state now (used after the logits)
  const bool resolve = fuse_resolve && rank == 0;
  int pre_slot[kPre], pre_exp[kPre];
  uint64_t pre_last[kPre], clock0 = 0;
  if (resolve) {
    const int32_t* g_slot_of = d.slot_of + (size_t)layer * E;
    const int32_t* g_expert_of = d.expert_of + (size_t)layer * d.S_alloc;
    const uint64_t* g_last = d.last_use + (size_t)layer * d.S_alloc;
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
      const int e = tid + i * kThreadsR;
      pre_slot[i] = e < E ? g_slot_of[e] : -1;
      pre_exp[i] = e < S ? g_expert_of[e] : -1;
      pre_last[i] = e < S ? g_last[e] : 0;
    }
    if (tid == 0) clock0 = d.clock[layer];
  }

  float* z0 = rank == 0 ? s_z : cluster.map_shared_rank(s_z, 0);  // block 0's logits
  for (int eb = e0; eb < e1; eb += ew) {  // block-uniform passes
    const int e = eb + warp / wpe;
    float ps = 0.f, pc = 0.f;
    if (e < e1 && warp / wpe < ew) {
      if (eb != e0) w_preload(wr + (size_t)e * H, n4, part * 32 + lane, wpe * 32, pre);
      logit_part(wr + (size_t)e * H, s_x, n4, part * 32 + lane, wpe * 32, pre, ps, pc);
    }
    if (lane == 0) {
      s_ps[warp] = ps;
      s_pc[warp] = pc;
    }
    __syncthreads();
    if (lane == 0 && part == 0 && e < e1 && warp / wpe < ew) {
      float zs = s_ps[warp], zc = s_pc[warp];
      for (int p = 1; p < wpe; ++p) pair_add(zs, zc, s_ps[warp + p], s_pc[warp + p]);
      float z = __fadd_rn(zs, zc);
      if (bias) z = __fadd_rn(z, bias[(size_t)t * E + e]);
      z0[e] = z;  // distributed shared memory store into block 0
    }
    __syncthreads();
  }
  if (resolve) {  // the prefetched cache state into shared memory (the loads have long landed)
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
      const int e = tid + i * kThreadsR;
      if (e < E) s_slot_of[e] = pre_slot[i];
      if (e < S) {
        s_expert_of[e] = pre_exp[i];
        s_lastuse[e] = pre_last[i];
      }
    }
  }
  // the logits are stored: the expert FFN (a programmatic launch) may start its prologue
  pdl_trigger();
  // every block's logits stores, before block 0 reads them; the other blocks leave
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  if (rank != 0) return;
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  rank_topk<kThreadsR>(s_z, E, k, s_sel, s_zsel);
  if (warp == 0) softmax_topk(d, t, k, s_sel, s_zsel);
  if (!resolve) return;

  // One token per call: the k chosen experts are distinct, so the accesses are the chosen
  // experts in rank order, all in one wave.
  if (tid == 0) d.info[2] = 0;
  __syncthreads();
  if (warp == 0) lru_warp(d, layer, k, s_sel, s_slot_of, s_expert_of, s_lastuse, s_uslot, __shfl_sync(0xffffffffu, clock0, 0));
  __syncthreads();
  if (tid < k) {  // one assignment per distinct expert: t = 0, j = u
    d.pos_slot[tid] = s_uslot[tid];
    d.asg[tid] = tid;
    d.asg_off[tid] = tid;
  }
  if (tid == 0) d.asg_off[k] = k;
  int32_t* g_slot_of = d.slot_of + (size_t)layer * E;
  int32_t* g_expert_of = d.expert_of + (size_t)layer * d.S_alloc;
  uint64_t* g_last = d.last_use + (size_t)layer * d.S_alloc;
  for (int e = tid; e < E; e += kThreadsR) g_slot_of[e] = s_slot_of[e];
  for (int q = tid; q < S; q += kThreadsR) {
    g_expert_of[q] = s_expert_of[q];
    g_last[q] = s_lastuse[q];
  }
}


// ---------------------------------------------------------------- many tokens per call
// Exact (Dot2) logits are needed only for the experts that can be chosen.  k_logits_fp32 computes every
// logit as a plain fp32 dot product (one FMA per product instead of Dot2's ten operations), k_topk_exact
// bounds each one's error, keeps the experts whose bound reaches the k-th largest logit, and computes
// those (k and the rare close call) with the compensated dot product, which alone decides: the routing
// and the weights are those of exact logits for every expert.  Bound: fp32 issue of the plain product (4096
// tokens, 128 experts, hidden 2048: 62 us), then the exact ones' re-reading of k rows of W_r per token (80
// us); compensated dot products for every expert took 385 + 31 us there.
//
// k_logits_fp32: block (expert tile, token tile, K split) computes a 64-token x 16 J-expert tile over its
// range of H, from shared-memory tiles of x and W_r that cp.async fills 16 columns at a time
// (double-buffered).  Thread (ty, tx) owns tokens 4 ty .. + 3 and experts tx + 16 j.  Columns are taken two
// at a time with f32x2 FMAs (one running sum for the even, one for the odd columns).  The blocks of the
// first token tile also sum the squares of the rows of W_r.
constexpr int kTT = 64, kHC = 16, kThreadsT = 256;
constexpr int kPadT = kHC + 4;  // shared row stride in floats: the 8 rows of a load phase use all banks

__device__ __forceinline__ uint64_t f2_op_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float2 f2_split(uint64_t a) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
  return make_float2(lo, hi);
}

__device__ __forceinline__ void cp_async16_zfill(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}

template <int J>
__global__ void __launch_bounds__(kThreadsT, 2)
    k_logits_fp32(const float* __restrict__ x, const float* __restrict__ wr, int T, int E, int H, int cps,
                  float* __restrict__ part, float* __restrict__ wsq) {
  constexpr int kTE = 16 * J;
  __shared__ __align__(16) float s_x[2][kTT][kPadT];
  __shared__ __align__(16) float s_w[2][kTE][kPadT];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int e0 = (int)blockIdx.x * kTE, t0 = (int)blockIdx.y * kTT;
  const int c0 = (int)blockIdx.z * cps, c1 = min(H / kHC, c0 + cps);
  // one 16-byte piece of the x tile and J / 4 of the W tile per thread; rows past T or E read zeros
  auto load = [&](int ch, int buf) {
    {
      const int r = tid >> 2, q = tid & 3, t = t0 + r;
      cp_async16_zfill(&s_x[buf][r][4 * q], x + (size_t)min(t, T - 1) * H + ch * kHC + 4 * q, t < T);
    }
#pragma unroll
    for (int i = 0; i < J / 4; ++i) {
      const int id = tid + i * kThreadsT, r = id >> 2, q = id & 3, e = e0 + r;
      cp_async16_zfill(&s_w[buf][r][4 * q], wr + (size_t)min(e, E - 1) * H + ch * kHC + 4 * q, e < E);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  pdl_trigger();
  pdl_wait();
  uint64_t S[4][J];  // [token][expert]: (even-column, odd-column) sums
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int j = 0; j < J; ++j) S[a][j] = 0;
  float sq = 0.f;  // this thread's part of its W row's square (row tid * J / 16, all columns / (16 / J))
  if (c0 < c1) load(c0, 0);
  for (int ch = c0; ch < c1; ++ch) {
    const int buf = (ch - c0) & 1;
    if (ch + 1 < c1) {
      load(ch + 1, buf ^ 1);  // that buffer was released by the barrier ending the previous chunk
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
#pragma unroll
    for (int k4 = 0; k4 < kHC; k4 += 4) {
      ulonglong2 xv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) xv[a] = *reinterpret_cast<const ulonglong2*>(&s_x[buf][4 * ty + a][k4]);
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&s_w[buf][tx + 16 * j][k4]);
#pragma unroll
        for (int a = 0; a < 4; ++a) S[a][j] = f2_op_fma(w.x, xv[a].x, S[a][j]);
#pragma unroll
        for (int a = 0; a < 4; ++a) S[a][j] = f2_op_fma(w.y, xv[a].y, S[a][j]);
      }
    }
    if (blockIdx.y == 0) {
      const float* w = &s_w[buf][tid * J / 16][(tid % (16 / J)) * J];
#pragma unroll
      for (int q = 0; q < J; ++q) sq = fmaf(w[q], w[q], sq);
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int t = t0 + 4 * ty + a;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int e = e0 + tx + 16 * j;
      const float2 v = f2_split(S[a][j]);
      if (t < T && e < E) part[((size_t)blockIdx.z * T + t) * E + e] = v.x + v.y;
    }
  }
  if (blockIdx.y == 0) {
#pragma unroll
    for (int o = 1; o < 16 / J; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    const int e = e0 + tid * J / 16;
    if (tid % (16 / J) == 0 && e < E) wsq[(size_t)blockIdx.z * E + e] = sq;
  }
}

constexpr int kThreadsTop = 256;

// One block per token.  The K splits' sums of an expert are added by P threads (as many as fit, eight loads
// in flight).  Then, with a the fp32 logit and |a - exact| <= B:
//   a sum of H products in two chains, added over the splits, is off by less than
//   (H / 2 + splits + 8) 2^-24 sum |x w| <= (H + 64) 2^-24 |x|_2 |w|_2 and H 2^-148 where products underflow;
//   a squared norm summed in fp32 may be short by 2^-150 for each of its H terms where squares underflow
//   (values below 2^-63 or so), and is taken H 2^-149 longer;
//   2^-21 of the logit's and the bias's magnitude covers the roundings after it (to fp32, the bias added).
// L = the k-th largest of a - B is at or below the k-th largest exact logit, so an expert with a + B < L is
// not chosen, not even on a tie.  The others are computed exactly, one warp each.  A bound that is not a
// number (overflow) keeps its expert.  Logits that are known exactly are not computed again, as they tie in
// numbers: those of a token that is zero (a padding row; every expert was a candidate, 4096 such tokens over
// 128 experts took 622 us in the router, now 102) are its biases, and a bias of -infinity is its expert's.
__global__ void __launch_bounds__(kThreadsTop, 4)
    k_topk_exact(Dev d, const float* __restrict__ x, const float* __restrict__ wr, const float* __restrict__ part,
                 const float* __restrict__ wsq, const float* __restrict__ bias, int T, int ks) {
  extern __shared__ __align__(16) float s_x[];  // the token's x
  __shared__ float s_a[kMaxExperts], s_b[kMaxExperts];  // a - B, a + B; later the exact logits in s_a
  __shared__ float s_p[2][kThreadsTop], s_n[kThreadsTop / 32];
  __shared__ int s_cand[kMaxExperts], s_sel[kMaxTopK], s_nc, s_all;
  __shared__ float s_zs[kMaxTopK], s_l;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, t = blockIdx.x, E = d.E, k = d.k, H = d.H;
  int P = 1;
  while (P * 2 <= ks && P * 2 * E <= kThreadsTop) P *= 2;
  const int per = kThreadsTop / P, p = tid / per;
  pdl_trigger();
  pdl_wait();
  float nx = 0.f;
  bool some = false;  // a value that is not zero
  {
    const float4* x4 = reinterpret_cast<const float4*>(x + (size_t)t * H);
    for (int i = tid; i < H / 4; i += kThreadsTop) {
      const float4 v = x4[i];
      reinterpret_cast<float4*>(s_x)[i] = v;
      nx += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
      some |= v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nx += __shfl_xor_sync(0xffffffffu, nx, o);
  if (lane == 0) s_n[warp] = nx;
  if (tid == 0) s_nc = s_all = 0;
  const bool zero = !__syncthreads_or(some);
  nx = 0.f;
#pragma unroll
  for (int i = 0; i < kThreadsTop / 32; ++i) nx += s_n[i];
  // (factors of 1.01: the roundings of the norms and of this expression)
  const float under = (float)H * 0x1p-149f;
  const float scale = (float)(H + 64) * 0x1p-24f * 1.01f * sqrtf(nx + under) * 1.01f;
  for (int e0 = 0; e0 < E; e0 += per) {  // block-uniform
    const int e = e0 + tid % per;
    float a = 0.f, w2 = 0.f;
    if (e < E) {
      for (int s0 = p; s0 < ks; s0 += 8 * P) {
        float q[8], r[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (s0 + u * P < ks) {
            q[u] = part[((size_t)(s0 + u * P) * T + t) * E + e];
            r[u] = wsq[(size_t)(s0 + u * P) * E + e];
          }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (s0 + u * P < ks) {
            a += q[u];
            w2 += r[u];
          }
      }
    }
    s_p[0][tid] = a;
    s_p[1][tid] = w2;
    __syncthreads();
    if (p == 0 && e < E) {
      for (int i = 1; i < P; ++i) {
        a += s_p[0][tid + i * per];
        w2 += s_p[1][tid + i * per];
      }
      const float b = bias ? bias[(size_t)t * E + e] : 0.f;
      const float B0 = scale * sqrtf(w2 + under) + 0x1p-21f * fabsf(a) + (float)H * 0x1p-148f;
      if (b == -INFINITY && fabsf(a) + B0 < INFINITY) {  // an expert masked out: its logit is exactly that
        s_a[e] = s_b[e] = b;
      } else {
        const float B = zero ? 0.f : B0 + 0x1p-21f * fabsf(b);
        s_a[e] = (a + b) - B;
        s_b[e] = (a + b) + B;
        if (!(fabsf(s_b[e]) < INFINITY)) s_all = 1;
      }
    }
    __syncthreads();
  }
  {  // L: the a - B of rank k - 1 (rank by counting, ties to the lower id)
    int tpe = 1;
    while (tpe < 32 && tpe * 2 * E <= kThreadsTop) tpe *= 2;
    const int per_pass = kThreadsTop / tpe, q = tid % tpe;
    for (int e0 = 0; e0 < E; e0 += per_pass) {  // block-uniform
      const int e = e0 + tid / tpe;
      const float z = e < E ? s_a[e] : 0.f;
      int r = 0;
      if (e < E)
        for (int e2 = q; e2 < E; e2 += tpe) {
          const float z2 = s_a[e2];
          r += (z2 > z) || (z2 == z && e2 < e);
        }
      for (int off = tpe >> 1; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
      if (e < E && q == 0 && r < k) {
        if (r == k - 1) s_l = z;
        s_sel[r] = e;  // the choice where x is zero
        s_zs[r] = z;
      }
    }
  }
  __syncthreads();
  const float L = s_l;
  const bool all = s_all != 0;
  if (zero && !all) {
    if (warp == 0) softmax_topk(d, t, k, s_sel, s_zs);
    return;
  }
  for (int e = tid; e < E; e += kThreadsTop)
    if (all || !(s_b[e] < L)) s_cand[atomicAdd(&s_nc, 1)] = e;
  __syncthreads();
  const int nc = s_nc;
  for (int c = warp; c < nc; c += kThreadsTop / 32) {
    const float* w = wr + (size_t)s_cand[c] * H;
    const float4* w4 = reinterpret_cast<const float4*>(w);
    const float4* x4 = reinterpret_cast<const float4*>(s_x);
    float zs = 0.f, zc = 0.f;
    for (int q0 = lane; q0 < H / 4; q0 += 4 * 32) {  // four loads in flight: few registers, many blocks
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (q0 + u * 32 < H / 4) v[u] = ld_hint(w4 + q0 + u * 32, l2_evict_last());
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (q0 + u * 32 < H / 4) {
          const float4 xv = x4[q0 + u * 32];
          dot2(zs, zc, v[u].x, xv.x);
          dot2(zs, zc, v[u].y, xv.y);
          dot2(zs, zc, v[u].z, xv.z);
          dot2(zs, zc, v[u].w, xv.w);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pair_add(zs, zc, __shfl_xor_sync(0xffffffffu, zs, o), __shfl_xor_sync(0xffffffffu, zc, o));
    if (lane == 0) {
      float z = __fadd_rn(zs, zc);
      if (bias) z = __fadd_rn(z, bias[(size_t)t * E + s_cand[c]]);
      s_a[c] = z;  // (the bounds in s_a are no longer read)
    }
  }
  __syncthreads();
  for (int c = tid; c < nc; c += kThreadsTop) {  // rank the candidates, ties to the lower id
    const float z = rank_key(s_a[c]);
    const int e = s_cand[c];
    int r = 0;
    for (int c2 = 0; c2 < nc; ++c2) {
      const float z2 = rank_key(s_a[c2]);
      r += (z2 > z) || (z2 == z && s_cand[c2] < e);
    }
    if (r < k) {
      s_sel[r] = e;
      s_zs[r] = s_a[c];
    }
  }
  __syncthreads();
  if (warp == 0) softmax_topk(d, t, k, s_sel, s_zs);
}

// K splits for T tokens.  At least about kTiledBlocks blocks (two per SM) when the tiles alone are fewer;
// from there to twice as many splits, the number whose busiest SM walks the fewest chunks: 64 token tiles
// (4096 tokens) in 5 splits left 16 of 320 blocks to a round of their own, in 7 the call is 17 us shorter.
// Constants (of a 152-SM part), not the device's count, so that the planner, which runs without a GPU,
// sizes the scratch exactly as the context does.
constexpr int kTiledSms = 152, kTiledBlocks = 2 * kTiledSms, kMaxSplits = 64;
int tile_experts(int E) { return E > 64 ? 128 : 64; }
int tiled_splits(int T, int E, int H) {
  const int tiles = ((T + kTT - 1) / kTT) * ((E + tile_experts(E) - 1) / tile_experts(E));
  const int nch = H / kHC;
  const int want = std::min(kMaxSplits, std::max(1, (kTiledBlocks + tiles - 1) / tiles));
  int best = 0, best_cost = 0;
  for (int w = want; w <= std::min(kMaxSplits, 2 * want); ++w) {
    const int cps = (nch + w - 1) / w, ks = (nch + cps - 1) / cps;
    const int cost = (tiles * ks + kTiledSms - 1) / kTiledSms * cps;
    if (best == 0 || cost < best_cost) best = ks, best_cost = cost;
  }
  return best;
}

cudaError_t launch_router_tiled(const Dev& d, const float* x, const float* wr, const float* bias, int T,
                                cudaStream_t s) {
  const int ks = tiled_splits(T, d.E, d.H), te = tile_experts(d.E);
  const int nch = d.H / kHC, cps = (nch + ks - 1) / ks;
  float* wsq = d.zpart + (size_t)ks * T * d.E;
  const dim3 grid((d.E + te - 1) / te, (T + kTT - 1) / kTT, ks);
  cudaError_t e = te == 128 ? launch_pdl(true, k_logits_fp32<8>, grid, dim3(kThreadsT), 0, s, x, wr, T, d.E, d.H, cps, d.zpart, wsq)
                            : launch_pdl(true, k_logits_fp32<4>, grid, dim3(kThreadsT), 0, s, x, wr, T, d.E, d.H, cps, d.zpart, wsq);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)d.H * sizeof(float);
  if (smem > 24 * 1024 &&
      (e = cudaFuncSetAttribute(k_topk_exact, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return e;
  return launch_pdl(true, k_topk_exact, dim3(T), dim3(kThreadsTop), smem, s, d, x, wr, (const float*)d.zpart,
                    (const float*)wsq, bias, T, ks);
}

}  // namespace

size_t router_part_floats(int T_max, int E, int H) {
  size_t most = 0;
  for (int t0 = 0; t0 < T_max; t0 += kTT) {  // the splits depend on the number of token tiles only
    const int T = std::min(t0 + kTT, T_max);
    if (T < kTiledMinT) continue;
    const size_t n = (size_t)tiled_splits(T, E, H) * ((size_t)T + 1) * E;
    if (n > most) most = n;
  }
  return most;
}

cudaError_t launch_router(const Dev& d, const float* x, const float* wr, const float* bias, int T, int layer,
                          cudaStream_t s, float* x_copy) {
  if (T >= kTiledMinT) return launch_router_tiled(d, x, wr, bias, T, s);
  const size_t smem = (size_t)d.H * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(k_router, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreadsR);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // cluster size: 16 where the GPU can hold such a cluster (asked once), else the portable 8
  static int nc = 0;
  if (nc == 0) {
    nc = 8;
    if (cudaFuncSetAttribute(k_router, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      cfg.gridDim = dim3(16, 1);
      attr[0].val.clusterDim.x = 16;
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, k_router, &cfg) == cudaSuccess && clusters >= 1) nc = 16;
    }
    cudaGetLastError();
  }
  cfg.gridDim = dim3(nc, T);
  attr[0].val.clusterDim.x = nc;
  // programmatic: the launch may begin while the previous kernel of the stream finishes (the
  // kernel waits for it before touching global memory); plain where the driver refuses that
  static bool pdl_ok = true;
  if (pdl_ok) {
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, k_router, d, x, wr, bias, T, layer, T == 1 ? 1 : 0, x_copy, nc);
    if (e == cudaSuccess) return e;
    cudaGetLastError();
    pdl_ok = false;
    cfg.numAttrs = 1;
  }
  e = cudaLaunchKernelEx(&cfg, k_router, d, x, wr, bias, T, layer, T == 1 ? 1 : 0, x_copy, nc);
  return e;
}

}  // namespace mf
