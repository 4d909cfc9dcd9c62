// Slot resolve: the per-layer bounded expert cache (section "Native Serving Path": a miss
// materialises the expert block into an available slot and updates the route-to-slot
// metadata).
//
// One block of 1024 threads per call.  Steps:
//  1. the distinct experts of the call's T*k routes, in (token, rank) first-occurrence
//     order (or, with MF_ORDER_RESIDENT_FIRST, the resident ones first), and for each the list
//     of assignments t*k+j it serves;
//  2. least-recently-used replacement over those accesses in waves of S: all accesses at once where
//     they all hit or where no miss can take a slot that a later access still hits (lru_parallel),
//     else one after the other (lru_block);
//  3. counters (accesses, hits, misses, evictions, bytes = misses * payload) and the
//     access record of the call.
// Each warp counts its routes into its own copy of the per-expert counters, so that a hot
// expert's counter (skewed routing) is not contended across warps.  Everything here is latency: the
// scans and the rank counts use every thread (several per expert where E is small), and nothing but
// the rare ordered walk runs on one thread: 7 us for 64 tokens x 8 routes over 128 experts (20-34 with the
// order kept by a walk over a linked list), 25 us for 4096 tokens (55).
// With one token per call the router's last block does this itself (mf_router.cu).
#include "mf_lru.cuh"
#include "mf_stream.cuh"

namespace mf {
namespace {

constexpr int kThreadsRes = 1024;
static_assert(kThreadsRes >= kMaxExperts, "one thread per expert, access and slot");
constexpr int kRouteChunk = 8;  // routes a thread loads before using them (their loads overlap)
constexpr int kNone = 0x7fffffff;

// histogram copies: one per warp where E allows (no two warps update the same counter), fewer
// for large E (shared memory)
__host__ __device__ inline int n_segments(int E) {
  const int n = 8192 / E;
  return n < 1 ? 1 : (n > kThreadsRes / 32 ? kThreadsRes / 32 : n);
}

// threads that share one of n items (a power of two, at most a warp)
__device__ __forceinline__ int threads_per(int n) {
  int t = 1;
  while (t < 32 && t * 2 * n <= kThreadsRes) t *= 2;
  return t;
}

// Exclusive prefix sum of v over the block's threads; *total (shared) gets the sum.  s_w: 32 words.
__device__ __forceinline__ uint64_t block_scan(uint64_t v, uint64_t* s_w, uint64_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const uint64_t w0 = s_w[lane];
    uint64_t w = w0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    s_w[lane] = w - w0;
    if (lane == 31) *total = w;
  }
  __syncthreads();
  const uint64_t r = s_w[warp] + x - v;
  __syncthreads();  // s_w may be reused
  return r;
}

// r(i) = number of j < n with less(j, i), for every i < n at once: threads_per(n) lanes per item, each
// counting over every that-many-th j.  put(i, r) is called by one thread per item.
template <class Less, class Put>
__device__ __forceinline__ void rank_all(int n, Less less, Put put) {
  const int tpe = threads_per(n), per = kThreadsRes / tpe, p = threadIdx.x % tpe;
  for (int i0 = 0; i0 < n; i0 += per) {  // block-uniform
    const int i = i0 + threadIdx.x / tpe;
    int r = 0;
    if (i < n)
      for (int j = p; j < n; j += tpe) r += less(j, i);
    for (int o = tpe >> 1; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (i < n && p == 0) put(i, r);
  }
}

// The record of access u (expert e, slot s) by the thread that owns it.
__device__ __forceinline__ void record(const Dev& d, int layer, int u, int e, int s, bool miss) {
  d.uniq[u] = e;
  d.uslot[u] = s;
  d.umiss[u] = miss ? 1 : 0;
  const size_t o = (size_t)layer * d.E + u;
  d.tr_expert[o] = e;
  d.tr_slot[o] = s;
  d.tr_hit[o] = miss ? 0 : 1;
}

// One thread: the call's totals.
__device__ __forceinline__ void totals(const Dev& d, int layer, int U, uint64_t clock, uint64_t misses,
                                       uint64_t evictions) {
  d.clock[layer] = clock + (uint64_t)U;
  unsigned long long* st = reinterpret_cast<unsigned long long*>(d.stats + (size_t)layer * 5);
  atomicAdd(st + 0, (unsigned long long)U);
  atomicAdd(st + 1, (unsigned long long)(U - misses));
  atomicAdd(st + 2, (unsigned long long)misses);
  atomicAdd(st + 3, (unsigned long long)evictions);
  atomicAdd(st + 4, (unsigned long long)(misses * d.lay.canonical));
  d.info[0] = U;
  d.info[1] = (U + d.S_active - 1) / d.S_active;
  d.tr_n[layer] = U;
}

struct LruMem {  // shared memory of the replacement
  int *slot_of, *uniq, *uslot, *mr;          // [E] expert -> slot; accesses: expert, slot, misses before
  int *expert_of, *order, *rank, *base, *acc;  // [S] slots: expert; by last use; place in that order; victims; accessed
  uint64_t* last;                             // [S]
  uint64_t *w, *tot;                          // block_scan's words
};

// Every access of the call decided at once; false (with nothing written) where that is not known to
// give the order-by-order decisions.
//
// Let the accesses that find their expert resident at the call's start all hit.  Then the m-th miss
// takes the m-th entry of the list
//   free slots (lowest first), the occupied slots that no access of the call hits (oldest use first),
//   then the slots of the accesses themselves in access order (a call of several waves),
// because replacement always takes the least recently used slot and an accessed slot is younger than
// every one not accessed yet.  The assumption holds if for each such access u, with E_u evictions
// before it (misses before it less the free slots), p slots of older last use and A of those accessed
// before u, E_u <= p - A: that many older slots that no access has touched stand in front of it.
__device__ __forceinline__ bool lru_parallel(const Dev& d, int layer, int U, const LruMem& m, uint64_t clock) {
  const int S = d.S_active, tid = threadIdx.x;
  const int e = tid < U ? m.uniq[tid] : 0;
  const int own = tid < U ? m.slot_of[e] : -1;  // its slot at the start
  const bool miss = tid < U && own < 0;
  const int n_miss = __syncthreads_count(miss);
  if (n_miss == 0) {  // nothing is placed: access u takes clock value clock + u + 1
    if (tid < U) {
      d.last_use[(size_t)layer * d.S_alloc + own] = clock + (uint64_t)tid + 1;
      record(d, layer, tid, e, own, false);
    }
    if (tid == 0) totals(d, layer, U, clock, 0, 0);
    return true;
  }
  const bool occ = tid < S && m.expert_of[tid] >= 0;
  const int n_occ = __syncthreads_count(occ), n_free = S - n_occ;
  if (tid < S) m.acc[tid] = 0;
  if (tid < U) m.uslot[tid] = own;
  // occupied slots by (last use, slot), free ones by slot: place r of its class
  rank_all(
      S,
      [&](int j, int i) {
        const bool oj = m.expert_of[j] >= 0;
        if (oj != (m.expert_of[i] >= 0)) return 0;
        return oj ? (int)(m.last[j] < m.last[i] || (m.last[j] == m.last[i] && j < i)) : (int)(j < i);
      },
      [&](int i, int r) {
        if (m.expert_of[i] >= 0) {
          m.order[r] = i;
          m.rank[i] = r;
        } else {
          m.base[r] = i;
        }
      });
  const int mu = (int)block_scan(miss ? 1 : 0, m.w, m.tot);  // misses before access tid
  if (tid < U) m.mr[tid] = mu;
  __syncthreads();
  bool fine = true;
  rank_all(
      U,
      [&](int v, int u) {  // A of access u
        const int su = m.uslot[u], sv = m.uslot[v];
        return (int)(su >= 0 && v < u && sv >= 0 && m.rank[sv] < m.rank[su]);
      },
      [&](int u, int a) {
        const int su = m.uslot[u];
        if (su >= 0) {
          fine = max(0, m.mr[u] - n_free) <= m.rank[su] - a && fine;
          m.acc[su] = 1;
        }
      });
  if (!__syncthreads_and(fine)) return false;
  // the list's second part: slots not accessed, in order of last use
  const bool never = tid < n_occ && !m.acc[m.order[tid]];
  const int nv = (int)block_scan(never ? 1 : 0, m.w, m.tot);
  if (never) m.base[n_free + nv] = m.order[tid];
  const int F = n_free + (int)*m.tot;
  __syncthreads();
  int slot = own;
  if (miss) {
    int q = mu;
    while (q >= F) {  // the slot of access q - F: its own if that hit, else what it took
      const int s = m.uslot[q - F];
      if (s >= 0) {
        slot = s;
        break;
      }
      q = m.mr[q - F];
    }
    if (q < F) slot = m.base[q];
  }
  int32_t* g_slot_of = d.slot_of + (size_t)layer * d.E;
  int32_t* g_expert_of = d.expert_of + (size_t)layer * d.S_alloc;
  uint64_t* g_last = d.last_use + (size_t)layer * d.S_alloc;
  if (tid >= n_free && tid < min(n_miss, F)) g_slot_of[m.expert_of[m.base[tid]]] = -1;  // evicted, not accessed
  if (tid < U) {
    if (F + tid >= n_miss) {  // the last access of its slot in this call
      g_expert_of[slot] = e;
      g_slot_of[e] = slot;
      g_last[slot] = clock + (uint64_t)tid + 1;
    } else {
      g_slot_of[e] = -1;  // evicted again within the call
    }
    record(d, layer, tid, e, slot, miss);
    const int w = tid / S;
    if (miss) d.miss_list[w * S + mu - m.mr[w * S]] = tid;
    if (tid % S == 0) d.info[2 + w] = (tid + S < U ? m.mr[tid + S] : n_miss) - mu;
  }
  if (tid == 0) totals(d, layer, U, clock, (uint64_t)n_miss, (uint64_t)max(0, n_miss - n_free));
  return true;
}

// Block 0 resolves; blocks 1 .. T, where launched, split token blockIdx.x - 1 of x into the pieces the
// streaming expert kernels read (their work hides behind block 0's latency).
__global__ void __launch_bounds__(kThreadsRes, 1) k_resolve(Dev d, int layer, int T, const float* __restrict__ x) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (blockIdx.x > 0) {
    pdl_trigger();
    pdl_wait();
    float* s_m = reinterpret_cast<float*>(smem);
    if (d.qtype == dq::kQ8)
      split_token<dq::kQ8, kThreadsRes>(d, x, (int)blockIdx.x - 1, s_m);
    else
      split_token<dq::kQ4, kThreadsRes>(d, x, (int)blockIdx.x - 1, s_m);
    return;
  }
  const int E = d.E, k = d.k, S = d.S_active, n = T * k, NSEG = n_segments(E);
  uint64_t* s_last = reinterpret_cast<uint64_t*>(smem);           // [S_alloc]
  int* seg_first = reinterpret_cast<int*>(s_last + d.S_alloc);     // [NSEG][E] first route per copy
  int* seg_cnt = seg_first + NSEG * E;                              // [NSEG][E] routes per copy, then next position
  int* cnt = seg_cnt + NSEG * E;                                    // [E]
  int* s_slot_of = cnt + E;                                         // [E]
  int* s_uniq = s_slot_of + E;                                      // [E]
  int* s_uslot = s_uniq + E;                                        // [E]
  int* firstpos = s_uslot + E;                                      // [E], then misses before each access
  int* s_expert_of = firstpos + E;                                  // [S_alloc]
  int* s_order = s_expert_of + d.S_alloc;                           // [S_alloc] LRU scratch
  int* s_prev = s_order + d.S_alloc;                                // [S_alloc]
  int* s_next = s_prev + d.S_alloc;                                 // [S_alloc]
  int* s_acc = s_next + d.S_alloc;                                  // [S_alloc]
  __shared__ uint64_t s_w[32], s_tot;
  __shared__ int s_n[2];

  const int tid = threadIdx.x, nt = kThreadsRes;
  const int seg = (tid >> 5) % NSEG;
  int32_t* g_slot_of = d.slot_of + (size_t)layer * E;
  int32_t* g_expert_of = d.expert_of + (size_t)layer * d.S_alloc;
  uint64_t* g_last = d.last_use + (size_t)layer * d.S_alloc;

  for (int i = tid; i < NSEG * E; i += nt) {
    seg_first[i] = kNone;
    seg_cnt[i] = 0;
  }
  pdl_trigger();  // the next kernel's blocks may set up while this one works (they wait for its end)
  pdl_wait();     // the routes are complete
  const uint64_t clock = d.clock[layer];
  if (tid < E) s_slot_of[tid] = g_slot_of[tid];
  if (tid < S) {
    s_expert_of[tid] = g_expert_of[tid];
    s_last[tid] = g_last[tid];
  }
  {  // every wave the host may launch for this call starts with no misses and no work drawn
    const int acc_max = n < E ? n : E;
    if (tid < (acc_max + S - 1) / S) {
      d.info[2 + tid] = 0;
      d.sched[2 * tid] = d.sched[2 * tid + 1] = 0;
    }
  }
  __syncthreads();
  // routes c0 + j * nt of this thread (j < kRouteChunk) are loaded first, then counted into
  // this warp's histogram copy (a warp's 32 consecutive routes hold an expert at most once per
  // token, so few lanes share a counter)
  for (int c0 = tid; c0 < n; c0 += nt * kRouteChunk) {
    int ev[kRouteChunk];
#pragma unroll
    for (int j = 0; j < kRouteChunk; ++j) {
      const int p = c0 + j * nt;
      ev[j] = p < n ? d.idx[p] : 0;
    }
#pragma unroll
    for (int j = 0; j < kRouteChunk; ++j) {
      const int p = c0 + j * nt;
      if (p < n) {
        atomicMin(&seg_first[seg * E + ev[j]], p);
        atomicAdd(&seg_cnt[seg * E + ev[j]], 1);
      }
    }
  }
  __syncthreads();
  if (tid < E) {
    int f = kNone, c = 0;
#pragma unroll 8
    for (int g = 0; g < NSEG; ++g) {
      f = min(f, seg_first[g * E + tid]);
      c += seg_cnt[g * E + tid];
    }
    firstpos[tid] = f;
    cnt[tid] = c;
  }
  // access order: the distinct experts by first occurrence (resident ones first where asked)
  const bool res_first = d.order == MF_ORDER_RESIDENT_FIRST;
  const int U = __syncthreads_count(tid < E && firstpos[tid] != kNone);
  rank_all(
      E,
      [&](int j, int i) {
        const int fj = firstpos[j], fi = firstpos[i];
        if (fj == kNone) return 0;
        if (res_first) {
          const bool rj = s_slot_of[j] >= 0, ri = s_slot_of[i] >= 0;
          if (rj != ri) return (int)rj;
        }
        return (int)(fj < fi);
      },
      [&](int i, int r) {
        if (firstpos[i] != kNone) s_uniq[r] = i;
      });
  __syncthreads();
  {  // assignment offsets and 128-assignment blocks, in access order
    const int e = tid < U ? s_uniq[tid] : 0, c = tid < U ? cnt[e] : 0;
    const uint64_t p = block_scan((uint64_t)c << 32 | (uint64_t)((c + 127) / 128), s_w, &s_tot);
    if (tid < U) {
      d.asg_off[tid] = (int)(p >> 32);
      d.tb_off[tid] = (int)(uint32_t)p;
      int at = (int)(p >> 32);  // where each histogram copy's routes of this expert start
#pragma unroll 8
      for (int g = 0; g < NSEG; ++g) {
        const int c1 = seg_cnt[g * E + e];
        seg_cnt[g * E + e] = at;
        at += c1;
      }
    }
    if (tid == 0) {
      d.asg_off[U] = (int)(s_tot >> 32);
      d.tb_off[U] = (int)(uint32_t)s_tot;
    }
  }
  __syncthreads();
  for (int c0 = tid; c0 < n; c0 += nt * kRouteChunk) {  // the same walk as the count
    int ev[kRouteChunk];
#pragma unroll
    for (int j = 0; j < kRouteChunk; ++j) {
      const int p = c0 + j * nt;
      ev[j] = p < n ? d.idx[p] : 0;
    }
#pragma unroll
    for (int j = 0; j < kRouteChunk; ++j) {
      const int p = c0 + j * nt;
      if (p < n) d.asg[atomicAdd(&seg_cnt[seg * E + ev[j]], 1)] = p;
    }
  }

  const LruMem m = {s_slot_of, s_uniq, s_uslot, firstpos, s_expert_of, s_order, s_next, s_prev, s_acc, s_last, s_w, &s_tot};
  if (lru_parallel(d, layer, U, m, clock)) return;
  lru_block(d, layer, U, s_uniq, s_slot_of, s_expert_of, s_last, s_uslot, clock, s_order, s_prev, s_next, s_n);
  for (int e = tid; e < E; e += nt) g_slot_of[e] = s_slot_of[e];
  for (int q = tid; q < S; q += nt) {
    g_expert_of[q] = s_expert_of[q];
    g_last[q] = s_last[q];
  }
}

__global__ void k_reset(Dev d) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t nE = (size_t)d.L * d.E, nS = (size_t)d.L * d.S_alloc;
  if (i < nE) d.slot_of[i] = -1;
  if (i < nS) {
    d.expert_of[i] = -1;
    d.last_use[i] = 0;
  }
  if (i < (size_t)d.L) {
    d.clock[i] = 0;
    d.tr_n[i] = 0;
  }
  if (i < (size_t)d.L * 5) d.stats[i] = 0;
}

}  // namespace

size_t resolve_smem_bytes(const Dev& d) {
  return (size_t)d.S_alloc * sizeof(uint64_t) + ((size_t)2 * n_segments(d.E) + 5) * d.E * sizeof(int) +
         (size_t)5 * d.S_alloc * sizeof(int);
}

cudaError_t launch_resolve(const Dev& d, int layer, int T, const float* x, bool split, cudaStream_t s) {
  const size_t smem = resolve_smem_bytes(d);
  cudaError_t e = cudaFuncSetAttribute(k_resolve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(true, k_resolve, dim3(split ? 1 + T : 1), dim3(kThreadsRes), smem, s, d, layer, T, x);
}

cudaError_t launch_reset(const Dev& d, cudaStream_t s) {
  size_t n = (size_t)d.L * (d.E > d.S_alloc ? d.E : d.S_alloc);
  if (n < (size_t)d.L * 5) n = (size_t)d.L * 5;
  k_reset<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d);
  return cudaGetLastError();
}

}  // namespace mf
