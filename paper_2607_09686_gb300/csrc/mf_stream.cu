// Expert FFN of calls with a few to a few hundred tokens (2 <= T below the GEMM threshold): each
// wave's experts streamed once from their HBM slots through the warp-level tensor-core MMA.
//
//   gate/up:  h[a][r] = silu(Wg_e[r,:] . x_t) * (Wu_e[r,:] . x_t)     a = (t, j) routed to expert e
//   down:     part[a][c] = Wd_e[c,:] . h[a]                            then y = sum_j g part (combine)
// (SwiGLU experts with separate gate, up and down tensors, section "Native Serving Path".)
//
// Arithmetic.  A weight is d * q with q an integer of at most 8 bits: q is exact in bfloat16, so the
// codes go to the MMA as they are and no weight is rounded.  An activation is split exactly into three
// bfloat16 pieces (3 x 8 bits: the top bits of v, of the remainder, and the rest), so all 24 bits take
// part.  Each 32-weight block is two fresh fp32 accumulators, two m16n8k16 MMAs of the top pieces and four
// of the others; its scale is then applied to the block's sums as an FMA into the running sums, as the
// GGUF formats define (one scale per 32 weights).  The tensor cores round each MMA's sum towards zero, a
// bias of about 4e-8 of it where bits are lost: the top pieces' sums (16-bit products of values within
// 2^8 of each other) have nearly none to lose, and the others' sums are 2^8 smaller.  Every kSeg stages
// the running sums move to a second level, as a long chain of additions rounds at the size of its result.
// Against 64 bits the layer's error stays that of fp32 dot products (1.9e-7 of the result at hidden 2048;
// with one accumulator and one level 2.5e-7).
//
// Range.  A token's x is first scaled by the power of two 2^-e that brings its largest magnitude into
// [0.5, 1), which is exact; G and U below are the scaled products.  The activations are kept as
// G U sigmoid(2^e G), which is h 2^-2e, and the down sums are scaled back by 2^2e: no piece leaves the
// normal range of bfloat16 however small or large the inputs are.
//
// Work unit = (expert, 64 row records, up to 32 assignments): 128 weight rows, for gate/up 64 gate and
// the same 64 up rows, so that one thread ends with gate and up of the same output feature.  One CTA per
// SM takes units one after another from a counter (their costs differ with the assignments; dealt out in
// turn, the last SM ended 13 % after the average) and walks each in K chunks of 128 weights: a producer
// warp fills a ring of stages (TMA boxes of codes, 128-byte / 64-byte swizzled so that the fragment loads are
// conflict free; TMA boxes of scales; one bulk copy of 768 bytes per assignment's activation pieces), 16
// consumer warps take 16 rows x 64 K each (8 row groups x 2 K halves of the stage) and convert the codes
// in registers.  The halves' sums meet in shared memory once per unit.
//
// Bound: with few assignments per expert, HBM (the wave's quantised weights, read once per 32
// assignments of an expert); above about 16 assignments per expert the MMA (m16n8k16 runs at 2 cycles
// per SM).  The codes stay in registers between the conversion and the MMA, and the unit's rows are the
// MMA's M side, so a lightly loaded expert wastes only MMA columns, of which there are 8.
// Measured, 64 tokens over 128 Q8_0 experts of 2816 x 1408 (1.5 GB of weights when all are routed to): the
// whole call 450 us, where one warp per weight row on fp32 FMAs took 2090 (k_gateup 1330, down 735); 5
// tokens, 40 assignments over 2048 x 768: 65 us against 176.  At 64 tokens neither memory (copies alone
// 340 us) nor the MMA (31 % of its cycles) binds by itself but the latency of the 4 warps a scheduler has
// (half of its issue slots are filled): units of 8 or 16 columns with more stages (500, 464), copies by
// cp.async (521), a prefetch into L2 (501), other splits of rows and K over the warps (453-493) were slower.
#include "mf_stream.cuh"

namespace mf {
namespace {

using dq::codes_q4;
using dq::codes_q8;
using dq::kQ4;
using dq::kQ8;

constexpr int kRecs = 64;                       // row records per box
constexpr int kKC = kStreamK;                   // weights of K per stage
constexpr int kSeg = 4;                         // stages whose blocks are summed before they join the row's sum
constexpr int kSCols = kStreamCols;             // assignments per unit
constexpr int kSWarps = 16;                     // consumer warps
constexpr int kSThreads = (kSWarps + 1) * 32;   // + the producer warp
constexpr uint32_t kColBytes = kStreamChunkBytes;  // one assignment's pieces of one K chunk: 3 x 128 bf16
constexpr uint32_t kColStride = kColBytes + 64;  // in shared memory: neighbouring columns use different banks
constexpr int kSMaxStages = 8;
constexpr uint32_t kScaleBoxBytes = 16;         // 8 scales (256 weights) of a row
constexpr size_t kSSmem = 224 * 1024;

template <int QT>
struct SL {  // shared-memory stage: codes of two boxes, their scales, the activation pieces
  static constexpr uint32_t kRow = QT == kQ8 ? 128 : 64;  // code bytes of a row per stage
  static constexpr uint32_t kBox = kRecs * kRow;
  static constexpr uint32_t kOffScale = 2 * kBox;
  static constexpr uint32_t kOffB = kOffScale + 2 * kRecs * kScaleBoxBytes;
};

struct StreamCfg {
  int NS, cols;          // stages; assignments per unit (a multiple of 8, at most kSCols): no unit holds more,
                         // whatever the routes are, as a stage and the exchange buffers have room for these
  uint32_t stage;        // bytes per stage (a multiple of 1024)
  uint32_t off_bar, off_red, off_tab, total;
};

StreamCfg stream_cfg(const Dev& d, int T) {
  StreamCfg c;
  c.cols = T >= kSCols ? kSCols : (T + 7) & ~7;  // one unit per row block: a token takes an expert at most once
  const uint32_t a = d.qtype == MF_Q8_0 ? SL<kQ8>::kOffB : SL<kQ4>::kOffB;
  c.stage = (a + (uint32_t)c.cols * kColStride + 1023) & ~1023u;
  const uint32_t red = 2u * 8 * 32 * (c.cols / 8) * 16;  // two buffers of the K halves' sums
  const uint32_t tab = (uint32_t)(3 * (d.S_active + 1)) * 4;
  const uint32_t bars = (2 * kSMaxStages + 32) * 8 + kSMaxStages * 4;
  const uint32_t fixed = 1024 + bars + red + tab;
  const uint32_t ns = ((uint32_t)kSSmem - fixed) / c.stage;
  c.NS = ns > (uint32_t)kSMaxStages ? kSMaxStages : (int)ns;
  c.off_bar = (uint32_t)c.NS * c.stage;
  c.off_red = c.off_bar + bars;
  c.off_tab = c.off_red + red;
  c.total = c.off_tab + tab;
  return c;
}

__device__ __forceinline__ void tma_3d(void* dst, const CUtensorMap* tmap, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A fragments of one 32-weight block for the two K halves m = 0, 1 (k slots 2t, 2t + 1, 2t + 8, 2t + 9 of
// lane (g, t)): rows g of the box at `lo` and of the box at `hi`.  Q8_0: lane t holds weights 8t .. 8t + 7.
// Q4_0: its four code bytes hold weights 4t .. 4t + 3 (low nibbles) and 16 + 4t .. + 3 (high nibbles).
// The activation pieces are stored in the same order (stream_pos).
template <int QT>
__device__ __forceinline__ void load_a(const unsigned char* lo, const unsigned char* hi, uint32_t (&a)[2][4]) {
  if constexpr (QT == kQ8) {
    const uint2 u = *reinterpret_cast<const uint2*>(lo), v = *reinterpret_cast<const uint2*>(hi);
    codes_q8(u.x, a[0][0], a[0][2]);
    codes_q8(u.y, a[1][0], a[1][2]);
    codes_q8(v.x, a[0][1], a[0][3]);
    codes_q8(v.y, a[1][1], a[1][3]);
  } else {
    const uint32_t u = *reinterpret_cast<const uint32_t*>(lo), v = *reinterpret_cast<const uint32_t*>(hi);
    codes_q4(u & 0x0F0F0F0Fu, a[0][0], a[0][2]);
    codes_q4((u >> 4) & 0x0F0F0F0Fu, a[1][0], a[1][2]);
    codes_q4(v & 0x0F0F0F0Fu, a[0][1], a[0][3]);
    codes_q4((v >> 4) & 0x0F0F0F0Fu, a[1][1], a[1][3]);
  }
}

struct SUnit {
  int z, y, a0, n;  // slot plane, first row, first assignment (into asg), assignments
};

// One consumer warp's place in the ring, and its row group's exchange of the K halves' sums
struct SRing {
  int stage = 0, unit = 0;
  uint32_t phase = 0;
};

// kB consecutive 32-weight blocks of one stage, from block kb: the A fragments are converted once, every
// tile's MMAs go to fresh accumulators, the scales are applied in fp32.  All kB blocks form one straight
// line of code: their MMA chains overlap.
template <int QT, int NTL, int kB>
__device__ __forceinline__ void stream_blocks(const unsigned char* st, const unsigned char* bp, const uint32_t (&off)[2],
                                              int kb, const float (&dl)[2], const float (&dh)[2], float (&acc)[NTL][4]) {
  uint32_t a[kB][2][4];
#pragma unroll
  for (int b = 0; b < kB; ++b) load_a<QT>(st + off[b], st + SL<QT>::kBox + off[b], a[b]);
#pragma unroll
  for (int i = 0; i < NTL; ++i) {
#pragma unroll
    for (int b = 0; b < kB; ++b) {
      const unsigned char* bc = bp + (uint32_t)i * 8 * kColStride + (kb + b) * 64;
      const uint4 v0 = *reinterpret_cast<const uint4*>(bc);
      const uint4 v1 = *reinterpret_cast<const uint4*>(bc + kKC * 2);
      const uint4 v2 = *reinterpret_cast<const uint4*>(bc + kKC * 4);
      float c[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f};
      mma16816(c, a[b][0], v0.x, v0.y);  // top pieces
      mma16816(e, a[b][0], v2.x, v2.y);  // the others, the smallest first
      mma16816(c, a[b][1], v0.z, v0.w);
      mma16816(e, a[b][1], v2.z, v2.w);
      mma16816(e, a[b][0], v1.x, v1.y);
      mma16816(e, a[b][1], v1.z, v1.w);
      acc[i][0] = fmaf(dl[b], c[0] + e[0], acc[i][0]);
      acc[i][1] = fmaf(dl[b], c[1] + e[1], acc[i][1]);
      acc[i][2] = fmaf(dh[b], c[2] + e[2], acc[i][2]);
      acc[i][3] = fmaf(dh[b], c[3] + e[3], acc[i][3]);
    }
  }
}

// One unit's K loop and epilogue for one consumer warp (its first stage has arrived); NTL = MMA column
// tiles.  False once a bounded wait gave up.
template <int QT, int NT, int NTL>
__device__ __forceinline__ bool stream_unit(const Dev& d, const SUnit& un, unsigned char* smem, uint64_t* full,
                                            uint64_t* empty, uint64_t* rbar, const StreamCfg& f, float4* red, int KC,
                                            int nb, int rows, SRing& r, int warp, int lane) {
  using L = SL<QT>;
  const int grp = warp & 7, half = warp >> 3, g = lane >> 2, t = lane & 3;
  const int row = grp * 8 + g;  // record row inside each box
  uint32_t off[2];  // this lane's codes of its two blocks inside a box: the TMA swizzle XORs the 16-byte chunk with the row
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int kb = half * 2 + b;
    if constexpr (QT == kQ8)
      off[b] = (uint32_t)row * 128 + ((uint32_t)((kb * 2 + (t >> 1)) ^ (row & 7)) << 4) + (t & 1) * 8;
    else
      off[b] = (uint32_t)row * 64 + ((uint32_t)(kb ^ ((row >> 1) & 3)) << 4) + t * 4;
  }
  int pl = -1, el = 0;  // assignment of column `lane` and the scale exponent of its token
  if (half == 0 && lane < un.n) {
    pl = d.asg[un.a0 + lane];
    el = d.xe[pl / d.k];
  }
  float acc[NTL][4], tot[NTL][4];  // sums of a segment of kSeg stages, of the row
#pragma unroll
  for (int i = 0; i < NTL; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[i][q] = tot[i][q] = 0.f;

  for (int kc = 0; kc < KC; ++kc) {
    if (kc > 0 && !mbar_wait(&full[r.stage], r.phase, d.wait_ns)) return false;
    const unsigned char* st = smem + (size_t)r.stage * f.stage;
    const uint32_t so = L::kOffScale + (uint32_t)row * kScaleBoxBytes + ((kc & 1) * 2 + half) * 4;
    const __half2 s_lo = *reinterpret_cast<const __half2*>(st + so);
    const __half2 s_hi = *reinterpret_cast<const __half2*>(st + so + kRecs * kScaleBoxBytes);
    const unsigned char* bp = st + L::kOffB + (uint32_t)g * kColStride + t * 16;
    const float dl[2] = {__low2float(s_lo), __high2float(s_lo)}, dh[2] = {__low2float(s_hi), __high2float(s_hi)};
    const int kb = half * 2, left = nb - kc * 4 - kb;  // blocks of the row from this warp's first on
    if (left >= 2)
      stream_blocks<QT, NTL, 2>(st, bp, off, kb, dl, dh, acc);
    else if (left == 1)
      stream_blocks<QT, NTL, 1>(st, bp, off, kb, dl, dh, acc);
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[r.stage]);
    if ((kc & (kSeg - 1)) == kSeg - 1) {
#pragma unroll
      for (int i = 0; i < NTL; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          tot[i][q] += acc[i][q];
          acc[i][q] = 0.f;
        }
    }
    if (++r.stage == f.NS) {
      r.stage = 0;
      r.phase ^= 1u;
    }
  }
#pragma unroll
  for (int i = 0; i < NTL; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) tot[i][q] += acc[i][q];

  // the two K halves of a row group meet: half 1 leaves its sums in one of the group's two buffers
  const int buf = r.unit & 1;
  const uint32_t par = (uint32_t)(r.unit >> 1) & 1u;
  uint64_t* filled = rbar + grp * 4 + buf;
  uint64_t* taken = filled + 2;
  float4* rp = red + (size_t)(buf * 8 + grp) * (f.cols / 8) * 32 + lane;
  if (half == 1) {
    if (r.unit >= 2 && !mbar_wait(taken, par ^ 1u, d.wait_ns)) return false;
#pragma unroll
    for (int i = 0; i < NTL; ++i) rp[i * 32] = make_float4(tot[i][0], tot[i][1], tot[i][2], tot[i][3]);
    __syncwarp();
    if (lane == 0) mbar_arrive(filled);
    return true;
  }
  if (!mbar_wait(filled, par, d.wait_ns)) return false;
#pragma unroll
  for (int i = 0; i < NTL; ++i) {
    const float4 o = rp[i * 32];
    const float v[4] = {tot[i][0] + o.x, tot[i][1] + o.y, tot[i][2] + o.z, tot[i][3] + o.w};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int pos = __shfl_sync(0xffffffffu, pl, i * 8 + 2 * t + q), e = __shfl_sync(0xffffffffu, el, i * 8 + 2 * t + q);
      if (pos < 0) continue;
      if constexpr (NT == 2) {
        const int o_row = un.y + row;  // v[q]: gate, v[q + 2]: up, of output feature o_row
        if (o_row < rows) {
          const float h = v[q] / (1.0f + expf(-dq::scale2(v[q], e))) * v[q + 2];
          uint16_t p[3];
          split3(h, p);
          uint16_t* hp = reinterpret_cast<uint16_t*>(d.hs + ((size_t)pos * ((d.I + kKC - 1) / kKC) + o_row / kKC) * kColBytes) +
                         ((o_row & (kKC - 1) & ~31) | stream_pos<QT>(o_row & 31));
          hp[0] = p[0];
          hp[kKC] = p[1];
          hp[2 * kKC] = p[2];
        }
      } else {
        float* o2 = d.part + (size_t)pos * d.H + un.y + row;
        if (un.y + row < rows) o2[0] = dq::scale2(dq::scale2(v[q], e), e);
        if (un.y + kRecs + row < rows) o2[kRecs] = dq::scale2(dq::scale2(v[q + 2], e), e);
      }
    }
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(taken);
  return true;
}

// NT = 2: gate and up rows of the same 64 records; NT = 1: 128 down rows (two boxes of 64 records).
template <int QT, int NT>
__global__ void __launch_bounds__(kSThreads, 1)
    k_stream(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap smap, Dev d, int layer,
             int wave, StreamCfg f) {
  using L = SL<QT>;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + f.off_bar);
  uint64_t* empty = full + kSMaxStages;
  uint64_t* rbar = empty + kSMaxStages;  // [8 row groups]: filled x 2, taken x 2
  int* s_q = reinterpret_cast<int*>(rbar + 32);  // [kSMaxStages] the block's j-th unit at j % kSMaxStages
  float4* red = reinterpret_cast<float4*>(smem + f.off_red);
  int* s_units = reinterpret_cast<int*>(smem + f.off_tab);  // [nu + 1] units before expert i of the wave
  int* s_asg = s_units + d.S_active + 1;                    // [nu + 1] its first assignment
  int* s_slot = s_asg + d.S_active + 1;                     // [nu] its slot
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int K = NT == 2 ? d.H : d.I, rows = NT == 2 ? d.I : d.H;
  const int nb = K / 32, KC = (K + kKC - 1) / kKC;
  constexpr int kUnitRows = NT == 2 ? kRecs : 2 * kRecs;
  const int nrb = (rows + kUnitRows - 1) / kUnitRows;
  if (tid == 0) {
    for (int s = 0; s < f.NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kSWarps);
    }
    for (int i = 0; i < 32; ++i) mbar_init(&rbar[i], 1);
    mbar_fence_init();
  }
  pdl_wait();
  const int u0 = wave * d.S_active, nu = max(0, min(d.S_active, d.info[0] - u0));
  for (int i = tid; i <= nu; i += kSThreads) {
    s_asg[i] = d.asg_off[u0 + i];
    if (i < nu) s_slot[i] = d.uslot[u0 + i];
  }
  __syncthreads();
  if (warp == 0) {  // units before expert i: row blocks x groups of up to f.cols assignments
    int base = 0;
    for (int i0 = 0; i0 < nu; i0 += 32) {
      const int i = i0 + lane;
      int v = i < nu ? (s_asg[i + 1] - s_asg[i] + f.cols - 1) / f.cols * nrb : 0;
      const int own = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int w = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += w;
      }
      if (i < nu) s_units[i] = base + v - own;
      base += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) s_units[nu] = base;
  }
  __syncthreads();
  const int total = s_units[nu];
  auto unit_at = [&](int i) -> SUnit {
    int lo = 0, hi = nu - 1;
    while (lo < hi) {  // the last expert whose units begin at or before i
      const int mid = (lo + hi + 1) >> 1;
      if (s_units[mid] <= i) lo = mid;
      else hi = mid - 1;
    }
    const int r = i - s_units[lo], cb = r / nrb, n = s_asg[lo + 1] - s_asg[lo] - cb * f.cols;
    return {layer * d.S_alloc + s_slot[lo], (r - cb * nrb) * kUnitRows, s_asg[lo] + cb * f.cols, min(n, f.cols)};
  };

  if (warp == kSWarps) {  // ---- producer warp
    int stage = 0, it = 0, next = (int)blockIdx.x;
    uint32_t phase = 0;
    bool ok = true;
    const uint8_t* src = NT == 2 ? d.xs : d.hs;
    const size_t cstride = (size_t)KC * kColBytes;
    unsigned* ctr = d.sched + 2 * wave + (NT == 1);
    for (int j = 0; ok; ++j) {
      const int i = next;
      const bool end = i >= total;
      SUnit un = {0, 0, 0, 0};
      const uint8_t* col = nullptr;  // this lane's assignment: its activation pieces
      if (!end) {
        if (lane == 0) next = (int)gridDim.x + (int)atomicAdd(ctr, 1u);  // the unit after this one
        un = unit_at(i);
        if (lane < un.n) {
          const int a = __ldg(&d.asg[un.a0 + lane]);
          col = src + (size_t)(NT == 2 ? a / d.k : a) * cstride;
        }
      }
      const int n_kc = end ? 1 : KC;
      for (int kc = 0; kc < n_kc; ++kc, ++it) {
        if (it >= f.NS) ok = mbar_wait(&empty[stage], phase ^ 1u, d.wait_ns);
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        unsigned char* st = smem + (size_t)stage * f.stage;
        if (lane == 0) {
          if (kc == 0) s_q[j % kSMaxStages] = end ? -1 : i;
          if (end) {
            mbar_arrive(&full[stage]);
          } else {
            mbar_arrive_tx(&full[stage], 2 * L::kBox + 2 * kRecs * kScaleBoxBytes + (uint32_t)un.n * kColBytes);
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              const int x = (NT == 2 && b ? (int)d.lay.o_up : 0) + kc * (int)L::kRow;
              const int xs = (int)(NT == 2 ? (b ? d.lay.o_us : d.lay.o_gs) : d.lay.o_ds) + (kc >> 1) * (int)kScaleBoxBytes;
              const int y = un.y + (NT == 1 && b ? kRecs : 0);
              tma_3d(st + b * L::kBox, &tmap, x, y, un.z, &full[stage]);
              tma_3d(st + L::kOffScale + b * kRecs * kScaleBoxBytes, &smap, xs, y, un.z, &full[stage]);
            }
          }
        }
        __syncwarp();
        if (col) bulk_g2s(st + L::kOffB + (uint32_t)lane * kColStride, col + (size_t)kc * kColBytes, kColBytes, &full[stage]);
        if (++stage == f.NS) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (end) break;
      next = __shfl_sync(0xffffffffu, next, 0);
    }
    if (lane == 0) {
      if (!ok) atomicExch(d.err, 1u);
      // no copy may be in flight when the block exits: wait for the last use of every stage
      for (int s = 0; s < f.NS && s < it; ++s)
        if (!mbar_wait(&full[s], (uint32_t)((it - 1 - s) / f.NS) & 1u, d.wait_ns)) atomicExch(d.err, 2u);
    }
  } else {  // ---- consumers: units in the order the producer drew them
    SRing r;
    bool ok = true;
    while ((ok = mbar_wait(&full[r.stage], r.phase, d.wait_ns))) {
      const int i = s_q[r.unit % kSMaxStages];
      if (i < 0) break;
      const SUnit un = unit_at(i);
#define MF_UNIT(N) stream_unit<QT, NT, N>(d, un, smem, full, empty, rbar, f, red, KC, nb, rows, r, warp, lane)
      switch ((un.n + 7) >> 3) {
        case 1: ok = MF_UNIT(1); break;
        case 2: ok = MF_UNIT(2); break;
        case 3: ok = MF_UNIT(3); break;
        default: ok = MF_UNIT(4); break;
      }
#undef MF_UNIT
      if (!ok) break;
      ++r.unit;
    }
    if (!ok && lane == 0) atomicExch(d.err, 6u);
  }
  __syncthreads();
}

int sm_count_s() {
  static int n = 0;
  if (!n) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    n = v > 0 ? v : 1;
  }
  return n;
}

template <int QT, int NT>
cudaError_t launch_s(const Dev& d, const CUtensorMap* tm, int layer, int wave, int T, bool overlap,
                     cudaStream_t s) {
  const StreamCfg f = stream_cfg(d, T);
  cudaError_t e = cudaFuncSetAttribute(k_stream<QT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.total);
  if (e != cudaSuccess) return e;
  return launch_pdl(overlap, k_stream<QT, NT>, dim3(sm_count_s()), dim3(kSThreads), f.total, s, tm[0], tm[1], d, layer, wave, f);
}

}  // namespace

size_t stream_bytes(int n, int K) { return (size_t)n * ((K + kKC - 1) / kKC) * kColBytes; }

int stream_tensor_maps(mf_ctx* c) {
  const Dev& d = c->d;
  const uint32_t row = d.qtype == MF_Q8_0 ? SL<kQ8>::kRow : SL<kQ4>::kRow;
  const uint64_t planes = (uint64_t)d.L * d.S_alloc;
  for (int m = 0; m < 2; ++m) {  // boxes of codes (swizzled by their row bytes) and of scales
    const uint32_t box = m ? kScaleBoxBytes : row;
    const int sw = m ? 0 : (int)row;
    if (encode_slot_region(&c->ts_gu[m], d.pool, d.lay.rs_gu, (uint64_t)d.I, planes, d.lay.stride, box, kRecs, sw)) return -1;
    if (encode_slot_region(&c->ts_d[m], d.pool + d.lay.d_off, d.lay.rs_d, (uint64_t)d.H, planes, d.lay.stride, box, kRecs, sw))
      return -1;
  }
  return 0;
}

cudaError_t launch_stream_gateup(const Dev& d, const CUtensorMap* tm, int layer, int wave, int T, bool overlap,
                                 cudaStream_t s) {
  return d.qtype == MF_Q8_0 ? launch_s<kQ8, 2>(d, tm, layer, wave, T, overlap, s)
                            : launch_s<kQ4, 2>(d, tm, layer, wave, T, overlap, s);
}

cudaError_t launch_stream_down(const Dev& d, const CUtensorMap* tm, int layer, int wave, int T, cudaStream_t s) {
  return d.qtype == MF_Q8_0 ? launch_s<kQ8, 1>(d, tm, layer, wave, T, true, s)
                            : launch_s<kQ4, 1>(d, tm, layer, wave, T, true, s);
}

}  // namespace mf
