// Prefill expert FFN: grouped GEMMs on the fifth-generation tensor cores (tcgen05).
//
// When many tokens route to each expert (a prefill chunk), the expert FFN of a wave is a set
// of dense products, one per expert e of the wave with the n_e assignments it serves:
//   gate/up:  G = Wg_e X_e^T, U = Wu_e X_e^T,  h = silu(G) * U                 [I x n_e]
//   down:     P = Wd_e h                                                        [H x n_e]
// then y[t] = sum_j g[t,j] P_{e_j}[:, t] (the batched combine kernel).  (SwiGLU experts with
// separate gate, up and down tensors, section "Native Serving Path".)
//
// Precision.  Operands are split into two bfloat16 parts, v = hi + lo with hi = bf16(v) and
// lo = bf16(v - hi), so hi + lo carries 16 significant bits (relative error <= 2^-17).  Each
// product is formed as hi*hi + hi*lo + lo*hi with fp32 accumulation in tensor memory; the
// dropped lo*lo term is below 2^-16 of the product.  Per product the relative error is thus
// a few times 1e-5, far inside the output tolerance, while the tensor cores do the work.
//
// Operand B never needs a gather inside the GEMM: once per call k_tile_x writes x, split, in
// the MMA's shared-memory order per (128-assignment block, K step of 32) -- 16 KiB tiles that
// one bulk copy moves -- and the gate/up epilogue writes h the same way for the down GEMM.
//
// Work unit = (expert of the wave, block of 128 assignments, 256 weight rows as two M blocks: gate and
// up of the same 128 records, or 256 down rows); one CTA of 27 warps per SM walks its units as a flat
// sequence of K steps of 32 (one quantisation block), with warp-specialised roles linked by mbarriers:
//   producer (1 warp)    per step bulk copies of the B tile into a 6-slot ring; every 128 code bytes
//                        of K a TMA load per M block (128 rows, from a 3-D tensor map over the slot
//                        pool) into one of 3 raw buffers; every 8 steps one TMA load per M block of
//                        the rows' next 8 scales (lane 0 issues; a TMA box costs 2 cycles a row up to
//                        128 bytes, so a box per step kept the copy engine as busy as the MMAs);
//   converters (2 x 8 warps, even and odd steps) turn the raw codes into exact bf16 integers, form
//                        hi and lo of their products with the scale in packed bf16 arithmetic and
//                        write the A operand into tensor memory (tcgen05.st; one lane per row, hi and
//                        lo of 32 weights = 2 x 16 columns per M block);
//   MMA (2 warps)        issue the step's tcgen05.mma, one M block each (A in tensor memory, B in shared memory;
//                        M = 128, K = 16, N = the block's assignments rounded up to a multiple of
//                        16) into the unit's TMEM accumulators and commits them to the slot's and
//                        the A stage's mbarriers;
//   epilogue (8 warps)   reads the finished accumulators with tcgen05.ld (two warps per 32 TMEM
//                        lanes, half of the columns each); the next unit's MMAs wait for that, the
//                        converters and copies run ahead.
// Tensor memory: 256 columns of accumulators, 4 A stages of 64 columns.  What bounds it: the MMAs
// (three products per weight: 768 cycles of a step's 1200 at 128 assignments) and, between two units, the
// epilogue's reading of the one accumulator set there is room for (150-280 cycles a step).  4096 tokens,
// 128 Q4_0 experts of 2048 x 768: gate/up 456 us and down 294 us, where units of 128 rows with A in shared
// memory took 638 and 446.  With A in shared memory the MMAs' operand reads, the converters'
// stores and the B copies together filled the shared-memory pipe (an M = 128, N = 128, K = 16 MMA
// reads 8 KiB of it per 64 tensor cycles; down units of 128 rows also loaded a B tile per 128 rows).
// Every wait is bounded; a wait that gives up sets the block's flag and the device error word,
// the roles leave their loops, and the block drains its copies and MMAs (bounded) and frees
// its tensor memory before returning.
#include <cuda_bf16.h>

#include "mf_dequant.cuh"

namespace mf {
namespace {

using dq::f2_fma;
using dq::f2_pack;

constexpr int kBM = 128, kBN = 128, kBK = 32;
constexpr int kStages = 4;  // A operand stages in tensor memory
constexpr int kSlots = 6;   // B ring slots
constexpr int kRaws = 3;    // raw-code buffers, 128 code bytes of K per row each
constexpr uint32_t kTile = kBM * kBK * 2;  // one bf16 tile: 128 rows x 32 k = 8 KiB
constexpr uint32_t kBTile = 2 * kTile;     // B hi + lo, one bulk copy

// warp roles of the 864-thread CTA
constexpr int kConvWarps = 8;   // warps 0-7 dequantise the even steps, 8-15 the odd ones; M block (warp / 4) % 2,
                                // TMEM lane quarter warp % 4
constexpr int kProdWarp = 16;   // warp 16: copies
constexpr int kMmaWarp = 17;    // warps 17 and 18: MMA issue, one M block each
constexpr int kEpiWarp0 = 19;   // warps 19-26: epilogue; TMEM lane quarter = warp % 4
constexpr int kEpiWarps = 8;
constexpr int kThreadsW = 27 * 32;
static_assert(kEpiWarp0 == kMmaWarp + 2 && kEpiWarp0 + kEpiWarps == kThreadsW / 32, "warp roles");
constexpr uint32_t kAcc0 = 0, kA0 = 256, kAStage = 64;  // TMEM columns: accumulators, A stages
constexpr uint32_t kCols = 512;
static_assert(kA0 + kStages * kAStage == kCols, "tensor memory");

// Byte offset of element (row r, k) in a K-major no-swizzle tile of 128 x 32: 8x8 core
// matrices of 128 contiguous bytes, K-adjacent core matrices 128 B apart (the descriptor's
// leading byte offset), 8-row groups 512 B apart (its stride byte offset).
__host__ __device__ __forceinline__ uint32_t core_off(int r, int k) {
  return (uint32_t)((r >> 3) * 512 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// shared-memory matrix descriptor: start >> 4, LBO >> 4 at bit 16, SBO >> 4 at bit 32,
// descriptor version 1 at bit 46, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(512u >> 4) << 32) |
         ((uint64_t)1 << 46);
}

// kind::f16 instruction descriptor: fp32 accumulator, bf16 A and B, both K-major, M = 128 x N
// (N a multiple of 16, at most 128 here)
__device__ __forceinline__ uint32_t idesc_n(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}
constexpr uint32_t kNegateA = 1u << 13;  // the descriptor's bit that negates A
// the MMA width of a block with n assignments: n rounded up to a multiple of 16
__device__ __forceinline__ int n_eff(int n) { return max(16, (n + 15) & ~15); }

// D[tmem] (+)= A[tmem] * B[smem descriptor]
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{ .reg .pred p; setp.ne.u32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p; }" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate));
}
// 1 on one lane of the (converged) warp
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile("{ .reg .pred p; elect.sync _|p, 0xffffffff; selp.u32 %0, 1, 0, p; }" : "=r"(r));
  return r;
}
// the six MMAs of one M block and K step of 32: (hi + lo) B's hi and hi times B's lo, two K = 16 halves (of B two
// core matrices, of A 8 columns); A's low part is stored negated (split_pair)
__device__ __forceinline__ void mma_step(uint32_t d_tmem, uint32_t a, uint64_t bh, uint64_t bl, uint32_t idesc,
                                         uint32_t accumulate) {
  constexpr uint64_t ko = 256 >> 4;
  mma_bf16(d_tmem, a, bh, idesc, accumulate);
  mma_bf16(d_tmem, a, bl, idesc, 1);
  mma_bf16(d_tmem, a + 16, bh, idesc | kNegateA, 1);
  mma_bf16(d_tmem, a + 8, bh + ko, idesc, 1);
  mma_bf16(d_tmem, a + 8, bl + ko, idesc, 1);
  mma_bf16(d_tmem, a + 24, bh + ko, idesc | kNegateA, 1);
}
// arrive on the barrier once every MMA this thread issued so far has completed
__device__ __forceinline__ void mma_commit_at(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) { mma_commit_at(smem_u32(bar)); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 3-D tiled TMA load of a box at (x, y, z) of `tmap` into shared memory, completing on `bar`
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tmap, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// 16 consecutive fp32 accumulator columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t bf2_bits(__nv_bfloat162 v) { return *reinterpret_cast<uint32_t*>(&v); }

// Two values (packed fp32 pair) -> bf16x2 words hi = bf16(v), lo = bf16(v - hi).
__device__ __forceinline__ void split2(uint64_t w, uint32_t& hi, uint32_t& lo) {
  uint32_t a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(w));
  const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(a), __uint_as_float(b));
  const float2 hf = __bfloat1622float2(h);
  const uint64_t r = f2_fma(f2_pack(__float_as_uint(hf.x), __float_as_uint(hf.y)), f2_pack(0xBF800000u, 0xBF800000u), w);
  uint32_t ra, rb;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(ra), "=r"(rb) : "l"(r));
  hi = bf2_bits(h);
  lo = bf2_bits(__floats2bfloat162_rn(__uint_as_float(ra), __uint_as_float(rb)));
}

// A scale d as the sum of two bf16 values dh + dl (exact: 11 bits; dl at most four units of d's last place).
struct ScaleParts {
  uint32_t h, nh, l, nl, l2;  // pairs of dh, -dh, dl, -dl, 2 dl
  __device__ __forceinline__ explicit ScaleParts(float d) {
    const __nv_bfloat16 hb = __float2bfloat16_rn(d), lb = __float2bfloat16_rn(d - __bfloat162float(hb));
    h = __bfloat16_as_ushort(hb) * 0x10001u;
    l = __bfloat16_as_ushort(lb) * 0x10001u;
    nh = h ^ 0x80008000u;
    nl = l ^ 0x80008000u;
    l2 = __bfloat16_as_ushort(lb + lb) * 0x10001u;
  }
};

// A pair of codes q (exact bf16) times a scale -> the bf16 parts hi = RN(q d) of the weights and -lo, lo =
// RN(q d - hi), in packed instructions of the FMA pipe: hi - q dh is exact (it fits 8 bits), so each part is
// rounded once.  (-lo: a sign change in between would cost an instruction; the MMA negates it.)  t = q dl is
// exact for Q4_0.  For Q8_0 it may take nine bits and is then rounded by one unit, to a multiple of four units:
// where that makes q dh + t a tie between two values of hi, hi could be the farther one (for ten pairs of code
// and mantissa hi + lo was off by up to 9.2e-6 of q d, in place of 7.6e-6).  2 q dl - t is off by one unit to the other
// side, no multiple of four, and meets no tie: hi is the nearest for every code and mantissa.
// Converting q d to fp32 and splitting it there kept the ALU pipe busy with byte permutes and unpacking: 1000
// tokens over 64 Q8_0 experts took 324 us a call, so 338 (with the split in f32x2 arithmetic 340; with hi from
// q dh + RN(q dl), 318), each before the epilogue's division was exact (329 us).
template <int QT>
__device__ __forceinline__ void split_pair(uint32_t q, const ScaleParts& d, uint32_t& hi, uint32_t& nlo) {
  uint32_t t;
  if constexpr (QT == MF_Q8_0)
    asm("{ .reg .b32 m;\n"
        "mul.rn.bf16x2 m, %1, %2;\n"
        "fma.rn.bf16x2 %0, %1, %3, m; }"
        : "=r"(t)
        : "r"(q), "r"(d.nl), "r"(d.l2));
  else
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(t) : "r"(q), "r"(d.l));
  asm("{ .reg .b32 e;\n"
      "fma.rn.bf16x2 %0, %2, %3, %6;\n"
      "fma.rn.bf16x2 e, %2, %4, %0;\n"
      "fma.rn.bf16x2 %1, %2, %5, e; }"
      : "=&r"(hi), "=r"(nlo)
      : "r"(q), "r"(d.h), "r"(d.nh), "r"(d.nl), "r"(t));
}

// Four codes (Q8_0: bytes q + 128; Q4_0: nibbles masked to bytes) -> two words of hi and of -lo.
template <int QT>
__device__ __forceinline__ void dequant4(uint32_t w, const ScaleParts& d, uint32_t* h, uint32_t* l) {
  uint32_t q01, q23;
  if constexpr (QT == MF_Q8_0)
    dq::codes_q8(w, q01, q23);
  else
    dq::codes_q4(w, q01, q23);
  split_pair<QT>(q01, d, h[0], l[0]);
  split_pair<QT>(q23, d, h[1], l[1]);
}

// 8 consecutive columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

struct Unit {
  int u;   // unique-expert index (access order)
  int tb;  // block of 128 assignments
  int rb;  // block of 128 records (gate/up) or 256 rows (down)
};

// The wave's units, expert by expert: expert u0 + e has ceil(n / 128) assignment blocks times
// `nrb` row blocks, row blocks innermost (CTAs working on the same assignment block at once
// share its B tiles in L2).  Unit i is row block i % nrb of the wave's assignment block i / nrb,
// found in the exclusive prefix of assignment blocks per unique expert (tb_off).
struct UnitMap {
  int u0, nu, nrb, total;
  const int* tb_off;
  __device__ __forceinline__ Unit at(int i) const {
    const int ti = __ldg(&tb_off[u0]) + i / nrb;
    int lo = u0, hi = u0 + nu - 1;
    while (lo < hi) {  // last expert whose first assignment block is at or before ti
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(&tb_off[mid]) <= ti) lo = mid;
      else hi = mid - 1;
    }
    return {lo, ti - __ldg(&tb_off[lo]), i % nrb};
  }
};

// Scales travel in groups of kGroup K steps: one 16-byte TMA box per (M block, row) holds the
// group's 8 binary16 scales, which the converters read into registers at their first step of the group
// (its first or second).  A group's buffer is loaded again two groups later, once the producer has seen
// the B slot of the step kSlots + 1 before freed: every group has 4 or 8 steps (K is a multiple of 128),
// so that step does not lie before the second step of the buffer's previous group while kSlots <= 6.
constexpr int kGroup = 8;
constexpr uint32_t kScaleBox = 16;
static_assert(kSlots <= 6 && kStages % 2 == 0 && kGroup * 2 == (int)kScaleBox, "scale groups");

// Shared memory of one CTA: B ring, raw buffers (two M blocks of 128 rows x 128 code bytes, 16-byte
// chunks XORed with the row by the TMA swizzle), scale ring, barriers.
constexpr uint32_t kRawRow = 128;
constexpr uint32_t kRawBuf = 2 * kBM * kRawRow;
constexpr uint32_t kScaleBuf = 2 * kBM * kScaleBox;  // scales of one group (TMA boxes)
constexpr int kBarFull = 0, kBarDone = kSlots, kBarRawFull = 2 * kSlots, kBarRawFree = kBarRawFull + kRaws,
              kBarSFull = kBarRawFree + kRaws, kBarAReady = kBarSFull + 2, kBarAccFull = kBarAReady + 2 * kStages, kBarAccEmpty = kBarAccFull + 2, kBarDrain = kBarAccEmpty + 2,
              kBars = kBarDrain + 1;
constexpr uint32_t kOffRaw = kSlots * kBTile;
constexpr uint32_t kOffScale = kOffRaw + kRaws * kRawBuf;
constexpr uint32_t kOffBar = kOffScale + 2 * kScaleBuf;
constexpr uint32_t kOffMisc = kOffBar + kBars * 8;
constexpr uint32_t kSmemW = kOffMisc + 16;
static_assert(kOffRaw % 1024 == 0 && kRawBuf % 1024 == 0 && kOffScale % 128 == 0 && kScaleBuf % 128 == 0,
              "TMA destinations");

// Gate/up (NT = 2) or down (NT = 1) projection of wave `wave` for every assignment of the wave.
//   gate/up: A = gate / up rows of the slot's gate/up region, B = x tiles; epilogue
//            h = silu(G) * U, split, into the h tiles
//   down:    A = down rows, B = h tiles; epilogue part[assignment][hidden]
// Pipeline (mbarriers): producer --raw_full--> converters --a_ready--> MMA --done--> converters, producer;
// converters --raw_free--> producer --full--> MMA; MMA --acc_full--> epilogue --acc_empty--> MMA.
// (Launch bounds of 1024 threads: 64 registers, which leaves the materialiser room beside a GEMM block; with 72
// its blocks waited for the GEMM's end and a cold call of several waves took 3.2 instead of 2.9 ms.)
template <int QT, int NT>
__global__ void __launch_bounds__(1024, 1)
    k_prefill(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ CUtensorMap smap, Dev d, int layer,
              int wave) {
  constexpr int CB = QT == MF_Q8_0 ? 32 : 16;
  constexpr int RG = (int)kRawRow / CB;  // K steps of a raw buffer
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOffBar);
  uint64_t* full = bars + kBarFull;           // [kSlots]  1 expect-tx arrival (B tile)
  uint64_t* done = bars + kBarDone;           // [kSlots]  tcgen05.commit of both MMA warps: the step's slot and A stage are free
  uint64_t* raw_full = bars + kBarRawFull;    // [kRaws]   1 expect-tx arrival (codes)
  uint64_t* raw_free = bars + kBarRawFree;    // [kRaws]   one arrival per converter warp
  uint64_t* s_full = bars + kBarSFull;        // [2]       1 expect-tx arrival (a group's scales)
  uint64_t* a_ready = bars + kBarAReady;      // [kStages][M block] one arrival per converter warp of the block
  uint64_t* acc_full = bars + kBarAccFull;    // [M block] tcgen05.commit
  uint64_t* acc_empty = bars + kBarAccEmpty;  // [M block] one arrival per epilogue warp
  uint64_t* drain = bars + kBarDrain;         // [1]       tcgen05.commit of both MMA warps
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* s_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  const int K = NT == 2 ? d.H : d.I;  // reduction length
  const int nk = K / kBK;             // steps per unit
  const int rows = NT == 2 ? d.I : d.H;
  constexpr int kURows = NT == 2 ? kBM : 2 * kBM;  // records per unit
  const int nrb = (rows + kURows - 1) / kURows;    // row blocks per expert

  // ---- prologue: barriers, tensor memory, the wave's unit prefix
  if (tid == 0) {
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&done[i], 2);
    }
    for (int i = 0; i < kRaws; ++i) {
      mbar_init(&raw_full[i], 1);
      mbar_init(&raw_free[i], 2 * kConvWarps);
    }
    for (int i = 0; i < 2; ++i) mbar_init(&s_full[i], 1);
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&a_ready[2 * i], kConvWarps / 2);
      mbar_init(&a_ready[2 * i + 1], kConvWarps / 2);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], kEpiWarps);
    }
    mbar_init(drain, 2);
    *s_flag = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  UnitMap um;
  um.u0 = wave * d.S_active;
  um.nu = max(0, min(d.S_active, d.info[0] - um.u0));
  um.nrb = nrb;
  um.tb_off = d.tb_off;
  um.total = um.nu > 0 ? (d.tb_off[um.u0 + um.nu] - d.tb_off[um.u0]) * nrb : 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem0 = *s_tmem;
  const int bid = (int)blockIdx.x, nb = (int)gridDim.x;
  const int n_units = um.total > bid ? (um.total - 1 - bid) / nb + 1 : 0;
  const int n_steps = n_units * nk;

  // bounded wait; false (and the block's flag and the device error word set) once any wait gave up
  auto wait = [&](uint64_t* bar, uint32_t parity, unsigned code) -> bool {
    if (mbar_try_wait(bar, parity)) return true;  // the common case: no flag read on the fast path
    if (*s_flag) return false;
    if (mbar_wait(bar, parity, d.wait_ns)) return true;
    *s_flag = 1;
    atomicExch(d.err, code);
    return false;
  };
  // true where the unit's second M block lies past the last row (down, hidden not a multiple of 256)
  auto half_unit = [&](const Unit& un) -> bool { return NT == 1 && un.rb * kURows + kBM >= rows; };

  if (warp < 2 * kConvWarps) {
    // ================= converters: raw codes of step s -> A stage s % kStages; thread = (M block, row)
    const int ten = (warp >> 2) & 1, grp = warp >> 3, tr = ten * kBM + (tid & (kBM - 1));
    const uint32_t a_addr = tmem0 + kA0 + (uint32_t)ten * 32 + ((uint32_t)((warp & 3) * 32) << 16);
    int kk = grp, stage = grp, gb = 1, rb = kRaws - 1;  // steps grp, grp + 2, ... (nk is even)
    int before = grp;                    // slot of the step kStages before (from step kStages on)
    uint32_t bph = 0, gph = 1, rph = 1;  // phase parities of that slot, the scale ring, the raw buffers
    uint4 sv = make_uint4(0, 0, 0, 0);  // this row's scales of the current group
    bool alive = true;
    for (int s = grp; s < n_steps; s += 2) {
      if ((kk & (kGroup - 1)) == grp) {  // this warp's first step of a scale group
        gb ^= 1;
        if (gb == 0) gph ^= 1;
        if (!wait(&s_full[gb], gph, 1u)) break;
        sv = *reinterpret_cast<const uint4*>(smem + kOffScale + gb * kScaleBuf + tr * kScaleBox);
      }
      const int ri = kk % RG;  // the step's place in its raw buffer
      if (ri == grp) {
        if (++rb == kRaws) rb = 0, rph ^= 1;
        if (!wait(&raw_full[rb], rph, 1u)) break;
      }
      const unsigned char* codes = smem + kOffRaw + rb * kRawBuf + (uint32_t)tr * kRawRow;
      const int q = (kk >> 1) & 3;
      const uint32_t sw = q == 0 ? sv.x : q == 1 ? sv.y : q == 2 ? sv.z : sv.w;
      const float dsc = __half2float(__ushort_as_half((unsigned short)((kk & 1) ? (sw >> 16) : (sw & 0xFFFFu))));
      const ScaleParts ds(dsc);
      // 16 weights at a time (elements 0-15, 16-31: the two K halves of the step)
      uint32_t w[8];
      if constexpr (QT == MF_Q8_0) {
        const uint4 c0 = *reinterpret_cast<const uint4*>(codes + (((2 * ri) ^ (tr & 7)) << 4));
        const uint4 c1 = *reinterpret_cast<const uint4*>(codes + (((2 * ri + 1) ^ (tr & 7)) << 4));
        w[0] = c0.x, w[1] = c0.y, w[2] = c0.z, w[3] = c0.w, w[4] = c1.x, w[5] = c1.y, w[6] = c1.z, w[7] = c1.w;
      } else {
        // byte j: element j (low nibble), element j + 16 (high nibble)
        const uint4 c = *reinterpret_cast<const uint4*>(codes + ((ri ^ (tr & 7)) << 4));
        w[0] = c.x, w[1] = c.y, w[2] = c.z, w[3] = c.w;
#pragma unroll
        for (int i = 0; i < 4; ++i) w[4 + i] = (w[i] >> 4) & 0x0F0F0F0Fu, w[i] &= 0x0F0F0F0Fu;
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint32_t h[8], l[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) dequant4<QT>(w[4 * half + i], ds, h + 2 * i, l + 2 * i);
        if (half == 0) {  // the MMAs have read the stage
          if (s >= kStages) {
            if (!wait(&done[before], bph, 2u)) {
              alive = false;
              break;
            }
            if ((before += 2) >= kSlots) before -= kSlots, bph ^= 1;
          }
          __syncwarp();
          tc_fence_after();
        }
        tmem_st8(a_addr + stage * kAStage + half * 8, h);
        tmem_st8(a_addr + stage * kAStage + 16 + half * 8, l);
      }
      if (!alive) break;
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&a_ready[2 * stage + ten]);
        if (ri == RG - 2 + grp || kk == nk - 2 + grp) mbar_arrive(&raw_free[rb]);  // its last step of the buffer
      }
      if ((kk += 2) >= nk) kk -= nk;
      if ((stage += 2) >= kStages) stage -= kStages;
    }
  } else if (warp == kProdWarp) {
    // ================= producer (lane 0; the warp's other lanes have no role): TMA boxes of codes
    // and scales, bulk B tile
    if (lane == 0) {
      const uint8_t* tiles = NT == 2 ? d.xt : d.ht;
      int y0 = 0, z0 = 0;    // the unit's TMA coordinates: first row, slot plane
      size_t b0 = 0;         // its first B tile
      uint32_t b_bytes = 0;  // bytes of each B half the MMAs read: n_eff columns
      int kk = 0, slot = 0, j = 0, gb = 1, rb = kRaws - 1, issued = 0, groups = 0, raws = 0;
      uint32_t ph = 0, rph = 0;
      for (int s = 0; s < n_steps; ++s) {
        if (kk == 0) {
          const Unit un = um.at(bid + j * nb);
          z0 = layer * d.S_alloc + d.uslot[un.u];
          y0 = un.rb * kURows;
          b0 = (size_t)(d.tb_off[un.u] + un.tb) * nk;
          const int a0 = d.asg_off[un.u] + un.tb * kBN;
          b_bytes = (uint32_t)n_eff(min(kBN, d.asg_off[un.u + 1] - a0)) * (kBK * 2);
        }
        const bool raw = kk % RG == 0, group = kk % kGroup == 0;
        if (raw) {
          if (++rb == kRaws) rb = 0, rph ^= 1;
          if (raws >= kRaws && !wait(&raw_free[rb], rph, 3u)) break;
          mbar_arrive_tx(&raw_full[rb], kRawBuf);
          ++raws;
        }
        if (group) {
          gb ^= 1;
          mbar_arrive_tx(&s_full[gb], kScaleBuf);
          ++groups;
        }
#pragma unroll
        for (int tn = 0; tn < 2; ++tn) {  // gate and up records, or two blocks of down rows
          const int y = y0 + (NT == 1 ? tn * kBM : 0);
          if (raw)
            tma_load_3d(smem + kOffRaw + rb * kRawBuf + tn * kBM * kRawRow, &tmap, (NT == 2 && tn ? (int)d.lay.o_up : 0) + kk * CB,
                        y, z0, &raw_full[rb]);
          // x = the scale region's start (16-byte aligned in the slot layout) + 16 bytes per group
          const uint32_t so = NT == 2 ? (tn ? d.lay.o_us : d.lay.o_gs) : d.lay.o_ds;
          if (group)
            tma_load_3d(smem + kOffScale + gb * kScaleBuf + tn * kBM * kScaleBox, &smap,
                        (int)(so + (uint32_t)(kk / kGroup) * kScaleBox), y, z0, &s_full[gb]);
        }
        if (s >= kSlots && !wait(&done[slot], ph ^ 1, 4u)) break;
        unsigned char* base = smem + slot * kBTile;
        const uint8_t* bsrc = tiles + (b0 + kk) * kBTile;
        mbar_arrive_tx(&full[slot], 2 * b_bytes);
        bulk_g2s(base, bsrc, b_bytes, &full[slot]);                  // hi: the first n_eff columns
        bulk_g2s(base + kTile, bsrc + kTile, b_bytes, &full[slot]);  // lo
        ++issued;
        if (++kk == nk) kk = 0, ++j;
        if (++slot == kSlots) slot = 0, ph ^= 1;
      }
      // no copy may be in flight when the block exits: wait for the last use of every buffer
      for (int i = 0; i < kSlots && i < issued; ++i)
        if (!mbar_wait(&full[i], (uint32_t)((issued - 1 - i) / kSlots) & 1u, d.wait_ns)) atomicExch(d.err, 4u);
      for (int i = 0; i < kRaws && i < raws; ++i)
        if (!mbar_wait(&raw_full[i], (uint32_t)((raws - 1 - i) / kRaws) & 1u, d.wait_ns)) atomicExch(d.err, 4u);
      for (int i = 0; i < 2 && i < groups; ++i)
        if (!mbar_wait(&s_full[i], (uint32_t)((groups - 1 - i) / 2) & 1u, d.wait_ns)) atomicExch(d.err, 4u);
    }
  } else if (warp < kEpiWarp0) {
    // ================= MMA issue, one warp per M block: the whole warp walks the steps, one elected lane
    // issues.  Warp-uniform operands stay in uniform registers: from a single thread's branch every MMA
    // cost 72 cycles to issue whatever its N, against 64 at N = 128 and 28 at N = 16 this way.  The MMA
    // queue is too short to cover a step's waits and commits, so two warps take turns in them.
    const int tn = warp - kMmaWarp;
    int kk = 0, slot = 0, stage = 0, j = 0;
    uint32_t sph = 0, ph = 0, idesc = 0, next = 0;  // instruction descriptor of the unit (0: this M block is empty), of the next
    const uint32_t t0 = __shfl_sync(0xffffffffu, tmem0, 0);
    const uint32_t acc = t0 + kAcc0 + tn * kBN, smem0 = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
    const uint32_t bars0 = __shfl_sync(0xffffffffu, smem_u32(bars), 0);
    const int steps = __shfl_sync(0xffffffffu, n_steps, 0);
    auto unit_desc = [&](int i) -> uint32_t {
      const Unit un = um.at(bid + i * nb);
      const int a0 = d.asg_off[un.u] + un.tb * kBN;
      const uint32_t v = idesc_n(n_eff(min(kBN, d.asg_off[un.u + 1] - a0)));
      return __shfl_sync(0xffffffffu, tn == 1 && half_unit(un) ? 0u : v, 0);
    };
    if (steps > 0) next = unit_desc(0);
    for (int s = 0; s < steps; ++s) {
      if (kk == 0) idesc = next;
      bool ok = kk != 0 || j == 0 || wait(&acc_empty[tn], (j - 1) & 1, 8u);
      // both barriers polled at once: their latencies overlap
      const bool f = mbar_try_wait(&full[slot], ph), a = mbar_try_wait(&a_ready[2 * stage + tn], sph);
      ok = ok && (f || wait(&full[slot], ph, 9u)) && (a || wait(&a_ready[2 * stage + tn], sph, 9u));
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const uint32_t base = smem0 + slot * kBTile, a0 = t0 + kA0 + stage * kAStage + tn * 32;
      if (elect_one()) {
        if (idesc) mma_step(acc, a0, smem_desc(base), smem_desc(base + kTile), idesc, kk != 0);
        mma_commit_at(bars0 + (uint32_t)(kBarDone + slot) * 8);
        if (kk == nk - 1) mma_commit_at(bars0 + (uint32_t)(kBarAccFull + tn) * 8);
      }
      __syncwarp();
      if (kk == 0 && j + 1 < n_units) next = unit_desc(j + 1);  // while this unit's MMAs run
      if (++kk == nk) kk = 0, ++j;
      if (++slot == kSlots) slot = 0, ph ^= 1;
      if (++stage == kStages) stage = 0, sph ^= 1;
    }
    // nothing may be in flight when the tensor memory is freed
    if (elect_one()) mma_commit(drain);
    __syncwarp();
    if (!mbar_wait(drain, 0, d.wait_ns)) atomicExch(d.err, 10u);
  } else {
    // ================= epilogue: the unit's accumulators -> outputs
    const int q4 = warp & 3;                                     // TMEM lanes 32 q4 .. 32 q4 + 31
    const int ch = (warp - kEpiWarp0) >> 2;                      // columns 64 ch .. 64 ch + 63
    const uint32_t lane_addr = tmem0 + kAcc0 + ((uint32_t)(q4 * 32) << 16);
    for (int j = 0; j < n_units; ++j) {
      const Unit un = um.at(bid + j * nb);
      const int a0 = d.asg_off[un.u] + un.tb * kBN;
      const int n = min(kBN, d.asg_off[un.u + 1] - a0), ne = n_eff(n);
      if constexpr (NT == 2) {
        if (!wait(&acc_full[0], j & 1, 11u) || !wait(&acc_full[1], j & 1, 11u)) break;
        __syncwarp();
        tc_fence_after();
        const int r = un.rb * kBM + q4 * 32 + lane;  // weight row = output feature
        // h tile of K step r / 32 of the down GEMM: this lane's row is its k = r % 32
        uint8_t* ht = d.ht + ((size_t)(d.tb_off[un.u] + un.tb) * (d.I / kBK) + (r >> 5)) * kBTile;
        for (int c0 = ch * 64; c0 < min(ne, ch * 64 + 64); c0 += 16) {  // the columns the down MMAs read
          // (the division is the IEEE one: __fdividef is 0 above 2^126, for gates below -87.3; 1000 tokens 324 -> 329 us)
          float g[16], u[16];
          tmem_ld16(lane_addr + c0, g);
          tmem_ld16(lane_addr + kBN + c0, u);
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int col = c0 + q;
            const float hv = col < n ? g[q] / (1.0f + expf(-g[q])) * u[q] : 0.0f;
            const __nv_bfloat16 hi = __float2bfloat16_rn(hv);
            const uint32_t o = core_off(col, r & 31);
            *reinterpret_cast<uint16_t*>(ht + o) = __bfloat16_as_ushort(hi);
            *reinterpret_cast<uint16_t*>(ht + kTile + o) =
                __bfloat16_as_ushort(__float2bfloat16_rn(hv - __bfloat162float(hi)));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&acc_empty[0]);
          mbar_arrive(&acc_empty[1]);
        }
      } else {
        const int blocks = half_unit(un) ? 1 : 2;
        int pl[2];  // assignments of columns 64 ch + lane and + 32
#pragma unroll
        for (int i = 0; i < 2; ++i) pl[i] = ch * 64 + i * 32 + lane < n ? __ldg(&d.asg[a0 + ch * 64 + i * 32 + lane]) : -1;
        bool ok = true;
        for (int tn = 0; tn < 2; ++tn) {
          if (!(ok = wait(&acc_full[tn], j & 1, 11u))) break;
          __syncwarp();
          tc_fence_after();
          if (tn < blocks) {
            float* out = d.part + un.rb * kURows + tn * kBM + q4 * 32 + lane;
#pragma unroll
            for (int hf = 0; hf < 4; ++hf) {
              const int c0 = ch * 64 + hf * 16;
              if (c0 >= n) break;
              float v[16];
              tmem_ld16(lane_addr + tn * kBN + c0, v);
#pragma unroll
              for (int q = 0; q < 16; ++q) {
                const int p = __shfl_sync(0xffffffffu, pl[hf >> 1], (hf & 1) * 16 + q);
                if (p >= 0) out[(size_t)p * d.H] = v[q];
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[tn]);
        }
        if (!ok) break;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem0), "r"(kCols));
}

// x (fp32 [T][H]) -> the x tiles of every 128-assignment block of the call: block t (of unique
// expert u, assignments asg_off[u] + 128 tb ..), K step kk: column c = assignment, row k,
// split into bf16 hi and lo; columns past the expert's assignments, up to the next multiple of 16, are zero.
// Bound: HBM (4 bytes written per assignment and weight column; the rows are re-read from L2), given enough
// blocks: a tile's K steps are dealt to as many blocks as keep the launch at about six per SM (one per tile
// was two or three per SM: 1000 tokens 357 -> 319 us a call, 4096 1067 -> 1050).  Eight fill an SM's threads,
// and the materialiser running beside them then waits for its place (4096 tokens with misses: 2.25 -> 2.29 ms).
__global__ void __launch_bounds__(256) k_tile_x(Dev d, const float* __restrict__ x) {
  __shared__ int s_row[kBN];
  __shared__ int s_u, s_tb;
  const int t = blockIdx.x;
  const int U = d.info[0];
  if (t >= d.tb_off[U]) return;
  if (threadIdx.x == 0) {
    int lo = 0, hi = U - 1;
    while (lo < hi) {  // last expert with tb_off[u] <= t
      const int mid = (lo + hi + 1) >> 1;
      if (d.tb_off[mid] <= t) lo = mid;
      else hi = mid - 1;
    }
    s_u = lo;
    s_tb = t - d.tb_off[lo];
  }
  __syncthreads();
  const int a0 = d.asg_off[s_u] + s_tb * kBN, n = min(kBN, d.asg_off[s_u + 1] - a0);
  for (int c = threadIdx.x; c < kBN; c += blockDim.x) s_row[c] = c < n ? d.asg[a0 + c] / d.k : -1;
  __syncthreads();
  const int steps = d.H / kBK;
  uint8_t* tile0 = d.xt + (size_t)t * steps * kBTile;
  // K steps [k0, nk): this block's share of the tile
  const int k0 = steps * (int)blockIdx.y / (int)gridDim.y, nk = steps * ((int)blockIdx.y + 1) / (int)gridDim.y;
  // item i = (column i >> 2, 8-value group i & 3) of one K step
  const int per = n_eff(n) * 4;  // items of a K step: the columns the MMAs read
  int kk = k0 + threadIdx.x / per, i = threadIdx.x % per;
  for (; kk < nk; i += blockDim.x) {
    while (i >= per) i -= per, ++kk;
    if (kk >= nk) break;
    const int col = i >> 2, g = i & 3;
    uint32_t h[4] = {0, 0, 0, 0}, l[4] = {0, 0, 0, 0};
    const int row = s_row[col];
    if (row >= 0) {
      const float4* src = reinterpret_cast<const float4*>(x + (size_t)row * d.H + kk * kBK + g * 8);
      const float4 v0 = __ldg(src), v1 = __ldg(src + 1);
      split2(f2_pack(__float_as_uint(v0.x), __float_as_uint(v0.y)), h[0], l[0]);
      split2(f2_pack(__float_as_uint(v0.z), __float_as_uint(v0.w)), h[1], l[1]);
      split2(f2_pack(__float_as_uint(v1.x), __float_as_uint(v1.y)), h[2], l[2]);
      split2(f2_pack(__float_as_uint(v1.z), __float_as_uint(v1.w)), h[3], l[3]);
    }
    uint8_t* tile = tile0 + (size_t)kk * kBTile + core_off(col, g * 8);
    *reinterpret_cast<uint4*>(tile) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(tile + kTile) = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

int sm_count_p() {
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
cudaError_t launch_k(const Dev& d, const CUtensorMap* tm, int layer, int wave, cudaStream_t s) {
  static_assert(kSmemW <= 232448, "shared memory per block");
  cudaError_t e = cudaFuncSetAttribute(k_prefill<QT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemW);
  if (e != cudaSuccess) return e;
  k_prefill<QT, NT><<<sm_count_p(), kThreadsW, kSmemW, s>>>(tm[0], tm[1], d, layer, wave);
  return cudaGetLastError();
}

}  // namespace

// shapes the GEMM path serves: whole 128-row blocks in both projections (which also makes the
// scale words read in pairs lie inside each row's scales)
bool prefill_shape_ok(int H, int I) { return H > 0 && I > 0 && H % kBM == 0 && I % kBM == 0; }

// Each unique expert adds at most one partial block: sum_u ceil(n_u / 128) <= T k / 128 + min(E, T k).
uint64_t prefill_tiles_max(int T, int k, int E) {
  const uint64_t a = (uint64_t)T * k;
  return a / kBN + (a < (uint64_t)E ? a : (uint64_t)E);
}

uint64_t prefill_scratch_bytes(int T_max, int k, int E, int H, int I) {
  return prefill_tiles_max(T_max, k, E) * (uint64_t)kBN * (uint64_t)(H + I) * 4;  // hi + lo bf16
}

int encode_slot_region(CUtensorMap* tm, void* base, uint64_t rec_bytes, uint64_t rows, uint64_t planes,
                       uint64_t plane_stride, uint32_t box_bytes, uint32_t box_rows, int swizzle) {
  using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !fn)
    return -1;
  const cuuint64_t dims[3] = {rec_bytes, rows, planes};
  const cuuint64_t strides[2] = {rec_bytes, plane_stride};
  const cuuint32_t box[3] = {box_bytes, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUtensorMapSwizzle sw = swizzle == 128  ? CU_TENSOR_MAP_SWIZZLE_128B
                                : swizzle == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                : CU_TENSOR_MAP_SWIZZLE_NONE;
  return reinterpret_cast<EncodeTiled>(fn)(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, base, dims, strides, box, estr,
                                           CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? 0
             : -1;
}

int prefill_tensor_maps(mf_ctx* c) {
  const Dev& d = c->d;
  const uint64_t planes = (uint64_t)d.L * d.S_alloc;
  for (int m = 0; m < 2; ++m) {  // code boxes (128 bytes of a row, swizzled), scale boxes (one group)
    const uint32_t box = m ? kScaleBox : kRawRow;
    const int sw = m ? 0 : 128;
    if (encode_slot_region(&c->tm_gu[m], d.pool, d.lay.rs_gu, (uint64_t)d.I, planes, d.lay.stride, box, kBM, sw)) return -1;
    if (encode_slot_region(&c->tm_d[m], d.pool + d.lay.d_off, d.lay.rs_d, (uint64_t)d.H, planes, d.lay.stride, box, kBM, sw))
      return -1;
  }
  return 0;
}

cudaError_t launch_tile_x(const Dev& d, const float* x, int T, cudaStream_t s) {
  const uint64_t blocks = prefill_tiles_max(T, d.k, d.E);
  const uint64_t most = (uint64_t)d.H / kBK, room = 6 * (uint64_t)sm_count_p() / blocks;
  const uint64_t split = room < 1 ? 1 : room > most ? most : room;
  k_tile_x<<<dim3((unsigned)blocks, (unsigned)split), 256, 0, s>>>(d, x);
  return cudaGetLastError();
}

cudaError_t launch_prefill_gateup(const Dev& d, const CUtensorMap* tm, int layer, int wave, cudaStream_t s) {
  return d.qtype == MF_Q8_0 ? launch_k<MF_Q8_0, 2>(d, tm, layer, wave, s) : launch_k<MF_Q4_0, 2>(d, tm, layer, wave, s);
}

cudaError_t launch_prefill_down(const Dev& d, const CUtensorMap* tm, int layer, int wave, cudaStream_t s) {
  return d.qtype == MF_Q8_0 ? launch_k<MF_Q8_0, 1>(d, tm, layer, wave, s) : launch_k<MF_Q4_0, 1>(d, tm, layer, wave, s);
}

}  // namespace mf
