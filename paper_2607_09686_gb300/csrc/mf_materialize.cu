// Materialisation of missed experts: pinned host pack -> HBM slot (section "Native Serving
// Path": on a miss the runtime copies the requested expert block into an available slot).  With
// a file-backed split-pack the host first reads the wave's misses from the file into pinned
// staging (in miss order) and the same kernel copies them from there.
//
// The misses are decided on the device (slot resolve), so the copy is driven by the GPU
// itself: SMs load 16-byte vectors straight from the pinned, device-mapped pack over the
// CPU-GPU link and store them into the slot, with no host round trip.  The wave's missed
// payloads are dealt to the blocks in chunks, 12 16-byte loads in flight per thread, so that every block
// has copies in flight however small a payload is (one payload after another left most blocks idle: 35
// misses of 418 KB took 393 us, 37 GB/s).  A call of one wave has nothing beside the copy: a few large
// blocks on the call's own stream.  In a call of several waves the copy runs on the context's side
// stream beside the persistent expert kernels (one block per SM with a fixed share of the work): one
// block of 64 threads per SM, with at most 64 registers a thread, so that it fits beside a GEMM block
// (which has all but 2048 registers of each SM sub-partition) or a streaming block.  4096 Q4_0 tokens
// on a cold 15 % cache: 2.26 ms a call; 64 streams in waves: 1.31 ms (1.50 with 128 threads, of which
// the streaming blocks leave no room for four warps).  The kernels here ask
// for the largest shared-memory carveout although they use none: an SM runs blocks of one
// carveout at a time, so only then can they share SMs with a running expert-FFN kernel (which
// needs most of the shared memory) instead of holding those SMs until they finish.
//
// Calls with several waves stage the misses of wave w + 1 (one payload per miss, in miss
// order) while wave w computes: the slots they go to may still be read by wave w.  Once wave w
// is done, k_stage_commit copies the staged payloads HBM -> HBM into their slots.
#include "mf_internal.cuh"

namespace mf {
namespace {

constexpr int kUnroll = 12;
constexpr int kMatThreadsSpread = 64;  // one block per SM
constexpr int kMatThreadsDense = 512;  // one block per 8 SMs

// dst_stage: null to write each miss into its slot, else miss m of the wave goes to
// dst_stage + m * stride
// (Launch bounds of 1024 threads: at most 64 registers.)
__global__ void __launch_bounds__(1024) k_materialize(Dev d, int layer, int wave, uint8_t* dst_stage) {
  pdl_trigger();
  pdl_wait();
  const int n_miss = d.info[2 + wave];
  const uint32_t nvec = (uint32_t)(d.lay.stride / 16);  // 16-byte vectors per payload
  const uint32_t chunk = blockDim.x * kUnroll, per = (nvec + chunk - 1) / chunk;
#pragma unroll 1
  for (uint32_t c = blockIdx.x; c < (uint32_t)n_miss * per; c += gridDim.x) {
    const uint32_t m = c / per, i0 = (c - m * per) * chunk + threadIdx.x;
    const int u = d.miss_list[wave * d.S_active + m];
    const uint4* src = reinterpret_cast<const uint4*>(
        d.fstage ? d.fstage + (size_t)m * d.fstride  // a file-backed pack: the host staged miss m here
                 : d.pack + ((size_t)layer * d.E + d.uniq[u]) * d.lay.stride);
    uint4* dst = reinterpret_cast<uint4*>(dst_stage ? dst_stage + (size_t)m * d.lay.stride
                                                    : d.pool + ((size_t)layer * d.S_alloc + d.uslot[u]) * d.lay.stride);
    uint4 v[kUnroll];
#pragma unroll
    for (int r = 0; r < kUnroll; ++r) {  // all loads first: kUnroll transfers in flight per thread
      const uint32_t i = i0 + r * blockDim.x;
      if (i < nvec) v[r] = ld_stream(src + i);
    }
#pragma unroll
    for (int r = 0; r < kUnroll; ++r) {
      const uint32_t i = i0 + r * blockDim.x;
      if (i < nvec) dst[i] = v[r];
    }
  }
}

// the wave's staged payloads into their slots (HBM -> HBM)
__global__ void __launch_bounds__(256) k_stage_commit(Dev d, int layer, int wave, const uint8_t* __restrict__ stage) {
  const int n_miss = d.info[2 + wave];
  const size_t nvec = d.lay.stride / 16;
  const size_t step = (size_t)gridDim.x * blockDim.x * 4;
  for (int m = 0; m < n_miss; ++m) {
    const int u = d.miss_list[wave * d.S_active + m];
    const uint4* src = reinterpret_cast<const uint4*>(stage + (size_t)m * d.lay.stride);
    uint4* dst = reinterpret_cast<uint4*>(d.pool + ((size_t)layer * d.S_alloc + d.uslot[u]) * d.lay.stride);
    for (size_t i0 = (size_t)blockIdx.x * blockDim.x * 4 + threadIdx.x; i0 < nvec; i0 += step) {
      uint4 v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const size_t i = i0 + (size_t)r * blockDim.x;
        if (i < nvec) v[r] = src[i];
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const size_t i = i0 + (size_t)r * blockDim.x;
        if (i < nvec) dst[i] = v[r];
      }
    }
  }
}

int n_sm() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

}  // namespace

cudaError_t max_shared_carveout() {
  static cudaError_t e = [] {
    cudaError_t r = cudaFuncSetAttribute(k_materialize, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(k_stage_commit, cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
    return r;
  }();
  return e;
}

cudaError_t launch_materialize(const Dev& d, int layer, int wave, int max_miss, cudaStream_t s, uint8_t* dst_stage,
                               bool spread, bool overlap) {
  if (max_miss <= 0) return cudaSuccess;
  cudaError_t e = max_shared_carveout();
  if (e != cudaSuccess) return e;
  if (spread)
    return launch_pdl(overlap, k_materialize, dim3(n_sm()), dim3(kMatThreadsSpread), 0, s, d, layer, wave, dst_stage);
  return launch_pdl(overlap, k_materialize, dim3((n_sm() + 7) / 8), dim3(kMatThreadsDense), 0, s, d, layer, wave, dst_stage);
}

cudaError_t launch_stage_commit(const Dev& d, int layer, int wave, const uint8_t* stage, cudaStream_t s) {
  cudaError_t e = max_shared_carveout();
  if (e != cudaSuccess) return e;
  k_stage_commit<<<2 * n_sm(), 256, 0, s>>>(d, layer, wave, stage);
  return cudaGetLastError();
}

}  // namespace mf
