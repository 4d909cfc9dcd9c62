// Activations of calls with several tokens below the GEMM threshold, in the form the streaming expert
// kernels read (mf_stream.cu): three exact bfloat16 pieces per value, per K chunk of kStreamK values
// [piece][kStreamK], in the kernels' K order (internal).
#pragma once

#include "mf_dequant.cuh"

namespace mf {

constexpr int kStreamK = 128;
static_assert(kStreamChunkBytes == 3 * kStreamK * 2, "pieces of one K chunk");

// position of element e (of a 32-weight block) in the activation pieces
template <int QT>
__device__ __forceinline__ int stream_pos(int e) {
  if constexpr (QT == dq::kQ8) return e;
  return ((e & 12) << 1) | ((e & 16) >> 2) | (e & 3);
}

// v = p0 + p1 + p2 exactly, each a bfloat16 (the top 8 bits of v, of the remainder, and the last 8)
__device__ __forceinline__ void split3(float v, uint16_t (&p)[3]) {
  const uint32_t b0 = __float_as_uint(v) & 0xFFFF0000u;
  const float r1 = v - __uint_as_float(b0);
  const uint32_t b1 = __float_as_uint(r1) & 0xFFFF0000u;
  const float r2 = r1 - __uint_as_float(b1);
  p[0] = (uint16_t)(b0 >> 16);
  p[1] = (uint16_t)(b1 >> 16);
  p[2] = (uint16_t)(__float_as_uint(r2) >> 16);
}

// Token t of x [T][H] -> the pieces of 2^-e x and e (d.xs, d.xe), by one block of kThreads threads;
// s_m: kThreads / 32 floats of shared memory.
template <int QT, int kThreads>
__device__ __forceinline__ void split_token(const Dev& d, const float* __restrict__ x, int t, float* s_m) {
  const int H = d.H, KC = (H + kStreamK - 1) / kStreamK;
  const float4* row = reinterpret_cast<const float4*>(x + (size_t)t * H);
  uint8_t* out = d.xs + (size_t)t * KC * kStreamChunkBytes;
  float m = 0.f;
  for (int i = threadIdx.x; i < H / 4; i += kThreads) {
    const float4 v = row[i];
    m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kThreads / 32; ++i) m = fmaxf(m, s_m[i]);
  const int e = dq::vec_exponent(m);
  if (threadIdx.x == 0) d.xe[t] = e;
  for (int i = threadIdx.x; i < H / 4; i += kThreads) {  // four values in a row stay together in the pieces
    const float4 f = row[i];
    const float v[4] = {f.x, f.y, f.z, f.w};
    uint16_t p[4][3];
#pragma unroll
    for (int q = 0; q < 4; ++q) split3(dq::scale2(v[q], -e), p[q]);
    const int el = 4 * i;
    uint16_t* o = reinterpret_cast<uint16_t*>(out + (size_t)(el / kStreamK) * kStreamChunkBytes) +
                  ((el & (kStreamK - 1) & ~31) | stream_pos<QT>(el & 31));
#pragma unroll
    for (int c = 0; c < 3; ++c)
      *reinterpret_cast<uint2*>(o + c * kStreamK) =
          make_uint2(p[0][c] | (uint32_t)p[1][c] << 16, p[2][c] | (uint32_t)p[3][c] << 16);
  }
}

}  // namespace mf
