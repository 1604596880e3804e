// The transform of one real row by a group of T = L/V <= 32 threads on the
// register FFTs: 16 values per thread (shf_fft16.cuh; half widths 32, 64, 128,
// 256, 512) or 12, 20 or 32 (shf_fftv.cuh: 3 2^a, 5 2^a, 1024), behind one interface
// for the kernels that take any of them.
#pragma once

#include "shf_fast.h"
#include "shf_fft16.cuh"
#include "shf_fftv.cuh"

namespace shf {
namespace fast {

__host__ __device__ constexpr bool half16(int L) { return L == 32 || L == 64 || L == 128 || L == 256 || L == 512; }
__host__ __device__ constexpr bool half_ok(int L) { return half16(L) || rv::supported(L); }
__host__ __device__ constexpr int even2(int n) { return (n + 1) & ~1; }

// The transform of one row: 16 values per thread or V.
template <int L, bool R16 = half16(L)>
struct Rows;
template <int L>
struct Rows<L, true> {
  static constexpr int V = 16;
  static constexpr int BUF = even2(reg::row_buf(L));
  static constexpr int PT = even2(r16::Passes<L>::TWSIZE);
  __device__ static void tables(float2* pt, const float2* tw) {
    r16::build_pass_twiddles<L, 2>(pt, tw, threadIdx.x, blockDim.x);
  }
  template <int S>
  __device__ static void fft(float2 (&v)[16], int tt, float2* fb, const float2* pt) {
    r16::row_fft<L, S>(v, tt, fb, pt, 0);
  }
  __device__ static void pack(float2 (&v)[16], int k, int tt, float2 ra, float2 rb, float2& prev, const float2* tw) {
    r16::pack_step<L>(v, k, tt, ra, rb, prev, tw);
  }
  __device__ static float2 unpack(const float2 (&v)[16], int q, int tt, float2 r, const float2* tw) {
    return r16::unpack_value<L>(v, q, tt, r, tw);
  }
};
template <int L>
struct Rows<L, false> {
  static constexpr int V = rv::vals_for(L);
  static constexpr int BUF = even2(rv::row_buf(L));
  static constexpr int PT = even2(rv::Passes<L>::TWSIZE);
  __device__ static void tables(float2* pt, const float2* tw) {
    rv::build_pass_twiddles<L, 2>(pt, tw, threadIdx.x, blockDim.x);
  }
  template <int S>
  __device__ static void fft(float2 (&v)[V], int tt, float2* fb, const float2* pt) {
    rv::row_fft<L, S>(v, tt, fb, pt);
  }
  __device__ static void pack(float2 (&v)[V], int k, int tt, float2 ra, float2 rb, float2& prev, const float2* tw) {
    rv::pack_step<L>(v, k, tt, ra, rb, prev, tw);
  }
  __device__ static float2 unpack(const float2 (&v)[V], int q, int tt, float2 r, const float2* tw) {
    return rv::unpack_value<L>(v, q, tt, r, tw);
  }
};

// Inverse packing of the registers X_{tt + k T} (prev: X_L) in place, the
// partners by shuffle; every lane of the warp takes part.
template <int L>
__device__ __forceinline__ void pack_row(float2 (&v)[Rows<L>::V], int tt, int partner, float2 prev, const float2* tw) {
  constexpr int V = Rows<L>::V;
#pragma unroll
  for (int k = 0; k < V / 2; ++k) {
    float2 ra, rb;
    ra.x = __shfl_sync(0xffffffffu, v[V - 1 - k].x, partner);
    ra.y = __shfl_sync(0xffffffffu, v[V - 1 - k].y, partner);
    rb.x = __shfl_sync(0xffffffffu, v[k].x, partner);
    rb.y = __shfl_sync(0xffffffffu, v[k].y, partner);
    Rows<L>::pack(v, k, tt, ra, rb, prev, tw);
  }
}

}  // namespace fast
}  // namespace shf
