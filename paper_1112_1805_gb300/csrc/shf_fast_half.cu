// Single row transforms on the register FFTs of the v-step: half spectra ->
// real rows and real rows -> half spectra, for the half widths with 16 values
// per thread (32, 64, 128, 256, 512) and with 12, 20 or 32 (shf_fftv.cuh: 3 2^a,
// 5 2^a and 1024 with groups inside a warp).  The analysis, the synthesis, the
// reverse sweep's S Qbar and S^T and the readouts use them; other half widths
// take the staged kernels of shf_transform.cu.
//
// Resident CTAs of row groups of T = L/V threads (32/T per warp) loop over the
// rows r = fl H + row of the wave's planes.  The inverse reads the spectrum
// columns of the filter's range from L2 (the next row's prefetched into L1) and
// streams the real row out; the forward keeps the next real row in registers
// while the current one is transformed (V <= 16).  Both move 8 B per value of
// DRAM and are bound by that and by instruction issue (half of the v-step's
// instructions).  CTAs shrink to 128, 64 or 32 threads when the rows would not
// give every SM two of 256.
#include <algorithm>

#include "shf_fast.h"
#include "shf_rows.cuh"

namespace shf {
namespace fast {
namespace {

template <int L>
struct HalfGeo {
  static constexpr int V = Rows<L>::V;
  static constexpr int T = L / V;  // threads per row, at most a warp
  static_assert(T <= 32 && 32 % T == 0, "row groups inside a warp");
  static constexpr int RAW = Rows<L>::BUF;
  static constexpr int STRIDE = T >= 16 ? RAW : RAW + ((T - RAW % 16) % 16 + 16) % 16;
  static constexpr int TW = even2(L + 1);
  static constexpr int PT = Rows<L>::PT;
  static constexpr int MINB = V == 32 ? 1 : 2;
  __host__ static size_t smem(int threads) {
    return sizeof(float2) * (static_cast<size_t>(TW) + PT + static_cast<size_t>(threads / T) * STRIDE);
  }
};

// Rows of a wave: planes fl = (channel - l0) nf + (f - f0) of the spectra at
// `pitch`; their real planes are channel eta + f.
struct RowSet {
  const int2* ranges;  // columns that are not zero, per filter (nullptr: all)
  int H, pitch, eta, l0, f0, nf, nv;
};

template <int L>
__device__ __forceinline__ void half_tables(float2* tw, float2* pt, const float2* __restrict__ twW) {
  load_table(tw, twW, L + 1);
  Rows<L>::tables(pt, twW);
}

// The group's position and its walk over the rows.
template <int L>
struct Walk {
  int tt, grp, partner, fl, row, gq, gr, niter;
  __device__ Walk(const RowSet& a) {
    constexpr int T = HalfGeo<L>::T;
    const int lane = threadIdx.x & 31;
    tt = threadIdx.x & (T - 1);
    grp = threadIdx.x / T;
    partner = (lane - tt) + ((T - tt) & (T - 1));
    const int rpc = blockDim.x / T, G = gridDim.x * rpc, gid = blockIdx.x * rpc + grp;
    const long long rows = static_cast<long long>(a.nv) * a.H;
    niter = static_cast<int>((rows + G - 1) / G);  // the same for every group: all lanes take part in the shuffles
    fl = gid / a.H;
    row = gid - fl * a.H;
    gq = G / a.H;
    gr = G - gq * a.H;
  }
  __device__ void next(int H, int& f, int& r) const {
    f += gq;
    r += gr;
    if (r >= H) {
      r -= H;
      ++f;
    }
  }
};
__device__ __forceinline__ int filter_of(const RowSet& a, int fl, int& chan) {
  const int q = fl / a.nf;
  chan = a.l0 + q;
  return a.f0 + fl - q * a.nf;
}

// out = scale * row-inverse of the half spectra X.
template <int L>
__global__ void __launch_bounds__(256, HalfGeo<L>::MINB)
    k_wrow_inv(const float2* __restrict__ X, float2* __restrict__ out, const RowSet a, float scale,
               const float2* __restrict__ twW) {
  using G = HalfGeo<L>;
  constexpr int T = G::T, V = G::V;
  extern __shared__ __align__(16) float2 sm[];
  float2* tw = sm;
  float2* pt = tw + G::TW;
  Walk<L> wk(a);
  float2* fb = pt + G::PT + wk.grp * G::STRIDE;
  half_tables<L>(tw, pt, twW);
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  const int tt = wk.tt;
  auto span = [&](int fl, int& c0, int& c1) {
    int ch;
    const int f = filter_of(a, fl, ch);
    c0 = 0;
    c1 = L;
    if (a.ranges) {
      const int2 r = a.ranges[f];
      c0 = r.x;
      c1 = min(r.y, L);
    }
  };
  for (int it = 0; it < wk.niter; ++it) {
    const bool live = wk.fl < a.nv;
    const int fl = live ? wk.fl : 0, row = live ? wk.row : 0;
    int fln = wk.fl, rown = wk.row, c0, c1;
    wk.next(a.H, fln, rown);
    span(fl, c0, c1);
    const float2* x = X + (static_cast<size_t>(fl) * a.H + row) * a.pitch;
    if (fln < a.nv) {  // the next row's columns into L1
      int n0, n1;
      span(fln, n0, n1);
      const char* base = reinterpret_cast<const char*>(X + (static_cast<size_t>(fln) * a.H + rown) * a.pitch + n0);
      const int bytes = (n1 - n0 + 1) * 8;
      for (int o = 128 * tt; o < bytes; o += 128 * T) asm volatile("prefetch.global.L1 [%0];" ::"l"(base + o));
    }
    float2 v[V];
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int n = tt + k * T;
      v[k] = live && n >= c0 && n <= c1 ? __ldca(x + n) : make_float2(0.f, 0.f);
    }
    const float2 prev = live && c1 >= L ? __ldca(x + L) : make_float2(0.f, 0.f);
    pack_row<L>(v, tt, wk.partner, prev, tw);
    Rows<L>::template fft<+1>(v, tt, fb, pt);
    if (live) {
      int ch;
      const int f = filter_of(a, fl, ch);
      float2* o = out + ((static_cast<size_t>(ch) * a.eta + f) * a.H + row) * L + tt;
#pragma unroll
      for (int k = 0; k < V; ++k) __stcs(o + k * T, c_scale(v[k], scale));
    }
    wk.fl = fln;
    wk.row = rown;
  }
}

// X = row-forward of the real rows, on the column tiles (8 columns, or 4 for
// heights above 1024) that the filter's range touches.
template <int L>
__global__ void __launch_bounds__(256, HalfGeo<L>::MINB)
    k_wrow_fwd(const float2* __restrict__ in, float2* __restrict__ X, const RowSet a, const float2* __restrict__ twW) {
  using G = HalfGeo<L>;
  constexpr int T = G::T, V = G::V;
  constexpr bool AHEAD = V <= 16;  // the next row's values in registers (20 would spill)
  extern __shared__ __align__(16) float2 sm[];
  float2* tw = sm;
  float2* pt = tw + G::TW;
  Walk<L> wk(a);
  float2* fb = pt + G::PT + wk.grp * G::STRIDE;
  half_tables<L>(tw, pt, twW);
  pdl_wait();
  pdl_trigger();
  const int tt = wk.tt, cmask = reg::col_batch(a.H) - 1;
  auto load = [&](float2 (&v)[V], int fl, int row) {
    int ch;
    const int f = filter_of(a, fl < a.nv ? fl : 0, ch);
    const float2* p = in + ((static_cast<size_t>(ch) * a.eta + f) * a.H + (fl < a.nv ? row : 0)) * L + tt;
#pragma unroll
    for (int k = 0; k < V; ++k) v[k] = fl < a.nv ? __ldcs(p + k * T) : make_float2(0.f, 0.f);
  };
  float2 nx[AHEAD ? V : 1];
  if constexpr (AHEAD) load(nx, wk.fl, wk.row);
  __syncthreads();
  for (int it = 0; it < wk.niter; ++it) {
    const bool live = wk.fl < a.nv;
    const int fl = live ? wk.fl : 0, row = live ? wk.row : 0;
    int fln = wk.fl, rown = wk.row, ch, c0 = 0, c1 = L;
    wk.next(a.H, fln, rown);
    if (a.ranges) {
      const int2 r = a.ranges[filter_of(a, fl, ch)];
      c0 = r.x <= r.y ? r.x & ~cmask : L + 1;
      c1 = r.x <= r.y ? min(L, r.y | cmask) : -1;
    }
    float2 v[V];
    if constexpr (AHEAD) {
#pragma unroll
      for (int k = 0; k < V; ++k) v[k] = nx[k];
      load(nx, fln, rown);
    } else {
      load(v, wk.fl, wk.row);
    }
    Rows<L>::template fft<-1>(v, tt, fb, pt);
    float2* x = X + (static_cast<size_t>(fl) * a.H + row) * a.pitch;
#pragma unroll
    for (int q = 0; q < V; ++q) {
      float2 r;
      r.x = __shfl_sync(0xffffffffu, v[V - 1 - q].x, wk.partner);
      r.y = __shfl_sync(0xffffffffu, v[V - 1 - q].y, wk.partner);
      const int i = tt + q * T;
      if (live && i >= c0 && i <= c1) x[i] = Rows<L>::unpack(v, q, tt, r, tw);
    }
    if (live && tt == 0 && c1 >= L) x[L] = make_float2(v[0].x - v[0].y, 0.f);  // i = L: e^{-i pi} = -1
    wk.fl = fln;
    wk.row = rown;
  }
}

template <int L>
cudaError_t prepare_half_t() {
  if constexpr (half_ok(L)) {
    cudaError_t e = allow_smem(k_wrow_inv<L>, HalfGeo<L>::smem(256));
    return e == cudaSuccess ? allow_smem(k_wrow_fwd<L>, HalfGeo<L>::smem(256)) : e;
  }
  return cudaSuccess;
}

int half_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 152;
  return sms;
}

// CTA size and grid: 256 threads while that gives every SM two CTAs, else
// smaller; at most the resident CTAs.
template <int L, class K>
cudaError_t half_shape(K kern, long long rows, int* threads, int* ctas) {
  const int sms = half_sms();
  int nt = 256;
  while (nt > 32 && (rows * HalfGeo<L>::T + nt - 1) / nt < 2 * sms) nt /= 2;
  int fit = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, nt, HalfGeo<L>::smem(nt));
  if (e != cudaSuccess) return e;
  const long long rpc = nt / HalfGeo<L>::T;
  *threads = nt;
  *ctas = static_cast<int>(std::min<long long>((rows + rpc - 1) / rpc, static_cast<long long>(std::max(fit, 1)) * sms));
  return cudaSuccess;
}

template <int L>
cudaError_t inv_t(const RowSet& a, const float2* X, float* out, float scale, const float2* twW, cudaStream_t st) {
  if constexpr (half_ok(L)) {
    int nt = 0, nc = 0;
    cudaError_t e = half_shape<L>(k_wrow_inv<L>, static_cast<long long>(a.nv) * a.H, &nt, &nc);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_wrow_inv<L>, dim3(nc), dim3(nt), HalfGeo<L>::smem(nt), st, X, reinterpret_cast<float2*>(out), a,
                      scale, twW);
  }
  return cudaErrorInvalidValue;
}

template <int L>
cudaError_t fwd_t(const RowSet& a, const float* in, float2* X, const float2* twW, cudaStream_t st) {
  if constexpr (half_ok(L)) {
    int nt = 0, nc = 0;
    cudaError_t e = half_shape<L>(k_wrow_fwd<L>, static_cast<long long>(a.nv) * a.H, &nt, &nc);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_wrow_fwd<L>, dim3(nc), dim3(nt), HalfGeo<L>::smem(nt), st, reinterpret_cast<const float2*>(in), X,
                      a, twW);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool half_rows_ok(int L) {
  switch (L) {
#define SHF_CASE(N) \
  case N:           \
    return half_ok(N);
    SHF_FAST_SIZES(SHF_CASE)
#undef SHF_CASE
    default: return false;
  }
}

cudaError_t prepare_half_kernels(int N) {
  switch (N) {
#define SHF_CASE(M) \
  case M:           \
    return prepare_half_t<M>();
    SHF_FAST_SIZES(SHF_CASE)
#undef SHF_CASE
    default: return cudaSuccess;
  }
}

cudaError_t rows_inv(const Geo& g, const float2* X, int pitch, float* out, const int2* ranges, int eta, const Wave& wv,
                     float scale, cudaStream_t st) {
  const RowSet a{ranges, g.H, pitch, eta, wv.l0, wv.f0, wv.nf, wv.nv};
  switch (g.L) {
#define SHF_CASE(N) \
  case N:           \
    return inv_t<N>(a, X, out, scale, g.twW, st);
    SHF_FAST_SIZES(SHF_CASE)
#undef SHF_CASE
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t rows_fwd(const Geo& g, const float* in, float2* X, int pitch, const int2* ranges, int eta, const Wave& wv,
                     cudaStream_t st) {
  const RowSet a{ranges, g.H, pitch, eta, wv.l0, wv.f0, wv.nf, wv.nv};
  switch (g.L) {
#define SHF_CASE(N) \
  case N:           \
    return fwd_t<N>(a, in, X, g.twW, st);
    SHF_FAST_SIZES(SHF_CASE)
#undef SHF_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fast
}  // namespace shf
