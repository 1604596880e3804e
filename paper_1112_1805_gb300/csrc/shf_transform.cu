// Row kernels of the general lengths (Haeuser & Steidl, arXiv:1112.1805): sizes
// H, W/2 = 2^a 3^b 5^c that the register-FFT path (shf_fast_*.cu) does not
// take, and the transforms of single planes at any size.
//
// A 2-D transform of an H x W real plane is split into row transforms (real
// length W, packed into complex length W/2) and column transforms (complex
// length H) over the W/2+1 columns of the half spectrum.  The filters are real
// and even, so every product of a filter with the spectrum of a real plane is
// again the half spectrum of a real plane.  They also vanish outside a column
// range (compact support, Sec. 2, Remark 1): coefficient spectra are computed,
// stored and read on that range only.
//
// Analysis S (eq. wichtig) in waves of (channel, filter) pairs whose spectra
// stay near the L2 between the launches:
//   row-forward -> column-forward (in place) -> per wave [fan: times W_f,
//   column-inverse] -> row-inverse.
// Synthesis S^T (Fourier-domain form after the Theorem), per wave:
//   row-forward of the coefficient planes -> [gather: column-forward, times
//   W_f, sum over a filter group]; then [reduce: sum over groups in fixed
//   order, column-inverse] -> row-inverse.
// ADMM iteration (Sec. 3), state (b_v, T = column-inverse of the synthesis
// spectrum of v - b_v, w, b_w):
//   k_row_ustep   : T -> S^T(v-b_v); u-step; w-step; b_w; row-forward of u
//   column-forward of u's row spectra
//   per wave: fan; k_row_shrink: row-inverse -> g = b_v + Su; b_v <- clip(g);
//     d = soft(g) - clip(g) = v - b_v; row-forward of d (in place); gather
//   reduce        : synthesis spectrum of d -> T
// Every transform runs on the staged FFTs of shf_gfft.cuh.  Measured against
// full-width spectra of all channels at once and radix-2/3/4/5/8 stages that
// each crossed shared memory: an iteration at 480 x 640, K = 5, J = 4 3.14 ->
// 1.09 ms (u/w-step 70 -> 59 us, fan 776 -> 157, v-step 955 -> 613, gather
// 1213 -> 200, reduce 34 -> 26, column-forward 12); synthesis of three 1080 x
// 1920 channels 7.8 -> 2.5 ms (row-forward 2224 -> 1200 us, gather 5227 ->
// 1180).  The v-step and the row transforms are bound by instruction issue and
// latency (issue slots 40% busy, 127 registers, two CTAs per SM).
#include <algorithm>

#include "shf_fast.h"
#include "shf_gfft.cuh"
#include "shf_internal.h"
#include "shf_simplex.cuh"

namespace shf {

namespace {

using fast::launch_pdl;
using fast::pdl_trigger;
using fast::pdl_wait;

// ---------------------------------------------------------------------------
// One CTA owns RB consecutive rows of one plane.  A real row of length W = 2L
// is handled as the complex row z[n] = x[2n] + i x[2n+1].
// ---------------------------------------------------------------------------

// A plane of a launch: its index, and where its data and its filter are.  A
// plain launch has planes 0, 1, ...; a wave's plane p is filter f0 + p mod nf of
// channel c0 + p / nf, whose coefficients are plane c eta + f.
struct Plane {
  size_t data;  // plane of the real data
  int f;        // filter (waves)
  int c0, c1;   // columns of the half spectrum that are not zero by construction
};
template <bool FILT>
__device__ __forceinline__ Plane plane_of(const Geo& g, const FilterWave& wv) {
  Plane p{blockIdx.y, 0, 0, g.L};
  if constexpr (FILT) {
    const int q = static_cast<int>(blockIdx.y) / wv.nf;
    p.f = wv.f0 + static_cast<int>(blockIdx.y) - q * wv.nf;
    p.data = static_cast<size_t>(wv.c0 + q) * g.eta + p.f;
    if (g.ranges) {
      const int2 r = g.ranges[p.f];
      p.c0 = r.x;
      p.c1 = min(r.y, g.L);
    }
  }
  return p;
}

// Element k of the inverse packing of half-spectrum row X, zero outside [c0, c1].
__device__ __forceinline__ float2 packed(const float2* X, int L, int k, int c0, int c1, const float2* __restrict__ twW) {
  const int m = L - k;
  const float2 a = (k >= c0 && k <= c1) ? X[k] : make_float2(0.f, 0.f);
  const float2 b = (m >= c0 && m <= c1) ? c_conj(X[m]) : make_float2(0.f, 0.f);
  const float2 s = c_add(a, b), d = c_sub(a, b);
  return pack_combine(s, d, twW[k]);
}

// Writes columns [c0, c1] of the half spectra of RB rows from their complex
// transforms Z (rows of L), times `scale`.
__device__ __forceinline__ void store_half(const float2* Z, float2* dst, int pitch, int L, int row0, int rows, int c0,
                                           int c1, float scale, const float2* __restrict__ twW) {
  const int n = c1 - c0 + 1;
  if (n <= 0) return;
  const unsigned m = fdiv_mul(static_cast<unsigned>(n));
  for (int e = threadIdx.x; e < rows * n; e += blockDim.x) {
    const int r = static_cast<int>(fdiv(static_cast<unsigned>(e), m)), k = c0 + e - r * n;
    dst[static_cast<size_t>(row0 + r) * pitch + k] = c_scale(r2c_unpack(Z + r * L, L, k, twW), scale);
  }
}

template <bool FILT>
__global__ void __launch_bounds__(kRowThreads, 2)
    k_row_r2c(const __grid_constant__ Geo g, const float* __restrict__ in, float2* __restrict__ out, int pitch, int RB,
              const __grid_constant__ gf::Batch ba, int bufn, const FilterWave wv, float scale) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int L = g.L, row0 = blockIdx.x * RB, rows = min(RB, g.H - row0);
  pdl_wait();
  pdl_trigger();
  Plane p = plane_of<FILT>(g, wv);
  if (p.c1 < p.c0) return;  // an empty filter: nothing reads its spectrum
  if (FILT) {  // whole column tiles: the register-FFT gather reads those
    const int mask = reg::col_batch(g.H) - 1;
    p.c0 &= ~mask;
    p.c1 = min(g.L, p.c1 | mask);
  }
  const float2* src = reinterpret_cast<const float2*>(in) + p.data * g.H * L + static_cast<size_t>(row0) * L;
  const auto ld = [&](int i, int b) { return b < rows ? src[static_cast<size_t>(b) * L + i] : make_float2(0.f, 0.f); };
  const float2* y = gf::fft_head<-1, false>(g.planL, ba, x, g.ptL, ld);
  float2* Z = x.next();
  const auto st = [&](int i, int b, float2 v) { Z[b * L + i] = v; };
  gf::NoLd nl;
  if (g.planL.nst == 1)
    gf::run_stage<-1, false, gf::kOnly>(g.planL, 0, ba, nullptr, nullptr, g.ptL, ld, st, threadIdx.x, blockDim.x);
  else
    gf::run_stage<-1, false, gf::kLast>(g.planL, g.planL.nst - 1, ba, y, nullptr, g.ptL, nl, st, threadIdx.x, blockDim.x);
  __syncthreads();
  store_half(Z, out + static_cast<size_t>(blockIdx.y) * g.H * pitch, pitch, L, row0, rows, p.c0, p.c1, scale, g.twW);
}

template <bool FILT>
__global__ void __launch_bounds__(kRowThreads, 2)
    k_row_c2r(const __grid_constant__ Geo g, const float2* __restrict__ in, float* __restrict__ out, int pitch, int RB,
              const __grid_constant__ gf::Batch ba, int bufn, const FilterWave wv, float scale) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int L = g.L, row0 = blockIdx.x * RB, rows = min(RB, g.H - row0);
  pdl_wait();
  pdl_trigger();
  const Plane p = plane_of<FILT>(g, wv);
  const float2* src = in + (static_cast<size_t>(blockIdx.y) * g.H + row0) * pitch;
  float2* dst = reinterpret_cast<float2*>(out) + p.data * g.H * L + static_cast<size_t>(row0) * L;
  gf::fft<+1, false>(
      g.planL, ba, x, g.ptL,
      [&](int i, int b) {
        return b < rows ? packed(src + static_cast<size_t>(b) * pitch, L, i, p.c0, p.c1, g.twW) : make_float2(0.f, 0.f);
      },
      [&](int i, int b, float2 v) {
        if (b < rows) {
          if constexpr (FILT)
            __stcs(dst + static_cast<size_t>(b) * L + i, c_scale(v, scale));
          else
            dst[static_cast<size_t>(b) * L + i] = c_scale(v, scale);
        }
      });
}

// The v-step's middle: the inverse transform's last stage, the shrinkage on
// its results and the forward transform's first stage, on the same registers
// (the forward plan is the inverse one reversed, so both stages have the same
// radix and hold the values j + q L/R of a row).
struct Turn {
  const Geo& g;
  const gf::Batch &bi, &bf;
  const float2* in;
  float2* out;
  const float2* src;  // spectra rows (single-stage plans)
  int pitch, rows, c0, c1;
  float2 *b2, *gout;  // b_v rows, optional g rows (pitch L)
  float t, scale;
  template <int R>
  __device__ __forceinline__ void run() {
    const FftStage& gi = g.planL.st[g.planL.nst - 1];
    const FftStage& gfw = g.planLr.st[0];
    const int total = gi.nb * bi.B, L = g.L;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
      int j, b, k = 0;
      gf::item_of<false>(gi, bi, idx, j, b);
      const bool live = b < rows;
      float2* br = b2 + static_cast<size_t>(live ? b : 0) * L;
      float2 bo[R], v[R];
#pragma unroll
      for (int q = 0; q < R; ++q) bo[q] = live ? __ldcs(br + j + q * gi.nb) : make_float2(0.f, 0.f);
      if (g.planL.nst == 1) {
#pragma unroll
        for (int q = 0; q < R; ++q)
          v[q] = live ? packed(src + static_cast<size_t>(b) * pitch, L, j + q * gi.nb, c0, c1, g.twW) : make_float2(0.f, 0.f);
      } else {
        gf::stage_in<R, +1, false>(gi, bi, g.planL.nst == 2, j, b, in, g.ptL, v, k);
      }
      gf::dft<R, +1>(v);
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const float2 gv = c_fma2(make_float2(scale, scale), v[q], bo[q]);
        const float2 c = make_float2(fminf(fmaxf(gv.x, -t), t), fminf(fmaxf(gv.y, -t), t));
        if (live) {
          __stcs(br + j + q * gi.nb, c);
          if (gout) gout[static_cast<size_t>(b) * L + j + q * gi.nb] = gv;
        }
        v[q] = c_fma2(make_float2(-2.f, -2.f), c, gv);  // g - 2 clip(g)
      }
      gf::dft<R, -1>(v);
      gf::stage_out<R, false>(gfw, bf, true, j, b, 0, out, v);
    }
  }
};

// v-step and b_v update (Sec. 3): with c = (S u)_f on this row,
// g = b_v + c, b_v <- clip(g, -t, t) = g - soft(g, t), d = soft(g) - clip(g);
// d (= v - b_v of the new iterate) is transformed back in place.
__global__ void __launch_bounds__(kRowThreads, 2)
    k_row_shrink(const __grid_constant__ Geo g, float2* __restrict__ Y, float* __restrict__ bv,
                 const float* __restrict__ thr, int pitch, int RB, const __grid_constant__ gf::Batch bi,
                 const __grid_constant__ gf::Batch bf, int bufn, const FilterWave wv, float scale,
                 float* __restrict__ gout) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int L = g.L, row0 = blockIdx.x * RB, rows = min(RB, g.H - row0);
  pdl_wait();
  pdl_trigger();
  const Plane p = plane_of<true>(g, wv);
  float2* X = Y + (static_cast<size_t>(blockIdx.y) * g.H + row0) * pitch;
  const size_t off = (p.data * g.H + row0) * L;
  const float2* y = gf::fft_head<+1, false>(g.planL, bi, x, g.ptL, [&](int i, int b) {
    return b < rows ? packed(X + static_cast<size_t>(b) * pitch, L, i, p.c0, p.c1, g.twW) : make_float2(0.f, 0.f);
  });
  float2* z = x.next();
  Turn turn{g,  bi,     bf,   y,    z,    X, pitch, rows, p.c0, p.c1, reinterpret_cast<float2*>(bv) + off,
            gout ? reinterpret_cast<float2*>(gout) + off : nullptr, thr[p.f], scale};
  gf::with_radix(g.planL.st[g.planL.nst - 1].R, turn);
  __syncthreads();
  gf::NoLd nl;
  gf::NoSt ns;
  const float2* in = z;
  for (int s = 1; s + 1 < g.planLr.nst; ++s) {
    float2* o = x.next();
    gf::run_stage<-1, false, gf::kMid>(g.planLr, s, bf, in, o, g.ptLr, nl, ns, threadIdx.x, blockDim.x);
    __syncthreads();
    in = o;
  }
  if (g.planLr.nst > 1) {
    float2* Z = x.next();
    const auto st = [&](int i, int b, float2 v) { Z[b * L + i] = v; };
    gf::run_stage<-1, false, gf::kLast>(g.planLr, g.planLr.nst - 1, bf, in, nullptr, g.ptLr, nl, st, threadIdx.x,
                                        blockDim.x);
    __syncthreads();
    in = Z;
  }
  store_half(in, X - static_cast<size_t>(row0) * pitch, pitch, L, row0, rows, p.c0, p.c1, 1.f, g.twW);
}

constexpr int kL1Threads = kRowThreads;

// Weighted l1 norm of the real planes behind the half spectra: one FP64
// partial per block, fixed summation order.
__global__ void __launch_bounds__(kRowThreads, 2)
    k_row_l1(const __grid_constant__ Geo g, const float2* __restrict__ in, const float* __restrict__ lam, int pitch,
             int RB, const __grid_constant__ gf::Batch ba, int bufn, const FilterWave wv, float scale,
             double* __restrict__ partial) {
  extern __shared__ float2 sm[];
  __shared__ double red[kL1Threads];
  gf::Exchange x{{sm, sm + bufn}};
  const int L = g.L, row0 = blockIdx.x * RB, rows = min(RB, g.H - row0);
  pdl_wait();
  pdl_trigger();
  const Plane p = plane_of<true>(g, wv);
  const float2* src = in + (static_cast<size_t>(blockIdx.y) * g.H + row0) * pitch;
  double acc = 0.0;
  gf::fft<+1, false>(
      g.planL, ba, x, g.ptL,
      [&](int i, int b) {
        return b < rows ? packed(src + static_cast<size_t>(b) * pitch, L, i, p.c0, p.c1, g.twW) : make_float2(0.f, 0.f);
      },
      [&](int, int b, float2 v) {
        if (b < rows) acc += static_cast<double>(fabsf(scale * v.x)) + static_cast<double>(fabsf(scale * v.y));
      });
  red[threadIdx.x] = acc * static_cast<double>(lam[p.f]);
  __syncthreads();
  for (int s = kL1Threads / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[p.data * gridDim.x + blockIdx.x] = red[0];
}

// The v-step with its transforms apart (sweep plans, whose forward transform
// starts with another radix than the inverse one ends with).
__global__ void __launch_bounds__(kRowThreads, 2)
    k_row_shrink_apart(const __grid_constant__ Geo g, float2* __restrict__ Y, float* __restrict__ bv,
                       const float* __restrict__ thr, int pitch, int RB, const __grid_constant__ gf::Batch ba, int bufn,
                       const FilterWave wv, float scale, float* __restrict__ gout) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int L = g.L, row0 = blockIdx.x * RB, rows = min(RB, g.H - row0);
  pdl_wait();
  pdl_trigger();
  const Plane p = plane_of<true>(g, wv);
  float2* X = Y + (static_cast<size_t>(blockIdx.y) * g.H + row0) * pitch;
  const size_t off = (p.data * g.H + row0) * L;
  float2* b2 = reinterpret_cast<float2*>(bv) + off;
  float2* g2 = gout ? reinterpret_cast<float2*>(gout) + off : nullptr;
  const float t = thr[p.f];
  const auto ldx = [&](int i, int b) {
    return b < rows ? packed(X + static_cast<size_t>(b) * pitch, L, i, p.c0, p.c1, g.twW) : make_float2(0.f, 0.f);
  };
  const float2* y = gf::fft_head<+1, false>(g.planL, ba, x, g.ptL, ldx);
  float2* D = x.next();
  const auto shrink = [&](int i, int b, float2 v) {
    float2 d = make_float2(0.f, 0.f);
    if (b < rows) {
      const int e = b * L + i;
      const float2 gv = c_fma2(make_float2(scale, scale), v, b2[e]);
      const float2 c = make_float2(fminf(fmaxf(gv.x, -t), t), fminf(fmaxf(gv.y, -t), t));
      b2[e] = c;
      if (g2) g2[e] = gv;
      d = c_fma2(make_float2(-2.f, -2.f), c, gv);  // g - 2 clip(g)
    }
    D[b * L + i] = d;
  };
  gf::NoLd nl;
  if (g.planL.nst == 1)
    gf::run_stage<+1, false, gf::kOnly>(g.planL, 0, ba, nullptr, nullptr, g.ptL, ldx, shrink, threadIdx.x, blockDim.x);
  else
    gf::run_stage<+1, false, gf::kLast>(g.planL, g.planL.nst - 1, ba, y, nullptr, g.ptL, nl, shrink, threadIdx.x, blockDim.x);
  __syncthreads();
  const auto ldd = [&](int i, int b) { return D[b * L + i]; };
  y = gf::fft_head<-1, false>(g.planL, ba, x, g.ptL, ldd);
  float2* Z = x.next();
  const auto st = [&](int i, int b, float2 v) { Z[b * L + i] = v; };
  if (g.planL.nst == 1)
    gf::run_stage<-1, false, gf::kOnly>(g.planL, 0, ba, nullptr, nullptr, g.ptL, ldd, st, threadIdx.x, blockDim.x);
  else
    gf::run_stage<-1, false, gf::kLast>(g.planL, g.planL.nst - 1, ba, y, nullptr, g.ptL, nl, st, threadIdx.x, blockDim.x);
  __syncthreads();
  store_half(Z, X - static_cast<size_t>(row0) * pitch, pitch, L, row0, rows, p.c0, p.c1, 1.f, g.twW);
}

// u-step (u = 1/2 [S^T(v - b_v) + (w - b_w) - gamma s], A^T A = 2I), w-step
// (pixelwise projection of g_w = b_w + u onto the simplex), b_w = g_w - w,
// and the row-forward transform of u for the next analysis.  KG labels' RB rows
// are transformed as one batch (all labels where shared memory allows: label
// after label the K transforms were a chain of 2 K times the barriers).  Shared
// memory: the exchange buffers and U (K x RB x L complex).
__global__ void __launch_bounds__(kRowThreads)
    k_row_ustep(const __grid_constant__ Geo g, const float2* __restrict__ T, const float* __restrict__ s,
                float* __restrict__ w, float* __restrict__ bw, float* __restrict__ u, float2* __restrict__ Ur,
                float* __restrict__ stv, int K, int RB, int KG, unsigned mRB, const __grid_constant__ gf::Batch ba, int bufn,
                float scale, float gamma) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  float2* U = sm + 2 * bufn;
  const int L = g.L, E = RB * L, Wh = g.Wh, row0 = blockIdx.x * RB, rows = min(RB, g.H - row0);
  const size_t HL = static_cast<size_t>(g.H) * L, HWh = static_cast<size_t>(g.H) * Wh;
  pdl_wait();
  pdl_trigger();
  // sequence b of a batch: row r of label k0 + kk
  const auto split = [&](int b, int& kk) {
    kk = static_cast<int>(fdiv(static_cast<unsigned>(b), mRB));
    return b - kk * RB;
  };
  for (int k0 = 0; k0 < K; k0 += KG) {
    const float2* src = T + k0 * HWh + static_cast<size_t>(row0) * Wh;
    float2* Uk = U + k0 * E;
    gf::fft<+1, false>(
        g.planL, ba, x, g.ptL,
        [&](int i, int b) {
          int kk;
          const int r = split(b, kk);
          return r < rows && k0 + kk < K ? packed(src + kk * HWh + static_cast<size_t>(r) * Wh, L, i, 0, L, g.twW)
                                         : make_float2(0.f, 0.f);
        },
        [&](int i, int b, float2 v) {
          int kk;
          const int r = split(b, kk);
          if (k0 + kk < K) Uk[kk * E + r * L + i] = c_scale(v, scale);
        });
  }
  __syncthreads();
  const float2* s2 = reinterpret_cast<const float2*>(s);
  float2* w2 = reinterpret_cast<float2*>(w);
  float2* bw2 = reinterpret_cast<float2*>(bw);
  float2* u2 = reinterpret_cast<float2*>(u);
  float2* stv2 = reinterpret_cast<float2*>(stv);
  const float hg = 0.5f * gamma;
  for (int e = threadIdx.x; e < E; e += kRowThreads) {
    if (e >= rows * L) {
      for (int k = 0; k < K; ++k) U[k * E + e] = make_float2(0.f, 0.f);
      continue;
    }
    const size_t off = static_cast<size_t>(row0) * L + e;
    float gx[kMaxK], gy[kMaxK];
#pragma unroll
    for (int k = 0; k < kMaxK; ++k) {
      gx[k] = 0.f;
      gy[k] = 0.f;
      if (k < K) {
        const float2 st = U[k * E + e];
        const float2 wv = w2[k * HL + off], bv = bw2[k * HL + off], sv = s2[k * HL + off];
        const float ux = 0.5f * (st.x + (wv.x - bv.x)) - hg * sv.x;
        const float uy = 0.5f * (st.y + (wv.y - bv.y)) - hg * sv.y;
        u2[k * HL + off] = make_float2(ux, uy);
        if (stv) stv2[k * HL + off] = st;
        U[k * E + e] = make_float2(ux, uy);
        gx[k] = bv.x + ux;
        gy[k] = bv.y + uy;
      }
    }
    float px[kMaxK], py[kMaxK];
#pragma unroll
    for (int k = 0; k < kMaxK; ++k) {
      px[k] = gx[k];
      py[k] = gy[k];
    }
    simplex_project<kMaxK>(px, K);
    simplex_project<kMaxK>(py, K);
#pragma unroll
    for (int k = 0; k < kMaxK; ++k) {
      if (k < K) {
        w2[k * HL + off] = make_float2(px[k], py[k]);
        bw2[k * HL + off] = make_float2(gx[k] - px[k], gy[k] - py[k]);
      }
    }
  }
  __syncthreads();
  for (int k0 = 0; k0 < K; k0 += KG) {
    const float2* Uk = U + k0 * E;
    const int nk = min(KG, K - k0);
    const auto ld = [&](int i, int b) {
      int kk;
      const int r = split(b, kk);
      return kk < nk ? Uk[kk * E + r * L + i] : make_float2(0.f, 0.f);
    };
    const float2* y = gf::fft_head<-1, false>(g.planL, ba, x, g.ptL, ld);
    float2* Z = x.next();
    const auto st = [&](int i, int b, float2 v) { Z[b * L + i] = v; };
    gf::NoLd nl;
    if (g.planL.nst == 1)
      gf::run_stage<-1, false, gf::kOnly>(g.planL, 0, ba, nullptr, nullptr, g.ptL, ld, st, threadIdx.x, blockDim.x);
    else
      gf::run_stage<-1, false, gf::kLast>(g.planL, g.planL.nst - 1, ba, y, nullptr, g.ptL, nl, st, threadIdx.x,
                                          blockDim.x);
    __syncthreads();
    for (int kk = 0; kk < nk; ++kk)
      store_half(Z + kk * E, Ur + (k0 + kk) * HWh, Wh, L, row0, rows, 0, L, 1.f, g.twW);
  }
}

template <typename K>
cudaError_t set_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// Rows of a u/w-step CTA that a tile shape is accepted by.
int ustep_rows(const Geo& g, int K) {
  int rb = 65536 / (g.L * (8 * K + 16));
  if (rb < 1) rb = 1;
  if (rb > g.RB) rb = g.RB;
  return rb;
}

// Padding of the first exchange of a row plan: only even first radices need
// it, and only where the padded buffers still fit.
constexpr size_t kRowSmemMax = 227 * 1024 - sizeof(double) * kL1Threads;
int row_pad(const FftPlan& p, int rb, int extra) {
  const size_t need = sizeof(float2) * (2 * static_cast<size_t>(gf::buf_elems(p, rb, 1)) + static_cast<size_t>(extra));
  return p.nst > 1 && p.st[0].R % 2 == 0 && need <= kRowSmemMax ? 1 : 0;
}

// Launch shape of a row kernel: the batch of the plan and its buffers.
struct RowShape {
  gf::Batch ba;
  int bufn;
  size_t smem;
};
RowShape row_shape(const FftPlan& p, int rb) {
  const int pad = row_pad(p, rb, 0), n = gf::buf_elems(p, rb, pad);
  return RowShape{gf::make_batch(p, rb, pad), n, sizeof(float2) * 2 * static_cast<size_t>(n)};
}

}  // namespace

cudaError_t prepare_col_general(int optin);

// Raises the dynamic shared-memory limits of the kernels that g's transforms
// launch, outside any capture: the staged kernels' to the device's opt-in
// maximum (an upper bound only), the single row transforms' of g's width.
cudaError_t prepare_kernels(const Geo& g) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const cudaError_t errs[] = {
      set_smem(k_row_r2c<false>, optin), set_smem(k_row_r2c<true>, optin), set_smem(k_row_c2r<false>, optin),
      set_smem(k_row_c2r<true>, optin),  set_smem(k_row_shrink, optin),
      set_smem(k_row_shrink_apart, optin),
      set_smem(k_row_l1, optin - static_cast<int>(sizeof(double)) * kL1Threads),
      set_smem(k_row_ustep, optin),      prepare_col_general(optin),
      fast::prepare_half_kernels(g.L)};
  for (cudaError_t x : errs)
    if (x != cudaSuccess) return x;
  return cudaSuccess;
}

int max_dynamic_smem_needed(const Geo& g, int K) {
  const int col = static_cast<int>(2 * sizeof(float2) * g.H * g.TC);
  const int row = static_cast<int>(2 * sizeof(float2) * g.RB * g.L);
  const int us = static_cast<int>(sizeof(float2) * static_cast<size_t>(ustep_rows(g, K)) * g.L * (2 + K));
  return std::max(col, std::max(row, us));
}

bool set_generic_tiles(Geo* g, int TC, int RB, int K, int smem_limit) {
  if (TC < 1 || RB < 1 || TC > g->Wh || RB > g->H) return false;
  const int per = (g->H * TC + kColThreads - 1) / kColThreads;
  if (per > 32) return false;
  Geo t = *g;
  t.TC = TC;
  t.ntiles = (t.Wh + TC - 1) / TC;
  t.RB = RB;
  const size_t col = 2 * sizeof(float2) * static_cast<size_t>(t.H) * t.TC;
  const size_t row = 2 * sizeof(float2) * static_cast<size_t>(t.RB) * t.L;
  const size_t us = sizeof(float2) * static_cast<size_t>(ustep_rows(t, K)) * t.L * (2 + K);
  const size_t lim = static_cast<size_t>(smem_limit);
  if (col > lim || row + sizeof(double) * kL1Threads > lim || us > lim) return false;
  *g = t;
  return true;
}

namespace {
// A plain launch's planes as one wave of single-filter channels.
fast::Wave plain(int planes) { return fast::Wave{0, 0, 1, planes}; }
bool half_rows(const Geo& g) { return !g.staged && fast::half_rows_ok(g.L); }
fast::Wave fast_wave_of(const FilterWave& wv) { return fast::Wave{wv.c0, wv.f0, wv.nf, wv.nc * wv.nf}; }
}  // namespace

cudaError_t run_row_r2c(const Geo& g, const float* in, float2* out, int planes, float scale, cudaStream_t st) {
  if (scale == 1.f && half_rows(g)) return fast::rows_fwd(g, in, out, g.Wh, nullptr, 1, plain(planes), st);
  const RowShape s = row_shape(g.planL, g.RB);
  return launch_pdl(k_row_r2c<false>, dim3((g.H + g.RB - 1) / g.RB, planes), dim3(kRowThreads), s.smem, st, g, in, out,
                    g.Wh, g.RB, s.ba, s.bufn, FilterWave{}, scale);
}

cudaError_t run_row_c2r(const Geo& g, const float2* in, float* out, int planes, float scale, cudaStream_t st) {
  if (half_rows(g)) return fast::rows_inv(g, in, g.Wh, out, nullptr, 1, plain(planes), scale, st);
  const RowShape s = row_shape(g.planL, g.RB);
  return launch_pdl(k_row_c2r<false>, dim3((g.H + g.RB - 1) / g.RB, planes), dim3(kRowThreads), s.smem, st, g, in, out,
                    g.Wh, g.RB, s.ba, s.bufn, FilterWave{}, scale);
}

cudaError_t run_wave_r2c(const Geo& g, const float* coef, float2* Y, const FilterWave& wv, cudaStream_t st) {
  if (half_rows(g)) return fast::rows_fwd(g, coef, Y, g.Wy, g.ranges, g.eta, fast_wave_of(wv), st);
  const RowShape s = row_shape(g.planL, g.RB);
  return launch_pdl(k_row_r2c<true>, dim3((g.H + g.RB - 1) / g.RB, wv.nc * wv.nf), dim3(kRowThreads), s.smem, st, g,
                    coef, Y, g.Wy, g.RB, s.ba, s.bufn, wv, 1.f);
}

cudaError_t run_wave_c2r(const Geo& g, const float2* Y, float* coef, const FilterWave& wv, float scale,
                         cudaStream_t st) {
  if (half_rows(g)) return fast::rows_inv(g, Y, g.Wy, coef, g.ranges, g.eta, fast_wave_of(wv), scale, st);
  const RowShape s = row_shape(g.planL, g.RB);
  return launch_pdl(k_row_c2r<true>, dim3((g.H + g.RB - 1) / g.RB, wv.nc * wv.nf), dim3(kRowThreads), s.smem, st, g, Y,
                    coef, g.Wy, g.RB, s.ba, s.bufn, wv, scale);
}

cudaError_t run_wave_shrink(const Geo& g, float2* Y, float* bv, const float* thr, const FilterWave& wv, float scale,
                            cudaStream_t st, float* gout) {
  if (fast_shrink_ok(g) && !gout) {  // the register-FFT v-step of this half width
    const fast::Wave f = fast_wave_of(wv);
    const int rpc = fast::row_groups_per_cta(g), groups = (f.nv * g.H + rpc - 1) / rpc;
    return fast::row_shrink(g, std::min(groups, std::max(1, fast_row_ctas(g))), Y, bv, thr, g.Wy, f, scale, nullptr, 0, st);
  }
  if (g.staged) {
    const RowShape s = row_shape(g.planL, g.RB);
    return launch_pdl(k_row_shrink_apart, dim3((g.H + g.RB - 1) / g.RB, wv.nc * wv.nf), dim3(kRowThreads), s.smem, st, g, Y,
                      bv, thr, g.Wy, g.RB, s.ba, s.bufn, wv, scale, gout);
  }
  const RowShape s = row_shape(g.planL, g.RB), r = row_shape(g.planLr, g.RB);
  const int bufn = std::max(s.bufn, r.bufn);
  return launch_pdl(k_row_shrink, dim3((g.H + g.RB - 1) / g.RB, wv.nc * wv.nf), dim3(kRowThreads),
                    2 * sizeof(float2) * static_cast<size_t>(bufn), st, g, Y, bv, thr, g.Wy, g.RB, s.ba, r.ba, bufn, wv,
                    scale, gout);
}

cudaError_t run_wave_l1(const Geo& g, const float2* Y, const float* lam, const FilterWave& wv, float scale,
                        double* partial, cudaStream_t st) {
  const RowShape s = row_shape(g.planL, g.RB);
  return launch_pdl(k_row_l1, dim3((g.H + g.RB - 1) / g.RB, wv.nc * wv.nf), dim3(kRowThreads), s.smem, st, g, Y, lam,
                    g.Wy, g.RB, s.ba, s.bufn, wv, scale, partial);
}

int l1_blocks(const Geo& g, int nch) { return ((g.H + g.RB - 1) / g.RB) * nch * g.eta; }

namespace {
// Rows and labels per batch of a u/w-step CTA: rows for two CTAs per SM, all
// labels as one batch while that takes at most half of the shared memory.
struct UstepShape {
  int rb, kg, pad, bufn;
  size_t smem;
};
UstepShape ustep_shape(const Geo& g, int K) {
  UstepShape u{std::max(1, std::min(ustep_rows(g, K), g.H / (2 * 152))), K, 0, 0, 0};
  for (;; --u.kg) {
    const int B = u.kg * u.rb;
    u.pad = row_pad(g.planL, B, K * u.rb * g.L);
    u.bufn = gf::buf_elems(g.planL, B, u.pad);
    u.smem = sizeof(float2) * (2 * static_cast<size_t>(u.bufn) + static_cast<size_t>(K) * u.rb * g.L);
    if (u.kg == 1 || u.smem <= 113 * 1024) return u;
  }
}
}  // namespace

cudaError_t run_row_ustep(const Geo& g, const float2* T, const float* s, float* w, float* bw, float* u, float2* Ur,
                          float* stv, int K, float gamma, float scale, cudaStream_t st) {
  const UstepShape us = ustep_shape(g, K);
  return launch_pdl(k_row_ustep, dim3((g.H + us.rb - 1) / us.rb), dim3(kRowThreads), us.smem, st, g, T, s, w, bw, u, Ur,
                    stv, K, us.rb, us.kg, fdiv_mul(static_cast<unsigned>(us.rb)),
                    gf::make_batch(g.planL, us.kg * us.rb, us.pad), us.bufn, scale, gamma);
}

}  // namespace shf
