// Column kernels of the general lengths (heights H = 2^a 3^b 5^c): the fan-out
// over the filters, the synthesis gather and the passes of single planes, on
// the staged FFTs of shf_gfft.cuh.  One CTA owns a tile of TC consecutive
// half-spectrum columns over all H rows, consecutive threads on consecutive
// columns.  Filter tiles outside a filter's column range are skipped (the
// spectra of a range hold about half of the columns at four scales), and
// columns of a tile outside the range count as zero without being read.
// Bound by latency (ncu at 480 rows, 8 columns: issue slots 35% busy, stalls on
// global loads and barriers, 16 warps per SM by registers).
#include <algorithm>

#include "shf_fast.h"
#include "shf_gfft.cuh"
#include "shf_internal.h"

namespace shf {

namespace {

using fast::launch_pdl;
using fast::pdl_trigger;
using fast::pdl_wait;

// Column range of filter f.
__device__ __forceinline__ int2 range_of(const Geo& g, int f) {
  return g.ranges ? g.ranges[f] : make_int2(0, g.L);
}

// Column-forward of row spectra, in place: U [nch][H][Wh].
__global__ void __launch_bounds__(kColThreads, 2)
    k_gcol_fwd(const __grid_constant__ Geo g, float2* U, const __grid_constant__ gf::Batch ba, int bufn) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int col0 = blockIdx.x * g.TC, Wh = g.Wh;
  pdl_wait();
  pdl_trigger();
  float2* P = U + static_cast<size_t>(blockIdx.y) * g.H * Wh + col0;
  const int n = min(g.TC, Wh - col0);
  const auto ld = [&](int i, int b) { return b < n ? P[static_cast<size_t>(i) * Wh + b] : make_float2(0.f, 0.f); };
  const auto st = [&](int i, int b, float2 v) {
    if (b < n) P[static_cast<size_t>(i) * Wh + b] = v;
  };
  // every load of the tile is in the first stage; a single-stage butterfly
  // reads and writes its own column only
  gf::fft<-1, true>(g.planH, ba, x, g.ptH, ld, st);
}

// Column-forward, times the one filter g.bank, column-inverse: in [nch][H][Wh]
// -> out [nch][H][Wh].
__global__ void __launch_bounds__(kColThreads, 2)
    k_gcol_filter(const __grid_constant__ Geo g, const float2* __restrict__ in, float2* __restrict__ out,
                  const __grid_constant__ gf::Batch ba, int bufn) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int col0 = blockIdx.x * g.TC, Wh = g.Wh, n = min(g.TC, Wh - col0);
  pdl_wait();
  pdl_trigger();
  const size_t off = static_cast<size_t>(blockIdx.y) * g.H * Wh + col0;
  const float2* src = in + off;
  float2* dst = out + off;
  const float* wf = g.bank + col0;
  const auto ld = [&](int i, int b) { return b < n ? src[static_cast<size_t>(i) * Wh + b] : make_float2(0.f, 0.f); };
  const float2* y = gf::fft_head<-1, true>(g.planH, ba, x, g.ptH, ld);
  float2* Z = x.next();
  const auto mul = [&](int i, int b, float2 v) {
    Z[i * ba.B + b] = c_scale(v, b < n ? __ldg(wf + static_cast<size_t>(i) * Wh + b) : 0.f);
  };
  gf::NoLd nl;
  if (g.planH.nst == 1)
    gf::run_stage<-1, true, gf::kOnly>(g.planH, 0, ba, nullptr, nullptr, g.ptH, ld, mul, threadIdx.x, blockDim.x);
  else
    gf::run_stage<-1, true, gf::kLast>(g.planH, g.planH.nst - 1, ba, y, nullptr, g.ptH, nl, mul, threadIdx.x, blockDim.x);
  __syncthreads();
  gf::fft<+1, true>(
      g.planH, ba, x, g.ptH, [&](int i, int b) { return Z[i * ba.B + b]; },
      [&](int i, int b, float2 v) {
        if (b < n) dst[static_cast<size_t>(i) * Wh + b] = v;
      });
}

// Analysis fan-out of a wave: Y plane (c - c0) nf + (f - f0) = column-inverse of
// W_f times uhat [nch][H][Wh], fg filters per CTA (uhat's tile then comes from
// L1 after the first).
__global__ void __launch_bounds__(kColThreads, 2)
    k_gcol_fan(const __grid_constant__ Geo g, const float2* __restrict__ uhat, float2* __restrict__ Y, int fg, int mask,
               const FilterWave wv, const __grid_constant__ gf::Batch ba, int bufn) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int col0 = blockIdx.x * g.TC, Wh = g.Wh, Wy = g.Wy, H = g.H;
  const int fb = wv.f0 + blockIdx.z * fg, fe = min(wv.f0 + wv.nf, fb + fg);
  pdl_wait();
  pdl_trigger();
  const float2* src = uhat + static_cast<size_t>(wv.c0 + blockIdx.y) * H * Wh + col0;
  for (int f = fb; f < fe; ++f) {
    // columns b0..b1 of the tile are in the range; s0..s1 are stored: the range
    // widened to whole tiles of mask + 1 columns (0: not widened)
    const int2 r = range_of(g, f);
    if (r.x > r.y) continue;
    const int b0 = max(r.x - col0, 0), b1 = min(min(r.y, g.L) - col0, g.TC - 1);
    const int s0 = max((r.x & ~mask) - col0, 0), s1 = min(min(r.y | mask, g.L) - col0, g.TC - 1);
    if (s0 > s1) continue;
    const float* wf = g.bank + static_cast<size_t>(f) * H * Wh + col0;
    float2* dst = Y + static_cast<size_t>(blockIdx.y * wv.nf + (f - wv.f0)) * H * Wy + col0;
    gf::fft<+1, true>(
        g.planH, ba, x, g.ptH,
        [&](int i, int b) {
          if (b < b0 || b > b1) return make_float2(0.f, 0.f);
          const size_t e = static_cast<size_t>(i) * Wh + b;
          return c_scale(src[e], __ldg(wf + e));
        },
        [&](int i, int b, float2 v) {
          if (b >= s0 && b <= s1) dst[static_cast<size_t>(i) * Wy + b] = v;
        });
  }
}

// The gather's last stage: adds W_f times the butterflies' results to the
// accumulators (butterfly m of the thread: acc[m R ..]); its final store.
template <int MAXV>
struct GatherLast {
  const Geo& g;
  const gf::Batch& ba;
  const float2 *in, *src;  // the exchange buffer; the tile itself (single-stage plans)
  const float* wf;
  int b0, b1;
  float2 (&acc)[MAXV];
  template <int R>
  __device__ __forceinline__ void run() {
    const FftStage& s = g.planH.st[g.planH.nst - 1];
    const int total = s.nb * ba.B;
#pragma unroll
    for (int m = 0; m < MAXV / R; ++m) {
      const int idx = threadIdx.x + m * kColThreads;
      if (idx < total) {
        int j, b, k;
        gf::item_of<true>(s, ba, idx, j, b);
        if (b < b0 || b > b1) continue;
        float2 v[R];
        float w[R];
#pragma unroll
        for (int q = 0; q < R; ++q) w[q] = __ldg(wf + static_cast<size_t>(j + q * s.nb) * g.Wh + b);
        if (g.planH.nst == 1) {
#pragma unroll
          for (int q = 0; q < R; ++q) v[q] = src[static_cast<size_t>(j + q * s.nb) * g.Wy + b];
        } else {
          gf::stage_in<R, -1, true>(s, ba, g.planH.nst == 2, j, b, in, g.ptH, v, k);
        }
        gf::dft<R, -1>(v);
#pragma unroll
        for (int q = 0; q < R; ++q) acc[m * R + q] = c_fma2(make_float2(w[q], w[q]), v[q], acc[m * R + q]);
      }
    }
  }
};
template <int MAXV>
struct GatherStore {
  const Geo& g;
  const gf::Batch& ba;
  float2* dst;  // the tile's partial sums, row pitch Wh
  int n;
  float2 (&acc)[MAXV];
  template <int R>
  __device__ __forceinline__ void run() {
    const FftStage& s = g.planH.st[g.planH.nst - 1];
    const int total = s.nb * ba.B;
#pragma unroll
    for (int m = 0; m < MAXV / R; ++m) {
      const int idx = threadIdx.x + m * kColThreads;
      if (idx < total) {
        int j, b;
        gf::item_of<true>(s, ba, idx, j, b);
#pragma unroll
        for (int q = 0; q < R; ++q)
          if (b < n) dst[static_cast<size_t>(j + q * s.nb) * g.Wh + b] = acc[m * R + q];
      }
    }
  }
};

// Synthesis gather of a wave's filter groups: partial[grp][ch] = sum over the
// group's filters, in order, of W_f * column-forward(Y).
template <int MAXV>
__global__ void __launch_bounds__(kColThreads, MAXV <= 24 ? 2 : 1)
    k_gcol_gather(const __grid_constant__ Geo g, const float2* __restrict__ Y, float2* __restrict__ partial, int nch,
                  int fg, int g0, const FilterWave wv, const __grid_constant__ gf::Batch ba, int bufn) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int col0 = blockIdx.x * g.TC, Wh = g.Wh, Wy = g.Wy, H = g.H, grp = g0 + blockIdx.z;
  const int fb = grp * fg, fe = min(wv.f0 + wv.nf, fb + fg);
  pdl_wait();
  pdl_trigger();
  float2 acc[MAXV];
#pragma unroll
  for (int m = 0; m < MAXV; ++m) acc[m] = make_float2(0.f, 0.f);
  const int R = g.planH.st[g.planH.nst - 1].R;
  for (int f = fb; f < fe; ++f) {
    const int2 r = range_of(g, f);
    const int b0 = max(r.x - col0, 0), b1 = min(min(r.y, g.L) - col0, g.TC - 1);
    if (b0 > b1) continue;
    const float2* src = Y + static_cast<size_t>(blockIdx.y * wv.nf + (f - wv.f0)) * H * Wy + col0;
    const float2* y = gf::fft_head<-1, true>(g.planH, ba, x, g.ptH, [&](int i, int b) {
      return b >= b0 && b <= b1 ? src[static_cast<size_t>(i) * Wy + b] : make_float2(0.f, 0.f);
    });
    GatherLast<MAXV> last{g, ba, y, src, g.bank + static_cast<size_t>(f) * H * Wh + col0, b0, b1, acc};
    gf::with_radix(R, last);
  }
  GatherStore<MAXV> store{g, ba, partial + (static_cast<size_t>(grp) * nch + wv.c0 + blockIdx.y) * H * Wh + col0,
                          min(g.TC, Wh - col0), acc};
  gf::with_radix(R, store);
}

// out[nch] = column-inverse of the sum of the groups' partial sums, in order.
__global__ void __launch_bounds__(kColThreads, 2)
    k_gcol_reduce_inv(const __grid_constant__ Geo g, const float2* __restrict__ partial, float2* __restrict__ out,
                      int nch, int groups, const __grid_constant__ gf::Batch ba, int bufn) {
  extern __shared__ float2 sm[];
  gf::Exchange x{{sm, sm + bufn}};
  const int col0 = blockIdx.x * g.TC, Wh = g.Wh, n = min(g.TC, Wh - col0);
  pdl_wait();
  pdl_trigger();
  const size_t off = static_cast<size_t>(blockIdx.y) * g.H * Wh + col0, step = static_cast<size_t>(nch) * g.H * Wh;
  const float2* src = partial + off;
  float2* dst = out + off;
  gf::fft<+1, true>(
      g.planH, ba, x, g.ptH,
      [&](int i, int b) {
        float2 s = make_float2(0.f, 0.f);
        if (b < n) {
          const float2* p = src + static_cast<size_t>(i) * Wh + b;
          for (int k = 0; k < groups; ++k) s = c_add(s, p[k * step]);
        }
        return s;
      },
      [&](int i, int b, float2 v) {
        if (b < n) dst[static_cast<size_t>(i) * Wh + b] = v;
      });
}

template <typename K>
cudaError_t set_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

struct ColShape {
  gf::Batch ba;
  int bufn;
  size_t smem;
};
// The padded first exchange where it pays (fewer than 16 columns: rows of two
// or more butterflies share a half-warp) and fits.
ColShape col_shape(const Geo& g) {
  const FftPlan& p = g.planH;
  int pad = p.nst > 1 && p.st[0].R % 2 == 0 && g.TC < 16 ? 1 : 0;
  if (2 * sizeof(float2) * static_cast<size_t>(gf::buf_elems(p, g.TC, pad)) > 227 * 1024) pad = 0;
  const int n = gf::buf_elems(p, g.TC, pad);
  return ColShape{gf::make_batch(p, g.TC, pad), n, sizeof(float2) * 2 * static_cast<size_t>(n)};
}

template <int MAXV>
cudaError_t gather_t(const Geo& g, const float2* Y, float2* partial, int nch, int fg, int g0, int ng,
                     const FilterWave& wv, const ColShape& s, cudaStream_t st) {
  return launch_pdl(k_gcol_gather<MAXV>, dim3(g.ntiles, wv.nc, ng), dim3(kColThreads), s.smem, st, g, Y, partial, nch,
                    fg, g0, wv, s.ba, s.bufn);
}

// Y bytes of a wave (full-width planes): the filters' ranges hold about half of
// them, so that a wave's spectra stay near the 129 MB L2 between its launches
// (DRAM reads 24 MB and 95 MB in the fan and the gather of a 154 MB wave).
constexpr size_t kWaveBytes = size_t(192) << 20;

}  // namespace

cudaError_t prepare_col_general(int optin) {
  const cudaError_t errs[] = {set_smem(k_gcol_fwd, optin),        set_smem(k_gcol_filter, optin),
                              set_smem(k_gcol_fan, optin),        set_smem(k_gcol_gather<16>, optin),
                              set_smem(k_gcol_gather<24>, optin), set_smem(k_gcol_gather<32>, optin),
                              set_smem(k_gcol_gather<48>, optin), set_smem(k_gcol_reduce_inv, optin)};
  for (cudaError_t x : errs)
    if (x != cudaSuccess) return x;
  return cudaSuccess;
}

namespace {
size_t plane_bytes(const Geo& g) { return sizeof(float2) * static_cast<size_t>(g.H) * g.Wy; }
int wave_channels(const Geo& g, int nch) {
  const size_t per = plane_bytes(g) * static_cast<size_t>(g.eta);
  return static_cast<int>(std::max<size_t>(1, std::min<size_t>(nch, kWaveBytes / per)));
}
}  // namespace

int default_groups(const Geo& g, int nch) {
  // enough CTAs for the SMs in one wave's gather, and groups small enough that
  // one channel's filters can be split into waves
  const int base = g.ntiles * wave_channels(g, nch);
  int G = (4 * 152 + base - 1) / base;
  const size_t per = plane_bytes(g) * static_cast<size_t>(g.eta);
  G = std::max(G, static_cast<int>((per + kWaveBytes - 1) / kWaveBytes));
  if (G < 1) G = 1;
  if (G > g.eta) G = g.eta;
  const int fg = (g.eta + G - 1) / G;
  return (g.eta + fg - 1) / fg;
}

std::vector<FilterWave> general_waves(const Geo& g, int nch, int groups) {
  std::vector<FilterWave> out;
  const int fg = (g.eta + groups - 1) / groups;
  const int nc = wave_channels(g, nch);
  const size_t per = plane_bytes(g) * static_cast<size_t>(g.eta);
  if (per <= kWaveBytes) {  // whole channels, balanced over the waves
    const int nw = (nch + nc - 1) / nc, b = (nch + nw - 1) / nw;
    for (int c = 0; c < nch; c += b) out.push_back(FilterWave{c, std::min(b, nch - c), 0, g.eta});
  } else {  // runs of whole filter groups of one channel
    const int most = std::max<int>(1, static_cast<int>(kWaveBytes / (plane_bytes(g) * static_cast<size_t>(fg))));
    const int nw = (groups + most - 1) / most, ng = (groups + nw - 1) / nw;
    for (int c = 0; c < nch; ++c)
      for (int k = 0; k < groups; k += ng) {
        const int f0 = k * fg, f1 = std::min(g.eta, (k + ng) * fg);
        if (f1 > f0) out.push_back(FilterWave{c, 1, f0, f1 - f0});
      }
  }
  return out;
}

size_t wave_planes(const std::vector<FilterWave>& waves) {
  size_t n = 1;
  for (const FilterWave& w : waves) n = std::max(n, static_cast<size_t>(w.nc) * w.nf);
  return n;
}

cudaError_t run_col_fwd(const Geo& g, float2* U, int nch, cudaStream_t st) {
  const ColShape s = col_shape(g);
  return launch_pdl(k_gcol_fwd, dim3(g.ntiles, nch), dim3(kColThreads), s.smem, st, g, U, s.ba, s.bufn);
}

cudaError_t run_col_filter(const Geo& g, const float2* in, float2* out, int nch, cudaStream_t st) {
  const ColShape s = col_shape(g);
  return launch_pdl(k_gcol_filter, dim3(g.ntiles, nch), dim3(kColThreads), s.smem, st, g, in, out, s.ba, s.bufn);
}

cudaError_t run_wave_fan(const Geo& g, const float2* uhat, float2* Y, const FilterWave& wv, cudaStream_t st) {
  const ColShape s = col_shape(g);
  // up to 4 filters per CTA (one load of uhat's tile from L2 for all of them)
  // while that leaves eight CTAs per SM
  const long all = static_cast<long>(g.ntiles) * wv.nc * wv.nf;
  const int fg = static_cast<int>(std::max<long>(1, std::min<long>(4, all / (8 * 152))));
  return launch_pdl(k_gcol_fan, dim3(g.ntiles, wv.nc, (wv.nf + fg - 1) / fg), dim3(kColThreads), s.smem, st, g, uhat, Y,
                    fg, fast_shrink_ok(g) ? reg::col_batch(g.H) - 1 : 0, wv, s.ba, s.bufn);
}

cudaError_t run_wave_gather(const Geo& g, const float2* Y, float2* partial, int nch, int groups, const FilterWave& wv,
                            cudaStream_t st) {
  const ColShape s = col_shape(g);
  const int fg = (g.eta + groups - 1) / groups;
  const int g0 = wv.f0 / fg, ng = (wv.nf + fg - 1) / fg;
  const FftStage& l = g.planH.st[g.planH.nst - 1];
  const int need = (l.nb * g.TC + kColThreads - 1) / kColThreads * l.R;
  if (need <= 16) return gather_t<16>(g, Y, partial, nch, fg, g0, ng, wv, s, st);
  if (need <= 24) return gather_t<24>(g, Y, partial, nch, fg, g0, ng, wv, s, st);
  if (need <= 32) return gather_t<32>(g, Y, partial, nch, fg, g0, ng, wv, s, st);
  if (need <= 48) return gather_t<48>(g, Y, partial, nch, fg, g0, ng, wv, s, st);
  return cudaErrorInvalidValue;
}

cudaError_t run_col_reduce_inv(const Geo& g, const float2* partial, float2* out, int nch, int groups,
                               cudaStream_t st) {
  const ColShape s = col_shape(g);
  return launch_pdl(k_gcol_reduce_inv, dim3(g.ntiles, nch), dim3(kColThreads), s.smem, st, g, partial, out, nch, groups,
                    s.ba, s.bufn);
}

}  // namespace shf
