// The row half of a TV iteration in one kernel (Sec. 4, eq. TVreg): inverse row
// transforms of the u-step's spectra, the v-, w- and b-updates, the next
// right-hand side and its forward row transforms, for the half widths of the
// register row transforms (shf_rows.cuh) up to 640.  With the column kernel an
// iteration is then two launches, and d = v - b_v, q = (w - b_w) - gamma s, u and
// w stay on the chip: per pixel and label 28 B of b_v, b_w and s and 16 B of
// spectra move instead of 96 B.
//
// A CTA owns R rows of all K labels.  Row r's update needs u of rows r and r + 1
// and its right-hand side d of rows r - 1 and r, so the CTA inverts R + 2 rows
// and repeats the update of the row above its first one; b_v is read from one
// buffer and written to another for that reason.  Every (row, column pair) is an
// item of its own: the CTA's loads are all in flight at once, where walking down
// the rows with the row above in registers left one row's latency after the
// other (with the staged transforms: 31 us a launch at 512 x 512, K = 4).
//
// Its arithmetic is that of the separate kernels, operation by operation (the row
// transforms are the same functions, and the right-hand side is summed in this
// kernel's order there too): n iterations in one call give the bits of n calls.
#include <algorithm>

#include "shf_fast.h"
#include "shf_rows.cuh"
#include "shf_simplex.cuh"

namespace shf {
namespace tvfast {
namespace {

using fast::even2;
using fast::launch_pdl;
using fast::load_table;
using fast::pack_row;
using fast::pdl_trigger;
using fast::pdl_wait;
using fast::Rows;

__host__ __device__ constexpr bool len_ok(int L) { return fast::half_ok(L) && L <= 640 && L >= 32; }

template <int L, int NT>
struct BandGeo {
  static constexpr int V = Rows<L>::V, T = L / V;
  static constexpr int NG = NT / T;  // row groups
  static constexpr int RAW = Rows<L>::BUF;
  static constexpr int STRIDE = T >= 16 ? RAW : RAW + ((T - RAW % 16) % 16 + 16) % 16;
  static constexpr int TW = even2(L + 1), PT = Rows<L>::PT;
  static constexpr int FIXED = TW + PT + NG * STRIDE;  // float2: tables and exchange buffers
  // + u [K][R + 2][L], d0 of the rows above and the rest of the right-hand side
  // [K][R][L] each, d1 of the pairs' second pixels [K][R][L] floats
  __host__ static size_t smem(int K, int R) {
    return sizeof(float2) * (FIXED + static_cast<size_t>(K) * L * (3 * R + 2)) + sizeof(float) * static_cast<size_t>(K) * L * R;
  }
};

struct BandArgs {
  const float2* Y;  // spectra of u [K][H][pitch]
  float2* Ur;       // spectra of the next right-hand side
  const float *bv_in, *s;
  float *bv_out, *bw;
  int H, pitch, K, R, per_label;
  float t, gamma, scale;
};

template <int L, int KM, int NT, bool FULL>
__global__ void __launch_bounds__(NT, 512 / NT) k_tv_band(const BandArgs a, const float2* __restrict__ twW) {
  using G = BandGeo<L, NT>;
  constexpr int V = G::V, T = G::T;
  extern __shared__ __align__(16) float2 sm[];
  float2* tw = sm;
  float2* pt = tw + G::TW;
  const int H = a.H, K = FULL ? KM : a.K, R = a.R, R2 = R + 2;
  const int lane = threadIdx.x & 31, tt = threadIdx.x & (T - 1), grp = threadIdx.x / T;
  const int partner = (lane - tt) + ((T - tt) & (T - 1));
  float2* fb = pt + G::PT + grp * G::STRIDE;
  float2* U = sm + G::FIXED;                               // [K][R + 2][L]
  float2* D0 = U + static_cast<size_t>(K) * R2 * L;        // [K][R][L]: d0 of slots 0 .. R - 1
  float2* Q = D0 + static_cast<size_t>(K) * R * L;         // [K][R][L]
  float* D1 = reinterpret_cast<float*>(Q + static_cast<size_t>(K) * R * L);  // [K][R][L]
  const int r0 = blockIdx.x * R, nr = min(R, H - r0);
  const size_t HL = static_cast<size_t>(H) * L;
  load_table(tw, twW, L + 1);
  Rows<L>::tables(pt, twW);
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  const auto row_at = [&](int rr) {  // row of u slot rr (periodic)
    const int r = r0 - 1 + rr;
    return r < 0 ? H - 1 : (r >= H ? r - H : r);
  };
  // u on rows r0 - 1 .. r0 + nr: sequence q is slot rr of label k
  for (int q0 = 0; q0 < K * R2; q0 += G::NG) {
    const int q = q0 + grp, k = q / R2, rr = q - k * R2;
    const bool live = k < K && rr <= nr + 1;
    const float2* X = a.Y + (static_cast<size_t>(live ? k : 0) * H + row_at(live ? rr : 0)) * a.pitch;
    float2 v[V];
#pragma unroll
    for (int j = 0; j < V; ++j) v[j] = live ? __ldcg(X + tt + j * T) : make_float2(0.f, 0.f);
    const float2 last = live ? __ldcg(X + L) : make_float2(0.f, 0.f);
    pack_row<L>(v, tt, partner, last, tw);
    Rows<L>::template fft<+1>(v, tt, fb, pt);
    if (live) {
      float2* u = U + static_cast<size_t>(q) * L + tt;
#pragma unroll
      for (int j = 0; j < V; ++j) u[j * T] = c_scale(v[j], a.scale);
    }
  }
  __syncthreads();
  const float2* bv2 = reinterpret_cast<const float2*>(a.bv_in);
  float2* bo2 = reinterpret_cast<float2*>(a.bv_out);
  const float2* s2 = reinterpret_cast<const float2*>(a.s);
  float2* bw2 = reinterpret_cast<float2*>(a.bw);
  for (int e = threadIdx.x; e < (nr + 1) * L; e += NT) {
    const int rr = e / L, p = e - rr * L;  // slot 0 is the row above: only its d0 is used
    const size_t off = static_cast<size_t>(row_at(rr)) * L + p;
    float2 uk[KM], g0[KM], g1[KM];
    float nx = 0.f, ny = 0.f;
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (k < K) {
        const float2* Uk = U + (static_cast<size_t>(k) * R2 + rr) * L;
        const float2 u = Uk[p], down = Uk[L + p];
        const float right = Uk[p + 1 == L ? 0 : p + 1].x;
        const float2 b0 = bv2[2 * k * HL + off], b1 = bv2[(2 * k + 1) * HL + off];
        uk[k] = u;
        g0[k] = make_float2(b0.x + (down.x - u.x), b0.y + (down.y - u.y));
        g1[k] = make_float2(b1.x + (u.y - u.x), b1.y + (right - u.y));
        nx = fmaf(g1[k].x, g1[k].x, fmaf(g0[k].x, g0[k].x, nx));
        ny = fmaf(g1[k].y, g1[k].y, fmaf(g0[k].y, g0[k].y, ny));
      }
    nx = sqrtf(nx);
    ny = sqrtf(ny);
    const float fx = nx > a.t ? a.t / nx : 1.f, fy = ny > a.t ? a.t / ny : 1.f;
    float2 q[KM];
    if (rr > 0) {
      float gx[KM], gy[KM], wx[KM], wy[KM];
#pragma unroll
      for (int k = 0; k < KM; ++k) {
        const float2 b = k < K ? bw2[k * HL + off] : make_float2(0.f, 0.f);
        gx[k] = k < K ? b.x + uk[k].x : 0.f;
        gy[k] = k < K ? b.y + uk[k].y : 0.f;
        wx[k] = gx[k];
        wy[k] = gy[k];
      }
      simplex_project_sorted<KM>(wx, K);
      simplex_project_sorted<KM>(wy, K);
#pragma unroll
      for (int k = 0; k < KM; ++k)
        if (k < K) {
          const float2 bn = make_float2(gx[k] - wx[k], gy[k] - wy[k]), sv = s2[k * HL + off];
          bw2[k * HL + off] = bn;
          q[k] = make_float2(fmaf(-a.gamma, sv.x, wx[k] - bn.x), fmaf(-a.gamma, sv.y, wy[k] - bn.y));
        }
    }
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (k < K) {
        float kx = fx, ky = fy;
        if (a.per_label) {
          const float mx = sqrtf(fmaf(g0[k].x, g0[k].x, g1[k].x * g1[k].x));
          const float my = sqrtf(fmaf(g0[k].y, g0[k].y, g1[k].y * g1[k].y));
          kx = mx > a.t ? a.t / mx : 1.f;
          ky = my > a.t ? a.t / my : 1.f;
        }
        const float2 b0 = make_float2(kx * g0[k].x, ky * g0[k].y), b1 = make_float2(kx * g1[k].x, ky * g1[k].y);
        const float2 d0 = make_float2(g0[k].x - 2.f * b0.x, g0[k].y - 2.f * b0.y);
        const float2 d1 = make_float2(g1[k].x - 2.f * b1.x, g1[k].y - 2.f * b1.y);
        if (rr < R) D0[(static_cast<size_t>(k) * R + rr) * L + p] = d0;
        if (rr > 0) {
          bo2[2 * k * HL + off] = b0;
          bo2[(2 * k + 1) * HL + off] = b1;
          // the right-hand side q + (d0 above - d0) + (d1 left - d1), but for d0
          // above and the left pair's d1
          Q[(static_cast<size_t>(k) * R + rr - 1) * L + p] = make_float2(q[k].x - (d0.x + d1.x), q[k].y + ((d1.x - d1.y) - d0.y));
          D1[(static_cast<size_t>(k) * R + rr - 1) * L + p] = d1.y;
        }
      }
  }
  __syncthreads();
  for (int q0 = 0; q0 < K * R; q0 += G::NG) {
    const int q = q0 + grp, k = q / R, r = q - k * R;
    const bool live = k < K && r < nr;
    const size_t at = static_cast<size_t>(live ? q : 0) * L;
    float2 v[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
      const int i = tt + j * T;
      const float2 b = Q[at + i], up = D0[at + i];
      const float left = D1[at + (i == 0 ? L - 1 : i - 1)];
      v[j] = make_float2(b.x + (up.x + left), b.y + up.y);
    }
    Rows<L>::template fft<-1>(v, tt, fb, pt);
    float2* X = a.Ur + (static_cast<size_t>(live ? k : 0) * H + r0 + (live ? r : 0)) * a.pitch;
#pragma unroll
    for (int j = 0; j < V; ++j) {
      float2 z;
      z.x = __shfl_sync(0xffffffffu, v[V - 1 - j].x, partner);
      z.y = __shfl_sync(0xffffffffu, v[V - 1 - j].y, partner);
      if (live) X[tt + j * T] = Rows<L>::unpack(v, j, tt, z, tw);
    }
    if (live && tt == 0) X[L] = make_float2(v[0].x - v[0].y, 0.f);  // i = L: e^{-i pi} = -1
  }
}

constexpr size_t kMost = 226 * 1024, kHalf = 113 * 1024;  // one CTA per SM, two

// Threads and rows per CTA: two CTAs of 256 threads per SM where two rows fit so
// (the phases of one hide the latencies of the other: 512 x 512, K = 4 20.3 us an
// iteration, 23 with one CTA of 512 and R = 4, 29 with the four kernels), else one
// of 512; enough rows for every SM, at least two (the rows above and below are
// extra work), as many as fit.  R = 0, and the four kernels, where the band does
// not fit, where its last round of CTAs is mostly empty (384 x 640, K = 5, 192
// CTAs: 48 us against 43) and where the image is large enough for the extra work
// to cost what the launches and passes save (in us: 1024 x 1024, K = 4 84 against
// 92, but 2048 x 1024 172 against 169, 720 x 1280 128 both; smaller ones: 128 x
// 128 12 against 25, 256 x 256 17 against 27, 90 x 160 13 against 25).
struct BandShape {
  int threads, R;
};
template <int L>
BandShape shape_t(int H, int K) {
  if constexpr (len_ok(L)) {
    if (2l * L * H * K > (9l << 19)) return BandShape{0, 0};
    const auto filled = [&](int R, int slots) {  // the rounds of CTAs are 70% full
      const int n = (H + R - 1) / R, rounds = (n + slots - 1) / slots;
      return rounds == 1 || 10 * n >= 7 * rounds * slots;
    };
    for (int R = std::min(8, std::max(2, (H + 303) / 304)); R >= 2; --R)
      if (BandGeo<L, 256>::smem(K, R) <= kHalf && filled(R, 304)) return BandShape{256, R};
    for (int R = std::min(8, std::max(2, (H + 151) / 152)); R >= 2; --R)
      if (BandGeo<L, 512>::smem(K, R) <= kMost && filled(R, 152)) return BandShape{512, R};
  }
  return BandShape{0, 0};
}
BandShape band_shape(int L, int H, int K) {
  if (K > 8 || H < 2) return BandShape{0, 0};
  switch (L) {
#define SHF_CASE(N) \
  case N:           \
    return shape_t<N>(H, K);
    SHF_FAST_SIZES(SHF_CASE)
#undef SHF_CASE
    default: return BandShape{0, 0};
  }
}

template <int L, int NT>
cudaError_t prepare_nt() {
  const size_t most = NT == 256 ? kHalf : kMost;
  cudaError_t e = fast::allow_smem(k_tv_band<L, 4, NT, true>, most);
  if (e == cudaSuccess) e = fast::allow_smem(k_tv_band<L, 4, NT, false>, most);
  return e == cudaSuccess ? fast::allow_smem(k_tv_band<L, 8, NT, false>, most) : e;
}
template <int L>
cudaError_t prepare_t() {
  if constexpr (len_ok(L)) {
    cudaError_t e = prepare_nt<L, 256>();
    return e == cudaSuccess ? prepare_nt<L, 512>() : e;
  }
  return cudaSuccess;
}

template <int L, int NT>
cudaError_t band_nt(const BandArgs& a, const float2* twW, cudaStream_t st) {
  const dim3 grid((a.H + a.R - 1) / a.R), block(NT);
  const size_t smem = BandGeo<L, NT>::smem(a.K, a.R);
  if (a.K == 4) return launch_pdl(k_tv_band<L, 4, NT, true>, grid, block, smem, st, a, twW);
  if (a.K < 4) return launch_pdl(k_tv_band<L, 4, NT, false>, grid, block, smem, st, a, twW);
  return launch_pdl(k_tv_band<L, 8, NT, false>, grid, block, smem, st, a, twW);
}
template <int L>
cudaError_t band_t(const BandArgs& a, int threads, const float2* twW, cudaStream_t st) {
  if constexpr (len_ok(L)) return threads == 256 ? band_nt<L, 256>(a, twW, st) : band_nt<L, 512>(a, twW, st);
  return cudaErrorInvalidValue;
}

}  // namespace

bool tv_band_ok(int H, int W, int K) { return band_shape(W / 2, H, K).R > 0; }

cudaError_t tv_band_prepare(int W) {
  switch (W / 2) {
#define SHF_CASE(N) \
  case N:           \
    return prepare_t<N>();
    SHF_FAST_SIZES(SHF_CASE)
#undef SHF_CASE
    default: return cudaSuccess;
  }
}

cudaError_t tv_band(const float2* Y, float2* Ur, int pitch, const float* bv_in, float* bv_out, float* bw, const float* s,
                    int K, int H, int W, float t, float gamma, int per_label, const float2* twW, cudaStream_t st) {
  const BandShape sh = band_shape(W / 2, H, K);
  const BandArgs a{Y, Ur, bv_in, s, bv_out, bw, H, pitch, K, sh.R, per_label, t, gamma, 1.f / (static_cast<float>(H) * W)};
  if (a.R < 2) return cudaErrorInvalidValue;
  switch (W / 2) {
#define SHF_CASE(N) \
  case N:           \
    return band_t<N>(a, sh.threads, twW, st);
    SHF_FAST_SIZES(SHF_CASE)
#undef SHF_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace tvfast
}  // namespace shf
