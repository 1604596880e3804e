// Transforms of small images, whole planes in shared memory (any height and half
// width 2^a 3^b 5^c whose plane fits twice): one CTA per (channel, filter) runs a
// plane's row and column transforms back to back on the staged FFTs of
// shf_gfft.cuh, so that an analysis is one launch without temporaries and a
// synthesis two.
//
// At these sizes a transform is a chain of launches, each a few microseconds of
// latency for a fraction of a microsecond of work, behind a stream-ordered
// allocation.  The transforms of a whole column range and of all rows run as one
// batch from shared memory to shared memory through one function per direction
// and orientation (a few KB of code that the kernels share: instruction fetch
// would otherwise cost as much as the arithmetic), with element-wise passes
// between them.  One 64 x 64 channel, 13 filters: analysis 31 -> 22 us in a row
// (17 where the caller has the stream's handle at hand) and 270 -> 85 us for the
// first on a bank (four launches on the staged or register-FFT kernels: 33 us).
// The ADMM iteration was tried the same way (a
// cluster of one CTA per label for the u/w-step, a CTA per label and filter for
// the rest) and is slower than its six or seven short launches: 41 against 25 us
// at 64 x 64, K = 3, 62 against 56 at 50 x 216, K = 5; a CTA needs about 20 us for
// its eight batch stages, latency-bound (issue slots 12% busy).
#include <cooperative_groups.h>

#include <algorithm>

#include "shf_fast.h"
#include "shf_gfft.cuh"
#include "shf_internal.h"

namespace cg = cooperative_groups;

namespace shf {

namespace {

using fast::pdl_trigger;
using fast::pdl_wait;

constexpr int kFilterCluster = 8;
constexpr size_t kSmallMost = 220 * 1024;  // dynamic shared memory of a CTA

// The plans of a launch in shared memory and its two plane buffers.
struct Plane2 {
  FftPlan planH, planL;
};
struct Bufs {
  float2 *a, *b;  // a holds the data, b is free
  __device__ __forceinline__ void swap() {
    float2* t = a;
    a = b;
    b = t;
  }
};

// One stage of a batch in shared memory (the general stage of shf_gfft.cuh with
// its place in the plan at run time).
template <int S, bool COLS>
struct PlaneStage {
  const FftStage& g;
  const gf::Batch& a;
  int s;
  bool last;
  const float2* in;
  float2* out;
  const float2* pt;
  template <int R>
  __device__ __forceinline__ void run() {
    const int total = g.nb * a.B;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
      int j, b, k = 0;
      gf::item_of<COLS>(g, a, idx, j, b);
      float2 v[R];
      if (s == 0) {
        const float2* p = COLS ? in + j * a.B + b : in + b * g.nb * R + j;  // natural order, rows of L
        const int d = COLS ? g.nb * a.B : g.nb;
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = p[t * d];
      } else {
        gf::stage_in<R, S, COLS>(g, a, s == 1, j, b, in, pt, v, k);
      }
      gf::dft<R, S>(v);
      if (last) {
        float2* p = COLS ? out + j * a.B + b : out + b * g.nb * R + j;
        const int d = COLS ? g.nb * a.B : g.nb;
#pragma unroll
        for (int q = 0; q < R; ++q) p[q * d] = v[q];
      } else {
        gf::stage_out<R, COLS>(g, a, s == 0, j, b, k, out, v);
      }
    }
  }
};

// The transform of a batch of B sequences in p.a (natural order: columns
// i B + b, rows b L + i), in place of p.a / p.b; starts and ends with a barrier.
template <int S, bool COLS>
__device__ __noinline__ Bufs plane_fft(const FftPlan& plan, int B, int pad, Bufs p, const float2* pt) {
  const gf::Batch a{B, fdiv_mul(static_cast<unsigned>(B)), plan.L + (pad ? plan.L / plan.st[0].R : 0), pad};
  __syncthreads();
  for (int s = 0; s < plan.nst; ++s) {
    PlaneStage<S, COLS> f{plan.st[s], a, s, s + 1 == plan.nst, p.a, p.b, pt};
    gf::with_radix(plan.st[s].R, f);
    __syncthreads();
    p.swap();
  }
  return p;
}

// Columns [c0, c0 + n) of filter f's support (n = 0: none).
struct Cols {
  int c0, n;
};
__device__ __forceinline__ Cols cols_of(const Geo& g, int f) {
  Cols c{0, 0};
  if (f < g.eta) {
    const int2 r = g.ranges[f];
    c.c0 = r.x;
    c.n = max(0, min(r.y, g.L) - r.x + 1);
  }
  return c;
}

// Element k of the inverse packing of a row of X, of which columns [c0, c0 + n)
// are stored.
__device__ __forceinline__ float2 packed_cols(const float2* X, int L, int k, int c0, int n, const float2* __restrict__ twW) {
  const int i = k - c0, m = L - k - c0;
  const float2 a = (i >= 0 && i < n) ? X[i] : make_float2(0.f, 0.f);
  const float2 b = (m >= 0 && m < n) ? c_conj(X[m]) : make_float2(0.f, 0.f);
  return pack_combine(c_add(a, b), c_sub(a, b), twW[k]);
}

// Calls f(row, position, element) over rows of n elements.
template <class F>
__device__ __forceinline__ void each(int rows, int n, F&& f) {
  const unsigned m = fdiv_mul(static_cast<unsigned>(n));
  for (int e = threadIdx.x; e < rows * n; e += blockDim.x) {
    const int r = static_cast<int>(fdiv(static_cast<unsigned>(e), m));
    f(r, e - r * n, e);
  }
}

// The launch's context: plans in shared memory, pads of the row plan.
struct Ctx {
  const Geo& g;
  const Plane2& pl;
  int padL;
  Bufs p;
  template <int S>
  __device__ __forceinline__ void cols(int n) {
    p = plane_fft<S, true>(pl.planH, n, 0, p, g.ptH);
  }
  template <int S>
  __device__ __forceinline__ void rows() {
    p = plane_fft<S, false>(pl.planL, g.H, padL, p, g.ptL);
  }
  // spectrum rows (columns [c0, c0 + n) at pitch n) -> packed rows of L
  __device__ __forceinline__ void pack(int c0, int n) {
    const float2* X = p.a;
    float2* o = p.b;
    each(g.H, g.L, [&](int r, int i, int e) { o[e] = packed_cols(X + r * n, g.L, i, c0, n, g.twW); });
    p.swap();
  }
  // complex rows of L -> columns [c0, c0 + n) of their half spectra at pitch n
  __device__ __forceinline__ void unpack(int c0, int n) {
    const float2* Z = p.a;
    float2* o = p.b;
    each(g.H, n, [&](int r, int b, int e) { o[e] = r2c_unpack(Z + r * g.L, g.L, c0 + b, g.twW); });
    p.swap();
  }
};

// Prologue of a kernel: the plans into shared memory (before the wait).
__device__ __forceinline__ void load_plans(const Geo& g, Plane2& s) {
  const int n = sizeof(FftPlan) / 4;
  for (int e = threadIdx.x; e < 2 * n; e += blockDim.x)
    reinterpret_cast<int*>(&s)[e] = e < n ? reinterpret_cast<const int*>(&g.planH)[e] : reinterpret_cast<const int*>(&g.planL)[e - n];
  __syncthreads();
}

// The cluster's sum of R (its CTAs' filtered spectra, columns span[0] ..
// span[0] + span[1] - 1 at pitch span[1], the same buffer in each CTA), in
// filter order, into dst [H][Wh]: each CTA adds its share of the elements.
__device__ __forceinline__ void cluster_sum(const Geo& g, float2* R, const int* span, float2* __restrict__ dst) {
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();  // every CTA's R and span are written
  const int q0 = cl.block_rank(), nq = cl.num_blocks(), E = g.H * g.Wh;
  const unsigned m = fdiv_mul(static_cast<unsigned>(g.Wh));
  const int e0 = static_cast<int>(static_cast<long long>(E) * q0 / nq), e1 = static_cast<int>(static_cast<long long>(E) * (q0 + 1) / nq);
  int c0[kFilterCluster], n[kFilterCluster];
  const float2* src[kFilterCluster];
#pragma unroll
  for (int q = 0; q < kFilterCluster; ++q) {
    const int r = q < nq ? q : 0;
    const int* s = cl.map_shared_rank(span, r);
    c0[q] = s[0];
    n[q] = q < nq ? s[1] : 0;
    src[q] = cl.map_shared_rank(R, r);
  }
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int r = static_cast<int>(fdiv(static_cast<unsigned>(e), m)), col = e - r * g.Wh;
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kFilterCluster; ++q) {
      const int b = col - c0[q];
      if (b >= 0 && b < n[q]) s = c_add(s, src[q][r * n[q] + b]);
    }
    dst[e] = s;
  }
  cl.sync();  // nobody leaves while its R is read
}

// p.a (columns [c0, c0 + n)) times W_f, in place; each thread its own elements.
__device__ __forceinline__ void filter_cols(const Ctx& x, const Cols& c, int f) {
  const float* wf = x.g.bank + static_cast<size_t>(f) * x.g.H * x.g.Wh + c.c0;
  float2* R = x.p.a;
  each(x.g.H, c.n, [&](int i, int b, int e) { R[e] = c_scale(R[e], __ldg(wf + static_cast<size_t>(i) * x.g.Wh + b)); });
}

#define SHF_SMALL_PROLOGUE                  \
  extern __shared__ float2 sm[];            \
  __shared__ Plane2 plans;                  \
  Ctx x{g, plans, padL, Bufs{sm, sm + bufn}}; \
  load_plans(g, plans);

// The sum of np partial spectra [np][nch][H][Wh] of channel k into p.a.
__device__ __forceinline__ void sum_partials(const Ctx& x, const float2* __restrict__ partial, int np, int nch, int k) {
  const size_t E = static_cast<size_t>(x.g.H) * x.g.Wh;
  const float2* p0 = partial + k * E;
  for (int e = threadIdx.x; e < static_cast<int>(E); e += blockDim.x) {
    float2 a = p0[e];
    for (int q = 1; q < np; ++q) a = c_add(a, p0[static_cast<size_t>(q) * nch * E + e]);
    x.p.a[e] = a;
  }
}

// 2-D inverse of the sum of np partial spectra [np][nch][H][Wh], times scale:
// out [nch][H][W].
__global__ void __launch_bounds__(512, 1)
    k_small_sum(const __grid_constant__ Geo g, const float2* __restrict__ partial, int np, float* __restrict__ out, int padL, int bufn, float scale) {
  SHF_SMALL_PROLOGUE
  const int k = blockIdx.x, HL = g.H * g.L;
  pdl_wait();
  pdl_trigger();
  sum_partials(x, partial, np, gridDim.x, k);
  x.cols<+1>(g.Wh);
  x.pack(0, g.Wh);
  x.rows<+1>();
  float2* o = reinterpret_cast<float2*>(out) + static_cast<size_t>(k) * HL;
  for (int e = threadIdx.x; e < HL; e += blockDim.x) o[e] = c_scale(x.p.a[e], scale);
}

// Coefficients of filter blockIdx.x of channel blockIdx.y: every CTA forms the
// filter's columns of the channel's spectrum itself.
__global__ void __launch_bounds__(512, 1)
    k_small_analyze(const __grid_constant__ Geo g, const float* __restrict__ u, float* __restrict__ coef, int padL, int bufn,
                    float scale) {
  SHF_SMALL_PROLOGUE
  const int f = blockIdx.x, HL = g.H * g.L;
  const Cols c = cols_of(g, f);
  pdl_wait();
  pdl_trigger();
  float2* o = reinterpret_cast<float2*>(coef) + (static_cast<size_t>(blockIdx.y) * g.eta + f) * HL;
  if (c.n == 0) {
    for (int e = threadIdx.x; e < HL; e += blockDim.x) o[e] = make_float2(0.f, 0.f);
    return;
  }
  const float2* src = reinterpret_cast<const float2*>(u) + static_cast<size_t>(blockIdx.y) * HL;
  for (int e = threadIdx.x; e < HL; e += blockDim.x) x.p.a[e] = src[e];
  x.rows<-1>();
  x.unpack(c.c0, c.n);
  x.cols<-1>(c.n);
  filter_cols(x, c, f);
  x.cols<+1>(c.n);
  x.pack(c.c0, c.n);
  x.rows<+1>();
  for (int e = threadIdx.x; e < HL; e += blockDim.x) o[e] = c_scale(x.p.a[e], scale);
}

// Filtered spectrum of coefficient plane blockIdx.x of channel blockIdx.y, added
// over the cluster's filters: partial [clusters][nch][H][Wh].
__global__ void __launch_bounds__(512, 1)
    k_small_gather(const __grid_constant__ Geo g, const float* __restrict__ coef, float2* __restrict__ partial, int padL,
                   int bufn) {
  SHF_SMALL_PROLOGUE
  __shared__ int span[2];
  const int f = blockIdx.x, HL = g.H * g.L;
  const Cols c = cols_of(g, f);
  if (threadIdx.x == 0) {
    span[0] = c.c0;
    span[1] = c.n;
  }
  pdl_wait();
  pdl_trigger();
  if (c.n > 0) {
    const float2* src = reinterpret_cast<const float2*>(coef) + (static_cast<size_t>(blockIdx.y) * g.eta + f) * HL;
    for (int e = threadIdx.x; e < HL; e += blockDim.x) x.p.a[e] = src[e];
    x.rows<-1>();
    x.unpack(c.c0, c.n);
    x.cols<-1>(c.n);
    filter_cols(x, c, f);
  } else if ((g.planL.nst + g.planH.nst + 1) & 1) {
    x.p.swap();  // the buffer that the others' sums are in
  }
  cluster_sum(g, x.p.a, span, partial + (static_cast<size_t>(blockIdx.x / kFilterCluster) * gridDim.y + blockIdx.y) * g.H * g.Wh);
}

// Launch shape: the row plan's padding and the buffers of a plane.
struct Shape {
  int padL, bufn, threads;
  size_t smem;
};
Shape shape_of(const Geo& g) {
  const int pad = g.planL.nst > 1 && g.planL.st[0].R % 2 == 0 ? 1 : 0;
  const int n = std::max(gf::buf_elems(g.planL, g.H, pad), g.H * g.Wh);
  return Shape{pad, n, g.H * g.Wh > 3072 ? 512 : 256, 2 * sizeof(float2) * static_cast<size_t>(n)};
}

template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*kernel)(KArgs...), dim3 grid, int cluster, const Shape& s, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(s.threads);
  cfg.dynamicSmemBytes = s.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (pdl_enabled()) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

int clusters(const Geo& g) { return (g.eta + kFilterCluster - 1) / kFilterCluster; }

}  // namespace

// The whole plane twice in a CTA's shared memory.
bool small_ok(const Geo& g) { return g.ranges && shape_of(g).smem <= kSmallMost; }

size_t small_partials(const Geo& g, int nch) { return static_cast<size_t>(clusters(g)) * nch * g.H * g.Wh; }

cudaError_t prepare_small(const Geo& g) {
  if (!small_ok(g)) return cudaSuccess;
  // one limit for every size: banks of several sizes (and threads) share the kernels
  const auto set = [](const void* k) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmallMost));
  };
  for (const void* k : {reinterpret_cast<const void*>(k_small_sum), reinterpret_cast<const void*>(k_small_analyze), reinterpret_cast<const void*>(k_small_gather)}) {
    cudaError_t e = set(k);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t run_small_analyze(const Geo& g, const float* u, float* coef, int nch, float scale, cudaStream_t st) {
  const Shape sh = shape_of(g);
  return launch_cluster(k_small_analyze, dim3(g.eta, nch), 1, sh, st, g, u, coef, sh.padL, sh.bufn, scale);
}

cudaError_t run_small_synthesize(const Geo& g, const float* coef, float* u, float2* partial, int nch, float scale,
                                 cudaStream_t st) {
  const Shape sh = shape_of(g);
  cudaError_t e = launch_cluster(k_small_gather, dim3(clusters(g) * kFilterCluster, nch), kFilterCluster, sh, st, g, coef,
                                 partial, sh.padL, sh.bufn);
  if (e != cudaSuccess) return e;
  return launch_cluster(k_small_sum, dim3(nch), 1, sh, st, g, partial, clusters(g), u, sh.padL,
                        sh.bufn, scale);
}

}  // namespace shf
