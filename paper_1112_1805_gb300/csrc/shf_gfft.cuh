// FFTs of the general lengths 2^a 3^b 5^c (up to 2048) for sm_103a: Stockham
// stages of radices 2 to 16 chosen at run time (FftPlan), a batch of sequences
// per CTA.
//
// A stage of radix R takes its R values from the previous stage's buffer in
// shared memory, does the butterfly in registers and writes to the other
// buffer.  The first stage takes its values from a functor (global memory, a
// filter product, the real-row packing) and the last one hands its results to
// a functor, so a transform of n stages crosses shared memory n - 1 times:
// with radices up to 16 that is once up to length 256 and twice up to 2048
// (nearly all lengths).  The loop is bound by instruction issue and the
// exchanges' latency, which is why the radices are as large as the registers
// of two to three resident CTAs of 256 threads allow.  The exchanges alternate between two
// buffers, so that one barrier per exchange is enough: a buffer is written
// again only after the barrier of the exchange in between, which every thread
// reaches after its reads of that buffer.
//
// Columns (COLS): element i of sequence b at i B + b, consecutive threads on
// consecutive sequences.  Rows: at b pitch + i, consecutive threads on
// consecutive butterflies.  The first stage writes i = j R + q; for an even R
// that stride maps half-warps onto few banks, so with `pad` index i of the
// first exchange is stored at i + i / R0 (R0 the first radix): the writes then
// go to j (R0 + 1) + q, and the second stage, whose span is R0, reads
// (j + j / R0) + t (nb + nb / R0): one base and a constant stride as without
// padding.
//
// The item functions are __host__ __device__: tests/gfft_host.cu runs every
// length through them on the CPU.
#pragma once

#include "shf_fft16.cuh"
#include "shf_fftv.cuh"

namespace shf {
namespace gf {

// R = A x B point DFT in registers, natural order in and out: DFT-A over a of
// v[a B + b] for each b, twiddles exp(S 2 pi i b q1 / R), DFT-B over b for each
// q1; output q1 + A q2.  c[m], s[m]: cos and sin of 2 pi m / R.
template <int A, int B, int S>
__host__ __device__ __forceinline__ void dft_ab(float2* v, const float* c, const float* s) {
  constexpr int R = A * B;
  float2 y[R];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    float2 x[A];
#pragma unroll
    for (int a = 0; a < A; ++a) x[a] = v[a * B + b];
    dft_small<A, S>(x);
#pragma unroll
    for (int q = 0; q < A; ++q)
      y[q * B + b] = b * q == 0 ? x[q] : r16::cmul_cs(x[q], c[b * q], static_cast<float>(S) * s[b * q]);
  }
#pragma unroll
  for (int q = 0; q < A; ++q) {
    dft_small<B, S>(y + q * B);
#pragma unroll
    for (int p = 0; p < B; ++p) v[q + A * p] = y[q * B + p];
  }
}

template <int R, int S>
__host__ __device__ __forceinline__ void dft(float2* v) {
  if constexpr (R == 16) {
    r16::dft16<S>(*reinterpret_cast<float2(*)[16]>(v));
  } else if constexpr (R == 12) {
    rv::dftv<12, S>(*reinterpret_cast<float2(*)[12]>(v));
  } else if constexpr (R == 6) {  // multiples of 60 degrees
    const float c[3] = {1.f, 0.5f, -0.5f}, s[3] = {0.f, 0.86602540378443864676f, 0.86602540378443864676f};
    dft_ab<3, 2, S>(v, c, s);
  } else if constexpr (R == 9) {  // multiples of 40 degrees (b q <= 4)
    const float c[5] = {1.f, 0.76604444311897803520f, 0.17364817766693034885f, -0.5f, -0.93969262078590838405f};
    const float s[5] = {0.f, 0.64278760968653932632f, 0.98480775301220805937f, 0.86602540378443864676f,
                        0.34202014332566873304f};
    dft_ab<3, 3, S>(v, c, s);
  } else if constexpr (R == 10) {  // multiples of 36 degrees (b q <= 4)
    const float c[5] = {1.f, 0.80901699437494742410f, 0.30901699437494742410f, -0.30901699437494742410f,
                        -0.80901699437494742410f};
    const float s[5] = {0.f, 0.58778525229247312917f, 0.95105651629515357212f, 0.95105651629515357212f,
                        0.58778525229247312917f};
    dft_ab<5, 2, S>(v, c, s);
  } else if constexpr (R == 15) {  // multiples of 24 degrees (b q <= 8)
    const float c[9] = {1.f, 0.91354545764260089550f, 0.66913060635885821383f, 0.30901699437494742410f,
                        -0.10452846326765347140f, -0.5f, -0.80901699437494742410f, -0.97814760073380563793f,
                        -0.97814760073380563793f};
    const float s[9] = {0.f, 0.40673664307580020775f, 0.74314482547739423501f, 0.95105651629515357212f,
                        0.99452189536827333692f, 0.86602540378443864676f, 0.58778525229247312917f,
                        0.20791169081775933710f, -0.20791169081775933710f};
    dft_ab<5, 3, S>(v, c, s);
  } else {
    dft_small<R, S>(v);
  }
}

// Which ends of the transform a stage touches.
enum StageKind { kMid = 0, kFirst = 1, kLast = 2, kOnly = 3 };

// A batch of B sequences: multiplier for B (columns), pitch of a sequence in
// the exchange buffers (rows), and the first exchange's padding.
struct Batch {
  int B;
  unsigned mB;
  int pitch;
  int pad;
};
// Elements of one exchange buffer (columns: B sequences interleaved).
inline int buf_elems(const FftPlan& p, int B, int pad) { return B * (p.L + (pad ? p.L / p.st[0].R : 0)); }
inline Batch make_batch(const FftPlan& p, int B, int pad) {
  return Batch{B, fdiv_mul(static_cast<unsigned>(B)), p.L + (pad ? p.L / p.st[0].R : 0), pad};
}

// Item idx of a stage -> butterfly j of sequence b.
template <bool COLS>
__host__ __device__ __forceinline__ void item_of(const FftStage& g, const Batch& a, int idx, int& j, int& b) {
  if (COLS) {
    j = static_cast<int>(fdiv(static_cast<unsigned>(idx), a.mB));
    b = idx - j * a.B;
  } else {
    b = static_cast<int>(fdiv(static_cast<unsigned>(idx), g.mNb));
    j = idx - b * g.nb;
  }
}

// The R inputs of butterfly j from the previous stage's buffer, times the
// stage's twiddles exp(S 2 pi i t (j mod Ns) / (Ns R)).
template <int R, int S, bool COLS>
__host__ __device__ __forceinline__ void stage_in(const FftStage& g, const Batch& a, bool second, int j, int b,
                                                  const float2* in, const float2* __restrict__ pt, float2 (&v)[R],
                                                  int& k) {
  const int q0 = static_cast<int>(fdiv(static_cast<unsigned>(j), g.mNs));
  k = j - q0 * g.Ns;
  const bool padded = second && a.pad;
  const int i0 = padded ? j + q0 : j;
  const int di = padded ? g.nb + static_cast<int>(fdiv(static_cast<unsigned>(g.nb), g.mNs)) : g.nb;
  const float2* p = COLS ? in + i0 * a.B + b : in + b * a.pitch + i0;
  const int d = COLS ? di * a.B : di;
#pragma unroll
  for (int t = 0; t < R; ++t) v[t] = p[t * d];
  const float2* w = pt + g.off + k;
#pragma unroll
  for (int t = 1; t < R; ++t) {
    float2 x = w[(t - 1) * g.Ns];
    if (S > 0) x.y = -x.y;
    v[t] = c_mul(v[t], x);
  }
}

// The R outputs of butterfly j into the next stage's buffer.
template <int R, bool COLS>
__host__ __device__ __forceinline__ void stage_out(const FftStage& g, const Batch& a, bool first, int j, int b, int k,
                                                   float2* out, const float2 (&v)[R]) {
  const int o = first ? j * (R + (a.pad ? 1 : 0)) : (j - k) * R + k;
  const int di = first ? 1 : g.Ns;
  float2* p = COLS ? out + o * a.B + b : out + b * a.pitch + o;
  const int d = COLS ? di * a.B : di;
#pragma unroll
  for (int q = 0; q < R; ++q) p[q * d] = v[q];
}

// Butterfly idx of a stage; ld(i, b) supplies element i of sequence b to a
// first stage, st(i, b, v) takes the results of a last one.
template <int R, int S, bool COLS, int KIND, class LD, class ST>
__host__ __device__ __forceinline__ void stage_item(const FftStage& g, const Batch& a, bool second, int idx,
                                                    const float2* in, float2* out, const float2* __restrict__ pt,
                                                    LD&& ld, ST&& st) {
  int j, b, k = 0;
  item_of<COLS>(g, a, idx, j, b);
  float2 v[R];
  if constexpr ((KIND & kFirst) != 0) {
#pragma unroll
    for (int t = 0; t < R; ++t) v[t] = ld(j + t * g.nb, b);
  } else {
    stage_in<R, S, COLS>(g, a, second, j, b, in, pt, v, k);
  }
  dft<R, S>(v);
  if constexpr ((KIND & kLast) != 0) {
#pragma unroll
    for (int q = 0; q < R; ++q) st(j + q * g.nb, b, v[q]);
  } else {
    stage_out<R, COLS>(g, a, (KIND & kFirst) != 0, j, b, k, out, v);
  }
}

// Calls f.template run<R>() for the plan's radix.
template <class F>
__host__ __device__ __forceinline__ void with_radix(int R, F&& f) {
  switch (R) {
    case 2: f.template run<2>(); break;
    case 3: f.template run<3>(); break;
    case 4: f.template run<4>(); break;
    case 5: f.template run<5>(); break;
    case 6: f.template run<6>(); break;
    case 8: f.template run<8>(); break;
    case 9: f.template run<9>(); break;
    case 10: f.template run<10>(); break;
    case 12: f.template run<12>(); break;
    case 15: f.template run<15>(); break;
    default: f.template run<16>(); break;
  }
}

// All butterflies of one stage, spread over items i0, i0 + step, ...
template <int S, bool COLS, int KIND, class LD, class ST>
struct StageLoop {
  const FftStage& g;
  const Batch& a;
  bool second;
  const float2* in;
  float2* out;
  const float2* pt;
  LD& ld;
  ST& st;
  int i0, step;
  template <int R>
  __host__ __device__ __forceinline__ void run() {
    const int total = g.nb * a.B;
    for (int idx = i0; idx < total; idx += step) stage_item<R, S, COLS, KIND>(g, a, second, idx, in, out, pt, ld, st);
  }
};
template <int S, bool COLS, int KIND, class LD, class ST>
__host__ __device__ __forceinline__ void run_stage(const FftPlan& p, int s, const Batch& a, const float2* in,
                                                   float2* out, const float2* pt, LD& ld, ST& st, int i0, int step) {
  StageLoop<S, COLS, KIND, LD, ST> f{p.st[s], a, s == 1, in, out, pt, ld, st, i0, step};
  with_radix(p.st[s].R, f);
}

#ifdef __CUDACC__
// The exchange buffers of a CTA; `cur` alternates with every exchange.
struct Exchange {
  float2* buf[2];
  int cur = 0;
  __device__ __forceinline__ float2* next() {
    float2* b = buf[cur];
    cur ^= 1;
    return b;
  }
};

struct NoLd {
  __host__ __device__ float2 operator()(int, int) const { return make_float2(0.f, 0.f); }
};
struct NoSt {
  __host__ __device__ void operator()(int, int, float2) const {}
};

// Every stage but the last one: ld -> ... -> the buffer the last stage reads
// (nullptr for a single-stage plan, whose last stage reads ld itself).
template <int S, bool COLS, class LD>
__device__ __forceinline__ const float2* fft_head(const FftPlan& p, const Batch& a, Exchange& x, const float2* pt,
                                                  LD&& ld) {
  if (p.nst == 1) return nullptr;
  NoSt ns;
  float2* b = x.next();
  run_stage<S, COLS, kFirst>(p, 0, a, nullptr, b, pt, ld, ns, threadIdx.x, blockDim.x);
  __syncthreads();
  NoLd nl;
  for (int s = 1; s + 1 < p.nst; ++s) {
    float2* c = x.next();
    run_stage<S, COLS, kMid>(p, s, a, b, c, pt, nl, ns, threadIdx.x, blockDim.x);
    __syncthreads();
    b = c;
  }
  return b;
}

// A whole transform of the batch: ld -> st.  Every thread of the CTA calls it;
// the caller orders what ld reads and st writes.
template <int S, bool COLS, class LD, class ST>
__device__ __forceinline__ void fft(const FftPlan& p, const Batch& a, Exchange& x, const float2* pt, LD&& ld, ST&& st) {
  const float2* b = fft_head<S, COLS>(p, a, x, pt, ld);
  if (p.nst == 1) {
    run_stage<S, COLS, kOnly>(p, 0, a, nullptr, nullptr, pt, ld, st, threadIdx.x, blockDim.x);
  } else {
    NoLd nl;
    run_stage<S, COLS, kLast>(p, p.nst - 1, a, b, nullptr, pt, nl, st, threadIdx.x, blockDim.x);
  }
}
#endif

}  // namespace gf
}  // namespace shf
