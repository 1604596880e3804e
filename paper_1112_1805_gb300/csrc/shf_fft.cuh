// FFT building blocks for sm_103a: complex helpers, the small DFTs, the stage
// plans of the general lengths (the transforms themselves are in shf_gfft.cuh),
// and the packing that turns a length-W real transform into a length-W/2
// complex one.  Conventions follow the paper's
// fft2/ifft2 (Sec. 2): forward exponent -1 without scaling, inverse exponent
// +1 (the 1/(H W) factor is applied by the caller).
#pragma once

#include <cuda_runtime.h>

namespace shf {

constexpr int kMaxStages = 8;

// One Stockham stage of a transform of length L: radix, span (product of the
// radices before it), butterflies L / radix, the offset of its twiddles in the
// pass table ([t - 1][j mod span], t = 1..radix - 1), and multipliers that
// divide small integers by the span and by the butterfly count (0: divisor 1).
struct FftStage {
  int R, Ns, nb, off;
  unsigned mNs, mNb;
};
struct FftPlan {
  int L;
  int nst;
  FftStage st[kMaxStages];
};

// x / d for x d < 2^32, from fdiv_mul(d) = floor(2^32 / d) + 1 (d > 1).
__host__ __device__ __forceinline__ unsigned fdiv_mul(unsigned d) {
  return d <= 1 ? 0u : static_cast<unsigned>((1ull << 32) / d) + 1u;
}
__host__ __device__ __forceinline__ unsigned fdiv(unsigned x, unsigned m) {
#ifdef __CUDA_ARCH__
  return m ? __umulhi(x, m) : x;
#else
  return m ? static_cast<unsigned>((static_cast<unsigned long long>(x) * m) >> 32) : x;
#endif
}

// Complex sums on the device use the packed FP32x2 adds of sm_100-class GPUs
// (one instruction for both components, IEEE round-to-nearest per component,
// the same values as two scalar adds); the host emulation keeps plain floats.
__host__ __device__ __forceinline__ float2 c_add(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ float2 c_sub(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "sub.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
#else
  return make_float2(a.x - b.x, a.y - b.y);
#endif
}
__host__ __device__ __forceinline__ float2 c_mul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// Component-wise a * b and a * b + c: packed FP32x2 multiply and fused
// multiply-add on the device (per component the same IEEE operation as the
// scalar one).
__host__ __device__ __forceinline__ float2 c_mul2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
#else
  return make_float2(a.x * b.x, a.y * b.y);
#endif
}
__host__ __device__ __forceinline__ float2 c_fma2(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mov.b64 rc, {%6, %7};\n\tfma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
#else
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
// The last step of the real-row packing, s + i conj(w) d with w = e^{-2 pi i k/W}
// (i conj w = (w.y, w.x): one complex product and one packed add).
__host__ __device__ __forceinline__ float2 pack_combine(float2 s, float2 d, float2 w) {
  return c_add(s, c_mul(make_float2(w.y, w.x), d));
}
// The last step of the real-row unpacking, (s - i w d) / 2 (-i w = (w.y, -w.x)).
__host__ __device__ __forceinline__ float2 unpack_combine(float2 s, float2 d, float2 w) {
  return c_mul2(c_add(s, c_mul(make_float2(w.y, -w.x), d)), make_float2(0.5f, 0.5f));
}
__host__ __device__ __forceinline__ float2 c_conj(float2 a) { return make_float2(a.x, -a.y); }
__host__ __device__ __forceinline__ float2 c_scale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// a * (S i) for S = +1 or -1
template <int S>
__host__ __device__ __forceinline__ float2 c_mul_si(float2 a) {
  return make_float2(-static_cast<float>(S) * a.y, static_cast<float>(S) * a.x);
}

// In-place R-point DFTs V_q = sum_t v_t exp(S 2 pi i t q / R).
template <int S>
__host__ __device__ __forceinline__ void dft2(float2* v) {
  const float2 t = c_sub(v[0], v[1]);
  v[0] = c_add(v[0], v[1]);
  v[1] = t;
}

template <int S>
__host__ __device__ __forceinline__ void dft4_vals(float2& a0, float2& a1, float2& a2, float2& a3) {
  const float2 s02 = c_add(a0, a2), d02 = c_sub(a0, a2);
  const float2 s13 = c_add(a1, a3), t = c_sub(a1, a3);
  a0 = c_add(s02, s13);
  a2 = c_sub(s02, s13);
  // d02 +- S i t with the swapped components in scalar adds (a packed add
  // would first have to move them into a register pair)
  const float s = static_cast<float>(S);
  a1 = make_float2(d02.x - s * t.y, d02.y + s * t.x);
  a3 = make_float2(d02.x + s * t.y, d02.y - s * t.x);
}

template <int S>
__host__ __device__ __forceinline__ void dft4(float2* v) {
  dft4_vals<S>(v[0], v[1], v[2], v[3]);
}

template <int S>
__host__ __device__ __forceinline__ void dft8(float2* v) {
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4_vals<S>(e0, e1, e2, e3);
  dft4_vals<S>(o0, o1, o2, o3);
  const float r = 0.70710678118654752440f;
  const float s = static_cast<float>(S);
  const float2 t1 = make_float2(r * (o1.x - s * o1.y), r * (o1.y + s * o1.x));    // * (1 + S i)/sqrt(2)
  const float2 t2 = c_mul_si<S>(o2);                                               // * S i
  const float2 t3 = make_float2(r * (-o3.x - s * o3.y), r * (-o3.y + s * o3.x));  // * (-1 + S i)/sqrt(2)
  v[0] = c_add(e0, o0);
  v[4] = c_sub(e0, o0);
  v[1] = c_add(e1, t1);
  v[5] = c_sub(e1, t1);
  v[2] = c_add(e2, t2);
  v[6] = c_sub(e2, t2);
  v[3] = c_add(e3, t3);
  v[7] = c_sub(e3, t3);
}

template <int S>
__host__ __device__ __forceinline__ void dft3(float2* v) {
  const float h = static_cast<float>(S) * 0.86602540378443864676f;  // S sin(2 pi / 3)
  const float2 t1 = c_add(v[1], v[2]), t2 = c_sub(v[1], v[2]);
  const float2 m = make_float2(v[0].x - 0.5f * t1.x, v[0].y - 0.5f * t1.y);
  const float2 n = make_float2(-h * t2.y, h * t2.x);
  v[0] = c_add(v[0], t1);
  v[1] = c_add(m, n);
  v[2] = c_sub(m, n);
}

template <int S>
__host__ __device__ __forceinline__ void dft5(float2* v) {
  const float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;  // cos(2pi/5), cos(4pi/5)
  const float s1 = static_cast<float>(S) * 0.95105651629515357212f;         // S sin(2pi/5)
  const float s2 = static_cast<float>(S) * 0.58778525229247312917f;         // S sin(4pi/5)
  const float2 a1 = c_add(v[1], v[4]), b1 = c_sub(v[1], v[4]);
  const float2 a2 = c_add(v[2], v[3]), b2 = c_sub(v[2], v[3]);
  const float2 p1 = make_float2(v[0].x + c1 * a1.x + c2 * a2.x, v[0].y + c1 * a1.y + c2 * a2.y);
  const float2 p2 = make_float2(v[0].x + c2 * a1.x + c1 * a2.x, v[0].y + c2 * a1.y + c1 * a2.y);
  const float2 r1 = make_float2(s1 * b1.x + s2 * b2.x, s1 * b1.y + s2 * b2.y);
  const float2 r2 = make_float2(s2 * b1.x - s1 * b2.x, s2 * b1.y - s1 * b2.y);
  const float2 q1 = make_float2(-r1.y, r1.x);  // i * r1 (S folded into s1, s2)
  const float2 q2 = make_float2(-r2.y, r2.x);
  v[0] = make_float2(v[0].x + a1.x + a2.x, v[0].y + a1.y + a2.y);
  v[1] = c_add(p1, q1);
  v[4] = c_sub(p1, q1);
  v[2] = c_add(p2, q2);
  v[3] = c_sub(p2, q2);
}

template <int R, int S>
__host__ __device__ __forceinline__ void dft_small(float2* v) {
  if (R == 2) dft2<S>(v);
  if (R == 3) dft3<S>(v);
  if (R == 4) dft4<S>(v);
  if (R == 5) dft5<S>(v);
  if (R == 8) dft8<S>(v);
}

// Real transforms of length W = 2L through one complex transform of length L.
// twW[m] = exp(-2 pi i m / W).
//
// Inverse packing: from the half spectrum X[0..L] of a real row, the complex
// sequence whose unscaled inverse DFT of length L has the even samples of the
// unscaled length-W inverse in its real part and the odd samples in its
// imaginary part:  Z[k] = (X[k] + conj X[L-k]) + i e^{+2 pi i k/W} (X[k] - conj X[L-k])
// (pack_combine, on what the row kernels load of X).
//
// Forward unpacking: Z = DFT_L(x[2n] + i x[2n+1]); returns X[k], k = 0..L,
// X[k] = 1/2 [ (Z_k + conj Z_{L-k}) - i e^{-2 pi i k/W} (Z_k - conj Z_{L-k}) ] (indices mod L).
__host__ __device__ __forceinline__ float2 r2c_unpack(const float2* Z, int L, int k, const float2* twW) {
  const float2 a = Z[k == L ? 0 : k];
  const float2 b = c_conj(Z[k == 0 ? 0 : L - k]);
  const float2 s = c_add(a, b), d = c_sub(a, b);
  return unpack_combine(s, d, twW[k]);
}

// Fills a plan from its radices in order.
inline void set_stages(FftPlan* p, int L, const int* radix, int n) {
  p->L = L;
  p->nst = n;
  int Ns = 1, off = 0;
  for (int s = 0; s < n; ++s) {
    FftStage& g = p->st[s];
    g.R = radix[s];
    g.Ns = Ns;
    g.nb = L / g.R;
    g.off = off;
    g.mNs = fdiv_mul(static_cast<unsigned>(Ns));
    g.mNb = fdiv_mul(static_cast<unsigned>(g.nb));
    if (s > 0) off += (g.R - 1) * Ns;
    Ns *= g.R;
  }
}

// Stage plan for L = 2^a 3^b 5^c: the fewest stages of radices up to 16, then
// the smallest sum of radices (registers and twiddles), in increasing order or,
// for `reversed`, in decreasing order (the forward transform of the v-step,
// whose first stage takes over the last stage's registers of the inverse one).
// False when L has another prime factor.
inline bool make_plan(int L, FftPlan* p, bool reversed = false) {
  constexpr int kRadices[] = {2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16};
  if (L < 1) return false;
  int best[kMaxStages], nbest = kMaxStages + 1, sbest = 0, cur[kMaxStages];
  auto search = [&](auto&& self, int rest, int depth, int from, int sum) -> void {
    if (rest == 1) {
      if (depth >= 1 && (depth < nbest || (depth == nbest && sum < sbest))) {
        nbest = depth;
        sbest = sum;
        for (int i = 0; i < depth; ++i) best[i] = cur[i];
      }
      return;
    }
    if (depth >= kMaxStages || depth >= nbest) return;
    for (int i = from; i < 11; ++i)
      if (rest % kRadices[i] == 0) {
        cur[depth] = kRadices[i];
        self(self, rest / kRadices[i], depth + 1, i, sum + kRadices[i]);
      }
  };
  search(search, L, 0, 0, 0);
  if (nbest > kMaxStages) return false;
  if (reversed)
    for (int i = 0; i < nbest / 2; ++i) {
      const int t = best[i];
      best[i] = best[nbest - 1 - i];
      best[nbest - 1 - i] = t;
    }
  set_stages(p, L, best, nbest);
  return true;
}

// The radices 8 (as many as fit), then 4 or 2, then 3s and 5s: the sequence of
// the unrolled sweeps, whose gradients hang on which side of the clip threshold
// a rounded coefficient falls, so that their iterates stay bit for bit what
// they have been.  False when L has another prime factor.
inline bool make_sweep_plan(int L, FftPlan* p) {
  int radix[16], n = 0, rest = L, a = 0;
  for (; rest % 2 == 0; rest /= 2) ++a;
  for (int i = 0; i < a / 3; ++i) radix[n++] = 8;
  if (a % 3) radix[n++] = a % 3 == 2 ? 4 : 2;
  for (; rest % 3 == 0; rest /= 3) radix[n++] = 3;
  for (; rest % 5 == 0; rest /= 5) radix[n++] = 5;
  if (rest != 1 || n < 1 || n > kMaxStages) return false;
  set_stages(p, L, radix, n);
  return true;
}

// Entries of a plan's pass table.
inline int plan_table(const FftPlan& p) {
  int n = 0;
  for (int s = 1; s < p.nst; ++s) n += (p.st[s].R - 1) * p.st[s].Ns;
  return n > 0 ? n : 1;
}

}  // namespace shf
