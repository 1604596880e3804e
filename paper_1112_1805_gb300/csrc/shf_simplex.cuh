// Pixelwise Euclidean projection onto the unit simplex (the w-step of the
// ADMM of Sec. 3), shared by the u/w-step kernels of both regularisers.
#pragma once

namespace shf {

// Projection of g[0..K) onto {x >= 0, sum x = 1}, as the paper constructs it:
// project onto the hyperplane sum = 1 (g + (1 - sum g)/q), set the negative
// components to zero and repeat on the remaining ones (at most K passes; the
// result is exact).  K <= KMAX <= 32.
template <int KMAX>
__device__ __forceinline__ void simplex_project(float (&g)[KMAX], int K) {
  unsigned act = (K >= 32) ? 0xffffffffu : ((1u << K) - 1u);
  float tau = 0.f;
  for (int pass = 0; pass < K; ++pass) {
    float sum = 0.f;
    int q = 0;
#pragma unroll
    for (int k = 0; k < KMAX; ++k)
      if ((act >> k) & 1u) {
        sum += g[k];
        ++q;
      }
    tau = (sum - 1.f) / static_cast<float>(q);
    unsigned nact = act;
#pragma unroll
    for (int k = 0; k < KMAX; ++k)
      if (((act >> k) & 1u) && g[k] - tau < 0.f) nact &= ~(1u << k);
    if (nact == act) break;
    act = nact;
  }
#pragma unroll
  for (int k = 0; k < KMAX; ++k) g[k] = ((act >> k) & 1u) ? g[k] - tau : 0.f;
}

// The same projection in closed form: with the values in decreasing order and
// their sums S_j, the threshold is the largest (S_j - 1) / j.  A sorting network
// and running sums without branches: about 25 instructions for four labels,
// where the passes above take some 200 with their divisions and the warp waits
// for its slowest lane (the TV band kernel at 512 x 512, K = 4: 6.6 to 5.6 M warp
// instructions, the iteration 26 -> 23 us).
// The sums run over the sorted values, so results agree to rounding; the unrolled
// sweeps' iterations keep the form above.  A NaN or infinity makes every result
// NaN.
template <int KMAX>
__device__ __forceinline__ void simplex_project_sorted(float (&g)[KMAX], int K) {
  static_assert(KMAX == 4 || KMAX == 8 || KMAX == 16, "sorting networks of 4, 8 and 16 values");
  float v[KMAX];
  float all = 0.f;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    v[k] = k < K ? g[k] : -INFINITY;
    all += k < K ? g[k] : 0.f;
  }
  // odd-even merge sort, decreasing
#pragma unroll
  for (int p = 1; p < KMAX; p *= 2)
#pragma unroll
    for (int h = p; h >= 1; h /= 2)
#pragma unroll
      for (int j = h % p; j + h < KMAX; j += 2 * h)
#pragma unroll
        for (int i = 0; i < h; ++i)
          if (i + j + h < KMAX && (i + j) / (2 * p) == (i + j + h) / (2 * p)) {
            const float a = v[i + j], b = v[i + j + h];
            v[i + j] = fmaxf(a, b);
            v[i + j + h] = fminf(a, b);
          }
  float s = 0.f, tau = -INFINITY;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    s += v[k];
    const float r = 1.f / static_cast<float>(k + 1), q = (s - 1.f) * r;
    // the rounded quotient (exact for powers of two)
    const float t = ((k + 1) & k) == 0 ? q : fmaf(fmaf(-static_cast<float>(k + 1), q, s - 1.f), r, q);
    tau = k < K ? fmaxf(tau, t) : tau;
  }
  tau += all - all;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const float x = g[k] - tau;
    g[k] = k < K && !(x < 0.f) ? x : 0.f;
  }
}

}  // namespace shf
