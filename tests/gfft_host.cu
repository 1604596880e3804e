// The staged FFTs of the general lengths (shf_gfft.cuh) on the host: every
// length 2^a 3^b 5^c up to 2048, both directions, rows and columns, the padded
// and the plain first exchange, and the reversed plan, item by item against an
// FP64 DFT; every exchange position stays inside its buffer and is written once.
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
#include <vector>

#include "shf_gfft.cuh"

namespace gf = shf::gf;
using cd = std::complex<double>;

static int g_bad = 0;

struct Load {
  const std::vector<float2>* x;
  int L;
  float2 operator()(int i, int b) const { return (*x)[static_cast<size_t>(b) * L + i]; }
};
struct Store {
  std::vector<float2>* y;
  std::vector<int>* hits;
  int L;
  void operator()(int i, int b, float2 v) const {
    (*y)[static_cast<size_t>(b) * L + i] = v;
    ++(*hits)[static_cast<size_t>(b) * L + i];
  }
};

template <int S, bool COLS>
static double run(const shf::FftPlan& p, int B, int pad, const std::vector<float2>& x, const std::vector<float2>& pt,
                  std::vector<float2>* y) {
  const gf::Batch ba = gf::make_batch(p, B, pad);
  const int n = gf::buf_elems(p, B, pad);
  const float2 mark = make_float2(NAN, NAN);
  std::vector<float2> buf[2] = {std::vector<float2>(n, mark), std::vector<float2>(n, mark)};
  std::vector<int> hits(static_cast<size_t>(B) * p.L, 0);
  Load ld{&x, p.L};
  Store st{y, &hits, p.L};
  gf::NoLd nl;
  gf::NoSt ns;
  if (p.nst == 1) {
    gf::run_stage<S, COLS, gf::kOnly>(p, 0, ba, nullptr, nullptr, pt.data(), ld, st, 0, 1);
  } else {
    int cur = 0;
    gf::run_stage<S, COLS, gf::kFirst>(p, 0, ba, nullptr, buf[0].data(), pt.data(), ld, ns, 0, 1);
    for (int s = 1; s + 1 < p.nst; ++s) {
      buf[cur ^ 1].assign(n, mark);
      gf::run_stage<S, COLS, gf::kMid>(p, s, ba, buf[cur].data(), buf[cur ^ 1].data(), pt.data(), nl, ns, 0, 1);
      cur ^= 1;
    }
    gf::run_stage<S, COLS, gf::kLast>(p, p.nst - 1, ba, buf[cur].data(), nullptr, pt.data(), nl, st, 0, 1);
  }
  for (int h : hits)
    if (h != 1) ++g_bad;
  return 0.0;
}

int main() {
  std::mt19937 rng(7);
  std::normal_distribution<float> nd;
  int lengths = 0;
  double worst = 0.0;
  for (int L = 4; L <= 2048; ++L) {
    shf::FftPlan plan, rev;
    if (!shf::make_plan(L, &plan)) continue;
    if (!shf::make_plan(L, &rev, true)) return 2;
    ++lengths;
    const int B = 3;
    std::vector<float2> x(static_cast<size_t>(B) * L), y(x.size());
    for (auto& v : x) v = make_float2(nd(rng), nd(rng));
    std::vector<cd> root(L);
    for (int m = 0; m < L; ++m) root[m] = std::polar(1.0, -2.0 * M_PI * m / L);
    for (int S = -1; S <= 1; S += 2) {
      // the DFT of the middle sequence at 40 indices
      std::vector<int> at;
      for (int q = 0; q < std::min(L, 40); ++q) at.push_back(static_cast<int>(static_cast<long>(q) * L / std::min(L, 40)));
      std::vector<cd> ref;
      double norm = 0.0;
      for (int i = 0; i < L; ++i) norm += std::norm(cd(x[L + i].x, x[L + i].y));
      norm = std::sqrt(norm);  // 2-norm of the input: the outputs' root mean square
      for (int k : at) {
        cd a = 0.0;
        for (int i = 0; i < L; ++i) {
          const cd w = root[static_cast<long>(i) * k % L];
          a += cd(x[L + i].x, x[L + i].y) * (S < 0 ? w : std::conj(w));
        }
        ref.push_back(a);
      }
      for (const shf::FftPlan* p : {&plan, &rev}) {
        std::vector<float2> pt(shf::plan_table(*p), make_float2(1.f, 0.f));
        for (int s = 1; s < p->nst; ++s) {
          const shf::FftStage& g = p->st[s];
          for (int t = 1; t < g.R; ++t)
            for (int k = 0; k < g.Ns; ++k) {
              const cd w = root[static_cast<long>(t) * k * (L / (g.Ns * g.R)) % L];
              pt[g.off + (t - 1) * g.Ns + k] = make_float2(static_cast<float>(w.real()), static_cast<float>(w.imag()));
            }
        }
        for (int pad = 0; pad <= 1; ++pad)
          for (int cols = 0; cols <= 1; ++cols) {
            y.assign(x.size(), make_float2(NAN, NAN));
            if (S < 0)
              cols ? run<-1, true>(*p, B, pad, x, pt, &y) : run<-1, false>(*p, B, pad, x, pt, &y);
            else
              cols ? run<+1, true>(*p, B, pad, x, pt, &y) : run<+1, false>(*p, B, pad, x, pt, &y);
            for (size_t q = 0; q < at.size(); ++q) {
              const float2 v = y[L + at[q]];
              const double err = std::abs(cd(v.x, v.y) - ref[q]) / norm;
              if (!(err <= 4.0 * 6e-8 * std::max(2.0, std::log2(static_cast<double>(L))))) {
                if (g_bad++ < 10) std::printf("L=%d S=%d pad=%d cols=%d k=%d err=%g\n", L, S, pad, cols, at[q], err);
              }
              worst = std::max(worst, err);
            }
          }
      }
    }
  }
  std::printf("%d lengths, worst %.3g, bad %d\n", lengths, worst, g_bad);
  return g_bad ? 1 : 0;
}
