// The library's states on the stand-in runtime of fake_cudart.h: every allocation
// of every call is made to fail once.  A call that runs out of memory says so,
// leaves the state usable, returns what it had taken in the order of the stream it
// was taken on, and nothing is left when everything is destroyed.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <string>
#include <vector>

#include "fake_cudart.h"
#include "shearseg.h"

namespace {

int failures = 0;
void expect(bool ok, const char* what, int n = 0) {
  if (!ok) {
    ++failures;
    std::printf("FAILED: %s (%d): %s\n", what, n, shf_last_error());
  }
}

struct Problem {
  int H, W, K, J;
  std::vector<float> f, cb, lam;
  shf_bank* bank = nullptr;
  Problem(int h, int w, int k, int j) : H(h), W(w), K(k), J(j), f(static_cast<size_t>(h) * w, 0.5f), lam(j + 1, 0.01f) {
    for (int i = 0; i < k; ++i) cb.push_back(0.1f * (i + 1));
    expect(shfilters_build(H, W, J, nullptr, &bank) == SHF_OK, "bank");
  }
  ~Problem() { shfilters_destroy(bank); }
  int init(seg_state** st) {
    seg_params p{};
    p.gamma = 1.f;
    p.Lambda = lam.data();
    p.J = J;
    p.max_iters = 10;
    return seg_admm_init(bank, f.data(), 1, cb.data(), K, &p, nullptr, st);
  }
};

// Calls `call` with its first, second, ... allocation failing, until none is left
// to fail; the number of calls that ran out of memory.  A call may do without the
// allocation that failed; `undo` then takes its result back.
template <typename F, typename U>
int exhaust(const char* what, F&& call, U&& undo) {
  int out = 0;
  for (int n = 1; n < 200; ++n) {
    fake::fail_alloc_at = n;
    const int rc = call();
    const bool none_failed = fake::fail_alloc_at > 0;
    fake::fail_alloc_at = 0;
    expect(rc == SHF_OK || (!none_failed && rc == SHF_ERR_OOM), what, n);
    if (none_failed) return out;
    if (rc == SHF_OK)
      undo();
    else
      ++out;
  }
  expect(false, what);
  return out;
}

void plans_and_sweeps(int H, int W) {
  Problem pb(H, W, 3, 2);
  seg_state* st = nullptr;
  expect(exhaust("init", [&] { return pb.init(&st); }, [&] { seg_admm_destroy(st); }) > 10, "init: failing allocations");
  seg_plan plan{};
  expect(seg_admm_get_plan(st, &plan) == SHF_OK, "get_plan");
  if (plan.fast) {
    plan.wave_mib = 1;
  } else {
    plan.groups = plan.groups > 1 ? 1 : 2;
  }
  expect(seg_admm_step(st, 2) == SHF_OK, "step");
  const auto nothing = [] {};
  expect(exhaust("set_plan", [&] { return seg_admm_set_plan(st, &plan); }, nothing) >= 2, "set_plan: failing allocations");
  expect(seg_admm_step(st, 2) == SHF_OK, "step");
  expect(exhaust("unrolled_fwd", [&] { return seg_admm_unrolled_fwd(st, 6, 2); }, nothing) >= 3, "unrolled_fwd: failing allocations");
  std::vector<float> g(static_cast<size_t>(H) * W * 3, 0.f);
  expect(exhaust("unrolled_bwd", [&] { return seg_admm_unrolled_bwd_enqueue(st, g.data()); }, nothing) >= 1,
         "unrolled_bwd: failing allocations");
  expect(seg_admm_destroy(st) == SHF_OK, "destroy");
}

// The unrolled sweeps' tables of the general path: a launch that fails is reported,
// and the next call makes them after all.
void failed_tables() {
  Problem pb(30, 50, 3, 2);
  seg_state* st = nullptr;
  expect(pb.init(&st) == SHF_OK, "init");
  const std::size_t before = fake::live();
  fake::fail_kernel = "k_pass_table";
  expect(seg_admm_unrolled_fwd(st, 4, 2) == SHF_ERR_CUDA, "unrolled_fwd: tables fail");
  expect(!fake::fail_kernel && fake::live() == before, "unrolled_fwd: buffers of a failed setup");
  const int tables = fake::launched("k_pass_table");
  expect(seg_admm_unrolled_fwd(st, 4, 2) == SHF_OK, "unrolled_fwd after a failed one");
  expect(fake::launched("k_pass_table") == tables + 3, "unrolled_fwd: the tables of three plans");
  expect(seg_admm_destroy(st) == SHF_OK, "destroy");
}

// The comparison models on a stream that can't be captured (the stand-in's never
// can): the iterations are launched directly.
const int kH = 64, kW = 128, kK = 3;
const std::vector<float> kImage(static_cast<size_t>(kH) * kW, 0.5f), kCodes{0.2f, 0.5f, 0.8f};
int tv_init(tv_state** st) {
  tv_params p{1.f, 0.1f, 0};
  return tv_admm_init(kH, kW, kImage.data(), 1, kCodes.data(), kK, &p, nullptr, st);
}
int nl_init(nl_state** st) {
  nl_params p{};
  p.gamma = 0.2f;
  p.lambda = 0.03f;
  p.patch = 5;
  p.window = 15;
  p.neighbours = 5;
  p.a = 2.f;
  return nl_admm_init(kH, kW, kImage.data(), 1, kCodes.data(), kK, &p, nullptr, st);
}
void no_capture() {
  tv_state* tv = nullptr;
  expect(tv_init(&tv) == SHF_OK && tv_admm_step(tv, 1) == SHF_OK, "tv: init, step");
  expect(tv_admm_step(tv, 3) == SHF_OK && tv_admm_destroy(tv) == SHF_OK, "tv: step, destroy");
  nl_state* nl = nullptr;
  expect(nl_init(&nl) == SHF_OK && nl_admm_step(nl, 1) == SHF_OK, "nl: init, step");
  expect(nl_admm_step(nl, 3) == SHF_OK && nl_admm_destroy(nl) == SHF_OK, "nl: step, destroy");
}

// An error is reported by the call that meets it and by no later one.
void reported_once() {
  Problem pb(270, 64, 3, 2);  // general path, more than one plane per CTA
  seg_state* st = nullptr;
  expect(pb.init(&st) == SHF_OK, "init");
  std::vector<float> u(3ul * 270 * 64, 0.f), c(13 * u.size(), 0.f);
  double energy = 0;
  const auto once = [](const char* what, auto&& call) {
    for (int n = 1; n <= 2; ++n) {
      fake::fail_alloc_at = n;
      const int rc = call();
      const bool failed = fake::fail_alloc_at == 0;
      fake::fail_alloc_at = 0;
      expect((rc != SHF_OK) == failed && call() == SHF_OK, what, n);
    }
    fake::fail_kernel = "k_";
    expect(call() == SHF_ERR_CUDA && call() == SHF_OK, what);
  };
  once("analyze", [&] { return shearlet_analyze(pb.bank, u.data(), 3, c.data(), nullptr); });
  once("synthesize", [&] { return shearlet_synthesize(pb.bank, c.data(), 3, u.data(), nullptr); });
  once("energy", [&] { return seg_admm_get(st, SEG_ENERGY, &energy, 1); });
  once("set v", [&] { return seg_admm_set(st, SEG_V, c.data(), 1); });
  expect(seg_admm_destroy(st) == SHF_OK, "destroy");
}

// A readout into memory that another stream may still use comes after that stream.
void readouts() {
  cudaStream_t other = nullptr;
  cudaStreamCreateWithFlags(&other, cudaStreamNonBlocking);
  std::vector<float> out(3ul * 64 * 128, 0.f), in(out);
  Problem pb(64, 64, 3, 2);
  seg_state* st = nullptr;
  tv_state* tv = nullptr;
  nl_state* nl = nullptr;
  expect(pb.init(&st) == SHF_OK && tv_init(&tv) == SHF_OK && nl_init(&nl) == SHF_OK, "init");
  const auto check = [&](const char* what, auto&& read) {
    cudaMemcpyAsync(out.data(), in.data(), 4, cudaMemcpyDeviceToDevice, other);
    const int n = fake::waits();
    expect(read() == SHF_OK && fake::waits() == n + 1, what);
    expect(cudaGetLastError() == cudaSuccess, what);
  };
  check("seg_admm_read", [&] { return seg_admm_read(st, SEG_W, out.data(), other); });
  check("tv_admm_read", [&] { return tv_admm_read(tv, SEG_W, out.data(), other); });
  check("nl_admm_read", [&] { return nl_admm_read(nl, SEG_W, out.data(), other); });
  expect(seg_admm_read(st, 99, out.data(), other) == SHF_ERR_ARG, "unknown selector");
  expect(seg_admm_destroy(st) == SHF_OK && tv_admm_destroy(tv) == SHF_OK && nl_admm_destroy(nl) == SHF_OK, "destroy");
}

// A batch's iterations run as a graph on the batch's stream, tuning and readouts on
// the images' own.
struct Batch {
  std::vector<float> f, cb{0.2f, 0.5f, 0.8f}, lam;
  seg_batch* b = nullptr;
  Batch() : f(64 * 64, 0.5f), lam(3, 0.01f) {
    const int H[2] = {64, 30}, W[2] = {64, 50}, C[2] = {1, 1}, K[2] = {3, 3};
    const float* fs[2] = {f.data(), f.data()};
    const float* cbs[2] = {cb.data(), cb.data()};
    seg_params p[2] = {};
    for (seg_params& x : p) {
      x.gamma = 1.f;
      x.Lambda = lam.data();
      x.J = 2;
      x.max_iters = 10;
    }
    expect(seg_admm_batch_init(2, H, W, C, K, fs, cbs, p, nullptr, &b) == SHF_OK, "batch init");
  }
  ~Batch() { expect(seg_admm_batch_destroy(b) == SHF_OK, "batch destroy"); }
};
void batch_order() {
  fake::capture = true;
  {
    Batch ba;
    expect(seg_admm_batch_step(ba.b, 4) == SHF_OK && seg_admm_batch_tune(ba.b, 2) == SHF_OK, "tune after iterations");
    expect(seg_admm_batch_step(ba.b, 2) == SHF_OK && seg_admm_batch_sync(ba.b) == SHF_OK, "iterations after tune");
    // what a call leaves on an image's stream is not beside the next iterations
    std::vector<float> x(3ul * 13 * 64 * 64, 0.f);
    for (int i = 0; i < 2; ++i) {
      seg_state* st = nullptr;
      expect(seg_admm_batch_image(ba.b, i, &st) == SHF_OK, "image", i);
      for (int what : {SEG_W, SEG_STV, SEG_V}) {
        expect(seg_admm_set(st, what, x.data(), 0) == SHF_OK, "set", what);
        expect(seg_admm_batch_step(ba.b, 1) == SHF_OK && seg_admm_batch_sync(ba.b) == SHF_OK, "iteration");
      }
      for (int what : {SEG_W, SEG_STV, SEG_LABELS}) {
        expect(seg_admm_get(st, what, x.data(), 0) == SHF_OK, "get", what);
        expect(seg_admm_batch_step(ba.b, 1) == SHF_OK && seg_admm_batch_sync(ba.b) == SHF_OK, "iteration");
      }
    }
    expect(fake::violations == 0, "batch: streams in order", fake::violations);
  }
  fake::capture = false;
}

// What a state takes only to be faster it does without when memory is short: the
// larger waves of the default plans, TV's second b_v, NL-means ranks of all rows at
// once.
void short_of_memory() {
  {
    // coefficient spectra of all labels: 264 MB in one wave, b_v 256 MB
    Problem pb(512, 512, 4, 4);
    seg_state* st = nullptr;
    seg_plan plan{};
    expect(pb.init(&st) == SHF_OK && seg_admm_get_plan(st, &plan) == SHF_OK && plan.wave_mib > 128, "default waves");
    expect(seg_admm_destroy(st) == SHF_OK, "destroy");
    fake::fail_over = 260000000;
    expect(pb.init(&st) == SHF_OK, "init with little memory");
    fake::fail_over = 0;
    if (st) {
      expect(seg_admm_get_plan(st, &plan) == SHF_OK && plan.wave_mib == 128, "waves of 128 MiB", plan.wave_mib);
      expect(seg_admm_step(st, 2) == SHF_OK && seg_admm_destroy(st) == SHF_OK, "step, destroy");
    }
  }
  const auto served = [](const char* what, auto&& init, auto&& destroy) {  // without the n-th allocation
    int out = 0;
    exhaust(what, init, [&] {
      ++out;
      destroy();
    });
    destroy();
    return out;
  };
  tv_state* tv = nullptr;
  expect(served("tv_init", [&] { return tv_init(&tv); },
                [&] { expect(tv_admm_step(tv, 3) == SHF_OK && tv_admm_destroy(tv) == SHF_OK, "tv step, destroy"); }) == 1,
         "tv: without the second b_v");
  nl_state* nl = nullptr;
  expect(served("nl_init", [&] { return nl_init(&nl); },
                [&] { expect(nl_admm_step(nl, 3) == SHF_OK && nl_admm_destroy(nl) == SHF_OK, "nl step, destroy"); }) == 1,
         "nl: ranks of fewer rows at a time");
}

}  // namespace

int main() {
  plans_and_sweeps(64, 64);  // register-FFT path
  plans_and_sweeps(30, 50);  // general path
  failed_tables();
  no_capture();
  reported_once();
  readouts();
  batch_order();
  short_of_memory();
  expect(fake::violations == 0, "buffers returned in order", fake::violations);
  expect(fake::live() == 0, "buffers left", static_cast<int>(fake::live()));
  std::printf("%s\n", failures ? "failed" : "all ok");
  return failures ? 1 : 0;
}
