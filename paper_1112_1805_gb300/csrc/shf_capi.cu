// C ABI of the shearlet segmentation library: filter banks, the shearlet
// transform and the ADMM state (Haeuser & Steidl, arXiv:1112.1805).  Argument
// checking, buffer ownership, CUDA-graph capture of one ADMM iteration,
// readouts and checkpoints.  All arithmetic runs in the kernels of
// shf_bank.cu and shf_transform.cu.
#include <cmath>
#include <cstdio>
#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "shearseg.h"
#include "shf_internal.h"

using shf::Geo;

namespace {

thread_local std::string g_err;

// An error of the runtime is reported once: left pending, it would be taken for
// that of the next kernel launched.
int fail(int code, const std::string& msg) {
  g_err = msg;
  if (code == SHF_ERR_CUDA || code == SHF_ERR_OOM) cudaGetLastError();
  return code;
}

#define SHF_CK(call)                                                                              \
  do {                                                                                            \
    cudaError_t e_ = (call);                                                                      \
    if (e_ != cudaSuccess) return fail(SHF_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

bool aligned8(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7u) == 0; }

template <typename T>
int dev_alloc(T** p, size_t count, const char* what) {
  *p = nullptr;
  if (count == 0) return SHF_OK;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), count * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return fail(e == cudaErrorMemoryAllocation ? SHF_ERR_OOM : SHF_ERR_CUDA,
                std::string("cudaMalloc(") + what + "): " + cudaGetErrorString(e));
  }
  return SHF_OK;
}

int check_sizes(int H, int W, int J) {
  if (J < 1 || J > shf::kMaxJ) return fail(SHF_ERR_ARG, "J must be in [1, 6]");
  if (H < 8 || W < 8 || H > shf::kMaxSide || W > shf::kMaxSide)
    return fail(SHF_ERR_SIZE, "H and W must be in [8, 2048]");
  if (W & 1) return fail(SHF_ERR_SIZE, "W must be even");
  shf::FftPlan p;
  if (!shf::make_plan(H, &p) || !shf::make_plan(W / 2, &p))
    return fail(SHF_ERR_SIZE, "H and W/2 must be products of powers of 2, 3 and 5");
  return SHF_OK;
}

}  // namespace

struct shf_bank {
  Geo g;
  float* bank = nullptr;
  int2* ranges = nullptr;
  std::vector<int2> ranges_host;  // the filters' column ranges
  float2* twH = nullptr;
  float2* twW = nullptr;
  float2* pt = nullptr;  // the plans' pass tables
  shf::FilterDesc* descs = nullptr;
  int device = 0;
  cudaMemPool_t pool = nullptr;  // the device's (DevicePool), shared by its banks
  // Heights with register-FFT column kernels: the work list of one channel's
  // filters, used by the transforms for every channel (its device arrays in
  // `chan_mem`).
  bool chan_ok = false;
  shf::FastPlan chan;
  int* chan_mem = nullptr;
};

struct seg_state {
  const shf_bank* bank = nullptr;
  cudaMemPool_t pool = nullptr;  // the device's, shared
  std::vector<void*> direct;     // buffers too large for it (cudaMalloc)
  int device = 0;
  seg_batch* batch = nullptr;  // the batch whose graphs replay this state, if any
  Geo g;
  int K = 0, C = 0;
  float gamma = 1.f;
  std::vector<float> Lambda;
  std::vector<float> codebook;  // [K][C], host copy for seg_admm_reset
  int max_iters = 0;
  float tol = 0.f;
  int check_every = 1;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float *f = nullptr, *s = nullptr, *bv = nullptr, *w = nullptr, *bw = nullptr, *u = nullptr, *stv = nullptr;
  float2 *Ur = nullptr, *Y = nullptr, *partial = nullptr, *T = nullptr;
  float *thr = nullptr, *lam = nullptr, *gap = nullptr;
  int* labels = nullptr;
  int* bad = nullptr;  // pinned host memory, written by the restart kernel
  double* red = nullptr;
  int groups = 1;
  std::vector<shf::FilterWave> waves;  // general path: the waves of `groups` filter groups
  cudaGraphExec_t exec = nullptr;        // one iteration
  cudaGraphExec_t exec_timed = nullptr;  // the same with an event before every launch
  bool graph_tried = false;
  bool untimed = false;  // steps record no per-kernel events (the tuner's trials)
  bool fast = false;          // power-of-two sizes: the shf_fast.cu kernels
  bool fast_ustep = false;    // ... including the u/w-step (K <= 8)
  shf::FastPlan plan;         // fast path: static per-wave work list
  int* d_lists = nullptr;     // fast path: the plan's work lists
  float2* uhat = nullptr;     // fast path: 2-D spectra of u [K][H][Wh]
  // Events recorded before every launch of an iteration (graph event nodes),
  // with the kind of the launch that follows each.
  // created when a timed iteration is first captured, as many as it has marks
  static constexpr int kMaxMarks = 8192;
  std::vector<cudaEvent_t> ev;
  std::vector<int> kinds;
  int nmarks = 0;
  bool marks_ok = true;
  // unrolled mode (reverse-mode differentiation): generic-path scratch and
  // the states kept every un_ck iterations
  int un_T = 0, un_ck = 0;
  float2* un_Y = nullptr;        // a wave's spectra [planes][H][Wy]
  float2* un_partial = nullptr;  // [un_groups][K][H][Wh]
  int un_groups = 0;
  std::vector<shf::FilterWave> un_waves;
  Geo un_g;                      // general path: the geometry on sweep plans
  float2* un_pt = nullptr;       // ... and their pass tables
  std::vector<float*> ck_bv, ck_w, ck_bw;
  std::vector<float2*> ck_T;
  // the forward and reverse sweeps captured as graphs for (T, ckpt) = un_key;
  // the reverse sweep's temporaries live in un_mem (un_mem_bytes)
  cudaGraphExec_t un_fwd_exec = nullptr, un_bwd_exec = nullptr;
  int un_fwd_key[2] = {0, 0}, un_bwd_key[2] = {0, 0};
  char* un_mem = nullptr;
  size_t un_mem_bytes = 0;
  bool un_bwd_pending = false;  // a reverse sweep was enqueued (its results are in un_mem)
  long long iter = 0;
  size_t P() const { return static_cast<size_t>(g.H) * g.W; }
  size_t Ph() const { return static_cast<size_t>(g.H) * g.Wh; }
};

namespace shf {
void bank_geo(const shf_bank* b, Geo* g) { *g = b->g; }

cudaError_t order_after(cudaStream_t st, cudaStream_t earlier) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = st == earlier ? cudaSuccess : cudaStreamIsCapturing(earlier, &cs);
  if (e != cudaSuccess || st == earlier || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return cudaSuccess;
  }
  // (an event and a wait take the host 0.8 us, asking first whether they are needed 1.5)
  cudaEvent_t ev = nullptr;
  e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  if (e != cudaSuccess) return e;
  e = cudaEventRecord(ev, earlier);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev, 0);
  cudaEventDestroy(ev);
  return e;
}

int bank_device(const shf_bank* b) { return b->device; }
int set_error(int code, const std::string& msg) { return fail(code, msg); }
}  // namespace shf

namespace {

// Stream-ordered temporary memory from the bank's pool.
cudaError_t scratch_alloc(const shf_bank* b, float2** p, size_t count, cudaStream_t st) {
  const size_t bytes = sizeof(float2) * count;
  return b->pool ? cudaMallocFromPoolAsync(reinterpret_cast<void**>(p), bytes, b->pool, st)
                 : cudaMallocAsync(reinterpret_cast<void**>(p), bytes, st);
}

// The library's memory pool of a device, for the transforms' temporaries and the
// states' buffers: made with the first bank there and destroyed with the last
// bank or state.  It keeps up to kPoolKeep bytes between calls: the device's default pool
// gives its memory back whenever the device is waited for, and a call after that
// pays for mapping it again (a 64 x 64 analysis: 256 us against 30 us in a row).
// Without one (an older driver) the default pool and cudaMalloc serve.
constexpr unsigned long long kPoolKeep = 512ull << 20;
constexpr int kMaxDevices = 64;
struct DevicePool {
  cudaMemPool_t pool = nullptr;
  int users = 0;
  // pinned host integers for the states' flags (one page for kFlags of them)
  int* flags = nullptr;
  std::vector<int*> free_flags;
};
constexpr int kFlags = 1024;
std::mutex g_pool_mu;
DevicePool g_pools[kMaxDevices];

cudaMemPool_t acquire_pool(int device) {
  if (device < 0 || device >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  DevicePool& d = g_pools[device];
  if (!d.pool) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    unsigned long long keep = kPoolKeep;
    if (cudaMemPoolCreate(&d.pool, &props) != cudaSuccess) {
      d.pool = nullptr;
    } else if (cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      cudaMemPoolDestroy(d.pool);
      d.pool = nullptr;
    }
    cudaGetLastError();
    if (!d.pool) return nullptr;
  }
  ++d.users;
  return d.pool;
}

// After the device has been waited for.
void release_pool(int device) {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  DevicePool& d = g_pools[device];
  if (--d.users > 0) return;
  cudaStreamSynchronize(nullptr);  // the states' frees
  cudaMemPoolDestroy(d.pool);
  d.pool = nullptr;
  cudaFreeHost(d.flags);
  d.flags = nullptr;
  d.free_flags.clear();
}

// A pinned host integer: from the device's page, or its own allocation.
int acquire_flag(int device, int** flag) {
  if (device >= 0 && device < kMaxDevices) {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    DevicePool& d = g_pools[device];
    if (d.pool && !d.flags && cudaMallocHost(reinterpret_cast<void**>(&d.flags), sizeof(int) * kFlags) == cudaSuccess)
      for (int i = 0; i < kFlags; ++i) d.free_flags.push_back(d.flags + i);
    cudaGetLastError();
    if (!d.free_flags.empty()) {
      *flag = d.free_flags.back();
      d.free_flags.pop_back();
      return SHF_OK;
    }
  }
  SHF_CK(cudaMallocHost(reinterpret_cast<void**>(flag), sizeof(int)));
  return SHF_OK;
}

void release_flag(int device, int* flag) {
  if (!flag) return;
  if (device >= 0 && device < kMaxDevices) {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    DevicePool& d = g_pools[device];
    if (d.flags && flag >= d.flags && flag < d.flags + kFlags) {
      d.free_flags.push_back(flag);
      return;
    }
  }
  cudaFreeHost(flag);
}

// A work list's four arrays one after another (the items as four ints each);
// at[i]: where array i starts.
std::vector<int> pack_lists(const std::vector<shf::WorkItem>& items, const std::vector<int>& cta_begin,
                            const std::vector<int>& tile_begin, const std::vector<int>& tile_slots, size_t (&at)[3]) {
  std::vector<int> all(4 * items.size());
  std::memcpy(all.data(), items.data(), sizeof(shf::WorkItem) * items.size());
  const std::vector<int>* parts[] = {&cta_begin, &tile_begin, &tile_slots};
  for (int i = 0; i < 3; ++i) {
    at[i] = all.size();
    all.insert(all.end(), parts[i]->begin(), parts[i]->end());
  }
  return all;
}
void set_lists(shf::FastPlan* p, const int* mem, const size_t (&at)[3]) {
  p->items = reinterpret_cast<const shf::WorkItem*>(mem);
  p->cta_begin = mem + at[0];
  p->tile_begin = mem + at[1];
  p->tile_slots = mem + at[2];
}

// The single-channel work list of a bank whose ranges are known; synchronous.
int build_channel_plan(shf_bank* b, const std::vector<int2>& ranges) {
  const Geo& g = b->g;
  shf::FastPlan& p = b->chan;
  p.wave_mib = shf::default_fast_plan(g).wave_mib;
  p.col_ctas = shf::fast_col_ctas(g, 0);
  p.fan_ctas = shf::fast_fan_ctas(g);
  if (p.col_ctas < 1 || p.fan_ctas < 1) return fail(SHF_ERR_CUDA, "shfilters_build: no resident CTA");
  std::vector<shf::WorkItem> items;
  std::vector<int> cta_begin, tile_begin, tile_slots;
  shf::build_fast_plan(g, ranges.data(), 1, &p, &items, &cta_begin, &tile_begin, &tile_slots);
  size_t at[3];
  const std::vector<int> all = pack_lists(items, cta_begin, tile_begin, tile_slots, at);
  int rc = dev_alloc(&b->chan_mem, all.size(), "work list");
  if (rc) return rc;
  SHF_CK(cudaMemcpy(b->chan_mem, all.data(), sizeof(int) * all.size(), cudaMemcpyHostToDevice));
  set_lists(&p, b->chan_mem, at);
  b->chan_ok = true;
  return SHF_OK;
}

// Transforms on whole planes in shared memory: small images, and no more CTAs
// (one per channel and filter) than a few per SM; an analysis CTA repeats the
// forward transform of its channel, a synthesis ends in one CTA per channel.
// Up to 5000 half-spectrum values a synthesis takes 30 us (four channels), less
// than four launches in a row; at 8320 57 us, more.
bool small_transform(const Geo& g, int nch, bool analysis) {
  return shf::small_ok(g) && static_cast<long long>(nch) * g.eta <= 4 * 152 && (analysis || g.H * g.Wh <= 5000);
}

// Channels of a launch over the single-channel plan: as many as keep the wave's
// spectra within the plan's budget.
int channels_per_launch(const shf_bank* b, int nch) {
  const size_t plane = sizeof(float2) * static_cast<size_t>(b->g.H) * b->g.Wy;
  const size_t per = plane * static_cast<size_t>(b->chan.y_planes);
  return static_cast<int>(std::max<size_t>(1, std::min<size_t>(nch, (static_cast<size_t>(b->chan.wave_mib) << 20) / per)));
}

}  // namespace

extern "C" {

int shf_version(void) { return 100; }

const char* shf_last_error(void) { return g_err.c_str(); }

int shfilters_build(int H, int W, int J, void* stream, shf_bank** out) {
  if (!out) return fail(SHF_ERR_ARG, "out is NULL");
  *out = nullptr;
  int rc = check_sizes(H, W, J);
  if (rc) return rc;
  Geo g;
  if (!shf::make_geo(H, W, J, &g)) return fail(SHF_ERR_SIZE, "unsupported geometry");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int device = 0, optin = 0;
  SHF_CK(cudaGetDevice(&device));
  SHF_CK(shf::prepare_kernels(g));
  SHF_CK(shf::prepare_fast_kernels(g));
  SHF_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
  if (shf::max_dynamic_smem_needed(g, shf::kMaxK) > optin)
    return fail(SHF_ERR_SIZE, "tile does not fit in shared memory");
  auto* b = new shf_bank();
  b->g = g;
  b->device = device;
  b->pool = acquire_pool(device);
  std::vector<shf::FilterDesc> d(g.eta);
  shf::filter_descs(J, d.data());
  if ((rc = dev_alloc(&b->bank, static_cast<size_t>(g.eta) * H * g.Wh, "bank")) ||
      (rc = dev_alloc(&b->twH, H, "twH")) || (rc = dev_alloc(&b->twW, W, "twW")) ||
      (rc = dev_alloc(&b->pt, shf::pass_table_entries(g), "pass tables")) ||
      (rc = dev_alloc(&b->descs, g.eta, "descs")) || (rc = dev_alloc(&b->ranges, g.eta, "ranges"))) {
    shfilters_destroy(b);
    return rc;
  }
  b->g.bank = b->bank;
  b->g.ranges = b->ranges;
  if (cudaError_t es = shf::prepare_small(b->g); es != cudaSuccess) {
    shfilters_destroy(b);
    return fail(SHF_ERR_CUDA, std::string("shfilters_build: ") + cudaGetErrorString(es));
  }
  b->g.twH = b->twH;
  b->g.twW = b->twW;
  cudaError_t e = cudaMemcpyAsync(b->descs, d.data(), sizeof(shf::FilterDesc) * g.eta, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = shf::launch_twiddles(b->twH, H, st);
  if (e == cudaSuccess) e = shf::launch_twiddles(b->twW, W, st);
  if (e == cudaSuccess) e = shf::launch_pass_tables(&b->g, b->pt, st);
  if (e == cudaSuccess) e = shf::launch_build_bank(b->bank, b->g, b->descs, st);
  if (e == cudaSuccess) e = shf::launch_filter_ranges(b->bank, b->g, b->ranges, st);
  std::vector<int2>& ranges = b->ranges_host;
  ranges.resize(g.eta);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ranges.data(), b->ranges, sizeof(int2) * g.eta, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // d and ranges are host temporaries
  if (e != cudaSuccess) {
    shfilters_destroy(b);
    return fail(SHF_ERR_CUDA, std::string("shfilters_build: ") + cudaGetErrorString(e));
  }
  if (shf::fast_columns_ok(b->g) && (rc = build_channel_plan(b, ranges))) {
    const std::string m = g_err;
    shfilters_destroy(b);
    return fail(rc, m);
  }
  *out = b;
  return SHF_OK;
}

int shfilters_destroy(shf_bank* b) {
  if (!b) return SHF_OK;
  cudaDeviceSynchronize();
  cudaFree(b->bank);
  cudaFree(b->twH);
  cudaFree(b->twW);
  cudaFree(b->pt);
  cudaFree(b->chan_mem);
  if (b->pool) release_pool(b->device);
  cudaFree(b->descs);
  cudaFree(b->ranges);
  delete b;
  return SHF_OK;
}

int shfilters_info(const shf_bank* b, int* eta, int* H, int* W, int* J) {
  if (!b) return fail(SHF_ERR_ARG, "bank is NULL");
  if (eta) *eta = b->g.eta;
  if (H) *H = b->g.H;
  if (W) *W = b->g.W;
  if (J) *J = b->g.J;
  return SHF_OK;
}

int shfilters_copy(const shf_bank* b, float* dst, void* stream) {
  if (!b || !dst) return fail(SHF_ERR_ARG, "NULL argument");
  SHF_CK(cudaMemcpyAsync(dst, b->bank, sizeof(float) * b->g.eta * b->g.H * b->g.Wh, cudaMemcpyDeviceToDevice,
                         static_cast<cudaStream_t>(stream)));
  return SHF_OK;
}

int shearlet_analyze(const shf_bank* b, const float* u, int nch, float* coef, void* stream) {
  if (!b || !u || !coef || nch < 1) return fail(SHF_ERR_ARG, "shearlet_analyze: bad argument");
  if (!aligned8(u) || !aligned8(coef)) return fail(SHF_ERR_ARG, "shearlet_analyze: pointers must be 8-byte aligned");
  const Geo& g = b->g;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t ph = static_cast<size_t>(g.H) * g.Wh;
  const float scale = 1.f / (static_cast<float>(g.H) * g.W);
  if (small_transform(g, nch, true)) {
    const cudaError_t e = shf::run_small_analyze(g, u, coef, nch, scale, st);
    if (e != cudaSuccess) return fail(SHF_ERR_CUDA, std::string("shearlet_analyze: ") + cudaGetErrorString(e));
    return SHF_OK;
  }
  if (b->chan_ok) {
    const size_t php = static_cast<size_t>(g.H) * g.Wy;
    const int nc = channels_per_launch(b, nch);
    const size_t ny = php * b->chan.y_planes * static_cast<size_t>(nc);
    float2* tmp = nullptr;
    cudaError_t e = scratch_alloc(b, &tmp, ny + (php + ph) * static_cast<size_t>(nch), st);
    if (e != cudaSuccess) return fail(SHF_ERR_OOM, std::string("shearlet_analyze: ") + cudaGetErrorString(e));
    float2 *Y = tmp, *uhat = tmp + ny, *Ur = uhat + php * nch;
    e = shf::run_row_r2c(g, u, Ur, nch, 1.f, st);
    if (e == cudaSuccess) e = shf::run_channel_fwd(g, Ur, uhat, nch, st);
    for (int w = 0; w < static_cast<int>(b->chan.wave_f0.size()); ++w)
      for (int c = 0; c < nch && e == cudaSuccess; c += nc) {
        const shf::FilterWave wv{c, std::min(nc, nch - c), b->chan.wave_f0[w], b->chan.wave_nf[w]};
        e = shf::run_channel_fan(g, b->chan, w, uhat, Y, wv, st);
        if (e == cudaSuccess) e = shf::run_wave_c2r(g, Y, coef, wv, scale, st);
      }
    cudaError_t e2 = cudaFreeAsync(tmp, st);
    if (e != cudaSuccess || e2 != cudaSuccess)
      return fail(SHF_ERR_CUDA, std::string("shearlet_analyze: ") + cudaGetErrorString(e != cudaSuccess ? e : e2));
    return SHF_OK;
  }
  const std::vector<shf::FilterWave> waves = shf::general_waves(g, nch, shf::default_groups(g, nch));
  float2* tmp = nullptr;
  cudaError_t e = scratch_alloc(b, &tmp, ph * nch + shf::wave_planes(waves) * g.H * g.Wy, st);
  if (e != cudaSuccess) return fail(SHF_ERR_OOM, std::string("shearlet_analyze: ") + cudaGetErrorString(e));
  float2* Ur = tmp + shf::wave_planes(waves) * g.H * g.Wy;
  float2* Y = tmp;
  e = shf::run_row_r2c(g, u, Ur, nch, 1.f, st);
  if (e == cudaSuccess) e = shf::run_col_fwd(g, Ur, nch, st);
  for (const shf::FilterWave& wv : waves) {
    if (e == cudaSuccess) e = shf::run_wave_fan(g, Ur, Y, wv, st);
    if (e == cudaSuccess) e = shf::run_wave_c2r(g, Y, coef, wv, scale, st);
  }
  cudaError_t e2 = cudaFreeAsync(tmp, st);
  if (e != cudaSuccess || e2 != cudaSuccess)
    return fail(SHF_ERR_CUDA, std::string("shearlet_analyze: ") + cudaGetErrorString(e != cudaSuccess ? e : e2));
  return SHF_OK;
}

namespace {
// T[nch][H][Wh] = column-inverse of sum_f W_f * fft2(coef_f) (unscaled).
cudaError_t synthesis_spectrum(const shf_bank* b, const Geo& g, const float* coef, int nch, float2* T,
                               cudaStream_t st) {
  if (b->chan_ok) {
    const size_t php = static_cast<size_t>(g.H) * g.Wy;
    const int nc = channels_per_launch(b, nch);
    const size_t ny = php * b->chan.y_planes * static_cast<size_t>(nc);
    const size_t np = static_cast<size_t>(std::max(b->chan.nslots, 1)) * g.H * shf::fast_tile(g);
    float2* tmp = nullptr;
    cudaError_t e = scratch_alloc(b, &tmp, ny + np * static_cast<size_t>(nch), st);
    if (e != cudaSuccess) return e;
    float2 *Z = tmp, *part = tmp + ny;
    for (int w = 0; w < static_cast<int>(b->chan.wave_f0.size()); ++w)
      for (int c = 0; c < nch && e == cudaSuccess; c += nc) {
        const shf::FilterWave wv{c, std::min(nc, nch - c), b->chan.wave_f0[w], b->chan.wave_nf[w]};
        e = shf::run_wave_r2c(g, coef, Z, wv, st);
        if (e == cudaSuccess) e = shf::run_channel_gather(g, b->chan, w, Z, part, wv, st);
      }
    if (e == cudaSuccess) e = shf::run_channel_reduce(g, b->chan, part, T, nch, st);
    cudaError_t e2 = cudaFreeAsync(tmp, st);
    return e != cudaSuccess ? e : e2;
  }
  const size_t ph = static_cast<size_t>(g.H) * g.Wh;
  const int groups = shf::default_groups(g, nch);
  const std::vector<shf::FilterWave> waves = shf::general_waves(g, nch, groups);
  const size_t ny = shf::wave_planes(waves) * g.H * g.Wy;
  float2* tmp = nullptr;
  cudaError_t e = scratch_alloc(b, &tmp, ny + ph * nch * static_cast<size_t>(groups), st);
  if (e != cudaSuccess) return e;
  float2* Z = tmp;
  float2* part = tmp + ny;
  for (const shf::FilterWave& wv : waves) {
    if (e == cudaSuccess) e = shf::run_wave_r2c(g, coef, Z, wv, st);
    if (e == cudaSuccess) e = shf::run_wave_gather(g, Z, part, nch, groups, wv, st);
  }
  if (e == cudaSuccess) e = shf::run_col_reduce_inv(g, part, T, nch, groups, st);
  cudaError_t e2 = cudaFreeAsync(tmp, st);
  return e != cudaSuccess ? e : e2;
}
}  // namespace

int shearlet_synthesize(const shf_bank* b, const float* coef, int nch, float* u, void* stream) {
  if (!b || !coef || !u || nch < 1) return fail(SHF_ERR_ARG, "shearlet_synthesize: bad argument");
  if (!aligned8(u) || !aligned8(coef))
    return fail(SHF_ERR_ARG, "shearlet_synthesize: pointers must be 8-byte aligned");
  const Geo& g = b->g;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (small_transform(g, nch, false)) {
    float2* part = nullptr;
    cudaError_t e = scratch_alloc(b, &part, shf::small_partials(g, nch), st);
    if (e != cudaSuccess) return fail(SHF_ERR_OOM, std::string("shearlet_synthesize: ") + cudaGetErrorString(e));
    e = shf::run_small_synthesize(g, coef, u, part, nch, 1.f / (static_cast<float>(g.H) * g.W), st);
    cudaError_t e2 = cudaFreeAsync(part, st);
    if (e == cudaSuccess) e = e2;
    if (e != cudaSuccess) return fail(SHF_ERR_CUDA, std::string("shearlet_synthesize: ") + cudaGetErrorString(e));
    return SHF_OK;
  }
  const size_t ph = static_cast<size_t>(g.H) * g.Wh;
  float2* T = nullptr;
  cudaError_t e = scratch_alloc(b, &T, ph * nch, st);
  if (e != cudaSuccess) return fail(SHF_ERR_OOM, std::string("shearlet_synthesize: ") + cudaGetErrorString(e));
  e = synthesis_spectrum(b, g, coef, nch, T, st);
  if (e == cudaSuccess) e = shf::run_row_c2r(g, T, u, nch, 1.f / (static_cast<float>(g.H) * g.W), st);
  cudaError_t e2 = cudaFreeAsync(T, st);
  if (e != cudaSuccess || e2 != cudaSuccess)
    return fail(SHF_ERR_CUDA, std::string("shearlet_synthesize: ") + cudaGetErrorString(e != cudaSuccess ? e : e2));
  return SHF_OK;
}

// ---------------------------------------------------------------------------
// ADMM state
// ---------------------------------------------------------------------------

namespace {

// Returns a state's buffer in the order of `order`: what that stream has queued by
// now runs before the pool hands the memory on.  A call that fails leaves no error
// behind for a later launch's check (in a broken context those fail by themselves).
void state_free_in(seg_state* st, void* p, cudaStream_t order) {
  if (!p) return;
  const auto it = std::find(st->direct.begin(), st->direct.end(), p);
  cudaError_t e;
  if (it == st->direct.end()) {
    e = cudaFreeAsync(p, order);
  } else {
    st->direct.erase(it);
    e = cudaFree(p);
  }
  if (e != cudaSuccess) cudaGetLastError();
}
// ... of its own stream, in which pool memory is allocated and used: a buffer that
// an unfinished call gives back has its allocation there, and maybe a user.
void state_free(seg_state* st, void* p) { state_free_in(st, p, st->stream); }

void free_state(seg_state* s) {
  // The caller's stream may be gone by now: everything is waited for, and the
  // buffers go back in the order of the legacy stream.
  cudaDeviceSynchronize();
  const auto give = [s](void* p) { state_free_in(s, p, nullptr); };
  if (s->exec) cudaGraphExecDestroy(s->exec);
  if (s->exec_timed) cudaGraphExecDestroy(s->exec_timed);
  for (cudaEvent_t e : s->ev)
    if (e) cudaEventDestroy(e);
  give(s->uhat);
  give(s->d_lists);
  give(s->un_Y);
  give(s->un_partial);
  give(s->un_pt);
  if (s->un_fwd_exec) cudaGraphExecDestroy(s->un_fwd_exec);
  if (s->un_bwd_exec) cudaGraphExecDestroy(s->un_bwd_exec);
  give(s->un_mem);
  for (float* p : s->ck_bv) give(p);
  for (float* p : s->ck_w) give(p);
  for (float* p : s->ck_bw) give(p);
  for (float2* p : s->ck_T) give(p);
  float* fl[] = {s->f, s->s, s->bv, s->w, s->bw, s->u, s->stv, s->thr, s->lam, s->gap};
  for (float* p : fl) give(p);
  give(s->Ur);
  give(s->Y);
  give(s->partial);
  give(s->T);
  give(s->labels);
  release_flag(s->device, s->bad);
  give(s->red);
  if (s->own_stream && s->stream) cudaStreamDestroy(s->stream);
  if (s->pool) release_pool(s->device);
  delete s;
}

// Data term from st->f and a zero state; checks f for NaN/Inf (synchronises).
int restart(seg_state* st, const float* codebook) {
  const Geo& g = st->g;
  const size_t P = st->P();
  *st->bad = 0;
  SHF_CK(shf::launch_restart(st->f, st->C, codebook, st->K, st->s, st->w, st->bw, st->u, static_cast<int>(P), st->T,
                             static_cast<long long>(st->Ph()) * st->K, st->bad, st->stream));
  SHF_CK(cudaMemsetAsync(st->bv, 0, sizeof(float) * P * st->K * g.eta, st->stream));
  SHF_CK(cudaStreamSynchronize(st->stream));
  st->iter = 0;
  if (*st->bad) return fail(SHF_ERR_NONFINITE, "image contains NaN or Inf");
  return SHF_OK;
}

// Launches of one iteration, plus the closing mark.
int marks_needed(const seg_state* st) {
  if (!st->fast) return 4 + 3 * static_cast<int>(st->waves.size());
  int n = 4;  // u/w-step, column forward, reduction, end
  n += 3 * static_cast<int>(st->plan.wave_f0.size());  // fan, v-step, gather per wave
  return n;
}

// Creates the timing events an iteration of the current plan needs (at most
// kMaxMarks); a failure leaves the timing disabled.
void ensure_marks(seg_state* st) {
  const size_t need = static_cast<size_t>(std::min(marks_needed(st), static_cast<int>(seg_state::kMaxMarks)));
  while (st->ev.size() < need) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) {
      cudaGetLastError();
      break;
    }
    st->ev.push_back(e);
  }
  st->kinds.resize(st->ev.size());
}

// Records the event of the next mark; during stream capture it becomes an
// event-record node of the graph (cudaEventRecordExternal), so that each
// replay timestamps it.  A failed record only disables the timing (its error
// is cleared, not left for a later call to report).
void mark_launch(void* ctx, int kind) {
  auto* st = static_cast<seg_state*>(ctx);
  if (st->nmarks >= static_cast<int>(st->ev.size())) {
    st->marks_ok = false;
    return;
  }
  const int i = st->nmarks++;
  st->kinds[i] = kind;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st->stream, &cs);
  if (e == cudaSuccess)
    e = cs == cudaStreamCaptureStatusActive ? cudaEventRecordWithFlags(st->ev[i], st->stream, cudaEventRecordExternal)
                                            : cudaEventRecord(st->ev[i], st->stream);
  if (e != cudaSuccess) {
    st->marks_ok = false;
    cudaGetLastError();
  }
}

// One ADMM iteration; `timed`: with an event recorded before every launch and
// after the last one; `code` (fast path, optional): the per-coefficient codes
// of the v-step for the reverse mode.
cudaError_t enqueue_iteration(seg_state* st, bool timed, signed char* code = nullptr) {
  const Geo& g = st->g;
  const shf::PdlScope pdl(!(st->fast && st->plan.serial));
  const float scale = 1.f / (static_cast<float>(g.H) * g.W);
  cudaStream_t s = st->stream;
  shf::LaunchHook hook;
  if (timed) {
    hook.fn = mark_launch;
    hook.ctx = st;
    st->nmarks = 0;
    st->marks_ok = true;
  }
  hook.mark(shf::kKindUstep);
  cudaError_t e =
      st->fast_ustep
          ? shf::run_fast_ustep(g, st->T, st->s, st->w, st->bw, st->u, st->Ur, st->K, st->gamma, scale, s)
          : shf::run_row_ustep(g, st->T, st->s, st->w, st->bw, st->u, st->Ur, nullptr, st->K, st->gamma, scale, s);
  if (st->fast) {
    if (e == cudaSuccess)
      e = shf::run_fast_iteration_body(g, st->plan, st->Ur, st->uhat, st->Y, st->bv, st->thr, st->partial, st->T,
                                       st->K, scale, s, hook, code);
  } else {
    hook.mark(shf::kKindColFwd);
    if (e == cudaSuccess) e = shf::run_col_fwd(g, st->Ur, st->K, s);
    for (const shf::FilterWave& wv : st->waves) {
      hook.mark(shf::kKindFan);
      if (e == cudaSuccess) e = shf::run_wave_fan(g, st->Ur, st->Y, wv, s);
      hook.mark(shf::kKindShrink);
      if (e == cudaSuccess) e = shf::run_wave_shrink(g, st->Y, st->bv, st->thr, wv, scale, s);
      hook.mark(shf::kKindGather);
      if (e == cudaSuccess) e = shf::run_wave_gather(g, st->Y, st->partial, st->K, st->groups, wv, s);
    }
    hook.mark(shf::kKindReduce);
    if (e == cudaSuccess) e = shf::run_col_reduce_inv(g, st->partial, st->T, st->K, st->groups, s);
  }
  hook.mark(shf::kKindEnd);
  return e;
}

// One iteration on the general path's sweep plans with the unrolled mode's
// scratch; gout (optional) records g = b_v + S u.
cudaError_t enqueue_generic_iteration(seg_state* st, float* gout) {
  const Geo& g = st->un_g;
  const float scale = 1.f / (static_cast<float>(g.H) * g.W);
  cudaStream_t s = st->stream;
  cudaError_t e =
      shf::run_row_ustep(g, st->T, st->s, st->w, st->bw, st->u, st->Ur, nullptr, st->K, st->gamma, scale, s);
  if (e == cudaSuccess) e = shf::run_col_fwd(g, st->Ur, st->K, s);
  for (const shf::FilterWave& wv : st->un_waves) {
    if (e == cudaSuccess) e = shf::run_wave_fan(g, st->Ur, st->un_Y, wv, s);
    if (e == cudaSuccess) e = shf::run_wave_shrink(g, st->un_Y, st->bv, st->thr, wv, scale, s, gout);
    if (e == cudaSuccess) e = shf::run_wave_gather(g, st->un_Y, st->un_partial, st->K, st->un_groups, wv, s);
  }
  if (e == cudaSuccess) e = shf::run_col_reduce_inv(g, st->un_partial, st->T, st->K, st->un_groups, s);
  return e;
}

cudaGraphExec_t capture_iteration(seg_state* st, bool timed) {
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  if (cudaStreamBeginCapture(st->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  cudaError_t e = enqueue_iteration(st, timed);
  cudaError_t e2 = cudaStreamEndCapture(st->stream, &graph);
  if (e == cudaSuccess && e2 == cudaSuccess && graph && (!timed || st->marks_ok)) {
    if (cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) exec = nullptr;
  }
  if (graph) cudaGraphDestroy(graph);
  cudaGetLastError();
  return exec;
}

// Captures one iteration into two graphs (plain, and with the timing events)
// when the stream can be captured (not the legacy default stream); otherwise
// iterations are launched directly.  An iteration with more launches than
// timing marks keeps only the plain graph (seg_admm_kernel_times then reports
// the timing as unavailable).
void try_capture(seg_state* st) {
  st->graph_tried = true;
  ensure_marks(st);
  if (st->stream == nullptr) return;
  st->exec = capture_iteration(st, false);
  if (st->exec) st->exec_timed = capture_iteration(st, true);
}

void drop_batch_graphs(seg_batch* b);

void drop_graphs(seg_state* st) {
  // a batch's graphs hold this state's buffers: they go too (a new plan
  // reallocates them)
  if (st->batch) drop_batch_graphs(st->batch);
  if (st->exec) cudaGraphExecDestroy(st->exec);
  if (st->exec_timed) cudaGraphExecDestroy(st->exec_timed);
  if (st->un_fwd_exec) cudaGraphExecDestroy(st->un_fwd_exec);
  if (st->un_bwd_exec) cudaGraphExecDestroy(st->un_bwd_exec);
  st->exec = st->exec_timed = st->un_fwd_exec = st->un_bwd_exec = nullptr;
  st->un_fwd_key[0] = st->un_fwd_key[1] = st->un_bwd_key[0] = st->un_bwd_key[1] = 0;
  st->graph_tried = false;
}

// Captures the work `enqueue` puts on the state's stream into an executable
// graph; nullptr when the stream cannot be captured or the work failed.
extern "C++" template <typename F>
cudaGraphExec_t capture_work(seg_state* st, F enqueue) {
  if (st->stream == nullptr) return nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  if (cudaStreamBeginCapture(st->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  cudaError_t e = enqueue();
  cudaError_t e2 = cudaStreamEndCapture(st->stream, &graph);
  if (e == cudaSuccess && e2 == cudaSuccess && graph && cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess)
    exec = nullptr;
  if (graph) cudaGraphDestroy(graph);
  cudaGetLastError();
  return exec;
}

// A state's buffers come from the device's pool in the order of its stream: a training step that makes a state per image then
// maps no memory.  Buffers that the pool would not keep anyway are mapped by
// cudaMalloc, which takes fewer and larger pages (the 17 GB of a 2048 x 2048, K =
// 8 state: 43 ms of preparation against 59).
extern "C++" template <typename T>
int state_alloc(seg_state* st, T** p, size_t count, const char* what) {
  *p = nullptr;
  if (count == 0) return SHF_OK;
  if (!st->pool || count * sizeof(T) > kPoolKeep / 2) {
    const int rc = dev_alloc(p, count, what);
    if (!rc) st->direct.push_back(*p);
    return rc;
  }
  cudaError_t e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(p), count * sizeof(T), st->pool, st->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return fail(e == cudaErrorMemoryAllocation ? SHF_ERR_OOM : SHF_ERR_CUDA,
                std::string("cudaMallocFromPoolAsync(") + what + "): " + cudaGetErrorString(e));
  }
  return SHF_OK;
}

// Fast path: builds the work list for (wave_mib, col_ctas_per_sm) and
// allocates what depends on it (one wave of coefficient spectra Y, the
// partial tiles, the device work list); the previous buffers are released
// only once the new ones exist.  Synchronises the state's stream.
int install_fast_plan(seg_state* st, int wave_mib, int col_ctas_per_sm, int row_kernel = shf::kRowDefault,
                      int col_kernel = shf::kColDefault, int serial = 0, int sms = 0) {
  const Geo& g = st->g;
  shf::FastPlan plan;
  plan.wave_mib = wave_mib;
  plan.col_ctas_per_sm = col_ctas_per_sm;
  plan.row_kernel = row_kernel;
  plan.col_kernel = col_kernel;
  plan.serial = serial;
  plan.sms = sms;
  plan.col_ctas = shf::fast_col_ctas(g, col_ctas_per_sm, col_kernel, sms);
  plan.fan_ctas = shf::fast_fan_ctas(g, col_kernel, sms);
  plan.row_ctas = shf::fast_row_ctas(g, row_kernel, sms);
  if (plan.col_ctas < 1 || plan.fan_ctas < 1 || plan.row_ctas < 1)
    return fail(SHF_ERR_CUDA, "install_fast_plan: no resident CTA");
  std::vector<shf::WorkItem> h_items;
  std::vector<int> h_cta_begin, h_tile_begin, h_tile_slots;
  shf::build_fast_plan(g, st->bank->ranges_host.data(), st->K, &plan, &h_items, &h_cta_begin, &h_tile_begin,
                       &h_tile_slots);
  const size_t Phs = static_cast<size_t>(g.H) * shf::fast_pitch(g);
  const size_t y_elems = Phs * static_cast<size_t>(std::max(plan.y_planes, 1));
  const size_t partial_elems = static_cast<size_t>(std::max(plan.nslots, 1)) * g.H * shf::fast_tile(g);
  size_t at[3];
  const std::vector<int> lists = pack_lists(h_items, h_cta_begin, h_tile_begin, h_tile_slots, at);
  float2 *Y = nullptr, *partial = nullptr;
  int* d_lists = nullptr;
  auto release = [&]() {
    state_free(st, Y);
    state_free(st, partial);
    state_free(st, d_lists);
  };
  int rc;
  if ((rc = state_alloc(st, &Y, y_elems, "Y")) || (rc = state_alloc(st, &partial, partial_elems, "partial")) ||
      (rc = state_alloc(st, &d_lists, lists.size(), "work lists"))) {
    release();
    return rc;
  }
  cudaError_t e = cudaMemcpyAsync(d_lists, lists.data(), sizeof(int) * lists.size(), cudaMemcpyHostToDevice, st->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st->stream);  // the old buffers may still be in use
  if (e != cudaSuccess) {
    release();
    return fail(SHF_ERR_CUDA, std::string("install_fast_plan: ") + cudaGetErrorString(e));
  }
  drop_graphs(st);
  state_free(st, st->Y);
  state_free(st, st->partial);
  state_free(st, st->d_lists);
  st->Y = Y;
  st->partial = partial;
  st->d_lists = d_lists;
  set_lists(&plan, d_lists, at);
  st->plan = plan;
  return SHF_OK;
}

// The plan that a new state starts with; where its larger waves do not fit in
// memory, waves of kWaveMiB.  (Waves of 1024 MiB hold all spectra of most states,
// another b_v: a 512 x 512, K = 4, J = 4 state takes 570 MB in place of 440.)
int install_default_plan(seg_state* st) {
  const shf::FastPlan def = shf::default_fast_plan(st->g);
  const auto install = [&](int mib) {
    return install_fast_plan(st, mib, 0, def.row_kernel, def.col_kernel, def.serial);
  };
  const int rc = install(def.wave_mib);
  return rc == SHF_ERR_OOM && def.wave_mib > shf::kWaveMiB ? install(shf::kWaveMiB) : rc;
}

// Filter groups as the general-path kernels use them: groups of ceil(eta/G)
// filters, no group empty.
int normalise_groups(int eta, int G) {
  if (G < 1) G = 1;
  if (G > eta) G = eta;
  const int fg = (eta + G - 1) / G;
  return (eta + fg - 1) / fg;
}

// General path: tile shape (TC, RB) and filter groups; reallocates the
// partial sums.  Synchronises the state's stream.
int install_generic_plan(seg_state* st, int TC, int RB, int groups) {
  int dev = 0, optin = 0;
  SHF_CK(cudaGetDevice(&dev));
  SHF_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  Geo g = st->g;
  if (!shf::set_generic_tiles(&g, TC, RB, st->K, optin))
    return fail(SHF_ERR_ARG, "tile shape not supported for this image size");
  groups = normalise_groups(g.eta, groups);
  std::vector<shf::FilterWave> waves = shf::general_waves(g, st->K, groups);
  float2 *partial = nullptr, *Y = nullptr;
  int rc = state_alloc(st, &partial, st->Ph() * st->K * static_cast<size_t>(groups), "partial");
  if (!rc) rc = state_alloc(st, &Y, shf::wave_planes(waves) * g.H * g.Wy, "Y");
  if (rc) {
    state_free(st, partial);
    return rc;
  }
  cudaError_t e = cudaStreamSynchronize(st->stream);
  if (e != cudaSuccess) {
    state_free(st, partial);
    state_free(st, Y);
    return fail(SHF_ERR_CUDA, std::string("install_generic_plan: ") + cudaGetErrorString(e));
  }
  drop_graphs(st);
  state_free(st, st->partial);
  state_free(st, st->Y);
  st->partial = partial;
  st->Y = Y;
  st->g = g;
  st->groups = groups;
  st->waves = std::move(waves);
  return SHF_OK;
}

int energy_of_w(seg_state* st, double* out_host) {
  const Geo& g = st->g;
  const size_t P = st->P();
  const float scale = 1.f / (static_cast<float>(g.H) * g.W);
  // <w, s>
  SHF_CK(shf::launch_dot(st->w, st->s, static_cast<long>(P * st->K), st->red + 2, 512, st->red, st->stream));
  // sum_f Lambda_f ||(S w)_f||_1: row- and column-forward of w, then per wave
  // the fan-out and the l1 of the row-inverse, in stream-ordered temporaries
  const size_t ph = st->Ph();
  const std::vector<shf::FilterWave> waves = shf::general_waves(g, st->K, shf::default_groups(g, st->K));
  const size_t ny = shf::wave_planes(waves) * g.H * g.Wy;
  const int nb = shf::l1_blocks(g, st->K);
  float2* tmp = nullptr;
  SHF_CK(scratch_alloc(st->bank, &tmp, ph * st->K + ny + static_cast<size_t>(nb), st->stream));
  float2* Yw = tmp;
  float2* Uw = Yw + ny;
  double* part = reinterpret_cast<double*>(Uw + ph * st->K);  // float2 units: 8-byte aligned
  cudaError_t e = shf::run_row_r2c(g, st->w, Uw, st->K, 1.f, st->stream);
  if (e == cudaSuccess) e = shf::run_col_fwd(g, Uw, st->K, st->stream);
  for (const shf::FilterWave& wv : waves) {
    if (e == cudaSuccess) e = shf::run_wave_fan(g, Uw, Yw, wv, st->stream);
    if (e == cudaSuccess) e = shf::run_wave_l1(g, Yw, st->lam, wv, scale, part, st->stream);
  }
  if (e == cudaSuccess) e = shf::launch_sum_partials(part, nb, st->red + 1, st->stream);
  cudaError_t e2 = cudaFreeAsync(tmp, st->stream);
  SHF_CK(e);
  SHF_CK(e2);
  double h[2];
  SHF_CK(cudaMemcpyAsync(h, st->red, sizeof(h), cudaMemcpyDeviceToHost, st->stream));
  SHF_CK(cudaStreamSynchronize(st->stream));
  *out_host = h[0] + h[1];
  return SHF_OK;
}

int residual_uw(seg_state* st, double* out_host) {
  const size_t n = st->P() * st->K;
  SHF_CK(shf::launch_sqdiff(st->u, st->w, static_cast<long>(n), st->red + 2, 512, st->red, st->stream));
  double h = 0;
  SHF_CK(cudaMemcpyAsync(&h, st->red, sizeof(double), cudaMemcpyDeviceToHost, st->stream));
  SHF_CK(cudaStreamSynchronize(st->stream));
  *out_host = std::sqrt(h / static_cast<double>(n));
  return SHF_OK;
}

int copy_out(seg_state* st, void* dst, const void* src, size_t bytes, int to_host) {
  SHF_CK(cudaMemcpyAsync(dst, src, bytes, to_host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st->stream));
  if (to_host) SHF_CK(cudaStreamSynchronize(st->stream));
  return SHF_OK;
}

int copy_in(seg_state* st, void* dst, const void* src, size_t bytes, int from_host) {
  SHF_CK(cudaMemcpyAsync(dst, src, bytes, from_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st->stream));
  if (from_host) SHF_CK(cudaStreamSynchronize(st->stream));
  return SHF_OK;
}

}  // namespace

int seg_admm_init(const shf_bank* b, const float* f, int C, const float* codebook, int K, const seg_params* p,
                  void* stream, seg_state** out) {
  if (!out) return fail(SHF_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!b || !f || !codebook || !p || !p->Lambda) return fail(SHF_ERR_ARG, "seg_admm_init: NULL argument");
  if (K < 2 || K > shf::kMaxK) return fail(SHF_ERR_ARG, "K must be in [2, 16]");
  if (C != 1 && C != 3) return fail(SHF_ERR_ARG, "C must be 1 or 3");
  if (p->J != b->g.J) return fail(SHF_ERR_STATE, "params->J differs from the bank's J");
  if (!(p->gamma > 0.f) || !std::isfinite(p->gamma)) return fail(SHF_ERR_ARG, "gamma must be positive and finite");
  if (!aligned8(f)) return fail(SHF_ERR_ARG, "f must be 8-byte aligned");
  for (int i = 0; i < K * C; ++i)
    if (!std::isfinite(codebook[i])) return fail(SHF_ERR_NONFINITE, "codebook contains NaN or Inf");
  for (int j = 0; j <= p->J; ++j)
    if (!std::isfinite(p->Lambda[j]) || p->Lambda[j] < 0.f)
      return fail(SHF_ERR_ARG, "Lambda must be finite and non-negative");
  auto* st = new seg_state();
  st->bank = b;
  st->device = b->device;
  st->pool = acquire_pool(b->device);
  st->g = b->g;
  st->K = K;
  st->C = C;
  st->gamma = p->gamma;
  st->Lambda.assign(p->Lambda, p->Lambda + p->J + 1);
  st->codebook.assign(codebook, codebook + K * C);
  st->max_iters = p->max_iters;
  st->tol = p->tol;
  st->check_every = p->check_every > 0 ? p->check_every : 1;
  if (stream) {
    st->stream = static_cast<cudaStream_t>(stream);
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&st->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      free_state(st);
      return fail(SHF_ERR_CUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e));
    }
    st->own_stream = true;
  }
  const Geo& g = st->g;
  const size_t P = st->P(), Ph = st->Ph();
  st->groups = shf::default_groups(g, K);
  st->fast = shf::fast_path_ok(g);
  st->fast_ustep = shf::fast_ustep_ok(g, K);
  if (!st->fast) st->waves = shf::general_waves(g, K, st->groups);
  int rc;
  if ((rc = state_alloc(st, &st->f, P * C, "f")) || (rc = state_alloc(st, &st->s, P * K, "s")) ||
      (rc = state_alloc(st, &st->bv, P * K * g.eta, "b_v")) || (rc = state_alloc(st, &st->w, P * K, "w")) ||
      (rc = state_alloc(st, &st->bw, P * K, "b_w")) || (rc = state_alloc(st, &st->u, P * K, "u")) ||
      (rc = state_alloc(st, &st->stv, P * K, "stv")) || (rc = state_alloc(st, &st->Ur, Ph * K, "Ur")) ||
      (rc = state_alloc(st, &st->T, Ph * K, "T")) ||
      (st->fast && (rc = state_alloc(st, &st->uhat, static_cast<size_t>(g.H) * shf::fast_pitch(g) * K, "uhat"))) ||
      // one wave's coefficient spectra and one partial sum per filter group on
      // the general path (the fast path's come with its plan)
      (!st->fast && (rc = state_alloc(st, &st->Y, shf::wave_planes(st->waves) * g.H * g.Wy, "Y"))) ||
      (!st->fast && (rc = state_alloc(st, &st->partial, Ph * K * static_cast<size_t>(st->groups), "partial"))) ||
      (rc = state_alloc(st, &st->thr, g.eta, "thr")) || (rc = state_alloc(st, &st->lam, g.eta, "lam")) ||
      (rc = state_alloc(st, &st->gap, P, "gap")) || (rc = state_alloc(st, &st->labels, P, "labels")) ||
      (rc = acquire_flag(st->device, &st->bad)) || (rc = state_alloc(st, &st->red, 2 + 512, "red")) ||
      // last: its size depends on what is left
      (st->fast && (rc = install_default_plan(st)))) {
    free_state(st);
    return rc;
  }
  std::vector<shf::FilterDesc> d(g.eta);
  shf::filter_descs(g.J, d.data());
  std::vector<float> thr(g.eta), lam(g.eta);
  for (int i = 0; i < g.eta; ++i) {
    lam[i] = d[i].kind == 0 ? st->Lambda[0] : st->Lambda[d[i].j + 1];
    thr[i] = st->gamma * lam[i];
  }
  cudaError_t e = cudaMemcpyAsync(st->thr, thr.data(), sizeof(float) * g.eta, cudaMemcpyHostToDevice, st->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(st->lam, lam.data(), sizeof(float) * g.eta, cudaMemcpyHostToDevice, st->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(st->f, f, sizeof(float) * P * C, cudaMemcpyDeviceToDevice, st->stream);
  if (e != cudaSuccess) {
    free_state(st);
    return fail(SHF_ERR_CUDA, std::string("seg_admm_init: ") + cudaGetErrorString(e));
  }
  rc = restart(st, codebook);  // synchronises: thr/lam host vectors stay valid until here
  if (rc) {
    free_state(st);
    return rc;
  }
  *out = st;
  return SHF_OK;
}

int seg_admm_reset(seg_state* st, const float* f, int f_on_host) {
  if (!st || !f) return fail(SHF_ERR_ARG, "seg_admm_reset: NULL argument");
  if (!f_on_host && !aligned8(f)) return fail(SHF_ERR_ARG, "f must be 8-byte aligned");
  SHF_CK(cudaMemcpyAsync(st->f, f, sizeof(float) * st->P() * st->C,
                         f_on_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st->stream));
  return restart(st, st->codebook.data());
}

}  // extern "C"

namespace {
// Whether a state's iterations are launched one by one instead of as graphs: then
// an iteration's first kernel overlaps the end of the iteration before (graph
// launches follow one another with a gap) and a new state pays for no capture.
// In us per iteration and for the first 20 of a state: 64 x 64, K = 3 27.7 -> 25.2
// and 606 -> 489; 128 x 128, K = 4 37.2 -> 34.6; 256 x 256, K = 4 58.1 -> 55.5; the
// general path 1-2% (480 x 640, K = 5 755 -> 753).  Where the iteration is long
// the graph is ahead (512 x 512, K = 4 257.8 against 262.8).
bool launched_directly(const seg_state* st) {
  return !st->fast || static_cast<double>(st->P()) * st->K * st->g.eta <= 3.3e7;
}
}  // namespace

extern "C" {

int seg_admm_step(seg_state* st, int n) {
  if (!st || n < 0) return fail(SHF_ERR_ARG, "seg_admm_step: bad argument");
  if (n == 0) return SHF_OK;
  if (launched_directly(st)) {
    ensure_marks(st);
    for (int i = 0; i < n; ++i) SHF_CK(enqueue_iteration(st, i == n - 1 && !st->untimed));
    st->iter += n;
    return SHF_OK;
  }
  if (!st->graph_tried) try_capture(st);
  // the last iteration of the call records the per-kernel timing events
  for (int i = 0; i < n; ++i) {
    const bool timed = i == n - 1 && !st->untimed;
    if (st->exec) {
      SHF_CK(cudaGraphLaunch(timed && st->exec_timed ? st->exec_timed : st->exec, st->stream));
    } else {
      SHF_CK(enqueue_iteration(st, timed));
    }
  }
  st->iter += n;
  return SHF_OK;
}

int seg_admm_get_plan(const seg_state* st, seg_plan* out) {
  if (!st || !out) return fail(SHF_ERR_ARG, "seg_admm_get_plan: NULL argument");
  out->fast = st->fast ? 1 : 0;
  out->wave_mib = st->fast ? st->plan.wave_mib : 0;
  out->col_ctas_per_sm = st->fast ? st->plan.col_ctas_per_sm : 0;
  out->tile_cols = st->fast ? 0 : st->g.TC;
  out->tile_rows = st->fast ? 0 : st->g.RB;
  out->groups = st->fast ? 0 : st->groups;
  out->us_per_iter = 0.f;
  out->row_kernel = st->fast ? st->plan.row_kernel : 0;
  out->col_kernel = st->fast ? st->plan.col_kernel : 0;
  out->serial = st->fast ? st->plan.serial : 0;
  out->sms = st->fast ? st->plan.sms : 0;
  return SHF_OK;
}

int seg_admm_set_plan(seg_state* st, const seg_plan* p) {
  if (!st || !p) return fail(SHF_ERR_ARG, "seg_admm_set_plan: NULL argument");
  if (st->fast) {
    if (p->col_ctas_per_sm < 0 || p->col_ctas_per_sm > 32 || p->wave_mib < 1 || p->wave_mib > 4096)
      return fail(SHF_ERR_ARG, "seg_admm_set_plan: col_ctas_per_sm must be in [0, 32] and wave_mib in [1, 4096]");
    if (!shf::fast_row_kernel_ok(st->g, p->row_kernel) || !shf::fast_col_kernel_ok(st->g, p->col_kernel))
      return fail(SHF_ERR_ARG, "seg_admm_set_plan: row_kernel or col_kernel not available at this size");
    if (p->serial != 0 && p->serial != 1) return fail(SHF_ERR_ARG, "seg_admm_set_plan: serial must be 0 or 1");
    if (p->sms < 0 || p->sms > 65536) return fail(SHF_ERR_ARG, "seg_admm_set_plan: sms must be in [0, 65536]");
    if (p->col_ctas_per_sm == st->plan.col_ctas_per_sm && p->wave_mib == st->plan.wave_mib &&
        p->row_kernel == st->plan.row_kernel && p->col_kernel == st->plan.col_kernel && p->sms == st->plan.sms) {
      if (p->serial != st->plan.serial) {  // same buffers, other launches: capture the graphs again
        st->plan.serial = p->serial;
        drop_graphs(st);
      }
      return SHF_OK;
    }
    return install_fast_plan(st, p->wave_mib, p->col_ctas_per_sm, p->row_kernel, p->col_kernel, p->serial, p->sms);
  }
  if (p->tile_cols < 1 || p->tile_rows < 1 || p->groups < 1)
    return fail(SHF_ERR_ARG, "seg_admm_set_plan: tile_cols, tile_rows and groups must be positive");
  if (p->tile_cols == st->g.TC && p->tile_rows == st->g.RB && normalise_groups(st->g.eta, p->groups) == st->groups)
    return SHF_OK;
  return install_generic_plan(st, p->tile_cols, p->tile_rows, p->groups);
}

}  // extern "C"

namespace {

// Mean time (microseconds) of one iteration over `iters` replays, after one
// warm-up iteration that also captures the graphs.
// Average time of `iters` iterations of the plain graph (without the event
// nodes of the timed iteration, which cost differently per plan).
int time_iterations(seg_state* st, int iters, float* us) {
  st->untimed = true;
  struct Restore {
    seg_state* st;
    ~Restore() { st->untimed = false; }
  } restore{st};
  int rc = seg_admm_step(st, 1);
  if (rc) return rc;
  cudaEvent_t a = nullptr, b = nullptr;
  SHF_CK(cudaEventCreate(&a));
  cudaError_t e = cudaEventCreate(&b);
  if (e == cudaSuccess) e = cudaEventRecord(a, st->stream);
  if (e == cudaSuccess) rc = seg_admm_step(st, iters);
  if (e == cudaSuccess && !rc) e = cudaEventRecord(b, st->stream);
  if (e == cudaSuccess && !rc) e = cudaEventSynchronize(b);
  float ms = 0.f;
  if (e == cudaSuccess && !rc) e = cudaEventElapsedTime(&ms, a, b);
  cudaEventDestroy(a);
  if (b) cudaEventDestroy(b);
  if (rc) return rc;
  SHF_CK(e);
  *us = 1000.f * ms / static_cast<float>(iters);
  return SHF_OK;
}

// Candidate plans around the current one, for coordinate-wise search: stage 0
// varies the first parameter, stage 1 the second, stage 2 the third, each
// around the best found so far.
std::vector<seg_plan> plan_candidates(const seg_state* st, const seg_plan& base, int stage) {
  std::vector<seg_plan> out;
  const Geo& g = st->g;
  if (st->fast) {
    if (stage == 0) {
      // wave budgets that give distinct waves (filters per wave of one label,
      // or labels per wave)
      std::vector<int> seen;
      for (int mib : {16, 32, 64, 96, 128, 192, 256, 384, 512, 1024}) {
        const int w = shf::fast_wave(g, mib), nl = shf::fast_wave_labels(g, mib, st->K);
        const int sig = nl > 1 ? -nl : (g.eta + w - 1) / w;
        if (std::find(seen.begin(), seen.end(), sig) != seen.end()) continue;
        seen.push_back(sig);
        seg_plan p = base;
        p.wave_mib = mib;
        out.push_back(p);
      }
    } else if (stage == 2) {
      // the FFT kernel of the forward v-step: 8 or 16 values per thread, one
      // row or a pair of rows per group, or 12 / 20 / 32 values per thread
      // (odd factor 3 or 5, or 1024 = 32 x 32); each with the iteration's
      // launches overlapped (programmatic dependent launch) and serial
      for (int rk : {shf::kRow8, shf::kRow16, shf::kRowPair, shf::kRowV}) {
        if (!shf::fast_row_kernel_ok(g, rk)) continue;
        for (int serial : {0, 1}) {  // with and without programmatic dependent launch
          seg_plan p = base;
          p.row_kernel = rk;
          p.serial = serial;
          out.push_back(p);
        }
      }
    } else if (stage == 3) {
      // the FFT kernel of the fan and the gather: 8 or 16 values per thread
      for (int ck : {shf::kCol8, shf::kCol16, shf::kColV}) {
        if (!shf::fast_col_kernel_ok(g, ck)) continue;
        seg_plan p = base;
        p.col_kernel = ck;
        out.push_back(p);
      }
    } else if (stage == 1) {
      // resident column CTAs per SM: every count up to what fits (0 = all)
      const int fit = shf::fast_col_ctas(g, 0, base.col_kernel) / std::max(1, shf::fast_col_ctas(g, 1, base.col_kernel));
      for (int c = 1; c < fit; ++c) {
        seg_plan p = base;
        p.col_ctas_per_sm = c;
        out.push_back(p);
      }
      seg_plan p = base;
      p.col_ctas_per_sm = 0;
      out.push_back(p);
    }
    return out;
  }
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return out;
  if (stage == 0) {
    std::vector<int> seen;
    for (int G : {base.groups / 2, base.groups, 2 * base.groups, 4 * base.groups}) {
      const int n = normalise_groups(g.eta, G);
      if (std::find(seen.begin(), seen.end(), n) != seen.end()) continue;
      seen.push_back(n);
      seg_plan p = base;
      p.groups = n;
      out.push_back(p);
    }
  } else if (stage == 1 || stage == 2) {
    const int vals1[] = {4, 8, 16, 32};
    const int vals2[] = {base.tile_rows / 2, base.tile_rows, 2 * base.tile_rows};
    const int* vals = stage == 1 ? vals1 : vals2;
    const int nv = stage == 1 ? 4 : 3;
    for (int i = 0; i < nv; ++i) {
      seg_plan p = base;
      (stage == 1 ? p.tile_cols : p.tile_rows) = vals[i];
      Geo t = g;
      if (!shf::set_generic_tiles(&t, p.tile_cols, p.tile_rows, st->K, optin)) continue;
      out.push_back(p);
    }
  }
  return out;
}

// A copy of a state's iterate (b_v, w, b_w, u and the u-spectra) and
// iteration count, taken on the state's stream before trial iterations and
// put back after them.
struct IterateCopy {
  seg_state* st = nullptr;
  float* buf = nullptr;
  long long iter0 = 0;

  // SHF_ERR_OOM when there is no memory for the copy
  int save(seg_state* s) {
    st = s;
    iter0 = s->iter;
    const size_t KP = s->P() * s->K, NC = KP * s->g.eta, TH = s->Ph() * s->K;
    if (cudaMallocAsync(reinterpret_cast<void**>(&buf), sizeof(float) * (NC + 3 * KP + 2 * TH), s->stream) !=
        cudaSuccess) {
      cudaGetLastError();
      buf = nullptr;
      return fail(SHF_ERR_OOM, "no memory to save the iterate for the tuning trials");
    }
    return copy(true) == cudaSuccess ? SHF_OK : fail(SHF_ERR_CUDA, "saving the iterate failed");
  }
  // copies the iterate back, frees the copy and synchronises the stream
  cudaError_t restore() {
    if (!buf) return cudaSuccess;
    cudaError_t e = copy(false);
    cudaError_t e2 = cudaFreeAsync(buf, st->stream);
    cudaError_t e3 = cudaStreamSynchronize(st->stream);
    buf = nullptr;
    st->iter = iter0;
    return e != cudaSuccess ? e : (e2 != cudaSuccess ? e2 : e3);
  }

 private:
  cudaError_t copy(bool save) {
    const size_t KP = st->P() * st->K, NC = KP * st->g.eta, TH = st->Ph() * st->K;
    struct Piece {
      void* p;
      size_t bytes;
    };
    const Piece pieces[] = {{st->bv, sizeof(float) * NC},
                            {st->w, sizeof(float) * KP},
                            {st->bw, sizeof(float) * KP},
                            {st->u, sizeof(float) * KP},
                            {st->T, sizeof(float2) * TH}};
    char* q = reinterpret_cast<char*>(buf);
    cudaError_t e = cudaSuccess;
    for (const Piece& pc : pieces) {
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(save ? q : pc.p, save ? pc.p : q, pc.bytes, cudaMemcpyDeviceToDevice, st->stream);
      q += pc.bytes;
    }
    return e;
  }
};

}  // namespace

extern "C" {

int seg_admm_tune(seg_state* st, int iters, seg_plan* best_out) {
  if (!st || iters < 1) return fail(SHF_ERR_ARG, "seg_admm_tune: bad argument");
  // the iterate is saved and restored around the trial iterations
  IterateCopy snap;
  int rc0 = snap.save(st);
  if (rc0) {
    snap.restore();
    return rc0;
  }
  seg_plan best;
  seg_admm_get_plan(st, &best);
  best.us_per_iter = INFINITY;
  int rc = SHF_OK;
  for (int stage = 0; stage < 4 && !rc; ++stage) {
    const seg_plan base = best;
    for (const seg_plan& cand : plan_candidates(st, base, stage)) {
      int r = seg_admm_set_plan(st, &cand);
      if (r == SHF_ERR_OOM || r == SHF_ERR_ARG) continue;  // not feasible here: skip
      if (r) {
        rc = r;
        break;
      }
      // the better of two timings: plans a few percent apart must not swap
      // places on one noisy trial
      float us = 0.f, us2 = 0.f;
      r = time_iterations(st, iters, &us);
      if (!r) r = time_iterations(st, iters, &us2);
      if (r) {
        rc = r;
        break;
      }
      us = std::min(us, us2);
      if (us < best.us_per_iter) {
        best = cand;
        best.us_per_iter = us;
      }
    }
  }
  if (!rc) rc = seg_admm_set_plan(st, &best);
  const cudaError_t e = snap.restore();
  if (rc) return rc;
  if (e != cudaSuccess) return fail(SHF_ERR_CUDA, "seg_admm_tune: restoring the iterate failed");
  if (best_out) *best_out = best;
  return SHF_OK;
}

int seg_admm_solve(seg_state* st, int* iters_done, float* final_residual) {
  if (!st) return fail(SHF_ERR_ARG, "state is NULL");
  double res = INFINITY;
  int done = 0;
  while (done < st->max_iters) {
    const int n = std::min(st->check_every, st->max_iters - done);
    int rc = seg_admm_step(st, n);
    if (rc) return rc;
    done += n;
    rc = residual_uw(st, &res);
    if (rc) return rc;
    if (res < st->tol) break;
  }
  if (iters_done) *iters_done = done;
  if (final_residual) *final_residual = static_cast<float>(res);
  return SHF_OK;
}

}  // extern "C"

namespace {

// An image of a batch: what a call left on the image's stream has ended before the
// batch's next iterations, which run as a graph on the batch's.
int settled(seg_state* st, int rc) {
  if (!rc && st->batch) SHF_CK(cudaStreamSynchronize(st->stream));
  return rc;
}

int get_component(seg_state* st, int what, void* dst, int on_host) {
  const Geo& g = st->g;
  const size_t P = st->P(), KP = P * st->K;
  switch (what) {
    case SEG_U: return copy_out(st, dst, st->u, sizeof(float) * KP, on_host);
    case SEG_W: return copy_out(st, dst, st->w, sizeof(float) * KP, on_host);
    case SEG_BW: return copy_out(st, dst, st->bw, sizeof(float) * KP, on_host);
    case SEG_BV: return copy_out(st, dst, st->bv, sizeof(float) * KP * g.eta, on_host);
    case SEG_S: return copy_out(st, dst, st->s, sizeof(float) * KP, on_host);
    case SEG_STV:
      SHF_CK(shf::run_row_c2r(g, st->T, st->stv, st->K, 1.f / (static_cast<float>(g.H) * g.W), st->stream));
      return copy_out(st, dst, st->stv, sizeof(float) * KP, on_host);
    case SEG_LABELS:
    case SEG_GAP:
      SHF_CK(shf::launch_labels(st->w, st->K, static_cast<int>(P), st->labels, st->gap, st->stream));
      if (what == SEG_LABELS) return copy_out(st, dst, st->labels, sizeof(int) * P, on_host);
      return copy_out(st, dst, st->gap, sizeof(float) * P, on_host);
    case SEG_ENERGY: {
      double e = 0;
      int rc = energy_of_w(st, &e);
      if (rc) return rc;
      if (on_host) {
        *static_cast<double*>(dst) = e;
        return SHF_OK;
      }
      SHF_CK(cudaMemcpy(dst, &e, sizeof(double), cudaMemcpyHostToDevice));
      return SHF_OK;
    }
    case SEG_ITER:
      if (!on_host) return fail(SHF_ERR_ARG, "SEG_ITER is host only");
      *static_cast<int*>(dst) = static_cast<int>(st->iter);
      return SHF_OK;
    default: return fail(SHF_ERR_ARG, "unknown selector");
  }
}

int set_component(seg_state* st, int what, const void* src, int on_host) {
  const Geo& g = st->g;
  const size_t P = st->P(), KP = P * st->K;
  switch (what) {
    case SEG_W: return copy_in(st, st->w, src, sizeof(float) * KP, on_host);
    case SEG_BW: return copy_in(st, st->bw, src, sizeof(float) * KP, on_host);
    case SEG_BV: return copy_in(st, st->bv, src, sizeof(float) * KP * g.eta, on_host);
    case SEG_STV: {
      int rc = copy_in(st, st->stv, src, sizeof(float) * KP, on_host);
      if (rc) return rc;
      // T = H * row-forward(stv), so that the u-step's 1/(HW) row-inverse returns stv.
      SHF_CK(shf::run_row_r2c(g, st->stv, st->T, st->K, static_cast<float>(g.H), st->stream));
      return SHF_OK;
    }
    case SEG_V: {
      float* d = nullptr;
      SHF_CK(cudaMallocAsync(reinterpret_cast<void**>(&d), sizeof(float) * KP * g.eta, st->stream));
      cudaError_t e = cudaMemcpyAsync(d, src, sizeof(float) * KP * g.eta,
                                      on_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st->stream);
      if (e == cudaSuccess) e = shf::launch_sub(d, st->bv, d, static_cast<long>(KP * g.eta), st->stream);
      if (e == cudaSuccess) e = synthesis_spectrum(st->bank, g, d, st->K, st->T, st->stream);
      cudaError_t e2 = cudaFreeAsync(d, st->stream);
      if (e == cudaSuccess) e = e2;
      if (e == cudaSuccess && on_host) e = cudaStreamSynchronize(st->stream);
      if (e != cudaSuccess) return fail(SHF_ERR_CUDA, std::string("seg_admm_set(SEG_V): ") + cudaGetErrorString(e));
      return SHF_OK;
    }
    default: return fail(SHF_ERR_ARG, "selector cannot be set");
  }
}

}  // namespace

extern "C" {

int seg_admm_get(seg_state* st, int what, void* dst, int on_host) {
  if (!st || !dst) return fail(SHF_ERR_ARG, "seg_admm_get: NULL argument");
  return settled(st, get_component(st, what, dst, on_host));
}

int seg_admm_read(seg_state* st, int what, void* dst, void* earlier) {
  if (!st || !dst) return fail(SHF_ERR_ARG, "seg_admm_read: NULL argument");
  SHF_CK(shf::order_after(st->stream, static_cast<cudaStream_t>(earlier)));
  const int rc = get_component(st, what, dst, 0);
  return rc ? rc : seg_admm_sync(st);
}

int seg_admm_set(seg_state* st, int what, const void* src, int on_host) {
  if (!st || !src) return fail(SHF_ERR_ARG, "seg_admm_set: NULL argument");
  return settled(st, set_component(st, what, src, on_host));
}

namespace {
struct CkptHeader {
  char magic[8];
  int32_t H, W, K, J, eta, C;
  int64_t iter;
  float gamma;
  float Lambda[shf::kMaxJ + 1];
};
}  // namespace

int seg_admm_save(seg_state* st, const char* path) {
  if (!st || !path) return fail(SHF_ERR_ARG, "seg_admm_save: NULL argument");
  const Geo& g = st->g;
  const size_t KP = st->P() * st->K;
  CkptHeader h{};
  std::memcpy(h.magic, "SHFCKPT1", 8);
  h.H = g.H;
  h.W = g.W;
  h.K = st->K;
  h.J = g.J;
  h.eta = g.eta;
  h.C = st->C;
  h.iter = st->iter;
  h.gamma = st->gamma;
  for (int j = 0; j <= g.J; ++j) h.Lambda[j] = st->Lambda[j];
  std::vector<float> buf(KP * g.eta);
  FILE* fp = std::fopen(path, "wb");
  if (!fp) return fail(SHF_ERR_IO, std::string("cannot open ") + path);
  bool ok = std::fwrite(&h, sizeof(h), 1, fp) == 1;
  // the carried synthesis spectrum T, raw, so that a resumed run continues bit for bit
  const size_t nT = 2 * st->Ph() * st->K;
  std::vector<float> tbuf(nT);
  int rc0 = copy_out(st, tbuf.data(), st->T, sizeof(float) * nT, 1);
  if (rc0) {
    std::fclose(fp);
    return rc0;
  }
  ok = ok && std::fwrite(tbuf.data(), sizeof(float), nT, fp) == nT;
  const int parts[] = {SEG_BV, SEG_W, SEG_BW, SEG_S, SEG_U};
  for (int what : parts) {
    const size_t n = what == SEG_BV ? KP * g.eta : KP;
    int rc = seg_admm_get(st, what, buf.data(), 1);
    if (rc) {
      std::fclose(fp);
      return rc;
    }
    ok = ok && std::fwrite(buf.data(), sizeof(float), n, fp) == n;
  }
  ok = (std::fclose(fp) == 0) && ok;
  return ok ? SHF_OK : fail(SHF_ERR_IO, std::string("write failed: ") + path);
}

int seg_admm_load(seg_state* st, const char* path) {
  if (!st || !path) return fail(SHF_ERR_ARG, "seg_admm_load: NULL argument");
  const Geo& g = st->g;
  const size_t KP = st->P() * st->K;
  FILE* fp = std::fopen(path, "rb");
  if (!fp) return fail(SHF_ERR_IO, std::string("cannot open ") + path);
  CkptHeader h{};
  if (std::fread(&h, sizeof(h), 1, fp) != 1 || std::memcmp(h.magic, "SHFCKPT1", 8) != 0) {
    std::fclose(fp);
    return fail(SHF_ERR_IO, "not a checkpoint file");
  }
  if (h.H != g.H || h.W != g.W || h.K != st->K || h.J != g.J) {
    std::fclose(fp);
    return fail(SHF_ERR_STATE, "checkpoint sizes differ from the state's");
  }
  std::vector<float> buf(KP * g.eta);
  const size_t nT = 2 * st->Ph() * st->K;
  std::vector<float> tbuf(nT);
  if (std::fread(tbuf.data(), sizeof(float), nT, fp) != nT) {
    std::fclose(fp);
    return fail(SHF_ERR_IO, "truncated checkpoint");
  }
  int rc0 = copy_in(st, st->T, tbuf.data(), sizeof(float) * nT, 1);
  if (rc0) {
    std::fclose(fp);
    return rc0;
  }
  const int parts[] = {SEG_BV, SEG_W, SEG_BW};
  for (int what : parts) {
    const size_t n = what == SEG_BV ? KP * g.eta : KP;
    if (std::fread(buf.data(), sizeof(float), n, fp) != n) {
      std::fclose(fp);
      return fail(SHF_ERR_IO, "truncated checkpoint");
    }
    int rc = seg_admm_set(st, what, buf.data(), 1);
    if (rc) {
      std::fclose(fp);
      return rc;
    }
  }
  // s and u
  for (float* dstp : {st->s, st->u}) {
    if (std::fread(buf.data(), sizeof(float), KP, fp) != KP) {
      std::fclose(fp);
      return fail(SHF_ERR_IO, "truncated checkpoint");
    }
    int rc = copy_in(st, dstp, buf.data(), sizeof(float) * KP, 1);
    if (rc) {
      std::fclose(fp);
      return rc;
    }
  }
  std::fclose(fp);
  st->iter = h.iter;
  return SHF_OK;
}

}  // extern "C"

namespace {

// Layout of the reverse sweep's temporaries in st->un_mem (byte offsets, each
// region on a 256-byte boundary: the fast kernels copy rows of bvbar and of
// the codes with 16-byte asynchronous copies).
struct UnLayout {
  size_t tpart, tbar, cbpart, cbout;      // doubles
  size_t Uw, Tt;                          // float2 [K][H][Wh]
  size_t bvbar, dbar, Qbar, wbar, bwbar, sbar, gwbar, stv, fbar, grec, wrec;  // floats
  size_t code;                            // bytes
  size_t total;
};

UnLayout un_layout(const seg_state* st, int ck) {
  const Geo& g = st->g;
  const int K = st->K, C = st->C, eta = g.eta;
  const size_t P = st->P(), Ph = st->Ph(), KP = P * K, NC = KP * eta;
  const bool fast = st->fast;
  const size_t nblk = static_cast<size_t>(shf::adj_part_blocks());
  UnLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = (off + bytes + 255) & ~static_cast<size_t>(255);
    return at;
  };
  L.tpart = take(sizeof(double) * K * eta * (fast ? static_cast<size_t>(g.H) : nblk));
  L.tbar = take(sizeof(double) * eta);
  L.cbpart = take(sizeof(double) * K * C * nblk);
  L.cbout = take(sizeof(double) * K * C);
  L.Uw = take(sizeof(float2) * Ph * K);
  L.Tt = take(sizeof(float2) * Ph * K);
  L.bvbar = take(sizeof(float) * NC);
  L.dbar = fast ? 0 : take(sizeof(float) * NC);
  L.Qbar = take(sizeof(float) * KP);
  L.wbar = take(sizeof(float) * KP);
  L.bwbar = take(sizeof(float) * KP);
  L.sbar = take(sizeof(float) * KP);
  L.gwbar = take(sizeof(float) * KP);
  L.stv = take(sizeof(float) * KP);
  L.fbar = take(sizeof(float) * P * C);
  L.grec = fast ? 0 : take(sizeof(float) * NC * ck);
  L.wrec = take(sizeof(float) * KP * ck);
  L.code = fast ? take(NC * ck) : 0;
  L.total = off;
  return L;
}

// T iterations from the zero state, keeping (b_v, w, b_w, T) before every
// ckpt-th iteration.
cudaError_t enqueue_unrolled_fwd(seg_state* st, int T, int ck) {
  const size_t P = st->P(), Ph = st->Ph(), KP = P * st->K, NC = KP * st->g.eta;
  cudaStream_t s = st->stream;
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
  };
  ok(cudaMemsetAsync(st->bv, 0, sizeof(float) * NC, s));
  ok(cudaMemsetAsync(st->w, 0, sizeof(float) * KP, s));
  ok(cudaMemsetAsync(st->bw, 0, sizeof(float) * KP, s));
  ok(cudaMemsetAsync(st->u, 0, sizeof(float) * KP, s));
  ok(cudaMemsetAsync(st->T, 0, sizeof(float2) * Ph * st->K, s));
  for (int i = 0; i < T && e == cudaSuccess; ++i) {
    if (i % ck == 0) {
      const int c = i / ck;
      ok(cudaMemcpyAsync(st->ck_bv[c], st->bv, sizeof(float) * NC, cudaMemcpyDeviceToDevice, s));
      ok(cudaMemcpyAsync(st->ck_w[c], st->w, sizeof(float) * KP, cudaMemcpyDeviceToDevice, s));
      ok(cudaMemcpyAsync(st->ck_bw[c], st->bw, sizeof(float) * KP, cudaMemcpyDeviceToDevice, s));
      ok(cudaMemcpyAsync(st->ck_T[c], st->T, sizeof(float2) * Ph * st->K, cudaMemcpyDeviceToDevice, s));
    }
    ok(st->fast ? enqueue_iteration(st, false) : enqueue_generic_iteration(st, nullptr));
  }
  return e;
}

// The reverse sweep, from wbar (already holding dL/dw) to sbar, fbar, tbar
// and cbout in st->un_mem.
cudaError_t enqueue_unrolled_bwd(seg_state* st, const UnLayout& U) {
  const Geo& g = st->g;
  const int K = st->K, C = st->C, eta = g.eta, T = st->un_T, ck = st->un_ck;
  const size_t P = st->P(), Ph = st->Ph(), KP = P * K, NC = KP * eta;
  const float scale = 1.f / (static_cast<float>(g.H) * g.W);
  cudaStream_t s = st->stream;
  const bool fast = st->fast;
  char* m = st->un_mem;
  double* tpart = reinterpret_cast<double*>(m + U.tpart);
  double* tbar = reinterpret_cast<double*>(m + U.tbar);
  double* cbpart = reinterpret_cast<double*>(m + U.cbpart);
  double* cbout = reinterpret_cast<double*>(m + U.cbout);
  float2* Uw = reinterpret_cast<float2*>(m + U.Uw);
  float2* Tt = reinterpret_cast<float2*>(m + U.Tt);
  auto F = [&](size_t o) { return reinterpret_cast<float*>(m + o); };
  float *bvbar = F(U.bvbar), *dbar = fast ? nullptr : F(U.dbar), *Qbar = F(U.Qbar), *wbar = F(U.wbar),
        *bwbar = F(U.bwbar), *sbar = F(U.sbar), *gwbar = F(U.gwbar), *stv = F(U.stv), *fbar = F(U.fbar),
        *grec = fast ? nullptr : F(U.grec), *wrec = F(U.wrec);
  signed char* crec = fast ? reinterpret_cast<signed char*>(m + U.code) : nullptr;
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
    return e == cudaSuccess;
  };
  ok(cudaMemsetAsync(bvbar, 0, sizeof(float) * NC, s));
  ok(cudaMemsetAsync(Qbar, 0, sizeof(float) * KP, s));
  ok(cudaMemsetAsync(bwbar, 0, sizeof(float) * KP, s));
  ok(cudaMemsetAsync(sbar, 0, sizeof(float) * KP, s));
  ok(cudaMemsetAsync(tbar, 0, sizeof(double) * eta, s));
  const int nseg = (T + ck - 1) / ck;
  for (int seg = nseg - 1; seg >= 0 && e == cudaSuccess; --seg) {
    const int n = std::min(ck, T - seg * ck);
    ok(cudaMemcpyAsync(st->bv, st->ck_bv[seg], sizeof(float) * NC, cudaMemcpyDeviceToDevice, s));
    ok(cudaMemcpyAsync(st->w, st->ck_w[seg], sizeof(float) * KP, cudaMemcpyDeviceToDevice, s));
    ok(cudaMemcpyAsync(st->bw, st->ck_bw[seg], sizeof(float) * KP, cudaMemcpyDeviceToDevice, s));
    ok(cudaMemcpyAsync(st->T, st->ck_T[seg], sizeof(float2) * Ph * K, cudaMemcpyDeviceToDevice, s));
    for (int i = 0; i < n && e == cudaSuccess; ++i) {  // recompute the segment, recording g (or its codes) and w'
      if (fast)
        ok(enqueue_iteration(st, false, crec + static_cast<size_t>(i) * NC));
      else
        ok(enqueue_generic_iteration(st, grec + static_cast<size_t>(i) * NC));
      ok(cudaMemcpyAsync(wrec + static_cast<size_t>(i) * KP, st->w, sizeof(float) * KP, cudaMemcpyDeviceToDevice, s));
    }
    for (int i = n - 1; i >= 0 && e == cudaSuccess; --i) {
      ok(shf::launch_adj_proj(wrec + static_cast<size_t>(i) * KP, wbar, bwbar, gwbar, K, static_cast<int>(P), s));
      if (fast) {
        // S Qbar, the v-step adjoint and S^T bvbar, fused per wave of filters
        ok(shf::run_row_r2c(g, Qbar, Uw, K, 1.f, s));
        ok(shf::run_fast_adjoint_body(g, st->plan, Uw, st->uhat, st->Y, bvbar, st->thr, st->partial, Tt, K, scale,
                                      crec + static_cast<size_t>(i) * NC, tpart, s));
        ok(shf::launch_adj_tsum_rows(tpart, K, eta, g.H, tbar, s));
      } else {
        // dbar = S Qbar
        ok(shf::run_row_r2c(g, Qbar, Uw, K, 1.f, s));
        ok(shf::run_col_fwd(g, Uw, K, s));
        for (const shf::FilterWave& wv : st->un_waves) {
          ok(shf::run_wave_fan(g, Uw, st->un_Y, wv, s));
          ok(shf::run_wave_c2r(g, st->un_Y, dbar, wv, scale, s));
        }
        ok(shf::launch_adj_shrink(grec + static_cast<size_t>(i) * NC, dbar, bvbar, st->thr, K, eta,
                                  static_cast<long>(P), tpart, tbar, s));
        // stv = S^T bvbar
        for (const shf::FilterWave& wv : st->un_waves) {
          ok(shf::run_wave_r2c(g, bvbar, st->un_Y, wv, s));
          ok(shf::run_wave_gather(g, st->un_Y, st->un_partial, K, st->un_groups, wv, s));
        }
        ok(shf::run_col_reduce_inv(g, st->un_partial, Tt, K, st->un_groups, s));
      }
      ok(shf::run_row_c2r(g, Tt, stv, K, scale, s));
      ok(shf::launch_adj_u(gwbar, stv, Qbar, wbar, bwbar, sbar, st->gamma, static_cast<long>(KP), s));
    }
  }
  ok(shf::adj_codebook(sbar, st->f, st->codebook.data(), K, C, static_cast<long>(P), cbpart, cbout, fbar, s));
  return e;
}

// The general path's sweep plans, their tables and scratch; the state has them all
// or, after a failure, none.
int make_sweep_scratch(seg_state* st) {
  const Geo& g = st->g;
  const size_t Ph = st->Ph();
  // filter groups for four CTAs per SM over all labels, unless the plan says otherwise
  int groups = st->groups;
  if (groups == shf::default_groups(g, st->K)) {
    const int base = g.ntiles * st->K;
    groups = normalise_groups(g.eta, (4 * 152 + base - 1) / base);
  }
  Geo sg = g;
  sg.staged = 1;
  if (!shf::make_sweep_plan(g.H, &sg.planH) || !shf::make_sweep_plan(g.L, &sg.planL))
    return fail(SHF_ERR_SIZE, "unsupported geometry");
  sg.planLr = sg.planL;
  std::vector<shf::FilterWave> waves = shf::general_waves(g, st->K, groups);
  float2 *pt = nullptr, *Y = nullptr, *partial = nullptr;
  int rc;
  if (!(rc = state_alloc(st, &pt, shf::pass_table_entries(sg), "pass tables")) &&
      !(rc = state_alloc(st, &Y, shf::wave_planes(waves) * g.H * g.Wy, "unrolled scratch")) &&
      !(rc = state_alloc(st, &partial, Ph * st->K * static_cast<size_t>(groups), "unrolled partials"))) {
    const cudaError_t e = shf::launch_pass_tables(&sg, pt, st->stream);
    if (e != cudaSuccess) rc = fail(SHF_ERR_CUDA, std::string("pass tables: ") + cudaGetErrorString(e));
  }
  if (rc) {
    state_free(st, pt);
    state_free(st, Y);
    state_free(st, partial);
    return rc;
  }
  st->un_g = sg;
  st->un_waves = std::move(waves);
  st->un_groups = groups;
  st->un_pt = pt;
  st->un_Y = Y;
  st->un_partial = partial;
  return SHF_OK;
}

}  // namespace

extern "C" {

int seg_admm_unrolled_fwd(seg_state* st, int T, int ckpt_every) {
  if (!st || T < 1 || ckpt_every < 1) return fail(SHF_ERR_ARG, "seg_admm_unrolled_fwd: bad argument");
  const Geo& g = st->g;
  const size_t P = st->P(), Ph = st->Ph(), KP = P * st->K, NC = KP * g.eta;
  int rc;
  // the fast path iterates with its plan's wave scratch; the general path has a
  // wave of its own (another number of filter groups, sweep plans)
  if (!st->fast && !st->un_Y && (rc = make_sweep_scratch(st))) return rc;
  const int nseg = (T + ckpt_every - 1) / ckpt_every;
  while (static_cast<int>(st->ck_bv.size()) < nseg) {
    float *bv = nullptr, *w = nullptr, *bw = nullptr;
    float2* Tt = nullptr;
    if ((rc = state_alloc(st, &bv, NC, "checkpoint")) || (rc = state_alloc(st, &w, KP, "checkpoint")) ||
        (rc = state_alloc(st, &bw, KP, "checkpoint")) || (rc = state_alloc(st, &Tt, Ph * st->K, "checkpoint"))) {
      state_free(st, bv);
      state_free(st, w);
      state_free(st, bw);
      state_free(st, Tt);
      return rc;
    }
    st->ck_bv.push_back(bv);
    st->ck_w.push_back(w);
    st->ck_bw.push_back(bw);
    st->ck_T.push_back(Tt);
  }
  // the first sweep of a (T, ckpt) is launched directly (a state made for one
  // training step never pays for a graph: capturing and instantiating takes the
  // host longer than launching), the second one captured, later ones replayed.
  // A forward and reverse pass in us, first / second / third, and with the capture
  // in the first: 64 x 64, K = 3, T = 10 1029 / 1266 / 811 (1652 / 895 / 887); 256 x
  // 256, K = 4, T = 10 2162 / 2153 / 1957 (3155 / 2142 / 2137), T = 50 9890 / 9933 /
  // 9232 (13554 / 10144 / 10137).  So the second pass of a small state can take
  // longer, but no number of passes does.
  const bool again = st->un_fwd_key[0] == T && st->un_fwd_key[1] == ckpt_every;
  if (!again && st->un_fwd_exec) {
    cudaGraphExecDestroy(st->un_fwd_exec);
    st->un_fwd_exec = nullptr;
  }
  if (again && !st->un_fwd_exec)
    st->un_fwd_exec = capture_work(st, [&]() { return enqueue_unrolled_fwd(st, T, ckpt_every); });
  st->un_fwd_key[0] = T;
  st->un_fwd_key[1] = ckpt_every;
  if (st->un_fwd_exec)
    SHF_CK(cudaGraphLaunch(st->un_fwd_exec, st->stream));
  else
    SHF_CK(enqueue_unrolled_fwd(st, T, ckpt_every));
  st->iter = T;
  st->un_T = T;
  st->un_ck = ckpt_every;
  return SHF_OK;
}

int seg_admm_unrolled_bwd_enqueue(seg_state* st, const float* dL_dw) {
  if (!st || !dL_dw) return fail(SHF_ERR_ARG, "seg_admm_unrolled_bwd_enqueue: NULL argument");
  if (st->un_T < 1) return fail(SHF_ERR_STATE, "seg_admm_unrolled_fwd has not run");
  const size_t KP = st->P() * st->K;
  cudaStream_t s = st->stream;
  const UnLayout U = un_layout(st, st->un_ck);
  if (st->un_mem_bytes < U.total) {
    SHF_CK(cudaStreamSynchronize(s));
    if (st->un_bwd_exec) cudaGraphExecDestroy(st->un_bwd_exec);
    st->un_bwd_exec = nullptr;
    state_free(st, st->un_mem);
    st->un_mem = nullptr;
    st->un_mem_bytes = 0;
    int rc = state_alloc(st, &st->un_mem, U.total, "reverse-sweep scratch");
    if (rc) return rc;
    st->un_mem_bytes = U.total;
  }
  SHF_CK(cudaMemcpyAsync(st->un_mem + U.wbar, dL_dw, sizeof(float) * KP, cudaMemcpyDeviceToDevice, s));
  // as the forward sweep: directly, then captured, then replayed
  const bool again = st->un_bwd_key[0] == st->un_T && st->un_bwd_key[1] == st->un_ck;
  if (!again && st->un_bwd_exec) {
    cudaGraphExecDestroy(st->un_bwd_exec);
    st->un_bwd_exec = nullptr;
  }
  if (again && !st->un_bwd_exec) st->un_bwd_exec = capture_work(st, [&]() { return enqueue_unrolled_bwd(st, U); });
  st->un_bwd_key[0] = st->un_T;
  st->un_bwd_key[1] = st->un_ck;
  SHF_CK(st->un_bwd_exec ? cudaGraphLaunch(st->un_bwd_exec, s) : enqueue_unrolled_bwd(st, U));
  st->un_bwd_pending = true;
  return SHF_OK;
}

int seg_admm_unrolled_grads(seg_state* st, float* dL_dcodebook, float* dL_dLambda, float* dL_df, float* dL_ds) {
  if (!st || !dL_dcodebook || !dL_dLambda) return fail(SHF_ERR_ARG, "seg_admm_unrolled_grads: NULL argument");
  if (!st->un_bwd_pending) return fail(SHF_ERR_STATE, "no reverse sweep has been enqueued");
  const Geo& g = st->g;
  const int K = st->K, C = st->C, eta = g.eta;
  const size_t P = st->P(), KP = P * K;
  cudaStream_t s = st->stream;
  const UnLayout U = un_layout(st, st->un_ck);
  char* m = st->un_mem;
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
  };
  if (dL_df) ok(cudaMemcpyAsync(dL_df, m + U.fbar, sizeof(float) * P * C, cudaMemcpyDeviceToDevice, s));
  if (dL_ds) ok(cudaMemcpyAsync(dL_ds, m + U.sbar, sizeof(float) * KP, cudaMemcpyDeviceToDevice, s));
  std::vector<double> th(eta), cb(static_cast<size_t>(K) * C);
  ok(cudaMemcpyAsync(th.data(), m + U.tbar, sizeof(double) * eta, cudaMemcpyDeviceToHost, s));
  ok(cudaMemcpyAsync(cb.data(), m + U.cbout, sizeof(double) * K * C, cudaMemcpyDeviceToHost, s));
  ok(cudaStreamSynchronize(s));
  if (e != cudaSuccess) return fail(SHF_ERR_CUDA, std::string("seg_admm_unrolled_grads: ") + cudaGetErrorString(e));
  std::vector<shf::FilterDesc> d(eta);
  shf::filter_descs(g.J, d.data());
  std::vector<double> lam(g.J + 1, 0.0);
  for (int f = 0; f < eta; ++f) lam[d[f].kind == 0 ? 0 : d[f].j + 1] += st->gamma * th[f];
  for (int j = 0; j <= g.J; ++j) dL_dLambda[j] = static_cast<float>(lam[j]);
  for (int i = 0; i < K * C; ++i) dL_dcodebook[i] = static_cast<float>(cb[i]);
  return SHF_OK;
}

int seg_admm_unrolled_bwd(seg_state* st, const float* dL_dw, float* dL_dcodebook, float* dL_dLambda, float* dL_df,
                          float* dL_ds) {
  if (!st || !dL_dw || !dL_dcodebook || !dL_dLambda) return fail(SHF_ERR_ARG, "seg_admm_unrolled_bwd: NULL argument");
  int rc = seg_admm_unrolled_bwd_enqueue(st, dL_dw);
  if (rc) return rc;
  return seg_admm_unrolled_grads(st, dL_dcodebook, dL_dLambda, dL_df, dL_ds);
}

int seg_admm_kernel_times(seg_state* st, float* ms, int* launches, int* nk) {
  if (!st || !ms) return fail(SHF_ERR_ARG, "seg_admm_kernel_times: NULL argument");
  if (st->iter == 0 || st->nmarks < 2) return fail(SHF_ERR_STATE, "no iteration has run yet");
  if (!st->marks_ok) return fail(SHF_ERR_STATE, "iteration has more launches than timing marks");
  for (int k = 0; k < shf::kNumKinds; ++k) {
    ms[k] = 0.f;
    if (launches) launches[k] = 0;
  }
  SHF_CK(cudaEventSynchronize(st->ev[st->nmarks - 1]));
  for (int i = 0; i + 1 < st->nmarks; ++i) {
    float t = 0.f;
    SHF_CK(cudaEventElapsedTime(&t, st->ev[i], st->ev[i + 1]));
    ms[st->kinds[i]] += t;
    if (launches) ++launches[st->kinds[i]];
  }
  if (nk) *nk = shf::kNumKinds;
  return SHF_OK;
}

const char* seg_admm_kernel_name(int i) {
  static const char* names[] = {"row_ustep", "col_fwd", "col_fan", "row_shrink", "col_gather", "col_reduce_inv"};
  return (i >= 0 && i < shf::kNumKinds) ? names[i] : "";
}

// ---------------------------------------------------------------------------
// Batches
// ---------------------------------------------------------------------------
}  // extern "C"

struct seg_batch {
  std::vector<shf_bank*> banks;
  std::vector<seg_state*> states;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  cudaEvent_t fork = nullptr;
  std::vector<cudaEvent_t> joins;
  cudaGraphExec_t exec = nullptr;
  bool graph_tried = false;
  int lanes = 0;  // chains of images run side by side (0: one image per chain)
};

namespace {

void drop_batch_graphs(seg_batch* b) {
  if (b->stream) cudaStreamSynchronize(b->stream);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  b->exec = nullptr;
  b->graph_tried = false;
}

int tune_batch_layout(seg_batch* b, int iters);

void free_batch(seg_batch* b) {
  if (b->stream) cudaStreamSynchronize(b->stream);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  b->exec = nullptr;
  for (seg_state* s : b->states)
    if (s) s->batch = nullptr;
  for (seg_state* s : b->states)
    if (s) seg_admm_destroy(s);
  for (shf_bank* k : b->banks)
    if (k) shfilters_destroy(k);
  if (b->fork) cudaEventDestroy(b->fork);
  for (cudaEvent_t e : b->joins)
    if (e) cudaEventDestroy(e);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
  delete b;
}

// Forks from the batch stream, enqueues one iteration of every image on its
// own stream and joins back.  With b->lanes = L in [1, n) the images form L
// chains that run side by side: in decreasing order of their work (H W K eta)
// each image joins the chain with the least work so far and starts after the
// chain's previous image; with 0 (or L >= n) every image is a chain of its own.
cudaError_t enqueue_batch_iteration(seg_batch* b) {
  const int n = static_cast<int>(b->states.size());
  const int nl = b->lanes > 0 && b->lanes < n ? b->lanes : n;
  auto work = [&](int i) {
    const seg_state* s = b->states[i];
    return static_cast<double>(s->P()) * s->K * s->g.eta;
  };
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  if (nl < n) std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return work(x) > work(y); });
  std::vector<double> load(nl, 0.0);
  std::vector<int> last(nl, -1);  // the chain's latest image
  cudaError_t e = cudaEventRecord(b->fork, b->stream);
  for (int k = 0; k < n && e == cudaSuccess; ++k) {
    const int i = order[k];
    int l = nl < n ? 0 : k;
    if (nl < n)
      for (int c = 1; c < nl; ++c)
        if (load[c] < load[l]) l = c;
    load[l] += work(i);
    seg_state* st = b->states[i];
    e = cudaStreamWaitEvent(st->stream, last[l] < 0 ? b->fork : b->joins[last[l]], 0);
    if (e == cudaSuccess) e = enqueue_iteration(st, false);
    if (e == cudaSuccess) e = cudaEventRecord(b->joins[i], st->stream);
    last[l] = i;
  }
  for (int l = 0; l < nl && e == cudaSuccess; ++l)
    if (last[l] >= 0) e = cudaStreamWaitEvent(b->stream, b->joins[last[l]], 0);
  return e;
}

}  // namespace

extern "C" {

int seg_admm_batch_init(int n, const int* H, const int* W, const int* C, const int* K, const float* const* f,
                        const float* const* codebooks, const seg_params* params, void* stream, seg_batch** out) {
  if (!out) return fail(SHF_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (n < 1 || !H || !W || !C || !K || !f || !codebooks || !params)
    return fail(SHF_ERR_ARG, "seg_admm_batch_init: bad argument");
  auto* b = new seg_batch();
  if (stream) {
    b->stream = static_cast<cudaStream_t>(stream);
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      delete b;
      return fail(SHF_ERR_CUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e));
    }
    b->own_stream = true;
  }
  cudaError_t e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    free_batch(b);
    return fail(SHF_ERR_CUDA, std::string("cudaEventCreate: ") + cudaGetErrorString(e));
  }
  b->joins.assign(n, nullptr);
  for (int i = 0; i < n; ++i) {
    e = cudaEventCreateWithFlags(&b->joins[i], cudaEventDisableTiming);
    if (e != cudaSuccess) {
      free_batch(b);
      return fail(SHF_ERR_CUDA, std::string("cudaEventCreate: ") + cudaGetErrorString(e));
    }
  }
  b->states.assign(n, nullptr);
  for (int i = 0; i < n; ++i) {
    shf_bank* bank = nullptr;
    for (shf_bank* k : b->banks)
      if (k->g.H == H[i] && k->g.W == W[i] && k->g.J == params[i].J) bank = k;
    if (!bank) {
      int rc = shfilters_build(H[i], W[i], params[i].J, b->stream, &bank);
      if (rc) {
        const std::string m = g_err;
        free_batch(b);
        return fail(rc, "image " + std::to_string(i) + ": " + m);
      }
      b->banks.push_back(bank);
    }
    int rc = seg_admm_init(bank, f[i], C[i], codebooks[i], K[i], &params[i], nullptr, &b->states[i]);
    if (rc) {
      const std::string m = g_err;
      free_batch(b);
      return fail(rc, "image " + std::to_string(i) + ": " + m);
    }
    b->states[i]->batch = b;
  }
  *out = b;
  return SHF_OK;
}

int seg_admm_batch_step(seg_batch* b, int n) {
  if (!b || n < 0) return fail(SHF_ERR_ARG, "seg_admm_batch_step: bad argument");
  if (n == 0) return SHF_OK;
  if (!b->graph_tried) {
    b->graph_tried = true;
    cudaGraph_t graph = nullptr;
    if (b->stream && cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
      cudaError_t e = enqueue_batch_iteration(b);
      cudaError_t e2 = cudaStreamEndCapture(b->stream, &graph);
      if (e == cudaSuccess && e2 == cudaSuccess && graph &&
          cudaGraphInstantiate(&b->exec, graph, 0) != cudaSuccess)
        b->exec = nullptr;
      if (graph) cudaGraphDestroy(graph);
    }
    cudaGetLastError();
  }
  for (int i = 0; i < n; ++i) {
    if (b->exec) {
      SHF_CK(cudaGraphLaunch(b->exec, b->stream));
    } else {
      SHF_CK(enqueue_batch_iteration(b));
    }
  }
  for (seg_state* st : b->states) st->iter += n;
  return SHF_OK;
}

int seg_admm_batch_set_lanes(seg_batch* b, int lanes) {
  if (!b || lanes < 0) return fail(SHF_ERR_ARG, "seg_admm_batch_set_lanes: bad argument");
  if (lanes != b->lanes) {
    b->lanes = lanes;
    drop_batch_graphs(b);
  }
  return SHF_OK;
}

int seg_admm_batch_get_lanes(const seg_batch* b, int* lanes) {
  if (!b || !lanes) return fail(SHF_ERR_ARG, "seg_admm_batch_get_lanes: NULL argument");
  *lanes = b->lanes;
  return SHF_OK;
}

int seg_admm_batch_image(seg_batch* b, int i, seg_state** out) {
  if (!b || !out || i < 0 || i >= static_cast<int>(b->states.size()))
    return fail(SHF_ERR_ARG, "seg_admm_batch_image: bad argument");
  *out = b->states[i];
  return SHF_OK;
}

}  // extern "C"

namespace {

// Mean time (microseconds) of one batch iteration over `iters` replays of the
// batch's graph, after one that also captures it.
int time_batch_iterations(seg_batch* b, int iters, float* us) {
  int rc = seg_admm_batch_step(b, 1);
  if (rc) return rc;
  cudaEvent_t a = nullptr, c = nullptr;
  SHF_CK(cudaEventCreate(&a));
  cudaError_t e = cudaEventCreate(&c);
  if (e == cudaSuccess) e = cudaEventRecord(a, b->stream);
  if (e == cudaSuccess) rc = seg_admm_batch_step(b, iters);
  if (e == cudaSuccess && !rc) e = cudaEventRecord(c, b->stream);
  if (e == cudaSuccess && !rc) e = cudaEventSynchronize(c);
  float ms = 0.f;
  if (e == cudaSuccess && !rc) e = cudaEventElapsedTime(&ms, a, c);
  cudaEventDestroy(a);
  if (c) cudaEventDestroy(c);
  if (rc) return rc;
  SHF_CK(e);
  *us = 1000.f * ms / static_cast<float>(iters);
  return SHF_OK;
}

// The fast images' fan, v-step and gather grids sized for `sms` SMs (0: all).
int set_batch_share(seg_batch* b, int sms) {
  for (seg_state* st : b->states) {
    if (!st->fast) continue;
    seg_plan p;
    seg_admm_get_plan(st, &p);
    p.sms = sms;
    const int rc = seg_admm_set_plan(st, &p);
    if (rc) return rc;
  }
  return SHF_OK;
}

// Batch-wide stages of the tuner, timed on the batch's graph (each candidate
// twice, the better time kept; the iterates saved before and restored after,
// or the stages skipped without memory for the copies): first the number of
// image chains (one image per chain, or 1 to 4 chains), then every fast
// image's persistent grids sized for all SMs or for a half, a third or a
// quarter of them.
int tune_batch_layout(seg_batch* b, int iters) {
  const int n = static_cast<int>(b->states.size());
  if (n < 2) return SHF_OK;
  int nfast = 0;
  for (seg_state* st : b->states) nfast += st->fast ? 1 : 0;
  int dev = 0, nsm = 0;
  SHF_CK(cudaGetDevice(&dev));
  SHF_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  std::vector<IterateCopy> snaps(b->states.size());
  int rc = SHF_OK;
  for (size_t i = 0; i < b->states.size() && !rc; ++i) rc = snaps[i].save(b->states[i]);
  for (seg_state* st : b->states) cudaStreamSynchronize(st->stream);  // copies before the batch's streams
  auto timed = [&](float* best_us) {
    float us = INFINITY;
    for (int t = 0; t < 2 && !rc; ++t) {
      float u = 0.f;
      rc = time_batch_iterations(b, iters, &u);
      us = std::min(us, u);
    }
    const bool better = !rc && us < *best_us;
    if (better) *best_us = us;
    return better;
  };
  int best_lanes = b->lanes, best_share = 0;
  if (!rc) {
    float best_us = INFINITY;
    for (int lanes : {0, 1, 2, 3, 4}) {
      if (lanes >= n) continue;
      b->lanes = lanes;
      drop_batch_graphs(b);
      if (timed(&best_us)) best_lanes = lanes;
      if (rc) break;
    }
    b->lanes = best_lanes;
    drop_batch_graphs(b);
    best_us = INFINITY;
    for (int share : {0, nsm / 2, nsm / 3, nsm / 4}) {
      if (rc || nfast == 0 || (share > 0 && share < 8)) continue;
      rc = set_batch_share(b, share);
      if (!rc && timed(&best_us)) best_share = share;
    }
  }
  const bool skipped = rc == SHF_ERR_OOM;
  if (skipped) rc = SHF_OK;
  b->lanes = best_lanes;
  drop_batch_graphs(b);
  if (!rc) rc = set_batch_share(b, best_share);
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (IterateCopy& sn : snaps)
    if (sn.restore() != cudaSuccess && !rc) rc = fail(SHF_ERR_CUDA, "seg_admm_batch_tune: restoring an iterate failed");
  return rc;
}

}  // namespace

extern "C" {

int seg_admm_batch_tune(seg_batch* b, int iters) {
  if (!b || iters < 1) return fail(SHF_ERR_ARG, "seg_admm_batch_tune: bad argument");
  // the images' iterates are saved on their own streams: the batch's iterations end first
  SHF_CK(cudaStreamSynchronize(b->stream));
  // every image back on grids for all SMs before its shape is tuned alone
  for (seg_state* st : b->states) {
    if (!st->fast || st->plan.sms == 0) continue;
    seg_plan p;
    seg_admm_get_plan(st, &p);
    p.sms = 0;
    const int rc = seg_admm_set_plan(st, &p);
    if (rc) return rc;
  }
  // one tuning run per distinct problem shape; the other images take its plan
  struct Key {
    int fast, H, W, J, K;
    bool operator==(const Key& o) const {
      return fast == o.fast && H == o.H && W == o.W && J == o.J && K == o.K;
    }
  };
  std::vector<std::pair<Key, seg_plan>> done;
  for (seg_state* st : b->states) {
    const Key k{st->fast ? 1 : 0, st->g.H, st->g.W, st->g.J, st->K};
    auto it = std::find_if(done.begin(), done.end(), [&](const std::pair<Key, seg_plan>& d) { return d.first == k; });
    int rc;
    if (it == done.end()) {
      seg_plan p;
      rc = seg_admm_tune(st, iters, &p);
      if (!rc) done.emplace_back(k, p);
    } else {
      rc = seg_admm_set_plan(st, &it->second);
    }
    if (rc) return rc;
  }
  drop_batch_graphs(b);
  return tune_batch_layout(b, iters);
}

int seg_admm_batch_sync(seg_batch* b) {
  if (!b) return fail(SHF_ERR_ARG, "batch is NULL");
  SHF_CK(cudaStreamSynchronize(b->stream));
  return SHF_OK;
}

int seg_admm_batch_destroy(seg_batch* b) {
  if (!b) return SHF_OK;
  free_batch(b);
  return SHF_OK;
}

int seg_admm_sync(seg_state* st) {
  if (!st) return fail(SHF_ERR_ARG, "state is NULL");
  SHF_CK(cudaStreamSynchronize(st->stream));
  return SHF_OK;
}

int seg_admm_destroy(seg_state* st) {
  if (!st) return SHF_OK;
  cudaStreamSynchronize(st->stream);
  free_state(st);
  return SHF_OK;
}

}  // extern "C"
