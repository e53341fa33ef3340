// MSM entry points shared by all curves: window-width table (cost model and
// autotuner overrides), resident bases, and dispatch to the per-curve
// translation units (k_msm_bn254.cu, k_msm_bls12_381.cu).
#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>

#include "msm_host.cuh"

namespace ecc {

cudaError_t msm_points_bn254(uint32_t num, const uint64_t* offsets, const uint32_t* points,
                             const uint32_t* scalars, uint32_t* out, cudaStream_t st);
cudaError_t msm_points_bls12_381(uint32_t num, const uint64_t* offsets, const uint32_t* points,
                                 const uint32_t* scalars, uint32_t* out, cudaStream_t st);
cudaError_t msm_bases_bn254(void* bases, uint32_t num_vectors, const uint64_t* sizes,
                            const uint32_t* scalars,
                            uint32_t* out, cudaStream_t st);
cudaError_t msm_bases_bls12_381(void* bases, uint32_t num_vectors, const uint64_t* sizes,
                                const uint32_t* scalars,
                                uint32_t* out, cudaStream_t st);
cudaError_t points_to_mont(int curve, const uint32_t* in, uint64_t n, uint32_t* out, uint64_t phi,
                           cudaStream_t st);
cudaError_t bases_precompute_bn254(void* bases, int c, cudaStream_t st);
cudaError_t msm_points_dev_bn254(uint32_t num, uint64_t cap, const uint64_t* offsets, int c,
                                 const uint32_t* points, const uint32_t* scalars, uint32_t* out,
                                 cudaStream_t st);
cudaError_t msm_points_dev_bls12_381(uint32_t num, uint64_t cap, const uint64_t* offsets, int c,
                                     const uint32_t* points, const uint32_t* scalars, uint32_t* out,
                                     cudaStream_t st);
cudaError_t msm_bases_dev_bn254(void* bases, uint32_t num, uint64_t cap, const uint64_t* sizes, int c,
                                const uint32_t* scalars, uint32_t* out, cudaStream_t st);
cudaError_t msm_bases_dev_bls12_381(void* bases, uint32_t num, uint64_t cap, const uint64_t* sizes, int c,
                                    const uint32_t* scalars, uint32_t* out, cudaStream_t st);
cudaError_t bases_precompute_bls12_381(void* bases, int c, cudaStream_t st);

namespace {

std::mutex g_win_mu;
std::map<std::pair<int, int>, int> g_window_table;  // (curve, floor(log2 n)) -> c
std::map<std::pair<int, int>, int> g_chunk_table;   // (curve, floor(log2 n)) -> red_log

// Cost model, in products: 6 per (point, window) digit and 15 per bucket (of the
// affine form; the Jacobian form's 11 and 27 or more are in the same proportion);
// 100 (about 5 ns) for every digit in its way when the top window has only `top` bits
// and its points share 2^top buckets; and for a single call the latency of its tail,
// two steps of the reduction for each bit of c and one of the combination for each
// window (8 and 2.8 us with 8 limbs), which the instances of a batch share.  Batches of
// tiny MSMs are all buckets: 65536 BLS12-381 MSMs of 4 points take 38 ms with 2 bits and
// 58 with 4, 262144 of one point 100 and 161.
int model_window(int curve, uint64_t n, uint64_t num, bool split) {
  const int bits = split ? BN254::GLV_BITS : msm_detail::scalar_bits(curve);
  int best = 2;
  double best_cost = 1e300;
  for (int c = 2; c <= 20; ++c) {
    const double W = (bits + 1 + c - 1) / c, digits = (double)n * W * (split ? 2 : 1);
    const int top = bits - c * ((int)W - 1);
    double cost = digits * 6.0 + W * (double)(1u << (c - 1)) * 15.0;
    cost += digits / W / (double)(1u << std::max(top, 0)) * 100.0;
    cost += (150e3 * c + 59e3 * W) / (double)std::max<uint64_t>(num, 1);
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
  }
  return best;
}

// The same for the choice between split and whole scalars of an n-point BN254 MSM, from
// the phase times of both forms at 2^16 to 2^25 points and 13 to 20 bits: 20 a bucket; a
// tenth more for a digit of a split scalar past 2^21 points, where the points and their
// images no longer share the L2; for a digit of the top window what its bucket's x
// entries wait for each other in the sort, at most 12 (5 of a whole scalar: half as many
// meet); the doublings of the combination.
constexpr uint64_t kSplitPoints = 1u << 21;

double form_cost(uint64_t n, uint64_t num, int c, bool split) {
  const int bits = split ? BN254::GLV_BITS : BN254::SCALAR_BITS;
  const double W = (bits + 1 + c - 1) / c, top_digits = (double)n * (split ? 2 : 1);
  const int top = bits - c * ((int)W - 1);
  const double x = top_digits / (double)(1u << std::max(top, 0));
  double cost = top_digits * W * (split && n > kSplitPoints ? 6.6 : 6.0) + W * (double)(1u << (c - 1)) * 20.0;
  cost += top_digits * (split ? std::min(12.0, x / 128) : std::min(5.0, x / 256));
  return cost + (150e3 * c + 59e3 * W + 41.5e3 * bits) / (double)std::max<uint64_t>(num, 1);
}

int whole_window(uint64_t n, uint64_t num) {
  int best = 2;
  for (int c = 3; c <= 20; ++c)
    if (form_cost(n, num, c, false) < form_cost(n, num, best, false)) best = c;
  return best;
}

// The width by which sizes are admitted: whole scalars, 6 products per digit and 15
// per bucket.
int admitted_model(int curve, uint64_t n) {
  int best = 4;
  double best_cost = 1e300;
  for (int c = 4; c <= 20; ++c) {
    const double W = msm_detail::windows_for(curve, c);
    const double cost = (double)n * W * 6.0 + W * (double)(1u << (c - 1)) * 15.0;
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
  }
  return best;
}

int ilog2(uint64_t n) {
  int l = 0;
  while ((n >> 1) > 0) {
    n >>= 1;
    ++l;
  }
  return l;
}

}  // namespace

namespace {

// the caller's width for the size class of n (0: none)
int window_override(int curve, uint64_t n) {
  std::lock_guard<std::mutex> lock(g_win_mu);
  auto it = g_window_table.find({curve, ilog2(n)});
  return it != g_window_table.end() ? it->second : 0;
}

}  // namespace

int msm_window(int curve, uint64_t n, uint64_t num, bool split) {
  if (n < 2) n = 2;
  const int c = window_override(curve, n);
  if (c > 0) return c;
  return curve == 2 && !split ? whole_window(n, num) : model_window(curve, n, num, split);
}

double msm_split_gain(uint64_t n, uint64_t num, int c) {
  if (n < 2) n = 2;
  if (c <= 0) c = window_override(2, n);
  if (c > 0) return form_cost(n, num, c, false) - form_cost(n, num, c, true);
  const double gain = form_cost(n, num, whole_window(n, num), false) -
                      form_cost(n, num, model_window(2, n, num, true), true);
  return n <= kSplitPoints ? std::max(gain, 0.0) : gain;
}

int msm_admitted_window(int curve, uint64_t n) {
  if (n < 2) n = 2;
  const int c = window_override(curve, n);
  return c > 0 ? c : admitted_model(curve, n);
}

void msm_set_window(int curve, int log2n, int c) {
  std::lock_guard<std::mutex> lock(g_win_mu);
  if (c <= 0) {
    g_window_table.erase({curve, log2n});
  } else {
    g_window_table[{curve, log2n}] = c;
  }
}

namespace {

std::atomic<bool> g_phase_on{false};

// One set of boundary events per host thread (and device), created on first use.
struct PhaseClock {
  int dev = -1;
  cudaEvent_t ev[kMsmPhases + 1] = {};
  bool marked[kMsmPhases + 1] = {};
  ~PhaseClock() {
    for (auto& e : ev)
      if (e) cudaEventDestroy(e);
  }
};
thread_local PhaseClock t_clock;

}  // namespace

void set_phase_timing(bool on) { g_phase_on.store(on); }

void phase_mark(int i, cudaStream_t st) {
  if (!g_phase_on.load() || i < 0 || i > kMsmPhases) return;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return;
  }
  int dev = 0;
  cudaGetDevice(&dev);
  PhaseClock& pc = t_clock;
  if (pc.dev != dev) {
    for (auto& e : pc.ev) {
      if (e) cudaEventDestroy(e);
      e = nullptr;
    }
    pc.dev = dev;
  }
  if (!pc.ev[i] && cudaEventCreate(&pc.ev[i]) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  if (i == 0)
    for (auto& m : pc.marked) m = false;
  pc.marked[i] = cudaEventRecord(pc.ev[i], st) == cudaSuccess;
}

bool phase_times(float* ms) {
  PhaseClock& pc = t_clock;
  for (int i = 0; i <= kMsmPhases; ++i)
    if (!pc.marked[i]) return false;
  if (cudaEventSynchronize(pc.ev[kMsmPhases]) != cudaSuccess) return false;
  for (int i = 0; i < kMsmPhases; ++i)
    if (cudaEventElapsedTime(&ms[i], pc.ev[i], pc.ev[i + 1]) != cudaSuccess) return false;
  return true;
}

int msm_reduce_override(int curve, uint64_t n) {
  if (n < 2) n = 2;
  std::lock_guard<std::mutex> lock(g_win_mu);
  auto it = g_chunk_table.find({curve, ilog2(n)});
  return it != g_chunk_table.end() ? it->second : 0;
}

int msm_reduce_log(int curve, uint64_t n) {
  const int k = msm_reduce_override(curve, n);
  return k > 0 ? k : kRedLog1Default;
}

void msm_set_reduce_log(int curve, int log2n, int v) {
  std::lock_guard<std::mutex> lock(g_win_mu);
  if (v <= 0) {
    g_chunk_table.erase({curve, log2n});
  } else {
    g_chunk_table[{curve, log2n}] = v;
  }
}

cudaError_t launch_msm_dev(int curve, uint32_t num, uint64_t cap, const uint64_t* offsets, int c,
                           const uint32_t* points, const uint32_t* scalars, uint32_t* out,
                           cudaStream_t st) {
  switch (curve) {
    case 2: return msm_points_dev_bn254(num, cap, offsets, c, points, scalars, out, st);
    case 3: return msm_points_dev_bls12_381(num, cap, offsets, c, points, scalars, out, st);
  }
  return cudaErrorNotSupported;
}

cudaError_t launch_msm_bases_dev(void* handle, uint32_t num, uint64_t cap, const uint64_t* sizes, int c,
                                 const uint32_t* scalars, uint32_t* out, cudaStream_t st) {
  const int curve = bases_curve(handle);
  switch (curve) {
    case 2: return msm_bases_dev_bn254(handle, num, cap, sizes, c, scalars, out, st);
    case 3: return msm_bases_dev_bls12_381(handle, num, cap, sizes, c, scalars, out, st);
  }
  return cudaErrorNotSupported;
}

cudaError_t launch_msm(int curve, uint32_t num, const uint64_t* offsets, const uint32_t* points,
                       const uint32_t* scalars, uint32_t* out, cudaStream_t st) {
  switch (curve) {
    case 2: return msm_points_bn254(num, offsets, points, scalars, out, st);
    case 3: return msm_points_bls12_381(num, offsets, points, scalars, out, st);
  }
  return cudaErrorNotSupported;
}

cudaError_t bases_create(int curve, uint64_t n, const uint32_t* points, void** handle,
                         cudaStream_t st) {
  if (curve != 2 && curve != 3) return cudaErrorNotSupported;
  const int N = curve == 3 ? 12 : 8;
  uint32_t* m = nullptr;
  // BN254: the points' images beside them (glv.cuh), where there is room
  uint64_t phi = curve == 2 ? n : 0;
  size_t room = 0, all = 0;
  if (phi && (cudaMemGetInfo(&room, &all) != cudaSuccess || !images_fit(n, room))) {
    cudaGetLastError();
    phi = 0;
  }
  cudaError_t e = cudaMalloc(&m, std::max<uint64_t>(phi + n, 1) * 2 * N * 4);
  if (e == cudaErrorMemoryAllocation && phi) {
    cudaGetLastError();
    phi = 0;
    e = cudaMalloc(&m, std::max<uint64_t>(n, 1) * 2 * N * 4);
  }
  if (e != cudaSuccess) return e;
  if (n) e = points_to_mont(curve, points, n, m, phi, st);
  if (e != cudaSuccess) {
    cudaFree(m);
    return e;
  }
  *handle = new msm_detail::Bases{curve, n, m, phi};
  return cudaSuccess;
}

int bases_curve(void* handle) { return static_cast<msm_detail::Bases*>(handle)->curve; }
uint64_t bases_count(void* handle) { return static_cast<msm_detail::Bases*>(handle)->n; }

cudaError_t bases_destroy(void* handle) {
  auto* b = static_cast<msm_detail::Bases*>(handle);
  cudaError_t e = cudaFree(b->mont);
  if (b->pre) {
    const cudaError_t e2 = cudaFree(b->pre);
    if (e == cudaSuccess) e = e2;
  }
  delete b;
  return e;
}

int bases_window(void* handle) { return static_cast<msm_detail::Bases*>(handle)->pre_c; }

void msm_counts(int curve, uint64_t num, const uint64_t* sizes, uint64_t size_all, int pre_c,
                uint64_t* digits, uint64_t* buckets) {
  uint64_t d = 0, b = 0;
  BySize<int> admitted;
  for (uint64_t i = 0; i < num; ++i) {
    const uint64_t n = sizes ? sizes[i] : size_all;
    const int c = pre_c > 0 ? pre_c : admitted.get(n, [&] { return msm_admitted_window(curve, n); });
    const uint64_t W = (uint64_t)msm_detail::windows_for(curve, c);
    d += W * n;
    b += (pre_c > 0 ? 1 : W) << (c - 1);
  }
  *digits = d;
  *buckets = b;
}

cudaError_t bases_precompute(void* handle, int c, cudaStream_t st) {
  switch (bases_curve(handle)) {
    case 2: return bases_precompute_bn254(handle, c, st);
    case 3: return bases_precompute_bls12_381(handle, c, st);
  }
  return cudaErrorNotSupported;
}

cudaError_t launch_msm_bases(void* handle, uint32_t num_vectors, const uint64_t* sizes,
                             const uint32_t* scalars,
                             uint32_t* out, cudaStream_t st) {
  switch (bases_curve(handle)) {
    case 2: return msm_bases_bn254(handle, num_vectors, sizes, scalars, out, st);
    case 3: return msm_bases_bls12_381(handle, num_vectors, sizes, scalars, out, st);
  }
  return cudaErrorNotSupported;
}

}  // namespace ecc
