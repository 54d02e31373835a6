// Host side of the libcunbody C ABI (include/cunbody.h): argument checks,
// launch-shape selection, workspaces, dispatch to the kernels, batched
// plans, host-memory forms, tuning and status.
#include "cunbody.h"
#include "cn_guard.h"
#include "cn_kernels.h"
#include "cn_rows.h"
#include "cn_sym.h"

#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <optional>
#include <string>
#include <tuple>
#include <vector>

namespace cn {
cudaError_t device_status_address(int** p);
cudaError_t static_scratch_setup();
cudaError_t launch_timeout_probe(int* status, uint64_t wait_ns, cudaStream_t s);
cudaError_t run_probes(cudaStream_t s, double* out);
size_t energy_workspace_doubles();
}  // namespace cn

using cn::Plan;
using cn::PairArgs;

struct cn_batch_plan {
  int dev = -1;
  bool lists = false;       // interaction-list plan: separate i and j arrays
  bool zero_first = false;  // some group has i-particles but an empty list: clear outputs first
  int32_t n_clusters = 0;
  int64_t n_total = 0;      // i-particles (cluster plans: also the j records)
  int64_t n_j_total = 0;    // j records a list plan reads (max of begin + count)
  double pairs = 0.0;
  Plan plan;
  bool guard = false;
  bool pot = false;
  cn::TileDesc* d_tiles = nullptr;
  int32_t* d_index = nullptr;  // gathering list plans: the list entries (indices into the source records)
  int64_t n_index = 0;
  int32_t n_tiles = 0;
  int64_t units = 0;
  int64_t n_chunks = 0;
  int grid = 0;
  size_t ws_bytes = 0;
  size_t ctrl_bytes = 0;
  size_t data_bytes = 0;
  // The symmetric form of an ensemble, where it is expected to be the faster
  // one (sym_rows > 0); the above stays for calls without room for its slots.
  int32_t sym_rows = 0;
  int32_t sym_merge = 0;  // merge CTAs
  int sym_k = 0, sym_threads = 0, sym_chunk = 0, sym_stages = 0;
  size_t sym_smem = 0, sym_jslot_b = 0, sym_bytes = 0;
  int64_t sym_seg = 0;
  cn::SymGrid sym_grid{};
  cn::SymRow* d_rows = nullptr;
  cn::SymMergeBlock* d_blocks = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

namespace {

constexpr size_t kCtrlBytes = 4096;  // queue words and spare control space at the head of a workspace
constexpr uint64_t kDefaultWaitNs = 2000000000ull;
constexpr size_t kMaxSmem = 227 * 1024;
constexpr int32_t kNoIndex = 0;  // stands for the index array of a gathering plan whose lists are all empty
constexpr size_t kSymSlotCap = static_cast<size_t>(512) << 20;  // symmetric-form slot memory before banding

thread_local std::string g_last_error;
std::atomic<uint64_t> g_wait_ns{kDefaultWaitNs};

cn_status fail(cn_status st, const std::string& msg) {
  g_last_error = msg;
  return st;
}

cn_status fail_cuda(cudaError_t e, const char* what) {
  g_last_error = std::string(what) + ": " + cudaGetErrorString(e);
  return CN_ERR_CUDA;
}

// A step that a call can do without: what fails in it is no error of the call
// and leaves the thread's message as it was.
struct Attempt {
  std::string kept = g_last_error;
  ~Attempt() { g_last_error.swap(kept); }
};

// An NVTX range around each entry point (visible to Nsight tools; a few
// nanoseconds when no tool is attached).
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// CN_LOG=1 (read once, at the first call) prints each launch plan to stderr.
bool log_enabled() {
  static const bool on = [] {
    const char* v = std::getenv("CN_LOG");
    return v && *v && std::strcmp(v, "0") != 0;
  }();
  return on;
}

const char* variant_name(int v) {
  static const char* names[] = {"f32", "f32_pot", "dd", "dd_pot", "adjoint", "batched", "batched_pot",
                                "jerk", "jerk_pot", "symmetric", "f32_eps_i", "f32_eps_i_pot"};
  return (v >= 0 && v < 12) ? names[v] : "?";
}

// Host-side fault injection for tests: CN_FAULT_INJECT holds a comma list of
// "alloc", "launch", "capture"; the matching step then fails as if the CUDA
// call had failed. Nothing is done on the device.
bool inject(const char* point) {
  const char* v = std::getenv("CN_FAULT_INJECT");
  return v && std::strstr(v, point) != nullptr;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
  if (!a || !b || na == 0 || nb == 0) return false;
  const auto pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
  return pa < pb + nb && pb < pa + na;
}

// ------------------------------------------------------------------ devices
struct DeviceInfo {
  int sms = 0;
  int major = 0;
  int minor = 0;
  int* status = nullptr;
  bool supported = false;
};

std::mutex g_mu;  // guards the maps below and the creation of device entries

// Device entries, created once per device ordinal by the first call there
// (under g_mu) and never freed; read without a lock afterwards.
constexpr int kMaxDevices = 64;
std::atomic<DeviceInfo*> g_dev_table[kMaxDevices];

// Bumped whenever something a cached launch plan depends on changes: a
// tuning entry, or the address of a library workspace. Calls compare it
// with the generation their per-thread plan cache was filled under.
std::atomic<uint64_t> g_plan_gen{1};
thread_local uint64_t t_own_bumps = 0;  // generation bumps made by this thread's own workspace growth

// The launch plan of this thread's last single-system call, reused while the
// call's key and the generation match (the common loop of identical calls
// then skips the tuning, occupancy and workspace lookups).
struct PlanCache {
  bool valid = false;
  uint64_t gen = 0;
  int dev = -1;
  int variant = -1;
  int64_t n_i = -1, n_j = -1;
  bool guard = false;
  cudaStream_t stream = nullptr;
  bool hit(uint64_t g, int dv, int v, int64_t ni, int64_t nj, bool gd, cudaStream_t s) const {
    return valid && gen == g && dev == dv && variant == v && n_i == ni && n_j == nj && guard == gd && stream == s;
  }
};

DeviceInfo* device_entry(int dev) {
  return (dev >= 0 && dev < kMaxDevices) ? g_dev_table[dev].load(std::memory_order_acquire) : nullptr;
}

cn_status current_device(int* dev_out, DeviceInfo** info) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return fail(CN_ERR_UNSUPPORTED_DEVICE, "device ordinal out of range");
  DeviceInfo* d = device_entry(dev);
  if (!d) {
    std::lock_guard<std::mutex> lock(g_mu);
    d = g_dev_table[dev].load(std::memory_order_acquire);
    if (!d) {
      DeviceInfo nd;
      if ((e = cudaDeviceGetAttribute(&nd.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
          (e = cudaDeviceGetAttribute(&nd.major, cudaDevAttrComputeCapabilityMajor, dev)) != cudaSuccess ||
          (e = cudaDeviceGetAttribute(&nd.minor, cudaDevAttrComputeCapabilityMinor, dev)) != cudaSuccess)
        return fail_cuda(e, "cudaDeviceGetAttribute");
      nd.supported = (nd.major == 10 && nd.minor == 3);
      if (nd.supported && (e = cn::device_status_address(&nd.status)) != cudaSuccess)
        return fail_cuda(e, "cudaGetSymbolAddress(device status)");
      // the static scratch of cn_force_noalloc: its address, and its device
      // module loaded, on the library's first call on this device
      if (nd.supported && (e = cn::static_scratch_setup()) != cudaSuccess)
        return fail_cuda(e, "cudaGetSymbolAddress(static scratch)");
      d = new DeviceInfo(nd);
      g_dev_table[dev].store(d, std::memory_order_release);
    }
  }
  if (!d->supported)
    return fail(CN_ERR_UNSUPPORTED_DEVICE, "libcunbody is built for sm_103a (GB300); device " + std::to_string(dev) +
                                               " is sm_" + std::to_string(d->major) + std::to_string(d->minor));
  if (dev_out) *dev_out = dev;
  *info = d;
  return CN_OK;
}

// Launches that hand data from one to the next through a workspace of their
// stream are issued under this lock: calls of several threads on one stream
// follow one another there, and do not mix their launches (as calls of one
// launch cannot). Streams share the locks by hash.
std::recursive_mutex& launch_order(cudaStream_t s) {
  static std::recursive_mutex locks[64];
  return locks[(reinterpret_cast<uintptr_t>(s) / 64) % 64];
}

// ------------------------------------------------------------------ library workspaces
// Per (device, stream): `ctrl` holds the queue words and the split-tile
// arrival counters (zeroed when allocated, left zero by every kernel); `data`
// holds partial sums and packed weights (no initialisation needed).
struct LibWorkspace {
  void* ctrl = nullptr;
  size_t ctrl_bytes = 0;
  void* data = nullptr;
  size_t data_bytes = 0;
  double* aux = nullptr;  // potential-energy block sums + counter
  // slots and segments of the symmetric forms. A buffer that became too
  // small is kept until the stream's workspace is released: a captured graph
  // may still launch kernels on it. Each is at least 1.5 times the one
  // before, so that the retired ones together stay below twice the last.
  void* sym = nullptr;
  size_t sym_bytes = 0;
  std::vector<void*> retired;
};
std::map<std::pair<int, cudaStream_t>, LibWorkspace> g_ws;

bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cs) != cudaSuccess) return false;
  return cs != cudaStreamCaptureStatusNone;
}

cn_status grow(cudaStream_t s, void** buf, size_t* bytes, size_t need, bool zero, const char* what) {
  if (*buf && *bytes >= need) return CN_OK;
  if (inject("capture") || capturing(s))
    return fail(CN_ERR_WORKSPACE,
                "the library workspace of this stream must grow, which allocates; not allowed during graph "
                "capture (make one call before capturing, or pass a workspace)");
  cudaError_t e;
  if (*buf) {
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail_cuda(e, "cudaStreamSynchronize");
    cudaFree(*buf);
    *buf = nullptr;
    *bytes = 0;
    // cached plans hold its address, also when no new one can be had
    g_plan_gen.fetch_add(1, std::memory_order_acq_rel);
    ++t_own_bumps;
  }
  if (inject("alloc")) return fail(CN_ERR_CUDA, "cudaMalloc: injected allocation failure");
  const size_t nb = align_up(std::max(need, static_cast<size_t>(1) << 16), static_cast<size_t>(1) << 16);
  void* p = nullptr;
  if ((e = cudaMalloc(&p, nb)) != cudaSuccess) return fail_cuda(e, what);
  if (zero && (e = cudaMemsetAsync(p, 0, nb, s)) != cudaSuccess) {
    cudaFree(p);
    return fail_cuda(e, "cudaMemsetAsync(workspace)");
  }
  *buf = p;
  *bytes = nb;
  g_plan_gen.fetch_add(1, std::memory_order_acq_rel);
  ++t_own_bumps;
  return CN_OK;
}

cn_status library_workspace(cudaStream_t s, size_t ctrl_need, size_t data_need, char** ctrl, char** data) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
  std::lock_guard<std::mutex> lock(g_mu);
  LibWorkspace& w = g_ws[{dev, s}];
  cn_status st = grow(s, &w.ctrl, &w.ctrl_bytes, ctrl_need, true, "cudaMalloc(workspace control)");
  if (st != CN_OK) return st;
  if ((st = grow(s, &w.data, &w.data_bytes, std::max<size_t>(data_need, 256), false, "cudaMalloc(workspace)")) != CN_OK)
    return st;
  *ctrl = static_cast<char*>(w.ctrl);
  *data = static_cast<char*>(w.data);
  return CN_OK;
}

// The symmetric forms' buffer of a stream (no initialisation needed).
cn_status sym_workspace(cudaStream_t s, size_t need, char** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
  std::lock_guard<std::mutex> lock(g_mu);
  LibWorkspace& w = g_ws[{dev, s}];
  if (w.sym_bytes < need) {
    if (inject("capture") || capturing(s))
      return fail(CN_ERR_WORKSPACE,
                  "the symmetric form's slots of this stream must grow, which allocates; not allowed during graph "
                  "capture (make one call before capturing)");
    if (inject("alloc")) return fail(CN_ERR_CUDA, "cudaMalloc: injected allocation failure");
    const size_t nb = align_up(std::max(need, w.sym_bytes + w.sym_bytes / 2), static_cast<size_t>(1) << 16);
    void* p = nullptr;
    if (w.sym) w.retired.reserve(w.retired.size() + 1);
    if ((e = cudaMalloc(&p, nb)) != cudaSuccess) {
      cudaGetLastError();  // not left behind for a caller that then takes another path
      if (e == cudaErrorMemoryAllocation)
        return fail(CN_ERR_WORKSPACE, "symmetric form: the slot arrays do not fit in device memory");
      return fail_cuda(e, "cudaMalloc(symmetric slots)");
    }
    if (w.sym) w.retired.push_back(w.sym);
    w.sym = p;
    w.sym_bytes = nb;
    g_plan_gen.fetch_add(1, std::memory_order_acq_rel);
    ++t_own_bumps;
  }
  *out = static_cast<char*>(w.sym);
  return CN_OK;
}

// Frees the library workspace of a stream that is about to be destroyed.
void release_library_workspace(cudaStream_t s) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  std::lock_guard<std::mutex> lock(g_mu);
  auto it = g_ws.find({dev, s});
  if (it == g_ws.end()) return;
  if (it->second.ctrl) cudaFree(it->second.ctrl);
  if (it->second.data) cudaFree(it->second.data);
  if (it->second.aux) cudaFree(it->second.aux);
  if (it->second.sym) cudaFree(it->second.sym);
  for (void* p : it->second.retired) cudaFree(p);
  g_ws.erase(it);
  g_plan_gen.fetch_add(1, std::memory_order_acq_rel);
}

cn_status library_aux(cudaStream_t s, double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
  std::lock_guard<std::mutex> lock(g_mu);
  LibWorkspace& w = g_ws[{dev, s}];
  if (!w.aux) {
    if (inject("capture") || capturing(s))
      return fail(CN_ERR_WORKSPACE, "first potential-energy call on a stream allocates; not allowed during capture");
    if (inject("alloc")) return fail(CN_ERR_CUDA, "cudaMalloc: injected allocation failure");
    const size_t nb = (cn::energy_workspace_doubles() + 1) * sizeof(double);
    if ((e = cudaMalloc(reinterpret_cast<void**>(&w.aux), nb)) != cudaSuccess) return fail_cuda(e, "cudaMalloc(aux)");
    if ((e = cudaMemsetAsync(w.aux, 0, nb, s)) != cudaSuccess) return fail_cuda(e, "cudaMemsetAsync(aux)");
  }
  *out = w.aux;
  return CN_OK;
}

// ------------------------------------------------------------------ tuning
// Which calls a stored shape was timed on. It keeps those, or the calls of any
// sets (cn_tune_set), in the pair kernel where they would take another one;
// a size class holds one set against itself and two sets alike.
enum TunedOn : int { kTunedAny = 0, kTunedOneSet = 1, kTunedTwoSets = 2 };
struct Tuned {
  cn_tune t;
  TunedOn on;
};
std::map<std::tuple<int, int, int, int>, Tuned> g_tune;

int bucket(int64_t n) {
  int b = 0;
  while (b < 62 && (static_cast<int64_t>(1) << b) < n) ++b;
  return b;
}

bool valid_k(int variant, int k) {
  if (variant == cn::kSym) return k == 1 || k == 2 || k == 4 || k == 8;
  if (variant == cn::kDD || variant == cn::kDDPot || variant == cn::kAdjoint || variant == cn::kJerk ||
      variant == cn::kJerkPot)
    return k == 1 || k == 2 || k == 4;
  return k == 1 || k == 2 || k == 4 || k == 8;
}

int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Launch shape of the symmetric forms. Larger tiles run closer to the pipe
// (8 x 256 2.2e12 unordered pairs/s in the inner loop, 4 x 128 2.0e12, both
// at 16 warps per SM); smaller ones cut the work finer over the CTAs and
// waste less on the diagonal tiles, which are evaluated one-sided. Measured
// (us, equal masses, 152 SMs, folds as sym_fold has them; another SM count moves
// the lines by the work per SM):
//   n       2x128/128  4x128/256  4x256/128  8x128/128  8x256/128
//   5000      16.7       16.8        -         19.3+      19.3+
//   7000      25.3       22.9        -         25.0       25.2
//   9001       -         31.3       33.3         -          -
//   10007      -          -         37.7       39.7       39.7
//   14000      -          -         62.6       64.9       64.8
//   16384      -          -         80.8       79.7         -
//   18000      -          -         95.4       99.1         -
//   24000      -          -        159.6      157.8         -
//   24576      -          -          -        161.9      156.5
//   50001      -          -          -        623        605
//   131072     -          -          -       4159       3985
// (threads x K / records per stage). With the potential 4 x 256 stay ahead up to
// 24576 (20000 142.4 us, 8 x 128 142.7, unequal masses 156.2 / 171.6), and
// above the fourth sum takes 64-record stages for two CTAs of 256 threads per
// SM: 50001 798 -> 790, 131072 5343 -> 5250 against 8 x 128.
constexpr double kSymShort = 9700.0;   // where folds are short (sym_fold)
constexpr double kSymLarge = 24576.0;  // from here 8 x 256

cn_tune sym_default_tune(int64_t n, int sms, bool pot) {
  const double n_eff = static_cast<double>(n) * std::sqrt(152.0 / std::max(sms, 1));
  const bool mid = n_eff >= kSymShort && n_eff < (pot ? kSymLarge : 16000.0);
  cn_tune t{};
  t.i_per_thread = n_eff < 6000 ? 2 : n_eff < kSymShort || mid ? 4 : 8;
  t.threads = mid || n_eff >= kSymLarge ? 256 : 128;
  t.j_tile = n_eff >= 6000 && n_eff < kSymShort ? 256 : pot && n_eff >= kSymLarge ? 64 : 128;
  t.stages = 3;
  t.j_lanes = 1;
  return t;
}

// Shapes given by a tune are accepted up to the shared memory that a row of
// j-side sums per warp over the whole tile would take (three or four floats
// per particle), the limit that the entry point has always had.
size_t sym_tile_bytes(const Plan& p, bool pot) {
  const size_t b = static_cast<size_t>(p.threads) * p.k;
  return 256 + static_cast<size_t>(p.stages) * p.j_tile * 16 + (p.threads / 32) * b * (pot ? 4 : 3) * sizeof(float);
}

// The packed shapes of 256 threads with four or eight i-particles per lane
// (split-j or not) run one CTA per SM, and the static schedule gives each
// CTA ceil(units / CTAs) units of j_tile records (a ragged last j-tile is
// padded with zero masses, so every unit costs the same). For the shape's
// i-tile this picks the j-tile, a multiple of `step` in [lo, hi] and no
// longer than the j set, with the least work on the busiest CTA, counting
// `unit_cost` records of overhead per unit (64 for the 12-operation FP32
// pair, proportionally fewer for costlier pairs); ties take the smaller
// tile. Measured at N = 8192 .. 131072 (graph-replayed launches), it picked
// the fastest or a tile within 1% of it at each size of the sweeps
// (N = 14000: 0.44 -> 0.72 of the FP32 bound, 28000: 0.72 -> 0.80,
// 98304: 0.836 -> 0.852).
int32_t fit_j_tile(int64_t n_i, int64_t n_j, int64_t i_tile, int32_t lo, int32_t hi, int32_t step, int64_t ctas,
                   int32_t unit_cost = 64) {
  const int64_t n_it = (n_i + i_tile - 1) / i_tile;
  // the padding of a short tile is written by one thread
  const int64_t nj_up = (std::max<int64_t>(n_j, 1) + step - 1) / step * step;
  hi = static_cast<int32_t>(std::min<int64_t>(std::min(hi, 4096), nj_up)) / step * step;
  hi = std::max(hi, step);
  lo = std::min(hi, std::max(step, lo / step * step));
  int32_t best_t = hi;
  double best = -1.0;
  for (int32_t t = lo; t <= hi; t += step) {
    const int64_t units = n_it * ((std::max<int64_t>(n_j, 1) + t - 1) / t);
    const int64_t g = std::max<int64_t>(1, std::min(units, ctas));
    const double c = static_cast<double>((units + g - 1) / g) * static_cast<double>(t + unit_cost);
    if (best < 0.0 || c < best) {
      best = c;
      best_t = t;
    }
  }
  return best_t;
}

constexpr int64_t kDDSmall = 10500;  // particles from which the compensated form has fixed shapes

// The j-tile of a small compensated call in tiles of 64 i-particles (one per
// thread). Such a call is a chain of latencies, not work: a pair term takes
// about 0.06 us of one warp, and one warp per scheduler (two CTAs of 64
// threads per SM) runs at full speed, further units queue behind it; the CTA
// that arrives last adds its tile's parts one after the other, each as long
// as 13 records, and a unit's start costs about 24. Of the multiples of 32 this picks the
// j-tile with the least of the sum; in a sweep of 13 j-tiles it was the
// fastest one at every size tried up to 2600 (us, 2 x 64 threads with 128
// records before / now: 256 22.3 / 11.5, 1100 31.8 / 19.6, 2048 41.6 / 27.6, 2600
// 61.6 / 35.3, 100 x 4000 59.7 / 31.2). From 1.4e7 pairs on the eight CTAs of an
// SM are all busy, and the smallest tile is taken that leaves each one unit: a
// second unit for some of them costs a whole one (7982 x 2140, 1216 CTAs: 256
// records, 1125 units 69.2 us, 192, 1500 units 94.7; 4095: 256 records 72 us,
// 512 91, 480 102; 8947 x 1658 224 records 61.7, 128 70.0).
int32_t dd_small_j_tile(int64_t n_i, int64_t n_j, int sms) {
  const int64_t rows = (n_i + 63) / 64;
  const int64_t hi = std::min<int64_t>(768, (std::max<int64_t>(n_j, 1) + 31) / 32 * 32);
  if (static_cast<double>(n_i) * static_cast<double>(n_j) > 1.4e7) {
    int64_t t = 32;
    while (t < hi && rows * ((n_j + t - 1) / t) > 8 * static_cast<int64_t>(sms)) t += 32;
    return static_cast<int32_t>(t);
  }
  int32_t best_t = 32;
  int64_t best = -1;
  for (int64_t t = 32; t <= hi; t += 32) {
    const int64_t parts = (std::max<int64_t>(n_j, 1) + t - 1) / t;
    const int64_t rounds = (rows * parts + 2 * sms - 1) / (2 * sms);
    const int64_t c = rounds * (t + 24) + 13 * parts;
    if (best < 0 || c < best) {
      best = c;
      best_t = static_cast<int32_t>(t);
    }
  }
  return best_t;
}

// Default launch shape of a variant for these sizes on a device with `sms`
// multiprocessors (queried, never assumed).
cn_tune default_tune(int variant, int64_t n_i, int64_t n_j, int sms) {
  cn_tune t{};
  const int64_t n = std::max(n_i, n_j);
  const bool dd = variant == cn::kDD || variant == cn::kDDPot;
  // the adjoint and the force-jerk form stream two 16-byte records per j
  const bool adj = variant == cn::kAdjoint || variant == cn::kJerk || variant == cn::kJerkPot;
  const bool f32 = variant == cn::kF32 || variant == cn::kF32Pot || variant == cn::kF32EpsI ||
                   variant == cn::kF32EpsIPot;
  t.stages = 4;
  t.threads = 128;
  t.j_lanes = 1;
  if (f32 && n_i <= 4096) {
    // small systems (measured at N = 1024 .. 4096, packed form): lane groups
    // of 32 (16 at N = 4096) share two i-particles and, where it fits, the
    // whole j set sits in one single-stage tile, so that each CTA covers
    // whole i-tiles and nothing is merged
    const int jl = n_i > 2048 ? 16 : 32;
    t.i_per_thread = 2;
    t.j_lanes = jl;
    t.threads = n_i <= 1024 ? 128 : 256;
    const int64_t unit = 8 * jl;
    t.j_tile = static_cast<int32_t>(std::min<int64_t>(round_up(std::max<int64_t>(n_j, 1), unit), 4096));
    t.stages = n_j <= t.j_tile ? 1 : 3;
    return t;
  }
  if (f32) {
    // Mid-size systems (measured on GB300, 152 SMs, N = 4200 .. 40000,
    // graph-replayed launches): split-j lane groups of 4 or 8 holding two,
    // four or eight i-particles keep the i-tiles small enough to fill the
    // SMs while each j record feeds several packed pair terms. Sizes are compared by the
    // work per SM, n_eff = sqrt(n_i n_j) sqrt(152 / sms), so another SM count
    // moves the bands.
    const double n_eff = std::sqrt(static_cast<double>(n_i) * static_cast<double>(std::max<int64_t>(n_j, 1))) *
                         std::sqrt(152.0 / std::max(sms, 1));
    struct Band {
      double upto;
      int k, threads, j_lanes, jt_lo, jt_hi;
    };
    // (K, threads, lane groups) per band and the window of the j-tile fit;
    // fractions of the FP32 bound measured with the fitted j-tile
    static const Band bands[] = {
        {6500.0, 2, 256, 4, 512, 4096},    // N = 4500: 0.397, 6000: 0.503, 6400: 0.552
        {8600.0, 4, 256, 8, 512, 4096},    // N = 7000: 0.516, 8000: 0.562, 8192: 0.557
        {40000.0, 8, 256, 8, 512, 4096},   // 9000: 0.60, 14000: 0.72, 16384: 0.74, 20000: 0.76,
                                           // 24576: 0.80, 32768: 0.82, 40000: 0.81
    };
    if (n_i > 4096 && n_eff <= bands[2].upto) {
      for (const Band& b : bands) {
        if (n_eff > b.upto) continue;
        // with the potential the K = 8 split-j kernel runs short of registers
        // (N = 16384: 0.561 of its 14-operation bound); K = 4 with lane groups
        // of 4 keeps the 256-particle i-tile (0.689; 24576: 0.731, 32768: 0.744)
        const bool pot_k8 = variant == cn::kF32Pot && b.k == 8;
        const int k = pot_k8 ? 4 : b.k;
        const int jl = pot_k8 ? 4 : b.j_lanes;
        t.i_per_thread = k;
        t.threads = b.threads;
        t.j_lanes = jl;
        t.j_tile = fit_j_tile(n_i, n_j, static_cast<int64_t>(k) * b.threads / jl, b.jt_lo, b.jt_hi, 8 * jl, sms);
        t.stages = n_j <= t.j_tile ? 1 : 3;
        return t;
      }
    }
  }
  if ((variant == cn::kJerk || variant == cn::kJerkPot || variant == cn::kAdjoint) && n_i <= 8192) {
    // small systems, measured at N = 1024 .. 8192 (force + jerk + potential,
    // and the adjoint, with the same optima): packed split-j, two
    // i-particles per lane group of 32 (16 at N = 8192, 8 at N = 4096), up
    // to 2048 two-record j entries per stage
    const int jl = n_i <= 2048 ? 32 : (n_i <= 4096 ? 8 : 16);
    t.i_per_thread = 2;
    t.j_lanes = jl;
    t.threads = n_i <= 1024 ? 128 : 256;
    t.j_tile = static_cast<int32_t>(std::min<int64_t>(round_up(std::max<int64_t>(n_j, 1), 8 * jl), 2048));
    t.stages = n_j <= t.j_tile ? 1 : 3;
    return t;
  }
  if ((variant == cn::kJerk || variant == cn::kJerkPot || variant == cn::kAdjoint) && n < 32768) {
    // mid-size systems, measured at N = 16384 and 24576 (force + jerk +
    // potential and the adjoint): packed split-j, two i-particles per lane
    // group of 4, 512 two-record j entries per stage (N = 16384: 0.715 and
    // 0.707 of their FP32 bounds, against 0.694 and 0.667 for K = 2 x 128
    // without lane groups)
    t.i_per_thread = 2;
    t.threads = 256;
    t.j_lanes = 4;
    t.j_tile = static_cast<int32_t>(std::min<int64_t>(round_up(std::max<int64_t>(n_j, 1), 32), 512));
    t.stages = n_j <= t.j_tile ? 1 : 3;
    return t;
  }
  if (variant == cn::kSym) return sym_default_tune(n, sms, false);
  if (variant == cn::kBatched || variant == cn::kBatchedPot) {
    t.i_per_thread = 4;
    t.j_tile = 256;
  } else if (f32 && n > 4096) {
    // packed FP32, measured at N = 49152 .. 131072 (smaller systems take the
    // bands above): K = 4 x 256 below ~96K, K = 8 x 256 above, with the
    // j-tile fitted to the schedule from 512 or 1024 records. With the
    // potential K = 4 stays ahead at large N too (131072: 0.793 of its
    // 14-operation bound against 0.778 for K = 8)
    const bool k4 = n < 98304 || variant == cn::kF32Pot;
    t.i_per_thread = k4 ? 4 : 8;
    t.threads = 256;
    const int32_t jt0 = k4 ? 512 : 1024;
    t.j_tile = fit_j_tile(n_i, n_j, static_cast<int64_t>(t.i_per_thread) * t.threads, jt0 / 2, 2 * jt0, 16, sms);
  } else if (dd && n >= 20000) {
    // compensated form, K = 4 x 256 (measured at N = 24576 .. 131072), the
    // j-tile fitted to the schedule within 256 .. 1024 records; its pair
    // costs 82 FP32 lane operations, so a unit's overhead is about 9
    // records (N = 32768: 256-record tiles, 0.801 of its bound against
    // 0.782 with 1024; 24576: 1024, 0.758)
    t.i_per_thread = 4;
    t.threads = 256;
    t.j_tile = fit_j_tile(n_i, n_j, 1024, 256, 1024, 16, sms, 9);
  } else if (dd && n < kDDSmall) {
    // compensated form, small systems: one i-particle per thread in CTAs of 64
    // threads fills the SMs and its CTAs are many enough to even out the last
    // round. Up to 1.894e7 pairs the j-tile is fitted (dd_small_j_tile); above,
    // 96 records are within 8% of the best of 13 at every size tried (us, 1 x
    // 128 threads with 256 records / this: 4500 114.5 / 84.4, 5400 133.1 /
    // 103.7, 7200 181.5 / 165.1, 9000 281.6 / 249.6, 10000 335 / 312, but
    // 12000 416 / 438)
    // Where the units of 128 x 256 fill 94% of whole rounds of four CTAs per
    // SM, those stay ahead by 2 to 3% (6144 131.5 / 135.7, 8704 238 / 244)
    t.i_per_thread = 1;
    t.threads = 64;
    const int64_t units = (n_i + 127) / 128 * ((n_j + 255) / 256), round = 4 * static_cast<int64_t>(sms);
    if (static_cast<double>(n_i) * static_cast<double>(n_j) <= 1.894e7) {
      t.j_tile = dd_small_j_tile(n_i, n_j, sms);
    } else if (static_cast<double>(units) >= 0.94 * static_cast<double>((units + round - 1) / round * round)) {
      t.threads = 128;
      t.j_tile = 256;
    } else {
      t.j_tile = 96;
    }
  } else if (dd && n < 12000) {
    // K = 1 x 128, the j-tile of 256 records (11000: 373 us)
    t.i_per_thread = 1;
    t.j_tile = 256;
  } else if (n >= 32768) {
    // measured optima of the adjoint (N = 65536) and the force-jerk form
    // (N = 131072): K = 4 x 256 with j-tiles of 256 two-record j entries
    t.i_per_thread = adj ? 4 : 8;
    t.threads = 256;
    t.j_tile = adj ? 256 : 1024;
  } else if (n >= 4096) {
    // the compensated form between N = 12000 and 20000 (measured at 16384:
    // K = 2 x 128 threads x 256 records, 0.755 of its bound)
    t.i_per_thread = 2;
    t.j_tile = 256;
  } else {
    t.i_per_thread = adj ? 1 : 2;
    t.threads = 64;
    t.j_tile = 128;
  }
  return t;
}

cn_status check_tune(int variant, const cn_tune& t) {
  if (t.i_per_thread && !valid_k(variant, t.i_per_thread))
    return fail(CN_ERR_INVALID_ARG, "i_per_thread must be 1, 2, 4 or 8 (compensated and adjoint forms: 1, 2, 4)");
  if (t.threads && t.threads != 64 && t.threads != 128 && t.threads != 256)
    return fail(CN_ERR_INVALID_ARG, "threads must be 64, 128 or 256");
  if (t.j_tile && (t.j_tile < 16 || t.j_tile > 4096 || t.j_tile % 16))
    return fail(CN_ERR_INVALID_ARG, "j_tile must be a multiple of 16 in 16..4096");
  if (t.stages && (t.stages < 1 || t.stages > 8)) return fail(CN_ERR_INVALID_ARG, "stages must be 1..8");
  if (t.ctas_per_sm < 0 || t.chunk_units < 0) return fail(CN_ERR_INVALID_ARG, "negative tuning field");
  if (t.j_lanes < 0 || t.j_lanes > 32 || (t.j_lanes & (t.j_lanes - 1)))
    return fail(CN_ERR_INVALID_ARG, "j_lanes must be 0 or a power of two up to 32");
  if (t.j_lanes > 1) {
    const bool jerk = variant == cn::kJerk || variant == cn::kJerkPot || variant == cn::kAdjoint;
    const bool eps_i = variant == cn::kF32EpsI || variant == cn::kF32EpsIPot;
    const bool f32 = variant == cn::kF32 || variant == cn::kF32Pot || variant == cn::kBatched ||
                     variant == cn::kBatchedPot;
    if (!f32 && !eps_i && !jerk)
      return fail(CN_ERR_INVALID_ARG, "j_lanes > 1 is offered for the FP32 (single, batched, per-i softening), "
                                      "force-jerk and adjoint forms");
    if (eps_i && t.i_per_thread > 2)
      return fail(CN_ERR_INVALID_ARG, "the per-i-softening form takes j_lanes > 1 with i_per_thread = 1 or 2");
    if (jerk && t.i_per_thread != 2)
      return fail(CN_ERR_INVALID_ARG, "the force-jerk and adjoint forms take j_lanes > 1 with i_per_thread = 2");
    if (t.j_tile && t.j_tile % (8 * t.j_lanes))
      return fail(CN_ERR_INVALID_ARG, "with j_lanes > 1, j_tile must be a multiple of 8 x j_lanes");
  }
  return CN_OK;
}

bool two_records(int variant) {
  return variant == cn::kAdjoint || variant == cn::kJerk || variant == cn::kJerkPot;
}

// Whether a stored shape keeps calls of these sets in the pair kernel.
bool registered_tune(int dev, int variant, int64_t n_i, int64_t n_j, TunedOn sets) {
  std::lock_guard<std::mutex> lock(g_mu);
  const auto it = g_tune.find({dev, variant, bucket(n_i), bucket(n_j)});
  return it != g_tune.end() && (it->second.on == kTunedAny || it->second.on == sets);
}

cn_status store_tune(int variant, int64_t n_i, int64_t n_j, const cn_tune* tune, TunedOn on) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
  std::lock_guard<std::mutex> lock(g_mu);
  const auto key = std::make_tuple(dev, variant, bucket(n_i), bucket(n_j));
  if (tune)
    g_tune[key] = Tuned{*tune, on};
  else
    g_tune.erase(key);
  g_plan_gen.fetch_add(1, std::memory_order_acq_rel);
  return CN_OK;
}

cn_status resolve_plan(int dev, int variant, int64_t n_i, int64_t n_j, bool guard, const cn_tune* explicit_tune,
                       Plan* p) {
  int sms = 0;
  if (const DeviceInfo* d = device_entry(dev)) sms = d->sms;
  if (sms <= 0 && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return fail(CN_ERR_CUDA, "cudaDeviceGetAttribute(multiprocessor count)");
  cn_tune t = default_tune(variant, n_i, n_j, sms);
  cn_tune chosen{};
  bool have = false;
  if (explicit_tune) {
    chosen = *explicit_tune;
    have = true;
  } else {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_tune.find({dev, variant, bucket(n_i), bucket(n_j)});
    if (it != g_tune.end()) {
      chosen = it->second.t;
      have = true;
    }
  }
  if (have) {
    cn_status st = check_tune(variant, chosen);
    if (st != CN_OK) return st;
    if (chosen.i_per_thread) t.i_per_thread = chosen.i_per_thread;
    if (chosen.threads) t.threads = chosen.threads;
    if (chosen.j_tile) t.j_tile = chosen.j_tile;
    if (chosen.stages) t.stages = chosen.stages;
    t.ctas_per_sm = chosen.ctas_per_sm;
    t.chunk_units = chosen.chunk_units;
    t.j_lanes = chosen.j_lanes > 1 ? chosen.j_lanes : 1;
  }
  p->k = guard ? 1 : t.i_per_thread;
  p->threads = t.threads;
  p->j_tile = t.j_tile;
  p->stages = t.stages;
  p->ctas_per_sm = t.ctas_per_sm;
  p->chunk_units = t.chunk_units;
  p->j_lanes = t.j_lanes > 1 ? t.j_lanes : 1;
  if (p->j_lanes > 1 && variant == cn::kSym) return fail(CN_ERR_INVALID_ARG, "the symmetric form takes no j_lanes");
  if (p->j_lanes > 1 && (variant == cn::kJerk || variant == cn::kJerkPot || variant == cn::kAdjoint) && guard) {
    p->j_lanes = 1;  // the guarded force-jerk and adjoint kernels hold one i-particle per thread, without split-j
    p->k = 1;
  }
  if (p->j_lanes > 1) {
    // split-j: K i-particles per lane group (packed for K >= 2; the guarded
    // kernels hold one, the per-i-softening ones at most two)
    const bool eps_i = variant == cn::kF32EpsI || variant == cn::kF32EpsIPot;
    if (guard) p->k = 1;
    else if (eps_i && p->k > 2) p->k = 2;
    if (p->j_tile % (8 * p->j_lanes)) return fail(CN_ERR_INVALID_ARG, "j_tile must be a multiple of 8 x j_lanes");
  }
  const size_t smem = variant == cn::kSym
                          ? sym_tile_bytes(*p, false)
                          : (two_records(variant) ? cn::adjoint_smem_bytes(*p) : cn::ring_smem_bytes(*p));
  if (smem > kMaxSmem) return fail(CN_ERR_INVALID_ARG, "the launch shape exceeds the shared memory of one CTA");
  if (variant == cn::kSym && p->i_tile() % p->j_tile) p->j_tile = std::min(p->j_tile, p->i_tile());
  if (variant == cn::kSym && (p->i_tile() % p->j_tile || p->j_tile % 8))
    return fail(CN_ERR_INVALID_ARG, "symmetric form: j_tile must divide threads x i_per_thread and be a multiple of 8");
  return CN_OK;
}

// ------------------------------------------------------------------ geometry
struct Geometry {
  int64_t n_tiles = 0;
  int64_t njt = 0;
  int64_t units = 0;
  int64_t n_chunks = 0;
  int grid = 0;
  size_t smem = 0;
  size_t ctrl_bytes = 0;  // queue words + arrival counters (must be zero at launch)
  size_t data_bytes = 0;  // partial sums (+ packed weights)
  size_t off_wrec = 0;    // packed weights, from the start of the data region
  size_t ws_bytes = 0;    // one caller buffer: control region, then data region
};

std::map<std::tuple<int, int, bool, int, int, int, size_t>, int> g_occ;

// One line per launch on stderr when CN_LOG is set: the variant, sizes,
// launch shape, grid, units, chunks and how many i-tiles are split across
// chunks (those take the FP64 merge). Single-system schedules only count
// split tiles; batched plans pass n_tiles_split < 0.
void log_plan(const char* entry, int variant, int64_t n_i, int64_t n_j, bool guard, const Plan& p, const Geometry& g,
              int64_t njt) {
  if (!log_enabled()) return;
  int64_t split = -1;
  if (njt > 0 && g.units > 0 && p.chunk_units == 0) {
    split = 0;
    const int64_t U = g.units, Q = g.n_chunks;
    auto chunk_of = [&](int64_t u) { return ((u + 1) * Q - 1) / U; };
    for (int64_t t = 0; t < g.n_tiles; ++t)
      if (chunk_of(t * njt) != chunk_of(t * njt + njt - 1)) ++split;
  }
  std::fprintf(stderr,
               "[cunbody] %s: variant %s n_i %lld n_j %lld%s | K %d threads %d j_tile %d stages %d j_lanes %d "
               "chunk_units %lld ctas_per_sm %d | grid %d units %lld chunks %lld i_tiles %lld split_tiles %lld "
               "smem %zu ws %zu\n",
               entry, variant_name(variant), static_cast<long long>(n_i), static_cast<long long>(n_j),
               guard ? " (guarded)" : "", p.k, p.threads, p.j_tile, p.stages, p.j_lanes,
               static_cast<long long>(p.chunk_units), p.ctas_per_sm, g.grid, static_cast<long long>(g.units),
               static_cast<long long>(g.n_chunks), static_cast<long long>(g.n_tiles), static_cast<long long>(split),
               g.smem, g.ws_bytes);
}

cn_status occupancy(int dev, int variant, bool guard, const Plan& p, size_t smem, int* ctas, bool gather = false) {
  const auto key = std::make_tuple(dev, variant + (gather ? 100 : 0), guard, p.j_lanes, p.k, p.threads, smem);
  {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_occ.find(key);
    if (it != g_occ.end()) {
      *ctas = it->second;
      return CN_OK;
    }
  }
  int c = 0;
  cudaError_t e;
  switch (variant) {
    case cn::kF32: e = cn::occupancy_f32(p, false, guard, false, smem, &c); break;
    case cn::kF32Pot: e = cn::occupancy_f32(p, true, guard, false, smem, &c); break;
    case cn::kDD: e = cn::occupancy_dd(p, false, guard, smem, &c); break;
    case cn::kDDPot: e = cn::occupancy_dd(p, true, guard, smem, &c); break;
    case cn::kAdjoint: e = cn::occupancy_adjoint(p, guard, smem, &c); break;
    case cn::kBatched:
      e = gather ? cn::occupancy_f32_gather(p, false, guard, smem, &c) : cn::occupancy_f32(p, false, guard, true, smem, &c);
      break;
    case cn::kBatchedPot:
      e = gather ? cn::occupancy_f32_gather(p, true, guard, smem, &c) : cn::occupancy_f32(p, true, guard, true, smem, &c);
      break;
    case cn::kJerk: e = cn::occupancy_jerk(p, false, guard, smem, &c); break;
    case cn::kJerkPot: e = cn::occupancy_jerk(p, true, guard, smem, &c); break;
    case cn::kF32EpsI: e = cn::occupancy_f32(p, false, true, false, smem, &c, true); break;
    case cn::kF32EpsIPot: e = cn::occupancy_f32(p, true, true, false, smem, &c, true); break;
    default: return fail(CN_ERR_INVALID_ARG, "unknown variant");
  }
  if (e != cudaSuccess) return fail_cuda(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
  if (c <= 0) return fail(CN_ERR_INVALID_ARG, "launch shape does not fit on one SM");
  std::lock_guard<std::mutex> lock(g_mu);
  g_occ[key] = c;
  *ctas = c;
  return CN_OK;
}

int slot_f4(int variant) {
  return (variant == cn::kDD || variant == cn::kDDPot || variant == cn::kJerk || variant == cn::kJerkPot) ? 2 : 1;
}

// Grid and workspace layout for `units` units over `n_tiles` i-tiles
// (gather: the gathering list kernel).
cn_status layout(int dev, const DeviceInfo& d, int variant, bool guard, const Plan& p, int64_t n_tiles,
                 int64_t units, int64_t n_wrec, Geometry* g, bool gather = false) {
  g->n_tiles = n_tiles;
  g->units = units;
  g->smem = gather ? cn::gather_smem_bytes(p) : two_records(variant) ? cn::adjoint_smem_bytes(p) : cn::ring_smem_bytes(p);
  if (g->smem > kMaxSmem) return fail(CN_ERR_INVALID_ARG, "the launch shape exceeds the shared memory of one CTA");
  int occ = 0;
  cn_status st = occupancy(dev, variant, guard, p, g->smem, &occ, gather);
  if (st != CN_OK) return st;
  const int ctas = p.ctas_per_sm > 0 ? std::min(p.ctas_per_sm, occ) : occ;
  const int64_t slots = static_cast<int64_t>(ctas) * d.sms;
  if (p.chunk_units == 0) {
    g->n_chunks = std::min<int64_t>(slots, units);
    g->grid = static_cast<int>(g->n_chunks);
  } else {
    g->n_chunks = ceil_div(units, p.chunk_units);
    g->grid = static_cast<int>(std::min<int64_t>(slots, g->n_chunks));
  }
  if (g->n_tiles > INT32_MAX || g->n_chunks > INT32_MAX)
    return fail(CN_ERR_INVALID_ARG, "problem too large for one launch");
  g->ctrl_bytes = align_up(kCtrlBytes + static_cast<size_t>(n_tiles) * 4, 256);
  const size_t partial_bytes =
      static_cast<size_t>(g->n_chunks) * 2 * static_cast<size_t>(p.i_tile()) * 16 * slot_f4(variant);
  g->off_wrec = align_up(partial_bytes, 256);
  g->data_bytes = g->off_wrec + static_cast<size_t>(n_wrec) * 16;
  g->ws_bytes = g->ctrl_bytes + g->data_bytes;
  return CN_OK;
}

cn_status single_geometry(int dev, const DeviceInfo& d, int variant, bool guard, const Plan& p, int64_t n_i,
                          int64_t n_j, Geometry* g) {
  const int64_t n_tiles = ceil_div(n_i, p.i_tile());
  const int64_t njt = ceil_div(n_j, p.j_tile);
  if (njt > INT32_MAX) return fail(CN_ERR_INVALID_ARG, "n_j too large");
  g->njt = njt;
  return layout(dev, d, variant, guard, p, n_tiles, n_tiles * njt, variant == cn::kAdjoint ? n_i : 0, g);
}

PairArgs base_args(char* ctrl, char* data, const Geometry& g, const Plan& p, int* status) {
  PairArgs a{};
  a.queue = reinterpret_cast<int*>(ctrl);
  a.counters = reinterpret_cast<unsigned int*>(ctrl + kCtrlBytes);
  a.partials = reinterpret_cast<float4*>(data);
  a.status = status;
  a.total_units = g.units;
  a.chunk_units = p.chunk_units;
  a.n_chunks = g.n_chunks;
  a.n_tiles = static_cast<int32_t>(g.n_tiles);
  a.njt = static_cast<int32_t>(g.njt);
  a.j_tile = p.j_tile;
  a.stages = p.stages;
  a.j_lanes = p.j_lanes;
  a.wait_ns = g_wait_ns.load();
  return a;
}

// Resolves the workspace of a launch: the library's (per stream) or one
// caller buffer whose control head is cleared here, on the stream.
cn_status launch_workspace(cudaStream_t s, const Geometry& g, void* ws, size_t ws_bytes, bool lib_ws, char** ctrl,
                           char** data) {
  if (lib_ws) return library_workspace(s, g.ctrl_bytes, g.data_bytes, ctrl, data);
  if (!ws || ws_bytes < g.ws_bytes) return fail(CN_ERR_WORKSPACE, "workspace smaller than the size this call needs");
  if (!aligned(ws, 256)) return fail(CN_ERR_MISALIGNED, "workspace must be 256-byte aligned");
  cudaError_t e = cudaMemsetAsync(ws, 0, g.ctrl_bytes, s);
  if (e != cudaSuccess) return fail_cuda(e, "cudaMemsetAsync(workspace control)");
  *ctrl = static_cast<char*>(ws);
  *data = static_cast<char*>(ws) + g.ctrl_bytes;
  return CN_OK;
}

cn_status check_eps2(float eps2) {
  if (!std::isfinite(eps2) || eps2 < 0.f) return fail(CN_ERR_INVALID_ARG, "eps2 must be finite and >= 0");
  return CN_OK;
}

// eps2 below the smallest normal float can make s flush to zero: take the guarded kernels.
bool needs_guard(float eps2) { return !(eps2 >= FLT_MIN); }

cn_status check_records(const float* p, int64_t n, const char* name) {
  if (n > 0 && !p) return fail(CN_ERR_INVALID_ARG, std::string(name) + " is NULL");
  if (p && !aligned(p, 16)) return fail(CN_ERR_MISALIGNED, std::string(name) + " must be 16-byte aligned");
  return CN_OK;
}

// ------------------------------------------------------------------ symmetric forms
// Shape, workspace and layout of a symmetric launch.
struct SymPlan {
  PlanCache key;
  int k = 0, threads = 0, chunk = 0, stages = 0, fold = 0;
  bool guard = false;
  int64_t tile = 0, tiles = 0, n_blocks = 0, n_pad = 0;
  int64_t band = 0;  // tile rows per launch
  int64_t slots = 0;  // resident CTAs
  size_t smem = 0, jslot_b = 0, seg_b = 0, need = 0;
  char* data = nullptr;
};

cn_status sym_occupancy(int dev, cn::SymForm form, const SymPlan& sp, int* ctas) {
  const auto key = std::make_tuple(dev, 1000 + static_cast<int>(form), sp.guard, 1, sp.k, sp.threads, sp.smem);
  {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_occ.find(key);
    if (it != g_occ.end()) {
      *ctas = it->second;
      return CN_OK;
    }
  }
  const cudaError_t e = cn::sym_ops(form).occupancy(sp.k, sp.guard, sp.threads, sp.smem, ctas);
  if (e != cudaSuccess) return fail_cuda(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
  if (*ctas <= 0) return fail(CN_ERR_INVALID_ARG, "launch shape does not fit on one SM");
  std::lock_guard<std::mutex> lock(g_mu);
  g_occ[key] = *ctas;
  return CN_OK;
}

// j blocks between the folds of register sums. Where the pair kernel's lane
// groups split a j-tile into short chains, 256 records left a larger error than
// it did (2-norm against 64 bits, geometric mean over 16 sets, cusps of unequal
// masses: force 10007 1.20 of it, 13001 1.05, 18000 1.06, jerk 12000 1.07; now 0.99,
// 0.96, 0.92, 0.88; Plummer spheres 0.58 .. 0.98). Below and above, 256 are at 0.5 ..
// 0.99 of it and cost 1 to 2% less. Up to 26000 also against the reduce-scatter
// kernel that cn_force_symmetric had, whose tiles are small until there (24577 1.13
// of its error, now 1.01; 28000 0.66 with 256).
int sym_fold(cn::SymForm form, int64_t n, int sms) {
  const double n_eff = static_cast<double>(n) * std::sqrt(152.0 / std::max(sms, 1));
  const bool force = form == cn::kSymForce || form == cn::kSymForcePot;
  const bool jerk = form == cn::kSymJerk || form == cn::kSymJerkPot;
  const bool few = force ? n_eff >= kSymShort && n_eff < 26000.0 : jerk && n_eff >= 7500.0 && n_eff < 16000.0;
  return (few ? 128 : 256) / cn::kSymBlock;  // the adjoint's kernel folds within a stage
}

// Fits the plan of `form` for n particles (p: the shape); `need` bytes of
// workspace go into data. The j-side slots of every off-diagonal unit take one
// [rows][n_pad] array (half of it written) when that fits in kSymSlotCap,
// else bands of fewer rows, each merged into running sums; plus the i-side
// segments, one per (CTA, row). The shape's chunk_units, when set, fixes the
// rows per band.
cn_status sym_fit(int dev, const DeviceInfo& d, cn::SymForm form, int64_t n, bool guard, const Plan& p, SymPlan* sp) {
  const cn::SymOps ops = cn::sym_ops(form);
  sp->k = guard ? 2 : std::min(ops.max_k, std::max(2, p.k));
  sp->threads = p.threads;
  sp->guard = guard;
  sp->fold = sym_fold(form, n, d.sms);
  sp->chunk = static_cast<int>(std::min<int64_t>(round_up(p.j_tile, cn::kSymBlock), std::min(ops.max_stage, sp->fold * cn::kSymBlock)));
  sp->stages = std::max(2, p.stages);  // a stage is refilled a chunk after it was read
  sp->tile = static_cast<int64_t>(sp->k) * sp->threads;
  sp->tiles = ceil_div(n, sp->tile);
  sp->n_blocks = ceil_div(n, cn::kSymBlock);
  sp->n_pad = sp->n_blocks * cn::kSymBlock;
  if (sp->tiles > 65535) return fail(CN_ERR_INVALID_ARG, "too many tiles for the symmetric form");
  while ((sp->smem = ops.smem(sp->threads, sp->k, sp->chunk, sp->stages)) > kMaxSmem) {
    if (sp->stages > 2)
      --sp->stages;
    else if (sp->chunk > cn::kSymBlock)
      sp->chunk = static_cast<int>(round_up(sp->chunk / 2, cn::kSymBlock));
    else
      return fail(CN_ERR_INVALID_ARG, "the launch shape exceeds the shared memory of one CTA");
  }
  int occ = 0;
  cn_status st = sym_occupancy(dev, form, *sp, &occ);
  if (st != CN_OK) return st;
  sp->slots = static_cast<int64_t>(p.ctas_per_sm > 0 ? std::min(p.ctas_per_sm, occ) : occ) * d.sms;
  const size_t word = sizeof(float) * static_cast<size_t>(ops.sums);
  const size_t row_b = static_cast<size_t>(sp->n_pad) * word;
  sp->band = sp->tiles;
  if (p.chunk_units > 0)
    sp->band = std::min<int64_t>(p.chunk_units, sp->tiles);
  else if (static_cast<double>(sp->tiles) * static_cast<double>(row_b) > static_cast<double>(kSymSlotCap))
    sp->band = std::max<int64_t>(1, std::min<int64_t>(sp->tiles, static_cast<int64_t>(kSymSlotCap / row_b)));
  sp->jslot_b = align_up(static_cast<size_t>(sp->band) * row_b, 256);
  sp->seg_b = align_up(static_cast<size_t>(sp->slots + sp->band) * static_cast<size_t>(sp->tile) * sizeof(float) *
                           static_cast<size_t>(ops.planes),
                       256);
  sp->need = sp->jslot_b + sp->seg_b + (sp->band < sp->tiles ? 2 * row_b : 0);
  return CN_OK;
}

cn_status sym_launch(const std::string& what, const DeviceInfo& d, cn::SymForm form, const SymPlan& sp, int64_t n,
                     const float* pos, const float* rec2, float eps2, float* const (&out)[3], cudaStream_t s) {
  cn::SymArgs a{};
  a.g.n = n;
  a.g.n_tiles = static_cast<int32_t>(sp.tiles);
  a.g.n_blocks = static_cast<int32_t>(sp.n_blocks);
  a.g.tile_blocks = static_cast<int32_t>(sp.tile / cn::kSymBlock);
  a.pos = reinterpret_cast<const float4*>(pos);
  a.rec2 = reinterpret_cast<const float4*>(rec2);
  a.slots_j = reinterpret_cast<float*>(sp.data);
  a.slots_seg = reinterpret_cast<float*>(sp.data + sp.jslot_b);
  a.n_seg = sp.slots + sp.band;
  a.status = d.status;
  a.n_pad = sp.n_pad;
  a.chunk = sp.chunk;
  a.fold = sp.fold;
  a.stages = sp.stages;
  a.eps2 = eps2;
  // a mass-free term of these forms is at most 4 eps^-3 |w| with |w| <= 2 sqrt(3) of the largest component, and
  // at most 256 of them are added before they are scaled
  a.fast = static_cast<float>(std::min(3e38, 5e34 * std::pow(static_cast<double>(eps2), 1.5)));
  a.wait_ns = g_wait_ns.load();
  cn::SymMerge m{};
  m.slots_seg = a.slots_seg;
  m.slots_j = a.slots_j;
  m.carry = sp.band < sp.tiles ? reinterpret_cast<double*>(sp.data + sp.jslot_b + sp.seg_b) : nullptr;
  for (int o = 0; o < 3; ++o) m.out[o] = out[o];
  m.n_pad = sp.n_pad;
  m.tile = static_cast<int32_t>(sp.tile);
  m.n_merge = static_cast<int32_t>(sp.n_blocks);
  std::lock_guard<std::recursive_mutex> order(launch_order(s));
  for (int64_t r0 = 0; r0 < sp.tiles; r0 += sp.band) {
    const int64_t r1 = std::min(sp.tiles, r0 + sp.band);
    a.g.row0 = static_cast<int32_t>(r0);
    a.g.row1 = static_cast<int32_t>(r1);
    a.g.cost0 = a.g.row_start(r0);
    a.g.cost = a.g.row_start(r1) - a.g.cost0;
    a.g.grid = static_cast<int32_t>(std::max<int64_t>(1, std::min<int64_t>(sp.slots, a.g.cost / cn::kSymCostPair)));
    m.g = a.g;
    // parts of more than 1024 records
    a.both_words = a.g.cost > static_cast<int64_t>(a.g.grid) * cn::kSymCostPair * (1024 / cn::kSymBlock);
    m.first = r0 == 0;
    m.last = r1 == sp.tiles;
    if (log_enabled()) {
      int64_t units = 0;
      for (int64_t I = r0; I < r1; ++I) units += sp.n_blocks - I * a.g.tile_blocks;
      std::fprintf(stderr,
                   "[cunbody] %s%s | symmetric: K %d threads %d chunk %d stages %d | tile %lld tiles %lld band rows "
                   "%lld..%lld units %lld grid %d smem %zu slots %zu bytes\n",
                   what.c_str(), sp.guard ? " (guarded)" : "", sp.k, sp.threads, sp.chunk, sp.stages,
                   static_cast<long long>(sp.tile), static_cast<long long>(sp.tiles), static_cast<long long>(r0),
                   static_cast<long long>(r1), static_cast<long long>(units), a.g.grid, sp.smem, sp.need);
    }
    if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
    const cudaError_t e = cn::sym_ops(form).launch(a, m, sp.k, sp.guard, sp.threads, sp.smem, s);
    if (e != cudaSuccess) return fail_cuda(e, "symmetric kernel launch");
  }
  return CN_OK;
}

// Size from which one particle set against itself (the same pointer as i and
// j set) takes the symmetric form: just above the one-launch split-j shapes
// of the smallest systems, which merge nothing. Measured (us, one-sided /
// symmetric): force 4096 11.1 / 14.1, 5000 20.5 / 16.7, 16384 108 / 78;
// force + jerk + potential 2048 10.4 / 12.1, 3000 31.2 / 16.8, 16384 271 /
// 178; adjoint (folded every 64 records, now 32) 2048 12.3 / 14.4, 3000 34.9 /
// 18.5, 16384 284 / 174.
bool sym_pays(cn::SymForm form, int64_t n, int sms) {
  const int64_t from = form == cn::kSymForce || form == cn::kSymForcePot ? 4096 : 2048;
  return n > from && static_cast<double>(n) * std::sqrt(152.0 / std::max(sms, 1)) > static_cast<double>(from);
}

// Launch shape of a symmetric form (the force: sym_default_tune). The jerk's
// eight particles per thread (248 registers, one CTA of 256 per SM) share
// the 14 shuffles of a step among twice the pairs: with the potential 65536
// 2571 us against 2739 for four, 32768 659 / 687, 16384 184 / 178. Eight for
// the adjoint (folded every 64 records, now 32: 65536 2485): 65536 2392 /
// 2431, 50000 1484 / 1435, so it stays at four.
// Below, two or four particles in smaller tiles: jerk 4096 21.9 us (2 x 256)
// / 22.4 (4 x 128), 6000 37.7 / 36.3; adjoint 6000 36.9 (2 x 128) / 39.0 (4 x
// 128), 10000 81.9 / 77.8, 24576 373 (4 x 128) / 371 (4 x 256).
Plan sym_default_plan(cn::SymForm form, int64_t n, int sms) {
  Plan p;
  p.stages = 3;
  if (form == cn::kSymForce || form == cn::kSymForcePot) {
    const cn_tune t = sym_default_tune(n, sms, form == cn::kSymForcePot);
    p.k = t.i_per_thread;
    p.threads = t.threads;
    p.j_tile = t.j_tile;
    return p;
  }
  const double n_eff = static_cast<double>(n) * std::sqrt(152.0 / std::max(sms, 1));
  p.j_tile = 128;
  if (form == cn::kSymAdjoint) {
    p.k = n_eff < 6500 ? 2 : 4;
    p.threads = n_eff < 20000 ? 128 : 256;
  } else {
    p.k = n_eff < 5000 ? 2 : n_eff < 20000 ? 4 : 8;
    p.threads = 256;
  }
  return p;
}

// ------------------------------------------------------------------ one-sided rows
struct RowPlan {
  int k = 0, wi = 0, chunk = 0, stages = 0;
  size_t smem = 0, need = 0;
  int64_t tile = 0, rows = 0, blocks = 0, units = 0;
  int grid = 0;
};

// Shape of the row kernel. Small tiles (four particles per thread, all warps
// on the same 128) waste the least on small sets: 4000 x 16384 31.6 us against
// 32.6 for 8 x 32 and 56 for eight warps along i. Large plain sets take eight
// per thread (2048 x 262144 209 against 213 us) where they fill those tiles as
// well (1145 x 146556 86.2 us in the pair kernel, 87.2 with eight, 75.8 with four); with the potential or
// per-particle softening the registers of four suit better, and the latter's
// large sets take the warps along i (32768 x 32768 with the potential 461 us,
// 466 with all warps on the same, 482 with eight per thread).
cn_status rows_fit(int dev, const DeviceInfo& d, cn::RowForm form, int64_t n_i, int64_t n_j, RowPlan* rp) {
  const double pairs = static_cast<double>(n_i) * static_cast<double>(n_j);
  rp->k = form == cn::kRowForce && pairs >= 1.5e8 && 20 * round_up(n_i, 256) <= 21 * round_up(n_i, 128) ? 8 : 4;
  rp->wi = form != cn::kRowForce && pairs >= 5e8 && n_i >= 16384 ? 8 : 1;
  rp->stages = 3;
  rp->chunk = rp->wi == 8 ? 256 : 1024;
  rp->tile = static_cast<int64_t>(32) * rp->k * rp->wi;
  rp->rows = ceil_div(n_i, rp->tile);
  rp->blocks = ceil_div(n_j, cn::kRowBlock);
  rp->units = rp->rows * rp->blocks;
  if (rp->rows > INT32_MAX / 2 || rp->blocks > INT32_MAX / 2) return fail(CN_ERR_INVALID_ARG, "problem too large for one launch");
  rp->smem = cn::rows_smem_bytes(form, rp->k, rp->chunk, rp->stages);
  const auto key = std::make_tuple(dev, 2000 + static_cast<int>(form), false, 1, rp->k, 256, rp->smem);
  int occ = 0;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_occ.find(key);
    if (it != g_occ.end()) occ = it->second;
  }
  if (occ == 0) {
    const cudaError_t e = cn::occupancy_rows(form, rp->k, rp->smem, &occ);
    if (e != cudaSuccess) return fail_cuda(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    if (occ <= 0) return fail(CN_ERR_INVALID_ARG, "launch shape does not fit on one SM");
    std::lock_guard<std::mutex> lock(g_mu);
    g_occ[key] = occ;
  }
  rp->grid = static_cast<int>(std::min<int64_t>(static_cast<int64_t>(occ) * d.sms, rp->units));
  const bool pot = form == cn::kRowForcePot || form == cn::kRowEpsIPot;
  rp->need = static_cast<size_t>(2) * rp->grid * (pot ? 4 : 3) * rp->tile * sizeof(float);
  return CN_OK;
}

cn_status rows_launch(const std::string& what, const DeviceInfo& d, cn::RowForm form, const RowPlan& rp, int64_t n_i,
                      const float* pos_i, int64_t n_j, const float* pos_j, float eps2, float* acc_out, float* pot_out,
                      char* data, cudaStream_t s) {
  cn::RowArgs a{};
  a.pos_i = reinterpret_cast<const float4*>(pos_i);
  a.pos_j = reinterpret_cast<const float4*>(pos_j);
  a.acc_out = acc_out;
  a.pot_out = pot_out;
  a.segs = reinterpret_cast<float*>(data);
  a.status = d.status;
  a.n_i = n_i;
  a.n_j = n_j;
  a.units = rp.units;
  a.n_rows = static_cast<int32_t>(rp.rows);
  a.blocks = static_cast<int32_t>(rp.blocks);
  a.grid = rp.grid;
  a.tile = static_cast<int32_t>(rp.tile);
  a.wi = rp.wi;
  a.chunk = rp.chunk;
  a.stages = rp.stages;
  a.eps2 = eps2;
  a.wait_ns = g_wait_ns.load();
  if (log_enabled())
    std::fprintf(stderr, "[cunbody] %s | rows: K %d tile %lld rows %lld chunk %d stages %d | units %lld grid %d smem %zu ws %zu\n",
                 what.c_str(), rp.k, static_cast<long long>(rp.tile), static_cast<long long>(rp.rows), rp.chunk, rp.stages,
                 static_cast<long long>(rp.units), rp.grid, rp.smem, rp.need);
  if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
  std::lock_guard<std::recursive_mutex> order(launch_order(s));
  const cudaError_t e = cn::launch_rows(form, rp.k, a, rp.smem, s);
  return e == cudaSuccess ? CN_OK : fail_cuda(e, "row kernel launch");
}

// Whether the row kernel is the faster one for any masses, on a device with
// `sms` multiprocessors (pairs and particles counted per SM); p and g: the
// pair kernel's shape and schedule of the call. Below 2.4e7 pairs the pair
// kernel's small shapes are (4500 x 4500 15.6 us against 17.6, 8192 x 2500 15.7
// / 17.8), and fewer than 128 i-particles leave lanes idle (40 x 600000 38.2 /
// 60.8). Above, by 253 random shapes and 150 on a grid, unequal masses:
// - i-particles that fill their tiles badly (more than 1.28 times their number
//   in whole tiles, none from 401 on) keep the pair kernel: 135 x 180000 33.0 /
//   46.9, 145 x 450445 48.8 / 62.9, but 202 x 239087 48.8 / 42.5.
// - Up to 4096 of them the pair kernel's small shapes have large j-tiles: 300 x
//   70000 31.7 / 27.4, 4000 x 16384 39.8 / 33.6, 2048 x 262144 241 / 211.
// - More of them run at most 6% slower with the row kernel where the pair
//   kernel's schedule wastes nothing (5990 x 6938 24.1 / 25.5, 6136 x 7916 26.4 /
//   27.9) and up to 8% faster where it wastes a tenth: from 5% on it is taken
//   (6750 x 3592 20.2 / 18.8, 7009 x 11997 45.0 / 41.8).
// - Plain sets and those with the potential: large ones keep the pair kernel
//   (8192 x 100003 309 / 320, 10007 x 100003 376 / 388, 16384 x 16384 108.1 /
//   109.5).
// - Per-particle softening, whose pair kernel holds two particles per lane
//   group and a guard in every pair: always from 4.2e7 pairs (65536 x 65536 1713
//   / 1634, 2065368 x 22 756 / 369); below, more than 4096 i-particles as above,
//   and not on fewer than 1000 j records, which leave most of a row's warps idle
//   (95845 x 275 22.4 / 28.3, 17999 x 1343 15.9 / 20.7).
bool rows_pays(cn::RowForm form, int64_t n_i, int64_t n_j, int sms, const Plan& p, const Geometry& g) {
  const double share = 152.0 / std::max(sms, 1);
  const double real = static_cast<double>(n_i) * static_cast<double>(n_j), pairs = real * share;
  if (n_i < 128 || pairs < 2.4e7 || static_cast<double>(round_up(n_i, 128)) > 1.28 * static_cast<double>(n_i)) return false;
  const bool eps_i = form == cn::kRowEpsI || form == cn::kRowEpsIPot;
  const double rows = static_cast<double>(n_i) * share;
  if (eps_i ? pairs >= 4.2e7 : rows <= 4096.0 && pairs <= 5.5e8) return true;
  if (eps_i ? n_j < 1000 : rows > 8192.0 || pairs > 1.5e8) return false;
  if (rows <= 4096.0) return true;
  // the useful part of what the pair kernel's busiest CTA would do, were they all that busy
  const double busiest = static_cast<double>(ceil_div(g.units, g.n_chunks)) * static_cast<double>(g.n_chunks);
  return real < 0.95 * busiest * static_cast<double>(p.i_tile()) * static_cast<double>(p.j_tile);
}

// ------------------------------------------------------------------ single-system force
// eps_i: the softening of each pair is its i-particle's, from the 4th slot
// of its record (eps2 is not used); the kernels then always take the s = 0
// guard.
cn_status force_common(bool dd, int64_t n_i, const float* pos_i, int64_t n_j, const float* pos_mass_j,
                       float eps2, void* acc_out, void* pot_out, void* ws, size_t ws_bytes, bool lib_ws,
                       cudaStream_t s, bool eps_i = false) {
  if (n_i < 0 || n_j < 0) return fail(CN_ERR_INVALID_ARG, "n_i and n_j must be >= 0");
  cn_status st;
  if (!eps_i && (st = check_eps2(eps2)) != CN_OK) return st;
  if ((st = check_records(pos_i, n_i, "pos_i")) != CN_OK) return st;
  if ((st = check_records(pos_mass_j, n_j, "pos_mass_j")) != CN_OK) return st;
  const size_t elt = dd ? sizeof(double) : sizeof(float);
  if (n_i > 0 && !acc_out) return fail(CN_ERR_INVALID_ARG, "acc_out is NULL");
  if ((acc_out && !aligned(acc_out, elt)) || (pot_out && !aligned(pot_out, elt)))
    return fail(CN_ERR_MISALIGNED, "outputs must be aligned to their element size");
  const size_t acc_b = static_cast<size_t>(n_i) * 3 * elt, pot_b = pot_out ? static_cast<size_t>(n_i) * elt : 0;
  const size_t pi_b = static_cast<size_t>(n_i) * 16, pj_b = static_cast<size_t>(n_j) * 16;
  if (overlaps(acc_out, acc_b, pos_i, pi_b) || overlaps(acc_out, acc_b, pos_mass_j, pj_b) ||
      overlaps(pot_out, pot_b, pos_i, pi_b) || overlaps(pot_out, pot_b, pos_mass_j, pj_b) ||
      overlaps(acc_out, acc_b, pot_out, pot_b))
    return fail(CN_ERR_INVALID_ARG, "outputs overlap inputs or each other");
  if (n_i == 0) return CN_OK;
  int dev = 0;
  DeviceInfo* d = nullptr;
  if ((st = current_device(&dev, &d)) != CN_OK) return st;
  cudaError_t e;
  if (n_j == 0) {
    if ((e = cudaMemsetAsync(acc_out, 0, acc_b, s)) != cudaSuccess) return fail_cuda(e, "cudaMemsetAsync");
    if (pot_out && (e = cudaMemsetAsync(pot_out, 0, pot_b, s)) != cudaSuccess) return fail_cuda(e, "cudaMemsetAsync");
    return CN_OK;
  }
  const bool pot = pot_out != nullptr;
  const bool guard = eps_i || needs_guard(eps2);
  const int variant = eps_i ? (pot ? cn::kF32EpsIPot : cn::kF32EpsI)
                            : (dd ? (pot ? cn::kDDPot : cn::kDD) : (pot ? cn::kF32Pot : cn::kF32));
  // One set against itself: each unordered pair once (the i record's 4th slot
  // is then the same mass the j side reads).
  const bool self = !dd && !eps_i && !guard && pos_i == pos_mass_j && n_i == n_j && sym_pays(cn::kSymForce, n_i, d->sms);
  const cn::RowForm row_form =
      eps_i ? (pot ? cn::kRowEpsIPot : cn::kRowEpsI) : (pot ? cn::kRowForcePot : cn::kRowForce);
  struct Cached {
    PlanCache key;
    bool sym = false;
    bool rows = false;
    SymPlan sp;
    RowPlan rp;
    Plan p;
    Geometry g;
    char* ctrl = nullptr;
    char* data = nullptr;
  };
  thread_local Cached t_last, t_now;  // of the last call; of a call that is planned anew
  const int key = variant + (self ? 64 : 0);
  const uint64_t gen0 = g_plan_gen.load(std::memory_order_acquire);
  const Cached* c = &t_last;
  if (!(lib_ws && t_last.key.hit(gen0, dev, key, n_i, n_j, guard, s))) {
    Cached& now = t_now = Cached{};
    c = &now;
    const uint64_t bumps0 = t_own_bumps;
    // the per-particle kernels are guarded in every shape, so K is not
    // restricted to 1. The one-sided plan is made in any case: it is what is
    // left when the symmetric form's slots cannot be had, and its kernel is
    // loaded with it.
    if ((st = resolve_plan(dev, variant, n_i, n_j, guard && !eps_i, nullptr, &now.p)) != CN_OK) return st;
    if ((st = single_geometry(dev, *d, variant, guard, now.p, n_i, n_j, &now.g)) != CN_OK) return st;
    std::optional<Attempt> attempt(std::in_place);
    bool wanted = self && !registered_tune(dev, variant, n_i, n_j, kTunedOneSet);
    const cn::SymForm form = pot ? cn::kSymForcePot : cn::kSymForce;
    if (wanted) wanted = sym_fit(dev, *d, form, n_i, false, sym_default_plan(form, n_i, d->sms), &now.sp) == CN_OK;
    if (wanted && lib_ws) {
      // not during a capture that would have to allocate, and not without memory
      now.sym = sym_workspace(s, now.sp.need, &now.sp.data) == CN_OK;
    } else if (wanted && ws && aligned(ws, 256) && ws_bytes >= std::max(now.sp.need, now.g.ws_bytes)) {
      now.sym = true;
      now.sp.data = static_cast<char*>(ws);
    }
    bool wanted_rows = !dd && (eps_i || !guard) && !self && rows_pays(row_form, n_i, n_j, d->sms, now.p, now.g) &&
                       !registered_tune(dev, variant, n_i, n_j, kTunedTwoSets);
    if (wanted_rows) wanted_rows = rows_fit(dev, *d, row_form, n_i, n_j, &now.rp) == CN_OK;
    if (wanted_rows && lib_ws) {
      now.rows = sym_workspace(s, now.rp.need, &now.data) == CN_OK;
    } else if (wanted_rows && ws && aligned(ws, 256) && ws_bytes >= std::max(now.rp.need, now.g.ws_bytes)) {
      now.rows = true;
      now.data = static_cast<char*>(ws);
    }
    // The library's workspace of the one-sided kernel is there after any call
    // of these sizes, also one that did without it: a capture may then make
    // a call that has to fall back on it.
    if (!now.sym && !now.rows) {
      attempt.reset();
      if ((st = launch_workspace(s, now.g, ws, ws_bytes, lib_ws, &now.ctrl, &now.data)) != CN_OK) return st;
    } else if (lib_ws) {
      char *ctrl = nullptr, *data = nullptr;
      library_workspace(s, now.g.ctrl_bytes, now.g.data_bytes, &ctrl, &data);
    }
    // cache only a plan that nothing changed under (another thread's tuning
    // or workspace change would show as a generation step not our own), and
    // not one that had to do without its slots
    const uint64_t gen1 = g_plan_gen.load(std::memory_order_acquire);
    if (lib_ws && now.sym == wanted && now.rows == wanted_rows && gen1 == gen0 + (t_own_bumps - bumps0)) {
      now.key = PlanCache{true, gen1, dev, key, n_i, n_j, guard, s};
      t_last = now;
    }
  }
  if (c->sym) {
    float* const out[3] = {static_cast<float*>(acc_out), static_cast<float*>(pot_out), nullptr};
    std::string what;
    if (log_enabled())
      what = std::string("cn_force: variant ") + variant_name(variant) + " n_i " + std::to_string(n_i) + " n_j " +
             std::to_string(n_j);
    return sym_launch(what, *d, pot ? cn::kSymForcePot : cn::kSymForce, c->sp, n_i, pos_i, nullptr, eps2, out, s);
  }
  if (c->rows) {
    std::string what;
    if (log_enabled())
      what = std::string(eps_i ? "cn_force_eps_i" : "cn_force") + ": variant " + variant_name(variant) + " n_i " +
             std::to_string(n_i) + " n_j " + std::to_string(n_j);
    return rows_launch(what, *d, row_form, c->rp, n_i, pos_i, n_j, pos_mass_j, eps2, static_cast<float*>(acc_out),
                       static_cast<float*>(pot_out), c->data, s);
  }
  const Plan& p = c->p;
  const Geometry& g = c->g;
  PairArgs a = base_args(c->ctrl, c->data, g, p, d->status);
  a.pos_i = reinterpret_cast<const float4*>(pos_i);
  a.pos_j = reinterpret_cast<const float4*>(pos_mass_j);
  a.acc_out = acc_out;
  a.pot_out = pot_out;
  a.n_i = n_i;
  a.n_j = n_j;
  a.eps2 = eps2;
  log_plan(dd ? "cn_force_dd" : (eps_i ? "cn_force_eps_i" : "cn_force"), variant, n_i, n_j, guard, p, g, g.njt);
  if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
  e = dd ? cn::launch_dd(a, p, pot, guard, g.grid, s) : cn::launch_f32(a, p, pot, guard, false, g.grid, s, eps_i);
  if (e != cudaSuccess) return fail_cuda(e, "pair kernel launch");
  return CN_OK;
}

// The symmetric plan of a jerk or adjoint call of one set against itself,
// with its workspace (extra: bytes after its slots, at data + need), or
// nullptr where the call takes the one-sided kernel: a small set, a
// registered tune, or no slots to be had (memory, a capture).
const SymPlan* sym_self_plan(int dev, const DeviceInfo& d, cn::SymForm form, int variant, int64_t n, size_t extra,
                             cudaStream_t s) {
  if (!sym_pays(form, n, d.sms)) return nullptr;
  thread_local SymPlan t_last;
  const uint64_t gen0 = g_plan_gen.load(std::memory_order_acquire);
  if (t_last.key.hit(gen0, dev, form, n, n, false, s)) return &t_last;
  if (registered_tune(dev, variant, n, n, kTunedOneSet)) return nullptr;
  const Attempt attempt;
  const uint64_t bumps0 = t_own_bumps;
  t_last.key.valid = false;
  if (sym_fit(dev, d, form, n, false, sym_default_plan(form, n, d.sms), &t_last) != CN_OK) return nullptr;
  if (sym_workspace(s, t_last.need + extra, &t_last.data) != CN_OK) return nullptr;
  // the one-sided kernel's workspace too, for a later call that has to fall back on it during a capture
  Plan one;
  Geometry g;
  char *ctrl = nullptr, *data = nullptr;
  if (resolve_plan(dev, variant, n, n, false, nullptr, &one) == CN_OK &&
      single_geometry(dev, d, variant, false, one, n, n, &g) == CN_OK)
    library_workspace(s, g.ctrl_bytes, g.data_bytes, &ctrl, &data);
  const uint64_t gen1 = g_plan_gen.load(std::memory_order_acquire);
  t_last.key = PlanCache{gen1 == gen0 + (t_own_bumps - bumps0), gen1, dev, form, n, n, false, s};
  return &t_last;
}

cn_status jerk_common(int64_t n_i, const float* pos_i, const float* vel_i, int64_t n_j, const float* pos_mass_j,
                      const float* vel_j, float eps2, float* acc_out, float* jerk_out, float* pot_out,
                      cudaStream_t s) {
  if (n_i < 0 || n_j < 0) return fail(CN_ERR_INVALID_ARG, "n_i and n_j must be >= 0");
  cn_status st;
  if ((st = check_eps2(eps2)) != CN_OK) return st;
  if ((st = check_records(pos_i, n_i, "pos_i")) != CN_OK) return st;
  if ((st = check_records(vel_i, n_i, "vel_i")) != CN_OK) return st;
  if ((st = check_records(pos_mass_j, n_j, "pos_mass_j")) != CN_OK) return st;
  if ((st = check_records(vel_j, n_j, "vel_j")) != CN_OK) return st;
  if (n_i > 0 && (!acc_out || !jerk_out)) return fail(CN_ERR_INVALID_ARG, "acc_out and jerk_out are required");
  if ((acc_out && !aligned(acc_out, 4)) || (jerk_out && !aligned(jerk_out, 4)) || (pot_out && !aligned(pot_out, 4)))
    return fail(CN_ERR_MISALIGNED, "outputs must be 4-byte aligned");
  const size_t ob = static_cast<size_t>(n_i) * 12, pb = pot_out ? static_cast<size_t>(n_i) * 4 : 0;
  const size_t ib = static_cast<size_t>(n_i) * 16, jb = static_cast<size_t>(n_j) * 16;
  const void* ins[4] = {pos_i, vel_i, pos_mass_j, vel_j};
  const size_t insz[4] = {ib, ib, jb, jb};
  const void* outs[3] = {acc_out, jerk_out, pot_out};
  const size_t outsz[3] = {ob, ob, pb};
  for (int o = 0; o < 3; ++o) {
    for (int q = 0; q < 4; ++q)
      if (overlaps(outs[o], outsz[o], ins[q], insz[q])) return fail(CN_ERR_INVALID_ARG, "outputs overlap inputs");
    for (int q = o + 1; q < 3; ++q)
      if (overlaps(outs[o], outsz[o], outs[q], outsz[q])) return fail(CN_ERR_INVALID_ARG, "outputs overlap each other");
  }
  if (n_i == 0) return CN_OK;
  int dev = 0;
  DeviceInfo* d = nullptr;
  if ((st = current_device(&dev, &d)) != CN_OK) return st;
  cudaError_t e;
  if (n_j == 0) {
    for (int o = 0; o < 3; ++o)
      if (outs[o] && (e = cudaMemsetAsync(const_cast<void*>(outs[o]), 0, outsz[o], s)) != cudaSuccess)
        return fail_cuda(e, "cudaMemsetAsync");
    return CN_OK;
  }
  const bool pot = pot_out != nullptr;
  const bool guard = needs_guard(eps2);
  const int variant = pot ? cn::kJerkPot : cn::kJerk;
  if (!guard && pos_i == pos_mass_j && vel_i == vel_j && n_i == n_j) {
    const cn::SymForm form = pot ? cn::kSymJerkPot : cn::kSymJerk;
    if (const SymPlan* sp = sym_self_plan(dev, *d, form, variant, n_i, 0, s)) {
      float* const out[3] = {acc_out, jerk_out, pot_out};
      std::string what;
      if (log_enabled()) what = std::string("cn_force_jerk: variant ") + variant_name(variant) + " n " + std::to_string(n_i);
      return sym_launch(what, *d, form, *sp, n_i, pos_i, vel_i, eps2, out, s);
    }
  }
  Plan p;
  if ((st = resolve_plan(dev, variant, n_i, n_j, guard, nullptr, &p)) != CN_OK) return st;
  Geometry g;
  if ((st = single_geometry(dev, *d, variant, guard, p, n_i, n_j, &g)) != CN_OK) return st;
  char *ctrl = nullptr, *data = nullptr;
  if ((st = library_workspace(s, g.ctrl_bytes, g.data_bytes, &ctrl, &data)) != CN_OK) return st;
  PairArgs a = base_args(ctrl, data, g, p, d->status);
  a.pos_i = reinterpret_cast<const float4*>(pos_i);
  a.pos_i2 = reinterpret_cast<const float4*>(vel_i);
  a.pos_j = reinterpret_cast<const float4*>(pos_mass_j);
  a.pos_j2 = reinterpret_cast<const float4*>(vel_j);
  a.acc_out = acc_out;
  a.jerk_out = jerk_out;
  a.pot_out = pot_out;
  a.n_i = n_i;
  a.n_j = n_j;
  a.eps2 = eps2;
  log_plan("cn_force_jerk", variant, n_i, n_j, guard, p, g, g.njt);
  if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
  e = cn::launch_jerk(a, p, pot, guard, g.grid, s);
  return e == cudaSuccess ? CN_OK : fail_cuda(e, "force-jerk kernel launch");
}

cn_status symmetric_common(int64_t n, const float* pos_mass, float eps2, float* acc_out, float* pot_out,
                           cudaStream_t s) {
  if (n < 0) return fail(CN_ERR_INVALID_ARG, "n must be >= 0");
  cn_status st;
  if ((st = check_eps2(eps2)) != CN_OK) return st;
  if ((st = check_records(pos_mass, n, "pos_mass")) != CN_OK) return st;
  if (n > 0 && !acc_out) return fail(CN_ERR_INVALID_ARG, "acc_out is NULL");
  if ((acc_out && !aligned(acc_out, 4)) || (pot_out && !aligned(pot_out, 4)))
    return fail(CN_ERR_MISALIGNED, "outputs must be 4-byte aligned");
  const size_t nb = static_cast<size_t>(n);
  if (overlaps(acc_out, nb * 12, pos_mass, nb * 16) || overlaps(pot_out, nb * 4, pos_mass, nb * 16) ||
      overlaps(acc_out, nb * 12, pot_out, nb * 4))
    return fail(CN_ERR_INVALID_ARG, "outputs overlap pos_mass or each other");
  const bool pot = pot_out != nullptr;
  if (n == 0) return CN_OK;
  int dev = 0;
  DeviceInfo* d = nullptr;
  if ((st = current_device(&dev, &d)) != CN_OK) return st;
  const bool guard = needs_guard(eps2);
  const cn::SymForm form = pot ? cn::kSymForcePot : cn::kSymForce;
  thread_local SymPlan t_last;
  const uint64_t gen0 = g_plan_gen.load(std::memory_order_acquire);
  if (!t_last.key.hit(gen0, dev, form, n, n, guard, s)) {
    const uint64_t bumps0 = t_own_bumps;
    cn_tune pot_tune{};
    const cn_tune* shape = nullptr;
    if (pot && !registered_tune(dev, cn::kSym, n, n, kTunedOneSet)) {
      pot_tune = sym_default_tune(n, d->sms, true);
      shape = &pot_tune;
    }
    Plan p;
    if ((st = resolve_plan(dev, cn::kSym, n, n, guard, shape, &p)) != CN_OK) return st;
    if (pot && !shape && sym_tile_bytes(p, true) > kMaxSmem)
      return fail(CN_ERR_INVALID_ARG, "the launch shape exceeds the shared memory of one CTA");
    t_last.key.valid = false;
    if ((st = sym_fit(dev, *d, form, n, guard, p, &t_last)) != CN_OK) return st;
    if ((st = sym_workspace(s, t_last.need, &t_last.data)) != CN_OK) return st;
    const uint64_t gen1 = g_plan_gen.load(std::memory_order_acquire);
    t_last.key = PlanCache{gen1 == gen0 + (t_own_bumps - bumps0), gen1, dev, form, n, n, guard, s};
  }
  float* const out[3] = {acc_out, pot_out, nullptr};
  const std::string what = log_enabled() ? "cn_force_symmetric: n " + std::to_string(n) : std::string();
  return sym_launch(what, *d, form, t_last, n, pos_mass, nullptr, eps2, out, s);
}

// ------------------------------------------------------------------ symmetric ensembles
cn_status launch_ensemble(const DeviceInfo& d, const cn_batch_plan* plan, const float* pos, float* acc_out,
                          float* pot_out, char* data, cudaStream_t s) {
  const cn::SymForm form = plan->pot ? cn::kSymBatchedPot : cn::kSymBatched;
  cn::SymArgs a{};
  a.g = plan->sym_grid;
  a.pos = reinterpret_cast<const float4*>(pos);
  a.slots_j = reinterpret_cast<float*>(data);
  a.slots_seg = reinterpret_cast<float*>(data + plan->sym_jslot_b);
  a.n_seg = plan->sym_seg;
  a.status = d.status;
  a.chunk = plan->sym_chunk;
  a.fold = cn::sym_ops(form).max_stage / cn::kSymBlock;
  a.stages = plan->sym_stages;
  a.wait_ns = g_wait_ns.load();
  a.rows = plan->d_rows;
  a.n_rows = plan->sym_rows;
  cn::SymMerge m{};
  m.g = a.g;
  m.slots_seg = a.slots_seg;
  m.slots_j = a.slots_j;
  m.out[0] = acc_out;
  m.out[1] = pot_out;
  m.tile = plan->sym_k * plan->sym_threads;
  m.first = m.last = 1;
  m.rows = plan->d_rows;
  m.blocks = plan->d_blocks;
  m.n_merge = plan->sym_merge;
  if (log_enabled())
    std::fprintf(stderr,
                 "[cunbody] cn_force_batched: variant %s n %lld clusters %d | symmetric: K %d threads %d chunk %d stages "
                 "%d | rows %d cost %lld grid %d smem %zu slots %zu bytes\n",
                 variant_name(plan->pot ? cn::kBatchedPot : cn::kBatched), static_cast<long long>(plan->n_total),
                 plan->n_clusters, plan->sym_k, plan->sym_threads, plan->sym_chunk, plan->sym_stages, plan->sym_rows,
                 static_cast<long long>(a.g.cost), a.g.grid, plan->sym_smem, plan->sym_bytes);
  if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
  std::lock_guard<std::recursive_mutex> order(launch_order(s));
  const cudaError_t e = cn::sym_ops(form).launch(a, m, plan->sym_k, false, plan->sym_threads, plan->sym_smem, s);
  return e == cudaSuccess ? CN_OK : fail_cuda(e, "symmetric ensemble launch");
}

cn_status run_batched(const cn_batch_plan* plan, const float* pos_i, const float* pos_j, float* acc_out,
                      float* pot_out, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!plan) return fail(CN_ERR_INVALID_ARG, "plan is NULL");
  cn_status st;
  if ((st = check_records(pos_i, plan->n_total, "pos_i")) != CN_OK) return st;
  if ((st = check_records(pos_j, plan->n_j_total, "pos_mass_j")) != CN_OK) return st;
  if (plan->n_total > 0 && !acc_out) return fail(CN_ERR_INVALID_ARG, "acc_out is NULL");
  if ((acc_out && !aligned(acc_out, 4)) || (pot_out && !aligned(pot_out, 4)))
    return fail(CN_ERR_MISALIGNED, "outputs must be 4-byte aligned");
  if (pot_out && !plan->pot) return fail(CN_ERR_INVALID_ARG, "plan was created without the potential form");
  const size_t n = static_cast<size_t>(plan->n_total), nj = static_cast<size_t>(plan->n_j_total);
  if (overlaps(acc_out, n * 12, pos_i, n * 16) || overlaps(pot_out, n * 4, pos_i, n * 16) ||
      overlaps(acc_out, n * 12, pos_j, nj * 16) || overlaps(pot_out, n * 4, pos_j, nj * 16) ||
      overlaps(acc_out, n * 12, pot_out, n * 4))
    return fail(CN_ERR_INVALID_ARG, "outputs overlap inputs or each other");
  int dev = 0;
  DeviceInfo* d = nullptr;
  if ((st = current_device(&dev, &d)) != CN_OK) return st;
  if (dev != plan->dev) return fail(CN_ERR_INVALID_ARG, "plan was built on another device");
  cudaError_t e;
  if (plan->units == 0 || plan->zero_first) {
    if (n && (e = cudaMemsetAsync(acc_out, 0, n * 12, s)) != cudaSuccess) return fail_cuda(e, "cudaMemsetAsync");
    if (n && pot_out && (e = cudaMemsetAsync(pot_out, 0, n * 4, s)) != cudaSuccess)
      return fail_cuda(e, "cudaMemsetAsync");
    if (plan->units == 0) return CN_OK;
  }
  if (plan->sym_rows > 0) {
    char* slots = nullptr;
    if (!ws) {
      const Attempt attempt;
      if (sym_workspace(s, plan->sym_bytes, &slots) != CN_OK) slots = nullptr;
    } else if (aligned(ws, 256) && ws_bytes >= std::max(plan->sym_bytes, plan->ws_bytes)) {
      slots = static_cast<char*>(ws);
    }
    if (slots) return launch_ensemble(*d, plan, pos_j, acc_out, pot_out, slots, s);
  }
  Geometry g;
  g.units = plan->units;
  g.n_chunks = plan->n_chunks;
  g.n_tiles = plan->n_tiles;
  g.ctrl_bytes = plan->ctrl_bytes;
  g.data_bytes = plan->data_bytes;
  g.ws_bytes = plan->ws_bytes;
  char *ctrl = nullptr, *data = nullptr;
  if ((st = launch_workspace(s, g, ws, ws_bytes, ws == nullptr, &ctrl, &data)) != CN_OK) return st;
  PairArgs a = base_args(ctrl, data, g, plan->plan, d->status);
  a.pos_i = reinterpret_cast<const float4*>(pos_i);
  a.pos_j = reinterpret_cast<const float4*>(pos_j);
  a.acc_out = acc_out;
  a.pot_out = pot_out;
  a.tiles = plan->d_tiles;
  a.n_i = plan->n_total;
  a.n_j = plan->n_j_total;
  a.j_index = plan->d_index;
  a.n_index = plan->n_index;
  if (log_enabled()) {
    Geometry lg = g;
    lg.grid = plan->grid;
    lg.smem = plan->d_index ? cn::gather_smem_bytes(plan->plan) : cn::ring_smem_bytes(plan->plan);
    log_plan(plan->lists ? (plan->d_index ? "cn_force_lists (index lists)" : "cn_force_lists") : "cn_force_batched",
             plan->pot ? cn::kBatchedPot : cn::kBatched, plan->n_total, plan->n_j_total, plan->guard, plan->plan, lg,
             0);
  }
  if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
  e = plan->d_index ? cn::launch_f32_gather(a, plan->plan, plan->pot, plan->guard, plan->grid, s)
                    : cn::launch_f32(a, plan->plan, plan->pot, plan->guard, true, plan->grid, s);
  if (e != cudaSuccess) return fail_cuda(e, "batched pair kernel launch");
  return CN_OK;
}

// One group of the work: i-particles [i_begin, i_begin + ni) against the j
// records [j_begin, j_begin + nj) with softening eps2.
struct Group {
  int64_t i_begin, ni, j_begin, nj;
  float eps2;
};

// The symmetric form of an ensemble: its shape by a model of its time, its
// table of rows and merge blocks, uploaded with the plan. Nothing is kept
// when the one-sided shape is expected to take less (`one_sided_s`), or when
// the slots would pass kSymEnsembleCap.
//
// The model is off-diagonal pairs / pairs + diagonal pairs / diag + fixed,
// padding counted as work (unordered pairs of whole 32-record blocks against
// whole tiles), least squares over 17 ensembles measured in every shape (8 ..
// 4096 clusters of 64 .. 65536; residuals 5-9%). Its choice is the fastest
// shape measured for 29 of the 34 (with and without the potential), 6% off at
// worst: 512 clusters of 256 .. 16384 8 x 128 4849 us (8 x 256 5010, 4 x 128
// 5274, one-sided 7010), 1000 of 1024 4 x 64 370 us (4 x 128 386, one-sided
// 428), 4096 of 256 one-sided 115 us (2 x 64 149).
constexpr size_t kSymEnsembleCap = static_cast<size_t>(1) << 30;

cn_status fit_ensemble(int dev, const DeviceInfo& d, const std::vector<Group>& groups, double one_sided_s,
                       cn_batch_plan* plan) {
  struct Shape {
    int k, threads, chunk;
    double pairs, diag, fixed_s;  // rates on 152 SMs
  };
  static const Shape plain[] = {{8, 256, 128, 2.15e12, 2.70e12, 16e-6}, {8, 128, 128, 2.06e12, 2.51e12, 20e-6},
                                {4, 128, 128, 1.81e12, 2.19e12, 13e-6}, {4, 64, 128, 1.70e12, 1.82e12, 14e-6},
                                {2, 128, 128, 1.45e12, 1.80e12, 9e-6},  {2, 64, 128, 1.32e12, 1.52e12, 11e-6}};
  static const Shape with_pot[] = {{8, 256, 64, 1.67e12, 2.12e12, 18e-6},  {8, 128, 128, 1.61e12, 1.95e12, 19e-6},
                                   {4, 128, 128, 1.46e12, 1.83e12, 15e-6}, {4, 64, 128, 1.24e12, 1.39e12, 16e-6},
                                   {2, 128, 128, 1.16e12, 1.54e12, 10e-6}, {2, 64, 128, 1.04e12, 1.34e12, 12e-6}};
  const cn::SymForm form = plan->pot ? cn::kSymBatchedPot : cn::kSymBatched;
  const cn::SymOps ops = cn::sym_ops(form);
  double best_s = one_sided_s;
  SymPlan best;
  for (const Shape& sh : plan->pot ? with_pot : plain) {
    SymPlan sp;
    sp.k = sh.k;
    sp.threads = sh.threads;
    sp.chunk = sh.chunk;
    sp.stages = 3;
    sp.tile = static_cast<int64_t>(sh.k) * sh.threads;
    sp.smem = ops.smem(sp.threads, sp.k, sp.chunk, sp.stages);
    const double block = static_cast<double>(sp.tile) * cn::kSymBlock;
    double work_s = 0.0, bytes = 0.0;
    for (const Group& gr : groups) {
      const int64_t tb = sp.tile / cn::kSymBlock, nb = ceil_div(gr.ni, cn::kSymBlock), t = ceil_div(nb, tb);
      // blocks behind the diagonal tiles of all the cluster's rows
      const double off = static_cast<double>(t) * nb - static_cast<double>(tb) * (static_cast<double>(t) * (t + 1) / 2) +
                         static_cast<double>(t * tb - nb);
      work_s += block * (off / sh.pairs + static_cast<double>(nb) / sh.diag);
      bytes += off * cn::kSymBlock * 4.0 * ops.sums;
    }
    const double time_s = work_s * 152.0 / d.sms + sh.fixed_s;
    if (bytes <= static_cast<double>(kSymEnsembleCap) && time_s < best_s) {
      best_s = time_s;
      best = sp;
    }
  }
  if (best.k == 0) return CN_OK;
  int occ = 0;
  cn_status st = sym_occupancy(dev, form, best, &occ);
  if (st != CN_OK) return st;
  best.slots = static_cast<int64_t>(occ) * d.sms;
  std::vector<cn::SymRow> rows;
  std::vector<cn::SymMergeBlock> blocks;
  const int64_t tb = best.tile / cn::kSymBlock;
  int64_t cost = 0, slot = 0;
  for (const Group& gr : groups) {
    if (gr.ni == 0) continue;
    const int64_t nb = ceil_div(gr.ni, cn::kSymBlock);
    const size_t first = rows.size();
    for (int64_t b0 = 0; b0 < nb; b0 += tb) {
      cn::SymRow r{};
      r.cost = cost;
      r.p0 = gr.i_begin;
      r.slot = slot;
      r.n = static_cast<int32_t>(gr.ni);
      r.n_blocks = static_cast<int32_t>(nb);
      r.blk0 = static_cast<int32_t>(b0);
      r.diag_end = static_cast<int32_t>(std::min(nb, b0 + tb));
      r.plane = static_cast<int32_t>((nb - r.diag_end) * cn::kSymBlock);
      r.eps2 = gr.eps2;
      cost += r.length();
      slot += static_cast<int64_t>(r.plane) * ops.sums;
      rows.push_back(r);
    }
    for (int64_t b = 0; b < nb; ++b)
      blocks.push_back(cn::SymMergeBlock{static_cast<int32_t>(first), static_cast<int32_t>(first + b / tb),
                                         static_cast<int32_t>(b)});
  }
  if (rows.empty() || rows.size() > static_cast<size_t>(INT32_MAX) || blocks.size() > static_cast<size_t>(INT32_MAX))
    return CN_OK;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&plan->d_rows), rows.size() * sizeof(cn::SymRow));
  if (e == cudaSuccess)
    e = cudaMalloc(reinterpret_cast<void**>(&plan->d_blocks), blocks.size() * sizeof(cn::SymMergeBlock));
  if (e == cudaSuccess)
    e = cudaMemcpy(plan->d_rows, rows.data(), rows.size() * sizeof(cn::SymRow), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(plan->d_blocks, blocks.data(), blocks.size() * sizeof(cn::SymMergeBlock), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cudaFree(plan->d_rows);
    cudaFree(plan->d_blocks);
    plan->d_rows = nullptr;
    plan->d_blocks = nullptr;
    cudaGetLastError();  // the plan goes on without them
    return fail_cuda(e, "uploading the ensemble's rows");
  }
  plan->sym_k = best.k;
  plan->sym_threads = best.threads;
  plan->sym_chunk = best.chunk;
  plan->sym_stages = best.stages;
  plan->sym_smem = best.smem;
  plan->sym_grid.n = plan->n_total;
  plan->sym_grid.cost = cost;
  plan->sym_grid.grid = static_cast<int32_t>(std::max<int64_t>(1, std::min<int64_t>(best.slots, cost / cn::kSymCostPair)));
  plan->sym_seg = plan->sym_grid.grid + static_cast<int64_t>(rows.size());
  plan->sym_jslot_b = align_up(static_cast<size_t>(slot) * sizeof(float), 256);
  plan->sym_bytes =
      plan->sym_jslot_b + static_cast<size_t>(plan->sym_seg) * best.tile * sizeof(float) * static_cast<size_t>(ops.sums);
  plan->sym_merge = static_cast<int32_t>(blocks.size());
  plan->sym_rows = static_cast<int32_t>(rows.size());
  return CN_OK;
}

// Builds the (group, i-tile, j-tile) unit table of a plan and uploads it.
// index_host (gathering list plans): n_index list entries, each the index of
// a j record; the groups' j ranges then count entries of this array.
cn_status build_group_plan(const std::vector<Group>& groups, bool lists, int64_t n_i_total, int64_t n_j_total,
                           const cn_tune* tune, int with_pot, cn_batch_plan** out, const int32_t* index_host = nullptr,
                           int64_t n_index = 0) {
  const bool gather = index_host != nullptr;
  bool guard = false, zero_first = false;
  double pairs = 0.0;
  for (const Group& gr : groups) {
    cn_status st = check_eps2(gr.eps2);
    if (st != CN_OK) return st;
    if (gr.ni > 0 && gr.nj > 0 && needs_guard(gr.eps2)) guard = true;
    if (gr.ni > 0 && gr.nj == 0) zero_first = true;
    pairs += static_cast<double>(gr.ni) * static_cast<double>(gr.nj);
  }
  int dev = 0;
  DeviceInfo* d = nullptr;
  cn_status st = current_device(&dev, &d);
  if (st != CN_OK) return st;
  const int variant = with_pot ? cn::kBatchedPot : cn::kBatched;
  const int64_t key_i = static_cast<int64_t>(groups.size());
  cn_tune fitted{};
  double one_sided_s = 0.0;
  if (!tune && !registered_tune(dev, variant, key_i, n_i_total, kTunedAny)) {
    // i-tile fitted to the group sizes: every group is cut into whole i-tiles,
    // so a tile larger than the typical group leaves lanes idle, and every
    // j range into whole j-tiles (padded with zero masses). Among the
    // shapes below take the one with the least evaluated-but-padded work,
    // weighted by each shape's relative pair rate, measured on GB300: the
    // packed K = 8 kernel 1.0, its split-j forms 0.95, K = 4 0.99, K = 2 x
    // 128 0.93, one particle per thread 0.80. Ensembles (eight of them, 64 ..
    // 65536 particles per cluster) add K = 4 x 64 at 0.99, ahead of 4 x 128
    // (the same rate with half the i-tile), K = 2 x 64 with 128-record
    // j-tiles at 0.93 (clusters of a few hundred), and rate the 128-thread split-j
    // form 0.75 (0.29 against 0.67 of the FP32 bound for 4096 clusters of
    // 256); interaction lists keep their measured set (groups of 256 against
    // 4096-record lists: the 256-thread split-j form 0.72, 4 x 64 below 0.70).
    struct Cand {
      int k, threads, j_lanes, j_tile;
      double rate;
      int use;  // 1: ensembles, 2: lists, 3: both
    };
    static const Cand cands[] = {{8, 256, 1, 512, 1.0, 3},   {8, 256, 2, 512, 0.95, 3}, {8, 256, 4, 512, 0.95, 3},
                                 {8, 256, 8, 512, 0.95, 3},  {8, 128, 8, 512, 0.94, 2}, {8, 128, 8, 512, 0.75, 1},
                                 {4, 64, 1, 256, 0.99, 1},   {4, 128, 1, 256, 0.99, 3}, {2, 128, 1, 256, 0.93, 3},
                                 {2, 64, 1, 128, 0.93, 1},   {1, 128, 1, 256, 0.80, 3}};
    double best = -1.0;
    for (const Cand& c : cands) {
      if (!(c.use & (lists ? 2 : 1))) continue;
      if (guard && (c.j_lanes > 1 || c.k > 1)) continue;  // the guarded kernels hold one particle, no split-j
      const int64_t it = static_cast<int64_t>(c.k) * c.threads / c.j_lanes;
      double padded = 0.0;
      for (const Group& gr : groups)
        padded += static_cast<double>(ceil_div(gr.ni, it) * it) * static_cast<double>(ceil_div(gr.nj, c.j_tile) * c.j_tile);
      const double score = padded > 0.0 ? pairs / padded * c.rate : c.rate;
      if (score > best) {
        best = score;
        fitted = default_tune(variant, key_i, n_i_total, d->sms);
        fitted.i_per_thread = c.k;
        fitted.threads = c.threads;
        fitted.j_lanes = c.j_lanes;
        fitted.j_tile = c.j_tile;
      }
    }
    // with the potential the K = 8 split-j kernel runs short of registers:
    // K = 4 with half the lane groups keeps the i-tile (lists of 4096 records
    // for groups of 256: 0.525 -> 0.712 of the 14-operation bound); the
    // gathering kernel, whose threads also stage records, does the same
    // (0.651 -> 0.673 of the FP32 bound on those lists as index arrays)
    if ((with_pot || gather) && fitted.i_per_thread == 8 && fitted.j_lanes > 1) {
      fitted.i_per_thread = 4;
      fitted.j_lanes /= 2;
      if (fitted.j_lanes < 2) fitted.j_lanes = 0;
    }
    tune = &fitted;
    // that shape's expected time: 0.78 of the FP32 bound times its score, 14
    // operations with the potential, and 10 us (4096 clusters of 256: 113 us
    // against 115 measured, 512 of 256 .. 16384: 7.4 ms against 7.0)
    one_sided_s =
        10e-6 + pairs / (std::max(best, 1e-3) * 0.78 * 3.356e12 * (with_pot ? 12.0 / 14.0 : 1.0) * d->sms / 152.0);
  }
  Plan p;
  if ((st = resolve_plan(dev, variant, key_i, n_i_total, guard, tune, &p)) != CN_OK) return st;
  // split-j batched kernels exist for K = 2, 4, 8 without the s = 0 guard
  if (p.j_lanes > 1 && (guard || p.k < 2)) p.j_lanes = 1;
  // tiles in order of decreasing work (largest first for the dynamic queue)
  std::vector<size_t> order(groups.size());
  for (size_t c = 0; c < groups.size(); ++c) order[c] = c;
  std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) {
    return groups[x].ni * groups[x].nj > groups[y].ni * groups[y].nj;
  });
  std::vector<cn::TileDesc> tiles;
  int64_t units = 0;
  const int it = p.i_tile();
  for (size_t c : order) {
    const Group& gr = groups[c];
    if (gr.ni == 0 || gr.nj == 0) continue;
    const int64_t njt = ceil_div(gr.nj, p.j_tile);
    if (njt > INT32_MAX) return fail(CN_ERR_INVALID_ARG, "a j set is too large");
    for (int64_t i0 = 0; i0 < gr.ni; i0 += it) {
      cn::TileDesc t{};
      t.i0 = gr.i_begin + i0;
      t.j0 = gr.j_begin;
      t.nj = gr.nj;
      t.unit0 = units;
      t.ni = static_cast<int32_t>(std::min<int64_t>(it, gr.ni - i0));
      t.njt = static_cast<int32_t>(njt);
      t.eps2 = gr.eps2;
      tiles.push_back(t);
      units += njt;
    }
  }
  Geometry g;
  if (!tiles.empty() &&
      (st = layout(dev, *d, variant, guard, p, static_cast<int64_t>(tiles.size()), units, 0, &g, gather)) != CN_OK)
    return st;
  // Ragged ensembles (cluster sizes spanning 4x or more) with the fitted
  // shape and many units per resident CTA take the dynamic queue in chunks
  // of 32 units (measured: 0.74 -> 0.78 of the FP32 bound on 512 clusters
  // of 256 .. 16384, 0.60 -> 0.63 on 2048 of 256 .. 2048, 0.77 -> 0.81 on
  // 256 of 128 .. 65536). Equal clusters keep the static schedule (1000 of
  // 1024: 0.73 static, 0.62 dynamic; 64 of 16384: 0.83 static, 0.72
  // dynamic), and so do launches with few units per slot, where the chunks
  // leave CTAs idle.
  int64_t ni_min = INT64_MAX, ni_max = 0;
  for (const Group& gr : groups)
    if (gr.ni > 0 && gr.nj > 0) {
      ni_min = std::min(ni_min, gr.ni);
      ni_max = std::max(ni_max, gr.ni);
    }
  if (!lists && tune == &fitted && !tiles.empty() && p.chunk_units == 0 && ni_max >= 4 * ni_min &&
      units >= 20 * static_cast<int64_t>(g.grid)) {
    p.chunk_units = 32;
    if ((st = layout(dev, *d, variant, guard, p, static_cast<int64_t>(tiles.size()), units, 0, &g, gather)) != CN_OK)
      return st;
  }
  auto* plan = new cn_batch_plan();
  plan->dev = dev;
  plan->lists = lists;
  plan->zero_first = zero_first;
  plan->n_clusters = static_cast<int32_t>(groups.size());
  plan->n_total = n_i_total;
  plan->n_j_total = n_j_total;
  plan->pairs = pairs;
  plan->plan = p;
  plan->guard = guard;
  plan->pot = with_pot != 0;
  plan->n_tiles = static_cast<int32_t>(tiles.size());
  plan->units = units;
  plan->n_chunks = g.n_chunks;
  plan->grid = g.grid;
  plan->ws_bytes = tiles.empty() ? 0 : g.ws_bytes;
  plan->ctrl_bytes = g.ctrl_bytes;
  plan->data_bytes = g.data_bytes;
  if (!tiles.empty()) {
    if (inject("alloc")) {
      delete plan;
      return fail(CN_ERR_CUDA, "cudaMalloc: injected allocation failure");
    }
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&plan->d_tiles), tiles.size() * sizeof(cn::TileDesc));
    if (e == cudaSuccess)
      e = cudaMemcpy(plan->d_tiles, tiles.data(), tiles.size() * sizeof(cn::TileDesc), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && gather) {
      plan->n_index = n_index;
      e = cudaMalloc(reinterpret_cast<void**>(&plan->d_index), static_cast<size_t>(n_index) * sizeof(int32_t));
      if (e == cudaSuccess)
        e = cudaMemcpy(plan->d_index, index_host, static_cast<size_t>(n_index) * sizeof(int32_t),
                       cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
      cudaFree(plan->d_tiles);
      cudaFree(plan->d_index);
      delete plan;
      return fail_cuda(e, "uploading the batched unit table");
    }
  }
  // an ensemble in its default shape: the symmetric form too, where it is
  // expected to be the faster one (a plan without it when its table cannot be had)
  if (!lists && !guard && tune == &fitted && !tiles.empty()) {
    const Attempt attempt;
    fit_ensemble(dev, *d, groups, one_sided_s, plan);
  }
  *out = plan;
  return CN_OK;
}

cn_status build_batch_plan(int32_t n_clusters, const int64_t* offsets, const float* eps2, const cn_tune* tune,
                           int with_pot, cn_batch_plan** out) {
  if (!out) return fail(CN_ERR_INVALID_ARG, "plan_out is NULL");
  *out = nullptr;
  if (n_clusters < 0 || (n_clusters > 0 && (!offsets || !eps2)))
    return fail(CN_ERR_INVALID_ARG, "n_clusters < 0 or NULL offsets/eps2");
  if (n_clusters > 0 && offsets[0] != 0) return fail(CN_ERR_INVALID_ARG, "offsets[0] must be 0");
  std::vector<Group> groups(static_cast<size_t>(n_clusters));
  for (int32_t c = 0; c < n_clusters; ++c) {
    if (offsets[c + 1] < offsets[c]) return fail(CN_ERR_INVALID_ARG, "offsets must be non-decreasing");
    const int64_t nc = offsets[c + 1] - offsets[c];
    groups[c] = Group{offsets[c], nc, offsets[c], nc, eps2[c]};
  }
  const int64_t n_total = n_clusters > 0 ? offsets[n_clusters] : 0;
  if (inject("hostmem")) throw std::bad_alloc();
  return build_group_plan(groups, false, n_total, n_total, tune, with_pot, out);
}

cn_status build_list_plan(int32_t n_groups, const int64_t* i_offsets, const int64_t* j_begin, const int64_t* j_count,
                          const float* eps2, const cn_tune* tune, int with_pot, cn_batch_plan** out) {
  if (!out) return fail(CN_ERR_INVALID_ARG, "plan_out is NULL");
  *out = nullptr;
  if (n_groups < 0 || (n_groups > 0 && (!i_offsets || !j_begin || !j_count || !eps2)))
    return fail(CN_ERR_INVALID_ARG, "n_groups < 0 or a NULL array");
  if (n_groups > 0 && i_offsets[0] != 0) return fail(CN_ERR_INVALID_ARG, "i_offsets[0] must be 0");
  std::vector<Group> groups(static_cast<size_t>(n_groups));
  int64_t n_j_total = 0;
  for (int32_t c = 0; c < n_groups; ++c) {
    if (i_offsets[c + 1] < i_offsets[c]) return fail(CN_ERR_INVALID_ARG, "i_offsets must be non-decreasing");
    if (j_begin[c] < 0 || j_count[c] < 0) return fail(CN_ERR_INVALID_ARG, "negative list begin or count");
    groups[c] = Group{i_offsets[c], i_offsets[c + 1] - i_offsets[c], j_begin[c], j_count[c], eps2[c]};
    if (j_count[c] > 0) n_j_total = std::max(n_j_total, j_begin[c] + j_count[c]);
  }
  const int64_t n_i_total = n_groups > 0 ? i_offsets[n_groups] : 0;
  if (inject("hostmem")) throw std::bad_alloc();
  return build_group_plan(groups, true, n_i_total, n_j_total, tune, with_pot, out);
}

// Gathering list plan: group g's list is the entries j_begin[g] ..
// j_begin[g] + j_count[g] - 1 of j_index, each the index of one of n_src
// records. Every entry a list reaches is checked here, on the host.
cn_status build_list_plan_indexed(int32_t n_groups, const int64_t* i_offsets, const int64_t* j_begin,
                                  const int64_t* j_count, const float* eps2, const int32_t* j_index, int64_t n_index,
                                  int64_t n_src, const cn_tune* tune, int with_pot, cn_batch_plan** out) {
  if (!out) return fail(CN_ERR_INVALID_ARG, "plan_out is NULL");
  *out = nullptr;
  if (n_groups < 0 || (n_groups > 0 && (!i_offsets || !j_begin || !j_count || !eps2)))
    return fail(CN_ERR_INVALID_ARG, "n_groups < 0 or a NULL array");
  if (n_index < 0 || n_src < 0 || (n_index > 0 && !j_index))
    return fail(CN_ERR_INVALID_ARG, "n_index < 0, n_src < 0 or a NULL j_index");
  if (n_src > INT32_MAX) return fail(CN_ERR_INVALID_ARG, "n_src exceeds the 32-bit index range");
  if (n_groups > 0 && i_offsets[0] != 0) return fail(CN_ERR_INVALID_ARG, "i_offsets[0] must be 0");
  std::vector<Group> groups(static_cast<size_t>(n_groups));
  std::vector<char> reached(static_cast<size_t>(n_index), 0);
  for (int32_t c = 0; c < n_groups; ++c) {
    if (i_offsets[c + 1] < i_offsets[c]) return fail(CN_ERR_INVALID_ARG, "i_offsets must be non-decreasing");
    if (j_begin[c] < 0 || j_count[c] < 0) return fail(CN_ERR_INVALID_ARG, "negative list begin or count");
    if (j_count[c] > 0 && j_begin[c] + j_count[c] > n_index)
      return fail(CN_ERR_INVALID_ARG, "a list runs past the end of j_index");
    groups[c] = Group{i_offsets[c], i_offsets[c + 1] - i_offsets[c], j_begin[c], j_count[c], eps2[c]};
    if (groups[c].ni > 0)
      for (int64_t e = j_begin[c]; e < j_begin[c] + j_count[c]; ++e) reached[static_cast<size_t>(e)] = 1;
  }
  for (int64_t e = 0; e < n_index; ++e)
    if (reached[static_cast<size_t>(e)] && (j_index[e] < 0 || j_index[e] >= n_src))
      return fail(CN_ERR_INVALID_ARG, "a j_index entry lies outside 0 .. n_src - 1");
  const int64_t n_i_total = n_groups > 0 ? i_offsets[n_groups] : 0;
  if (inject("hostmem")) throw std::bad_alloc();
  return build_group_plan(groups, true, n_i_total, n_src, tune, with_pot, out, j_index != nullptr ? j_index : &kNoIndex,
                          n_index);
}

// Host staging buffers of cn_force_host, per (device, stream).
struct HostStage {
  void* buf = nullptr;
  size_t bytes = 0;
};
std::map<std::pair<int, cudaStream_t>, HostStage> g_stage;

cn_status stage_buffer(cudaStream_t s, size_t need, void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
  std::lock_guard<std::mutex> lock(g_mu);
  HostStage& h = g_stage[{dev, s}];
  if (h.bytes < need) {
    if (inject("alloc")) return fail(CN_ERR_CUDA, "cudaMalloc: injected allocation failure");
    if (h.buf) {
      if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail_cuda(e, "cudaStreamSynchronize");
      cudaFree(h.buf);
      h.buf = nullptr;
      h.bytes = 0;
    }
    const size_t nb = align_up(need, static_cast<size_t>(1) << 20);
    if ((e = cudaMalloc(&h.buf, nb)) != cudaSuccess) return fail_cuda(e, "cudaMalloc(staging)");
    h.bytes = nb;
  }
  *out = h.buf;
  return CN_OK;
}

cn_status energy_common(int64_t n, const float* pos_mass, const float* pot_f, const double* pot_d, double* w_out,
                        cudaStream_t s) {
  if (n < 0) return fail(CN_ERR_INVALID_ARG, "n must be >= 0");
  if (!w_out || !aligned(w_out, 8)) return fail(CN_ERR_INVALID_ARG, "w_out must be a non-NULL aligned double pointer");
  cn_status st = check_records(pos_mass, n, "pos_mass");
  if (st != CN_OK) return st;
  if (n > 0 && !pot_f && !pot_d) return fail(CN_ERR_INVALID_ARG, "pot is NULL");
  int dev = 0;
  DeviceInfo* d = nullptr;
  if ((st = current_device(&dev, &d)) != CN_OK) return st;
  if (n == 0) {
    cudaError_t e = cudaMemsetAsync(w_out, 0, sizeof(double), s);
    return e == cudaSuccess ? CN_OK : fail_cuda(e, "cudaMemsetAsync");
  }
  double* aux = nullptr;
  if ((st = library_aux(s, &aux)) != CN_OK) return st;
  const size_t nb = cn::energy_workspace_doubles();
  if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
  cudaError_t e = cn::launch_energy(n, reinterpret_cast<const float4*>(pos_mass), pot_f, pot_d, aux,
                                    reinterpret_cast<int*>(aux + nb), w_out, s);
  return e == cudaSuccess ? CN_OK : fail_cuda(e, "potential-energy kernel launch");
}

// ------------------------------------------------------------------ tuning file
// A small reader for the JSON the library writes (objects, arrays, strings
// without escapes other than \" and \\, integers, true/false/null).
struct JsonValue {
  enum Kind { kNull, kBool, kNumber, kString, kArray, kObject } kind = kNull;
  double number = 0.0;
  bool boolean = false;
  std::string text;
  std::vector<JsonValue> items;
  std::vector<std::pair<std::string, JsonValue>> fields;
  const JsonValue* get(const char* key) const {
    for (const auto& f : fields)
      if (f.first == key) return &f.second;
    return nullptr;
  }
};

struct JsonReader {
  const std::string& src;
  size_t pos = 0;
  int depth = 0;
  void skip() {
    while (pos < src.size() && (src[pos] == ' ' || src[pos] == '\n' || src[pos] == '\r' || src[pos] == '\t')) ++pos;
  }
  bool literal(const char* word) {
    const size_t n = std::strlen(word);
    if (src.compare(pos, n, word) != 0) return false;
    pos += n;
    return true;
  }
  bool string(std::string* out) {
    if (pos >= src.size() || src[pos] != '"') return false;
    ++pos;
    out->clear();
    while (pos < src.size() && src[pos] != '"') {
      char c = src[pos++];
      if (c == '\\') {
        if (pos >= src.size()) return false;
        c = src[pos++];
        if (c != '"' && c != '\\' && c != '/') return false;
      }
      out->push_back(c);
    }
    if (pos >= src.size()) return false;
    ++pos;
    return true;
  }
  bool value(JsonValue* v) {
    if (++depth > 16) return false;
    skip();
    bool ok = false;
    if (pos >= src.size()) {
      ok = false;
    } else if (src[pos] == '{') {
      v->kind = JsonValue::kObject;
      ++pos;
      skip();
      if (pos < src.size() && src[pos] == '}') {
        ++pos;
        ok = true;
      } else {
        for (;;) {
          skip();
          std::pair<std::string, JsonValue> f;
          if (!string(&f.first)) break;
          skip();
          if (pos >= src.size() || src[pos] != ':') break;
          ++pos;
          if (!value(&f.second)) break;
          v->fields.push_back(std::move(f));
          skip();
          if (pos < src.size() && src[pos] == ',') {
            ++pos;
            continue;
          }
          if (pos < src.size() && src[pos] == '}') {
            ++pos;
            ok = true;
          }
          break;
        }
      }
    } else if (src[pos] == '[') {
      v->kind = JsonValue::kArray;
      ++pos;
      skip();
      if (pos < src.size() && src[pos] == ']') {
        ++pos;
        ok = true;
      } else {
        for (;;) {
          JsonValue item;
          if (!value(&item)) break;
          v->items.push_back(std::move(item));
          skip();
          if (pos < src.size() && src[pos] == ',') {
            ++pos;
            continue;
          }
          if (pos < src.size() && src[pos] == ']') {
            ++pos;
            ok = true;
          }
          break;
        }
      }
    } else if (src[pos] == '"') {
      v->kind = JsonValue::kString;
      ok = string(&v->text);
    } else if (literal("true")) {
      v->kind = JsonValue::kBool;
      v->boolean = true;
      ok = true;
    } else if (literal("false")) {
      v->kind = JsonValue::kBool;
      ok = true;
    } else if (literal("null")) {
      ok = true;
    } else {
      const char* start = src.c_str() + pos;
      char* end = nullptr;
      v->number = std::strtod(start, &end);
      if (end != start) {
        v->kind = JsonValue::kNumber;
        pos += static_cast<size_t>(end - start);
        ok = std::isfinite(v->number);
      }
    }
    --depth;
    return ok;
  }
};

int variant_from_name(const std::string& name) {
  for (int v = 0; v < 12; ++v)
    if (name == variant_name(v)) return v;
  return -1;
}

bool json_int(const JsonValue& o, const char* key, int64_t lo, int64_t hi, int64_t* out) {
  const JsonValue* v = o.get(key);
  if (!v || v->kind != JsonValue::kNumber || v->number != std::floor(v->number) || v->number < static_cast<double>(lo) ||
      v->number > static_cast<double>(hi))
    return false;
  *out = static_cast<int64_t>(v->number);
  return true;
}

cn_status device_identity(int dev, std::string* name, std::string* arch, int* sms) {
  cudaDeviceProp prop{};
  const cudaError_t e = cudaGetDeviceProperties(&prop, dev);
  if (e != cudaSuccess) return fail_cuda(e, "cudaGetDeviceProperties");
  *name = prop.name;
  *arch = "sm_" + std::to_string(prop.major) + std::to_string(prop.minor);
  *sms = prop.multiProcessorCount;
  return CN_OK;
}

}  // namespace

namespace cn {
// cn_force on a workspace the caller supplies, without touching the
// library-owned workspaces (used by the static-scratch entry point).
cn_status force_f32_on_workspace(int64_t n_i, const float* pos_i, int64_t n_j, const float* pos_mass_j, float eps2,
                                 float* acc_out, float* pot_out, void* ws, size_t ws_bytes, cudaStream_t s) {
  return force_common(false, n_i, pos_i, n_j, pos_mass_j, eps2, acc_out, pot_out, ws, ws_bytes, false, s);
}
// Workspace bytes of a call of `variant` in its one-sided form.
size_t one_sided_workspace_bytes(int variant, int64_t n_i, int64_t n_j) {
  if (n_i <= 0 || n_j <= 0 || variant < kF32 || variant > kF32EpsIPot || variant == kBatched || variant == kBatchedPot ||
      variant == kSym)
    return 0;
  int dev = 0;
  DeviceInfo* d = nullptr;
  if (current_device(&dev, &d) != CN_OK) return 0;
  Plan p;
  if (resolve_plan(dev, variant, n_i, n_j, false, nullptr, &p) != CN_OK) return 0;
  Geometry g;
  if (single_geometry(dev, *d, variant, false, p, n_i, n_j, &g) != CN_OK) return 0;
  // the guarded (eps2 = 0) shape uses one i-particle per thread: size for the larger of the two
  Plan pg = p;
  pg.k = 1;
  Geometry gg;
  if (single_geometry(dev, *d, variant, true, pg, n_i, n_j, &gg) != CN_OK) return g.ws_bytes;
  return std::max(g.ws_bytes, gg.ws_bytes);
}
cn_status set_error(cn_status st, const std::string& msg) { return fail(st, msg); }

cn_status fail_nothrow(cn_status st, const char* msg) noexcept {
  try {
    g_last_error = msg;
  } catch (...) {
    g_last_error.clear();  // no room even for the message
  }
  return st;
}
}  // namespace cn

// ====================================================================== C ABI
extern "C" {

cn_status cn_force(int64_t n_i, const float* pos_i, int64_t n_j, const float* pos_mass_j, float eps2, float* acc_out,
                   float* pot_out, cn_stream stream) {
  NvtxRange nvtx_range("cn_force");
  return cn::guard([&]() -> cn_status {
    return force_common(false, n_i, pos_i, n_j, pos_mass_j, eps2, acc_out, pot_out, nullptr, 0, true,
                        reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_force_eps_i(int64_t n_i, const float* pos_eps_i, int64_t n_j, const float* pos_mass_j, float* acc_out,
                         float* pot_out, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_eps_i");
  return cn::guard([&]() -> cn_status {
    return force_common(false, n_i, pos_eps_i, n_j, pos_mass_j, 0.f, acc_out, pot_out, nullptr, 0, true,
                        reinterpret_cast<cudaStream_t>(stream), true);
  });
}

cn_status cn_force_ws(int64_t n_i, const float* pos_i, int64_t n_j, const float* pos_mass_j, float eps2,
                      float* acc_out, float* pot_out, void* workspace, size_t ws_bytes, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_ws");
  return cn::guard([&]() -> cn_status {
    return force_common(false, n_i, pos_i, n_j, pos_mass_j, eps2, acc_out, pot_out, workspace, ws_bytes, false,
                        reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_force_dd(int64_t n_i, const float* pos_i, int64_t n_j, const float* pos_mass_j, float eps2,
                      double* acc_out, double* pot_out, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_dd");
  return cn::guard([&]() -> cn_status {
    return force_common(true, n_i, pos_i, n_j, pos_mass_j, eps2, acc_out, pot_out, nullptr, 0, true,
                        reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_force_dd_ws(int64_t n_i, const float* pos_i, int64_t n_j, const float* pos_mass_j, float eps2,
                         double* acc_out, double* pot_out, void* workspace, size_t ws_bytes, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_dd_ws");
  return cn::guard([&]() -> cn_status {
    return force_common(true, n_i, pos_i, n_j, pos_mass_j, eps2, acc_out, pot_out, workspace, ws_bytes, false,
                        reinterpret_cast<cudaStream_t>(stream));
  });
}

size_t cn_workspace_bytes(int variant, int64_t n_i, int64_t n_j) {
  return cn::guard_value<size_t>(0, [&]() -> size_t {
    size_t need = cn::one_sided_workspace_bytes(variant, n_i, n_j);
    if (need != 0 && (variant == cn::kDD || variant == cn::kDDPot)) {
      // enough for any part of these sets too: the small shapes' j-tiles are
      // fitted to the sizes, so a smaller call may be cut into more units. None
      // has more than tiles of 64 by 32.
      int dev = 0;
      DeviceInfo* d = nullptr;
      Plan p;
      p.k = 1;
      p.threads = 64;
      p.j_tile = 32;
      p.stages = 4;
      Geometry g;
      if (current_device(&dev, &d) == CN_OK &&
          single_geometry(dev, *d, variant, false, p, std::min(n_i, kDDSmall), std::min(n_j, kDDSmall), &g) == CN_OK)
        need = std::max(need, g.ws_bytes);
      return need;
    }
    if (need == 0 || (variant != cn::kF32 && variant != cn::kF32Pot)) return need;
    // the slots of the symmetric form (one set against itself) and the
    // segments of the row kernel; a smaller buffer that holds the above is
    // accepted, and takes the pair kernel
    int dev = 0;
    DeviceInfo* d = nullptr;
    if (current_device(&dev, &d) != CN_OK) return need;
    const bool pot = variant == cn::kF32Pot;
    const cn::SymForm form = pot ? cn::kSymForcePot : cn::kSymForce;
    const cn::RowForm rows = pot ? cn::kRowForcePot : cn::kRowForce;
    SymPlan sp;
    if (n_i == n_j && sym_pays(form, n_i, d->sms) && !registered_tune(dev, variant, n_i, n_j, kTunedOneSet) &&
        sym_fit(dev, *d, form, n_i, false, sym_default_plan(form, n_i, d->sms), &sp) == CN_OK)
      need = std::max(need, sp.need);
    Plan p;
    Geometry g;
    RowPlan rp;
    if (!registered_tune(dev, variant, n_i, n_j, kTunedTwoSets) &&
        resolve_plan(dev, variant, n_i, n_j, false, nullptr, &p) == CN_OK &&
        single_geometry(dev, *d, variant, false, p, n_i, n_j, &g) == CN_OK &&
        rows_pays(rows, n_i, n_j, d->sms, p, g) && rows_fit(dev, *d, rows, n_i, n_j, &rp) == CN_OK)
      need = std::max(need, rp.need);
    return need;
  });
}

cn_status cn_batch_plan_create(int32_t n_clusters, const int64_t* offsets_host, const float* eps2_host,
                               const cn_tune* tune, int with_potential, cn_batch_plan** plan_out) {
  NvtxRange nvtx_range("cn_batch_plan_create");
  return cn::guard([&]() -> cn_status {
    return build_batch_plan(n_clusters, offsets_host, eps2_host, tune, with_potential, plan_out);
  });
}

cn_status cn_batch_plan_destroy(cn_batch_plan* plan) {
  return cn::guard([&]() -> cn_status {
    if (!plan) return CN_OK;
    if (plan->exec) cudaGraphExecDestroy(plan->exec);
    if (plan->graph) cudaGraphDestroy(plan->graph);
    if (plan->d_tiles) cudaFree(plan->d_tiles);
    if (plan->d_index) cudaFree(plan->d_index);
    if (plan->d_rows) cudaFree(plan->d_rows);
    if (plan->d_blocks) cudaFree(plan->d_blocks);
    delete plan;
    return CN_OK;
  });
}

size_t cn_batch_plan_workspace_bytes(const cn_batch_plan* plan) {
  return plan ? std::max(plan->ws_bytes, plan->sym_bytes) : 0;
}

cn_status cn_batch_plan_info(const cn_batch_plan* plan, int64_t* n_total, double* pairs) {
  return cn::guard([&]() -> cn_status {
    if (!plan) return fail(CN_ERR_INVALID_ARG, "plan is NULL");
    if (n_total) *n_total = plan->n_total;
    if (pairs) *pairs = plan->pairs;
    return CN_OK;
  });
}

cn_status cn_force_batched(const cn_batch_plan* plan, const float* pos_mass, float* acc_out, float* pot_out,
                           void* workspace, size_t ws_bytes, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_batched");
  return cn::guard([&]() -> cn_status {
    if (plan && plan->lists) return fail(CN_ERR_INVALID_ARG, "an interaction-list plan runs with cn_force_lists");
    return run_batched(plan, pos_mass, pos_mass, acc_out, pot_out, workspace, ws_bytes,
                       reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_list_plan_create(int32_t n_groups, const int64_t* i_offsets_host, const int64_t* j_begin_host,
                              const int64_t* j_count_host, const float* eps2_host, const cn_tune* tune,
                              int with_potential, cn_batch_plan** plan_out) {
  NvtxRange nvtx_range("cn_list_plan_create");
  return cn::guard([&]() -> cn_status {
    return build_list_plan(n_groups, i_offsets_host, j_begin_host, j_count_host, eps2_host, tune, with_potential,
                           plan_out);
  });
}

cn_status cn_list_plan_create_indexed(int32_t n_groups, const int64_t* i_offsets_host, const int64_t* j_begin_host,
                                      const int64_t* j_count_host, const float* eps2_host,
                                      const int32_t* j_index_host, int64_t n_index, int64_t n_src,
                                      const cn_tune* tune, int with_potential, cn_batch_plan** plan_out) {
  NvtxRange nvtx_range("cn_list_plan_create_indexed");
  return cn::guard([&]() -> cn_status {
    return build_list_plan_indexed(n_groups, i_offsets_host, j_begin_host, j_count_host, eps2_host, j_index_host,
                                   n_index, n_src, tune, with_potential, plan_out);
  });
}

cn_status cn_force_lists(const cn_batch_plan* plan, const float* pos_i, const float* pos_mass_j, float* acc_out,
                         float* pot_out, void* workspace, size_t ws_bytes, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_lists");
  return cn::guard([&]() -> cn_status {
    if (plan && !plan->lists) return fail(CN_ERR_INVALID_ARG, "a cluster plan runs with cn_force_batched");
    return run_batched(plan, pos_i, pos_mass_j, acc_out, pot_out, workspace, ws_bytes,
                       reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status capture_plan(cn_batch_plan* plan, const float* pos_i, const float* pos_j, float* acc_out, float* pot_out,
                       void* workspace, size_t ws_bytes, cn_stream stream) {
  if (!plan) return fail(CN_ERR_INVALID_ARG, "plan is NULL");
  auto s = reinterpret_cast<cudaStream_t>(stream);
  if (!s) return fail(CN_ERR_INVALID_ARG, "graph capture needs a non-default stream");
  if (!workspace && plan->ws_bytes) return fail(CN_ERR_WORKSPACE, "graph capture needs a caller workspace");
  if (inject("capture")) return fail(CN_ERR_CUDA, "cudaStreamBeginCapture: injected capture failure");
  cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return fail_cuda(e, "cudaStreamBeginCapture");
  cn_status st = run_batched(plan, pos_i, pos_j, acc_out, pot_out, workspace, ws_bytes, s);
  cudaGraph_t graph = nullptr;
  e = cudaStreamEndCapture(s, &graph);
  if (st != CN_OK) {
    if (graph) cudaGraphDestroy(graph);
    return st;
  }
  if (e != cudaSuccess) return fail_cuda(e, "cudaStreamEndCapture");
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  if (e != cudaSuccess) {
    cudaGraphDestroy(graph);
    return fail_cuda(e, "cudaGraphInstantiate");
  }
  if (plan->exec) cudaGraphExecDestroy(plan->exec);
  if (plan->graph) cudaGraphDestroy(plan->graph);
  plan->graph = graph;
  plan->exec = exec;
  return CN_OK;
}

cn_status cn_batch_plan_capture(cn_batch_plan* plan, const float* pos_mass, float* acc_out, float* pot_out,
                                void* workspace, size_t ws_bytes, cn_stream stream) {
  NvtxRange nvtx_range("cn_batch_plan_capture");
  return cn::guard([&]() -> cn_status {
    if (plan && plan->lists) return fail(CN_ERR_INVALID_ARG, "an interaction-list plan is captured with cn_list_plan_capture");
    return capture_plan(plan, pos_mass, pos_mass, acc_out, pot_out, workspace, ws_bytes, stream);
  });
}

cn_status cn_list_plan_capture(cn_batch_plan* plan, const float* pos_i, const float* pos_mass_j, float* acc_out,
                               float* pot_out, void* workspace, size_t ws_bytes, cn_stream stream) {
  NvtxRange nvtx_range("cn_list_plan_capture");
  return cn::guard([&]() -> cn_status {
    if (plan && !plan->lists) return fail(CN_ERR_INVALID_ARG, "a cluster plan is captured with cn_batch_plan_capture");
    return capture_plan(plan, pos_i, pos_mass_j, acc_out, pot_out, workspace, ws_bytes, stream);
  });
}

cn_status cn_batch_plan_launch(const cn_batch_plan* plan, cn_stream stream) {
  NvtxRange nvtx_range("cn_batch_plan_launch");
  return cn::guard([&]() -> cn_status {
    if (!plan || !plan->exec) return fail(CN_ERR_INVALID_ARG, "plan has no captured graph");
    if (inject("launch")) return fail(CN_ERR_CUDA, "cudaGraphLaunch: injected launch failure");
    cudaError_t e = cudaGraphLaunch(plan->exec, reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? CN_OK : fail_cuda(e, "cudaGraphLaunch");
  });
}

cn_status cn_force_adjoint(int64_t n, const float* pos_mass, float eps2, const float* w, float* grad_pos,
                           float* grad_mass, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_adjoint");
  return cn::guard([&]() -> cn_status {
    auto s = reinterpret_cast<cudaStream_t>(stream);
    if (n < 0) return fail(CN_ERR_INVALID_ARG, "n must be >= 0");
    cn_status st;
    if ((st = check_eps2(eps2)) != CN_OK) return st;
    if ((st = check_records(pos_mass, n, "pos_mass")) != CN_OK) return st;
    if (n > 0 && (!w || !grad_pos || !grad_mass)) return fail(CN_ERR_INVALID_ARG, "w, grad_pos and grad_mass are required");
    if ((w && !aligned(w, 4)) || (grad_pos && !aligned(grad_pos, 4)) || (grad_mass && !aligned(grad_mass, 4)))
      return fail(CN_ERR_MISALIGNED, "w and the gradients must be 4-byte aligned");
    const size_t un = static_cast<size_t>(n);
    if (overlaps(grad_pos, un * 12, pos_mass, un * 16) || overlaps(grad_pos, un * 12, w, un * 12) ||
        overlaps(grad_mass, un * 4, pos_mass, un * 16) || overlaps(grad_mass, un * 4, w, un * 12) ||
        overlaps(grad_pos, un * 12, grad_mass, un * 4))
      return fail(CN_ERR_INVALID_ARG, "outputs overlap inputs or each other");
    if (n == 0) return CN_OK;
    int dev = 0;
    DeviceInfo* d = nullptr;
    if ((st = current_device(&dev, &d)) != CN_OK) return st;
    const bool guard = needs_guard(eps2);
    if (!guard) {
      if (const SymPlan* sp = sym_self_plan(dev, *d, cn::kSymAdjoint, cn::kAdjoint, n, un * 16 + 256, s)) {
        float* wrec = reinterpret_cast<float*>(sp->data + align_up(sp->need, 256));
        if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
        std::lock_guard<std::recursive_mutex> order(launch_order(s));
        const cudaError_t e = cn::launch_pack_w(w, reinterpret_cast<float4*>(wrec), n, s);
        if (e != cudaSuccess) return fail_cuda(e, "weight packing launch");
        float* const out[3] = {grad_pos, grad_mass, nullptr};
        const std::string what = log_enabled() ? "cn_force_adjoint: n " + std::to_string(n) : std::string();
        return sym_launch(what, *d, cn::kSymAdjoint, *sp, n, pos_mass, wrec, eps2, out, s);
      }
    }
    Plan p;
    if ((st = resolve_plan(dev, cn::kAdjoint, n, n, guard, nullptr, &p)) != CN_OK) return st;
    Geometry g;
    if ((st = single_geometry(dev, *d, cn::kAdjoint, guard, p, n, n, &g)) != CN_OK) return st;
    char *ctrl = nullptr, *data = nullptr;
    if ((st = library_workspace(s, g.ctrl_bytes, g.data_bytes, &ctrl, &data)) != CN_OK) return st;
    float4* wrec = reinterpret_cast<float4*>(data + g.off_wrec);
    if (inject("launch")) return fail(CN_ERR_CUDA, "kernel launch: injected launch failure");
    std::lock_guard<std::recursive_mutex> order(launch_order(s));
    cudaError_t e = cn::launch_pack_w(w, wrec, n, s);
    if (e != cudaSuccess) return fail_cuda(e, "weight packing launch");
    PairArgs a = base_args(ctrl, data, g, p, d->status);
    a.pos_i = reinterpret_cast<const float4*>(pos_mass);
    a.pos_j = reinterpret_cast<const float4*>(pos_mass);
    a.pos_i2 = wrec;
    a.pos_j2 = wrec;
    a.acc_out = grad_pos;
    a.pot_out = grad_mass;
    a.n_i = n;
    a.n_j = n;
    a.eps2 = eps2;
    log_plan("cn_force_adjoint", cn::kAdjoint, n, n, guard, p, g, g.njt);
    e = cn::launch_adjoint(a, p, guard, g.grid, s);
    return e == cudaSuccess ? CN_OK : fail_cuda(e, "adjoint kernel launch");
  });
}

cn_status cn_force_jerk(int64_t n_i, const float* pos_i, const float* vel_i, int64_t n_j, const float* pos_mass_j,
                        const float* vel_j, float eps2, float* acc_out, float* jerk_out, float* pot_out,
                        cn_stream stream) {
  NvtxRange nvtx_range("cn_force_jerk");
  return cn::guard([&]() -> cn_status {
    return jerk_common(n_i, pos_i, vel_i, n_j, pos_mass_j, vel_j, eps2, acc_out, jerk_out, pot_out,
                       reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_force_symmetric(int64_t n, const float* pos_mass, float eps2, float* acc_out, float* pot_out,
                             cn_stream stream) {
  NvtxRange nvtx_range("cn_force_symmetric");
  return cn::guard([&]() -> cn_status {
    return symmetric_common(n, pos_mass, eps2, acc_out, pot_out, reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_potential_energy(int64_t n, const float* pos_mass, const float* pot, double* w_out, cn_stream stream) {
  NvtxRange nvtx_range("cn_potential_energy");
  return cn::guard([&]() -> cn_status {
    return energy_common(n, pos_mass, pot, nullptr, w_out, reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_potential_energy_dd(int64_t n, const float* pos_mass, const double* pot, double* w_out,
                                 cn_stream stream) {
  NvtxRange nvtx_range("cn_potential_energy_dd");
  return cn::guard([&]() -> cn_status {
    return energy_common(n, pos_mass, nullptr, pot, w_out, reinterpret_cast<cudaStream_t>(stream));
  });
}

cn_status cn_force_host(int64_t n_i, const float* pos_i_host, int64_t n_j, const float* pos_mass_j_host, float eps2,
                        float* acc_host, float* pot_host, cn_stream stream) {
  NvtxRange nvtx_range("cn_force_host");
  return cn::guard([&]() -> cn_status {
    auto s = reinterpret_cast<cudaStream_t>(stream);
    if (n_i < 0 || n_j < 0) return fail(CN_ERR_INVALID_ARG, "n_i and n_j must be >= 0");
    if ((n_i > 0 && (!pos_i_host || !acc_host)) || (n_j > 0 && !pos_mass_j_host))
      return fail(CN_ERR_INVALID_ARG, "NULL host buffer");
    cn_status st = check_eps2(eps2);
    if (st != CN_OK) return st;
    if (n_i == 0) return CN_OK;
    int dev = 0;
    DeviceInfo* d = nullptr;
    if ((st = current_device(&dev, &d)) != CN_OK) return st;
    // i = j when the caller passes the same host array for both sets: copy it once
    const bool same = pos_i_host == pos_mass_j_host && n_i == n_j;
    const size_t bi = align_up(static_cast<size_t>(n_i) * 16, 256);
    const size_t bj = same ? 0 : align_up(static_cast<size_t>(n_j) * 16, 256);
    const size_t ba = align_up(static_cast<size_t>(n_i) * 12, 256);
    const size_t bp = pot_host ? align_up(static_cast<size_t>(n_i) * 4, 256) : 0;
    void* buf = nullptr;
    if ((st = stage_buffer(s, bi + bj + ba + bp, &buf)) != CN_OK) return st;
    char* base = static_cast<char*>(buf);
    float* d_pi = reinterpret_cast<float*>(base);
    float* d_pj = same ? d_pi : reinterpret_cast<float*>(base + bi);
    float* d_acc = reinterpret_cast<float*>(base + bi + bj);
    float* d_pot = pot_host ? reinterpret_cast<float*>(base + bi + bj + ba) : nullptr;
    cudaError_t e = cudaMemcpyAsync(d_pi, pos_i_host, static_cast<size_t>(n_i) * 16, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && !same && n_j > 0)
      e = cudaMemcpyAsync(d_pj, pos_mass_j_host, static_cast<size_t>(n_j) * 16, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return fail_cuda(e, "cudaMemcpyAsync(host to device)");
    if ((st = cn_force(n_i, d_pi, n_j, d_pj, eps2, d_acc, d_pot, stream)) != CN_OK) return st;
    e = cudaMemcpyAsync(acc_host, d_acc, static_cast<size_t>(n_i) * 12, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && pot_host)
      e = cudaMemcpyAsync(pot_host, d_pot, static_cast<size_t>(n_i) * 4, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return fail_cuda(e, "cudaMemcpyAsync(device to host)");
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail_cuda(e, "cudaStreamSynchronize");
    return CN_OK;
  });
}

cn_status cn_force_host_f64(const double* xj, const double* mj, const double* xi, double eps2, double* a, int ni,
                            int nj) {
  NvtxRange nvtx_range("cn_force_host_f64");
  return cn::guard([&]() -> cn_status {
    if (ni < 0 || nj < 0) return fail(CN_ERR_INVALID_ARG, "ni and nj must be >= 0");
    if ((ni > 0 && (!xi || !a)) || (nj > 0 && (!xj || !mj))) return fail(CN_ERR_INVALID_ARG, "NULL host array");
    if (!std::isfinite(eps2) || eps2 < 0.0) return fail(CN_ERR_INVALID_ARG, "eps2 must be finite and >= 0");
    if (ni == 0) return CN_OK;
    std::vector<float> pi(static_cast<size_t>(ni) * 4), pj(static_cast<size_t>(nj) * 4), acc(static_cast<size_t>(ni) * 3);
    for (int i = 0; i < ni; ++i) {
      for (int c = 0; c < 3; ++c) pi[4 * i + c] = static_cast<float>(xi[3 * i + c]);
      pi[4 * i + 3] = 0.f;
    }
    for (int j = 0; j < nj; ++j) {
      for (int c = 0; c < 3; ++c) pj[4 * j + c] = static_cast<float>(xj[3 * j + c]);
      pj[4 * j + 3] = static_cast<float>(mj[j]);
    }
    cn_status st = cn_force_host(ni, pi.data(), nj, nj ? pj.data() : nullptr, static_cast<float>(eps2), acc.data(),
                                 nullptr, nullptr);
    if (st != CN_OK) return st;
    for (size_t k = 0; k < acc.size(); ++k) a[k] = acc[k];
    return CN_OK;
  });
}

cn_status cn_tune_get(int variant, int64_t n_i, int64_t n_j, cn_tune* out) {
  return cn::guard([&]() -> cn_status {
    if (!out || variant < cn::kF32 || variant > cn::kF32EpsIPot || n_i < 0 || n_j < 0)
      return fail(CN_ERR_INVALID_ARG, "bad variant, size or NULL output");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
    Plan p;
    cn_status st = resolve_plan(dev, variant, n_i, n_j, false, nullptr, &p);
    if (st != CN_OK) return st;
    out->i_per_thread = p.k;
    out->threads = p.threads;
    out->j_tile = p.j_tile;
    out->stages = p.stages;
    out->ctas_per_sm = p.ctas_per_sm;
    out->chunk_units = static_cast<int32_t>(p.chunk_units);
    out->j_lanes = p.j_lanes;
    return CN_OK;
  });
}

cn_status cn_tune_set(int variant, int64_t n_i, int64_t n_j, const cn_tune* tune) {
  return cn::guard([&]() -> cn_status {
    if (variant < cn::kF32 || variant > cn::kF32EpsIPot || n_i < 0 || n_j < 0)
      return fail(CN_ERR_INVALID_ARG, "bad variant or size");
    if (tune) {
      cn_status st = check_tune(variant, *tune);
      if (st != CN_OK) return st;
    }
    return store_tune(variant, n_i, n_j, tune, kTunedAny);
  });
}

cn_status cn_tune_save(const char* path) {
  return cn::guard([&]() -> cn_status {
    if (!path) return fail(CN_ERR_INVALID_ARG, "path is NULL");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail_cuda(e, "cudaGetDevice");
    std::string name, arch;
    int sms = 0;
    cn_status st = device_identity(dev, &name, &arch, &sms);
    if (st != CN_OK) return st;
    std::string out = "{\"format\": \"cunbody-tune-1\", \"device\": \"";
    for (char c : name) {
      if (c == '"' || c == '\\') out.push_back('\\');
      out.push_back(c);
    }
    out += "\", \"arch\": \"" + arch + "\", \"sms\": " + std::to_string(sms) + ", \"entries\": [";
    {
      std::lock_guard<std::mutex> lock(g_mu);
      bool first = true;
      for (const auto& kv : g_tune) {
        if (std::get<0>(kv.first) != dev) continue;
        const cn_tune& t = kv.second.t;
        const char* const on[] = {"", ", \"sets\": \"one\"", ", \"sets\": \"two\""};
        char line[512];
        std::snprintf(line, sizeof(line),
                      "%s\n  {\"variant\": \"%s\", \"n_i_class\": %d, \"n_j_class\": %d, \"i_per_thread\": %d, "
                      "\"threads\": %d, \"j_tile\": %d, \"stages\": %d, \"ctas_per_sm\": %d, \"chunk_units\": %d, "
                      "\"j_lanes\": %d%s}",
                      first ? "" : ",", variant_name(std::get<1>(kv.first)), std::get<2>(kv.first), std::get<3>(kv.first),
                      t.i_per_thread, t.threads, t.j_tile, t.stages, t.ctas_per_sm, t.chunk_units, t.j_lanes, on[kv.second.on]);
        out += line;
        first = false;
      }
    }
    out += "\n]}\n";
    FILE* f = std::fopen(path, "w");
    if (!f) return fail(CN_ERR_INVALID_ARG, std::string("cannot write ") + path);
    const bool ok = std::fwrite(out.data(), 1, out.size(), f) == out.size();
    if (std::fclose(f) != 0 || !ok) return fail(CN_ERR_INVALID_ARG, std::string("writing ") + path + " failed");
    return CN_OK;
  });
}

cn_status cn_tune_load(const char* path, int32_t* n_loaded) {
  return cn::guard([&]() -> cn_status {
    if (n_loaded) *n_loaded = 0;
    if (!path) return fail(CN_ERR_INVALID_ARG, "path is NULL");
    FILE* f = std::fopen(path, "r");
    if (!f) return fail(CN_ERR_INVALID_ARG, std::string("cannot read ") + path);
    std::string text;
    char buf[4096];
    size_t got;
    while ((got = std::fread(buf, 1, sizeof(buf), f)) > 0 && text.size() < (static_cast<size_t>(1) << 24))
      text.append(buf, got);
    std::fclose(f);
    JsonValue root;
    JsonReader rd{text};
    if (!rd.value(&root) || root.kind != JsonValue::kObject) return fail(CN_ERR_INVALID_ARG, "tuning file: not a JSON object");
    rd.skip();
    if (rd.pos != text.size()) return fail(CN_ERR_INVALID_ARG, "tuning file: trailing characters");
    const JsonValue* fmt = root.get("format");
    const JsonValue* dname = root.get("device");
    const JsonValue* darch = root.get("arch");
    const JsonValue* entries = root.get("entries");
    int64_t file_sms = 0;
    if (!fmt || fmt->kind != JsonValue::kString || fmt->text != "cunbody-tune-1")
      return fail(CN_ERR_INVALID_ARG, "tuning file: unknown format");
    if (!dname || dname->kind != JsonValue::kString || !darch || darch->kind != JsonValue::kString ||
        !json_int(root, "sms", 1, 1 << 20, &file_sms) || !entries || entries->kind != JsonValue::kArray)
      return fail(CN_ERR_INVALID_ARG, "tuning file: device, arch, sms or entries missing");
    struct Entry {
      int variant, ci, cj;
      cn_tune t;
      TunedOn on;
    };
    std::vector<Entry> parsed;
    for (const JsonValue& e : entries->items) {
      if (e.kind != JsonValue::kObject) return fail(CN_ERR_INVALID_ARG, "tuning file: an entry is not an object");
      const JsonValue* vn = e.get("variant");
      const int variant = (vn && vn->kind == JsonValue::kString) ? variant_from_name(vn->text) : -1;
      int64_t ci, cj, k, th, jt, stg, cps, ch, jl;
      if (variant < 0 || !json_int(e, "n_i_class", 0, 62, &ci) || !json_int(e, "n_j_class", 0, 62, &cj) ||
          !json_int(e, "i_per_thread", 0, 8, &k) || !json_int(e, "threads", 0, 1024, &th) ||
          !json_int(e, "j_tile", 0, 4096, &jt) || !json_int(e, "stages", 0, 8, &stg) ||
          !json_int(e, "ctas_per_sm", 0, 64, &cps) || !json_int(e, "chunk_units", 0, INT32_MAX, &ch) ||
          !json_int(e, "j_lanes", 0, 32, &jl))
        return fail(CN_ERR_INVALID_ARG, "tuning file: an entry has a missing or out-of-range field");
      Entry en{variant, static_cast<int>(ci), static_cast<int>(cj),
               cn_tune{static_cast<int32_t>(k), static_cast<int32_t>(th), static_cast<int32_t>(jt),
                       static_cast<int32_t>(stg), static_cast<int32_t>(cps), static_cast<int32_t>(ch),
                       static_cast<int32_t>(jl)}, kTunedAny};
      if (const JsonValue* on = e.get("sets")) {
        if (on->kind != JsonValue::kString || (on->text != "one" && on->text != "two"))
          return fail(CN_ERR_INVALID_ARG, "tuning file: an entry has a missing or out-of-range field");
        en.on = on->text == "one" ? kTunedOneSet : kTunedTwoSets;
      }
      const cn_status st = check_tune(variant, en.t);
      if (st != CN_OK) return st;
      parsed.push_back(en);
    }
    int dev = 0;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess) return fail_cuda(ce, "cudaGetDevice");
    std::string name, arch;
    int sms = 0;
    cn_status st = device_identity(dev, &name, &arch, &sms);
    if (st != CN_OK) return st;
    if (name != dname->text || arch != darch->text || sms != file_sms)
      return fail(CN_ERR_UNSUPPORTED_DEVICE, "tuning file was written on " + dname->text + " (" + darch->text + ", " +
                                                 std::to_string(file_sms) + " SMs), this device is " + name + " (" +
                                                 arch + ", " + std::to_string(sms) + " SMs)");
    {
      std::lock_guard<std::mutex> lock(g_mu);
      for (const Entry& en : parsed) g_tune[std::make_tuple(dev, en.variant, en.ci, en.cj)] = Tuned{en.t, en.on};
      g_plan_gen.fetch_add(1, std::memory_order_acq_rel);
    }
    if (n_loaded) *n_loaded = static_cast<int32_t>(parsed.size());
    return CN_OK;
  });
}

cn_status cn_autotune(int variant, int64_t n_i, const float* pos_i, int64_t n_j, const float* pos_mass_j, float eps2,
                      void* acc_out, void* pot_out, int reps, cn_stream stream, cn_tune* best_out) {
  NvtxRange nvtx_range("cn_autotune");
  return cn::guard([&]() -> cn_status {
    if (variant < cn::kF32 || variant > cn::kDDPot) return fail(CN_ERR_INVALID_ARG, "cn_autotune covers the F32 and DD variants");
    if (n_i <= 0 || n_j <= 0) return fail(CN_ERR_INVALID_ARG, "autotuning needs n_i > 0 and n_j > 0");
    const bool dd = variant == cn::kDD || variant == cn::kDDPot;
    const bool pot = variant == cn::kF32Pot || variant == cn::kDDPot;
    if (pot && !pot_out) return fail(CN_ERR_INVALID_ARG, "the potential variants need pot_out");
    auto s = reinterpret_cast<cudaStream_t>(stream);
    if (reps < 1) reps = 1;
    const int ks[] = {1, 2, 4, 8};
    const int ths[] = {64, 128, 256};
    const int tiles[] = {128, 256, 512, 1024};
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best_ms = 1e30f;
    cn_tune best{};
    cn_status result = CN_OK;
    std::vector<cn_tune> cands;
    const TunedOn on = pos_i == pos_mass_j && n_i == n_j ? kTunedOneSet : kTunedTwoSets;
    bool other = false;  // the call without an entry takes another kernel than the pair kernel
    {
      // the default shape of these sizes first (its j-tile fitted to the
      // schedule, which the grid below does not contain), so that the result
      // is never slower than the default by more than the timing noise
      int dev = 0;
      DeviceInfo* d = nullptr;
      cn_status st = current_device(&dev, &d);
      if (st != CN_OK) return st;
      cands.push_back(default_tune(variant, n_i, n_j, d->sms));
      if (!dd && !needs_guard(eps2)) {
        Plan p;
        Geometry g;
        if (on == kTunedOneSet && sym_pays(cn::kSymForce, n_i, d->sms))
          other = true;
        else
          other = resolve_plan(dev, variant, n_i, n_j, false, &cands.front(), &p) == CN_OK &&
                  single_geometry(dev, *d, variant, false, p, n_i, n_j, &g) == CN_OK &&
                  rows_pays(pot ? cn::kRowForcePot : cn::kRowForce, n_i, n_j, d->sms, p, g);
      }
    }
    for (int k : ks) {
      if (!valid_k(variant, k)) continue;
      for (int th : ths) {
        if (static_cast<int64_t>(k) * th > 4 * std::max<int64_t>(n_i, 256)) continue;  // tile far larger than the i set
        for (int jt : tiles) {
          if (jt > 4 * std::max<int64_t>(n_j, 64)) continue;
          cands.push_back(cn_tune{k, th, jt, 4, 0, 0, 1});
        }
      }
    }
    if (!dd && n_i <= 16384) {  // split-j shapes for small systems
      for (int jl : {2, 4, 8, 16, 32}) {
        if (n_i * jl > 262144) continue;
        for (int th : {128, 256})
          for (int64_t jt : {static_cast<int64_t>(512), static_cast<int64_t>(2048), round_up(std::max<int64_t>(n_j, 1), 8 * jl),
                             static_cast<int64_t>(4096)}) {
            if (jt % (8 * jl) || jt > 4096 || jt < 8 * jl) continue;
            for (int k : {1, 2, 4, 8}) {  // i-particles per lane group (packed for K >= 2)
              if (static_cast<int64_t>(k) * th / jl > 4 * std::max<int64_t>(n_i, 64)) continue;
              cands.push_back(cn_tune{k, th, static_cast<int32_t>(jt), jt >= n_j ? 1 : 3, 0, 0, jl});
            }
          }
      }
    }
    // Candidates are timed as one CUDA graph of `reps` calls, so that the host
    // cost of a call does not hide the device time of small problems. Capture
    // needs a non-default stream: the legacy stream gets a private one.
    cudaStream_t ts = s;
    const bool own_stream = (s == nullptr);
    if (own_stream && cudaStreamCreateWithFlags(&ts, cudaStreamNonBlocking) != cudaSuccess) {
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      return fail(CN_ERR_CUDA, "autotune: cudaStreamCreate failed");
    }
    auto call = [&]() {
      return force_common(dd, n_i, pos_i, n_j, pos_mass_j, eps2, acc_out, pot ? pot_out : nullptr, nullptr, 0, true,
                          ts);
    };
    // Without an entry the symmetric or the row kernel may take the call: that
    // default is timed first, as the candidate without an entry.
    if (other) cands.insert(cands.begin(), cands.front());
    bool untuned = other, best_untuned = false;
    for (const cn_tune& t : cands) {
      if (check_tune(variant, t) != CN_OK) continue;
      const bool bare = untuned;
      untuned = false;
      store_tune(variant, n_i, n_j, bare ? nullptr : &t, on);
      cn_status st = call();  // warm-up (and workspace growth)
      if (st == CN_ERR_INVALID_ARG) continue;  // shape does not fit
      if (st != CN_OK) {
        result = st;
        break;
      }
      cudaGraph_t graph = nullptr;
      cudaGraphExec_t exec = nullptr;
      if (cudaStreamBeginCapture(ts, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        result = fail(CN_ERR_CUDA, "autotune: cudaStreamBeginCapture failed");
        break;
      }
      for (int r = 0; r < reps && st == CN_OK; ++r) st = call();
      cudaError_t e = cudaStreamEndCapture(ts, &graph);
      if (st == CN_OK && e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
      if (st == CN_OK && e == cudaSuccess) e = cudaGraphLaunch(exec, ts);  // warm
      if (st == CN_OK && e == cudaSuccess) e = cudaEventRecord(e0, ts);
      if (st == CN_OK && e == cudaSuccess) e = cudaGraphLaunch(exec, ts);
      if (st == CN_OK && e == cudaSuccess) e = cudaEventRecord(e1, ts);
      if (st == CN_OK && e == cudaSuccess) e = cudaEventSynchronize(e1);
      float ms = 0.f;
      if (st == CN_OK && e == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
      if (exec) cudaGraphExecDestroy(exec);
      if (graph) cudaGraphDestroy(graph);
      if (st != CN_OK) {
        result = st;
        break;
      }
      if (e != cudaSuccess) {
        result = fail_cuda(e, "autotune: timing a candidate");
        break;
      }
      if (ms < best_ms) {
        best_ms = ms;
        best = t;
        best_untuned = bare;
      }
    }
    if (own_stream) {
      cudaStreamSynchronize(ts);
      release_library_workspace(ts);
      cudaStreamDestroy(ts);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (result != CN_OK) {
      cn_tune_set(variant, n_i, n_j, nullptr);
      return result;
    }
    if (best_ms >= 1e30f) {
      cn_tune_set(variant, n_i, n_j, nullptr);
      return fail(CN_ERR_INVALID_ARG, "no candidate launch shape fits");
    }
    store_tune(variant, n_i, n_j, best_untuned ? nullptr : &best, on);
    if (best_out) *best_out = best;
    return CN_OK;
  });
}

cn_status cn_autotune_batched(int32_t n_clusters, const int64_t* offsets_host, const float* eps2_host,
                              const float* pos_mass, float* acc_out, float* pot_out, int reps, cn_stream stream,
                              cn_tune* best_out) {
  NvtxRange nvtx_range("cn_autotune_batched");
  return cn::guard([&]() -> cn_status {
    if (n_clusters <= 0 || !offsets_host) return fail(CN_ERR_INVALID_ARG, "empty ensemble");
    auto s = reinterpret_cast<cudaStream_t>(stream);
    if (reps < 1) reps = 1;
    const int variant = pot_out ? cn::kBatchedPot : cn::kBatched;
    const int ks[] = {2, 4, 8};
    const int ths[] = {64, 128, 256};
    const int tiles[] = {128, 256, 512};
    const int chunks[] = {0, 8, 32};
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best_ms = 1e30f;
    cn_tune best{};
    cn_status result = CN_OK;
    // The default first (a plan without a tune, which may take the symmetric
    // form): when nothing beats it, no entry is stored and best_out is its
    // one-sided shape.
    const int64_t n_total = offsets_host[n_clusters];
    int dev = 0;
    cudaGetDevice(&dev);
    cn_tune before{}, bare_shape{};
    const bool had = registered_tune(dev, variant, n_clusters, n_total, kTunedAny);
    if (had) cn_tune_get(variant, n_clusters, n_total, &before);
    cn_tune_set(variant, n_clusters, n_total, nullptr);
    bool best_bare = false;
    std::vector<cn_tune> cands{bare_shape};
    for (int k : ks)
      for (int th : ths)
        for (int jt : tiles)
          for (int ch : chunks) cands.push_back(cn_tune{k, th, jt, 4, 0, ch, 1});
    // split-j shapes: eight i-particles per lane group, small i-tiles
    for (int jl : {2, 4, 8})
      for (int jt : {256, 512})
        for (int ch : {0, 8}) cands.push_back(cn_tune{8, 256, jt, 4, 0, ch, jl});
    for (const cn_tune& t : cands) {
      if (result != CN_OK) break;
      cn_batch_plan* plan = nullptr;
      const bool is_bare = &t == &cands.front();
      cn_status st =
          build_batch_plan(n_clusters, offsets_host, eps2_host, is_bare ? nullptr : &t, pot_out != nullptr, &plan);
      if (st != CN_OK) {
        if (st == CN_ERR_INVALID_ARG) continue;
        result = st;
        break;
      }
      st = run_batched(plan, pos_mass, pos_mass, acc_out, pot_out, nullptr, 0, s);
      if (st == CN_OK) {
        cudaEventRecord(e0, s);
        for (int r = 0; r < reps; ++r) run_batched(plan, pos_mass, pos_mass, acc_out, pot_out, nullptr, 0, s);
        cudaEventRecord(e1, s);
        if (cudaEventSynchronize(e1) == cudaSuccess) {
          float ms = 0.f;
          cudaEventElapsedTime(&ms, e0, e1);
          if (ms < best_ms) {
            best_ms = ms;
            best = t;
            best_bare = is_bare;
            if (is_bare)
              best = cn_tune{plan->plan.k, plan->plan.threads, plan->plan.j_tile, plan->plan.stages, 0,
                             static_cast<int32_t>(plan->plan.chunk_units), plan->plan.j_lanes};
          }
        } else {
          st = fail(CN_ERR_CUDA, "autotune: event synchronisation failed");
        }
      }
      cn_batch_plan_destroy(plan);
      if (st != CN_OK) result = st;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (result != CN_OK || best_ms >= 1e30f) {
      if (had) cn_tune_set(variant, n_clusters, n_total, &before);
      if (result != CN_OK) return result;
      return fail(CN_ERR_INVALID_ARG, "no candidate launch shape fits");
    }
    if (!best_bare) cn_tune_set(variant, n_clusters, n_total, &best);
    if (best_out) *best_out = best;
    return CN_OK;
  });
}

cn_status cn_get_device_status(cn_stream stream) {
  NvtxRange nvtx_range("cn_get_device_status");
  return cn::guard([&]() -> cn_status {
    auto s = reinterpret_cast<cudaStream_t>(stream);
    int dev = 0;
    DeviceInfo* d = nullptr;
    cn_status st = current_device(&dev, &d);
    if (st != CN_OK) return st;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail_cuda(e, "cudaStreamSynchronize");
    int flag = 0;
    if ((e = cudaMemcpy(&flag, d->status, sizeof(int), cudaMemcpyDeviceToHost)) != cudaSuccess)
      return fail_cuda(e, "reading the device status word");
    if (flag == 0) return CN_OK;
    const int zero = 0;
    cudaMemcpy(d->status, &zero, sizeof(int), cudaMemcpyHostToDevice);
    {
      // arrival counters may have been left mid-protocol: clear every library workspace of this device
      std::lock_guard<std::mutex> lock(g_mu);
      for (auto& kv : g_ws)
        if (kv.first.first == dev) {
          if (kv.second.ctrl) cudaMemset(kv.second.ctrl, 0, kv.second.ctrl_bytes);
          if (kv.second.aux) cudaMemset(kv.second.aux, 0, (cn::energy_workspace_doubles() + 1) * sizeof(double));
        }
    }
    cudaDeviceSynchronize();
    return fail(CN_ERR_TIMEOUT, "a kernel wait timed out (device status bits " + std::to_string(flag) + ")");
  });
}

cn_status cn_set_wait_limit_ns(uint64_t ns) {
  return cn::guard([&]() -> cn_status {
    g_wait_ns.store(ns ? ns : kDefaultWaitNs);
    return CN_OK;
  });
}

cn_status cn_debug_timeout_probe(cn_stream stream) {
  return cn::guard([&]() -> cn_status {
    int dev = 0;
    DeviceInfo* d = nullptr;
    cn_status st = current_device(&dev, &d);
    if (st != CN_OK) return st;
    cudaError_t e = cn::launch_timeout_probe(d->status, g_wait_ns.load(), reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? CN_OK : fail_cuda(e, "timeout probe launch");
  });
}

cn_status cn_probe_peaks(cn_stream stream, double* out5) {
  return cn::guard([&]() -> cn_status {
    if (!out5) return fail(CN_ERR_INVALID_ARG, "out is NULL");
    int dev = 0;
    DeviceInfo* d = nullptr;
    cn_status st = current_device(&dev, &d);
    if (st != CN_OK) return st;
    cudaError_t e = cn::run_probes(reinterpret_cast<cudaStream_t>(stream), out5);
    return e == cudaSuccess ? CN_OK : fail_cuda(e, "issue-rate probes");
  });
}

const char* cn_status_string(cn_status status) {
  switch (status) {
    case CN_OK: return "CN_OK";
    case CN_ERR_INVALID_ARG: return "CN_ERR_INVALID_ARG";
    case CN_ERR_MISALIGNED: return "CN_ERR_MISALIGNED";
    case CN_ERR_CUDA: return "CN_ERR_CUDA";
    case CN_ERR_TIMEOUT: return "CN_ERR_TIMEOUT";
    case CN_ERR_UNSUPPORTED_DEVICE: return "CN_ERR_UNSUPPORTED_DEVICE";
    case CN_ERR_WORKSPACE: return "CN_ERR_WORKSPACE";
    case CN_ERR_HOST: return "CN_ERR_HOST";
  }
  return "CN_ERR_UNKNOWN";
}

const char* cn_last_error_message(void) { return g_last_error.c_str(); }

const char* cn_version(void) { return "cunbody 0.1.0 (sm_103a)"; }

}  // extern "C"
