// Process-wide autotuner table (see tune.h) and its C entry points.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <atomic>
#include <functional>
#include <mutex>
#include <set>

#include "lqcd_common.cuh"
#include "lqcd_internal.h"
#include "tune.h"

namespace lqcd {

static std::mutex g_tune_mutex;
static std::map<std::string, int> g_tune;
// Counts the table's changes (under the mutex): what was looked up under an older
// count may be out of date.
static std::atomic<uint64_t> g_tune_version{1};

bool tune_lookup(const std::string& key, int* value) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  auto it = g_tune.find(key);
  if (it == g_tune.end()) return false;
  *value = it->second;
  return true;
}

void tune_store(const std::string& key, int value) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  g_tune[key] = value;
  g_tune_version++;
}

// A hop's choice is an index into LQCD_HOP_SHAPES, so its line in a saved table also
// names the list's version: under another list the number means another kernel.
static bool is_hop_key(const std::string& key) { return key.compare(0, 4, "hop ") == 0; }
static const std::string& shapes_tag() {
  static const std::string tag = "shapes=" + std::to_string(HOP_SHAPES_VERSION);
  return tag;
}

}  // namespace lqcd

using namespace lqcd;

extern "C" {

int lqcd_tune_save(const char* path) {
  if (!path) return fail(LQCD_ERR_ARG, "lqcd_tune_save: null path");
  FILE* f = fopen(path, "w");
  if (!f) return fail(LQCD_ERR_ARG, "lqcd_tune_save: cannot open %s", path);
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  for (auto& kv : g_tune)
    fprintf(f, "%d\t%s%s%s\n", kv.second, kv.first.c_str(), is_hop_key(kv.first) ? "\t" : "",
            is_hop_key(kv.first) ? shapes_tag().c_str() : "");
  fclose(f);
  return LQCD_OK;
}

int lqcd_tune_load(const char* path) {
  if (!path) return fail(LQCD_ERR_ARG, "lqcd_tune_load: null path");
  FILE* f = fopen(path, "r");
  if (!f) return fail(LQCD_ERR_ARG, "lqcd_tune_load: cannot open %s", path);
  char line[4096];
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  while (fgets(line, sizeof(line), f)) {
    char* tab = strchr(line, '\t');
    if (!tab) continue;
    *tab = 0;
    char* end = nullptr;
    const long v = strtol(line, &end, 10);
    if (end == line || *end != 0) continue;
    std::string k(tab + 1);
    while (!k.empty() && (k.back() == '\n' || k.back() == '\r')) k.pop_back();
    if (is_hop_key(k) && k.find('\t') != std::string::npos) {
      const size_t end_of_key = k.find('\t');
      if (k.compare(end_of_key + 1, std::string::npos, shapes_tag()) != 0) continue;  // timed again on next use
      k.resize(end_of_key);
    }
    if (k.empty() || v < 0 || v > 64) continue;
    g_tune[k] = (int)v;
  }
  g_tune_version++;
  fclose(f);
  return LQCD_OK;
}

int lqcd_tune_entries(void) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  return (int)g_tune.size();
}

void lqcd_tune_clear(void) {
  {
    std::lock_guard<std::mutex> lock(g_tune_mutex);
    g_tune.clear();
    g_tune_version++;
  }
  lqcd::solver_tuning_reset();
}

}  // extern "C"

namespace lqcd {

static std::atomic<bool> g_autotune{true};
static thread_local bool g_tuning_pass = false;
static thread_local bool g_no_tuning = false;

std::string hop_key_string(const HopKey& k) {
  char buf[160];
  snprintf(buf, sizeof(buf), "hop prec=%d recon=%d dagger=%d epi=%d red=%d full=%d lat=%dx%dx%dx%d n5=%d", k.prec,
           k.recon, k.dagger, k.epi, k.red, k.full, k.X, k.Y, k.Z, k.T, k.n5);
  return buf;
}

static bool same_key(const HopKey& a, const HopKey& b) {
  return a.prec == b.prec && a.recon == b.recon && a.dagger == b.dagger && a.epi == b.epi && a.red == b.red &&
         a.full == b.full && a.X == b.X && a.Y == b.Y && a.Z == b.Z && a.T == b.T && a.n5 == b.n5;
}

// Every hop launch asks for its shape, so the answers are kept per thread until the
// table changes: formatting the key and finding its text took 0.3 of the 2.6 us that
// the host spends on a launch (it bounds M^dag M at 8^4).
bool hop_shape_lookup(const HopKey& k, int* idx) {
  struct Slot {
    uint64_t version = 0;
    HopKey key;
    int shape;
  };
  static thread_local Slot slots[64];
  const unsigned h = (unsigned)(k.prec + 3 * k.recon + 5 * k.dagger + 7 * k.epi + 29 * k.red + 31 * k.full + 37 * k.X +
                                41 * k.Y + 43 * k.Z + 47 * k.T + 53 * k.n5);
  Slot& s = slots[h % 64];
  const uint64_t version = g_tune_version.load();
  if (s.version != version || !same_key(s.key, k)) {
    int v = 0;
    if (!tune_lookup(hop_key_string(k), &v) || v < 0 || v >= HOP_SHAPES) return false;
    s.version = version;  // read before the table: a change since then is seen next time
    s.key = k;
    s.shape = v;
  }
  *idx = s.shape;
  return true;
}

bool hop_tuning_pass() { return g_tuning_pass; }

static std::mutex g_solver_mutex;
static std::set<std::string> g_solver_tuned;

bool solver_tuning_due(const std::string& key) {
  std::lock_guard<std::mutex> lock(g_solver_mutex);
  return g_solver_tuned.insert(key).second;
}

void solver_tuning_reset() {
  std::lock_guard<std::mutex> lock(g_solver_mutex);
  g_solver_tuned.clear();
}

TuningPass::TuningPass() : prev(g_tuning_pass) { g_tuning_pass = true; }
TuningPass::~TuningPass() { g_tuning_pass = prev; }
NoTuning::NoTuning() : prev(g_no_tuning) { g_no_tuning = true; }
NoTuning::~NoTuning() { g_no_tuning = prev; }

bool hop_autotune_ready(cudaStream_t s) {
  if (!g_autotune.load() || g_no_tuning) return false;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cs) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return cs == cudaStreamCaptureStatusNone;
}

int tune_hop_shapes(const HopKey& k, const std::function<int(int)>& launch, cudaStream_t s, int* best) {
  // Every shape is launched once to warm up, then timed in ROUNDS interleaved
  // rounds of PAIR back-to-back launches; a shape's time is its fastest round.
  // The default shape is kept unless another one is faster by at least MARGIN:
  // differences of a few per cent between shapes are within the spread of such
  // timings and would make the choice change from run to run.
  constexpr int ROUNDS = 3, PAIR = 2;
  constexpr float MARGIN = 0.97f;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return cuda_fail(cudaGetLastError(), "hop autotune: event create");
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return cuda_fail(cudaGetLastError(), "hop autotune: event create");
  }
  float t[HOP_SHAPES];
  int st = LQCD_OK;
  for (int i = 0; i < HOP_SHAPES && st == LQCD_OK; i++) {
    t[i] = 3.0e38f;
    if (hop_shape_applies(i, k.n5)) st = launch(i);
  }
  for (int r = 0; r < ROUNDS && st == LQCD_OK; r++) {
    for (int i = 0; i < HOP_SHAPES && st == LQCD_OK; i++) {
      if (!hop_shape_applies(i, k.n5)) continue;
      cudaEventRecord(e0, s);
      for (int q = 0; q < PAIR && st == LQCD_OK; q++) st = launch(i);
      cudaEventRecord(e1, s);
      if (st) break;
      cudaError_t e = cudaEventSynchronize(e1);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e != cudaSuccess) {
        st = cuda_fail(e, "hop autotune: timing");
        break;
      }
      if (ms < t[i]) t[i] = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st) return st;
  int b = HOP_SHAPE_DEFAULT;
  for (int i = 0; i < HOP_SHAPES; i++)
    if (t[i] < MARGIN * t[HOP_SHAPE_DEFAULT] && t[i] < t[b]) b = i;
  *best = b;
  tune_store(hop_key_string(k), b);
  return LQCD_OK;
}

}  // namespace lqcd

extern "C" {

void lqcd_tune_set_enabled(int on) { lqcd::g_autotune.store(on != 0); }

int lqcd_tune_get(const char* key) {
  int v = 0;
  if (!key || !lqcd::tune_lookup(key, &v)) return -1;
  return v;
}

}  // extern "C"
