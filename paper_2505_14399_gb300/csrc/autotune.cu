// Launch-shape autotuner: times each candidate once per problem key and caches the winner.
//
// The first call with a new (kernel, dtype, parity, dagger, volume, nrhs) key runs every
// candidate shape on the caller's own arguments (one warm-up and three timed launches
// each, CUDA events on the caller's stream) and keeps the fastest; later calls reuse the
// choice.  Calls made while the stream is being captured into a graph never tune (they use
// the default shape).  WMG_DSLASH_VARIANT=<i> in the environment forces a shape.
//
// Persistence: with WMG_AUTOTUNE_CACHE=<file> the choices are also kept in that file, one JSON
// object per line ({"device": ..., "shapes": ..., "dtype": ..., "parity": ..., "dagger": ...,
// "volume": ..., "nrhs": ..., "variant": ..., "ms": ..., "all_ms": [every candidate's time]}); the
// file is read once per process and every new choice is appended, so later processes on the same
// kind of GPU skip the timing.  Entries of other device names are ignored, and so are those of
// another shape table, whose variant numbers mean other kernels.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace wmg {

namespace {
// Version of the shape numbering (csrc/dslash.cu, csrc/krylov.cu): goes up with every change of what
// a variant number launches.  Tables 1 and 2 wrote no version.
constexpr int kShapeTable = 4;

typedef std::tuple<int, int, int, int, int> Key;
std::map<Key, std::pair<int, float>> g_cache;
std::mutex g_mu;
std::string g_report;
bool g_loaded = false;

std::string device_name() {
  int dev = 0;
  cudaDeviceProp pr{};
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&pr, dev) != cudaSuccess) {
    cudaGetLastError();
    return "unknown";
  }
  std::string n = pr.name;
  for (auto& ch : n)
    if (ch == '"' || ch == '\\') ch = '_';
  return n;
}

// caller holds g_mu
void load_cache_file() {
  if (g_loaded) return;
  g_loaded = true;
  const char* path = std::getenv("WMG_AUTOTUNE_CACHE");
  if (!path) return;
  FILE* f = std::fopen(path, "r");
  if (!f) return;
  const std::string want = "{\"device\":\"" + device_name() +
                           "\",\"shapes\":" + std::to_string(kShapeTable) + ",";
  char line[512];
  while (std::fgets(line, sizeof(line), f)) {
    std::string s(line);
    if (s.compare(0, want.size(), want) != 0) continue;
    int dt, par, dag, V, nrhs, var;
    float ms;
    if (std::sscanf(s.c_str() + want.size(),
                    "\"dtype\":%d,\"parity\":%d,\"dagger\":%d,\"volume\":%d,\"nrhs\":%d,"
                    "\"variant\":%d,\"ms\":%f",
                    &dt, &par, &dag, &V, &nrhs, &var, &ms) == 7)
      g_cache[Key(dt, par, dag, V, nrhs)] = std::make_pair(var, ms);
  }
  std::fclose(f);
}

// caller holds g_mu
void append_cache_file(const Key& k, int var, float ms, const std::vector<float>& all) {
  const char* path = std::getenv("WMG_AUTOTUNE_CACHE");
  if (!path) return;
  FILE* f = std::fopen(path, "a");
  if (!f) return;
  std::fprintf(f,
               "{\"device\":\"%s\",\"shapes\":%d,\"dtype\":%d,\"parity\":%d,\"dagger\":%d,"
               "\"volume\":%d,\"nrhs\":%d,\"variant\":%d,\"ms\":%.6g,\"all_ms\":[",
               device_name().c_str(), kShapeTable, std::get<0>(k), std::get<1>(k), std::get<2>(k),
               std::get<3>(k), std::get<4>(k), var, ms);
  for (size_t i = 0; i < all.size(); ++i) std::fprintf(f, i ? ",%.6g" : "%.6g", all[i]);
  std::fprintf(f, "]}\n");
  std::fclose(f);
}
}  // namespace

int tuned_variant(int dtype, int parity, int dagger, int V, int nrhs, cudaStream_t st, int nvar,
                  const std::function<void(int)>& run) {
  static int forced = [] {
    const char* e = std::getenv("WMG_DSLASH_VARIANT");
    return e ? std::atoi(e) : -1;
  }();
  if (forced >= 0 && forced < nvar) return forced;
  Key key(dtype, parity, dagger, V, nrhs);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    load_cache_file();
    auto it = g_cache.find(key);
    if (it != g_cache.end() && (it->second.first < 0 || it->second.first >= nvar)) {
      g_cache.erase(it);
      it = g_cache.end();
    }
    if (it != g_cache.end()) return it->second.first;
  }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return 0;
  }
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return -1;
  int best = 0;
  float best_ms = 1e30f;
  std::vector<float> all;
  for (int v = 0; v < nvar; ++v) {
    run(v);
    cudaEventRecord(e0, st);
    for (int r = 0; r < 3; ++r) run(v);
    cudaEventRecord(e1, st);
    if (cudaEventSynchronize(e1) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      return -1;
    }
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    count_launch(4);
    all.push_back(ms / 3.0f);
    if (ms < best_ms) {
      best_ms = ms;
      best = v;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  std::lock_guard<std::mutex> lk(g_mu);
  g_cache[key] = std::make_pair(best, best_ms / 3.0f);
  append_cache_file(key, best, best_ms / 3.0f, all);
  return best;
}

const char* tune_report() {
  std::lock_guard<std::mutex> lk(g_mu);
  std::ostringstream os;
  os << "[";
  bool first = true;
  for (auto& kv : g_cache) {
    if (!first) os << ",";
    first = false;
    // key ranges: stencil dtype codes below 1000, the fused stencil + projections from 1000
    const int dt = std::get<0>(kv.first);
    const char* kern = dt >= 1000 ? "dslash_proj" : "dslash";
    os << "{\"kernel\":\"" << kern << "\",\"dtype\":" << dt
       << ",\"parity\":" << std::get<1>(kv.first) << ",\"dagger\":" << std::get<2>(kv.first)
       << ",\"volume\":" << std::get<3>(kv.first) << ",\"nrhs\":" << std::get<4>(kv.first)
       << ",\"variant\":" << kv.second.first << ",\"ms\":" << kv.second.second << "}";
  }
  os << "]";
  g_report = os.str();
  return g_report.c_str();
}

}  // namespace wmg

extern "C" const char* mg_autotune_report(void) { return wmg::tune_report(); }
