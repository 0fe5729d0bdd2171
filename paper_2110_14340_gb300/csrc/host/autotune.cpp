// autotune.cpp - exhaustive autotuner over the 24 tile configurations.
//
// Auto-tuning is named as future work in the paper (§8); OptACC's grid
// search over OpenACC parallelism is the related prior art it cites (§7).
// For one descriptor the tuner specialises each valid tile, runs a
// graph-captured sweep sequence once to warm up, times `reps` further runs
// with CUDA events on the caller's stream and keeps the median per sweep.
// The fastest tile is remembered per shape, and whether it is ahead of the
// kernel that the library chooses by itself, timed in the same way: only then
// do later jacc_specialize calls with tile_id = -1 use it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <limits>
#include <string>
#include <vector>

#include "jacc_internal.h"

namespace jacc {

static std::map<std::string, TunedPick>& tune_cache() {
  static std::map<std::string, TunedPick> c;
  return c;
}

std::string shape_key(const jacc_kernel_desc& d) {
  jacc_kernel_desc c = d;
  c.tile_id = -1;
  c.flags = 0;
  c.reserved = 0;
  if (c.tblock == 0) c.tblock = 1;
  return std::string(reinterpret_cast<const char*>(&c), sizeof(c));
}

TunedPick tuned_pick(const jacc_kernel_desc& d) {
  std::lock_guard<std::mutex> lock(global_mutex());
  auto it = tune_cache().find(shape_key(d));
  return it == tune_cache().end() ? TunedPick() : it->second;
}

void remember_pick(const jacc_kernel_desc& d, const TunedPick& p) {
  std::lock_guard<std::mutex> lock(global_mutex());
  tune_cache()[shape_key(d)] = p;
}

}  // namespace jacc

using namespace jacc;

// A tile is ahead of the library's own kernel if its time is below this share
// of it: runs of one kernel differ by 1 or 2 %, and a pick timed on precompiled
// kernels is also the folded handles', where own kernels gain more (512^3 FP64,
// own and best tile, us a sweep: precompiled 382 and 388, folded 357 and 382).
constexpr double kAhead = 0.97;

// Median time per sweep (ms) of `reps` graph-launched runs after one to warm up.
static jacc_status time_sweeps(jacc_kernel k, void* u0, void* u1, int32_t sweeps, int32_t reps, uintptr_t stream,
                               cudaEvent_t e0, cudaEvent_t e1, double* out) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  std::vector<double> times;
  int32_t fb = 0;
  jacc_status st = ok();
  for (int r = 0; r <= reps && !st; ++r) {
    st = cuda_check(cudaEventRecord(e0, s), "cudaEventRecord");
    if (!st) st = jacc_sweep(k, u0, u1, sweeps, nullptr, JACC_SWEEP_GRAPH, stream, &fb);
    if (!st) st = cuda_check(cudaEventRecord(e1, s), "cudaEventRecord");
    if (!st) st = cuda_check(cudaEventSynchronize(e1), "cudaEventSynchronize");
    float ms = 0.f;
    if (!st) st = cuda_check(cudaEventElapsedTime(&ms, e0, e1), "cudaEventElapsedTime");
    if (!st && r > 0) times.push_back(static_cast<double>(ms) / sweeps);  // run 0 warms up
  }
  if (st) return st;
  std::sort(times.begin(), times.end());
  *out = times[times.size() / 2];
  return st;
}

// Times the tiles with want[t] set (each valid one), fills `out`, and remembers
// the fastest for the shape and whether it is ahead of the library's own kernel.
static jacc_status autotune_subset(const jacc_kernel_desc* desc, void* u0, void* u1, int32_t sweeps_per_rep,
                                   int32_t reps, uintptr_t stream, const bool* want, jacc_tune_result* out) {
  if (!desc || !out || sweeps_per_rep < 1 || reps < 1) return fail(JACC_ERR_INVALID_ARG, "bad autotune arguments");
  cudaEvent_t e0, e1;
  jacc_status st = cuda_check(cudaEventCreate(&e0), "cudaEventCreate");
  if (st) return st;
  st = cuda_check(cudaEventCreate(&e1), "cudaEventCreate");
  if (st) {
    cudaEventDestroy(e0);
    return st;
  }
  out->best_tile = -1;
  out->best_ms = std::numeric_limits<double>::infinity();
  jacc_kernel_desc d = *desc;
  d.flags &= ~JACC_SPEC_JIT;
  for (int t = 0; t < JACC_NUM_TILES && !st; ++t) {
    out->ms[t] = std::numeric_limits<double>::infinity();
    out->valid[t] = 0;
    d.tile_id = t;
    if (!want[t] || !tile_valid(d, t)) continue;
    jacc_kernel k = nullptr;
    st = jacc_specialize(&d, &k);
    if (st) break;
    st = time_sweeps(k, u0, u1, sweeps_per_rep, reps, stream, e0, e1, &out->ms[t]);
    jacc_release(k);
    if (st) break;
    out->valid[t] = 1;
    if (out->ms[t] < out->best_ms) {
      out->best_ms = out->ms[t];
      out->best_tile = t;
    }
  }
  TunedPick pick;
  pick.tile = out->best_tile;
  pick.ahead = true;
  if (!st && out->best_tile >= 0 && desc->tblock <= 1) {
    d.tile_id = -1;
    jacc_kernel k = nullptr;
    double own = 0.0;
    st = specialize_own(d, &k);
    if (!st) {
      st = time_sweeps(k, u0, u1, sweeps_per_rep, reps, stream, e0, e1, &own);
      jacc_release(k);
      pick.ahead = out->best_ms < kAhead * own;
    } else if (st == JACC_ERR_INVALID_ARG) {
      st = ok();  // its tile does not cover this many rows
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st) return st;
  if (out->best_tile < 0) return fail(JACC_ERR_UNSUPPORTED, "no tile configuration fits this shape");
  remember_pick(*desc, pick);
  return ok();
}

extern "C" jacc_status jacc_autotune(const jacc_kernel_desc* desc, void* u0, void* u1, int32_t sweeps_per_rep,
                                     int32_t reps, uintptr_t stream, jacc_tune_result* out) {
  bool all[JACC_NUM_TILES];
  std::fill(all, all + JACC_NUM_TILES, true);
  return autotune_subset(desc, u0, u1, sweeps_per_rep, reps, stream, all, out);
}

extern "C" jacc_status jacc_autotune_tiles(const jacc_kernel_desc* desc, void* u0, void* u1, int32_t sweeps_per_rep,
                                           int32_t reps, uintptr_t stream, const int32_t* tiles, int32_t ntiles,
                                           jacc_tune_result* out) {
  if (!tiles || ntiles < 1) return fail(JACC_ERR_INVALID_ARG, "no tiles to time");
  bool want[JACC_NUM_TILES];
  std::fill(want, want + JACC_NUM_TILES, false);
  for (int32_t i = 0; i < ntiles; ++i) {
    if (tiles[i] < 0 || tiles[i] >= JACC_NUM_TILES) return fail(JACC_ERR_INVALID_ARG, "tile id out of range");
    want[tiles[i]] = true;
  }
  return autotune_subset(desc, u0, u1, sweeps_per_rep, reps, stream, want, out);
}

extern "C" jacc_status jacc_autotune_forget(void) {
  std::lock_guard<std::mutex> lock(global_mutex());
  tune_cache().clear();
  return ok();
}
