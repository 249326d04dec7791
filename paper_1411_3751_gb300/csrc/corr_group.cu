// Groups of sub-arrays of the C ABI (corr_group_*): several contexts of different N and C with one
// block length, correlated by one call.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <tuple>
#include <vector>

#include "corr_ctx.cuh"
#include "corr_internal.cuh"

using namespace corr;
using namespace corr::host;

struct corr_group {
  int n;
  corr_ctx* ctx[kMaxGroupArrays];
  GroupWork work;
  cudaGraphExec_t graph;
  // members whose operand scratch the graph uses, and their op_released at the capture
  bool on_scratch[kMaxGroupArrays];
  unsigned released[kMaxGroupArrays];
  int T;
};

namespace {

// autotuner cache: (N, C, T, n_pol, SMs, launched by itself) -> tile plan; optionally mirrored in the file named by the
// CORR_AUTOTUNE_CACHE environment variable (lines "group N C T n_pol SMs by_itself plan"; lines without the tag are
// an earlier version's, whose plans were chosen among fewer and for launches that are no longer made)
typedef std::tuple<int, int, int, int, int, int> TuneKey;
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tune;
bool g_tune_loaded = false;

void tune_load() {
  if (g_tune_loaded) return;
  g_tune_loaded = true;
  const char* path = std::getenv("CORR_AUTOTUNE_CACHE");
  if (!path) return;
  FILE* fh = std::fopen(path, "r");
  if (!fh) return;
  char line[256];
  int a, b, c, d, e, f, p;
  while (std::fgets(line, sizeof line, fh))  // other lines in the file belong to other tuners
    if (std::sscanf(line, "group %d %d %d %d %d %d %d", &a, &b, &c, &d, &e, &f, &p) == 7) g_tune[TuneKey(a, b, c, d, e, f)] = p;
  std::fclose(fh);
}

void tune_store(const TuneKey& k, int plan) {
  g_tune[k] = plan;
  const char* path = std::getenv("CORR_AUTOTUNE_CACHE");
  if (!path) return;
  FILE* fh = std::fopen(path, "a");
  if (!fh) return;
  std::fprintf(fh, "group %d %d %d %d %d %d %d\n", std::get<0>(k), std::get<1>(k), std::get<2>(k), std::get<3>(k),
               std::get<4>(k), std::get<5>(k), plan);
  std::fclose(fh);
}

// Arrays that take two passes share one build and one X-engine launch on the one-SM kernel, where one array's last wave
// is filled by the next one's items (with their dumps, 4096 samples: eight arrays of 256 inputs x 4 channels 387 us
// each by itself, 177 so; four of 256 x 40 387 and 302; 32 to 512 inputs x 2400 to 109 channels 1285 and 1216). On SM
// pairs (plan 3) an array with long items is faster by itself: two of 512 x 109 911 us apart and 864 merged at 4096
// samples, 978 and 945 at 5120, but 1052 and 1072 at 6144 and 1267 and 1323 at 8192; three of 512 x 40 (5 items a
// pair) 817 and 770 there.
constexpr int kPairAloneSamples = 5632, kPairAloneItems = 8;  // longer blocks, at least so many items an SM pair
bool long_on_pairs(const corr_ctx* c) {
  return c->L.T_pad > kPairAloneSamples &&
         (long long)work_items(c->L, 3).size() >= (long long)kPairAloneItems * (c->num_sms / 2);
}
bool launches_alone(const corr_ctx* c) { return c->tile_plan == 3 && long_on_pairs(c); }

// The work lists of the arrays that take two passes: the merged ones', in order of decreasing N (short items last, where
// they even out the tail; plan 0 for 2 and 3), and the others', each on its tile plan. Replaces the group's
// lists, so a graph that reads these has to be dropped first.
int group_build_work(corr_group* g) {
  GroupWork w{};
  std::vector<WorkItem> items;
  std::vector<int> merged;
  for (int i = 0; i < g->n; ++i)
    if (takes_two_passes(g->ctx[i]) && !launches_alone(g->ctx[i])) merged.push_back(i);
  if (merged.size() < 2) merged.clear();
  std::stable_sort(merged.begin(), merged.end(), [&](int x, int y) { return g->ctx[x]->L.s.N > g->ctx[y]->L.s.N; });
  for (int i : merged) {
    const corr_ctx* c = g->ctx[i];
    w.in_merged[i] = true;
    for (WorkItem it : work_items(c->L, c->tile_plan >= 2 ? 0 : c->tile_plan)) {
      it.array = i;
      items.push_back(it);
    }
  }
  w.merged = GroupWork::List{0, (long long)items.size(), 0};
  for (int i = 0; i < g->n; ++i) {
    const corr_ctx* c = g->ctx[i];
    if (!takes_two_passes(c) || w.in_merged[i]) continue;
    const std::vector<WorkItem> own = work_items(c->L, c->tile_plan);
    w.own[i] = GroupWork::List{(long long)items.size(), (long long)own.size(), c->tile_plan};
    items.insert(items.end(), own.begin(), own.end());
  }
  if (!items.empty()) {
    if (cudaMalloc(&w.d_items, items.size() * sizeof(WorkItem)) != cudaSuccess) {
      cudaGetLastError();
      return fail(CORR_ERR_OOM, "group work list allocation failed");
    }
    const cudaError_t e = cudaMemcpy(w.d_items, items.data(), items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
      cudaFree(w.d_items);
      return cuda_fail(e, "group work list upload");
    }
  }
  cudaFree(g->work.d_items);
  g->work = w;
  return CORR_OK;
}

// One grouped accumulate.
int group_enqueue(corr_group* g, const uint8_t* const* in, cudaStream_t st) {
  for (int i = 0; i < g->n; ++i)
    if (!g->ctx[i]->d_op)
      return fail(CORR_ERR_STATE, "group member " + std::to_string(i) +
                                      " has no operand scratch (its path was set to FP32 or int8; set a tensor path)");
  return enqueue_group(g->ctx, g->n, g->work, in, st);
}

void group_count(corr_group* g) {
  for (int i = 0; i < g->n; ++i) {
    corr_ctx* c = g->ctx[i];
    c->n_cross += c->L.s.T;
    c->n_auto += c->L.s.T;
    c->n_off += c->L.s.T;
    c->n_off_auto += c->L.s.T;
  }
}

}  // namespace

extern "C" {

corr_group* corr_group_create(int n_arrays, const int* n_inputs, const int* n_chans, int n_time_per_block, int n_pol) {
  if (n_arrays < 1 || n_arrays > kMaxGroupArrays || !n_inputs || !n_chans) {
    fail(CORR_ERR_ARG, "corr_group_create: need 1.." + std::to_string(kMaxGroupArrays) + " sub-arrays");
    return nullptr;
  }
  corr_group* g = new (std::nothrow) corr_group{};
  if (!g) {
    fail(CORR_ERR_OOM, "corr_group_create: host allocation");
    return nullptr;
  }
  g->n = n_arrays;
  g->T = n_time_per_block;
  for (int i = 0; i < n_arrays; ++i) {
    g->ctx[i] = corr_create(n_inputs[i], n_chans[i], n_time_per_block, n_pol);
    if (!g->ctx[i]) {
      const std::string msg = corr_last_error();
      corr_group_destroy(g);
      fail(CORR_ERR_ARG, "corr_group_create: sub-array " + std::to_string(i) + ": " + msg);
      return nullptr;
    }
  }
  if (group_build_work(g) != CORR_OK) {
    const std::string msg = corr_last_error();
    corr_group_destroy(g);
    fail(CORR_ERR_OOM, "corr_group_create: " + msg);
    return nullptr;
  }
  return g;
}

corr_ctx* corr_group_member(corr_group* g, int i) {
  if (!g || i < 0 || i >= g->n) {
    fail(CORR_ERR_ARG, "corr_group_member: bad index");
    return nullptr;
  }
  return g->ctx[i];
}

int corr_group_accumulate(corr_group* g, const void* const* d_samples, int mode, void* stream) {
  if (!g || !d_samples) return fail(CORR_ERR_ARG, "corr_group_accumulate: NULL argument");
  for (int i = 0; i < g->n; ++i)
    if (!d_samples[i]) return fail(CORR_ERR_ARG, "corr_group_accumulate: NULL block " + std::to_string(i));
  cudaStream_t st = (cudaStream_t)stream;
  const uint8_t* const* in = reinterpret_cast<const uint8_t* const*>(d_samples);
  if (mode == 1) {
    for (int i = 0; i < g->n; ++i) {
      const int rc = corr_accumulate(g->ctx[i], d_samples[i], stream);
      if (rc != CORR_OK) return rc;
    }
    return CORR_OK;
  }
  if (mode != 0) return fail(CORR_ERR_ARG, "corr_group_accumulate: mode must be 0 (grouped) or 1 (separate)");
  const int rc = group_enqueue(g, in, st);
  if (rc != CORR_OK) return rc;
  group_count(g);
  return CORR_OK;
}

int corr_group_autotune(corr_group* g, const void* const* d_samples, int* plans_out, void* stream) {
  if (!g || !d_samples) return fail(CORR_ERR_ARG, "corr_group_autotune: NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> lock(g_tune_mu);
  tune_load();
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return cuda_fail(cudaGetLastError(), "corr_group_autotune: events");
  int rc = CORR_OK, n_two_pass = 0;
  for (int i = 0; i < g->n; ++i) n_two_pass += takes_two_passes(g->ctx[i]);
  for (int i = 0; i < g->n && rc == CORR_OK; ++i) {
    corr_ctx* c = g->ctx[i];
    if (!takes_two_passes(c)) {  // correlated without a tile plan in a group, and by itself on the default one
      if (c->tile_plan != c->plan_default) rc = set_tile_plan(c, c->plan_default);
      if (rc == CORR_OK) rc = corr_reset(c, CORR_WHAT_CROSS | CORR_WHAT_AUTO, stream);
      if (plans_out) plans_out[i] = c->plan_default;
      continue;
    }
    // the plans that the group's launch can run the array on: the one-SM ones, and SM pairs where that is the default
    // and the array would not be merged on it
    const bool by_itself = n_two_pass == 1 || long_on_pairs(c);
    std::vector<int> plans = {0, 1};
    if (by_itself && c->plan_default == 3) plans = {3, 0, 1};
    const TuneKey key(c->L.s.N, c->L.s.C, c->L.s.T, c->L.s.npol, c->num_sms, by_itself);
    auto it = g_tune.find(key);
    int best = plans[0];
    if (it != g_tune.end() && std::find(plans.begin(), plans.end(), it->second) != plans.end()) {
      best = it->second;
    } else {
      float best_ms = 1e30f;
      for (int plan : plans) {
        rc = set_tile_plan(c, plan);
        if (rc != CORR_OK) break;
        // one warm-up block, then three timed blocks through the tensor path of this array alone
        for (int rep = 0; rep < 4 && rc == CORR_OK; ++rep) {
          if (rep == 1) cudaEventRecord(e0, st);
          rc = accumulate_device(c, static_cast<const uint8_t*>(d_samples[i]), c->L.s.T, st);
        }
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) rc = cuda_fail(cudaGetLastError(), "corr_group_autotune");
        if (rc != CORR_OK) break;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best_ms) {
          best_ms = ms;
          best = plan;
        }
      }
      if (rc == CORR_OK) tune_store(key, best);
    }
    if (rc == CORR_OK) rc = set_tile_plan(c, best);
    if (rc == CORR_OK) rc = corr_reset(c, CORR_WHAT_CROSS | CORR_WHAT_AUTO, stream);
    if (plans_out) plans_out[i] = best;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != CORR_OK) return rc;
  // a captured graph would keep the old plans' launches: drop it (corr_group_capture records a new one)
  if (g->graph) {
    cudaGraphExecDestroy(g->graph);
    g->graph = nullptr;
  }
  return group_build_work(g);
}

int corr_group_capture(corr_group* g, const void* const* d_samples, void* stream) {
  if (!g || !d_samples) return fail(CORR_ERR_ARG, "corr_group_capture: NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  if (!st) return fail(CORR_ERR_ARG, "corr_group_capture: needs a non-default stream");
  bool prof[kMaxGroupArrays];
  for (int i = 0; i < g->n; ++i) {
    prof[i] = g->ctx[i]->profiling;
    g->ctx[i]->profiling = false;  // no timing events inside the graph
  }
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
  int rc = CORR_OK;
  if (e == cudaSuccess) {
    rc = group_enqueue(g, reinterpret_cast<const uint8_t* const*>(d_samples), st);
    e = cudaStreamEndCapture(st, &graph);
  }
  for (int i = 0; i < g->n; ++i) g->ctx[i]->profiling = prof[i];
  if (rc != CORR_OK) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return cuda_fail(e, "corr_group_capture: capture");
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return cuda_fail(e, "corr_group_capture: instantiate");
  if (g->graph) cudaGraphExecDestroy(g->graph);
  g->graph = exec;
  for (int i = 0; i < g->n; ++i) {
    g->on_scratch[i] = uses_operand_scratch(g->ctx[i], static_cast<const uint8_t*>(d_samples[i]));
    g->released[i] = g->ctx[i]->op_released;
  }
  return CORR_OK;
}

int corr_group_launch(corr_group* g, void* stream) {
  if (!g) return fail(CORR_ERR_ARG, "corr_group_launch: NULL group");
  if (!g->graph) return fail(CORR_ERR_STATE, "corr_group_launch: no captured graph (call corr_group_capture)");
  for (int i = 0; i < g->n; ++i)
    if (g->on_scratch[i] && g->released[i] != g->ctx[i]->op_released)
      return fail(CORR_ERR_STATE, "corr_group_launch: member " + std::to_string(i) +
                                      " has released the operand scratch that the graph uses (its path or blocks per "
                                      "launch changed): call corr_group_capture again");
  cudaError_t e = cudaGraphLaunch(g->graph, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "corr_group_launch");
  group_count(g);
  return CORR_OK;
}

int corr_group_destroy(corr_group* g) {
  if (!g) return CORR_OK;
  int rc = CORR_OK;
  if (g->graph) cudaGraphExecDestroy(g->graph);
  cudaFree(g->work.d_items);
  for (int i = 0; i < g->n; ++i)
    if (g->ctx[i] && corr_destroy(g->ctx[i]) != CORR_OK) rc = CORR_ERR_CUDA;
  delete g;
  return rc;
}

}  // extern "C"
