// Launch-shape autotuner for the fused sweeps.
//
// The paper derives its spatial blocking from machine properties (the layer
// condition, Sec. 3.1); here the launch shape of the z-marching sweep is
// chosen by measurement instead: threads per block, resident blocks per SM
// and z-slab depth are swept with CUDA events on the caller's stream, timing
// the sweeps of the operation that will run (KPM: recurrence update + fp64 dot
// products; series: the accumulating sweep and the two plain ones that
// follow it; apply: the plain sweep), and the fastest shape is stored in the
// lattice handle.
// With PVSC_TUNE_CACHE=<file> results are kept on disk, keyed by model,
// dimensions, boundary conditions, R, precision and device name.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"
#include "sweep.cuh"

namespace pvsc {

static std::string cache_key(const pvsc_lattice* lat, int R, int prec, int op) {
  cudaDeviceProp prop;
  std::string dev = "gpu";
  if (cudaGetDeviceProperties(&prop, lat->device) == cudaSuccess) dev = prop.name;
  for (auto& c : dev)
    if (c == ' ') c = '_';
  char buf[512];
  snprintf(buf, sizeof(buf), "%d %lld %lld %lld %d%d%d %d %d %s%s", lat->g.model, (long long)lat->g.L[0],
           (long long)lat->g.L[1], (long long)lat->g.L[2], lat->g.per[0], lat->g.per[1], lat->g.per[2], R,
           prec, dev.c_str(), op == PVSC_OP_KPM ? "" : (op == PVSC_OP_SERIES ? " series" : " apply"));
  return buf;
}

static bool cache_lookup(const std::string& key, pvsc_tuning* t) {
  const char* path = std::getenv("PVSC_TUNE_CACHE");
  if (!path || !path[0]) return false;
  FILE* f = std::fopen(path, "r");
  if (!f) return false;
  char line[1024];
  bool found = false;
  while (std::fgets(line, sizeof(line), f)) {
    char* bar = std::strchr(line, '|');
    if (!bar) continue;
    *bar = 0;
    if (key != line) continue;
    pvsc_tuning c;
    if (std::sscanf(bar + 1, "%d %d %d %f %d %d %d %d", &c.threads, &c.blocks_per_sm, &c.zslab,
                    &c.time_ms, &c.vpt, &c.tile_x, &c.tile_y, &c.kernel) == 8) {
      *t = c;
      found = true;
    }
  }
  std::fclose(f);
  return found;
}

static void cache_store(const std::string& key, const pvsc_tuning& t) {
  const char* path = std::getenv("PVSC_TUNE_CACHE");
  if (!path || !path[0]) return;
  FILE* f = std::fopen(path, "a");
  if (!f) return;
  std::fprintf(f, "%s|%d %d %d %.6f %d %d %d %d\n", key.c_str(), t.threads, t.blocks_per_sm, t.zslab,
               t.time_ms, t.vpt, t.tile_x, t.tile_y, t.kernel);
  std::fclose(f);
}

// The untuned sweeps as a candidate, where no tuning entry can select them: the TMA-staged tiles of a
// lattice with Lx no multiple of 4 and of complex128 vectors, and the mix of a series (plain sweeps on
// eight warps, accumulating ones on sixteen; an entry holds one count: a filter of 240x240x6 sites,
// R = 32, K = 100, 27.5 ms, 28.2 with the best entry).  kernel = PVSC_UNTUNED with threads = 0 stands for them
// in the list and in the cache file, and installing it removes the entry.  The caller is told what
// pvsc_get_tuning then reads.
constexpr pvsc_tuning kUntuned{0, 0, 0, 0.f, 0, 0, 0, PVSC_UNTUNED};
static bool untuned_is_its_own(const pvsc_lattice* lat, int R, int prec, int op) {
  if (default_kernel(lat, R, prec) != kKernelTma) return false;
  return prec == PVSC_C128 || op == PVSC_OP_SERIES || !tma_sweep_possible(lat, R, prec);
}

static void install(pvsc_lattice* lat, int R, int prec, const pvsc_tuning& t) {
  if (t.threads > 0 && t.kernel != PVSC_UNTUNED) lat->tuning[{R, prec}] = t;
  else lat->tuning.erase({R, prec});
}

static pvsc_tuning reported(pvsc_tuning t, int R, int prec) {
  if (t.threads == 0) {
    t.threads = 256;
    t.vpt = vpt_for(R, prec);
    t.kernel = PVSC_UNTUNED;
  }
  return t;
}

// The shapes that are timed: z-marching (all shapes), for TI the flat, prefetching and shared-memory
// staged sweeps in a few shapes each, the TMA-staged tiles, and the untuned sweeps as above.
static std::vector<pvsc_tuning> candidates(const pvsc_lattice* lat, int R, int prec, int op) {
  std::vector<int> vpt_c = {1};
  if (prec == PVSC_C64 && R >= 2) vpt_c.push_back(2);
  std::vector<int> zslab_c = {0};
  const bool march = lat->g.model == PVSC_TI || lat->g.model == PVSC_WSM;  // z-marching sweeps
  if (march)
    for (int z : {4, 8, 16, 32, 64})
      if (z < lat->g.L[2]) zslab_c.push_back(z);
  const std::vector<int> bps_c = {0, 1, 2};
  std::vector<pvsc_tuning> cands;
  if (untuned_is_its_own(lat, R, prec, op)) cands.push_back(kUntuned);
  for (int vpt : vpt_c) {
    const int C = R / vpt;
    for (int th : {64, 128, 256}) {
      if (th % C != 0 || th < C) continue;
      for (int bps : bps_c)
        for (int zs : zslab_c) cands.push_back(pvsc_tuning{th, bps, zs, 0.f, vpt, 0, 0, 0});
      if (march) cands.push_back(pvsc_tuning{th, 0, 0, 0.f, vpt, 0, 0, 1});  // flat variant
      if (lat->g.model == PVSC_TI) {
        // column tiles of this many threads (z-marching, kernel 5)
        const int tiles5[][2] = {{4, 4}, {8, 4}, {4, 8}, {8, 8}, {16, 4}, {16, 2}, {2, 8}};
        for (const auto& t : tiles5)
          if (t[0] * t[1] * C == th) cands.push_back(pvsc_tuning{th, 0, 0, 0.f, vpt, t[0], t[1], 5});
        // marching along x (lattices with a short z extent)
        if (lat->g.L[0] > lat->g.L[2]) cands.push_back(pvsc_tuning{th, 0, 0, 0.f, vpt, 0, 0, 6});
        if (!(prec == PVSC_C64 && vpt == 1 && R > 1)) {
          for (int zs : {0, 16}) cands.push_back(pvsc_tuning{th, 0, zs, 0.f, vpt, 0, 0, 2});
          cands.push_back(pvsc_tuning{th, 0, 0, 0.f, vpt, 0, 0, 3});
        }
      }
    }
  }
  // TMA-staged plane tiles (kernel 7): z-chunks chosen automatically or a few fixed depths
  if (tma_sweep_possible(lat, R, prec)) {
    // the half tiles of the deeper rings (R = 32, 64: slices on the tiles of R = 16)
    const int deep_y = R == 1 ? 16 : (R == 2 || R == 4) ? 8 : 4, deep_x = R >= 16 ? 8 : (R <= 2 ? 32 : 16);
    // blocks_per_sm 1: spread the planes over every SM when there are fewer units
    // than SMs (the same launch otherwise, and with automatic chunks, which spread anyway)
    for (int zs : {0, 16, 32, 64})
      if (zs == 0 || zs < lat->g.L[2])
        for (int spread = 0; spread < (zs == 0 ? 1 : 2); ++spread) {
          cands.push_back(pvsc_tuning{256, spread, zs, 0.f, 2, 0, 0, kKernelTma});
          cands.push_back(pvsc_tuning{256, spread, zs, 0.f, 2, deep_x, deep_y, kKernelTma});
          if (lat->g.model == PVSC_TI)  // the Weyl cells run eight warps only
            cands.push_back(pvsc_tuning{512, spread, zs, 0.f, 2, 0, 0, kKernelTma});
        }
    // the same tiles marching along x, where the z columns are the shorter
    if (lat->g.L[0] > lat->g.L[2] && tma_xm_possible(lat, R, prec))
      for (int zs : {0, 32, 64})
        if (zs == 0 || zs < lat->g.L[0]) {
          cands.push_back(pvsc_tuning{256, 0, zs, 0.f, 2, 0, 0, kKernelTmaX});
          if (lat->g.model == PVSC_TI) cands.push_back(pvsc_tuning{256, 0, zs, 0.f, 2, deep_x, deep_y, kKernelTmaX});
        }
  }
  if (lat->g.model == PVSC_TI)
    for (int th : {128, 256}) {
      if (th % R) continue;
      const int tiles[][2] = {{32, 8}, {16, 8}, {16, 4}, {8, 8}, {8, 4}, {4, 4}};
      for (const auto& t : tiles)
        if (t[0] * t[1] <= 2 * th && bulk_smem_bytes(t[0], t[1], R, prec) <= 200 * 1024)
          cands.push_back(pvsc_tuning{th, 0, 0, 0.f, 1, t[0], t[1], 0});
    }
  return cands;
}

}  // namespace pvsc

using namespace pvsc;

extern "C" int pvsc_autotune_op(pvsc_lattice* lat, int R, int prec, int op, pvsc_tuning* best, void* stream) {
  if (int rc = check_lattice(lat)) return rc;
  if (!valid_R(R)) return set_error(PVSC_ERR_ARG, "R = %d: must be 1, 2, 4, 8, 16, 32 or 64", R);
  if (prec != PVSC_C128 && prec != PVSC_C64) return set_error(PVSC_ERR_ARG, "unknown precision %d", prec);
  if (op != PVSC_OP_KPM && op != PVSC_OP_SERIES && op != PVSC_OP_APPLY)
    return set_error(PVSC_ERR_ARG, "autotune op must be PVSC_OP_KPM, PVSC_OP_SERIES or PVSC_OP_APPLY");
  const std::string key = cache_key(lat, R, prec, op);
  pvsc_tuning cached;
  if (cache_lookup(key, &cached)) {
    install(lat, R, prec, cached);
    drop_graphs(lat);
    if (best) *best = reported(cached, R, prec);
    return PVSC_OK;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t vb = vec_bytes(lat, R, prec), wb = dots_work_bytes(lat, R);
  void *x = nullptr, *y = nullptr, *work = nullptr, *acc = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  int rc = PVSC_OK;
  auto cleanup = [&]() {
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(x);
    cudaFree(y);
    cudaFree(work);
    cudaFree(acc);
  };
  const size_t ab = op == PVSC_OP_SERIES ? vec_bytes(lat, R, PVSC_C128) : 16;
  if (cudaMalloc(&x, vb) != cudaSuccess || cudaMalloc(&y, vb) != cudaSuccess ||
      cudaMalloc(&work, wb) != cudaSuccess || cudaMalloc(&acc, ab) != cudaSuccess) {
    cleanup();
    return set_error(PVSC_ERR_OOM, "autotune could not allocate its sweep vectors");
  }
  // random-phase vectors (and accumulator): the sweeps are timed on data like a run's
  {
    const int64_t D = lat->g.n_sites * orbitals_of(lat->g.model);
    rc = launch_random_phase(x, prec, D, R, 0x5eed1, st);
    if (rc == PVSC_OK) rc = launch_random_phase(y, prec, D, R, 0x5eed2, st);
    if (rc == PVSC_OK && op == PVSC_OP_SERIES) rc = launch_random_phase(acc, PVSC_C128, D, R, 0x5eed3, st);
    if (rc != PVSC_OK) {
      cleanup();
      return rc;
    }
  }
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  auto saved = lat->tuning.find({R, prec});
  const bool had = saved != lat->tuning.end();
  const pvsc_tuning old = had ? saved->second : pvsc_tuning{};
  pvsc_tuning win{256, 0, 0, 1e30f, 0, 0, 0, 0};
  // time one candidate shape: one warm run, then the best of three trials of
  // three runs each, with the sweep features of the operation: KPM (recurrence
  // + dots), series (the accumulating sweep and the two plain ones that follow
  // it), apply (plain)
  auto time_one = [&](const pvsc_tuning& cand, float* ms) -> int {
    install(lat, R, prec, cand);
    Sweep p;
    sweep_init(p, lat, R, prec);
    for (int r = 0; r < R; ++r) {
      p.coef[0][r] = 0.2;
      p.coef[1][r] = 0.0;
      p.coef[2][r] = op == PVSC_OP_APPLY ? 0.0 : -1.0;
    }
    p.x = x;
    p.yin = op == PVSC_OP_APPLY ? nullptr : y;
    p.yout = y;
    p.dot_flags = 3;
    p.dot_mode = 0;
    p.partials = reinterpret_cast<double*>(static_cast<char*>(work) + kWorkHeader);
    p.acc = static_cast<double2*>(acc);
    p.acc_out = static_cast<double2*>(acc);
    p.acc_mode = ACC_ADD | ACC_X | (op == PVSC_OP_APPLY ? 0 : ACC_YIN);
    p.cx_re = 0.3;  // real weights, the kinds of a filter's three-term touch
    p.cy_re = -0.2;
    p.cz_re = -0.1;
    auto one = [&]() -> int {
      if (op == PVSC_OP_KPM) return launch_sweep(lat, prec, F_KPM, p, st);
      if (op == PVSC_OP_APPLY) return launch_sweep(lat, prec, 0, p, st);
      if (int r = launch_sweep(lat, prec, F_ACC, p, st)) return r;
      if (int r = launch_sweep(lat, prec, F_REC, p, st)) return r;
      return launch_sweep(lat, prec, F_REC, p, st);
    };
    if (int r = one()) return r;
    // the best of three trials of three repetitions each: shapes a few per cent
    // apart are told apart despite clock and co-tenant noise
    float best = 1e30f;
    for (int trial = 0; trial < 3; ++trial) {
      PVSC_CUDA_TRY(cudaEventRecord(e0, st));
      for (int rep = 0; rep < 3; ++rep)
        if (int r = one()) return r;
      PVSC_CUDA_TRY(cudaEventRecord(e1, st));
      PVSC_CUDA_TRY(cudaEventSynchronize(e1));
      float t = 0.f;
      PVSC_CUDA_TRY(cudaEventElapsedTime(&t, e0, e1));
      if (t < best) best = t;
    }
    *ms = best / 3.f;
    return PVSC_OK;
  };
  const std::vector<pvsc_tuning> cands = candidates(lat, R, prec, op);
  for (const pvsc_tuning& cand : cands) {
    float ms = 0.f;
    if ((rc = time_one(cand, &ms)) != PVSC_OK) break;
    if (ms < win.time_ms) {
      win = cand;
      win.time_ms = ms;
    }
  }
  cleanup();
  if (rc != PVSC_OK) {
    if (had) lat->tuning[{R, prec}] = old; else lat->tuning.erase({R, prec});
    return rc;
  }
  install(lat, R, prec, win);
  drop_graphs(lat);
  cache_store(key, win);
  if (best) *best = reported(win, R, prec);
  return PVSC_OK;
}

extern "C" int pvsc_autotune(pvsc_lattice* lat, int R, int prec, pvsc_tuning* best, void* stream) {
  return pvsc_autotune_op(lat, R, prec, PVSC_OP_KPM, best, stream);
}

extern "C" int pvsc_debug_autotune_candidates(const pvsc_lattice* lat, int R, int prec, int op, pvsc_tuning* out,
                                              int max, int* n) {
  if (int rc = check_lattice(lat)) return rc;
  if (!valid_R(R) || (prec != PVSC_C128 && prec != PVSC_C64) || !n || (max > 0 && !out))
    return set_error(PVSC_ERR_ARG, "bad R, precision or output");
  const std::vector<pvsc_tuning> c = candidates(lat, R, prec, op);
  for (int i = 0; i < max && i < (int)c.size(); ++i) out[i] = c[i];
  *n = (int)c.size();
  return PVSC_OK;
}
