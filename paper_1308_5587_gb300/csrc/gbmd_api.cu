// gbmd_api.cu -- the C ABI of libgbmd (include/gbmd.h): systems, batches, CUDA
// graphs with a device-decided rebuild, overflow recovery, readouts, autotuning.
//
// A "group" is the unit that is stepped: one system alone, or a batch of systems.
// Its step is a CUDA graph per block of steps; per step:
//   step kernel (pair force K5 + integration K6) -> IF(any system needs a rebuild)
//   { bin -> scan -> scatter -> cellsort -> permute -> copyback -> [blocks] -> nlist }.
// The IF is a graph conditional node whose value the step kernel's last block sets
// on the device, so a step never returns to the host.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "launch.cuh"

using namespace gbmd;

namespace {

thread_local std::string g_err;

int fail(int code, const char* fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
  return code;
}

#define CK(call)                                                                         \
  do {                                                                                   \
    cudaError_t e_ = (call);                                                             \
    if (e_ != cudaSuccess) {                                                             \
      return fail(e_ == cudaErrorMemoryAllocation ? GBMD_ERR_OOM : GBMD_ERR_CUDA,          \
                  "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    }                                                                                    \
  } while (0)

#define RET(x)                 \
  do {                         \
    int r_ = (x);              \
    if (r_ != GBMD_OK) return r_; \
  } while (0)

constexpr int STEPS_PER_GRAPH = 16;
constexpr int STAGED_WINDOW_CAP = 3072;   // window particles in 48 KB of shared memory

size_t round_up(size_t v, size_t m) { return (v + m - 1) / m * m; }

// NVTX range over a host call (the timeline of a profiler shows the library's
// calls: enqueues, rebuild recoveries, readouts); a no-op unless a tool is attached
struct Range {
  explicit Range(const char* name) { nvtxRangePushA(name); }
  ~Range() { nvtxRangePop(); }
};

}  // namespace

struct Group;

struct gbmd_system {
  int device = 0;             // CUDA ordinal every call on this system uses
  SysDev h{};                 // master descriptor (device pointers)
  Flags* d_flags = nullptr;
  cudaStream_t stream = nullptr;     // the caller's stream
  std::map<void*, size_t> allocs;   // device memory and its bytes
  size_t footprint = 0;
  Group* own = nullptr;       // the system alone
  Group* batch = nullptr;
  int batch_slot = -1;
  long long target_step = 0;  // steps requested so far (absolute), host bookkeeping
  long long step_limit = -1;
  double cell_min = 0;        // smallest allowed cell width: r_list,max (cell list) or
                              // r_list,min (tree list, whose cells only order particles)
  double cell_scale = 1.0;    // cell width >= cell_scale * cell_min (autotuned)
  bool want_staged = false;   // GBMD_PATH_STAGED requested
  // staging for import/export (device)
  double *d_pos = nullptr, *d_vel = nullptr, *d_frc = nullptr;
  int *d_img = nullptr, *d_type = nullptr, *d_misc = nullptr;
  double *d_ppu = nullptr, *d_ppw = nullptr;   // per-particle readout staging (lazy)
  std::vector<char> bounce;   // host side of a small readout
};

constexpr int TEAM_SIDES = 4;   // cluster sizes 16, 8, 4, 2, 1: the first on the group's stream

// what a resident kernel may use of the device: SMs, its blocks on one, and how many of its
// clusters of 2^k blocks run at once (fewer than the SMs would hold: a cluster stays in one
// part of the chip, 18 or 20 SMs; of 1, 2, .. 16 blocks, one an SM: 152, 76, 36, 15, 7)
struct TeamFit { int sms = 0, blocks_per_sm = 0, max_cluster = 0, clusters[TEAM_SIDES + 1] = {}; };

struct StepGraphs {
  cudaGraphExec_t many = nullptr, one = nullptr;
  cudaGraph_t graph_one = nullptr;                 // kept alive for node updates
  cudaGraphNode_t ev_begin = nullptr, ev_end = nullptr;
  bool built = false;
};

// how a group's team members are stepped: the kernel, its lanes a particle, and its launches,
// members [first, last) of the team each by clusters of that many blocks (0: by the whole
// grid, as shares of it or a system alone)
struct TeamClass { int first, last, cluster; };
struct TeamPlan {
  void* func = nullptr;
  int lanes = 1;
  TeamFit fit;
  bool shares = false;
  std::vector<TeamClass> cls;
};

struct Group {
  int device = 0;
  std::vector<gbmd_system*> members;   // may contain nullptr (free slots of a batch)
  bool is_batch = false;
  int precision = GBMD_MIXED;
  int multi = 0;   // pair-table mode: 0 one type, 1 at most two, 2 more
  bool rel = true;     // every member has at least 3 cells on every axis
  cudaStream_t stream = nullptr;
  int tpp = 2, fblock = 128;
  // device tables
  SysDev* d_desc = nullptr;
  Tile *d_tp = nullptr, *d_tf = nullptr, *d_tc = nullptr, *d_ts = nullptr;
  Tile *d_tb = nullptr, *d_tbk = nullptr;   // staged force blocks; their window kernel
  Tile* d_te = nullptr;   // energy/virial launches: ev_tile(n) particles per tile, whatever
                          // the force block, so the FP64 sums depend on the lanes alone
  int ev_tile = EV_TILE_P;   // the largest of them
  Tile *d_tt = nullptr, *d_tg = nullptr;   // tree-list systems: tiles over their trees'
                                           // leaves, and over the groups that query them
  Tile* d_tn = nullptr;   // list build by four warps per cell (few cells): (cell, part) items
  int ntp = 0, ntf = 0, ntc = 0, nts = 0, ntb = 0, ntbk = 0, nte = 0, ntt = 0, ntg = 0, ntn = 0;
  size_t cap_desc = 0, cap_tp = 0, cap_tf = 0, cap_tc = 0, cap_ts = 0, cap_part = 0;
  size_t cap_tb = 0, cap_tbk = 0, cap_te = 0, cap_tt = 0, cap_tg = 0, cap_tn = 0;
  bool any_cell = true;   // some member builds its list from cells
  int window_cap = 0;                        // largest staged window among members
  bool nvt = false;                          // the members integrate NVT (all or none)
  int eval = EVAL_LJ;                        // the members' pair evaluator (all the same)
  double* d_nhpart = nullptr;                // NVT: v.v partial sums per chunk of a system
  size_t cap_nhpart = 0;
  double* d_partials = nullptr;
  GroupCtl* d_ctl = nullptr;
  // the step graphs; [1]: beside work on other streams (no launch that needs the whole chip)
  StepGraphs graphs[2];
  // optional event records around the force kernel of the single-step graphs
  cudaEvent_t ev_begin = nullptr, ev_end = nullptr;
  bool layout_dirty = true;
  bool use_graphs = true;
  // the members that the team kernel steps (positions among the live members, the
  // largest first) and how; the others, if any, are stepped by the graph of `rest`
  std::vector<int> team;
  std::vector<int> team_n;             // their particles
  TeamPlan plan;
  int* d_team = nullptr;
  size_t cap_team = 0;
  // a batch's teams as shares of one grid: per block (member, rank, blocks, team)
  std::vector<int4> share;
  int4* d_share = nullptr;
  TeamSync* d_sync = nullptr;
  size_t cap_share = 0, cap_sync = 0;
  cudaStream_t side[TEAM_SIDES] = {};
  cudaEvent_t side_ev[TEAM_SIDES + 1] = {};
  Group* rest = nullptr;
  bool is_rest = false;
};

namespace {

// make `dev` current for this thread in this library's CUDA runtime
int use_device(int dev) {
  int cur = -1;
  if (cudaGetDevice(&cur) == cudaSuccess && cur == dev) return GBMD_OK;
  CK(cudaSetDevice(dev));
  return GBMD_OK;
}

std::vector<gbmd_system*> live(const Group* g) {
  std::vector<gbmd_system*> v;
  for (auto* s : g->members)
    if (s) v.push_back(s);
  return v;
}

template <typename T>
int grow(T** p, size_t* cap, size_t need) {
  if (*cap >= need && *p) return GBMD_OK;
  if (*p) CK(cudaFree(*p));
  *p = nullptr;
  size_t n = std::max<size_t>(need, 1);
  CK(cudaMalloc((void**)p, n * sizeof(T)));
  *cap = n;
  return GBMD_OK;
}

void destroy_graphs(Group* g);

// the group's device tables and graphs
void free_group(Group* g) {
  if (g->rest) free_group(g->rest);
  destroy_graphs(g);
  for (cudaStream_t st : g->side)
    if (st) cudaStreamDestroy(st);
  for (cudaEvent_t e : g->side_ev)
    if (e) cudaEventDestroy(e);
  for (void* p : {(void*)g->d_desc, (void*)g->d_tp, (void*)g->d_tf, (void*)g->d_tc, (void*)g->d_te,
                  (void*)g->d_nhpart, (void*)g->d_ts, (void*)g->d_tb, (void*)g->d_tbk, (void*)g->d_tt,
                  (void*)g->d_tg, (void*)g->d_tn, (void*)g->d_team, (void*)g->d_share, (void*)g->d_sync, (void*)g->d_partials, (void*)g->d_ctl})
    cudaFree(p);
  delete g;
}

void destroy_graphs(Group* g) {
  for (StepGraphs& q : g->graphs) {
    if (q.many) cudaGraphExecDestroy(q.many);
    if (q.one) cudaGraphExecDestroy(q.one);
    if (q.graph_one) cudaGraphDestroy(q.graph_one);
    q = StepGraphs();
  }
}

// The streams with steps enqueued that the host has not waited for since.  A cooperative launch
// of the whole grid waits until every SM is free for it, and what other streams launch waits
// for it in turn, so systems on streams of their own would go one after another: while some
// other stream of the device has work, neither the team's grid nor the cooperative
// rebuild is used.  us for a step of all, side by side, with them / so: 4 of 4,000 44.6 /
// 28.3, 8 of 20,000 119 / 74, 8 of 150,000 515 / 367, FP64 8 of 20,000 340 / 197.  (Clusters
// take part of the chip and stay: 8 of 1,000 13 us, 52 by the graph.)  Kept on the host, so
// that nothing is asked of the device while some thread captures; a stream that was waited
// for by other means counts until the library's next wait for it.
std::mutex pending_mu;
std::vector<std::pair<int, cudaStream_t>> pending;

// nothing is pending on the device's other streams
bool alone(int dev, cudaStream_t st) {
  std::lock_guard<std::mutex> lock(pending_mu);
  for (const auto& p : pending)
    if (p.first == dev && p.second != st) return false;
  return true;
}
void enqueued(int dev, cudaStream_t st) {
  std::lock_guard<std::mutex> lock(pending_mu);
  const std::pair<int, cudaStream_t> me(dev, st);
  if (std::find(pending.begin(), pending.end(), me) == pending.end()) pending.push_back(me);
}
cudaError_t wait_for(int dev, cudaStream_t st) {
  const cudaError_t e = cudaStreamSynchronize(st);
  std::lock_guard<std::mutex> lock(pending_mu);
  pending.erase(std::remove(pending.begin(), pending.end(), std::make_pair(dev, st)), pending.end());
  return e;
}

// Which list builder serves the rebuild's own launch (the rows are the same): four warps
// per cell (k_nlist_split) while a launch has few cells, else one warp per cell (k_nlist).
// One build, ncu: 8 cells (N = 500) 25 against 107 us; 2,744 cells (N = 64,000) 81 against
// 51 us; the lines cross near the cells of a 20,000-particle system (729: 40.4 against
// 43.6 us a step with a build every eighth).
constexpr int SPLIT_MAX_CELLS = 1024;
bool use_split(const std::vector<gbmd_system*>& m) {
  long long cells = 0;
  for (auto* s : m) {
    if (s->h.staged) return false;   // staged rows hold window indices: k_nlist's
    if (!s->h.tree) cells += s->h.ncells;
  }
  return cells > 0 && cells <= SPLIT_MAX_CELLS;
}
// blocks per cell: one for every 32 particles of the mean occupation
int split_parts(const SysDev& d) { return std::max(1, (d.n / d.ncells + 31) / 32); }

// the query groups of type ty of a tree-list system
int tree_groups(const SysDev& d, int ty) {
  return d.tree_single[ty] ? d.tree_n[ty] : (d.tree_n[ty] + TREE_G - 1) / TREE_G;
}

// Systems that the team kernel may step: the cell list on the global force path,
// without ghosts (their rebuilds are the caller's).  Alone it pays while a step is short
// beside the launches it saves: up to one turn of its warps, in mixed precision with two
// lanes a particle done by one (k_team.cuh), and with more lanes up to TEAM_ALONE_N.  With
// readouts, us: N = 64,000 mixed, 50 steps, 1,789 by the step kernel and k_rebuild, 1,663
// by the team; FP64, 20 steps, 2,291 and 2,211; FP64 NVT, 20 steps, 2,690 and 2,397.
// (N = 200,000, several turns: 73 us a step by the team, 66 by the step kernel.)
// In a batch, where a shared launch makes every member wait for any member's rebuild, up
// to TEAM_MEMBER_N (measured to 30,000), as far as that pays (plan_team).
constexpr int TEAM_ALONE_N = 49152;
constexpr int TEAM_MEMBER_N = 32768;
constexpr int TEAM_STEPS = 64;   // steps of one launch
bool team_member(const Group* g, const SysDev& d, int sms) {
  if (d.tree || d.staged || d.n_ghost > 0) return false;
  if (g->is_batch) return d.n <= TEAM_MEMBER_N;
  const int lanes = g->precision == GBMD_MIXED && g->tpp == 2 ? 1 : g->tpp;
  return d.n <= std::max(TEAM_ALONE_N, sms * TEAM_T / lanes);
}

// The force tiles of a system, `per` particles each.  The particles of a wide type of a
// tree-list system (its order is type-major) come first, in wide tiles: one to each 32
// threads of a block of per * tpp.
void force_tiles(const SysDev& d, int sys, int prec, int tpp, int per, std::vector<Tile>* out) {
  auto add = [&](int first, int count, int p, int wide) {
    for (int f = 0; f < count; f += p) out->push_back({sys, first + f, std::min(p, count - f), wide});
  };
  const bool wide = d.tree && !d.nvt && has_wide(prec, tpp);
  if (!wide) return add(0, d.n, per, 0);
  for (int t = 0; t < d.ntypes; ++t)
    if (d.tree_wide[t]) add(d.tree_first[t], d.tree_n[t], std::max(1, per * tpp / 32), 1);
  for (int t = 0; t < d.ntypes;) {   // the others, across type boundaries
    if (d.tree_wide[t]) { ++t; continue; }
    const int first = d.tree_first[t];
    int count = 0;
    for (; t < d.ntypes && !d.tree_wide[t]; ++t) count += d.tree_n[t];
    add(first, count, per, 0);
  }
}

// TeamFit of a resident kernel, asked once per kernel and device
int team_fit(void* f, int threads, size_t smem, int dev, TeamFit* out) {
  static std::mutex mu;
  static std::map<std::pair<int, void*>, TeamFit> known;
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find({dev, f});
  if (it != known.end()) {
    *out = it->second;
    return GBMD_OK;
  }
  TeamFit t;
  CK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  CK(cudaDeviceGetAttribute(&t.sms, cudaDevAttrMultiProcessorCount, dev));
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t.blocks_per_sm, f, threads, smem));
  CK(cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  for (int k = 0; k <= TEAM_SIDES; ++k) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(1u << k);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim = {1u << k, 1, 1};
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&t.clusters[k], f, &cfg) != cudaSuccess) {
      cudaGetLastError();
      t.clusters[k] = 0;
    }
    if (t.clusters[k] > 0) t.max_cluster = 1 << k;
  }
  known[{dev, f}] = t;
  *out = t;
  return GBMD_OK;
}

// A system alone takes one cluster up to TEAM_CLUSTER_CHUNKS warps' work a step (FP64,
// bound by the SMs' FP64 pipes: one block's warps), and every SM beyond that (N = 2,000,
// mixed: 8.1 us a step either way; N = 4,000: 12 on a cluster of 16, 9 on the grid).
constexpr int TEAM_CLUSTER_CHUNKS = 128;
int team_cluster(int chunks, int per_block, int most) {
  int c = 1;
  while (c < most && (long long)c * per_block < chunks) c *= 2;
  return c;
}
// shares of `sms` blocks for the team's members: one each, then the next always to the
// member with the most work a block
std::vector<int4> team_shares(const std::vector<int>& work, int sms) {
  const int teams = (int)work.size();
  std::vector<int> blocks(teams, 1);
  auto less = [&](int a, int b) {   // work a block; the earlier of equals first
    const long long x = (long long)work[a] * blocks[b], y = (long long)work[b] * blocks[a];
    return x != y ? x < y : a > b;
  };
  std::vector<int> heap(teams);
  for (int t = 0; t < teams; ++t) heap[t] = t;
  std::make_heap(heap.begin(), heap.end(), less);
  for (int k = teams; k < sms; ++k) {
    std::pop_heap(heap.begin(), heap.end(), less);
    ++blocks[heap.back()];
    std::push_heap(heap.begin(), heap.end(), less);
  }
  std::vector<int4> out;
  for (int t = 0; t < teams; ++t)
    for (int r = 0; r < blocks[t]; ++r) out.push_back(make_int4(t, r, blocks[t], t));
  return out;
}

// How the group's team members (g->team, g->team_n) are stepped; without a plan that pays
// the list is emptied.
//
// A batch's members divide one grid: each gets a share of the SMs by its particles, and no SM
// waits for a cluster to fit or stands beside a power of two.  Its barriers go through
// memory (2 us a step) where a cluster's take 0.5: clusters of 16, 8, .. 1 blocks by a
// member's own size, one launch a size, side by side on streams of their own, the largest
// first, serve batches whose clusters all run at once with up to half a turn of its warps on
// a block, mixed also up to two turns where no member has more than CLUSTER_SMALL_N particles,
// FP64 (bound by the SMs' FP64 pipes) up to a quarter.  us a step by clusters / shares, mixed:
// 4 of 500 9.7 / 11.4, 32 of 500 11.1 / 12.3, 64 of 500 21.2 / 22.1; 8 of 2,000 16.5 / 12.5, 4
// of 4,000 16.9 / 12.8, 2 of 8,000 27.8 / 13.2, 2 of 20,000 59 / 23; FP64: 4 of 500 29.4 /
// 30.9, 16 of 500 35.5 / 31.0, 4 of 4,000 55 / 36, 2 of 20,000 213 / 80.  More members than
// SMs take clusters as they become free.
//
// Against the shared graph, whose kernels spread every member over the chip: the fullest block
// of the team has more than the mean to do, and the step waits for it (TEAM_US a particle);
// in the graph every step waits for any member's rebuild, and for the graph itself where no
// other members need it (GRAPH_US, GRAPH_US_MEMBER).  us a step by the graph / the team,
// mixed: 96 of 4,000 174 / 154, 100 of 8,000 266 / 332, 32 of 20,000 230 / 219, 48 of 20,000
// 308 / 302, 40 of 30,000 363 / 427, 150 of 1,000 139 / 46, 96 of 500 to 20,000 287 / 243,
// 200 of 500 193 / 44, 200 of 500 to 20,000 445 / 475; FP64: 96 of 4,000 524 / 650, 16 of
// 20,000 434 / 384, 32 of 20,000 797 / 831, 48 of 500 to 20,000 489 / 419; with others: eight
// of 4,000 and two of 64,000 88 / 70, four of 20,000 and four of 40,000 99 / 108.
constexpr int CLUSTER_SMALL_N = 1024;
constexpr double TEAM_US_MIXED = 0.041, TEAM_US_FP64 = 0.16;
constexpr double GRAPH_US = 22.0, GRAPH_US_MEMBER = 1.5, TEAM_BASE_US = 10.0;
constexpr int GRAPH_MEMBERS = 64;   // from here on some member rebuilds at every step
constexpr double TEAM_WAVES = 1.35; // clusters one after another: the last ones' SMs stand idle
// A member's share where the chip has less than a turn of its warps to do, mixed: by its
// chunks and this many more, since a small member's rebuild is a chain that more blocks
// shorten (12 of 500 to 3,000: 31 us a step without, 16 with).  FP64 forces, bound by their pipe,
// want blocks by the pairs alone (24 of 500 to 3,000: 62 without, 78 with).
constexpr int SHARE_EXTRA = 64;
int plan_team(Group* g, bool others) {
  TeamPlan& p = g->plan;
  p = TeamPlan();
  g->share.clear();
  if (g->team.empty()) return GBMD_OK;
  constexpr int warps = TEAM_T / 32;
  const int teams = (int)g->team_n.size();
  p.lanes = g->tpp;
  p.func = k_team_variant(g->eval, g->precision, g->tpp, g->multi, false);
  RET(team_fit(p.func, TEAM_T, TEAM_SMEM, g->device, &p.fit));
  // two lanes a particle as one where that leaves every warp of the chip a chunk: a
  // system with more than one turn of them at two lanes, a batch with more than two
  if (g->precision == GBMD_MIXED && g->tpp == 2) {
    long long total = 0;
    for (int nn : g->team_n) total += ((long long)nn * 2 + 31) / 32;
    if (total > (long long)(g->is_batch ? 2 : 1) * p.fit.sms * warps) {
      p.lanes = 1;
      p.func = k_team_variant(g->eval, g->precision, g->tpp, g->multi, true);
      RET(team_fit(p.func, TEAM_T, TEAM_SMEM, g->device, &p.fit));
    }
  }
  const TeamFit& fit = p.fit;
  auto drop = [&]() -> int {
    g->team.clear();
    g->team_n.clear();
    g->share.clear();
    p = TeamPlan();
    return GBMD_OK;
  };
  if (fit.max_cluster < 1 || fit.blocks_per_sm < 1) return drop();
  auto chunks_of = [&](int nn) { return (int)(((long long)nn * p.lanes + 31) / 32); };
  if (!g->is_batch && chunks_of(g->team_n[0]) > (g->precision == GBMD_FP64 ? warps : TEAM_CLUSTER_CHUNKS)) {
    p.cls.push_back({0, 1, 0});
    return GBMD_OK;
  }
  int per_block = 2;
  auto cluster_of = [&](int nn) { return team_cluster(chunks_of(nn), per_block, fit.max_cluster); };
  auto at_once = [&]() {
    double chip = 0;
    for (int nn : g->team_n) chip += 1.0 / fit.clusters[31 - __builtin_clz((unsigned)cluster_of(nn))];
    return chip <= 1.0 + 1e-9;
  };
  while (per_block < 4 * warps && !at_once()) per_block *= 2;
  const bool fits = at_once();
  double fullest = 0, sum = 0;   // particles of a block
  for (int nn : g->team_n) {
    fullest = std::max(fullest, (double)nn / cluster_of(nn));
    sum += nn;
  }
  const bool fp64 = g->precision == GBMD_FP64;
  const double turns = fp64 ? 0.25 : g->team_n[0] <= CLUSTER_SMALL_N ? 2.0 : 0.5;
  p.shares = g->is_batch && teams <= fit.sms && !(fits && fullest * p.lanes <= turns * TEAM_T);
  if (p.shares) {
    const int extra = !fp64 && sum * p.lanes < (double)fit.sms * TEAM_T ? SHARE_EXTRA : 0;
    std::vector<int> work;
    for (int nn : g->team_n) work.push_back(chunks_of(nn) + extra);
    g->share = team_shares(work, fit.sms);
    fullest = 0;
    for (const int4& q : g->share) fullest = std::max(fullest, (double)g->team_n[q.x] / q.z);
    p.cls.push_back({0, teams, 0});
  } else {
    if (!fits) fullest = std::max(fullest, TEAM_WAVES * sum / fit.sms);
    for (int k = 0; k < teams; ++k) {
      const int c = cluster_of(g->team_n[k]);
      if (p.cls.empty() || p.cls.back().cluster != c) p.cls.push_back({k, k, c});
      p.cls.back().last = k + 1;
    }
  }
  if (!g->is_batch) return GBMD_OK;
  const double more = (fullest - sum / fit.sms) * (fp64 ? TEAM_US_FP64 : TEAM_US_MIXED);
  const double less = (others ? 0.0 : GRAPH_US) + GRAPH_US_MEMBER * std::min(teams, GRAPH_MEMBERS) - TEAM_BASE_US;
  return more <= less ? GBMD_OK : drop();
}

// Which members the team kernel steps, and the group of the others
int split_members(Group* g, const std::vector<gbmd_system*>& m) {
  g->team.clear();
  g->team_n.clear();
  std::vector<gbmd_system*> others;
  int sms = 0;
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device));
  if (g->use_graphs && !g->is_rest)
    for (size_t k = 0; k < m.size(); ++k) {
      if (team_member(g, m[k]->h, sms)) g->team.push_back((int)k);
      else others.push_back(m[k]);
    }
  std::stable_sort(g->team.begin(), g->team.end(), [&](int a, int b) { return m[a]->h.n > m[b]->h.n; });
  for (int k : g->team) g->team_n.push_back(m[k]->h.n);
  RET(plan_team(g, !others.empty()));
  if (!g->team.empty() && !others.empty()) {
    if (!g->rest) {
      g->rest = new Group();
      g->rest->is_rest = true;
      g->rest->is_batch = true;
    }
    Group* r = g->rest;
    r->device = g->device;
    r->precision = g->precision;
    r->stream = g->stream;
    r->tpp = g->tpp;
    r->fblock = g->fblock;
    r->members = others;
    r->layout_dirty = true;
  } else if (g->rest) {
    g->rest->members.clear();
    g->rest->layout_dirty = true;
  }
  return GBMD_OK;
}

// Rebuild descriptor copies and tile tables for the group's current members.
int sync_layout(Group* g) {
  if (!g->layout_dirty) return GBMD_OK;
  std::vector<gbmd_system*> m = live(g);
  std::vector<SysDev> desc;
  std::vector<Tile> tp, tf, tc, ts, tb, tbk, te, tt, tg, tn;
  const int per_f = g->fblock / g->tpp;
  g->multi = 0;
  g->rel = true;
  g->window_cap = 0;
  g->nvt = !m.empty() && m[0]->h.nvt;
  g->eval = m.empty() ? EVAL_LJ : m[0]->h.eval;
  g->any_cell = false;
  const bool split = use_split(m);
  int nh_chunks = 0;
  for (size_t k = 0; k < m.size(); ++k) {
    SysDev d = m[k]->h;
    const int n = d.n;
    g->ev_tile = std::max(k ? g->ev_tile : 0, ev_tile(n));
    for (int f = 0; f < n; f += TILE_P) tp.push_back({(int)k, f, std::min(TILE_P, n - f), 0});
    if (d.staged) {   // one force tile per 2x2x2 block of cells
      d.tile_first_f = (int)tb.size();   // shifted past the global tiles below
      for (int b = 0; b < d.nblocks; ++b) tb.push_back({(int)k, b, 1, 0});
      d.tile_count_f = d.nblocks;
      for (int b = 0; b < d.nblocks; b += 8) tbk.push_back({(int)k, b, std::min(8, d.nblocks - b), 0});
      g->window_cap = std::max(g->window_cap, d.window_cap);
    } else {
      d.nh_blocks = -(int)tf.size();
      force_tiles(d, (int)k, g->precision, g->tpp, per_f, &tf);
      d.nh_blocks += (int)tf.size();
      d.nh_first = nh_chunks;
      d.nh_count = (int)(((long long)n * g->tpp + 31) / 32);
      nh_chunks += d.nh_count;
      d.tile_first_f = (int)te.size();   // partial sums come from the energy launches
      force_tiles(d, (int)k, g->precision, g->tpp, ev_tile(n), &te);
      d.tile_count_f = (int)te.size() - d.tile_first_f;
    }
    for (int c = 0; c < d.nbins; c += CELLS_PER_TILE)
      tc.push_back({(int)k, c, std::min(CELLS_PER_TILE, d.nbins - c), 0});
    if (split && !d.tree) {
      const int parts = split_parts(d);
      for (int c = 0; c < d.nbins * parts; ++c) tn.push_back({(int)k, c / parts, c % parts, parts});
    }
    ts.push_back({(int)k, 0, 0, 0});
    if (d.tree)
      for (int f = 0; f < d.tree_leaves_total; f += TILE_P)
        tt.push_back({(int)k, f, std::min(TILE_P, d.tree_leaves_total - f), 0});
    for (int q = 0; d.tree && q < d.ntypes; ++q) {
      const int ty = d.tree_qtype[q], groups = tree_groups(d, ty);
      for (int f = 0; f < groups; f += TREE_WARPS)
        tg.push_back({(int)k, f, std::min(TREE_WARPS, groups - f), ty | (d.tree_single[ty] ? 256 : 0)});
    }
    desc.push_back(d);
    if (d.ntypes > 1) g->multi = std::max(g->multi, d.ntypes > 2 ? 2 : 1);
    if (!d.tree) {
      g->any_cell = true;
      if (d.nc[0] < 3 || d.nc[1] < 3 || d.nc[2] < 3) g->rel = false;
    }
  }
  RET(split_members(g, m));
  for (auto& d : desc)
    if (d.staged) d.tile_first_f += (int)te.size();   // staged partial sums follow the global ones
  RET(grow(&g->d_partials, &g->cap_part, 8 * std::max<size_t>(te.size() + tb.size(), 1)));
  RET(grow(&g->d_nhpart, &g->cap_nhpart, std::max<size_t>(nh_chunks, 1)));
  for (auto& d : desc) {
    d.partials = g->d_partials;
    d.nh_part = g->d_nhpart;
  }
  RET(grow(&g->d_desc, &g->cap_desc, desc.size()));
  RET(grow(&g->d_tp, &g->cap_tp, tp.size()));
  RET(grow(&g->d_tf, &g->cap_tf, tf.size()));
  RET(grow(&g->d_tc, &g->cap_tc, tc.size()));
  RET(grow(&g->d_ts, &g->cap_ts, ts.size()));
  RET(grow(&g->d_tb, &g->cap_tb, tb.size()));
  RET(grow(&g->d_tbk, &g->cap_tbk, tbk.size()));
  RET(grow(&g->d_te, &g->cap_te, te.size()));
  RET(grow(&g->d_tt, &g->cap_tt, tt.size()));
  RET(grow(&g->d_tg, &g->cap_tg, tg.size()));
  RET(grow(&g->d_tn, &g->cap_tn, tn.size()));
  RET(grow(&g->d_team, &g->cap_team, g->team.size()));
  RET(grow(&g->d_share, &g->cap_share, g->share.size()));
  if (!g->share.empty()) RET(grow(&g->d_sync, &g->cap_sync, (size_t)g->plan.fit.sms));   // a team a block at most
  if (!g->d_ctl) {
    CK(cudaMalloc(&g->d_ctl, sizeof(GroupCtl)));
    CK(cudaMemsetAsync(g->d_ctl, 0, sizeof(GroupCtl), g->stream));
  }
  // a wait that was given up leaves arrivals behind.  Its system stays stopped, so nothing
  // meets them before the group's members change, which comes through here.  (GBMD_TEAM_POLLS=0:
  // a test lets every wait run out at once)
  const char* polls = getenv("GBMD_TEAM_POLLS");
  const TeamSync clean{polls && polls[0] == '0' ? TEAM_CLOSED : 0ull, 0ull};
  const std::vector<TeamSync> sync(std::max<size_t>(g->d_sync ? g->cap_sync : 0, 1), clean);
  CK(cudaMemcpyAsync(&g->d_ctl->team, sync.data(), sizeof(TeamSync), cudaMemcpyHostToDevice, g->stream));
  if (g->d_sync)
    CK(cudaMemcpyAsync(g->d_sync, sync.data(), g->cap_sync * sizeof(TeamSync), cudaMemcpyHostToDevice, g->stream));
  auto up = [&](void* dst, const std::vector<Tile>& v) -> cudaError_t {
    if (v.empty()) return cudaSuccess;
    return cudaMemcpyAsync(dst, v.data(), v.size() * sizeof(Tile), cudaMemcpyHostToDevice, g->stream);
  };
  if (!desc.empty()) CK(cudaMemcpyAsync(g->d_desc, desc.data(), desc.size() * sizeof(SysDev), cudaMemcpyHostToDevice, g->stream));
  CK(up(g->d_tp, tp));
  CK(up(g->d_tf, tf));
  CK(up(g->d_tc, tc));
  CK(up(g->d_ts, ts));
  CK(up(g->d_tb, tb));
  CK(up(g->d_tbk, tbk));
  CK(up(g->d_te, te));
  CK(up(g->d_tt, tt));
  CK(up(g->d_tg, tg));
  CK(up(g->d_tn, tn));
  if (!g->share.empty())
    CK(cudaMemcpyAsync(g->d_share, g->share.data(), g->share.size() * sizeof(int4), cudaMemcpyHostToDevice, g->stream));
  if (!g->team.empty())
    CK(cudaMemcpyAsync(g->d_team, g->team.data(), g->team.size() * sizeof(int), cudaMemcpyHostToDevice, g->stream));
  CK(cudaStreamSynchronize(g->stream));   // host vectors die here
  g->ntp = (int)tp.size();
  g->ntf = (int)tf.size();
  g->ntc = (int)tc.size();
  g->nts = (int)ts.size();
  g->ntb = (int)tb.size();
  g->ntbk = (int)tbk.size();
  g->nte = (int)te.size();
  g->ntt = (int)tt.size();
  g->ntg = (int)tg.size();
  g->ntn = (int)tn.size();
  g->layout_dirty = false;
  destroy_graphs(g);
  return GBMD_OK;
}

// update one member's descriptor in every group it belongs to (pointer/size change)
int refresh_desc(gbmd_system* s) {
  for (Group* g : {s->own, s->batch}) {
    if (!g) continue;
    g->layout_dirty = true;
    RET(sync_layout(g));
  }
  return GBMD_OK;
}

// the rebuild: cell sort (and re-sort), then the lists -- cell-list members by
// k_nlist (after the staged windows, if any), tree-list members by k_tree_*
std::vector<KernelCall> rebuild_calls(const Group* g) {
  std::vector<KernelCall> v = {bin_call(g->d_desc, g->d_tp, g->ntp, g->d_ctl),
                               scan_call(g->d_desc, g->d_ts, g->nts, g->d_ctl),
                               scatter_call(g->d_desc, g->d_tp, g->ntp, g->d_ctl),
                               cellsort_call(g->d_desc, g->d_tc, g->ntc, g->d_ctl),
                               permute_call(g->d_desc, g->d_tp, g->ntp, g->d_ctl),
                               copyback_call(g->d_desc, g->d_tp, g->ntp, g->d_ctl)};
  if (g->ntbk > 0) v.push_back(blocks_call(g->d_desc, g->d_tbk, g->ntbk, g->d_ctl));
  if (g->ntn > 0)
    v.push_back(nlist_split_call(g->d_desc, g->d_tn, g->ntn, g->d_ctl, g->multi > 0));
  else if (g->any_cell)
    v.push_back(nlist_call(g->d_desc, g->d_tc, g->ntc, g->d_ctl, g->rel, g->multi, g->ntbk > 0));
  if (g->ntt > 0) {
    v.push_back(tree_build_call(g->d_desc, g->d_tt, g->ntt, g->d_ctl));
    v.push_back(tree_nlist_call(g->d_desc, g->d_tg, g->ntg, g->d_ctl));
  }
  return v;
}

// forces at the current positions, outside the step (autotuning, readouts)
KernelCall plain_force_call(const Group* g, int readout = 0) {
  StepArgs sa;
  sa.readout = readout;
  return force_call(g->precision, g->multi, readout ? MODE_READ : MODE_FORCE, g->tpp, g->fblock, g->d_desc, g->d_tf,
                    g->ntf, g->d_ctl, sa, g->eval);
}

// energy/virial launch of the global-list systems: the step's threads per particle
// (so the FP32 forces it writes are bitwise the step's), ev_tile particles per block
KernelCall ev_force_call(const Group* g, const SysDev* desc) {
  return force_call(g->precision, g->multi, MODE_EV, g->tpp, g->ev_tile * g->tpp, desc, g->d_te,
                    g->nte, g->d_ctl, StepArgs{}, g->eval);
}

// readout force launches (ev = 0 forces, 1 also energy/virial): global-list systems,
// then staged ones
std::vector<KernelCall> force_calls(const Group* g, int ev, int readout = 0) {
  std::vector<KernelCall> v;
  if (g->ntf > 0) v.push_back(ev ? ev_force_call(g, g->d_desc) : plain_force_call(g, readout));
  if (g->ntb > 0)
    v.push_back(force_staged_call(g->multi, ev ? MODE_EV : MODE_FORCE, g->d_desc, g->d_tb, g->ntb,
                                  g->d_ctl, g->nte, g->window_cap, StepArgs{}));
  return v;
}

// the step kernels: force + integrate of every member, global-list systems then
// staged ones; the last of all their blocks makes the step's decisions and sets
// `cond` (when use_cond) for the rebuild that follows
std::vector<KernelCall> step_calls(const Group* g, cudaGraphConditionalHandle cond, int use_cond) {
  StepArgs sa;
  sa.nsys = (int)live(g).size();
  sa.total_blocks = g->ntf + g->ntb;
  sa.cond = cond;
  sa.use_cond = use_cond;
  std::vector<KernelCall> v;
  if (g->nvt) {   // forces + closing half + thermostat, then the opening half and drift
    StepArgs a = sa;
    a.total_blocks = g->ntf;
    a.cond = 0;
    a.use_cond = 0;
    v.push_back(force_call(g->precision, g->multi, MODE_NVT_A, g->tpp, g->fblock, g->d_desc, g->d_tf,
                           g->ntf, g->d_ctl, a, g->eval));
    StepArgs b = sa;
    b.total_blocks = g->ntp;
    v.push_back(nvt_b_call(g->precision, g->d_desc, g->d_tp, g->ntp, g->d_ctl, b));
    return v;
  }
  if (g->ntf > 0)
    v.push_back(force_call(g->precision, g->multi, MODE_STEP, g->tpp, g->fblock, g->d_desc, g->d_tf,
                           g->ntf, g->d_ctl, sa, g->eval));
  if (g->ntb > 0)
    v.push_back(force_staged_call(g->multi, MODE_STEP, g->d_desc, g->d_tb, g->ntb, g->d_ctl, g->nte,
                                  g->window_cap, sa));
  return v;
}

// The rebuild of a step of one system alone as one cooperative kernel after the step
// kernel (no conditional node); null func: the group does not take it.  Up to COOP_MAX_N
// particles, with several types on the cell list COOP_MAX_TYPES_N: the separate kernels of a
// big rebuild balance better over the SMs than resident warps do.  us a step with the
// conditional node / with this: one type, N = 250,000 83.7 / 78.1, 400,000 118.3 / 114.8,
// 700,000 163.8 / 164.6, 10^6 245 / 254; KA 90,000 55.9 / 52.7, 250,000 109.7 / 109.1, 400,000
// 163 / 171, 10^6 314 / 351; WCA 1:10 on the tree 250,000 59 / 51.
constexpr int COOP_MAX_N = 400000, COOP_MAX_TYPES_N = 262144;
int coop_rebuild(const Group* g, bool alone, KernelCall* out) {
  out->func = nullptr;
  std::vector<gbmd_system*> m = live(g);
  if (!alone || m.size() != 1 || m[0]->h.staged) return GBMD_OK;
  if (m[0]->h.n > (g->multi && !m[0]->h.tree ? COOP_MAX_TYPES_N : COOP_MAX_N)) return GBMD_OK;
  TeamFit fit;
  RET(team_fit(rebuild_func(g->multi > 0), REBUILD_T, REBUILD_SMEM, g->device, &fit));
  if (fit.blocks_per_sm < 1) return GBMD_OK;
  *out = rebuild_call(g->d_desc, fit.sms, g->d_ctl, g->multi > 0);
  return GBMD_OK;
}

int add_kernel(cudaGraph_t graph, const cudaGraphNode_t* dep, const KernelCall& k,
               cudaGraphNode_t* out) {
  cudaKernelNodeParams p{};
  p.func = k.func;
  p.gridDim = k.grid;
  p.blockDim = k.block;
  p.sharedMemBytes = (unsigned)k.smem;
  void* a[10];
  args_of(k, a);
  p.kernelParams = a;
  p.extra = nullptr;
  CK(cudaGraphAddKernelNode(out, graph, dep, dep ? 1 : 0, &p));
  if (k.cooperative) {
    cudaKernelNodeAttrValue v{};
    v.cooperative = 1;
    CK(cudaGraphKernelNodeSetAttribute(*out, cudaLaunchAttributeCooperative, &v));
  }
  return GBMD_OK;
}

int build_graph(Group* g, int nsteps, bool alone, StepGraphs* q, cudaGraphExec_t* exec) {
  cudaGraph_t graph;
  CK(cudaGraphCreate(&graph, 0));
  const bool events = nsteps == 1 && g->ev_begin && g->ev_end;
  cudaGraphNode_t prev = nullptr;
  KernelCall coop;
  int rc = coop_rebuild(g, alone, &coop);
  for (int st = 0; st < nsteps && rc == GBMD_OK; ++st) {
    cudaGraphConditionalHandle h = 0;
    cudaError_t e = coop.func ? cudaSuccess
                              : cudaGraphConditionalHandleCreate(&h, graph, 0, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) { rc = fail(GBMD_ERR_CUDA, "conditional handle: %s", cudaGetErrorString(e)); break; }
    // force + integrate (event nodes around them when asked), then IF(rebuild){lists}
    cudaGraphNode_t before = prev;
    if (events) {
      e = cudaGraphAddEventRecordNode(&q->ev_begin, graph, before ? &before : nullptr, before ? 1 : 0,
                                      g->ev_begin);
      if (e != cudaSuccess) { rc = fail(GBMD_ERR_CUDA, "event node: %s", cudaGetErrorString(e)); break; }
      before = q->ev_begin;
    }
    for (const KernelCall& k : step_calls(g, h, coop.func ? 0 : 1)) {
      cudaGraphNode_t n5;
      rc = add_kernel(graph, before ? &before : nullptr, k, &n5);
      if (rc) break;
      before = n5;
    }
    if (rc) break;
    if (events) {
      e = cudaGraphAddEventRecordNode(&q->ev_end, graph, &before, 1, g->ev_end);
      if (e != cudaSuccess) { rc = fail(GBMD_ERR_CUDA, "event node: %s", cudaGetErrorString(e)); break; }
      before = q->ev_end;
    }
    if (coop.func) {
      cudaGraphNode_t nr;
      rc = add_kernel(graph, &before, coop, &nr);
      if (rc) break;
      prev = nr;
      continue;
    }
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeIf;
    cp.conditional.size = 1;
    cudaGraphNode_t nc;
    e = cudaGraphAddNode(&nc, graph, &before, nullptr, 1, &cp);
    if (e != cudaSuccess) { rc = fail(GBMD_ERR_CUDA, "conditional node: %s", cudaGetErrorString(e)); break; }
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    cudaGraphNode_t bprev = nullptr;
    for (const KernelCall& k : rebuild_calls(g)) {
      cudaGraphNode_t bn;
      rc = add_kernel(body, bprev ? &bprev : nullptr, k, &bn);
      if (rc) break;
      bprev = bn;
    }
    if (rc) break;
    prev = nc;
  }
  if (rc == GBMD_OK) {
    cudaError_t e = cudaGraphInstantiate(exec, graph, 0);
    if (e != cudaSuccess) rc = fail(GBMD_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(e));
  }
  if (events && rc == GBMD_OK) q->graph_one = graph;   // node handles stay valid
  else cudaGraphDestroy(graph);
  return rc;
}

int ensure_graphs(Group* g, bool alone, StepGraphs** out) {
  RET(sync_layout(g));
  KernelCall coop;
  RET(coop_rebuild(g, true, &coop));
  StepGraphs& q = g->graphs[alone || !coop.func ? 0 : 1];   // the same without that kernel
  *out = &q;
  if (q.built) return GBMD_OK;
  RET(build_graph(g, STEPS_PER_GRAPH, alone, &q, &q.many));
  RET(build_graph(g, 1, alone, &q, &q.one));
  q.built = true;
  return GBMD_OK;
}

// the streams that a batch's classes run on beside the group's own, and their events
// (event 0: the fork)
int team_stream(Group* g, size_t q) {
  if (!g->side_ev[0]) CK(cudaEventCreateWithFlags(&g->side_ev[0], cudaEventDisableTiming));
  if (g->side[q - 1]) return GBMD_OK;
  CK(cudaEventCreateWithFlags(&g->side_ev[q], cudaEventDisableTiming));
  CK(cudaStreamCreateWithFlags(&g->side[q - 1], cudaStreamNonBlocking));
  return GBMD_OK;
}

// n steps of the group's team members by its plan, one launch per TEAM_STEPS steps
int launch_team(Group* g, long long n) {
  const TeamPlan& p = g->plan;
  TeamArgs a{};
  a.desc = g->d_desc;
  a.ctl = g->d_ctl;
  if (p.shares) {
    a.share = g->d_share;
    a.sync = g->d_sync;
  }
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = dim3(TEAM_T);
  cfg.dynamicSmemBytes = TEAM_SMEM;
  cudaLaunchAttribute at{};
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  void* args[1] = {&a};
  const std::vector<TeamClass>& cls = p.cls;
  for (long long k = 0; k < n; k += TEAM_STEPS) {
    a.nsteps = (int)std::min<long long>(TEAM_STEPS, n - k);
    for (size_t q = 0; q < cls.size(); ++q) {
      const TeamClass& c = cls[q];
      a.list = g->d_team + c.first;
      a.cluster = c.cluster;
      cfg.stream = g->stream;
      if (q > 0) {
        RET(team_stream(g, q));
        if (k == 0) CK(cudaStreamWaitEvent(g->side[q - 1], g->side_ev[0], 0));
        cfg.stream = g->side[q - 1];
      } else if (k == 0 && cls.size() > 1) {
        RET(team_stream(g, 1));
        CK(cudaEventRecord(g->side_ev[0], g->stream));
      }
      if (c.cluster) {
        cfg.gridDim = dim3((unsigned)(c.last - c.first) * c.cluster);
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim = {(unsigned)c.cluster, 1, 1};
      } else {
        cfg.gridDim = dim3(a.share ? (int)g->share.size() : p.fit.blocks_per_sm * p.fit.sms);
        at.id = cudaLaunchAttributeCooperative;
        at.val.cooperative = 1;
      }
      CK(cudaLaunchKernelExC(&cfg, p.func, args));
    }
  }
  for (size_t q = 1; q < cls.size(); ++q) {
    CK(cudaEventRecord(g->side_ev[q], g->side[q - 1]));
    CK(cudaStreamWaitEvent(g->stream, g->side_ev[q], 0));
  }
  return GBMD_OK;
}

// enqueue n steps of the group: by the team kernel, and (members it does not take; a single
// step with event records around its force kernel; a grid beside other streams' work; graphs
// switched off) graphs or direct launches
int enqueue_steps(Group* g, long long n, bool alone) {
  if (n <= 0 || live(g).empty()) return GBMD_OK;
  RET(sync_layout(g));
  const bool whole_grid = !g->plan.cls.empty() && g->plan.cls[0].cluster == 0;
  if (!g->team.empty() && !(n == 1 && g->ev_begin && g->ev_end) && (alone || !whole_grid)) {
    RET(launch_team(g, n));
    return g->rest ? enqueue_steps(g->rest, n, alone) : GBMD_OK;
  }
  if (g->use_graphs) {
    StepGraphs* q;
    RET(ensure_graphs(g, alone, &q));
    for (long long k = 0; k < n / STEPS_PER_GRAPH; ++k) CK(cudaGraphLaunch(q->many, g->stream));
    for (long long k = 0; k < n % STEPS_PER_GRAPH; ++k) CK(cudaGraphLaunch(q->one, g->stream));
    return GBMD_OK;
  }
  for (long long k = 0; k < n; ++k) {
    const bool events = n == 1 && g->ev_begin && g->ev_end;
    if (events) CK(cudaEventRecord(g->ev_begin, g->stream));
    {
      Range r("gbmd step kernel launches");
      for (const KernelCall& c : step_calls(g, 0, 0)) CK(launch(c, g->stream));
    }
    if (events) CK(cudaEventRecord(g->ev_end, g->stream));
    Range r("gbmd rebuild kernel launches");
    for (const KernelCall& c : rebuild_calls(g)) CK(launch(c, g->stream));
  }
  return GBMD_OK;
}

// the same for a caller, whose stream has work from here on
int take_steps(Group* g, long long n) {
  if (n <= 0) return GBMD_OK;
  const bool al = alone(g->device, g->stream);
  enqueued(g->device, g->stream);
  return enqueue_steps(g, n, al);
}

int read_flags(gbmd_system* s, Flags* f, cudaStream_t st) {
  CK(cudaMemcpyAsync(f, s->d_flags, sizeof(Flags), cudaMemcpyDeviceToHost, st));
  CK(wait_for(s->device, st));
  return GBMD_OK;
}

int write_flags(gbmd_system* s, const Flags* f, cudaStream_t st) {
  CK(cudaMemcpyAsync(s->d_flags, f, sizeof(Flags), cudaMemcpyHostToDevice, st));
  CK(cudaStreamSynchronize(st));
  return GBMD_OK;
}

// the Snapshot that the last readout kernel left
int read_snapshot(gbmd_system* s, Snapshot* o, cudaStream_t st) {
  CK(cudaMemcpyAsync(o, s->h.thermo, sizeof(Snapshot), cudaMemcpyDeviceToHost, st));
  CK(wait_for(s->device, st));
  return GBMD_OK;
}

// no error to recover from and no steps owed: what a readout enqueued behind the steps
// has read is the state they end in
bool settled(const gbmd_system* s, const Flags& f) {
  const long long want = s->step_limit >= 0 ? std::min(s->target_step, s->step_limit) : s->target_step;
  return f.error == 0 && f.step >= want;
}

cudaStream_t cur_stream(gbmd_system* s) { return s->own->stream; }

// rebuild lists (when flags->do_rebuild) + forces, outside any graph, for the system alone
int rebuild_and_force(gbmd_system* s, int ev) {
  Group* g = s->own;
  RET(sync_layout(g));
  KernelCall coop;
  coop.func = nullptr;
  if (g->use_graphs) RET(coop_rebuild(g, alone(g->device, g->stream), &coop));
  if (coop.func) CK(launch(coop, g->stream));
  else for (const KernelCall& c : rebuild_calls(g)) CK(launch(c, g->stream));
  for (const KernelCall& c : force_calls(g, ev)) CK(launch(c, g->stream));
  return GBMD_OK;
}

int dalloc(gbmd_system* s, void** p, size_t bytes) {
  bytes = std::max<size_t>(bytes, 16);
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) return fail(GBMD_ERR_OOM, "cudaMalloc(%zu) failed: %s", bytes, cudaGetErrorString(e));
  s->allocs[*p] = bytes;
  s->footprint += bytes;
  return GBMD_OK;
}

void dfree(gbmd_system* s, void* p) {
  auto it = s->allocs.find(p);
  if (it != s->allocs.end()) {
    s->footprint -= it->second;
    s->allocs.erase(it);
  }
  cudaFree(p);
}

// Grow the neighbour list to hold `need` neighbours per particle.
int grow_nlist(gbmd_system* s, int need) {
  const int cap = (int)round_up((size_t)need + need / 4 + 8, 8);
  CK(wait_for(s->device, cur_stream(s)));
  dfree(s, s->h.nl);
  s->h.nl = nullptr;
  RET(dalloc(s, (void**)&s->h.nl, (size_t)s->h.nl_stride * cap * sizeof(int)));
  s->h.cap = cap;
  return refresh_desc(s);
}

// the errors that nothing recovers from.  After DEV_TEAM the bins' counts and, in a
// re-sort, the particles' order may be half written, so that not even a new state (which
// keeps the types) can be taken
int stopped(const Flags& f) {
  if (f.error == DEV_NONFINITE)
    return fail(GBMD_ERR_NONFINITE, "non-finite coordinate or a particle moved more than L/2 in one step (step %lld)", f.step);
  if (f.error == DEV_TEAM)
    return fail(GBMD_ERR_TIMEOUT, "a wait between thread blocks ran out (step %lld)", f.step);
  if (f.error == DEV_TREE)
    return fail(GBMD_ERR_TIMEOUT, "a tree traversal passed its node bound (step %lld)", f.step);
  return GBMD_OK;
}

// Wait for the system's work; recover from overflow; run what remains of its steps.
int sync_system(gbmd_system* s) {
  cudaStream_t st = cur_stream(s);
  for (int round = 0; round < 64; ++round) {
    Flags f;
    RET(read_flags(s, &f, st));   // waits for the stream
    RET(stopped(f));
    if (f.error == DEV_WINDOW) {   // a staged window outgrew shared memory
      s->h.staged = 0;
      RET(refresh_desc(s));
      f.error = 0;
      f.do_rebuild = 1;
      RET(write_flags(s, &f, st));
      RET(rebuild_and_force(s, 0));
      continue;
    }
    if (f.error == DEV_OVERFLOW) {
      Range r("gbmd neighbour-list overflow recovery");
      RET(grow_nlist(s, std::max(f.overflow_need, s->h.cap + 1)));
      f.error = 0;
      f.overflow_need = 0;
      f.do_rebuild = 1;
      RET(write_flags(s, &f, st));
      RET(rebuild_and_force(s, 0));   // finishes the interrupted step
      continue;
    }
    if (f.error) return fail(GBMD_ERR_CUDA, "unknown device error %d", f.error);
    long long want = s->target_step;
    if (s->step_limit >= 0) want = std::min(want, s->step_limit);
    if (f.step < want) {
      RET(take_steps(s->own, want - f.step));
      continue;
    }
    return GBMD_OK;
  }
  return fail(GBMD_ERR_NLIST_OVERFLOW, "neighbour list kept overflowing");
}

// the cut-off radius of type pair p: the rcut table, except WCA's 2^(1/6) sigma
double cut_of(const gbmd_desc* d, int p) {
  return d->potential == GBMD_POT_WCA ? std::pow(2.0, 1.0 / 6.0) * d->sigma[p] : d->rcut[p];
}

// the pair tables the potential reads: present, finite, in range and symmetric
int validate_pairs(const gbmd_desc* d, double* rmax_out) {
  const int pot = d->potential;
  if (pot < GBMD_POT_LJ || pot > GBMD_POT_GAUSS) return fail(GBMD_ERR_BAD_ARG, "potential must be a gbmd_potential (0..4)");
  const bool need_sigma = pot != GBMD_POT_YUKAWA, need_rcut = pot != GBMD_POT_WCA;
  const bool signed_eps = pot == GBMD_POT_YUKAWA || pot == GBMD_POT_GAUSS;
  if (!d->eps || (need_sigma && !d->sigma) || (need_rcut && !d->rcut))
    return fail(GBMD_ERR_BAD_ARG, "a pair table the potential reads (eps, sigma, rcut) is NULL");
  if (pot == GBMD_POT_MIE && (!d->mie_n || !d->mie_m)) return fail(GBMD_ERR_BAD_ARG, "Mie needs mie_n and mie_m");
  if (pot == GBMD_POT_YUKAWA && !d->kappa) return fail(GBMD_ERR_BAD_ARG, "Yukawa needs kappa");
  const int nt = d->ntypes;
  double rmax = 0;
  for (int a = 0; a < nt; ++a)
    for (int b = 0; b < nt; ++b) {
      const int p = a * nt + b, q = b * nt + a;
      auto sym = [&](const double* t) { return !t || t[p] == t[q]; };
      const double e = d->eps[p];
      if (!std::isfinite(e) || (signed_eps ? e == 0 : !(e > 0)))
        return fail(GBMD_ERR_BAD_ARG, "eps must be finite and %s", signed_eps ? "nonzero" : "positive");
      if (need_sigma && (!(d->sigma[p] > 0) || !std::isfinite(d->sigma[p])))
        return fail(GBMD_ERR_BAD_ARG, "sigma must be positive and finite");
      if (need_rcut && (!(d->rcut[p] > 0) || !std::isfinite(d->rcut[p])))
        return fail(GBMD_ERR_BAD_ARG, "rcut must be positive and finite");
      if (pot == GBMD_POT_MIE && !(d->mie_m[p] > 0 && d->mie_n[p] > d->mie_m[p] && std::isfinite(d->mie_n[p])))
        return fail(GBMD_ERR_BAD_ARG, "Mie exponents need 0 < m < n (finite)");
      if (pot == GBMD_POT_YUKAWA && !(d->kappa[p] >= 0 && std::isfinite(d->kappa[p])))
        return fail(GBMD_ERR_BAD_ARG, "kappa must be >= 0 and finite");
      const bool s = sym(d->eps) && (!need_sigma || sym(d->sigma)) && (!need_rcut || sym(d->rcut)) &&
                     (pot != GBMD_POT_MIE || (sym(d->mie_n) && sym(d->mie_m))) &&
                     (pot != GBMD_POT_YUKAWA || sym(d->kappa));
      if (!s) return fail(GBMD_ERR_BAD_ARG, "pair parameter tables must be symmetric");
      rmax = std::max(rmax, cut_of(d, p));
    }
  *rmax_out = rmax;
  return GBMD_OK;
}

int validate(const gbmd_desc* d, bool device) {
  if (!d) return fail(GBMD_ERR_BAD_ARG, "desc is NULL");
  if (d->n < 1 || d->n > (1LL << 30)) return fail(GBMD_ERR_BAD_ARG, "n must be in [1, 2^30], got %lld", (long long)d->n);
  if (!d->pos || !d->vel) return fail(GBMD_ERR_BAD_ARG, "pos and vel must not be NULL");
  if (d->ntypes < 1 || d->ntypes > GBMD_MAX_TYPES) return fail(GBMD_ERR_BAD_ARG, "ntypes must be in [1, %d]", GBMD_MAX_TYPES);
  for (int a = 0; a < 3; ++a)
    if (!(d->box[a] > 0) || !std::isfinite(d->box[a])) return fail(GBMD_ERR_BAD_ARG, "box edges must be positive and finite");
  if (!(d->dt > 0) || !(d->mass > 0) || !(d->r_buff >= 0) || !std::isfinite(d->dt) || !std::isfinite(d->r_buff))
    return fail(GBMD_ERR_BAD_ARG, "need dt > 0, mass > 0, r_buff >= 0");
  if (d->precision != GBMD_FP64 && d->precision != GBMD_MIXED) return fail(GBMD_ERR_BAD_ARG, "precision must be GBMD_FP64 or GBMD_MIXED");
  if (d->sort_period < 0 || d->nlist_capacity < 0) return fail(GBMD_ERR_BAD_ARG, "sort_period and nlist_capacity must be >= 0");
  if (d->threads_per_particle != 0 && !tpp_supported(d->threads_per_particle))
    return fail(GBMD_ERR_BAD_ARG, "threads_per_particle must be 0, 1, 2 or 4");
  if (d->force_path != GBMD_PATH_GLOBAL && d->force_path != GBMD_PATH_STAGED)
    return fail(GBMD_ERR_BAD_ARG, "force_path must be GBMD_PATH_GLOBAL or GBMD_PATH_STAGED");
  if (d->integrator != GBMD_NVE && d->integrator != GBMD_NVT)
    return fail(GBMD_ERR_BAD_ARG, "integrator must be GBMD_NVE or GBMD_NVT");
  if (d->nlist != GBMD_NLIST_CELL && d->nlist != GBMD_NLIST_TREE)
    return fail(GBMD_ERR_BAD_ARG, "nlist must be GBMD_NLIST_CELL or GBMD_NLIST_TREE");
  if (d->integrator == GBMD_NVT &&
      (!(d->kT > 0) || !(d->tau > 0) || !std::isfinite(d->kT) || !std::isfinite(d->tau) || d->n < 2))
    return fail(GBMD_ERR_BAD_ARG, "NVT needs kT > 0, tau > 0 and at least 2 particles");
  if (d->n_ghost < 0 || d->n_ghost >= d->n) return fail(GBMD_ERR_BAD_ARG, "n_ghost must be in [0, n)");
  if (d->n_ghost > 0 && (d->integrator != GBMD_NVE || d->force_path != GBMD_PATH_GLOBAL))
    return fail(GBMD_ERR_BAD_ARG, "ghosts need the NVE integrator and the global force path");
  const int nt = d->ntypes;
  double rmax = 0;
  RET(validate_pairs(d, &rmax));
  const double rl = rmax + d->r_buff;
  for (int a = 0; a < 3; ++a)
    if (d->box[a] < 2.0 * rl)
      return fail(GBMD_ERR_BOX_TOO_SMALL, "box edge %d (%g) < 2 (r_cut,max + r_buff) = %g", a, d->box[a], 2 * rl);
  if (!device) {
    for (int64_t i = 0; i < 3 * d->n; ++i)
      if (!std::isfinite(d->pos[i]) || !std::isfinite(d->vel[i])) return fail(GBMD_ERR_BAD_ARG, "non-finite position or velocity");
    if (d->type)
      for (int64_t i = 0; i < d->n; ++i)
        if (d->type[i] < 0 || d->type[i] >= nt) return fail(GBMD_ERR_BAD_ARG, "type id out of range at %lld", (long long)i);
  }
  return GBMD_OK;
}

// the evaluator coefficients of type pair p (PairD's p0..p4 and the unshifted
// V(r_cut) as `shift`), cut at rc
void pair_coefficients(const gbmd_desc* d, int p, double rc, PairD* c) {
  const double e = d->eps[p];
  switch (d->potential) {
    case GBMD_POT_MIE: {
      const double sg = d->sigma[p], n = d->mie_n[p], m = d->mie_m[p];
      const double ce = n / (n - m) * std::pow(n / m, m / (n - m)) * e;
      const double x = sg * sg / (rc * rc);
      c->p0 = sg * sg;
      c->p1 = 0.5 * n;
      c->p2 = 0.5 * m;
      c->p3 = ce;
      c->shift = ce * (std::pow(x, 0.5 * n) - std::pow(x, 0.5 * m));
      break;
    }
    case GBMD_POT_YUKAWA: {
      const double k = d->kappa[p];
      c->p0 = e;
      c->p1 = k;
      c->shift = e * std::exp(-k * rc) / rc;
      break;
    }
    case GBMD_POT_GAUSS: {
      const double sg = d->sigma[p];
      c->p0 = e;
      c->p1 = 1.0 / (2.0 * sg * sg);
      c->p2 = e / (sg * sg);
      c->shift = e * std::exp(-rc * rc / (2.0 * sg * sg));
      break;
    }
    default: {   // LJ; WCA with rc = 2^(1/6) sigma
      const double sg = d->sigma[p];
      const double s6 = std::pow(sg, 6.0), s12 = s6 * s6;
      const double c2 = sg * sg / (rc * rc), c6 = c2 * c2 * c2, c12 = c6 * c6;
      c->p0 = 48.0 * e * s12;
      c->p1 = 24.0 * e * s6;
      c->p3 = 4.0 * e * s12;
      c->p4 = 4.0 * e * s6;
      c->shift = 4.0 * e * (c12 - c6);
    }
  }
}

struct Geometry {
  int nc[3];
  int ncells;
  int nbins;        // sort bins: ncells, or ntypes * ncells on the tree list
  int cap;
  double rl_max;
  double cell_min;  // smallest cell width
};

// cells per axis: as many as fit with a width of at least scale * cell_min (for the
// cell list cell_min = r_list,max: the 27-cell stencil then holds every neighbour),
// at most 1024
int cells_along(double L, double cell_min, double scale) {
  const int c = (int)std::floor(L / (cell_min * scale * (1.0 + 1e-6)));
  return std::min(std::max(c, 1), 1024);
}

// type_counts (particles per type, or NULL when unknown) refines the default list
// capacity of the tree list: sum over types t of rho_t (4/3) pi r_list(i, t)^3 for the
// worst type i, instead of rho (4/3) pi r_list,max^3
Geometry geometry(const gbmd_desc* d, const int64_t* type_counts = nullptr) {
  Geometry g;
  const int nt = d->ntypes;
  const bool tree = d->nlist == GBMD_NLIST_TREE;
  double rmax = 0, rmin = 1e300;
  for (int p = 0; p < nt * nt; ++p) {
    rmax = std::max(rmax, cut_of(d, p));
    rmin = std::min(rmin, cut_of(d, p));
  }
  const double vol = d->box[0] * d->box[1] * d->box[2];
  g.rl_max = rmax + d->r_buff;
  // the tree list's cells only order the particles (by Morton code inside a cell):
  // about 32 particles per cell, and no finer than the smallest r_list
  g.cell_min = tree ? std::max(rmin + d->r_buff, std::cbrt(32.0 * vol / (double)d->n)) : g.rl_max;
  g.ncells = 1;
  for (int a = 0; a < 3; ++a) {
    g.nc[a] = cells_along(d->box[a], g.cell_min, 1.0);
    g.ncells *= g.nc[a];
  }
  g.nbins = tree ? nt * g.ncells : g.ncells;
  if (d->nlist_capacity > 0) {
    g.cap = (int)round_up((size_t)d->nlist_capacity, 4);   // whole slot groups
  } else {
    const double rho = (double)d->n / vol;
    double nexp = rho * 4.0 / 3.0 * M_PI * g.rl_max * g.rl_max * g.rl_max;
    if (tree && type_counts) {
      nexp = 0;
      for (int a = 0; a < nt; ++a) {
        double e = 0;
        for (int b = 0; b < nt; ++b) {
          const double rl = cut_of(d, a * nt + b) + d->r_buff;
          e += (double)type_counts[b] / vol * 4.0 / 3.0 * M_PI * rl * rl * rl;
        }
        if (type_counts[a] > 0) nexp = std::max(nexp, e);
      }
    }
    g.cap = (int)round_up((size_t)(nexp * 1.4 + 24), 8);
    g.cap = std::min<int>(g.cap, (int)std::max<int64_t>(8, round_up((size_t)d->n, 8)));
  }
  return g;
}

uint32_t spread3(uint32_t v) {   // 10 bits -> every third bit
  v &= 0x3ff;
  v = (v | (v << 16)) & 0x030000FF;
  v = (v | (v << 8)) & 0x0300F00F;
  v = (v | (v << 4)) & 0x030C30C3;
  v = (v | (v << 2)) & 0x09249249;
  return v;
}

size_t footprint_of(const gbmd_desc* d, const Geometry& g) {
  const size_t n = (size_t)d->n;
  size_t b = 0;
  b += n * (8 * 3 * 2);          // x, v
  b += n * 4 * 3 + n * 4 * 3;    // img, rtag/tag/type
  b += n * 16 * 3;               // q (two step-parity buffers), q_build
  if (d->precision == GBMD_FP64) b += n * 32 * 2;   // p64 (two buffers)
  b += n * (d->precision == GBMD_FP64 ? 32 : 16);   // force
  b += n * 4 + round_up(n, 32) * 4 * (size_t)g.cap;  // nn, nl (ELL4)
  b += n * (4 * 5 + 16) + (size_t)(g.nbins + 1) * 4 * 3 + (size_t)g.ncells * 4 * 2;   // cells, keys
  if (d->nlist == GBMD_NLIST_TREE)   // tree boxes and arrival counters (<= n + 4 ntypes
    b += (n + 4 * (size_t)d->ntypes) * (sizeof(TreeBox) + 4) + n * 16;  // nodes), leaves
  b += (size_t)((g.nc[0] + 1) / 2) * ((g.nc[1] + 1) / 2) * ((g.nc[2] + 1) / 2) *
       (WIN_CELLS * 8 + 16);                                                      // staged blocks
  b += n * (8 * 3 * 2 + 4 * 3 + 4 * 2 + 16);         // re-sort scratch
  b += n * (8 * 3 * 3 + 4 * 3 + 4 * 2);              // import/export staging
  b += 4096;
  return b;
}

// staged force path possible: mixed precision, >= 4 cells per axis, expected windows
// well inside shared memory (a larger one at a rebuild falls back, see sync_system)
bool staged_ok(const SysDev& h, const int nc[3]) {
  const double per_cell = (double)h.n / ((double)nc[0] * nc[1] * nc[2]);
  return h.precision == GBMD_MIXED && nc[0] >= 4 && nc[1] >= 4 && nc[2] >= 4 &&
         WIN_CELLS * per_cell * 1.35 + 96 <= STAGED_WINDOW_CAP;
}

// The cell grid: nc cells per axis, the arrays sized by the cell count and the
// Morton rank of every cell.  Replaces an existing grid (its arrays are freed).
int setup_cells(gbmd_system* s, const int nc[3], cudaStream_t st) {
  SysDev& h = s->h;
  CK(cudaStreamSynchronize(st));
  if (h.cell_cnt) {
    for (void* p : {(void*)h.cell_cnt, (void*)h.cell_start, (void*)h.cell_cursor,
                    (void*)const_cast<int*>(h.rank2lin), (void*)const_cast<int*>(h.lin2rank),
                    (void*)h.blk_win, (void*)h.blk_info})
      dfree(s, p);
    h.cell_cnt = h.cell_start = h.cell_cursor = nullptr;
    h.rank2lin = h.lin2rank = nullptr;
    h.blk_win = nullptr;
    h.blk_info = nullptr;
  }
  int ncells = 1, nblocks = 1;
  for (int a = 0; a < 3; ++a) {
    h.nc[a] = nc[a];
    ncells *= nc[a];
    h.nb[a] = (nc[a] + 1) / 2;
    nblocks *= h.nb[a];
  }
  h.ncells = ncells;
  h.nblocks = nblocks;
  h.nbins = h.tree ? h.ntypes * ncells : ncells;   // the tree list sorts type-major
  const size_t nbins = (size_t)h.nbins;
  int rc = GBMD_OK;
  auto A = [&](void** p, size_t bytes) {
    if (rc == GBMD_OK) rc = dalloc(s, p, bytes);
  };
  A((void**)&h.blk_win, (size_t)nblocks * WIN_CELLS * sizeof(int2));
  A((void**)&h.blk_info, (size_t)nblocks * sizeof(int4));
  A((void**)&h.cell_cnt, (nbins + 1) * 4); A((void**)&h.cell_start, (nbins + 1) * 4);
  A((void**)&h.cell_cursor, (nbins + 1) * 4);
  int *r2l = nullptr, *l2r = nullptr;
  A((void**)&r2l, (size_t)ncells * 4); A((void**)&l2r, (size_t)ncells * 4);
  h.rank2lin = r2l;
  h.lin2rank = l2r;
  if (rc != GBMD_OK) return rc;
  std::vector<std::pair<uint32_t, int>> code(ncells);
  for (int z = 0; z < nc[2]; ++z)
    for (int y = 0; y < nc[1]; ++y)
      for (int x = 0; x < nc[0]; ++x) {
        const int lin = (z * nc[1] + y) * nc[0] + x;
        code[lin] = {spread3(x) | (spread3(y) << 1) | (spread3(z) << 2), lin};
      }
  std::sort(code.begin(), code.end());
  std::vector<int> rl(ncells), lr(ncells);
  for (int r = 0; r < ncells; ++r) {
    rl[r] = code[r].second;
    lr[code[r].second] = r;
  }
  CK(cudaMemcpyAsync(r2l, rl.data(), (size_t)ncells * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(l2r, lr.data(), (size_t)ncells * 4, cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(h.cell_cnt, 0, (nbins + 1) * 4, st));
  CK(cudaStreamSynchronize(st));   // the host tables die here
  return GBMD_OK;
}

int create_impl(const gbmd_desc* d, gbmd_system** out, bool device) {
  if (!out) return fail(GBMD_ERR_BAD_ARG, "out is NULL");
  *out = nullptr;
  RET(validate(d, device));
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) return fail(GBMD_ERR_NO_DEVICE, "no CUDA device");
  int dev = d->device;
  if (dev < 0) CK(cudaGetDevice(&dev));
  if (dev >= ndev) return fail(GBMD_ERR_BAD_ARG, "device %d does not exist (%d devices)", dev, ndev);
  RET(use_device(dev));
  const bool tree = d->nlist == GBMD_NLIST_TREE;
  int64_t tcount[GBMD_MAX_TYPES] = {0, 0, 0, 0};   // particles per type (tree list)
  if (tree) {
    std::vector<int32_t> ty;
    const int32_t* tp = d->type;
    if (tp && device) {   // the tree layout is fixed by the type counts: read them once
      ty.resize((size_t)d->n);
      CK(cudaMemcpy(ty.data(), tp, (size_t)d->n * 4, cudaMemcpyDeviceToHost));
      tp = ty.data();
    }
    for (int64_t i = 0; i < d->n; ++i) {
      const int t = tp ? tp[i] : 0;
      if (t < 0 || t >= d->ntypes) return fail(GBMD_ERR_BAD_ARG, "type id out of range at %lld", (long long)i);
      ++tcount[t];
    }
  }
  const Geometry geo = geometry(d, tree ? tcount : nullptr);
  gbmd_system* s = new gbmd_system();
  s->device = dev;
  s->stream = (cudaStream_t)d->stream;
  SysDev& h = s->h;
  const int n = (int)d->n, nt = d->ntypes;
  h.n = n;
  h.n_ghost = (int)d->n_ghost;
  h.ntypes = nt;
  h.precision = d->precision;
  h.sort_period = d->sort_period;
  h.cap = geo.cap;
  h.nl_stride = (int)round_up((size_t)n, 32);
  h.dt = d->dt;
  h.mass = d->mass;
  h.h = 0.5 * d->dt / d->mass;
  s->cell_min = geo.cell_min;
  s->want_staged = d->force_path == GBMD_PATH_STAGED && d->integrator == GBMD_NVE &&
                   eval_of(d->potential) == EVAL_LJ && !tree;
  h.tree = tree ? 1 : 0;
  int nodes = 0;
  if (tree) {   // type t: particles [first, first + n) of the sorted order, P leaves
    int first = 0, leaves = 0;
    for (int t = 0; t < nt; ++t) {
      h.tree_first[t] = first;
      h.tree_n[t] = (int)tcount[t];
      h.tree_P[t] = tree_leaves((int)tcount[t]);
      h.tree_leaf0[t] = leaves;
      h.tree_node0[t] = nodes;
      first += (int)tcount[t];
      leaves += h.tree_P[t];
      nodes += 2 * h.tree_P[t];   // boxes 1 .. 2P - 1 (0 unused)
    }
    h.tree_leaves_total = leaves;
    // query order: the types by decreasing expected work per particle
    double work[GBMD_MAX_TYPES];
    int ord[GBMD_MAX_TYPES];
    for (int t = 0; t < nt; ++t) {
      work[t] = 0;
      for (int u = 0; u < nt; ++u) {
        const double rl = cut_of(d, t * nt + u) + d->r_buff;
        work[t] += (double)tcount[u] * rl * rl * rl;
      }
      ord[t] = t;
    }
    std::stable_sort(ord, ord + nt, [&](int a, int b) { return work[a] > work[b]; });
    const double vol = d->box[0] * d->box[1] * d->box[2];
    for (int k = 0; k < nt; ++k) {
      h.tree_qtype[k] = ord[k];
      // a group of 8 spans about two spacings of its type: where that is more than the
      // type's reach, the group's box would mostly hold strangers
      double reach = 0;
      for (int u = 0; u < nt; ++u) reach = std::max(reach, cut_of(d, k * nt + u) + d->r_buff);
      h.tree_single[k] = tcount[k] > 0 && 2.0 * std::cbrt(vol / (double)tcount[k]) > reach;
      // few particles with long rows: their lanes' chains would outlive the rest
      h.tree_wide[k] = work[k] * 4.0 / 3.0 * M_PI / vol >= 64.0 && 32 * tcount[k] <= n;
    }
  }
  h.nvt = d->integrator == GBMD_NVT;
  h.kT = d->kT;
  h.tau = d->tau;
  h.gdof = 3.0 * (double)n - 3.0;
  h.staged = s->want_staged && staged_ok(h, geo.nc);
  h.window_cap = STAGED_WINDOW_CAP;
  for (int a = 0; a < 3; ++a) {
    h.L[a] = d->box[a];
    h.qscale[a] = 4294967296.0 / d->box[a];
    h.dtq[a] = d->dt * h.qscale[a];
    h.fscale[a] = (float)(d->box[a] / 4294967296.0);
  }
  // units of the FP64 gather's positions: half the longest edge is at most 2^61 of them
  int fix_e;
  const double half_max = 0.5 * std::max({d->box[0], d->box[1], d->box[2]});
  if (std::frexp(half_max, &fix_e) == 0.5) --fix_e;
  h.fix_bits = 61 - fix_e;   // half_max <= 2^fix_e
  for (int a = 0; a < 3; ++a) {
    h.fix_q[a] = std::ldexp(d->box[a], h.fix_bits - 32);
    h.fix_L[a] = std::llrint(std::ldexp(d->box[a], h.fix_bits));
    h.fix_half[a] = (unsigned)((unsigned long long)h.fix_L[a] >> 33);
  }
  const double hb = 0.5 * d->r_buff;
  h.rbuff_half2 = (float)(hb * hb * (1.0 - 1e-5));
  h.eval = eval_of(d->potential);
  for (int p = 0; p < nt * nt; ++p) {
    const double rc = cut_of(d, p), rl = rc + d->r_buff;
    PairD& pd = h.pd[p];
    pd = PairD{};
    pair_coefficients(d, p, rc, &pd);
    pd.rc2 = rc * rc;
    pd.rl2 = rl * rl;
    PairF& pf = h.pf[p];
    pf.p0 = (float)pd.p0;
    pf.p1 = (float)pd.p1;
    pf.p2 = (float)pd.p2;
    pf.p3 = (float)pd.p3;
    pf.p4 = (float)pd.p4;
    pf.rc2 = (float)pd.rc2;
    pf.shift = (float)pd.shift;
    pf.rl2 = (float)pd.rl2;
  }
  int rc = GBMD_OK;
  auto A = [&](void** p, size_t bytes) {
    if (rc == GBMD_OK) rc = dalloc(s, p, bytes);
  };
  const size_t N = (size_t)n;
  A((void**)&h.x, N * 24); A((void**)&h.v, N * 24); A((void**)&h.img, N * 12);
  A((void**)&h.type, N * 4); A((void**)&h.tag, N * 4); A((void**)&h.rtag, N * 4);
  A((void**)&h.q, N * 16); A((void**)&h.q1, N * 16); A((void**)&h.q_build, N * 16);
  if (d->precision == GBMD_FP64) {
    A((void**)&h.p64, N * 32); A((void**)&h.p64b, N * 32);
  }
  if (d->precision == GBMD_FP64) A((void**)&h.f64, N * 32); else A((void**)&h.f32, N * 16);
  A((void**)&h.nn, N * 4); A((void**)&h.nl, round_up(N, 32) * 4 * (size_t)geo.cap);
  A((void**)&h.key, N * 4); A((void**)&h.members, N * 4); A((void**)&h.members_tmp, N * 4);
  A((void**)&h.rmember, N * 4);
  A((void**)&h.x_alt, N * 24); A((void**)&h.v_alt, N * 24); A((void**)&h.img_alt, N * 12);
  A((void**)&h.type_alt, N * 4); A((void**)&h.tag_alt, N * 4); A((void**)&h.q_alt, N * 16);
  A((void**)&h.fkey, N * 4);   // fine Morton keys: the order inside a cell
  A((void**)&h.cpos, N * 16);  // positions in cell order (the list build's candidates)
  A((void**)&h.nh, 4 * 8);
  if (tree) {
    A((void**)&h.tree_box, (size_t)nodes * sizeof(TreeBox));
    A((void**)&h.tree_arrive, (size_t)nodes * 4);
    A((void**)&h.tree_q, N * 16);
  }
  A((void**)&s->d_flags, sizeof(Flags));
  // import/export staging behind the snapshot: a small readout comes back in one copy
  A((void**)&h.thermo, SNAPSHOT_BYTES + N * 84);
  s->d_frc = h.thermo + SNAPSHOT_BYTES / 8;
  s->d_vel = s->d_frc + 3 * N;
  s->d_pos = s->d_vel + 3 * N;
  s->d_img = (int*)(s->d_pos + 3 * N);
  s->d_misc = h.thermo ? &((Snapshot*)h.thermo)->bad : nullptr;
  A((void**)&s->d_type, N * 4);
  h.flags = s->d_flags;
  if (rc != GBMD_OK) { gbmd_destroy(s); return rc; }
  cudaStream_t st = s->stream;
  rc = setup_cells(s, geo.nc, st);
  if (rc != GBMD_OK) { std::string m = g_err; gbmd_destroy(s); g_err = m; return rc; }
  {
    const double nh0[4] = {0.0, 0.0, 1.0, 0.0};   // xi, eta, exp(-xi dt/2)
    cudaError_t e5 = cudaMemsetAsync(s->d_flags, 0, sizeof(Flags), st);
    if (!e5) e5 = cudaMemsetAsync(h.thermo, 0, SNAPSHOT_BYTES, st);
    cudaError_t e6 = cudaMemsetAsync(h.nn, 0, N * 4, st);
    if (tree && e6 == cudaSuccess) e6 = cudaMemsetAsync(h.tree_arrive, 0, (size_t)nodes * 4, st);
    cudaError_t e7 = cudaMemcpyAsync(h.nh, nh0, sizeof(nh0), cudaMemcpyHostToDevice, st);
    cudaError_t e4 = cudaStreamSynchronize(st);
    if (e7) { gbmd_destroy(s); return fail(GBMD_ERR_CUDA, "thermostat upload failed"); }
    if (e4 || e5 || e6) { gbmd_destroy(s); return fail(GBMD_ERR_CUDA, "clearing the flags failed"); }
  }
  // own group
  s->own = new Group();
  s->own->device = dev;
  s->own->stream = st;
  s->own->precision = d->precision;
  s->own->members.push_back(s);
  // default tuning (measured on GB300 with the L2 flushed between steps).  Mixed
  // precision: one lane per particle once there are enough particles to fill every
  // SM several times over, two below that; 128-thread blocks.  FP64 (bound by the
  // FP64 pipe): one lane in 64-thread blocks from 32k particles (the 64k fluid
  // steps 10% faster than with two lanes in 128-thread blocks), four lanes in
  // 128-thread blocks below (the 4,000-particle fluid 29% faster)
  const bool fp64 = d->precision == GBMD_FP64;
  // FP64: four lanes while the team's warps take them in one turn (152 SMs of 16 warps,
  // eight particles a warp: 19,456), us a step with 4 / 2 lanes: N = 4,000 22.0 / 30.6,
  // 16,000 33.0 / 35.7, 20,000 53.1 / 41.0, 28,000 54.7 / 45.3; one from 32,768 on (64,000:
  // 85.9, two lanes 91.0)
  const int auto_tpp = fp64 ? (d->n >= 32768 ? 1 : d->n > 19456 ? 2 : 4) : (d->n >= (1 << 19) ? 1 : 2);
  s->own->tpp = d->threads_per_particle ? d->threads_per_particle : auto_tpp;
  s->own->fblock = fp64 && s->own->tpp == 1 ? 64 : 128;
  if (const char* ev = getenv("GBMD_NO_GRAPHS")) s->own->use_graphs = ev[0] != '1';
  *out = s;
  return GBMD_OK;
}

// Upload positions/velocities/types/images (tag order, host or device memory),
// then build the lists (with the initial Morton sort) and compute the forces.  bad (on
// the device): the state is refused when it is set, and nothing of the system changes.
int load_state(gbmd_system* s, const double* pos, const double* vel, const int32_t* type,
               const int32_t* image, bool device, long long step, const int* bad = nullptr) {
  cudaStream_t st = cur_stream(s);
  const size_t N = (size_t)s->h.n;
  const double *dp = pos, *dv = vel;
  const int *dt = type, *di = image;
  if (!device) {
    CK(cudaMemcpyAsync(s->d_pos, pos, N * 24, cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(s->d_vel, vel, N * 24, cudaMemcpyHostToDevice, st));
    dp = s->d_pos;
    dv = s->d_vel;
    if (type) {
      CK(cudaMemcpyAsync(s->d_type, type, N * 4, cudaMemcpyHostToDevice, st));
      dt = s->d_type;
    }
    if (image) {
      CK(cudaMemcpyAsync(s->d_img, image, N * 12, cudaMemcpyHostToDevice, st));
      di = s->d_img;
    }
  }
  Group* g = s->own;
  RET(sync_layout(g));
  CK(launch(load_flags_call(g->d_desc, bad, step, s->step_limit), st));
  CK(launch(import_call(g->d_desc, g->d_tp, g->ntp, dp, dv, dt, di, bad), st));
  RET(rebuild_and_force(s, 0));
  CK(launch(snapshot_call(g->d_desc), st));
  Snapshot snap;
  RET(read_snapshot(s, &snap, st));
  if (bad && snap.bad) return fail(GBMD_ERR_BAD_ARG, "non-finite state");
  Flags after = snap.flags;
  if (after.error == DEV_BADTYPE) return fail(GBMD_ERR_BAD_ARG, "type id out of range in the device type array");
  s->target_step = step;
  RET(stopped(after));
  if (after.error == DEV_WINDOW) {
    s->h.staged = 0;
    RET(refresh_desc(s));
    after.error = 0;
    after.do_rebuild = 1;
    RET(write_flags(s, &after, st));
    RET(rebuild_and_force(s, 0));
    RET(read_flags(s, &after, st));
    RET(stopped(after));
  }
  if (after.error == DEV_OVERFLOW) {
    RET(grow_nlist(s, after.overflow_need));
    after.error = 0;
    after.overflow_need = 0;
    after.do_rebuild = 1;
    RET(write_flags(s, &after, st));
    RET(rebuild_and_force(s, 0));
    RET(read_flags(s, &after, st));
    RET(stopped(after));
    if (after.error) return fail(GBMD_ERR_NLIST_OVERFLOW, "neighbour list overflow at creation");
  }
  return GBMD_OK;
}

// NVT readout of the thermostat, as the state after the last completed step: the
// stored xi / eta are those of the step's opening half; the closing half adds
// dt/2 G(K) to xi and dt/2 xi to eta (nothing right after create / set_state).
// h_ext = K + U (+ g kT (tau^2 xi^2 / 2 + eta) for NVT) is the conserved quantity.
void fill_thermostat(gbmd_system* s, const Flags& f, const double* nh, gbmd_thermo* out) {
  out->xi = 0.0;
  out->eta = 0.0;
  out->h_ext = out->ke + out->pe;
  if (!s->h.nvt) return;
  const SysDev& h = s->h;
  double xi = nh[0], eta = nh[1];
  if (!f.v_full) {
    const double G = (2.0 * out->ke / (h.gdof * h.kT) - 1.0) / (h.tau * h.tau);
    eta += 0.5 * h.dt * xi;
    xi += 0.5 * h.dt * G;
  }
  out->xi = xi;
  out->eta = eta;
  out->h_ext += h.gdof * h.kT * (0.5 * h.tau * h.tau * xi * xi + eta);
}

// the thermodynamic state from a snapshot whose sums are of the current positions
void fill_thermo(gbmd_system* s, const Snapshot& snap, gbmd_thermo* out) {
  const double* t = snap.thermo;
  const double n = (double)s->h.n;
  const double vol = s->h.L[0] * s->h.L[1] * s->h.L[2];
  out->step = snap.flags.step;
  out->pe = t[0];
  out->ke = 0.5 * s->h.mass * t[1];
  out->temperature = n > 1 ? 2.0 * out->ke / (3.0 * n - 3.0) : 0.0;
  for (int c = 0; c < 6; ++c) out->virial[c] = t[2 + c];
  out->w = t[2] + t[5] + t[7];
  out->pressure = (n * out->temperature + out->w / 3.0) / vol;
  out->n_rebuilds = snap.flags.n_rebuilds;
  fill_thermostat(s, snap.flags, snap.nh, out);
}

// Readouts are enqueued behind the steps without waiting for them, with a snapshot of
// the flags as their last kernel saw them; what they read counts once the snapshot says
// that the steps ended well.  Otherwise the system is recovered and they run once more.
// So a readout costs one round trip to the device (two where its arrays are too big for
// one copy through `bounce`), not one for each thing it must know.
constexpr size_t BOUNCE_MAX = 256 * 1024;
// forces and rows by one kernel / by two: N = 64,000 frame 19.4 / 21.5 us, N = 199,999 frame
// 51.2 / 49.3, N = 10^6 forces 181 / 168 (and a launch)
constexpr size_t FUSED_READ_N = 131072;

int thermo_impl(gbmd_system* s, Snapshot* snap) {
  Group* g = s->own;
  cudaStream_t st = cur_stream(s);
  for (int turn = 0; turn < 2; ++turn) {
    RET(sync_layout(g));
    for (const KernelCall& c : force_calls(g, 1)) CK(launch(c, st));
    CK(launch(thermo_call(g->d_desc, g->d_ts, g->nts, g->d_ctl), st));
    RET(read_snapshot(s, snap, st));
    if (settled(s, snap->flags)) return GBMD_OK;
    RET(sync_system(s));
  }
  return fail(GBMD_ERR_STATE, "the system does not settle");
}

int export_impl(gbmd_system* s, double* pos, double* vel, int32_t* image, double* force,
                double* pp_u, double* pp_w, int64_t* step = nullptr) {
  Group* g = s->own;
  cudaStream_t st = cur_stream(s);
  const size_t N = (size_t)s->h.n;
  if ((pp_u || pp_w) && !s->d_ppw) return fail(GBMD_ERR_STATE, "per-particle arrays not allocated");
  for (int turn = 0; turn < 2; ++turn) {
    RET(sync_layout(g));
    // the global-list force kernel writes the rows of a readout itself; up to FUSED_READ_N,
    // beyond which its stores to scattered tags cost more than k_export's launch
    const int readout = !pp_u && !pp_w && (vel || force) && g->ntb == 0 && N <= FUSED_READ_N
                            ? (force ? READ_FORCE : 0) | (vel ? READ_VEL : 0) | (pos ? READ_POS : 0) |
                                  (image ? READ_IMAGE : 0)
                            : 0;
    // forces and full-step velocities need F at the current positions: the step kernel
    // does not store its force, so evaluate it here (per-particle arrays: the energy pass)
    if (pp_u || pp_w)
      for (const KernelCall& c : force_calls(g, 1)) CK(launch(c, st));
    else if (vel || force)
      for (const KernelCall& c : force_calls(g, 0, readout)) CK(launch(c, st));
    if (!readout) CK(launch(export_call(g->d_desc, g->d_tp, g->ntp, pos ? s->d_pos : nullptr,
                          vel ? s->d_vel : nullptr, image ? s->d_img : nullptr,
                          force ? s->d_frc : nullptr, pp_u ? s->d_ppu : nullptr,
                          pp_w ? s->d_ppw : nullptr), st));
    // snapshot, force, velocity, position and image lie one after the other
    const size_t bytes = SNAPSHOT_BYTES + N * (image ? 84 : pos ? 72 : vel ? 48 : force ? 24 : 0);
    Snapshot snap;
    const bool one = !pp_u && !pp_w && bytes <= BOUNCE_MAX;
    if (one) {
      s->bounce.resize(bytes);
      CK(cudaMemcpyAsync(s->bounce.data(), s->h.thermo, bytes, cudaMemcpyDeviceToHost, st));
      CK(wait_for(s->device, st));
      memcpy(&snap, s->bounce.data(), sizeof(snap));
    } else {
      RET(read_snapshot(s, &snap, st));
    }
    if (!settled(s, snap.flags)) {
      RET(sync_system(s));
      continue;
    }
    if (step) *step = snap.flags.step;
    if (one) {
      const char* b = s->bounce.data() + SNAPSHOT_BYTES;
      if (force) memcpy(force, b, N * 24);
      if (vel) memcpy(vel, b + N * 24, N * 24);
      if (pos) memcpy(pos, b + N * 48, N * 24);
      if (image) memcpy(image, b + N * 72, N * 12);
      return GBMD_OK;
    }
    if (pos) CK(cudaMemcpyAsync(pos, s->d_pos, N * 24, cudaMemcpyDeviceToHost, st));
    if (vel) CK(cudaMemcpyAsync(vel, s->d_vel, N * 24, cudaMemcpyDeviceToHost, st));
    if (image) CK(cudaMemcpyAsync(image, s->d_img, N * 12, cudaMemcpyDeviceToHost, st));
    if (force) CK(cudaMemcpyAsync(force, s->d_frc, N * 24, cudaMemcpyDeviceToHost, st));
    if (pp_u) CK(cudaMemcpyAsync(pp_u, s->d_ppu, N * 8, cudaMemcpyDeviceToHost, st));
    if (pp_w) CK(cudaMemcpyAsync(pp_w, s->d_ppw, N * 48, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    return GBMD_OK;
  }
  return fail(GBMD_ERR_STATE, "the system does not settle");
}

int time_force(Group* g, float* ms) {
  RET(sync_layout(g));
  if (g->ntf == 0) {
    *ms = 0.f;
    return GBMD_OK;
  }
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  for (int k = 0; k < 2; ++k) CK(launch(plain_force_call(g), g->stream));
  CK(cudaEventRecord(a, g->stream));
  const int reps = 5;
  for (int k = 0; k < reps; ++k) CK(launch(plain_force_call(g), g->stream));
  CK(cudaEventRecord(b, g->stream));
  CK(cudaEventSynchronize(b));
  float t = 0;
  CK(cudaEventElapsedTime(&t, a, b));
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  *ms = t / reps;
  return GBMD_OK;
}

// Cells at least scale * r_list,max wide: a new cell grid, then the lists (with a
// re-sort into the new Morton order) and the forces at the current positions.  The
// neighbour sets do not change (r_list does not); the order of a particle's
// neighbours, and so the FP32 summation order of its force, may.
int regrid(gbmd_system* s, double scale) {
  if (!(scale >= 1.0 && scale <= 4.0)) return fail(GBMD_ERR_BAD_ARG, "cell scale must be in [1, 4]");
  SysDev& h = s->h;
  int nc[3];
  for (int a = 0; a < 3; ++a) nc[a] = cells_along(h.L[a], s->cell_min, scale);
  s->cell_scale = scale;
  if (nc[0] == h.nc[0] && nc[1] == h.nc[1] && nc[2] == h.nc[2]) return GBMD_OK;
  RET(sync_system(s));   // nothing in flight, nothing owed
  cudaStream_t st = cur_stream(s);
  RET(setup_cells(s, nc, st));
  h.staged = s->want_staged && staged_ok(h, nc);
  RET(refresh_desc(s));
  for (int round = 0; round < 2; ++round) {
    Flags f;
    RET(read_flags(s, &f, st));
    if (round == 1 && f.error != DEV_WINDOW) break;
    if (f.error == DEV_WINDOW) {   // a staged window outgrew shared memory
      h.staged = 0;
      RET(refresh_desc(s));
      f.error = 0;
    }
    f.do_rebuild = 1;
    f.do_sort = 1;
    f.last_sort = f.step;
    f.n_sorts += 1;
    RET(write_flags(s, &f, st));
    RET(rebuild_and_force(s, 0));
    CK(cudaStreamSynchronize(st));
  }
  Flags f;
  RET(read_flags(s, &f, st));
  RET(stopped(f));
  if (f.error) return fail(GBMD_ERR_STATE, "device error %d after a new cell grid", f.error);
  f.do_rebuild = 0;
  f.do_sort = 0;
  return write_flags(s, &f, st);
}

// Mean time of a step, rebuilds included, as gbmd_step / gbmd_batch_step would run it: the
// members' memory is copied aside, steps run, and all of it is put back.  *ms < 0: no room
// for the copy.
int time_steps(Group* g, float* ms) {
  *ms = -1.f;
  RET(sync_layout(g));
  std::vector<gbmd_system*> m = live(g);
  size_t bytes = 0;
  auto step256 = [](size_t b) { return (b + 255) / 256 * 256; };
  for (auto* s : m)
    for (const auto& a : s->allocs) bytes += step256(a.second);
  char* aside = nullptr;
  if (cudaMalloc(&aside, bytes) != cudaSuccess) {
    cudaGetLastError();
    return GBMD_OK;
  }
  auto copy = [&](bool back) -> int {
    char* at = aside;
    for (auto* s : m)
      for (const auto& a : s->allocs) {
        CK(cudaMemcpyAsync(back ? a.first : at, back ? at : a.first, a.second, cudaMemcpyDeviceToDevice, g->stream));
        at += step256(a.second);
      }
    return GBMD_OK;
  };
  auto run = [&]() -> int {
    cudaEvent_t a, b;
    CK(cudaEventCreate(&a));
    CK(cudaEventCreate(&b));
    for (auto* s : m) {   // also where a limit holds the system
      Flags f;
      RET(read_flags(s, &f, g->stream));
      f.step_limit = -1;
      RET(write_flags(s, &f, g->stream));
    }
    constexpr int WARM = 16, STEPS = 64;
    RET(enqueue_steps(g, WARM, true));
    CK(cudaEventRecord(a, g->stream));
    RET(enqueue_steps(g, STEPS, true));
    CK(cudaEventRecord(b, g->stream));
    CK(cudaEventSynchronize(b));
    float t = 0;
    CK(cudaEventElapsedTime(&t, a, b));
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    *ms = t / STEPS;
    for (auto* s : m) {   // a system that stopped (a list that overflowed) was not timed
      Flags f;
      RET(read_flags(s, &f, g->stream));
      if (f.error) *ms = 1e30f;
    }
    return GBMD_OK;
  };
  int rc = copy(false);
  if (rc == GBMD_OK) {
    rc = run();
    const int rb = copy(true);
    if (rc == GBMD_OK) rc = rb;
  }
  cudaStreamSynchronize(g->stream);
  cudaFree(aside);
  return rc;
}

// Mean time of one full list rebuild (no re-sort) of every member of the group, by the
// kernels that the step graph takes.
int time_rebuild(Group* g, float* ms) {
  RET(sync_layout(g));
  std::vector<gbmd_system*> m = live(g);
  for (auto* s : m) {
    Flags f;
    RET(read_flags(s, &f, g->stream));
    f.do_rebuild = 1;
    f.do_sort = 0;
    RET(write_flags(s, &f, g->stream));
  }
  std::vector<KernelCall> calls = rebuild_calls(g);
  KernelCall coop;
  coop.func = nullptr;
  if (g->use_graphs) RET(coop_rebuild(g, true, &coop));
  if (coop.func) calls = {coop};
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  for (const KernelCall& c : calls) CK(launch(c, g->stream));
  CK(cudaEventRecord(a, g->stream));
  const int reps = 3;
  for (int k = 0; k < reps; ++k)
    for (const KernelCall& c : calls) CK(launch(c, g->stream));
  CK(cudaEventRecord(b, g->stream));
  CK(cudaEventSynchronize(b));
  float t = 0;
  CK(cudaEventElapsedTime(&t, a, b));
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  *ms = t / reps;
  for (auto* s : m) {   // the lists stand for the current positions
    Flags f;
    RET(read_flags(s, &f, g->stream));
    RET(stopped(f));
    if (f.error) return fail(GBMD_ERR_STATE, "device error %d while timing a rebuild", f.error);
    f.do_rebuild = 0;
    RET(write_flags(s, &f, g->stream));
  }
  return GBMD_OK;
}

std::string tune_key(const Group* g) {
  std::vector<gbmd_system*> m = live(g);
  long long np = 0;
  double vol = 0;
  for (auto* s : m) {
    np += s->h.n;
    vol += s->h.L[0] * s->h.L[1] * s->h.L[2];
  }
  const int lg = np > 0 ? (int)std::floor(std::log2((double)np)) : 0;
  const int rho10 = vol > 0 ? (int)std::lround(10.0 * np / vol) : 0;
  char buf[512];
  cudaDeviceProp p{};
  int dev = 0;
  cudaGetDevice(&dev);
  cudaGetDeviceProperties(&p, dev);
  snprintf(buf, sizeof(buf), "%s|prec=%d|multi=%d|eval=%d|members=%d|log2n=%d|rho10=%d", p.name,
           g->precision, g->multi, g->eval, (int)m.size(), lg, rho10);
  for (char* c = buf; *c; ++c)
    if (*c == ' ') *c = '_';
  return buf;
}

int set_tuning(Group* g, int tpp, int block) {
  if (!tpp_supported(tpp) || block < 32 || block > 512 || block % 32 || block % tpp)
    return fail(GBMD_ERR_BAD_ARG, "bad tuning tpp=%d block=%d", tpp, block);
  if (g->tpp == tpp && g->fblock == block) return GBMD_OK;
  g->tpp = tpp;
  g->fblock = block;
  g->layout_dirty = true;
  return sync_layout(g);
}

int autotune_group(Group* g, const char* cache) {
  RET(sync_layout(g));
  if (g->ntf == 0) return GBMD_OK;   // every member on the staged path (nothing to tune)
  const std::string key = tune_key(g);
  if (cache) {
    std::ifstream in(cache);
    std::string line;
    int bt = 0, bb = 0;
    double bs = 1.0;
    while (std::getline(in, line)) {
      std::istringstream ls(line);
      std::string k;
      int t, b;
      if (ls >> k >> t >> b && k == key) {
        bt = t;
        bb = b;
        double sc;
        bs = (ls >> sc) ? sc : 1.0;
      }
    }
    if (bt) {
      for (auto* s : live(g)) RET(regrid(s, bs));
      return set_tuning(g, bt, bb);
    }
  }
  // Where the team would step some member at one of the lane counts, what counts is the
  // step itself: the lanes that suit the step kernel need not suit the team, and may be too
  // many for it (team_member).  us a step by default / chosen by the step kernel's time /
  // by the step's: mixed N = 20,000 14.8 / 18.6 / 14.9, FP64 40,000 65.4 / 77.7 / 65.5,
  // FP64 64,000 82.6 / 92.1 / 82.6, 16 replicas of 2,000 30.8 / 20.3 / 20.0.  Otherwise the
  // step kernel and the rebuild are timed.
  const int tpp0 = g->tpp, block0 = g->fblock;
  bool by_steps = false;
  for (int tpp : {1, 2, 4}) {
    RET(set_tuning(g, tpp, block0));
    by_steps |= !g->team.empty();
  }
  RET(set_tuning(g, tpp0, block0));
  if (by_steps) {
    float ms;
    RET(time_steps(g, &ms));
    by_steps = ms >= 0.f;
  }
  // cell width: the list rebuild at each candidate width (the global force path does
  // not depend on it); a wider cell only wins if it is clearly faster
  double best_s = 1.0;
  {
    bool any_staged = false;
    for (auto* s : live(g)) any_staged |= s->h.staged != 0;
    if (!any_staged) {
      float best_r = 1e30f;
      std::vector<std::vector<int>> seen;
      for (double sc : {1.0, 1.1, 1.2, 1.35}) {
        std::vector<int> grid;
        for (auto* s : live(g))
          for (int a = 0; a < 3; ++a) grid.push_back(cells_along(s->h.L[a], s->cell_min, sc));
        if (std::find(seen.begin(), seen.end(), grid) != seen.end()) continue;
        seen.push_back(grid);
        for (auto* s : live(g)) RET(regrid(s, sc));
        float ms;
        if (by_steps) RET(time_steps(g, &ms));
        else RET(time_rebuild(g, &ms));
        if (by_steps && ms < 0.f) continue;
        if (getenv("GBMD_VERBOSE")) fprintf(stderr, "gbmd autotune %s cell_scale=%.2f %s %.4f ms\n", key.c_str(), sc, by_steps ? "step" : "rebuild", ms);
        if (ms < 0.97f * best_r) { best_r = ms; best_s = sc; }
      }
      for (auto* s : live(g)) RET(regrid(s, best_s));
    }
  }
  int best_t = g->tpp, best_b = g->fblock;
  float best = 1e30f;
  // FP64 also tries 64-thread blocks (its best step shape from 32k particles on)
  const bool fp64 = g->precision == GBMD_FP64;
  auto tried = [&](int tpp, int block, const char* what, float ms) {
    if (getenv("GBMD_VERBOSE")) fprintf(stderr, "gbmd autotune %s tpp=%d block=%d %s %.4f ms\n", key.c_str(), tpp, block, what, ms);
  };
  bool readouts_only = false;   // the best lanes' block size serves readouts alone
  for (int tpp : {1, 2, 4})
    for (int block : {64, 128, 256, 512}) {
      if (block == 64 && !fp64) continue;
      RET(set_tuning(g, tpp, block));
      float ms;
      if (by_steps) RET(time_steps(g, &ms));
      else RET(time_force(g, &ms));
      if (ms < 0.f) continue;
      tried(tpp, block, by_steps ? "step" : "force", ms);
      const bool whole = by_steps && g->team.size() == live(g).size();   // team.size() > 0
      if (ms < best) { best = ms; best_t = tpp; best_b = block; readouts_only = whole; }
      if (whole) break;   // the team's blocks are its own: every block size is the same
    }
  if (readouts_only) {
    best = 1e30f;
    for (int block : {64, 128, 256, 512}) {
      if (block == 64 && !fp64) continue;
      RET(set_tuning(g, best_t, block));
      float ms;
      RET(time_force(g, &ms));
      tried(best_t, block, "force", ms);
      if (ms < best) { best = ms; best_b = block; }
    }
  }
  RET(set_tuning(g, best_t, best_b));
  if (cache) {
    std::ofstream o(cache, std::ios::app);
    o << key << " " << best_t << " " << best_b << " " << best_s << "\n";
  }
  return GBMD_OK;
}

}  // namespace

// ============================================================================
// C ABI
// ============================================================================
extern "C" {

const char* gbmd_last_error(void) { return g_err.c_str(); }

int gbmd_abi_version(void) { return GBMD_ABI_VERSION; }

int gbmd_probe_arith(int32_t kind, int32_t iters, void* stream, double* ops, float* ms) {
  if (!ops || !ms) return fail(GBMD_ERR_BAD_ARG, "NULL output");
  if (kind != GBMD_PROBE_DFMA && kind != GBMD_PROBE_FFMA && kind != GBMD_PROBE_DRCP)
    return fail(GBMD_ERR_BAD_ARG, "unknown probe kind %d", kind);
  if (iters < 1) return fail(GBMD_ERR_BAD_ARG, "iters must be >= 1");
  CK(probe_run(kind, static_cast<cudaStream_t>(stream), iters, ops, ms));
  return GBMD_OK;
}

int gbmd_create(const gbmd_desc* d, gbmd_system** out) {
  Range nvtx_range("gbmd_create");
  RET(create_impl(d, out, false));
  int rc = load_state(*out, d->pos, d->vel, d->type, d->image, false, 0);
  if (rc != GBMD_OK) {
    std::string msg = g_err;
    gbmd_destroy(*out);
    *out = nullptr;
    g_err = msg;
  }
  return rc;
}

int gbmd_create_device(const gbmd_desc* d, gbmd_system** out) {
  Range nvtx_range("gbmd_create_device");
  RET(create_impl(d, out, true));
  int rc = load_state(*out, d->pos, d->vel, d->type, d->image, true, 0);
  if (rc != GBMD_OK) {
    std::string msg = g_err;
    gbmd_destroy(*out);
    *out = nullptr;
    g_err = msg;
  }
  return rc;
}

int gbmd_destroy(gbmd_system* s) {
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  use_device(s->device);
  if (s->batch) {
    Group* b = s->batch;
    for (auto& m : b->members)
      if (m == s) m = nullptr;
    b->layout_dirty = true;
    s->batch = nullptr;
  }
  if (s->own) wait_for(s->device, s->own->stream);
  for (const auto& p : s->allocs) cudaFree(p.first);
  if (s->own) {
    free_group(s->own);
  }
  delete s;
  return GBMD_OK;
}

int gbmd_step(gbmd_system* s, int64_t nsteps) {
  Range nvtx_range("gbmd_step");
  if (!s || nsteps < 0) return fail(GBMD_ERR_BAD_ARG, "bad system or nsteps");
  RET(use_device(s->device));
  if (s->batch) return fail(GBMD_ERR_STATE, "system belongs to a batch; use gbmd_batch_step");
  s->target_step += nsteps;
  return take_steps(s->own, nsteps);
}

int gbmd_sync(gbmd_system* s) {
  Range nvtx_range("gbmd_sync");
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  RET(use_device(s->device));
  return sync_system(s);
}

int gbmd_get_forces(gbmd_system* s, double* out) {
  Range nvtx_range("gbmd_get_forces");
  if (!s || !out) return fail(GBMD_ERR_BAD_ARG, "NULL argument");
  RET(use_device(s->device));
  return export_impl(s, nullptr, nullptr, nullptr, out, nullptr, nullptr);
}

int gbmd_get_thermo(gbmd_system* s, gbmd_thermo* out) {
  Range nvtx_range("gbmd_get_thermo");
  if (!s || !out) return fail(GBMD_ERR_BAD_ARG, "NULL argument");
  RET(use_device(s->device));
  Snapshot snap;
  RET(thermo_impl(s, &snap));
  fill_thermo(s, snap, out);
  return GBMD_OK;
}

int gbmd_get_per_particle(gbmd_system* s, double* energy, double* virial) {
  Range nvtx_range("gbmd_get_per_particle");
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  RET(use_device(s->device));
  if (!s->h.pp_u) {
    RET(sync_system(s));
    const size_t N = (size_t)s->h.n;
    RET(dalloc(s, (void**)&s->h.pp_u, N * 8));
    RET(dalloc(s, (void**)&s->h.pp_w, N * 48));
    RET(dalloc(s, (void**)&s->d_ppu, N * 8));
    RET(dalloc(s, (void**)&s->d_ppw, N * 48));
    RET(refresh_desc(s));
  }
  if (!energy && !virial) return sync_system(s);
  // the energy pass fills the per-particle arrays
  return export_impl(s, nullptr, nullptr, nullptr, nullptr, energy, virial);
}

int gbmd_get_state(gbmd_system* s, double* pos, double* vel, int32_t* image, int64_t* step) {
  Range nvtx_range("gbmd_get_state");
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  RET(use_device(s->device));
  return export_impl(s, pos, vel, image, nullptr, nullptr, nullptr, step);
}

int gbmd_set_state(gbmd_system* s, const double* pos, const double* vel, const int32_t* image,
                   int64_t step) {
  Range nvtx_range("gbmd_set_state");
  if (!s || !pos || !vel || step < 0) return fail(GBMD_ERR_BAD_ARG, "bad argument");
  RET(use_device(s->device));
  if (s->batch) return fail(GBMD_ERR_STATE, "remove the system from its batch first");
  RET(sync_system(s));
  const size_t N = (size_t)s->h.n;
  cudaStream_t st = cur_stream(s);
  Group* g = s->own;
  RET(sync_layout(g));
  // The new state goes to the staging buffers; its finiteness and the current types
  // in tag order are taken there on the device, and nothing of the system is
  // replaced unless every value is finite.
  CK(cudaMemcpyAsync(s->d_pos, pos, N * 24, cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(s->d_vel, vel, N * 24, cudaMemcpyHostToDevice, st));
  if (image) CK(cudaMemcpyAsync(s->d_img, image, N * 12, cudaMemcpyHostToDevice, st));
  CK(cudaMemsetAsync(s->d_misc, 0, 4, st));
  CK(launch(prep_state_call(g->d_desc, g->d_tp, g->ntp, s->d_pos, s->d_vel, s->d_type, s->d_misc),
            st));
  return load_state(s, s->d_pos, s->d_vel, s->d_type, image ? s->d_img : nullptr, true, step, s->d_misc);
}

int gbmd_get_neighbors(gbmd_system* s, int32_t* counts, int32_t* idx, int64_t cap) {
  Range nvtx_range("gbmd_get_neighbors");
  if (!s || !counts || !idx || cap < 1 || cap > (1 << 20)) return fail(GBMD_ERR_BAD_ARG, "bad argument");
  RET(use_device(s->device));
  RET(sync_system(s));
  Group* g = s->own;
  RET(sync_layout(g));
  cudaStream_t st = cur_stream(s);
  const size_t N = (size_t)s->h.n;
  int *dc = nullptr, *di = nullptr, *dflag = s->d_misc;
  CK(cudaMalloc(&dc, N * 4));
  cudaError_t e = cudaMalloc(&di, N * (size_t)cap * 4);
  if (e != cudaSuccess) {
    cudaFree(dc);
    return fail(GBMD_ERR_OOM, "no room for the neighbour readout");
  }
  int too_many = 0;
  int rc = GBMD_OK;
  if (cudaMemsetAsync(dflag, 0, 4, st) != cudaSuccess ||
      launch(nlist_export_call(g->d_desc, g->d_tp, g->ntp, dc, di, (int)cap, dflag), st) != cudaSuccess ||
      cudaMemcpyAsync(counts, dc, N * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaMemcpyAsync(idx, di, N * (size_t)cap * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaMemcpyAsync(&too_many, dflag, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    rc = fail(GBMD_ERR_CUDA, "neighbour readout failed");
  cudaFree(dc);
  cudaFree(di);
  if (rc == GBMD_OK && too_many) rc = fail(GBMD_ERR_BAD_ARG, "some particle has more than cap neighbours");
  return rc;
}

int gbmd_get_info(gbmd_system* s, gbmd_info* out) {
  if (!s || !out) return fail(GBMD_ERR_BAD_ARG, "NULL argument");
  RET(use_device(s->device));
  RET(sync_system(s));
  Flags f;
  RET(read_flags(s, &f, cur_stream(s)));
  Group* g = s->batch ? s->batch : s->own;
  out->n = s->h.n;
  out->precision = s->h.precision;
  out->ntypes = s->h.ntypes;
  for (int a = 0; a < 3; ++a) out->cells[a] = s->h.nc[a];
  out->nlist_capacity = s->h.cap;
  out->threads_per_particle = g->tpp;
  out->force_block = g->fblock;
  out->step = f.step;
  out->n_rebuilds = f.n_rebuilds;
  out->n_sorts = f.n_sorts;
  out->kernel_launches = (int64_t)f.launches;
  out->neighbors_total = (int64_t)f.nb_total;
  out->footprint_bytes = (int64_t)s->footprint;
  out->force_path = s->h.staged ? 1 : 0;
  out->max_window = f.max_window;
  out->cell_scale = s->cell_scale;
  out->nlist = s->h.tree ? GBMD_NLIST_TREE : GBMD_NLIST_CELL;
  out->rebuild_pending = s->h.n_ghost > 0 && f.rebuild_req ? 1 : 0;
  out->n_ghost = s->h.n_ghost;
  return GBMD_OK;
}

int gbmd_set_ghost_positions(gbmd_system* s, const double* pos, int32_t device) {
  if (!s || !pos) return fail(GBMD_ERR_BAD_ARG, "NULL argument");
  if (s->h.n_ghost <= 0) return fail(GBMD_ERR_BAD_ARG, "the system has no ghosts");
  if (s->batch) return fail(GBMD_ERR_STATE, "the system is in a batch");
  RET(use_device(s->device));
  Group* g = s->own;
  RET(sync_layout(g));
  cudaStream_t st = cur_stream(s);
  const double* dp = pos;
  if (!device) {   // staging: the import buffer holds n >= n_ghost rows
    CK(cudaMemcpyAsync(s->d_pos, pos, (size_t)s->h.n_ghost * 24, cudaMemcpyHostToDevice, st));
    dp = s->d_pos;
  }
  CK(launch(ghost_set_call(g->d_desc, s->h.n_ghost, dp), st));
  return GBMD_OK;
}

int gbmd_get_positions(gbmd_system* s, const int32_t* tags, int64_t m, double* out,
                       int32_t device) {
  if (!s || !tags || !out) return fail(GBMD_ERR_BAD_ARG, "NULL argument");
  if (m < 0 || m > s->h.n) return fail(GBMD_ERR_BAD_ARG, "m must be in [0, n]");
  if (!device)
    for (int64_t k = 0; k < m; ++k)
      if (tags[k] < 0 || tags[k] >= s->h.n) return fail(GBMD_ERR_BAD_ARG, "tag %d out of range", tags[k]);
  RET(use_device(s->device));
  RET(sync_system(s));
  if (m == 0) return GBMD_OK;
  Group* g = s->batch ? s->batch : s->own;
  RET(sync_layout(g));
  int idx = 0;   // the system's slot in its group's descriptor array
  for (size_t k = 0; k < g->members.size(); ++k)
    if (g->members[k] == s) idx = (int)k;
  cudaStream_t st = cur_stream(s);
  const int* dt = tags;
  double* dout = out;
  if (!device) {   // staging: the import buffers hold n >= m rows
    CK(cudaMemcpyAsync(s->d_type, tags, (size_t)m * 4, cudaMemcpyHostToDevice, st));
    dt = s->d_type;
    dout = s->d_pos;
  }
  CK(launch(gather_pos_call(g->d_desc + idx, dt, (int)m, dout), st));
  if (!device) CK(cudaMemcpyAsync(out, s->d_pos, (size_t)m * 24, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  return GBMD_OK;
}

int64_t gbmd_footprint_bytes(const gbmd_desc* d) {
  if (!d || d->n < 1 || d->ntypes < 1 || d->ntypes > GBMD_MAX_TYPES)
    return fail(GBMD_ERR_BAD_ARG, "bad description");
  double rmax = 0;
  RET(validate_pairs(d, &rmax));
  for (int a = 0; a < 3; ++a)
    if (!(d->box[a] > 0)) return fail(GBMD_ERR_BAD_ARG, "bad box");
  return (int64_t)footprint_of(d, geometry(d));
}

int gbmd_set_step_limit(gbmd_system* s, int64_t step) {
  if (!s || step < -1) return fail(GBMD_ERR_BAD_ARG, "bad argument");
  RET(use_device(s->device));
  cudaStream_t st = cur_stream(s);
  CK(cudaStreamSynchronize(st));
  Flags f;
  RET(read_flags(s, &f, st));
  f.step_limit = step;
  s->step_limit = step;
  return write_flags(s, &f, st);
}

int gbmd_set_thermostat(gbmd_system* s, double xi, double eta) {
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  if (!s->h.nvt) return fail(GBMD_ERR_BAD_ARG, "not an NVT system");
  if (!std::isfinite(xi) || !std::isfinite(eta)) return fail(GBMD_ERR_BAD_ARG, "non-finite thermostat");
  RET(use_device(s->device));
  RET(sync_system(s));
  cudaStream_t st = cur_stream(s);
  // the state of a completed step, as gbmd_get_thermo reports it: valid where the
  // velocities are full-step ones too (after create / set_state, before stepping)
  Flags f;
  RET(read_flags(s, &f, st));
  if (!f.v_full) return fail(GBMD_ERR_STATE, "set the thermostat after gbmd_set_state, before stepping");
  const double nh[3] = {xi, eta, std::exp(-0.5 * s->h.dt * xi)};
  CK(cudaMemcpyAsync(s->h.nh, nh, sizeof(nh), cudaMemcpyHostToDevice, st));
  CK(cudaStreamSynchronize(st));
  return GBMD_OK;
}

int gbmd_set_cell_scale(gbmd_system* s, double scale) {
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  RET(use_device(s->device));
  return regrid(s, scale);
}

int gbmd_set_force_events(gbmd_system* s, void* ev_begin, void* ev_end) {
  if (!s || (!ev_begin) != (!ev_end)) return fail(GBMD_ERR_BAD_ARG, "bad argument");
  RET(use_device(s->device));
  Group* g = s->batch ? s->batch : s->own;
  cudaEvent_t b = (cudaEvent_t)ev_begin, e = (cudaEvent_t)ev_end;
  const bool had = g->ev_begin != nullptr;
  g->ev_begin = b;
  g->ev_end = e;
  if (had && b) {   // the built graphs get the new events
    for (StepGraphs& q : g->graphs) {
      if (!q.built || !q.ev_begin) continue;
      CK(cudaGraphExecEventRecordNodeSetEvent(q.one, q.ev_begin, b));
      CK(cudaGraphExecEventRecordNodeSetEvent(q.one, q.ev_end, e));
    }
    return GBMD_OK;
  }
  destroy_graphs(g);   // rebuilt with (or without) the records at the next step
  return GBMD_OK;
}

int gbmd_autotune(gbmd_system* s, const char* cache_path) {
  Range nvtx_range("gbmd_autotune");
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  RET(use_device(s->device));
  if (s->batch) return fail(GBMD_ERR_STATE, "system belongs to a batch");
  RET(sync_system(s));
  return autotune_group(s->own, cache_path);
}

int gbmd_set_tuning(gbmd_system* s, int32_t tpp, int32_t block) {
  if (!s) return fail(GBMD_ERR_BAD_ARG, "system is NULL");
  RET(use_device(s->device));
  RET(sync_system(s));
  return set_tuning(s->own, tpp, block);
}

// ---- batches ----

int gbmd_batch_create(int32_t precision, void* stream, int32_t device, gbmd_batch** out) {
  if (!out || (precision != GBMD_FP64 && precision != GBMD_MIXED)) return fail(GBMD_ERR_BAD_ARG, "bad argument");
  int dev = device;
  if (dev < 0) CK(cudaGetDevice(&dev));
  RET(use_device(dev));
  Group* g = new Group();
  g->device = dev;
  g->is_batch = true;
  g->precision = precision;
  g->stream = (cudaStream_t)stream;
  if (const char* ev = getenv("GBMD_NO_GRAPHS")) g->use_graphs = ev[0] != '1';
  *out = reinterpret_cast<gbmd_batch*>(g);
  return GBMD_OK;
}

// A member's own readouts (forces, thermo, state) run on its single-system group;
// they take the batch's tuning, so that (with FP64 sums depending on the lanes per
// particle) a member reads back what a system stepped alone at that tuning does.
static void follow_batch_tuning(Group* b) {
  for (auto* m : live(b)) {
    if (m->own->tpp != b->tpp || m->own->fblock != b->fblock) {
      m->own->tpp = b->tpp;
      m->own->fblock = b->fblock;
      m->own->layout_dirty = true;
    }
  }
}

int gbmd_batch_add(gbmd_batch* bh, gbmd_system* s, int32_t* slot) {
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b || !s || !slot) return fail(GBMD_ERR_BAD_ARG, "NULL argument");
  RET(use_device(reinterpret_cast<Group*>(bh)->device));
  if (s->batch) return fail(GBMD_ERR_STATE, "system already in a batch");
  if (s->h.n_ghost > 0) return fail(GBMD_ERR_BAD_ARG, "a system with ghosts cannot join a batch");
  if (s->h.precision != b->precision) return fail(GBMD_ERR_BAD_ARG, "precision mismatch");
  for (auto* m : live(b)) {
    if (m->h.nvt != s->h.nvt) return fail(GBMD_ERR_BAD_ARG, "a batch holds NVE or NVT systems, not both");
    if (m->h.eval != s->h.eval)
      return fail(GBMD_ERR_BAD_ARG, "a batch holds systems of one pair evaluator (LJ and WCA share one)");
  }
  if (s->device != b->device) return fail(GBMD_ERR_BAD_ARG, "system and batch are on different devices");
  RET(sync_system(s));
  CK(wait_for(b->device, b->stream));
  int k = -1;
  for (size_t i = 0; i < b->members.size(); ++i)
    if (!b->members[i]) { k = (int)i; break; }
  if (k < 0) {
    k = (int)b->members.size();
    b->members.push_back(nullptr);
  }
  b->members[k] = s;
  s->batch = b;
  s->batch_slot = k;
  s->own->stream = b->stream;
  b->layout_dirty = true;
  follow_batch_tuning(b);
  *slot = k;
  return GBMD_OK;
}

int gbmd_batch_remove(gbmd_batch* bh, int32_t slot) {
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b || slot < 0 || slot >= (int)b->members.size() || !b->members[slot])
    return fail(GBMD_ERR_BAD_ARG, "bad slot");
  RET(use_device(reinterpret_cast<Group*>(bh)->device));
  gbmd_system* s = b->members[slot];
  RET(sync_system(s));
  CK(wait_for(b->device, b->stream));
  b->members[slot] = nullptr;
  s->batch = nullptr;
  s->batch_slot = -1;
  s->own->stream = s->stream;
  b->layout_dirty = true;
  return GBMD_OK;
}

int gbmd_batch_step(gbmd_batch* bh, int64_t nsteps) {
  Range nvtx_range("gbmd_batch_step");
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b || nsteps < 0) return fail(GBMD_ERR_BAD_ARG, "bad argument");
  RET(use_device(reinterpret_cast<Group*>(bh)->device));
  for (auto* s : live(b)) s->target_step += nsteps;
  return take_steps(b, nsteps);
}

int gbmd_batch_sync(gbmd_batch* bh) {
  Range nvtx_range("gbmd_batch_sync");
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b) return fail(GBMD_ERR_BAD_ARG, "NULL batch");
  RET(use_device(reinterpret_cast<Group*>(bh)->device));
  CK(wait_for(b->device, b->stream));
  int first = GBMD_OK;
  std::string msg;
  for (auto* s : live(b)) {
    int rc = sync_system(s);
    if (rc != GBMD_OK && first == GBMD_OK) {
      first = rc;
      msg = g_err;
    }
  }
  if (first != GBMD_OK) g_err = msg;
  return first;
}

int gbmd_batch_autotune(gbmd_batch* bh, const char* cache_path) {
  Range nvtx_range("gbmd_batch_autotune");
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b) return fail(GBMD_ERR_BAD_ARG, "NULL batch");
  RET(use_device(reinterpret_cast<Group*>(bh)->device));
  RET(gbmd_batch_sync(bh));
  if (live(b).empty()) return GBMD_OK;
  RET(autotune_group(b, cache_path));
  follow_batch_tuning(b);
  return GBMD_OK;
}

int gbmd_batch_set_tuning(gbmd_batch* bh, int32_t tpp, int32_t block) {
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b) return fail(GBMD_ERR_BAD_ARG, "NULL batch");
  RET(use_device(reinterpret_cast<Group*>(bh)->device));
  RET(gbmd_batch_sync(bh));
  RET(set_tuning(b, tpp, block));
  follow_batch_tuning(b);
  return GBMD_OK;
}

int gbmd_batch_info(gbmd_batch* bh, int32_t* members, int64_t* particles, int64_t* launches) {
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b) return fail(GBMD_ERR_BAD_ARG, "NULL batch");
  RET(use_device(reinterpret_cast<Group*>(bh)->device));
  std::vector<gbmd_system*> m = live(b);
  if (members) *members = (int32_t)m.size();
  if (particles) {
    int64_t np = 0;
    for (auto* s : m) np += s->h.n;
    *particles = np;
  }
  if (launches) {
    *launches = 0;
    for (const Group* g : {b, b->rest}) {   // the members outside the team count apart
      if (!g || !g->d_ctl) continue;
      GroupCtl c{};
      CK(cudaMemcpyAsync(&c, g->d_ctl, sizeof(c), cudaMemcpyDeviceToHost, b->stream));
      CK(wait_for(b->device, b->stream));
      *launches += (int64_t)c.launches;
    }
  }
  return GBMD_OK;
}

int gbmd_batch_destroy(gbmd_batch* bh) {
  Group* b = reinterpret_cast<Group*>(bh);
  if (!b) return fail(GBMD_ERR_BAD_ARG, "NULL batch");
  use_device(b->device);
  wait_for(b->device, b->stream);
  for (auto* s : live(b)) {
    s->batch = nullptr;
    s->batch_slot = -1;
    s->own->stream = s->stream;
  }
  free_group(b);
  return GBMD_OK;
}

}  // extern "C"

// ============================================================================
// Allocation-free thermo readout (gbmd_get_thermo_noalloc)
//
// For callers that may not allocate GPU memory.  The scratch the energy/virial
// kernels need -- per-tile FP64 partial sums and the descriptor copy they read --
// lives in the static device arrays below; host code only ever passes their
// device addresses (looked up once per device with cudaGetSymbolAddress), never
// the symbols themselves.
// ============================================================================
namespace {

// The limit is in tiles of EV_TILE_P particles.  A tree list's wide types (force_tiles) take
// more: each holds at most n / 32 particles, and a wide tile as few as EV_TILE_P / 32 of
// them (one lane a particle), so up to as many tiles again as the whole system for each
// type but the one that is not wide, and a partial one a type
constexpr int kNoallocMaxTiles = GBMD_NOALLOC_MAX_TILES;
constexpr int kNoallocTiles = MAXT * (kNoallocMaxTiles + 2);
constexpr int kNoallocMaxDevices = 64;

static __device__ __align__(256) double g_noalloc_partials[8 * kNoallocTiles];   // 8 MiB
static __device__ __align__(256) SysDev g_noalloc_desc;

struct NoallocAddrs {
  bool ready = false;
  double* partials = nullptr;
  SysDev* desc = nullptr;
};
NoallocAddrs g_noalloc_addrs[kNoallocMaxDevices];
std::mutex g_noalloc_mutex;

// once per device, with that device current
int noalloc_setup(int dev, NoallocAddrs* out) {
  if (dev < 0 || dev >= kNoallocMaxDevices) return fail(GBMD_ERR_BAD_ARG, "device ordinal %d too large", dev);
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  NoallocAddrs& a = g_noalloc_addrs[dev];
  if (!a.ready) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_partials);
    if (e != cudaSuccess) return fail(GBMD_ERR_CUDA, "cudaGetSymbolAddress(partials): %s", cudaGetErrorString(e));
    a.partials = static_cast<double*>(p);
    e = cudaGetSymbolAddress(&p, g_noalloc_desc);
    if (e != cudaSuccess) return fail(GBMD_ERR_CUDA, "cudaGetSymbolAddress(descriptor): %s", cudaGetErrorString(e));
    a.desc = static_cast<SysDev*>(p);
    a.ready = true;
  }
  *out = a;
  return GBMD_OK;
}

}  // namespace

extern "C" int gbmd_get_thermo_noalloc(gbmd_system* s, gbmd_thermo* out) {
  if (!s || !out) return fail(GBMD_ERR_BAD_ARG, "NULL argument");
  RET(use_device(s->device));
  NoallocAddrs addr;
  RET(noalloc_setup(s->device, &addr));
  Group* g = s->own;
  cudaStream_t st = g->stream;
  // finish queued work without any recovery that could allocate
  CK(cudaStreamSynchronize(st));
  Flags f;
  RET(read_flags(s, &f, st));
  if (f.error == DEV_NONFINITE) return fail(GBMD_ERR_NONFINITE, "non-finite state (step %lld)", f.step);
  if (f.error) return fail(GBMD_ERR_STATE, "pending device error %d: call gbmd_sync first", f.error);
  long long want = s->target_step;
  if (s->step_limit >= 0) want = std::min(want, s->step_limit);
  if (f.step < want) return fail(GBMD_ERR_STATE, "steps still owed after a recovery: call gbmd_sync first");
  if (g->layout_dirty) return fail(GBMD_ERR_STATE, "layout changed: call gbmd_sync or gbmd_get_thermo first");
  const int tiles = g->ntb > 0 ? g->ntb : (s->h.n + EV_TILE_P - 1) / EV_TILE_P;
  if (tiles > kNoallocMaxTiles || g->nte + g->ntb > kNoallocTiles)
    return fail(GBMD_ERR_BAD_ARG, "%d energy tiles exceed the allocation-free limit of %d",
                tiles, kNoallocMaxTiles);
  // the system's descriptor, pointed at the static partials (own group: tiles from 0)
  SysDev d = s->h;
  d.tile_first_f = 0;
  d.tile_count_f = g->nte + g->ntb;   // the system alone: one of the two is zero
  d.partials = addr.partials;
  CK(cudaMemcpyAsync(addr.desc, &d, sizeof(SysDev), cudaMemcpyHostToDevice, st));
  if (g->ntf > 0) CK(launch(ev_force_call(g, addr.desc), st));
  if (g->ntb > 0)
    CK(launch(force_staged_call(g->multi, MODE_EV, addr.desc, g->d_tb, g->ntb, g->d_ctl, 0,
                                g->window_cap, StepArgs{}), st));
  CK(launch(thermo_call(addr.desc, g->d_ts, g->nts, g->d_ctl), st));
  Snapshot snap;
  RET(read_snapshot(s, &snap, st));   // waits: `d` is host stack memory
  fill_thermo(s, snap, out);
  return GBMD_OK;
}
