// rsa.cu -- host engine and C ABI (include/rsa.h) of the GB300 RSA library.
//
// One handle = one lattice shape (L, k).  A run is one graph and one device to
// host read: where a sample's hot buffers fit a block's shared memory, one
// launch with a block per sample; else the slices of the deposition, the
// contact graph and the probes of the first-wrap search, every kernel over the
// whole batch (grid.y = sample), with per-sample "done" flags that let
// finished samples drop out.  The graph holds as many rounds and probes as a
// shape normally needs; samples that need more go on in small graphs with a
// read after each.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstddef>
#include <map>
#include <memory>
#include <mutex>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/rsa.h"
#include "rsa_rounds.cuh"
#include "rsa_sample.cuh"
#include "rsa_config.cuh"

using namespace rsak;

namespace {

// An NVTX range for the lifetime of a scope (a no-op unless a profiler that
// collects NVTX ranges is attached).
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
};

thread_local std::string g_err;

int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}

#define CUDA_TRY(call)                                                              \
  do {                                                                              \
    cudaError_t e_ = (call);                                                        \
    if (e_ != cudaSuccess)                                                          \
      return fail(RSA_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));   \
  } while (0)

constexpr size_t ALIGN = 256;
constexpr u32 ROUND_CHECK = 4;   // added rounds per graph and host check (default)
constexpr u32 PROBE_CAP = 96;    // a threshold bisection of 64-bit times, at its worst, and the last window

// The loop counters and, behind them, the work counters.
constexpr size_t READ_BYTES = ALIGN + 4 * WORK_SLOTS * 8;

size_t align_up(size_t v) { return (v + ALIGN - 1) / ALIGN * ALIGN; }

struct Layout {
  size_t region, rstride;                             // shared region of sample 0, bytes per sample
  size_t fine, block, heads, list, flat, act;         // rounds (in the region)
  size_t uf, etime, elink, ehist, win;                // contact graph and search (in the region)
  size_t anch, owner, base, node_key, node_idx, node_pos, rs, st, seeds, counters, work, keys, total;
  size_t bits_bytes;  // per sample, fine + block, zeroed together
  size_t heads_bytes, ehist_bytes;  // per sample
  size_t anch_bytes;
};

struct Geometry {
  bool sites;       // k = 1: one pass, no slices
  RoundCfg rc;
  size_t list_cap;  // listed candidates per sample
  SearchCfg sc;
  SearchCfg ssc;    // the same for a sample in one block (rsa_sample.cuh)
  u32 probes;       // probes that bring the window of a large graph to the last
  Shape hot;        // what of it a block keeps in shared memory (offsets only)
  bool one_block;   // that fits
  bool win128;      // shape of the 128-thread window setting (rsa_set_window_threads)
};

u32 cap_nodes_of(u32 L, u32 k) { return (u32)(((u64)L * L) / k); }
u32 cap_edges_of(u32 L, u32 k) {
  u64 LL = (u64)L * L;
  u64 c = std::min<u64>(2 * LL, 6ull * cap_nodes_of(L, k) + 4ull * L) + 64;
  return (u32)c;
}

u32 log2_floor(u64 v) {
  u32 r = 0;
  while (v >>= 1) ++r;
  return r;
}

// Shapes that accept rsa_set_window_threads(h, 128): 32 < k <= 4096 dividing
// spans of 2048 or 4096 cells.
bool window_shape(u32 L, u32 k) {
  if (L % 32 || k < 32 || k > 4096 || (k <= 32 && (k & (k - 1)) == 0)) return false;
  const u32 P = std::min<u32>(L, 4096), C = P / 256;
  return P % 256 == 0 && C >= 1 && C <= 16 && (C & (C - 1)) == 0 && L % P == 0 && P % k == 0 &&
         k % C == 0 && L / P <= 8 && (P == 4096 || P == 2048);
}

void plan_search(u32 L, u32 k, Geometry& G) {
  const u32 cn = cap_nodes_of(L, k), ce = cap_edges_of(L, k);
  SearchCfg& c = G.sc;
  c.win_cap = std::min(FIN_EDGES, ce);
  c.hashed = cn > 2 * FIN_EDGES;
  c.ids = c.hashed ? 2 * FIN_EDGES : cn;
  // n_c / n_j runs from 0.59 (k = 1) to 0.86 (k = 4096), within 0.04 either
  // way; an edge is there by then with about the square of that chance
  const double f = 0.59 + 0.0225 * std::log2((double)k);
  c.q0 = (u32)(65536 * (f - 0.04) * (f - 0.04));
  c.q1 = std::min(64000u, (u32)(65536 * (f + 0.04) * (f + 0.04)));
  // edges per k-mer of capacity: 2 at k = 1, 1.7 at k = 4, 1 from 32 on
  const double edges = (double)cn * (k == 1 ? 2.0 : k <= 8 ? 1.7 : 1.0) * 0.16 * f;
  G.probes = ce <= c.win_cap ? 0 : 3 + (u32)std::max(0.0, std::ceil(std::log2(edges / c.win_cap)));
  G.ssc = c;
}

// Shared memory of a sample in one block: cover bits, bins and active
// candidates, and the anchor bits if they fit as well.
void plan_hot(u32 L, Geometry& G) {
  const RoundCfg& c = G.rc;
  Shape& h = G.hot;
  h.fine = h.heads = h.act = h.anch = NO_HOT;
  h.hot_bytes = 0;
  G.one_block = !G.sites || L <= 96;
  if (G.sites) return;
  size_t off = 0;
  auto part = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 15) / 16 * 16;
    return (u32)at;
  };
  const size_t room = SMP_MAX - SMP_FIXED - SMP_SCRATCH;
  h.act = part((size_t)2 * c.cap_act * sizeof(Act));
  h.fine = part((size_t)2 * (L + c.nbl) * c.W * 4);
  h.heads = part((size_t)4 * c.nb * c.nb * 4);
  G.one_block = off <= room;
  const size_t before = off;
  h.anch = part((size_t)4 * L * c.WA * 4);
  if (off > room) {
    off = before;
    h.anch = NO_HOT;
  }
  h.hot_bytes = (u32)off;
}

// The search of a sample in one block: as many edges as fit beside the
// union-find words of all k-mers, so that most graphs need no probe at all.
void plan_block_search(u32 L, u32 k, Geometry& G) {
  const size_t cn = cap_nodes_of(L, k), room = SMP_MAX - SMP_FIXED;
  if (!G.one_block || cn * 16 >= room) return;
  SearchCfg w = G.sc;
  w.hashed = 0;
  w.ids = (u32)cn;
  w.win_cap = (u32)std::min<size_t>(cap_edges_of(L, k), (room - cn * 16) / 18 / 8 * 8);
  if (w.win_cap >= G.sc.win_cap) G.ssc = w;
}

Geometry plan(u32 L, u32 k) {
  Geometry G{};
  plan_search(L, k, G);
  G.sites = k == 1;
  G.win128 = window_shape(L, k);
  RoundCfg& c = G.rc;
  const u64 N = 2ull * L * L, D = (u64)k * k + 2 * k;
  const u32 lk = log2_floor(k);
  c.W = (L + k + 31) / 32 + 1;
  c.inv_L = ((1ull << 45) + L - 1) / L;
  c.WA = (L + 2 * k + 31) / 32 + 1;
  // lines per block line: 2^bs + k / 2^bs updates per k-mer, least at sqrt(k)
  c.bs = k < 16 ? 0 : std::max(3u, lk / 2);
  c.nbl = c.bs ? (L + (1u << c.bs) - 1) >> c.bs : 0;
  // bins about 4 sqrt(k) cells wide
  c.b = 2 + lk / 2;
  c.nb = ((L - 1) >> c.b) + 1;
  // Priorities below 2^(64 - a) are listed by the first pass: the fewer, the
  // more candidates are still live afterwards (1.5% at 2^-a = 4 / k).  A smaller
  // share costs more slices: L = 1024, k = 32, 1000 samples take 19.3 ms at
  // a = 3, 20.7 at 4 and 24.1 at 5.
  c.a = std::max(1u, (lk + 2) / 2);
  // the first slice holds two to four candidates per conflict neighbourhood
  // (one to two for short k, where it is a large part of all)
  const u32 ld = log2_floor(D), first = k < 16 ? ld : ld - 1;
  c.lzmax = std::max(c.a, std::min(first, RD_LEVELS - 1));
  c.nlev = c.lzmax - c.a + 1;
  size_t off = 0;
  for (u32 t = 0; t < c.nlev; ++t) {
    // slice 0: every priority with lzmax leading zeros or more; slice t: exactly lzmax - t
    const u32 lz = c.lzmax - t;
    const double mean = std::ldexp((double)N, -(int)(t == 0 ? lz : lz + 1));
    // eight standard deviations of the number of hashes that fall in it
    const u64 cap = std::min<u64>(N, (u64)(mean + 8.0 * std::sqrt(mean) + 64.0));
    c.lvl_off[t] = (u32)off;
    c.lvl_cap[t] = (u32)cap;
    off += cap;
  }
  G.list_cap = off;
  // neither limit is met by random priorities; past one, a round (a refill)
  // takes a narrower slice and the run only takes longer
  c.cap_flat = (u32)std::min<u64>(N, N / 4 + 32);
  c.cap_act = (u32)std::min<u64>(N, std::max(cap_nodes_of(L, k) / 2, c.lvl_cap[0]) + 32);
  plan_hot(L, G);
  plan_block_search(L, k, G);
  return G;
}

Layout layout_of(u32 L, u32 k, u32 n, bool with_keys, const Geometry& G) {
  Layout l{};
  const u64 LL = (u64)L * L;
  const RoundCfg& c = G.rc;
  const size_t cn = cap_nodes_of(L, k), ce = cap_edges_of(L, k);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t at = off;
    off = align_up(off + bytes);
    return at;
  };
  // one region per sample, first for the buffers of its rounds, then for those
  // of its contact graph and search; offsets in it
  size_t ro = 0;
  auto part = [&](size_t bytes) {
    size_t at = ro;
    ro = align_up(ro + bytes);
    return at;
  };
  if (!G.sites) {
    l.bits_bytes = (size_t)2 * (L + c.nbl) * c.W * 4;
    l.fine = part(l.bits_bytes);
    l.block = l.fine + (size_t)2 * L * c.W * 4;
    l.heads_bytes = (size_t)4 * c.nb * c.nb * 4;
    l.heads = part(l.heads_bytes);
    l.list = part(G.list_cap * 4);
    l.flat = part((size_t)c.cap_flat * 4);
    l.act = part((size_t)2 * c.cap_act * sizeof(Act));
  }
  const size_t rounds_end = ro;
  ro = 0;
  l.uf = part(cn * 16);
  l.etime = part(ce * 8);
  l.elink = part(ce * 16);
  // (graphs that a sample in one block starts on whole use it from 1024
  // k-mers on: two good thresholds are worth its 9 KB there)
  l.ehist_bytes = G.probes || cap_edges_of(L, k) > G.ssc.win_cap || cn >= 1024 ? (size_t)SEARCH_WORDS * 4 : 0;
  l.ehist = part(l.ehist_bytes);
  l.win = part(std::max(G.sc.win_cap, G.ssc.win_cap) * sizeof(WinEdge));
  l.rstride = std::max(ro, rounds_end);
  l.region = take(n * l.rstride);
  l.anch_bytes = G.sites ? 0 : (size_t)n * 4 * L * c.WA * 4;
  l.anch = take(l.anch_bytes);
  l.owner = take(G.sites ? 0 : n * LL * 4);  // written at anchors only
  l.base = take((size_t)n * 8);
  l.node_key = take(n * cn * 8);
  l.node_idx = take(n * cn * 4);
  l.node_pos = take(n * cn * 4);
  l.rs = take(G.sites ? 0 : (size_t)n * sizeof(RoundState));
  l.st = take((size_t)n * sizeof(SampleState));
  l.seeds = take((size_t)n * 8);
  // loop counters, work counters, key bins of the configuration passes: zeroed
  // together
  l.counters = take(READ_BYTES + CFG_BINS * 4);
  l.work = l.counters + ALIGN;
  l.keys = take(with_keys ? 2 * LL * 8 : 0);
  l.total = off;
  return l;
}

}  // namespace

// For the other translation unit of the library (rsa_mix.cu): the thread's
// error message, and what it needs of rsa_run_small.
namespace rsa_detail {
int set_error(int code, const std::string& msg) { return fail(code, msg); }
bool small_eligible(uint32_t L, uint32_t k);
unsigned long long take_small_launches();
void release_small();
}  // namespace rsa_detail

enum Kind {
  KD_INIT, KD_DENSE, KD_PICK, KD_RESOLVE, KD_REFILL, KD_CHECK, KD_SITES, KD_EDGES,
  KD_SEARCH_INIT, KD_PROBE_COPY, KD_PROBE, KD_COLLECT, KD_FINISH, KD_RANK, KD_SAMPLE, KD_COUNT
};
const char* const kKindNames[KD_COUNT] = {
    "k_init", "k_dense", "k_pick", "k_resolve", "k_refill", "k_round_check", "k_sites", "k_edges",
    "k_search_init", "k_probe_copy", "k_probe", "k_collect", "k_finish", "k_rank",
    "k_sample"};

// Optional per-kernel timing with CUDA events recorded around each launch
// on the launch stream, plus launch counts (always kept).
struct Prof {
  bool on = false;
  std::vector<cudaEvent_t> pool;
  std::vector<int> kinds;  // kind of record i uses events 2i, 2i+1
  unsigned long long launches[KD_COUNT] = {};
  double ms[KD_COUNT] = {};
};

struct rsa {
  u32 L, k;
  u64 seed;
  Geometry geo;
  // device memory owned by the library
  void* own_ptr = nullptr;
  size_t own_bytes = 0;
  // caller-bound workspace
  void* bound_ptr = nullptr;
  size_t bound_bytes = 0;
  // last run
  void* ws = nullptr;
  Layout lay{};
  u32 last_n = 0;
  // sample states of the last run, once read (fetch_states): readers on several
  // threads share them
  std::mutex states_mu;
  std::shared_ptr<const std::vector<SampleState>> states;
  bool with_keys = false;
  cudaStream_t stream = nullptr;
  u32* h_counter = nullptr;  // pinned, READ_BYTES: loop and work counters, configuration bits
  unsigned long long work[4] = {0, 0, 0, 0};  // accumulated round-pass work
  int device = -1;
  int sm_count = 0;
  Prof prof;
  // CUDA graphs of a whole run, of added rounds, of the search after them and of
  // added probes, captured once per (workspace, batch size, key source, caps) on
  // a private stream and replayed on the run's stream
  bool use_graphs = true;
  cudaStream_t cap_stream = nullptr;
  // rounds after the last slice in the run's first graph: more once a run
  // has needed more
  u32 drain = 3;
  u32 round_check = ROUND_CHECK;  // added rounds per graph and host check
  // test-only lowered caps of the device loops (0 = default; rsa_test_caps)
  u32 t_round = 0, t_uf = 0, t_probe = 0, t_edges = 0;
  struct GraphSlot {
    cudaGraphExec_t exec = nullptr;
    const void* ws = nullptr;
    u32 n = 0;
    bool keys = false;
    u32 caps[6] = {0, 0, 0, 0, 0, 0};  // caps, rounds per chunk and after the last slice
    unsigned long long launches[32] = {};
  } g_main, g_round, g_search, g_probe;
};

namespace {

int ensure_workspace(rsa_t* h, u32 n, bool with_keys) {
  Layout l = layout_of(h->L, h->k, n, with_keys, h->geo);
  if (h->bound_ptr) {
    if (l.total > h->bound_bytes)
      return fail(RSA_ENOMEM, "bound workspace too small: need " + std::to_string(l.total) +
                                  " bytes, have " + std::to_string(h->bound_bytes));
    h->ws = h->bound_ptr;
  } else {
    if (l.total > h->own_bytes) {
      if (h->own_ptr) cudaFree(h->own_ptr);
      h->own_ptr = nullptr;
      h->own_bytes = 0;
      cudaError_t e = cudaMalloc(&h->own_ptr, l.total);
      if (e != cudaSuccess) {
        cudaGetLastError();
        h->own_ptr = nullptr;
        return fail(RSA_ENOMEM, "cudaMalloc(" + std::to_string(l.total) +
                                    ") failed: " + cudaGetErrorString(e));
      }
      h->own_bytes = l.total;
    }
    h->ws = h->own_ptr;
  }
  h->lay = l;
  return 0;
}

Group group_of(rsa_t* h, u32 n) {
  char* b = static_cast<char*>(h->ws);
  const Layout& l = h->lay;
  Group g{};
  g.L = h->L;
  g.k = h->k;
  g.n = n;
  g.cap_nodes = cap_nodes_of(h->L, h->k);
  g.cap_edges = cap_edges_of(h->L, h->k);
  g.uf_cap = h->t_uf ? h->t_uf : UF_CAP;
  g.edge_limit = h->t_edges ? std::min(h->t_edges, g.cap_edges) : g.cap_edges;
  g.LL = (u64)h->L * h->L;
  g.owner = reinterpret_cast<u32*>(b + l.owner);
  g.base = reinterpret_cast<u64*>(b + l.base);
  g.keys = h->with_keys ? reinterpret_cast<const u64*>(b + l.keys) : nullptr;
  g.node_key = reinterpret_cast<u64*>(b + l.node_key);
  g.node_idx = reinterpret_cast<u32*>(b + l.node_idx);
  g.node_pos = reinterpret_cast<u32*>(b + l.node_pos);
  char* r = b + l.region;
  g.rstride = l.rstride;
  g.uf = reinterpret_cast<u64*>(r + l.uf);
  g.etime = reinterpret_cast<u64*>(r + l.etime);
  g.elink = reinterpret_cast<uint4*>(r + l.elink);
  g.ehist = l.ehist_bytes ? reinterpret_cast<u32*>(r + l.ehist) : nullptr;
  g.win = reinterpret_cast<WinEdge*>(r + l.win);
  g.st = reinterpret_cast<SampleState*>(b + l.st);
  g.work = reinterpret_cast<u64*>(b + l.work);
  return g;
}

RoundPtrs round_ptrs(rsa_t* h) {
  char* b = static_cast<char*>(h->ws);
  const Layout& l = h->lay;
  char* r = b + l.region;
  RoundPtrs p{};
  p.fine = reinterpret_cast<u32*>(r + l.fine);
  p.block = reinterpret_cast<u32*>(r + l.block);
  p.anch = reinterpret_cast<u32*>(b + l.anch);
  p.list = reinterpret_cast<u32*>(r + l.list);
  p.flat = reinterpret_cast<u32*>(r + l.flat);
  p.act = reinterpret_cast<Act*>(r + l.act);
  p.heads = reinterpret_cast<u32*>(r + l.heads);
  p.rs = reinterpret_cast<RoundState*>(b + l.rs);
  return p;
}

cudaEvent_t prof_event(Prof& p, size_t i) {
  while (p.pool.size() <= i) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    p.pool.push_back(e);
  }
  return p.pool[i];
}

// Launch wrapper: counts launches and, when profiling is on, brackets the
// launch with two events on its stream.
cudaEvent_t prof_begin(Prof& p, int kind, cudaStream_t st) {
  if (!p.on) return nullptr;
  const size_t i = p.kinds.size();
  cudaEvent_t e0 = prof_event(p, 2 * i), e1 = prof_event(p, 2 * i + 1);
  if (!e0 || !e1) return nullptr;
  cudaEventRecord(e0, st);
  p.kinds.push_back(kind);
  return e1;
}

template <typename... KArgs, typename... Args>
void launch(rsa_t* h, int kind, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
            Args... args) {
  Prof& p = h->prof;
  cudaEvent_t e1 = prof_begin(p, kind, st);
  kernel<<<grid, block, smem, st>>>(args...);
  if (e1) cudaEventRecord(e1, st);
  p.launches[kind] += 1;
}

// The shape of the one-block kernels.
Shape shape_of(const Geometry& G, const Group& g, const RoundCfg& c, const RoundPtrs& p,
               u32 probe_cap) {
  Shape s = G.hot;
  s.g = g;
  s.c = c;
  s.p = p;
  s.sc = G.ssc;
  s.probe_cap = probe_cap;
  s.sites = G.sites;
  return s;
}

int launch_check(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(RSA_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
  return 0;
}

int read_counters(rsa_t* h, u32* active, u32* open) {
  const char* from = static_cast<const char*>(h->ws) + h->lay.counters;
  CUDA_TRY(cudaMemcpyAsync(h->h_counter, from, READ_BYTES, cudaMemcpyDeviceToHost, h->stream));
  CUDA_TRY(cudaStreamSynchronize(h->stream));
  *active = h->h_counter[0];
  *open = h->h_counter[1];
  return 0;
}

void drop_graph(rsa_t::GraphSlot& gs) {
  if (gs.exec) cudaGraphExecDestroy(gs.exec);
  gs.exec = nullptr;
  gs.ws = nullptr;
}

// Run `body(stream)` once, either directly or through a captured graph.
template <typename B>
int run_chunk(rsa_t* h, rsa_t::GraphSlot& gs, cudaStream_t stream, u32 n, B body) {
  if (!h->use_graphs || h->prof.on) {
    body(stream);
    return launch_check("chunk launches");
  }
  const u32 caps[6] = {h->t_round, h->t_uf, h->t_probe, h->t_edges, h->round_check, h->drain};
  if (!(gs.exec && gs.ws == h->ws && gs.n == n && gs.keys == h->with_keys &&
        std::memcmp(gs.caps, caps, sizeof(caps)) == 0)) {
    drop_graph(gs);
    if (!h->cap_stream)
      CUDA_TRY(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    unsigned long long before[KD_COUNT];
    std::memcpy(before, h->prof.launches, sizeof(before));
    CUDA_TRY(cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
    body(h->cap_stream);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(h->cap_stream, &graph);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return fail(RSA_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
    }
    e = cudaGraphInstantiate(&gs.exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
      gs.exec = nullptr;
      return fail(RSA_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
    }
    for (int i = 0; i < KD_COUNT; ++i) {
      gs.launches[i] = h->prof.launches[i] - before[i];
      h->prof.launches[i] = before[i];
    }
    gs.ws = h->ws;
    gs.n = n;
    gs.keys = h->with_keys;
    std::memcpy(gs.caps, caps, sizeof(caps));
  }
  CUDA_TRY(cudaGraphLaunch(gs.exec, stream));
  for (int i = 0; i < KD_COUNT; ++i) h->prof.launches[i] += gs.launches[i];
  return 0;
}

int run_impl(rsa_t* h, const uint64_t* seeds, u32 n, const uint64_t* keys, cudaStream_t stream) {
  if (n == 0) return fail(RSA_EINVAL, "n_samples must be >= 1");
  NvtxRange run_range("rsa_run");
  int rc;
  CUDA_TRY(cudaGetDevice(&h->device));
  if (!h->h_counter) CUDA_TRY(cudaMallocHost(&h->h_counter, READ_BYTES));
  h->with_keys = keys != nullptr;
  if ((rc = ensure_workspace(h, n, h->with_keys))) return rc;
  h->stream = stream;
  h->last_n = n;
  {
    std::lock_guard<std::mutex> lock(h->states_mu);
    h->states.reset();
  }
  Group g = group_of(h, n);
  const Geometry& G = h->geo;
  const Layout& l = h->lay;
  char* b = static_cast<char*>(h->ws);
  u64* d_seeds = reinterpret_cast<u64*>(b + l.seeds);
  u32* d_counter = reinterpret_cast<u32*>(b + l.counters);
  const u64 LL = g.LL;

  CUDA_TRY(cudaMemcpyAsync(d_seeds, seeds, (size_t)n * 8, cudaMemcpyHostToDevice, stream));
  if (keys)
    CUDA_TRY(cudaMemcpyAsync(b + l.keys, keys, 2 * LL * 8, cudaMemcpyHostToDevice, stream));
  if (!h->sm_count)
    CUDA_TRY(cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device));
  RoundCfg c = G.rc;
  // every round with an active candidate accepts the smallest of them, so
  // n_j + 1 rounds always suffice
  c.round_cap = h->t_round ? h->t_round : cap_nodes_of(h->L, h->k) + 2;
  const u32 probe_cap = h->t_probe ? h->t_probe : PROBE_CAP;
  const RoundPtrs rp = round_ptrs(h);
  int body_rc = 0;
  auto check = [&](cudaError_t e) {
    if (e != cudaSuccess) body_rc = RSA_ECUDA;
  };
  // blocks per sample: what the work of a sample fills, at most `waves`
  // blocks per SM over the batch
  auto grid_x = [&](u64 blocks, u32 waves) {
    const u64 most = std::max<u64>(1, ((u64)h->sm_count * waves + n - 1) / n);
    return dim3((unsigned)std::max<u64>(1, std::min(blocks, most)), n);
  };
  const dim3 init_grid((n + 127) / 128);
  // Lanes per active candidate in k_resolve.  Long k has many bins to look at
  // (L = 8192, k = 512, 32 samples: the run takes 14.6 ms with 16 lanes, 15.8
  // with 8, 15.1 with 32; L = 32768, k = 4096: 20.5 and 20.2 with 16 and 32).
  // For short k one lane does the least work in all, which counts once the
  // candidates fill the GPU (L = 1024, k = 32, 1000 samples: 19.8 ms, with 8
  // lanes 24.1), and eight lanes have the shortest chain of loads, which
  // counts when they do not (L = 128, k = 8, 32 samples: 0.18 ms of k_resolve
  // against 0.49).
  const u32 lanes = h->k >= 2048                             ? 32
                    : h->k > 128                             ? 16
                    : (u64)n * g.cap_nodes >= (2u << 20) ? 1
                                                             : 8;
  auto round = [&](cudaStream_t st) {
    const dim3 pg = grid_x((c.lvl_cap[c.nlev - 1] + RD_THREADS - 1) / RD_THREADS, 16);
    if (h->k <= PICK_LONGK)
      launch(h, KD_PICK, k_pick<false>, pg, dim3(RD_THREADS), 0, st, g, c, rp);
    else
      launch(h, KD_PICK, k_pick<true>, pg, dim3(RD_THREADS), 0, st, g, c, rp);
    const dim3 rg = grid_x(((u64)(g.cap_nodes / 4 + 1) * lanes + RD_THREADS - 1) / RD_THREADS, 16);
    switch (lanes) {
      case 1: launch(h, KD_RESOLVE, k_resolve<1>, rg, dim3(RD_THREADS), 0, st, g, c, rp); break;
      case 8: launch(h, KD_RESOLVE, k_resolve<8>, rg, dim3(RD_THREADS), 0, st, g, c, rp); break;
      case 16: launch(h, KD_RESOLVE, k_resolve<16>, rg, dim3(RD_THREADS), 0, st, g, c, rp); break;
      default: launch(h, KD_RESOLVE, k_resolve<32>, rg, dim3(RD_THREADS), 0, st, g, c, rp); break;
    }
  };
  auto refill = [&](cudaStream_t st) {
    const u32 warps = std::min(RD_THREADS / 32, REFILL_WORDS / c.W);
    launch(h, KD_REFILL, k_refill, grid_x((2ull * h->L + warps - 1) / warps, 16), dim3(RD_THREADS),
           0, st, g, c, rp);
  };
  auto count_active = [&](cudaStream_t st) {
    check(cudaMemsetAsync(d_counter, 0, 4, st));
    launch(h, KD_CHECK, k_round_check, init_grid, dim3(128), 0, st, g, d_counter);
  };
  // the whole deposition: every slice once, and three more rounds for the
  // candidates left undecided by the last ones
  auto deposit = [&](cudaStream_t st) {
    check(cudaMemsetAsync(b + l.counters, 0, READ_BYTES + CFG_BINS * 4, st));
    launch(h, KD_INIT, k_init, init_grid, dim3(128), 0, st, g, (const u64*)d_seeds);
    if (G.sites) {
      launch(h, KD_SITES, k_sites, grid_x((LL + 255) / 256, 32), dim3(256), 0, st, g);
      return;
    }
    check(cudaMemset2DAsync(b + l.region + l.fine, l.rstride, 0, l.bits_bytes, n, st));
    check(cudaMemsetAsync(b + l.anch, 0, l.anch_bytes, st));
    check(cudaMemset2DAsync(b + l.region + l.heads, l.rstride, 0xFF, l.heads_bytes, n, st));
    launch(h, KD_INIT, k_round_init, init_grid, dim3(128), 0, st, g, c, rp);
    const u64 dense_tile = DENSE_THREADS * DENSE_PER;
    const dim3 dg = grid_x((2 * LL + dense_tile - 1) / dense_tile, 16);
    if (h->with_keys)
      launch(h, KD_DENSE, k_dense<true>, dg, dim3(DENSE_THREADS), 0, st, g, c, rp);
    else
      launch(h, KD_DENSE, k_dense<false>, dg, dim3(DENSE_THREADS), 0, st, g, c, rp);
    for (u32 t = 0; t < c.nlev; ++t) round(st);
    refill(st);
    for (u32 t = c.nlev; t <= c.lzmax + h->drain; ++t) round(st);
    count_active(st);
  };
  // a sample that is not through yet: more rounds
  auto more_rounds = [&](cudaStream_t st) {
    refill(st);
    for (u32 i = 0; i < h->round_check; ++i) round(st);
    count_active(st);
  };
  const SearchCfg& sc = G.sc;
  // blocks per sample over its k-mers and its edges
  const dim3 node_grid = grid_x(((u64)g.cap_nodes + 255) / 256, 32);
  const dim3 edge_grid = grid_x(((u64)g.cap_edges + 255) / 256, 16);
  const size_t fin_smem = finish_smem(sc);
  // the same limit for every shape: handles run on several threads at once
  CUDA_TRY(cudaFuncSetAttribute(k_finish, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)FIN_SMEM_MAX));
  auto probes = [&](cudaStream_t st) {
    check(cudaMemsetAsync(d_counter + 1, 0, 4, st));
    for (u32 i = 0; i < G.probes; ++i) {
      launch(h, KD_PROBE_COPY, k_probe_copy, node_grid, dim3(256), 0, st, g);
      launch(h, KD_PROBE, k_probe, edge_grid, dim3(256), 0, st, g, sc, probe_cap);
    }
    launch(h, KD_COLLECT, k_collect, edge_grid, dim3(256), 0, st, g, sc);
    launch(h, KD_FINISH, k_finish, dim3(n), dim3(FIN_THREADS), fin_smem, st, g, sc, probe_cap,
           d_counter + 1);
    launch(h, KD_RANK, k_rank, node_grid, dim3(256), 0, st, g);
  };
  // contact graph of the jammed lattice and the search for the first wrap
  auto search = [&](cudaStream_t st) {
    launch(h, KD_SEARCH_INIT, k_graph_init, dim3(n), dim3(256), 0, st, g, (const u32*)d_counter);
    if (G.sites) {
      launch(h, KD_EDGES, k_site_contacts, grid_x((LL + 255) / 256, 32), dim3(256), 0, st, g);
    } else {
      // lanes per k-mer: 1 for lines of a few words (L = 1024, k = 32, 1000
      // samples: 2.0 ms, with 4 lanes 2.8), 4 for longer ones (L = 32768,
      // k = 4096, 4 samples: 1.2 ms, with 1 lane 1.8, with 32 lanes 2.7)
      const u32 el = h->k <= 64 ? 1 : 4;
      const dim3 eg = grid_x(((u64)g.cap_nodes * el + 255) / 256, 32);
      if (el == 1)
        launch(h, KD_EDGES, k_contacts<1>, eg, dim3(256), 0, st, g, c, rp);
      else
        launch(h, KD_EDGES, k_contacts<4>, eg, dim3(256), 0, st, g, c, rp);
    }
    launch(h, KD_SEARCH_INIT, k_search_init, dim3(n), dim3(256), 0, st, g, sc);
    probes(st);
  };
  // One block per sample for the small lattices, and for those that still fit
  // a block when there are enough samples to fill half of the GPU with blocks.
  // ms in one block / over the grid:
  //   4 samples    L = 160, k = 10  0.260 / 0.264, L = 192, k = 12  0.300 / 0.267
  //   76 samples   L = 256, k = 16  0.39 / 0.53, L = 512, k = 64  0.72 / 0.74
  //   152 samples  L = 256, k = 16  0.40 / 0.75, L = 512, k = 64  0.73 / 1.04
  //   400 samples  L = 256, k = 16  1.05 / 1.42, L = 512, k = 64  2.02 / 2.12
  // Of 43 such batches (L = 170 .. 512) five are slower in one block, the worst of
  // them L = 400, k = 100, 400 samples, 1.72 / 1.32 (a third wave of blocks).  Runs without
  // graphs pay for every launch on the host and take one block wherever it fits:
  // 4 samples L = 256, k = 16  0.40 / 0.42, L = 320, k = 320  0.33 / 0.50; the
  // grid would be better from L = 320 on for short k (L = 512, k = 64  0.68 / 0.50).
  const bool by_sample =
      G.one_block && (h->L <= 160 || n >= (u32)h->sm_count / 2 || !h->use_graphs);
  const Shape shape = shape_of(G, g, c, rp, probe_cap);
  CUDA_TRY(cudaFuncSetAttribute(k_sample, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMP_MAX));
  auto whole = [&](cudaStream_t st) {
    if (by_sample) {
      check(cudaMemsetAsync(b + l.counters, 0, READ_BYTES + CFG_BINS * 4, st));
      launch(h, KD_SAMPLE, k_sample, dim3(std::min(n, (u32)h->sm_count)), dim3(SMP_THREADS),
             sample_smem(shape), st, shape, (const u64*)d_seeds);
      return;
    }
    deposit(st);
    search(st);
  };
  u32 active = 0, open = 0;
  if ((rc = run_chunk(h, h->g_main, stream, n, whole))) return rc;
  if (body_rc) return fail(body_rc, "launches failed");
  if ((rc = read_counters(h, &active, &open))) return rc;
  if (active) {
    // the search of the first graph was left out
    NvtxRange rounds_range("more rounds");
    if (h->drain < 16) h->drain += 2;
    while (active) {
      if ((rc = run_chunk(h, h->g_round, stream, n, more_rounds))) return rc;
      if (body_rc) return fail(body_rc, "round launches failed");
      if ((rc = read_counters(h, &active, &open))) return rc;
    }
    if ((rc = run_chunk(h, h->g_search, stream, n, search))) return rc;
    if (body_rc) return fail(body_rc, "search launches failed");
    if ((rc = read_counters(h, &active, &open))) return rc;
  }
  while (open) {
    NvtxRange wrap_range("more probes");
    if ((rc = run_chunk(h, h->g_probe, stream, n, probes))) return rc;
    if (body_rc) return fail(body_rc, "probe launches failed");
    if ((rc = read_counters(h, &active, &open))) return rc;
  }
  // round-pass work counters of this run (for throughput accounting)
  const unsigned long long* wk =
      reinterpret_cast<const unsigned long long*>(reinterpret_cast<const char*>(h->h_counter) + ALIGN);
  for (u32 i = 0; i < 4 * WORK_SLOTS; ++i) h->work[i / WORK_SLOTS] += wk[i];
  return 0;
}

int status_code(u32 bits) {
  if (bits & ST_NOWRAP) return RSA_ENOWRAP;
  if (bits & (ST_UF_CAP | ST_SEARCH_CAP | ST_ROUND_CAP)) return RSA_ETIMEOUT;
  if (bits & (ST_NODE_OVF | ST_EDGE_OVF)) return RSA_ENOMEM;
  return 0;
}

typedef std::shared_ptr<const std::vector<SampleState>> States;

// The sample states of the last run, read from the device once per run.  A
// reader keeps the ones it was given while it walks over them.
int fetch_states(rsa_t* h, States* out) {
  if (!h->ws || h->last_n == 0) return fail(RSA_ESTATE, "no run to read");
  std::lock_guard<std::mutex> lock(h->states_mu);
  if (!h->states) {
    auto v = std::make_shared<std::vector<SampleState>>(h->last_n);
    const char* b = static_cast<const char*>(h->ws);
    CUDA_TRY(cudaMemcpyAsync(v->data(), b + h->lay.st, sizeof(SampleState) * h->last_n,
                             cudaMemcpyDeviceToHost, h->stream));
    CUDA_TRY(cudaStreamSynchronize(h->stream));
    h->states = std::move(v);
  }
  *out = h->states;
  return 0;
}

// ---------------------------------------------------------------------
// Workspace-free runs.  Some callers cannot call cudaMalloc: a process whose
// device memory pool is owned by another allocator (a framework's caching
// allocator that has reserved the whole HBM), or a latency-critical serving
// loop that must not hit the device-wide synchronisation cudaMalloc and
// cudaFree can cause.  rsa_run_static serves them from this fixed array,
// which every GPU that loads the library holds until the process exits.
// ---------------------------------------------------------------------
constexpr size_t STATIC_WS_BYTES = 64ull << 20;  // 64 MiB
static __device__ __align__(256) unsigned char g_static_ws[STATIC_WS_BYTES];

constexpr int MAX_DEVICES = 64;
std::mutex g_static_mu;
void* g_static_ptr[MAX_DEVICES] = {};
unsigned long long g_static_ctx[MAX_DEVICES] = {};

// Unique id of the current CUDA context (cuCtxGetId, reached through the
// runtime's driver entry-point table so the library does not link libcuda),
// or 0 if there is none or the driver lacks the call.
unsigned long long current_context_id() {
  typedef int (*ctx_id_fn)(void*, unsigned long long*);
  static ctx_id_fn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    cudaGetLastError();
    return reinterpret_cast<ctx_id_fn>(f);
  }();
  unsigned long long id = 0;
  if (!fn || fn(nullptr, &id) != 0) return 0;
  return id;
}

// Device address of g_static_ws on the current device, looked up once per
// device (with that device current) and again whenever that device's context
// has changed since (a context destroyed by cudaDeviceReset and created anew
// may place the array elsewhere).  In host code the symbol itself is only a
// host-side stand-in, never a device address.
int static_workspace(void** out) {
  int dev = -1;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= MAX_DEVICES) return fail(RSA_EINVAL, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_static_mu);
  const unsigned long long ctx = current_context_id();
  if (!g_static_ptr[dev] || ctx == 0 || ctx != g_static_ctx[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_ws);
    if (e != cudaSuccess || !p)
      return fail(RSA_ECUDA, std::string("cudaGetSymbolAddress(static workspace): ") +
                                 cudaGetErrorString(e));
    g_static_ptr[dev] = p;
    g_static_ctx[dev] = current_context_id();  // the lookup made the context current
  }
  *out = g_static_ptr[dev];
  return 0;
}

// The configuration of the first m accepted k-mers of sample `sample` of
// the last run: winding bits into *wdirs, and, if counts is given, the
// cluster-size histogram counts[0 .. m] (cap >= m + 1).
int configuration(rsa_t* h, uint32_t sample, uint32_t m, uint32_t* counts, uint32_t cap,
                  uint32_t* wdirs) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  if (sample >= h->last_n) return fail(RSA_EINVAL, "sample out of range");
  if (counts && cap < (u64)m + 1) return fail(RSA_EINVAL, "counts needs m + 1 entries");
  States states;
  int rc = fetch_states(h, &states);
  if (rc) return rc;
  const std::vector<SampleState>& st = *states;
  if ((rc = status_code(st[sample].status))) {
    g_err = "sample " + std::to_string(sample) + " has no valid result";
    return rc;
  }
  const u32 nj = st[sample].n_nodes;
  if (m > nj) return fail(RSA_EINVAL, "m exceeds n_j of the sample");
  if (counts) std::memset(counts, 0, (size_t)cap * sizeof(uint32_t));
  *wdirs = 0;
  if (m == 0) return 0;
  cudaStream_t stream = h->stream;
  Group g = group_of(h, h->last_n);
  const u32 bx = (u32)std::min<u64>(((u64)st[sample].n_edges + 255) / 256 + 1, 2048);
  const u32 nb = (u32)std::min<u64>(((u64)nj + 256) / 256, 1024);
  const bool at_wrap = m == st[sample].nc;
  const char* b = static_cast<const char*>(h->ws);
  if (g.cap_nodes <= CFG_NODES && st[sample].n_edges <= CFG_EDGES) {
    const size_t smem = cfg_block_smem(g.cap_nodes);
    CUDA_TRY(cudaFuncSetAttribute(k_cfg_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)cfg_block_smem(CFG_NODES)));
    k_cfg_block<<<1, CFG_THREADS, smem, stream>>>(g, sample, m, at_wrap, counts != nullptr);
    CUDA_TRY(cudaGetLastError());
    u32* to = counts ? counts : h->h_counter + 12;
    CUDA_TRY(cudaMemcpyAsync(to, cfg_size(g, sample), (counts ? (size_t)m + 1 : 1) * sizeof(u32),
                             cudaMemcpyDeviceToHost, stream));
    CUDA_TRY(cudaStreamSynchronize(stream));
    h->h_counter[12] = to[0];
    if (counts) counts[0] = 0;
  } else {
    if (!at_wrap) {
      u32* bins = reinterpret_cast<u32*>(const_cast<char*>(b) + h->lay.counters + READ_BYTES);
      const u32 kb = std::min(nb, 152u);
      k_key_bins<<<kb, 256, 0, stream>>>(g, sample, m, bins);
      k_key_select<<<kb, SEL_THREADS, 0, stream>>>(g, sample, bins);
    }
    k_cfg_init<<<nb, 256, 0, stream>>>(g, sample, at_wrap);
    k_cfg_union<<<bx, 256, 0, stream>>>(g, sample);
    if (counts) {
      k_cfg_count<<<nb, 256, 0, stream>>>(g, sample);
      k_cfg_hist<<<nb, 256, 0, stream>>>(g, sample);
    }
    CUDA_TRY(cudaGetLastError());
    const size_t so = h->lay.st + (size_t)sample * sizeof(SampleState);
    CUDA_TRY(cudaMemcpyAsync(h->h_counter + 12, b + so + offsetof(SampleState, wdirs), 4,
                             cudaMemcpyDeviceToHost, stream));
    if (counts)
      CUDA_TRY(cudaMemcpyAsync(counts + 1, cfg_hist(g, sample), (size_t)m * sizeof(uint32_t),
                               cudaMemcpyDeviceToHost, stream));
    CUDA_TRY(cudaStreamSynchronize(stream));
  }
  const u32 w = h->h_counter[12];
  if (w & CFG_CAPPED) return fail(RSA_ETIMEOUT, "union-find walk cap reached");
  *wdirs = w & 3u;
  return 0;
}

// ---------------------------------------------------------------------
// Small lattices of any mix of shapes (rsa_run_small).  Every block has a
// workspace slot of the largest shape's size.  The slots come stream-ordered
// from a memory pool of the library's own, which keeps up to SMALL_POOL_KEEP
// bytes between calls (a serving loop calls this often) and gives them back
// in rsa_mix_release.
// ---------------------------------------------------------------------
constexpr u64 SMALL_LMAX = 128, SMALL_NMAX = 4096;
constexpr unsigned long long SMALL_POOL_KEEP = 512ull << 20;
std::atomic<unsigned long long> g_small_launches{0};
// By device and context: the pool of a context that cudaDeviceReset has
// destroyed is gone with it, and its handle is never used again.
std::mutex g_pool_mu;
std::map<std::pair<int, unsigned long long>, cudaMemPool_t> g_pools;

int small_pool(int dev, cudaMemPool_t* out) {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  unsigned long long ctx = current_context_id();
  if (!ctx) {
    CUDA_TRY(cudaSetDevice(dev));  // makes the device's context current
    ctx = current_context_id();
  }
  if (!ctx) {  // no ids to tell contexts apart: the device's own pool
    CUDA_TRY(cudaDeviceGetDefaultMemPool(out, dev));
    return 0;
  }
  cudaMemPool_t& pool = g_pools[{dev, ctx}];
  if (!pool) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t made = nullptr;
    CUDA_TRY(cudaMemPoolCreate(&made, &props));
    unsigned long long keep = SMALL_POOL_KEEP;
    cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep);
    pool = made;
  }
  *out = pool;
  return 0;
}

// A shape with the pointers of a workspace of one sample that starts at 0.
Shape slot_shape(uint32_t L, uint32_t k, size_t* bytes) {
  rsa h;
  h.L = L;
  h.k = k;
  h.geo = plan(L, k);
  h.lay = layout_of(L, k, 1, false, h.geo);
  h.ws = nullptr;
  *bytes = h.lay.total;
  Group g = group_of(&h, 1);
  RoundCfg c = h.geo.rc;
  c.round_cap = cap_nodes_of(L, k) + 2;
  return shape_of(h.geo, g, c, round_ptrs(&h), PROBE_CAP);
}

int run_small(const uint32_t* L, const uint32_t* k, const uint64_t* seeds, uint32_t n,
              uint32_t threads, uint32_t* n_j, uint32_t* n_c, cudaStream_t st) {
  NvtxRange range("rsa_run_small");
  std::vector<Shape> shapes;
  std::map<std::pair<uint32_t, uint32_t>, u32> known;
  std::vector<SmallJob> jobs(n);
  size_t slot = 0, smem = 0;
  for (uint32_t i = 0; i < n; ++i) {
    if (!rsa_detail::small_eligible(L[i], k[i]))
      return fail(RSA_EINVAL, "rsa_run_small: sample " + std::to_string(i) + " (L=" +
                                  std::to_string(L[i]) + ", k=" + std::to_string(k[i]) +
                                  ") needs L <= 128 and L^2/k <= 4096");
    auto it = known.find({L[i], k[i]});
    if (it == known.end()) {
      size_t bytes = 0;
      shapes.push_back(slot_shape(L[i], k[i], &bytes));
      it = known.emplace(std::make_pair(L[i], k[i]), (u32)shapes.size() - 1).first;
      slot = std::max(slot, align_up(bytes));
      smem = std::max(smem, sample_smem(shapes.back()));
    }
    jobs[i] = SmallJob{seeds[i], it->second, 0};
  }
  int dev = 0, sms = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  cudaMemPool_t pool = nullptr;
  int rc = small_pool(dev, &pool);
  if (rc) return rc;
  CUDA_TRY(cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMP_MAX));
  if (!threads) {
    // One sample per SM at a time: as many threads as a block takes.  More
    // samples than that: smaller blocks, as many as shared memory holds beside
    // each other (5000 samples of L = 16, k = 2: 0.77 ms by 256 threads, 1.25 by
    // 512, 2.40 by 1024; of L = 128, k = 128, two blocks per SM: 4.51, 4.36 and
    // 7.96; of L = 64, k = 4, one block: 5.28, 4.23 and 3.99).
    const size_t fit = n > (u32)sms ? (SMP_MAX + 1024) / (smem + 1024) : 1;
    threads = fit >= 4 ? SMP_THREADS / 4 : fit >= 2 ? SMP_THREADS / 2 : SMP_THREADS;
  }
  int per_sm = 0;
  CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_small, (int)threads, smem));
  u32 grid = (u32)std::min<u64>(n, (u64)sms * std::max(per_sm, 1));
  // shapes and jobs in one copy; then results, work counters, job counter, slots
  const size_t sb = align_up(sizeof(Shape) * shapes.size()), jb = align_up(sizeof(SmallJob) * n);
  const size_t ob = align_up(sizeof(SmallOut) * n), wb = 4 * WORK_SLOTS * 8 + ALIGN;
  std::vector<char> in(sb + jb);
  std::memcpy(in.data(), shapes.data(), sizeof(Shape) * shapes.size());
  std::memcpy(in.data() + sb, jobs.data(), sizeof(SmallJob) * n);
  std::vector<SmallOut> out(n);
  char* d = nullptr;
  cudaError_t e;
  // where a slot for every block does not fit the free memory, fewer blocks take
  // more samples each
  for (;; grid = (grid + 1) / 2) {
    e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&d), sb + jb + ob + wb + grid * slot, pool, st);
    if (e == cudaSuccess) break;
    cudaGetLastError();
    if (e != cudaErrorMemoryAllocation || grid == 1)
      return fail(RSA_ECUDA, std::string("rsa_run_small: ") + cudaGetErrorString(e));
  }
  char* work = d + sb + jb + ob;
  e = cudaMemcpyAsync(d, in.data(), in.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(work, 0, wb, st);
  if (e == cudaSuccess) {
    k_small<<<grid, threads, smem, st>>>(
        reinterpret_cast<const Shape*>(d), reinterpret_cast<const SmallJob*>(d + sb), n,
        reinterpret_cast<SmallOut*>(d + sb + jb), work + wb, slot, reinterpret_cast<u64*>(work),
        reinterpret_cast<u32*>(work + 4 * WORK_SLOTS * 8));
    e = cudaGetLastError();
    if (e == cudaSuccess) g_small_launches.fetch_add(1);
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out.data(), d + sb + jb, sizeof(SmallOut) * n, cudaMemcpyDeviceToHost, st);
  cudaFreeAsync(d, st);
  const cudaError_t e2 = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess)
    return fail(RSA_ECUDA, std::string("rsa_run_small: ") + cudaGetErrorString(e));
  int first = 0;
  for (uint32_t i = 0; i < n; ++i) {
    n_j[i] = out[i].n_j;
    n_c[i] = out[i].n_c;
    const int cd = status_code(out[i].status);
    if (cd && !first) {
      first = cd;
      g_err = "sample " + std::to_string(i) + " status bits " + std::to_string(out[i].status);
    }
  }
  return first;
}

}  // namespace

namespace rsa_detail {
bool small_eligible(uint32_t L, uint32_t k) {
  return k >= 1 && k <= L && L <= SMALL_LMAX && (uint64_t)L * L / k <= SMALL_NMAX;
}
unsigned long long take_small_launches() { return g_small_launches.exchange(0); }
void release_small() {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  int dev = 0, now = -1;
  unsigned long long ctx = 0;
  if (g_pools.empty() || cudaGetDevice(&dev) != cudaSuccess) return;
  for (auto& p : g_pools) {  // ordered by device
    if (p.first.first != now && cudaSetDevice(now = p.first.first) == cudaSuccess)
      ctx = current_context_id();
    if (p.second && p.first.second == ctx) cudaMemPoolTrimTo(p.second, 0);
  }
  cudaSetDevice(dev);
}
}  // namespace rsa_detail

extern "C" {

int rsa_run_small(const uint32_t* L, const uint32_t* k, const uint64_t* seeds, uint32_t n,
                  uint32_t threads, uint32_t* n_j, uint32_t* n_c, void* stream) {
  if (!L || !k || !seeds || !n_j || !n_c || n == 0)
    return fail(RSA_EINVAL, "rsa_run_small: null array or n == 0");
  if (threads % 32 || threads > 1024)
    return fail(RSA_EINVAL, "threads must be 32 .. 1024, a multiple of 32");
  // the search's set-up needs 256 threads
  if (threads) threads = std::max(threads, 256u);
  return run_small(L, k, seeds, n, threads, n_j, n_c, static_cast<cudaStream_t>(stream));
}

int rsa_create(uint32_t L, uint32_t k, uint64_t seed, rsa_t** out) {
  if (!out) return fail(RSA_EINVAL, "out is NULL");
  *out = nullptr;
  if (!(k >= 1 && k <= L && L <= 32768))
    return fail(RSA_EINVAL, "need 1 <= k <= L <= 32768");
  rsa_t* h = new (std::nothrow) rsa_t();
  if (!h) return fail(RSA_ENOMEM, "host allocation failed");
  h->L = L;
  h->k = k;
  h->seed = seed;
  h->geo = plan(L, k);
  *out = h;
  g_err.clear();
  return 0;
}

int rsa_run_seeds(rsa_t* h, const uint64_t* seeds, uint32_t n, void* stream) {
  if (!h || !seeds) return fail(RSA_EINVAL, "null handle or seeds");
  return run_impl(h, seeds, n, nullptr, static_cast<cudaStream_t>(stream));
}

int rsa_run_batch(rsa_t* h, uint32_t n_samples, void* stream) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  std::vector<uint64_t> seeds(n_samples);
  for (uint32_t i = 0; i < n_samples; ++i) seeds[i] = h->seed + i;
  return run_impl(h, seeds.data(), n_samples, nullptr, static_cast<cudaStream_t>(stream));
}

int rsa_run_keys(rsa_t* h, const uint64_t* keys, void* stream) {
  if (!h || !keys) return fail(RSA_EINVAL, "null handle or keys");
  const u64 n = 2ull * h->L * h->L;
  std::vector<u32> order(n);
  for (u64 i = 0; i < n; ++i) order[i] = (u32)i;
  std::sort(order.begin(), order.end(), [&](u32 a, u32 b) { return keys[a] < keys[b]; });
  // Only the order of the priorities matters.  The slices of the scan expect
  // them spread evenly over 64 bits, so the ranks, spread evenly, run in
  // their place.
  const u64 step = (KEY_NONE - 1) / n;
  std::vector<uint64_t> spread(n);
  for (u64 i = 0; i < n; ++i) {
    if (keys[order[i]] == KEY_NONE) return fail(RSA_EINVAL, "key 2^64-1 is reserved");
    if (i && keys[order[i]] == keys[order[i - 1]])
      return fail(RSA_EINVAL, "keys are not distinct");
    spread[order[i]] = i * step + step / 2;
  }
  uint64_t seed = h->seed;
  return run_impl(h, &seed, 1, spread.data(), static_cast<cudaStream_t>(stream));
}

int rsa_run_static(uint32_t L, uint32_t k, const uint64_t* seeds, uint32_t n, uint32_t* n_j,
                   uint32_t* n_c, void* stream) {
  if (!seeds || !n_j || !n_c) return fail(RSA_EINVAL, "null seeds or output array");
  if (!(k >= 1 && k <= L && L <= 32768)) return fail(RSA_EINVAL, "need 1 <= k <= L <= 32768");
  if (n == 0) return fail(RSA_EINVAL, "n must be >= 1");
  rsa h;
  h.L = L;
  h.k = k;
  h.seed = 0;
  h.geo = plan(L, k);
  const size_t need = layout_of(L, k, n, false, h.geo).total;
  if (need > STATIC_WS_BYTES)
    return fail(RSA_EINVAL, "rsa_run_static: L=" + std::to_string(L) + " k=" + std::to_string(k) +
                                " n=" + std::to_string(n) + " needs " + std::to_string(need) +
                                " bytes of workspace; the static workspace holds " +
                                std::to_string(STATIC_WS_BYTES));
  void* ws = nullptr;
  int rc = static_workspace(&ws);
  if (rc) return rc;
  h.use_graphs = false;  // plain launches only: nothing is created or allocated
  h.bound_ptr = ws;  // the run's buffers (all re-initialised by the run) live here
  h.bound_bytes = STATIC_WS_BYTES;
  alignas(8) u32 counter[READ_BYTES / 4] = {};  // pageable host words for the loop checks
  h.h_counter = counter;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  rc = run_impl(&h, seeds, n, nullptr, st);
  h.h_counter = nullptr;
  if (rc) return rc;
  // results straight from the per-sample state records (strided copies)
  const char* sts = static_cast<const char*>(ws) + h.lay.st;
  CUDA_TRY(cudaMemcpy2DAsync(n_c, sizeof(u32), sts + offsetof(SampleState, status),
                             sizeof(SampleState), sizeof(u32), n, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  int first = 0;
  for (u32 i = 0; i < n && !first; ++i) {
    first = status_code(n_c[i]);
    if (first) g_err = "sample " + std::to_string(i) + " status bits " + std::to_string(n_c[i]);
  }
  CUDA_TRY(cudaMemcpy2DAsync(n_j, sizeof(u32), sts + offsetof(SampleState, n_nodes),
                             sizeof(SampleState), sizeof(u32), n, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpy2DAsync(n_c, sizeof(u32), sts + offsetof(SampleState, nc),
                             sizeof(SampleState), sizeof(u32), n, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  return first;
}

int rsa_results(rsa_t* h, uint32_t* n_j, uint32_t* n_c, uint32_t n) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  if (n > h->last_n) return fail(RSA_EINVAL, "n exceeds samples of the last run");
  States states;
  int rc = fetch_states(h, &states);
  if (rc) return rc;
  const std::vector<SampleState>& st = *states;
  int first = 0;
  for (u32 i = 0; i < n; ++i) {
    if (n_j) n_j[i] = st[i].n_nodes;
    if (n_c) n_c[i] = st[i].nc;
    int c = status_code(st[i].status);
    if (c && !first) {
      first = c;
      g_err = "sample " + std::to_string(i) + " status bits " + std::to_string(st[i].status);
    }
  }
  return first;
}

int rsa_sample_stats(rsa_t* h, uint32_t* rounds, uint32_t* probes, uint32_t* edges,
                     int32_t* status, uint32_t n) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  if (n > h->last_n) return fail(RSA_EINVAL, "n exceeds samples of the last run");
  States states;
  int rc = fetch_states(h, &states);
  if (rc) return rc;
  const std::vector<SampleState>& st = *states;
  for (u32 i = 0; i < n; ++i) {
    if (rounds) rounds[i] = st[i].rounds;
    if (probes) probes[i] = st[i].w.probes;
    if (edges) edges[i] = st[i].n_edges;
    if (status) status[i] = status_code(st[i].status);
  }
  return 0;
}

int rsa_contacts(rsa_t* h, uint32_t* n_x, uint32_t* n_y, uint32_t* n_xy, uint32_t n) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  if (n > h->last_n) return fail(RSA_EINVAL, "n exceeds samples of the last run");
  States states;
  int rc = fetch_states(h, &states);
  if (rc) return rc;
  const std::vector<SampleState>& st = *states;
  for (u32 i = 0; i < n; ++i) {
    if (n_x) n_x[i] = st[i].contacts_x;
    if (n_y) n_y[i] = st[i].contacts_y;
    if (n_xy) n_xy[i] = st[i].contacts_xy;
  }
  return 0;
}

int rsa_accepted(rsa_t* h, uint32_t sample, uint32_t* idx, uint32_t cap, uint32_t* count) {
  if (!h || !count) return fail(RSA_EINVAL, "null argument");
  if (sample >= h->last_n) return fail(RSA_EINVAL, "sample out of range");
  States states;
  int rc = fetch_states(h, &states);
  if (rc) return rc;
  const std::vector<SampleState>& st = *states;
  const u32 cn = cap_nodes_of(h->L, h->k);
  const u32 nj = std::min(st[sample].n_nodes, cn);
  std::vector<uint32_t> v(nj);
  const char* b = static_cast<const char*>(h->ws);
  if (nj)
    CUDA_TRY(cudaMemcpy(v.data(), b + h->lay.node_idx + (size_t)sample * cn * 4, (size_t)nj * 4,
                        cudaMemcpyDeviceToHost));
  std::sort(v.begin(), v.end());
  *count = nj;
  if (idx) std::memcpy(idx, v.data(), (size_t)std::min(cap, nj) * 4);
  return 0;
}

int rsa_cluster_sizes(rsa_t* h, uint32_t sample, uint32_t m, uint32_t* counts, uint32_t cap) {
  if (!counts) return fail(RSA_EINVAL, "null counts");
  uint32_t w;
  return configuration(h, sample, m, counts, cap, &w);
}

int rsa_wrap_dirs(rsa_t* h, uint32_t sample, uint32_t m, uint32_t* wrap_x, uint32_t* wrap_y) {
  uint32_t w = 0;
  int rc = configuration(h, sample, m, nullptr, 0, &w);
  if (rc) return rc;
  if (wrap_x) *wrap_x = w & 1u;
  if (wrap_y) *wrap_y = (w >> 1) & 1u;
  return 0;
}

int rsa_workspace_bytes(uint32_t L, uint32_t k, uint32_t n_samples, uint64_t* bytes) {
  if (!bytes || !(k >= 1 && k <= L && L <= 32768) || n_samples == 0)
    return fail(RSA_EINVAL, "bad arguments");
  Geometry G = plan(L, k);
  *bytes = layout_of(L, k, n_samples, false, G).total;
  return 0;
}

int rsa_bind_workspace(rsa_t* h, void* dev_ptr, uint64_t bytes) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  if (dev_ptr && (reinterpret_cast<uintptr_t>(dev_ptr) % ALIGN))
    return fail(RSA_EINVAL, "workspace must be 256-byte aligned");
  h->bound_ptr = dev_ptr;
  h->bound_bytes = dev_ptr ? bytes : 0;
  return 0;
}

int rsa_test_caps(rsa_t* h, uint32_t round_cap, uint32_t uf_steps, uint32_t probe_cap,
                  uint32_t edge_cap) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  h->t_round = round_cap;
  h->t_uf = uf_steps;
  h->t_probe = probe_cap;
  h->t_edges = edge_cap;
  return 0;
}

int rsa_set_rounds_per_check(rsa_t* h, uint32_t rounds) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  if (rounds < 1 || rounds > 64) return fail(RSA_EINVAL, "rounds per check must be in 1 .. 64");
  h->round_check = rounds;
  return 0;
}

int rsa_set_window_threads(rsa_t* h, uint32_t threads) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  if (threads != 0 && threads != 256 && threads != 128)
    return fail(RSA_EINVAL, "window CTA size must be 128 or 256");
  if (threads == 128 && !h->geo.win128)
    return fail(RSA_EINVAL, "128-thread windows need 32 < k <= 4096 dividing spans of 2048 or 4096 cells");
  return 0;
}

int rsa_profile(rsa_t* h, int enable) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  h->prof.on = enable != 0;
  return 0;
}

int rsa_kernel_stats(rsa_t* h, double* ms, unsigned long long* launches, uint32_t n_kinds) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  Prof& p = h->prof;
  if (!p.kinds.empty()) {
    if (h->stream || h->device >= 0) CUDA_TRY(cudaStreamSynchronize(h->stream));
    for (size_t i = 0; i < p.kinds.size(); ++i) {
      float t = 0.f;
      if (cudaEventElapsedTime(&t, p.pool[2 * i], p.pool[2 * i + 1]) == cudaSuccess)
        p.ms[p.kinds[i]] += t;
    }
    p.kinds.clear();
  }
  for (uint32_t i = 0; i < n_kinds && i < (uint32_t)KD_COUNT; ++i) {
    if (ms) ms[i] = p.ms[i];
    if (launches) launches[i] = p.launches[i];
    p.ms[i] = 0.0;
    p.launches[i] = 0;
  }
  return 0;
}

int rsa_work_stats(rsa_t* h, unsigned long long* out, uint32_t n) {
  if (!h) return fail(RSA_EINVAL, "null handle");
  for (uint32_t i = 0; i < n && i < 4; ++i) {
    if (out) out[i] = h->work[i];
    h->work[i] = 0;
  }
  return 0;
}

const char* rsa_kernel_name(uint32_t kind) {
  return kind < (uint32_t)KD_COUNT ? kKindNames[kind] : "";
}

void rsa_destroy(rsa_t* h) {
  if (!h) return;
  drop_graph(h->g_main);
  drop_graph(h->g_round);
  drop_graph(h->g_search);
  drop_graph(h->g_probe);
  if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
  for (cudaEvent_t e : h->prof.pool) cudaEventDestroy(e);
  if (h->own_ptr) cudaFree(h->own_ptr);
  if (h->h_counter) cudaFreeHost(h->h_counter);
  delete h;
}

const char* rsa_last_error(void) { return g_err.c_str(); }

}  // extern "C"
