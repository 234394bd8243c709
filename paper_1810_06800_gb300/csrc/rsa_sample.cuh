// rsa_sample.cuh -- a whole sample in one block, sm_103a: deposition, contact
// graph and first-wrap search of one sample after another in one launch, for
// lattices whose cover bits, bins and active candidates fit a block's shared
// memory.
//
// The steps are those of rsa_rounds.cuh and rsa_search.cuh; what are kernel
// boundaries there are block barriers here.  A round of a small sample is a
// chain of a dozen dependent accesses (entry, cover words, counter, bin,
// chain of the bin, node counter), each 0.3 to 0.5 us from L2, plus launch,
// fence and ticket: 20 to 30 us a round over several launches.  In shared
// memory the chain costs about a tenth.  (Clusters of blocks over the same
// buffers in L2 were tried: 17 us a round, 64 us at L = 1024.)
// Two callers: a handle's batch (k_sample, sample s in the s-th part of every
// buffer) and rsa_run_small (k_small: samples of any mix of shapes, each
// block in a workspace slot of its own).
#pragma once
#include "rsa_rounds.cuh"

namespace rsak {

constexpr u32 SMP_THREADS = 1024;
constexpr u32 SMP_PER = 16;  // candidates per thread and tile of its first pass
constexpr u32 NO_HOT = 0xFFFFFFFFu;

struct Shape {       // everything a sample's run needs to know of its (L, k)
  Group g;
  RoundCfg c;
  RoundPtrs p;
  SearchCfg sc;
  u32 probe_cap, sites;
  // byte offsets of the buffers kept in shared memory (NO_HOT: in the
  // workspace), and their size
  u32 fine, heads, act, anch, hot_bytes;
};

struct SmallJob {    // one sample of rsa_run_small
  u64 seed;
  u32 shape, pad;
};
struct SmallOut {    // its results
  u32 n_j, n_c, rounds, status;
};

struct SampleSmem {
  Shape sh;
  RoundState r;
  Window w;
  u64 mids[2];
  u32 status, rounds, flag, taken;
  u64 work[4];
  u32 part[256];
  u32 nodes, edges;
  FinishSmem fin;
};
union SampleScratch {  // one use at a time
  DenseSmem<SMP_THREADS, SMP_PER> dense;
  u32 refill[REFILL_WORDS];
  u32 hist[EHIST];
  struct {
    u32 hist[SUB_WORDS], queue[queue_words(SMP_THREADS)];
  } probe;
};
constexpr size_t SMP_FIXED = (sizeof(SampleSmem) + 15) / 16 * 16;
constexpr size_t SMP_SCRATCH = (sizeof(SampleScratch) + 15) / 16 * 16;
constexpr size_t SMP_MAX = 227 * 1024;

// Dynamic shared memory of a shape: the hot buffers and the scratch, or the
// last window of the search in their place.
__host__ __device__ inline size_t sample_smem(const Shape& sh) {
  const size_t a = SMP_SCRATCH + sh.hot_bytes, b = finish_smem(sh.sc);
  return SMP_FIXED + (a > b ? a : b);
}

__device__ __forceinline__ void block_fill(u32* a, size_t n, u32 v) {
  for (size_t i = threadIdx.x; i < n; i += blockDim.x) a[i] = v;
}

// One sample; sm.sh is its shape with every pointer at this sample's part.
__device__ void run_sample(SampleSmem& sm, SampleScratch& scratch, unsigned char* finish,
                           u64 seed) {
  const Group& g = sm.sh.g;
  const RoundCfg& c = sm.sh.c;
  const RoundPtrs& p = sm.sh.p;
  RoundState& r = sm.r;
  const Team team{0, 1};
  const u32 tid = threadIdx.x, nt = blockDim.x, L = g.L, k = g.k;
  SampleState& st = g.st[0];
  if (tid == 0) {
    RoundState z = {};
    z.sl = first_slice(c);
    r = z;
    SampleState y = {};
    y.nc = NONE32;
    st = y;
    g.base[0] = mix64(seed + SM_GAMMA);
    sm.w = first_window();
    sm.rounds = sm.status = sm.flag = sm.taken = sm.nodes = sm.edges = 0;
    for (u32 i = 0; i < 4; ++i) sm.work[i] = 0;
    sm.work[0] = 2 * g.LL;
  }
  if (!sm.sh.sites) {
    block_fill(p.fine, (size_t)2 * (L + c.nbl) * c.W, 0);
    block_fill(p.anch, (size_t)4 * L * c.WA, 0);
    block_fill(p.heads, (size_t)4 * c.nb * c.nb, NONE32);
  }
  __syncthreads();
  // ---- deposition ----
  if (sm.sh.sites) {
    sites_body(g, 0, team);
    if (tid == 0) {
      st.n_nodes = (u32)g.LL;
      sm.rounds = 1;
      sm.work[3] = g.LL;
    }
    __syncthreads();
  } else {
    if (g.keys) dense_body<true>(g, c, p, 0, team, r, scratch.dense);
    else dense_body<false>(g, c, p, 0, team, r, scratch.dense);
    __syncthreads();
    for (;;) {
      const Slice sl = r.sl;
      const u32 n1 = slice_entries(c, r, sl), n2 = r.act[sl.par ^ 1u];
      // (k > PICK_LONGK: 300 KB of cover bits and more, never in one block)
      pick_body<false>(g, c, p, 0, team, sl, n1, n2, &r.act[sl.par]);
      __syncthreads();
      const u32 n = r.act[sl.par];
      const bool over = n > c.cap_act;
      clear_bins(g, c, p, 0, team, over ? sl.par : sl.par ^ 1u);
      u32 taken = 0;
      if (!over) {
        // one lane each: chains in shared memory are short, and a block that
        // runs alone on its SM is bound by the instructions it issues
        if (k > 128) resolve_body<32>(g, c, p, 0, team, sl.par, n, &sm.nodes, taken);
        else resolve_body<1>(g, c, p, 0, team, sl.par, n, &sm.nodes, taken);
      }
      taken = __reduce_add_sync(FULL, taken);
      if ((tid & 31) == 0 && taken) atomicAdd(&sm.taken, taken);
      __syncthreads();
      if (tid == 0) {
        u32 rounds = sm.rounds, status = sm.status;
        sm.flag = round_step(c, r.sl, n, n - sm.taken, rounds, status);
        r.act[r.sl.par] = 0;
        sm.rounds = rounds;
        sm.status = status;
        sm.work[1] += n1 + n2;
        sm.work[2] += over ? 0 : n;
        sm.work[3] += sm.taken;
        sm.taken = 0;
        if (r.sl.refill) r.flat_n = 0;
      }
      __syncthreads();
      if (sm.flag) break;
      while (r.sl.refill) {
        refill_body(g, c, p, 0, team, r.sl, &r.flat_n, scratch.refill, REFILL_WORDS);
        __syncthreads();
        if (tid == 0) {
          refill_step(c, r.sl, r.flat_n);
          if (r.sl.refill) r.flat_n = 0;
        }
        __syncthreads();
      }
    }
  }
  // ---- contact graph (in the region of the lists) ----
  if (g.ehist) block_fill(g.ehist, SEARCH_WORDS, 0);
  if (tid == 0) {
    sm.status |= st.status;
    if (!sm.sh.sites) st.n_nodes = sm.nodes;
  }
  __syncthreads();
  if (!(sm.status & (ST_NODE_OVF | ST_ROUND_CAP))) {
    if (sm.sh.sites) site_contacts_body(g, 0, team, scratch.hist);
    else if (k <= 64) contacts_body<1>(g, c, p, 0, team, &sm.edges, scratch.hist);
    else contacts_body<4>(g, c, p, 0, team, &sm.edges, scratch.hist);
  }
  __syncthreads();
  // ---- first wrap ----
  EdgeQueue& queue = *reinterpret_cast<EdgeQueue*>(scratch.probe.queue);
  const u32 ne = sm.sh.sites ? st.n_edges : sm.edges;
  if (tid == 0) {
    st.n_edges = ne;
    sm.status |= st.status;
    sm.flag = (sm.status & (ST_NODE_OVF | ST_ROUND_CAP | ST_EDGE_OVF)) != 0;
    sm.w.ready = ne <= sm.sh.sc.win_cap;
  }
  __syncthreads();
  if (!sm.flag) {
    if (g.ehist) {
      thresholds_body(g, sm.sh.sc, 0, ne, sm.part, sm.mids);
      if (tid == 0) {
        sm.w.mid = sm.mids[0];
        sm.w.next_mid = sm.mids[1];
      }
      __syncthreads();
    }
    u32* set = g.ehist + EHIST;
    while (!sm.w.ready && !sm.flag) {
      copy_body(g, 0, team, sm.w);
      __syncthreads();
      probe_body(g, 0, team, sm.w, scratch.probe.hist, queue, set);
      __syncthreads();
      if (tid < 32) {
        Window w = sm.w;
        u32 status = sm.status | st.status;
        const bool end = probe_step(w, set, sm.sh.sc.win_cap, sm.sh.probe_cap, status);
        __syncwarp();
        if (tid == 0) {
          sm.w = w;
          sm.status = status;
          sm.flag = end;
        }
      }
      __syncthreads();
      for (u32 i = tid; i < SUB_WORDS; i += nt) set[i] = 0;
    }
  }
  if (!sm.flag) {
    collect_body(g, sm.sh.sc, 0, team, sm.w, queue);
    __syncthreads();
    finish_body(g, sm.sh.sc, 0, sm.w, sm.sh.probe_cap, finish, sm.fin);
    __syncthreads();
    if (st.ranked == 1) rank_body(g, 0, team);
  }
  __syncthreads();
  if (tid == 0) {
    st.status |= sm.status;
    st.rounds = sm.rounds;
    if (sm.flag) st.w.probes = sm.w.probes;
    st.done = 1;
    st.sdone = 1;
    for (u32 i = 0; i < 4; ++i) work_add(g, i, sm.work[i]);
  }
}

// The shape's hot buffers, in shared memory from `hot` on.
__device__ __forceinline__ void place_hot(Shape& sh, unsigned char* hot) {
  RoundPtrs& p = sh.p;
  if (sh.fine != NO_HOT) {
    p.fine = reinterpret_cast<u32*>(hot + sh.fine);
    p.block = p.fine + (size_t)2 * sh.g.L * sh.c.W;
  }
  if (sh.heads != NO_HOT) p.heads = reinterpret_cast<u32*>(hot + sh.heads);
  if (sh.act != NO_HOT) p.act = reinterpret_cast<Act*>(hot + sh.act);
  if (sh.anch != NO_HOT) p.anch = reinterpret_cast<u32*>(hot + sh.anch);
}

template <typename T>
__device__ __forceinline__ void move_ptr(T*& ptr, size_t bytes) {
  ptr = reinterpret_cast<T*>(reinterpret_cast<char*>(ptr) + bytes);
}

// Sample s of a batch (or, with a slot's address as `extra`, of none): every
// pointer moved to its part.
__device__ __forceinline__ void place_sample(Shape& sh, u32 s, size_t extra) {
  Group& g = sh.g;
  RoundPtrs& p = sh.p;
  const size_t region = (size_t)s * g.rstride + extra;
  const size_t node = (size_t)s * g.cap_nodes;
  move_ptr(g.owner, (size_t)s * g.LL * 4 + extra);
  move_ptr(g.base, (size_t)s * 8 + extra);
  move_ptr(g.node_key, node * 8 + extra);
  move_ptr(g.node_idx, node * 4 + extra);
  move_ptr(g.node_pos, node * 4 + extra);
  move_ptr(g.st, (size_t)s * sizeof(SampleState) + extra);
  move_ptr(p.anch, (size_t)s * 4 * g.L * sh.c.WA * 4 + extra);
  move_ptr(g.uf, region);
  move_ptr(g.etime, region);
  move_ptr(g.elink, region);
  move_ptr(g.win, region);
  if (g.ehist) move_ptr(g.ehist, region);
  move_ptr(p.fine, region);
  move_ptr(p.block, region);
  move_ptr(p.list, region);
  move_ptr(p.flat, region);
  move_ptr(p.act, region);
  move_ptr(p.heads, region);
}

struct SampleParts {
  SampleSmem* sm;
  SampleScratch* scratch;
  unsigned char *hot, *finish;
  __device__ __forceinline__ explicit SampleParts(unsigned char* raw)
      : sm(reinterpret_cast<SampleSmem*>(raw)),
        scratch(reinterpret_cast<SampleScratch*>(raw + SMP_FIXED)),
        hot(raw + SMP_FIXED + SMP_SCRATCH), finish(raw + SMP_FIXED) {}
};

__global__ void __launch_bounds__(SMP_THREADS, 1)
    k_sample(const __grid_constant__ Shape shape, const u64* seeds) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SampleParts q(smem_raw);
  for (u32 s = blockIdx.x; s < shape.g.n; s += gridDim.x) {
    if (threadIdx.x == 0) {
      q.sm->sh = shape;
      place_sample(q.sm->sh, s, 0);
      place_hot(q.sm->sh, q.hot);
    }
    __syncthreads();
    run_sample(*q.sm, *q.scratch, q.finish, seeds[s]);
    __syncthreads();
  }
}

// The shapes' pointers are offsets into a block's slot.
__global__ void __launch_bounds__(SMP_THREADS, 1)
    k_small(const Shape* shapes, const SmallJob* jobs, u32 n_jobs, SmallOut* out, char* slots,
            size_t slot_bytes, u64* work, u32* next) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SampleParts q(smem_raw);
  for (;;) {
    if (threadIdx.x == 0) q.sm->flag = atomicAdd(next, 1u);
    __syncthreads();
    const u32 it = q.sm->flag;
    if (it >= n_jobs) return;
    const SmallJob job = jobs[it];
    if (threadIdx.x == 0) {
      Shape& sh = q.sm->sh;
      sh = shapes[job.shape];
      place_sample(sh, 0, reinterpret_cast<size_t>(slots) + (size_t)blockIdx.x * slot_bytes);
      place_hot(sh, q.hot);
      sh.g.work = work;
    }
    __syncthreads();
    run_sample(*q.sm, *q.scratch, q.finish, job.seed);
    __syncthreads();
    if (threadIdx.x == 0) {
      const SampleState& st = q.sm->sh.g.st[0];
      SmallOut r;
      r.n_j = st.n_nodes;
      r.n_c = st.ranked == 1 ? st.nc : NONE32;
      r.rounds = st.rounds;
      r.status = st.status;
      out[it] = r;
    }
    __syncthreads();
  }
}

}  // namespace rsak
