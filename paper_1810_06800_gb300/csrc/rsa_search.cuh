// rsa_search.cuh -- first wrap (Sec. II.D) on the contact graph, sm_103a.
//
// wrap(T): does the graph of the k-mers of priority <= T contain a cycle of
// non-zero winding?  It is monotone in T and changes at the priority T_c of
// one k-mer; n_c is the rank of T_c.  An edge exists from the larger priority
// of its two ends on (its time), so wrap(T) takes the edges of time <= T.
// The search keeps a window (lo, hi] of times that holds T_c, and the
// union-find state of the edges up to lo:
//   k_probe_copy, k_probe   unite the edges of (lo, mid]; a closed cycle of
//              non-zero winding moves hi to mid, otherwise lo moves there.
//              The first two thresholds are quantiles of the edge times just
//              below and above where T_c is expected (k-mers at the first wrap
//              over k-mers at jamming: 0.59 + 0.0225 log2 k), later ones
//              halve the edges of the window;
//   k_collect  once the window holds at most FIN_EDGES edges (or edges of one
//              time only): those, with the roots of their ends and the
//              displacement between the roots;
//   k_finish   one block per sample: the rest of the search in shared memory,
//              on the graph of the roots; the last 32 edges one by one, unless
//              the window has come down to one time, which then is T_c;
//   k_rank     n_c, the k-mers of priority <= T_c.
// Samples whose whole graph has at most FIN_EDGES edges need no probe.
// That hi itself wraps is assumed until a probe shows it (the jammed lattice
// must wrap) and tested at the end if none has.
// Union-find words: parent (bits 0-31) and the lifted offset of the node from
// its parent, dx (32-47), dy (48-63), modulo 2^16.  A wrap is a cycle of
// primitive winding (a, b) times L; for L < 65536 its offset is never 0
// modulo 2^16, so 16-bit offsets decide exactly.
#pragma once
#include "rsa_device.cuh"

namespace rsak {

constexpr u32 FIN_EDGES = 4096;
constexpr u32 FIN_THREADS = 1024;
constexpr u32 FIN_SLOTS = 4 * FIN_EDGES;  // hash slots for the roots of the window (4 B: as much
                                          // as 2 FIN_EDGES union-find words)
constexpr u32 SUB_BINS = 128;
// per sample: the time histogram, and the counts of a probe
constexpr u32 SUB_WRAP = SUB_BINS, SUB_A = SUB_BINS + 1, SUB_B = SUB_BINS + 2;
constexpr u32 SUB_WORDS = SUB_BINS + 4;
constexpr u32 SEARCH_WORDS = EHIST + SUB_WORDS;

struct WinEdge {  // an edge of the last window, between roots
  u64 time;
  u32 r1, r2, dxy, pad;
};

struct SearchCfg {
  u32 win_cap;      // window edges stored per sample (<= FIN_EDGES with hashed roots)
  u32 hashed;       // roots are renumbered through a hash table (else: node ids)
  u32 ids;          // union-find words in shared memory
  u32 q0, q1;       // first two thresholds, edge quantiles in 1/65536
};

// Root of x and x's offset from it, halving the path: every node passed gets
// its grandparent for parent by a plain store.  A node that is no root never
// becomes one, and every word stored for it is a true ancestor relation, so
// stores may overtake one another.  Global words are read from L2 (other SMs
// write them).
template <bool GLOBAL>
__device__ __forceinline__ u32 find_root(u64* W, u32 x, u32* ox, u32* oy, bool* capped, u32 cap) {
  auto load = [&](u32 i) { return GLOBAL ? __ldcg(W + i) : *(volatile u64*)(W + i); };
  u32 sx = 0, sy = 0, steps = 0;
  u64 w = load(x);
  for (;;) {
    const u32 p = (u32)w;
    if (p == x) break;
    if (++steps >= cap) {
      *capped = true;
      break;
    }
    const u64 wp = load(p);
    const u32 gp = (u32)wp, dx = (u32)(w >> 32), dy = (u32)(w >> 48);
    if (gp == p) {
      sx += dx;
      sy += dy;
      x = p;
      break;
    }
    const u64 nw = uf_pack(gp, dx + (u32)(wp >> 32), dy + (u32)(wp >> 48));
    *(volatile u64*)(W + x) = nw;
    sx += (u32)(nw >> 32);
    sy += (u32)(nw >> 48);
    x = gp;
    w = load(x);
  }
  *ox = sx;
  *oy = sy;
  return x;
}

__device__ __forceinline__ u32 uf_find(u64* W, u32 x, u32* ox, u32* oy, bool* capped, u32 cap) {
  return find_root<true>(W, x, ox, oy, capped, cap);
}

// Add edge "anchor(m2) = anchor(m1) + d"; returns true if it closes a cycle
// of non-zero winding, and then, if mis is given, stores the cycle's lifted
// mismatch (x in bits 0-15, y in 16-31, modulo 2^16).  Roots are linked
// larger-id under smaller-id, so the forest stays acyclic under concurrent
// unions.  (Linking in the order of mixed ids, for shallower trees where ids
// follow the lattice, was no faster: k = 1 probes 10.7 ms in all, 9.7 so.)
__device__ bool uf_union(u64* W, u32 m1, u32 m2, u32 dxy, bool* capped, u32 cap,
                         u32* mis = nullptr) {
  const u32 dx = dxy & 0xFFFFu, dy = dxy >> 16;
  for (u32 it = 0; it < cap; ++it) {
    u32 o1x, o1y, o2x, o2y;
    const u32 r1 = uf_find(W, m1, &o1x, &o1y, capped, cap);
    const u32 r2 = uf_find(W, m2, &o2x, &o2y, capped, cap);
    if (*capped) return false;
    // lifted position of r2 minus r1
    const u32 Dx = o1x + dx - o2x, Dy = o1y + dy - o2y;
    if (r1 == r2) {
      if (mis) *mis = (Dx & 0xFFFFu) | ((Dy & 0xFFFFu) << 16);
      return ((Dx | Dy) & 0xFFFFu) != 0;
    }
    if (r1 < r2) {
      if (atomicCAS(W + r2, uf_pack(r2, 0, 0), uf_pack(r1, Dx, Dy)) == uf_pack(r2, 0, 0))
        return false;
    } else {
      if (atomicCAS(W + r1, uf_pack(r1, 0, 0), uf_pack(r2, 0u - Dx, 0u - Dy)) ==
          uf_pack(r1, 0, 0))
        return false;
    }
  }
  *capped = true;
  return false;
}

// Smallest time of bin b of time_bin.
__device__ __forceinline__ u64 bin_floor(u32 b) {
  const u32 e = b >> 5, m = 32 + (b & 31u);
  return e >= 5 ? (u64)m << (e - 5) : (u64)m >> (5 - e);
}

__device__ __forceinline__ Window first_window() {
  Window w = {};
  w.hi = KEY_NONE;
  w.first = 1;
  return w;
}

// Start of the search of one batch; while a sample of it is still being
// deposited (*n_active) nothing of it runs.
__global__ void __launch_bounds__(256) k_graph_init(Group g, const u32* n_active) {
  const u32 s = blockIdx.x;
  const bool wait = *n_active != 0;  // the region still holds the rounds' lists
  if (g.ehist && !wait)
    for (u32 i = threadIdx.x; i < SEARCH_WORDS; i += 256) region_of(g, g.ehist, s)[i] = 0;
  if (threadIdx.x) return;
  SampleState& st = g.st[s];
  st.n_edges = 0;
  st.contacts_x = st.contacts_y = st.contacts_xy = 0;
  st.w = first_window();
  st.ticket = 0;
  st.win_n = 0;
  st.ranked = 0;
  st.nc = NONE32;
  st.sdone = (wait || (st.status & (ST_NODE_OVF | ST_ROUND_CAP))) ? 1u : 0u;
}

// The first two thresholds from the histogram of times, ends of the bins in
// which the quantiles fall.  part: 256 words; out: two thresholds (shared).
__device__ void thresholds_body(const Group& g, const SearchCfg& c, u32 s, u32 ne, u32* part,
                                u64* out) {
  const u32 tid = threadIdx.x;
  constexpr u32 PER = EHIST / 256;
  const u32* h = region_of(g, g.ehist, s);
  u32 v[PER], sum = 0;
  if (tid < 256) {
#pragma unroll
    for (u32 i = 0; i < PER; ++i) {
      v[i] = __ldcg(h + tid * PER + i);
      sum += v[i];
    }
    part[tid] = sum;
  }
  if (tid < 2) out[tid] = KEY_NONE / 2;
  __syncthreads();
  for (u32 d = 1; d < 256; d <<= 1) {
    const u32 o = tid < 256 && tid >= d ? part[tid - d] : 0u;
    __syncthreads();
    if (tid < 256) part[tid] += o;
    __syncthreads();
  }
  if (tid < 256) {
    const u32 r0 = (u32)((u64)ne * c.q0 >> 16), r1 = (u32)((u64)ne * c.q1 >> 16);
    u32 a = part[tid] - sum;
#pragma unroll
    for (u32 i = 0; i < PER; ++i) {
      const u32 b = a + v[i];
      const u64 top = tid * PER + i + 1 < EHIST ? bin_floor(tid * PER + i + 1) - 1 : KEY_NONE - 1;
      if (a <= r0 && r0 < b) out[0] = top;
      if (a <= r1 && r1 < b) out[1] = top;
      a = b;
    }
  }
  __syncthreads();
}

// After the contacts: one block per sample.  Few edges: straight to the last
// window.
__global__ void __launch_bounds__(256) k_search_init(Group g, SearchCfg c) {
  __shared__ u32 part[256];
  __shared__ u64 mids[2];
  const u32 s = blockIdx.x, tid = threadIdx.x;
  SampleState& st = g.st[s];
  if (st.sdone) return;
  const bool ovf = (st.status & ST_EDGE_OVF) != 0;
  const u32 ne = st.n_edges;
  __syncthreads();
  if (ovf) {
    if (tid == 0) st.sdone = 1;
    return;
  }
  if (g.ehist) thresholds_body(g, c, s, ne, part, mids);
  if (tid == 0) {
    if (g.ehist) {
      st.w.mid = mids[0];
      st.w.next_mid = mids[1];
    }
    st.w.ready = ne <= c.win_cap;
  }
}

// The word of node m with its root for parent.  No union runs meanwhile; a
// word that another thread flattens while it is read is a true ancestor
// relation before and after.
__device__ __forceinline__ u64 flat_word(u64* W, u32 m, u32 cap, bool* capped) {
  u64 w = *(volatile u64*)(W + m);
  u32 x = m, sx = 0, sy = 0;
  for (u32 it = 0; it < cap; ++it) {
    const u32 p = (u32)w;
    if (p == x) return uf_pack(x, sx, sy);
    sx += (u32)(w >> 32);
    sy += (u32)(w >> 48);
    x = p;
    w = *(volatile u64*)(W + x);
  }
  *capped = true;
  return uf_pack(x, sx, sy);
}

// Working copy of the union-find state at lo (single k-mers while lo = 0),
// flattened: the walks of a probe start at the roots of that state, and the
// state, if a wrap sends the search back to it, stays flat.
__device__ __forceinline__ void copy_body(const Group& g, u32 s, Team team, const Window& w) {
  const u32 nn = min(g.st[s].n_nodes, g.cap_nodes), nt = blockDim.x;
  u64* S = region_of(g, g.uf, s) + (size_t)w.cur * g.cap_nodes;
  u64* Wd = region_of(g, g.uf, s) + (size_t)(w.cur ^ 1u) * g.cap_nodes;
  bool capped = false;
  for (u32 m = team.rank * nt + threadIdx.x; m < nn; m += team.size * nt) {
    u64 v = uf_pack(m, 0, 0);
    if (w.lo) {
      v = flat_word(S, m, g.uf_cap, &capped);
      S[m] = v;
    }
    Wd[m] = v;
  }
  if (capped) atomicOr(&g.st[s].status, ST_UF_CAP);
}

__global__ void __launch_bounds__(256) k_probe_copy(Group g) {
  const u32 s = blockIdx.y;
  if (g.st[s].sdone) return;
  const Window w = g.st[s].w;
  if (!w.ready) copy_body(g, s, Team{blockIdx.x, gridDim.x}, w);
}

// Sub-bins of the window (lo, hi]: 2^shift times each, at most SUB_BINS.
__device__ __forceinline__ u32 sub_shift(const Window& w) {
  const u32 width = 64 - (u32)__clzll((long long)(w.hi - w.lo - 1));
  return width > 7 ? width - 7 : 0;
}

// A threshold that halves the `in` edges of the window, at an end of a sub-bin
// (sub-bins of 2^shift times from lo0 on), by a whole warp.  Of the last
// sub-bin that is its lower end: the window then shrinks to that sub-bin or
// loses half of its edges, so about three probes take seven bits off a window
// whose edges all share one time, where its middle would take one.
__device__ u64 halve_window(const Window& w, u64 lo0, u32 shift, const u32* set, u32 in) {
  const u32 lane = threadIdx.x & 31;
  const u64 span = (1ull << shift) - 1;
  u32 v[4], sum = 0;  // four sub-bins per lane
  u64 from[4];
#pragma unroll
  for (u32 i = 0; i < 4; ++i) {
    const u32 b = lane * 4 + i;
    from[i] = lo0 + 1 + ((u64)b << shift);
    const u64 end = from[i] + span < from[i] ? KEY_NONE : from[i] + span;
    const bool out = from[i] <= lo0 || end <= w.lo || from[i] > w.hi;
    v[i] = out ? 0u : set[b];
    sum += v[i];
  }
  u32 inc = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const u32 o = __shfl_up_sync(FULL, inc, d);
    if ((int)lane >= d) inc += o;
  }
  const u32 half = in / 2;
  const u32 m = __ballot_sync(FULL, inc >= half && sum);
  u32 a = inc - sum;
  u64 mine = 0;  // start of the sub-bin (at least 1)
#pragma unroll
  for (u32 i = 0; i < 4; ++i) {
    a += v[i];
    if (mine == 0 && v[i] && a >= half) mine = from[i];
  }
  u64 mid = 0;
  if (m) {
    mine = __shfl_sync(FULL, mine, __ffs(m) - 1);
    mid = mine + span;
    if (mid < mine || mid >= w.hi) mid = mine - 1;
  }
  if (mid <= w.lo || mid >= w.hi) mid = w.lo + (w.hi - w.lo) / 2;
  return mid;
}

// The edges of a k-mer to its earlier neighbours all have its priority for
// time (2 k of them where it meets the ends of others all along its sides), so
// a window of one time can hold any number of edges.  Once a probe has wrapped
// there, that time is T_c.
__device__ __forceinline__ bool one_time(const Window& w) { return w.hi - w.lo == 1 && w.hi_ok; }

// The next threshold of a window that is not the last one.
__device__ __forceinline__ u64 next_threshold(const Window& w, u64 lo0, u32 shift, const u32* set,
                                              u32 in) {
  return w.hi - w.lo == 1 ? w.hi : halve_window(w, lo0, shift, set, in);
}

// The step from one probe to the next, from the counts in `set`, by a whole
// warp (every lane holds the same w).  True if the search of the sample ends
// here.
__device__ bool probe_step(Window& w, const u32* set, u32 win_cap, u32 probe_cap, u32& status) {
  w.probes += 1;
  if (status & ST_UF_CAP) return true;
  const bool wrap = set[SUB_WRAP] != 0, first = w.first != 0;
  const u32 in = set[wrap ? SUB_A : SUB_B];
  const u64 lo0 = w.lo;
  const u32 shift = sub_shift(w);
  w.first = 0;
  if (wrap) {
    w.hi = w.mid;
    w.hi_ok = 1;
  } else {
    w.lo = w.mid;
    w.cur ^= 1u;
  }
  if (in <= win_cap || one_time(w)) {
    w.ready = 1;
    return false;
  }
  if (w.probes >= probe_cap) {
    status |= ST_SEARCH_CAP;
    return true;
  }
  if (first && !wrap && w.next_mid > w.lo && w.next_mid < w.hi) w.mid = w.next_mid;
  else w.mid = next_threshold(w, lo0, shift, set, in);
  return false;
}

// Edges picked out of a scan, packed so that whole warps work on them: an
// edge costs a chain of a dozen L2 accesses, and a warp with one such lane
// waits as long as one with 32 (L = 512, k = 1, 100 samples, a window of 5% of
// the edges: 1.9 ms by the lane that met the edge, 0.50 ms packed).
constexpr u32 QUEUE_TILE = 4;      // edges per thread between two looks at the queue
struct EdgeQueue {
  u32 n;
  u32 item[1];                     // (QUEUE_TILE + 1) x the block's threads
};
__host__ __device__ constexpr u32 queue_words(u32 threads) { return 1 + (QUEUE_TILE + 1) * threads; }

// Calls work(i) for every i < ne, spread over the team's blocks, for which
// want(i) holds.  Every thread of the block takes part.
template <typename Want, typename Work>
__device__ __forceinline__ void scan_packed(u32 ne, Team team, EdgeQueue& q, Want want, Work work) {
  const u32 tid = threadIdx.x, nt = blockDim.x;
  // few edges: fewer per thread, on more blocks
  const u32 per = min(QUEUE_TILE, max(1u, (ne + team.size * nt - 1) / (team.size * nt)));
  const u32 tile = per * nt;
  if (tid == 0) q.n = 0;
  __syncthreads();
  for (u32 i0 = team.rank * tile; i0 < ne; i0 += team.size * tile) {
#pragma unroll
    for (u32 j = 0; j < QUEUE_TILE; ++j) {
      if (j == per) break;
      const u32 i = i0 + j * nt + tid;
      const bool ok = i < ne && want(i);
      const u32 at = warp_append(&q.n, ok);
      if (ok) q.item[at] = i;
    }
    __syncthreads();
    const u32 n = q.n;
    if (n >= nt || ne - i0 <= team.size * tile) {  // full, or the last tile of this block
      for (u32 e = tid; e < n; e += nt) work(q.item[e]);
      __syncthreads();
      if (tid == 0) q.n = 0;
    }
    __syncthreads();
  }
}

// Unites the edges of (lo, mid] in the working copy; adds to `set` the edges
// of the window by sub-bin and by side of mid, and whether a wrap was closed.
// hist: SUB_WORDS words (shared).
__device__ void probe_body(const Group& g, u32 s, Team team, const Window& w, u32* hist,
                           EdgeQueue& q, u32* set) {
  const u32 tid = threadIdx.x, nt = blockDim.x;
  SampleState& st = g.st[s];
  const u64 lo = w.lo, mid = w.mid, hi = w.hi;
  const u32 shift = sub_shift(w);
  const u32 ne = min(st.n_edges, g.edge_limit);
  for (u32 i = tid; i < SUB_WORDS; i += nt) hist[i] = 0;
  __syncthreads();
  u64* Wd = region_of(g, g.uf, s) + (size_t)(w.cur ^ 1u) * g.cap_nodes;
  const u64* E = region_of(g, g.etime, s);
  const uint4* K = region_of(g, g.elink, s);
  bool wrap = false, capped = false;
  u32 na = 0, nb = 0;
  scan_packed(
      ne, team, q,
      [&](u32 i) {
        const u64 t = E[i];
        if (t <= lo || t > hi) return false;
        atomicAdd(&hist[(u32)((t - lo - 1) >> shift)], 1u);
        if (t > mid) {
          ++nb;
          return false;
        }
        ++na;
        return true;
      },
      [&](u32 i) {
        const uint4 e = K[i];
        if (uf_union(Wd, e.x, e.y, e.z, &capped, g.uf_cap)) wrap = true;
      });
  na = __reduce_add_sync(FULL, na);
  nb = __reduce_add_sync(FULL, nb);
  if ((tid & 31) == 0) {
    if (na) atomicAdd(&hist[SUB_A], na);
    if (nb) atomicAdd(&hist[SUB_B], nb);
  }
  if (wrap) hist[SUB_WRAP] = 1;
  if (capped) atomicOr(&st.status, ST_UF_CAP);
  __syncthreads();
  for (u32 i = tid; i < SUB_WORDS; i += nt)
    if (hist[i]) atomicAdd(set + i, hist[i]);
}

// Eight 256-thread blocks per SM (32 registers): probes are latency-bound
// union-find walks, and full occupancy hides more of that latency.
__global__ void __launch_bounds__(256, 8) k_probe(Group g, SearchCfg c, u32 probe_cap) {
  __shared__ u32 hist[SUB_WORDS];
  __shared__ u32 queue[queue_words(256)];
  __shared__ u32 last_sh;
  const u32 s = blockIdx.y, tid = threadIdx.x;
  SampleState& st = g.st[s];
  if (st.sdone) return;
  Window w = st.w;
  if (w.ready) return;
  u32* set = region_of(g, g.ehist, s) + EHIST;
  probe_body(g, s, Team{blockIdx.x, gridDim.x}, w, hist, *reinterpret_cast<EdgeQueue*>(queue), set);
  __threadfence();
  __syncthreads();
  if (tid == 0) last_sh = atomicAdd(&st.ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last_sh) return;
  __threadfence();
  if (tid < 32) {
    u32 status = __ldcg(&st.status);
    const bool end = probe_step(w, set, c.win_cap, probe_cap, status);
    if (tid == 0) {
      st.ticket = 0;
      st.w = w;
      st.status = status;
      if (end) st.sdone = 1;
    }
  }
  __syncthreads();
  for (u32 i = tid; i < SUB_WORDS; i += 256) set[i] = 0;
}

// The edges of the last window between the roots they join.  Edges inside one
// root without mismatch can close no wrap and are left out.
__device__ void collect_body(const Group& g, const SearchCfg& c, u32 s, Team team,
                             const Window& w, EdgeQueue& q) {
  SampleState& st = g.st[s];
  const u64 lo = w.lo, hi = w.hi;
  const u32 ne = min(st.n_edges, g.edge_limit);
  u64* W = region_of(g, g.uf, s) + (size_t)w.cur * g.cap_nodes;
  const u64* E = region_of(g, g.etime, s);
  const uint4* K = region_of(g, g.elink, s);
  WinEdge* out = region_of(g, g.win, s);
  bool capped = false;
  scan_packed(
      ne, team, q, [&](u32 i) { return E[i] > lo && E[i] <= hi; },
      [&](u32 i) {
        const uint4 e = K[i];
        WinEdge we;
        we.time = E[i];
        we.r1 = e.x;
        we.r2 = e.y;
        we.dxy = e.z;
        we.pad = 0;
        if (lo) {
          u32 ax, ay, bx, by;
          we.r1 = uf_find(W, e.x, &ax, &ay, &capped, g.uf_cap);
          we.r2 = uf_find(W, e.y, &bx, &by, &capped, g.uf_cap);
          we.dxy = ((ax + e.z - bx) & 0xFFFFu) | ((ay + (e.z >> 16) - by) << 16);
          if (we.r1 == we.r2 && we.dxy == 0) return;
        }
        const u32 at = atomicAdd(&st.win_n, 1u);
        if (at < c.win_cap) out[at] = we;
      });
  if (capped) atomicOr(&st.status, ST_UF_CAP);
}

__global__ void __launch_bounds__(256) k_collect(Group g, SearchCfg c) {
  const u32 s = blockIdx.y;
  if (g.st[s].sdone) return;
  const Window w = g.st[s].w;
  __shared__ u32 queue[queue_words(256)];
  if (w.ready)
    collect_body(g, c, s, Team{blockIdx.x, gridDim.x}, w, *reinterpret_cast<EdgeQueue*>(queue));
}

__device__ __forceinline__ bool fin_union(u64* W, u32 m1, u32 m2, u32 dxy, bool* capped, u32 cap,
                                          u32* mis = nullptr) {
  for (u32 it = 0; it < cap; ++it) {
    u32 ax, ay, bx, by;
    const u32 r1 = find_root<false>(W, m1, &ax, &ay, capped, cap);
    const u32 r2 = find_root<false>(W, m2, &bx, &by, capped, cap);
    if (*capped) return false;
    const u32 Dx = ax + dxy - bx, Dy = ay + (dxy >> 16) - by;
    if (r1 == r2) {
      if (mis) *mis = (Dx & 0xFFFFu) | ((Dy & 0xFFFFu) << 16);
      return ((Dx | Dy) & 0xFFFFu) != 0;
    }
    const u32 hi = r1 < r2 ? r2 : r1;
    const u64 want = uf_pack(hi, 0, 0);
    const u64 link = r1 < r2 ? uf_pack(r1, Dx, Dy) : uf_pack(r2, 0u - Dx, 0u - Dy);
    if (atomicCAS(W + hi, want, link) == want) return false;
  }
  *capped = true;
  return false;
}

// Shared memory of finish_body: two arrays of union-find words (the hash
// table before them), then per edge its time, displacement and two ids, and a
// list of edges.
__host__ __device__ inline size_t finish_smem(const SearchCfg& c) {
  return ((c.hashed ? (size_t)FIN_SLOTS * 4 : (size_t)c.ids * 8)) * 2 + (size_t)c.win_cap * 18;
}
constexpr size_t FIN_SMEM_MAX = (size_t)FIN_SLOTS * 8 + (size_t)FIN_EDGES * 18;  // 2 FIN_EDGES ids
constexpr u32 FIN_LAST = 32;  // edges united one after another in the end

struct FinishSmem {
  u32 set[SUB_WORDS];
  u32 wsum[34];
  u32 count, flag;
  u16 list[FIN_LAST];
  Window w;
  u32 status;
};

// The rest of the search by one block: probes as before on the edges in
// shared memory, halving the window by sub-bins, and once FIN_LAST edges are
// left these in the order of their times until one closes a wrap.  (Sorting
// the edges for an exact bisection took longer than the probes themselves.)
// Thread 0 writes the sample's results.
__device__ void finish_body(const Group& g, const SearchCfg& c, u32 s, const Window& w0,
                            u32 probe_cap, unsigned char* smem, FinishSmem& fs) {
  const u32 tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  SampleState& st = g.st[s];
  const size_t words = c.hashed ? (size_t)FIN_SLOTS * 4 : (size_t)c.ids * 8;
  u64* ua = reinterpret_cast<u64*>(smem);                 // working copy
  u64* ub = reinterpret_cast<u64*>(smem + words);         // state at lo
  u32* slots = reinterpret_cast<u32*>(smem);
  u64* tm = reinterpret_cast<u64*>(smem + 2 * words);     // by edge: time,
  u32* dxy = reinterpret_cast<u32*>(tm + c.win_cap);      // displacement,
  u32* ends = dxy + c.win_cap;                            // two 16-bit ids
  u16* todo = reinterpret_cast<u16*>(ends + c.win_cap);   // edges of this probe, packed
  const u32 n = min(st.win_n, c.win_cap);
  const WinEdge* in = region_of(g, g.win, s);
  u32 nid = min(st.n_nodes, g.cap_nodes);
  if (c.hashed)
    for (u32 i = tid; i < FIN_SLOTS; i += nt) slots[i] = NONE32;
  for (u32 i = tid; i < SUB_WORDS; i += nt) fs.set[i] = 0;
  if (tid == 0) {
    fs.w = w0;
    fs.w.ready = 0;
    fs.status = st.status;
    fs.flag = 0;
    fs.count = 0;
  }
  __syncthreads();
  // the first threshold, unless one is set: the middle of the window's edges
  const bool whole = w0.lo == 0 && w0.mid > 0 && w0.mid < w0.hi;
  const u32 shift0 = sub_shift(w0);
  for (u32 i = tid; i < n; i += nt) {
    const WinEdge e = in[i];
    tm[i] = e.time;
    dxy[i] = e.dxy;
    if (!whole) atomicAdd(&fs.set[(u32)((e.time - w0.lo - 1) >> shift0)], 1u);
    u32 id[2] = {e.r1, e.r2};
    if (c.hashed) {
#pragma unroll
      for (u32 j = 0; j < 2; ++j) {
        // at most 2 n <= FIN_SLOTS / 2 roots, so a free slot is met
        u32 q = ((id[j] * 0x9E3779B1u) >> 16) & (FIN_SLOTS - 1);
        for (u32 guard = 0; guard < FIN_SLOTS; ++guard, q = (q + 1) & (FIN_SLOTS - 1)) {
          const u32 was = atomicCAS(&slots[q], NONE32, id[j]);
          if (was == NONE32 || was == id[j]) break;
        }
        id[j] = q;
      }
    }
    ends[i] = id[0] | (id[1] << 16);
  }
  __syncthreads();
  if (c.hashed) {
    // number the slots in use
    const u32 per = (FIN_SLOTS + nt - 1) / nt, a = min(tid * per, FIN_SLOTS),
              b = min(a + per, FIN_SLOTS);
    u32 used = 0;
    for (u32 i = a; i < b; ++i) used += slots[i] != NONE32;
    u32 pre = used;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 o = __shfl_up_sync(FULL, pre, d);
      if ((int)lane >= d) pre += o;
    }
    if (lane == 31) fs.wsum[warp] = pre;
    __syncthreads();
    u32 at = pre - used;
    nid = 0;
    for (u32 q = 0; q < nwarp; ++q) {
      if (q < warp) at += fs.wsum[q];
      nid += fs.wsum[q];
    }
    for (u32 i = a; i < b; ++i)
      if (slots[i] != NONE32) slots[i] = at++;
    __syncthreads();
    for (u32 i = tid; i < n; i += nt)
      ends[i] = slots[ends[i] & 0xFFFFu] | (slots[ends[i] >> 16] << 16);
    __syncthreads();
  }
  for (u32 i = tid; i < nid; i += nt) ub[i] = uf_pack(i, 0, 0);
  if (tid < 32) {
    Window w = fs.w;
    if (n <= FIN_LAST || one_time(w)) w.ready = 1;
    else if (!whole) w.mid = next_threshold(w, w.lo, shift0, fs.set, n);
    if (tid == 0) fs.w = w;
  }
  __syncthreads();
  for (;;) {
    const Window w = fs.w;
    if (w.ready || fs.flag || (fs.status & ST_UF_CAP)) break;
    if (w.probes >= probe_cap) {
      __syncthreads();
      if (tid == 0) {
        fs.status |= ST_SEARCH_CAP;
        fs.flag = 1;
      }
      __syncthreads();
      break;
    }
    bool wrap = false, capped = false;
    for (u32 i = tid; i < nid; i += nt) {
      const u64 v = flat_word(ub, i, g.uf_cap, &capped);
      ub[i] = v;
      ua[i] = v;
    }
    for (u32 i = tid; i < SUB_WORDS; i += nt) fs.set[i] = 0;
    if (tid == 0) fs.count = 0;
    __syncthreads();
    const u32 shift = sub_shift(w);
    u32 na = 0, nb = 0;
    for (u32 i0 = 0; i0 < n; i0 += nt) {
      const u32 i = i0 + tid;
      const u64 t = i < n ? tm[i] : 0;
      const bool in_w = i < n && t > w.lo && t <= w.hi, now = in_w && t <= w.mid;
      if (in_w) atomicAdd(&fs.set[(u32)((t - w.lo - 1) >> shift)], 1u);
      const u32 at = warp_append(&fs.count, now);
      if (now) todo[at] = (u16)i;
      na += now;
      nb += in_w && !now;
    }
    na = __reduce_add_sync(FULL, na);
    nb = __reduce_add_sync(FULL, nb);
    if (lane == 0) {
      if (na) atomicAdd(&fs.set[SUB_A], na);
      if (nb) atomicAdd(&fs.set[SUB_B], nb);
    }
    __syncthreads();
    for (u32 q = tid; q < fs.count; q += nt) {
      const u32 e = todo[q];
      if (fin_union(ua, ends[e] & 0xFFFFu, ends[e] >> 16, dxy[e], &capped, g.uf_cap)) wrap = true;
    }
    if (wrap) fs.set[SUB_WRAP] = 1;
    if (capped) atomicOr(&fs.status, ST_UF_CAP);
    __syncthreads();
    const bool wrapped = fs.set[SUB_WRAP] != 0;
    if (tid < 32) {
      Window x = w;
      u32 status = fs.status;
      const bool end = probe_step(x, fs.set, FIN_LAST, probe_cap, status);
      __syncwarp();
      if (tid == 0) {
        fs.w = x;
        fs.status = status;
        fs.flag = end;
      }
    }
    __syncthreads();
    if (!wrapped) {
      u64* t = ua;
      ua = ub;
      ub = t;
    }
  }
  const Window w = fs.w;
  const bool go = w.ready && !fs.flag && !(fs.status & ST_UF_CAP);
  if (tid == 0) fs.count = 0;
  __syncthreads();
  if (go)
    for (u32 i = tid; i < n; i += nt)
      if (tm[i] > w.lo && tm[i] <= w.hi) {
        const u32 at = atomicAdd(&fs.count, 1u);
        if (at < FIN_LAST) fs.list[at] = (u16)i;
      }
  __syncthreads();
  if (warp == 0) {
    u32 status = fs.status, probes = w.probes;
    u64 tc = 0;
    if (go && one_time(w)) {
      tc = w.hi;
    } else if (go && probes >= probe_cap) {
      status |= ST_SEARCH_CAP;
    } else if (go) {
      ++probes;
      const u32 m = min(fs.count, FIN_LAST);
      const u32 mine = lane < m ? fs.list[lane] : 0u;
      const u64 t = lane < m ? tm[mine] : KEY_NONE;
      u32 rank = 0;
      for (u32 i = 0; i < 32; ++i) {
        const u64 o = __shfl_sync(FULL, t, i);
        rank += o < t || (o == t && i < lane);
      }
      if (lane < m) fs.list[rank] = (u16)mine;
      __syncwarp();
      if (lane == 0) {
        bool capped = false;
        u32 i = 0;
        for (; i < m && !capped; ++i) {
          const u32 e = fs.list[i];
          if (fin_union(ub, ends[e] & 0xFFFFu, ends[e] >> 16, dxy[e], &capped, g.uf_cap)) {
            tc = tm[e];
            break;
          }
        }
        if (capped) status |= ST_UF_CAP;
        else if (i == m) status |= ST_NOWRAP;
      }
    }
    if (lane == 0) {
      st.status = status;
      st.w.probes = probes;
      st.sdone = 1;
      if (tc) {
        st.tc = tc;
        st.nc = 0;
        st.ranked = 1;
      }
    }
  }
}

__global__ void __launch_bounds__(FIN_THREADS) k_finish(Group g, SearchCfg c, u32 probe_cap,
                                                        u32* n_open) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FinishSmem fs;
  const u32 s = blockIdx.x, tid = threadIdx.x;
  SampleState& st = g.st[s];
  if (st.sdone) {
    if (tid == 0 && st.ranked == 1) st.ranked = 2;
    return;
  }
  const Window w = st.w;
  __syncthreads();
  if (!w.ready) {
    if (tid == 0) atomicAdd(n_open, 1u);
    return;
  }
  finish_body(g, c, s, w, probe_cap, smem_raw, fs);
}

// n_c: the k-mers of priority <= T_c.
__device__ __forceinline__ void rank_body(const Group& g, u32 s, Team team) {
  SampleState& st = g.st[s];
  const u64 T = st.tc;
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  const u32 nn = min(st.n_nodes, g.cap_nodes), nt = blockDim.x;
  u32 cnt = 0;
  for (u32 i = team.rank * nt + threadIdx.x; i < nn; i += team.size * nt) cnt += K[i] <= T;
  cnt = __reduce_add_sync(FULL, cnt);
  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&st.nc, cnt);
}

__global__ void __launch_bounds__(256) k_rank(Group g) {
  if (g.st[blockIdx.y].ranked == 1) rank_body(g, blockIdx.y, Team{blockIdx.x, gridDim.x});
}

}  // namespace rsak
