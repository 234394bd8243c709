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
//   k_collect  once the window holds at most FIN_EDGES edges: those, with
//              the roots of their ends and the displacement between the roots;
//   k_finish   one block per sample: these edges sorted by time in shared
//              memory and the rest of the bisection there, on the graph of
//              the roots;
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
constexpr u32 FIN_THREADS = 512;
constexpr u32 FIN_SLOTS = 4 * FIN_EDGES;  // hash slots for the roots of the window (4 B: as much
                                          // as 2 FIN_EDGES union-find words)
constexpr u32 SUB_BINS = 128;

struct WinEdge {  // an edge of the last window, between roots
  u64 time;
  u32 r1, r2, dxy, pad;
};

struct SearchCfg {
  u32 win_cap;      // window edges stored per sample, <= FIN_EDGES
  u32 hashed;       // roots are renumbered through a hash table (else: node ids)
  u32 ids;          // union-find words in shared memory
  u32 q0, q1;       // first two thresholds, edge quantiles in 1/65536
};

// Root of x and x's offset from it.  Path halving by CAS; a failed CAS is
// harmless because every stored (parent, offset) pair stays a true ancestor
// relation.  Loads bypass L1 (other SMs write these words).
__device__ __forceinline__ u32 uf_find(u64* W, u32 x, u32* ox, u32* oy, bool* capped, u32 cap) {
  u32 sx = 0, sy = 0;
  for (u32 it = 0; it < cap; ++it) {
    const u64 wx = __ldcg(W + x);
    const u32 p = (u32)wx;
    if (p == x) {
      *ox = sx;
      *oy = sy;
      return x;
    }
    const u64 wp = __ldcg(W + p);
    const u32 gp = (u32)wp;
    if (gp != p) {
      const u64 nw = uf_pack(gp, (u32)(wx >> 32) + (u32)(wp >> 32),
                             (u32)(wx >> 48) + (u32)(wp >> 48));
      atomicCAS(W + x, wx, nw);
    }
    sx += (u32)(wx >> 32);
    sy += (u32)(wx >> 48);
    x = p;
  }
  *capped = true;
  *ox = sx;
  *oy = sy;
  return x;
}

// Add edge "anchor(m2) = anchor(m1) + d"; returns true if it closes a cycle
// of non-zero winding, and then, if mis is given, stores the cycle's lifted
// mismatch (x in bits 0-15, y in 16-31, modulo 2^16).  Roots are linked
// larger-id under smaller-id, so the forest stays acyclic under concurrent
// unions.
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

// Start of the search of one batch; while a sample of it is still being
// deposited (*n_active) nothing of it runs.
__global__ void k_graph_init(Group g, const u32* n_active) {
  const u32 s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.n) return;
  SampleState& st = g.st[s];
  st.n_edges = 0;
  st.contacts_x = st.contacts_y = st.contacts_xy = 0;
  st.lo = 0;
  st.hi = KEY_NONE;
  st.mid = 0;
  st.hi_ok = 0;
  st.ready = 0;
  st.step = 0;
  st.wrap = 0;
  st.cur = 0;
  st.count_a = st.count_b = 0;
  st.ticket = 0;
  st.win_n = 0;
  st.ranked = 0;
  st.nc = NONE32;
  st.probes = 0;
  st.sdone = (*n_active || (st.status & (ST_NODE_OVF | ST_ROUND_CAP))) ? 1u : 0u;
}

// After the contacts: one block per sample.  Few edges: straight to the last
// window.  Otherwise the first two thresholds from the histogram of times.
__global__ void __launch_bounds__(256) k_search_init(Group g, SearchCfg c) {
  __shared__ u32 part[256];
  const u32 s = blockIdx.x, tid = threadIdx.x;
  SampleState& st = g.st[s];
  if (st.sdone) return;
  if (st.status & ST_EDGE_OVF) {
    __syncthreads();
    if (tid == 0) st.sdone = 1;
    return;
  }
  const u32 ne = st.n_edges;
  if (ne <= c.win_cap) {
    if (tid == 0) st.ready = 1;
    return;
  }
  u32* h = g.ehist + (size_t)s * (EHIST + SUB_BINS);
  constexpr u32 PER = EHIST / 256;
  u32 v[PER], sum = 0;
#pragma unroll
  for (u32 i = 0; i < PER; ++i) {
    v[i] = h[tid * PER + i];
    sum += v[i];
  }
  part[tid] = sum;
  if (tid < SUB_BINS) h[EHIST + tid] = 0;
  __syncthreads();
  for (u32 d = 1; d < 256; d <<= 1) {
    const u32 o = tid >= d ? part[tid - d] : 0u;
    __syncthreads();
    part[tid] += o;
    __syncthreads();
  }
  // the bin in which each quantile falls ends at the threshold
  const u32 r0 = (u32)((u64)ne * c.q0 >> 16), r1 = (u32)((u64)ne * c.q1 >> 16);
  u32 a = part[tid] - sum;
#pragma unroll
  for (u32 i = 0; i < PER; ++i) {
    const u32 b = a + v[i];
    const u64 top = tid * PER + i + 1 < EHIST ? bin_floor(tid * PER + i + 1) - 1 : KEY_NONE - 1;
    if (a <= r0 && r0 < b) st.mid = top;
    if (a <= r1 && r1 < b) st.next_mid = top;
    a = b;
  }
  if (tid == 0) st.in_win = ne;
}

// Working copy of the union-find state at lo (single k-mers while lo = 0).
__global__ void __launch_bounds__(256) k_probe_copy(Group g) {
  const u32 s = blockIdx.y;
  const SampleState& st = g.st[s];
  if (st.sdone || st.ready) return;
  const u32 nn = min(st.n_nodes, g.cap_nodes);
  const bool fresh = st.lo == 0;
  const u64* S = g.uf + ((size_t)s * 2 + st.cur) * g.cap_nodes;
  u64* Wd = g.uf + ((size_t)s * 2 + (st.cur ^ 1u)) * g.cap_nodes;
  for (u32 m = blockIdx.x * blockDim.x + threadIdx.x; m < nn; m += gridDim.x * blockDim.x)
    Wd[m] = fresh ? uf_pack(m, 0, 0) : S[m];
}

// The step from one probe to the next (one thread per sample).
__device__ void probe_step(SampleState& st, u32* sub, u32 shift, u32 win_cap, u32 probe_cap) {
  st.probes += 1;
  const u64 lo0 = st.lo;
  const bool w = st.wrap != 0, first = st.step == 0;
  st.wrap = 0;
  st.step = 1;
  if (st.status & ST_UF_CAP) {
    st.sdone = 1;
    return;
  }
  if (w) {
    st.hi = st.mid;
    st.hi_ok = 1;
  } else {
    st.lo = st.mid;
    st.cur ^= 1u;
  }
  const u32 in = w ? st.count_a : st.count_b;
  st.in_win = in;
  st.count_a = st.count_b = 0;
  if (in <= win_cap) {
    st.ready = 1;
  } else if (st.probes >= probe_cap) {
    st.status |= ST_SEARCH_CAP;
    st.sdone = 1;
  } else {
    u64 mid = 0;
    if (first && !w && st.next_mid > st.lo && st.next_mid < st.hi) {
      mid = st.next_mid;
    } else {
      // halve the window's edges at a sub-bin boundary
      u32 sum = 0;
      for (u32 b = 0; b < SUB_BINS; ++b) {
        const u64 first_t = lo0 + 1 + ((u64)b << shift);
        const u64 last_t = first_t + ((1ull << shift) - 1);
        if (last_t <= st.lo || first_t > st.hi) continue;
        sum += sub[b];
        mid = last_t;
        if (sum >= in / 2) break;
      }
      if (mid <= st.lo || mid >= st.hi) mid = st.lo + (st.hi - st.lo) / 2;
    }
    st.mid = mid;
  }
  for (u32 b = 0; b < SUB_BINS; ++b) sub[b] = 0;
}

// Eight 256-thread blocks per SM (32 registers): probes are latency-bound
// union-find walks, and full occupancy hides more of that latency.
__global__ void __launch_bounds__(256, 8) k_probe(Group g, SearchCfg c, u32 probe_cap) {
  __shared__ u32 hist[SUB_BINS];
  __shared__ u32 na_sh, nb_sh;
  const u32 s = blockIdx.y, tid = threadIdx.x;
  SampleState& st = g.st[s];
  if (st.sdone || st.ready) return;
  const u64 lo = st.lo, mid = st.mid, hi = st.hi;
  // sub-bins of the window (lo, hi], as many as fit SUB_BINS
  const u64 span = hi - lo - 1;
  const u32 width = 64 - __clzll((long long)span), shift = width > 7 ? width - 7 : 0;
  const u32 ne = min(st.n_edges, g.edge_limit);
  if (tid < SUB_BINS) hist[tid] = 0;
  if (tid == 0) na_sh = nb_sh = 0;
  __syncthreads();
  u64* Wd = g.uf + ((size_t)s * 2 + (st.cur ^ 1u)) * g.cap_nodes;
  const u64* E = g.etime + (size_t)s * g.cap_edges;
  const uint4* K = g.elink + (size_t)s * g.cap_edges;
  bool wrap = false, capped = false;
  u32 na = 0, nb = 0;
  for (u32 i = blockIdx.x * 256 + tid; i < ne; i += gridDim.x * 256) {
    const u64 t = E[i];
    if (t <= lo || t > hi) continue;
    atomicAdd(&hist[(u32)((t - lo - 1) >> shift)], 1u);
    if (t > mid) {
      ++nb;
      continue;
    }
    ++na;
    const uint4 e = K[i];
    if (uf_union(Wd, e.x, e.y, e.z, &capped, g.uf_cap)) wrap = true;
  }
  na = __reduce_add_sync(FULL, na);
  nb = __reduce_add_sync(FULL, nb);
  if ((tid & 31) == 0) {
    if (na) atomicAdd(&na_sh, na);
    if (nb) atomicAdd(&nb_sh, nb);
  }
  const bool bw = __syncthreads_or(wrap);
  const bool bc = __syncthreads_or(capped);
  u32* sub = g.ehist + (size_t)s * (EHIST + SUB_BINS) + EHIST;
  if (tid < SUB_BINS && hist[tid]) atomicAdd(&sub[tid], hist[tid]);
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    if (bw) atomicOr(&st.wrap, 1u);
    if (bc) atomicOr(&st.status, ST_UF_CAP);
    if (na_sh) atomicAdd(&st.count_a, na_sh);
    if (nb_sh) atomicAdd(&st.count_b, nb_sh);
    __threadfence();
    if (atomicAdd(&st.ticket, 1u) == gridDim.x - 1) {
      __threadfence();
      st.ticket = 0;
      st.wrap = __ldcg(&st.wrap);
      st.status = __ldcg(&st.status);
      st.count_a = __ldcg(&st.count_a);
      st.count_b = __ldcg(&st.count_b);
      probe_step(st, sub, shift, c.win_cap, probe_cap);
    }
  }
}

// The edges of the last window between the roots they join.  Edges inside one
// root without mismatch can close no wrap and are left out.
__global__ void __launch_bounds__(256) k_collect(Group g, SearchCfg c) {
  const u32 s = blockIdx.y;
  SampleState& st = g.st[s];
  if (st.sdone || !st.ready) return;
  const u64 lo = st.lo, hi = st.hi;
  const u32 ne = min(st.n_edges, g.edge_limit);
  u64* W = g.uf + ((size_t)s * 2 + st.cur) * g.cap_nodes;
  const u64* E = g.etime + (size_t)s * g.cap_edges;
  const uint4* K = g.elink + (size_t)s * g.cap_edges;
  WinEdge* out = g.win + (size_t)s * c.win_cap;
  bool capped = false;
  for (u32 i = blockIdx.x * 256 + threadIdx.x; i < ne; i += gridDim.x * 256) {
    const u64 t = E[i];
    if (t <= lo || t > hi) continue;
    const uint4 e = K[i];
    WinEdge w;
    w.time = t;
    w.r1 = e.x;
    w.r2 = e.y;
    w.dxy = e.z;
    w.pad = 0;
    if (lo) {
      u32 ax, ay, bx, by;
      w.r1 = uf_find(W, e.x, &ax, &ay, &capped, g.uf_cap);
      w.r2 = uf_find(W, e.y, &bx, &by, &capped, g.uf_cap);
      w.dxy = ((ax + e.z - bx) & 0xFFFFu) | ((ay + (e.z >> 16) - by) << 16);
      if (w.r1 == w.r2 && w.dxy == 0) continue;
    }
    const u32 at = atomicAdd(&st.win_n, 1u);
    if (at < c.win_cap) out[at] = w;
  }
  if (capped) atomicOr(&st.status, ST_UF_CAP);
}

// Root of x on shared-memory words, with path halving as in uf_find.
__device__ __forceinline__ u32 fin_find(u64* W, u32 x, u32* ox, u32* oy, bool* capped, u32 cap) {
  u32 sx = 0, sy = 0;
  for (u32 it = 0; it < cap; ++it) {
    const u64 wx = *(volatile u64*)(W + x);
    const u32 p = (u32)wx;
    if (p == x) {
      *ox = sx;
      *oy = sy;
      return x;
    }
    const u64 wp = *(volatile u64*)(W + p);
    const u32 gp = (u32)wp;
    if (gp != p)
      atomicCAS(W + x, wx, uf_pack(gp, (u32)(wx >> 32) + (u32)(wp >> 32),
                                   (u32)(wx >> 48) + (u32)(wp >> 48)));
    sx += (u32)(wx >> 32);
    sy += (u32)(wx >> 48);
    x = p;
  }
  *capped = true;
  *ox = sx;
  *oy = sy;
  return x;
}

__device__ __forceinline__ bool fin_union(u64* W, u32 m1, u32 m2, u32 dxy, bool* capped, u32 cap) {
  for (u32 it = 0; it < cap; ++it) {
    u32 ax, ay, bx, by;
    const u32 r1 = fin_find(W, m1, &ax, &ay, capped, cap);
    const u32 r2 = fin_find(W, m2, &bx, &by, capped, cap);
    if (*capped) return false;
    const u32 Dx = ax + dxy - bx, Dy = ay + (dxy >> 16) - by;
    if (r1 == r2) return ((Dx | Dy) & 0xFFFFu) != 0;
    const u32 hi = r1 < r2 ? r2 : r1;
    const u64 want = uf_pack(hi, 0, 0);
    const u64 link = r1 < r2 ? uf_pack(r1, Dx, Dy) : uf_pack(r2, 0u - Dx, 0u - Dy);
    if (atomicCAS(W + hi, want, link) == want) return false;
  }
  *capped = true;
  return false;
}

__host__ __device__ inline size_t finish_smem(const SearchCfg& c, u32 pow2) {
  // union-find words (as large as the hash table they follow), then per edge
  // its time, displacement, two ids, place in the order and end of a time
  return (c.hashed ? (size_t)FIN_SLOTS * 4 : (size_t)c.ids * 8) + (size_t)pow2 * 20;
}

constexpr size_t FIN_SMEM_MAX = (size_t)FIN_SLOTS * 4 + (size_t)FIN_EDGES * 20;  // 2 FIN_EDGES ids

// The rest of the search in one block's shared memory.  pow2: win_cap rounded
// up to a power of two.
__global__ void __launch_bounds__(FIN_THREADS) k_finish(Group g, SearchCfg c, u32 pow2,
                                                        u32 probe_cap, u32* n_open) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ u32 wsum[FIN_THREADS / 32 + 1];
  __shared__ u32 ndist_sh;
  const u32 s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  SampleState& st = g.st[s];
  if (st.sdone) {
    if (tid == 0 && st.ranked == 1) st.ranked = 2;
    return;
  }
  if (!st.ready) {
    if (tid == 0) atomicAdd(n_open, 1u);
    return;
  }
  u64* uf = reinterpret_cast<u64*>(smem_raw);             // and, before, the hash table
  u32* slots = reinterpret_cast<u32*>(smem_raw);
  const size_t words = finish_smem(c, 0);
  u64* tm = reinterpret_cast<u64*>(smem_raw + words);     // times, sorted
  u32* dxy = reinterpret_cast<u32*>(tm + pow2);           // by edge
  u32* ends = dxy + pow2;                                 // by edge: two 16-bit ids
  u16* ord = reinterpret_cast<u16*>(ends + pow2);         // edge of each sorted time
  u16* last = ord + pow2;                                 // last position of each distinct time
  const u32 n = min(st.win_n, c.win_cap);
  const WinEdge* in = g.win + (size_t)s * c.win_cap;
  u32 P2 = 1;
  while (P2 < n) P2 <<= 1;
  u32 nid = min(st.n_nodes, g.cap_nodes);
  if (c.hashed) {
    for (u32 i = tid; i < FIN_SLOTS; i += FIN_THREADS) slots[i] = NONE32;
    __syncthreads();
  }
  for (u32 i = tid; i < P2; i += FIN_THREADS) {
    u64 t = KEY_NONE;
    if (i < n) {
      const WinEdge w = in[i];
      t = w.time;
      dxy[i] = w.dxy;
      u32 id[2] = {w.r1, w.r2};
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
    tm[i] = t;
    ord[i] = (u16)i;
  }
  __syncthreads();
  if (c.hashed) {
    // number the slots in use
    constexpr u32 PER = FIN_SLOTS / FIN_THREADS;
    u32 used = 0;
    for (u32 i = 0; i < PER; ++i) used += slots[tid * PER + i] != NONE32;
    u32 pre = used;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 o = __shfl_up_sync(FULL, pre, d);
      if ((int)lane >= d) pre += o;
    }
    if (lane == 31) wsum[warp] = pre;
    __syncthreads();
    u32 at = pre - used;
    for (u32 w = 0; w < warp; ++w) at += wsum[w];
    for (u32 i = 0; i < PER; ++i)
      if (slots[tid * PER + i] != NONE32) slots[tid * PER + i] = at++;
    nid = 0;
    for (u32 w = 0; w < FIN_THREADS / 32; ++w) nid += wsum[w];
    __syncthreads();
    for (u32 i = tid; i < n; i += FIN_THREADS)
      ends[i] = slots[ends[i] & 0xFFFFu] | (slots[ends[i] >> 16] << 16);
    __syncthreads();
  }
  // bitonic sort of the times with their edges
  for (u32 kk = 2; kk <= P2; kk <<= 1)
    for (u32 j = kk >> 1; j > 0; j >>= 1) {
      for (u32 q = tid; q < P2 / 2; q += FIN_THREADS) {
        const u32 i = 2 * q - (q & (j - 1)), p = i + j;
        const u64 a = tm[i], b = tm[p];
        if ((a > b) == ((i & kk) == 0)) {
          tm[i] = b;
          tm[p] = a;
          const u16 oa = ord[i];
          ord[i] = ord[p];
          ord[p] = oa;
        }
      }
      __syncthreads();
    }
  // positions where a time ends, in order
  {
    const u32 per = (n + FIN_THREADS - 1) / FIN_THREADS, a = min(tid * per, n), b = min(a + per, n);
    u32 cnt = 0;
    for (u32 i = a; i < b; ++i) cnt += i + 1 == n || tm[i] != tm[i + 1];
    u32 pre = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 o = __shfl_up_sync(FULL, pre, d);
      if ((int)lane >= d) pre += o;
    }
    if (lane == 31) wsum[warp] = pre;
    __syncthreads();
    u32 at = pre - cnt;
    for (u32 w = 0; w < warp; ++w) at += wsum[w];
    for (u32 i = a; i < b; ++i)
      if (i + 1 == n || tm[i] != tm[i + 1]) last[at++] = (u16)i;
    if (tid == FIN_THREADS - 1) ndist_sh = at;
    __syncthreads();
  }
  u32 probes = st.probes, status = st.status;
  // wrap after the first `m` distinct times of the window
  auto probe = [&](u32 m, bool* capped_out) -> bool {
    for (u32 i = tid; i < nid; i += FIN_THREADS) uf[i] = uf_pack(i, 0, 0);
    __syncthreads();
    bool wrap = false, capped = false;
    const u32 e1 = (u32)last[m - 1] + 1;
    for (u32 i = tid; i < e1; i += FIN_THREADS) {
      const u32 e = ord[i], ab = ends[e];
      if (fin_union(uf, ab & 0xFFFFu, ab >> 16, dxy[e], &capped, g.uf_cap)) wrap = true;
    }
    *capped_out = __syncthreads_or(capped);
    return __syncthreads_or(wrap);
  };
  u32 lo = 0, hi = ndist_sh;  // wrap(lo) is false; wrap(hi) if hi_ok
  bool hi_ok = st.hi_ok != 0, capped = (status & ST_UF_CAP) != 0, over = false;
  if (hi == 0) status |= ST_NOWRAP;  // no edge left that could close a wrap
  while (hi > 0 && !capped && !(hi - lo == 1 && hi_ok)) {
    if (probes >= probe_cap) {
      over = true;
      break;
    }
    ++probes;
    const u32 mid = hi - lo == 1 ? hi : lo + (hi - lo) / 2;
    if (probe(mid, &capped)) {
      hi = mid;
      hi_ok = true;
    } else if (mid == hi) {
      if (!capped) status |= ST_NOWRAP;
      break;
    } else {
      lo = mid;
    }
  }
  if (tid == 0) {
    if (capped) status |= ST_UF_CAP;
    if (over) status |= ST_SEARCH_CAP;
    st.status = status;
    st.probes = probes;
    st.sdone = 1;
    if (hi > 0 && !(status & (ST_UF_CAP | ST_SEARCH_CAP | ST_NOWRAP))) {
      st.tc = tm[last[hi - 1]];
      st.nc = 0;
      st.ranked = 1;
    }
  }
}

// n_c: the k-mers of priority <= T_c.
__global__ void __launch_bounds__(256) k_rank(Group g) {
  const u32 s = blockIdx.y;
  SampleState& st = g.st[s];
  if (st.ranked != 1) return;
  const u64 T = st.tc;
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  const u32 nn = min(st.n_nodes, g.cap_nodes);
  u32 cnt = 0;
  for (u32 i = blockIdx.x * 256 + threadIdx.x; i < nn; i += gridDim.x * 256) cnt += K[i] <= T;
  cnt = __reduce_add_sync(FULL, cnt);
  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&st.nc, cnt);
}

}  // namespace rsak
