// rsa_kernels.cuh -- round, contact-graph and bisection kernels (sm_103a).
#pragma once
#include "rsa_device.cuh"

namespace rsak {

// Per-sample set-up: stream base from the seed, state cleared.
__global__ void k_init(Group g, const u64* seeds) {
  const u32 s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.n) return;
  g.base[s] = mix64(seeds[s] + SM_GAMMA);
  SampleState z = {};
  g.st[s] = z;
}

// Group one sample's edges by time >> 56 and its node keys by key >> 56
// (counting sort into NBKT buckets), so that a bisection probe touches only
// the edges whose time can lie in its window.  One block per sample.
__global__ void __launch_bounds__(1024) k_bucket(Group g) {
  __shared__ u32 he[NBKT], hn[NBKT], ce[NBKT], cn[NBKT];
  const u32 s = blockIdx.x;
  SampleState& st = g.st[s];
  const u32 ne = min(st.n_edges, g.edge_limit), nn = min(st.n_nodes, g.cap_nodes);
  const Edge* E = g.edges + (size_t)s * g.cap_edges;
  Edge* E2 = g.edges_b + (size_t)s * g.cap_edges;
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  u64* K2 = g.nkey_b + (size_t)s * g.cap_nodes;
  u32* eb = g.ebkt + (size_t)s * (NBKT + 1);
  u32* nb = g.nbkt + (size_t)s * (NBKT + 1);
  for (u32 i = threadIdx.x; i < NBKT; i += blockDim.x) he[i] = hn[i] = 0;
  __syncthreads();
  for (u32 i = threadIdx.x; i < ne; i += blockDim.x) atomicAdd(&he[(u32)(E[i].time >> 56)], 1u);
  for (u32 i = threadIdx.x; i < nn; i += blockDim.x) atomicAdd(&hn[(u32)(K[i] >> 56)], 1u);
  __syncthreads();
  if (threadIdx.x == 0) {
    u32 a = 0, b = 0;
    for (u32 i = 0; i < NBKT; ++i) {
      eb[i] = a; ce[i] = a; a += he[i];
      nb[i] = b; cn[i] = b; b += hn[i];
    }
    eb[NBKT] = a;
    nb[NBKT] = b;
  }
  __syncthreads();
  for (u32 i = threadIdx.x; i < ne; i += blockDim.x) {
    const Edge e = E[i];
    E2[atomicAdd(&ce[(u32)(e.time >> 56)], 1u)] = e;
  }
  for (u32 i = threadIdx.x; i < nn; i += blockDim.x) {
    const u64 kk = K[i];
    K2[atomicAdd(&cn[(u32)(kk >> 56)], 1u)] = kk;
  }
}

// ---------------------------------------------------------------------
// First wrap by bisection over the number of placed k-mers (Sec. II.D).
// wrap(m): does the graph of the first m accepted k-mers (the m smallest
// keys) contain a cycle of non-zero winding?  It is monotone in m, and n_c
// is the smallest m with wrap(m).  The first probe takes every k-mer (the
// jammed lattice must wrap); later probes bisect the rank interval
// (cnt_lo, cnt_hi] and take mid = T_r, the key of rank r, so that the edges
// of a probe are those with time (the larger key of their two ends) <= T_r.
// Each probe starts from the union-find state of the last non-wrapping rank
// cnt_lo (threshold `lo`) and adds only edges with lo < time <= mid, so the
// probes after the first non-wrapping one touch a halving share of edges.  Union-find words: parent (bits 0-31) and the lifted
// offset of the node from its parent, dx (32-47), dy (48-63), modulo 2^16.
// A wrap is a cycle of primitive winding (a, b) times L; for L < 65536 its
// offset is never 0 modulo 2^16, so 16-bit offsets decide exactly.
// ---------------------------------------------------------------------

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

__global__ void k_search_init(Group g) {
  const u32 s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.n) return;
  SampleState& st = g.st[s];
  st.lo = 0;
  st.lo_valid = 0;
  st.cnt_lo = 0;
  st.hi = KEY_NONE;
  st.cnt_hi = min(st.n_nodes, g.cap_nodes);
  st.mid = KEY_NONE;  // first probe: the whole jammed lattice must wrap
  st.cnt_mid = st.cnt_hi;
  st.hi_ok = 0;
  st.cur = 0;
  st.sdone = (st.status & (ST_NODE_OVF | ST_EDGE_OVF | ST_ROUND_CAP)) ? 1u : 0u;
  st.nc = NONE32;
  st.probes = 0;
}

__global__ void k_uf_identity(Group g) {
  const u32 s = blockIdx.y;
  const u32 nn = min(g.st[s].n_nodes, g.cap_nodes);
  u64* U = g.uf + (size_t)s * 2 * g.cap_nodes;
  for (u32 m = blockIdx.x * blockDim.x + threadIdx.x; m < nn; m += gridDim.x * blockDim.x)
    U[m] = uf_pack(m, 0, 0);
}

// Working copy of the union-find state at `lo`.
__global__ void k_probe_copy(Group g) {
  const u32 s = blockIdx.y;
  SampleState& st = g.st[s];
  if (st.sdone) return;
  if (threadIdx.x == 0 && blockIdx.x == 0) st.wrap = 0;
  const u32 nn = min(st.n_nodes, g.cap_nodes);
  const u64* S = g.uf + ((size_t)s * 2 + st.cur) * g.cap_nodes;
  u64* Wd = g.uf + ((size_t)s * 2 + (st.cur ^ 1u)) * g.cap_nodes;
  for (u32 m = blockIdx.x * blockDim.x + threadIdx.x; m < nn; m += gridDim.x * blockDim.x)
    Wd[m] = S[m];
}

// Eight 256-thread blocks per SM (32 registers): probes are latency-bound
// union-find walks, and full occupancy hides more of that latency.
__global__ void __launch_bounds__(256, 8) k_probe(Group g) {
  const u32 s = blockIdx.y;
  SampleState& st = g.st[s];
  if (st.sdone) return;
  const u64 lo = st.lo, mid = st.mid;
  const bool lo_valid = st.lo_valid != 0;
  const u32* eb = g.ebkt + (size_t)s * (NBKT + 1);
  const u32 blo = lo_valid ? (u32)(lo >> 56) : 0u, bmid = (u32)(mid >> 56);
  const u32 e0 = eb[blo], e1 = eb[bmid + 1];
  u64* Wd = g.uf + ((size_t)s * 2 + (st.cur ^ 1u)) * g.cap_nodes;
  const Edge* E = g.edges_b + (size_t)s * g.cap_edges;
  bool wrap = false, capped = false;
  const u32 stride = gridDim.x * blockDim.x;
  for (u32 i = e0 + blockIdx.x * blockDim.x + threadIdx.x; i < e1; i += stride) {
    const Edge e = E[i];
    if (e.time > mid || (lo_valid && e.time <= lo)) continue;
    if (uf_union(Wd, e.m1, e.m2, e.dxy, &capped, g.uf_cap)) wrap = true;
  }
  const bool bw = __syncthreads_or(wrap);
  const bool bc = __syncthreads_or(capped);
  if (threadIdx.x == 0) {
    if (bw) atomicOr(&st.wrap, 1u);
    if (bc) atomicOr(&st.status, ST_UF_CAP);
  }
}

// One bisection step of sample s (one thread): read the probe's wrap flag,
// move lo or hi, finish or pick the next rank.  True if another probe follows.
__device__ bool search_step(Group& g, SampleState& st, u32 probe_cap, u32* n_open) {
  st.probes += 1;
  if (st.status & ST_UF_CAP) {
    st.sdone = 1;
    return false;
  }
  const bool w = st.wrap != 0;
  if (!st.hi_ok) {
    if (!w) {
      st.status |= ST_NOWRAP;
      st.nc = NONE32;
      st.sdone = 1;
      return false;
    }
    st.hi_ok = 1;
    st.cnt_hi = st.cnt_mid;
  } else if (w) {
    st.hi = st.mid;
    st.cnt_hi = st.cnt_mid;
  } else {
    st.lo = st.mid;
    st.lo_valid = 1;
    st.cnt_lo = st.cnt_mid;
    st.cur ^= 1u;
  }
  if (st.cnt_hi <= st.cnt_lo) {
    st.status |= ST_SEARCH_BAD;
    st.sdone = 1;
    return false;
  }
  if (st.cnt_hi - st.cnt_lo == 1) {
    st.nc = st.cnt_hi;
    st.sdone = 1;
    return false;
  }
  if (st.probes >= probe_cap) {
    st.status |= ST_SEARCH_CAP;
    st.sdone = 1;
    return false;
  }
  // next rank, strictly inside (cnt_lo, cnt_hi)
  st.cnt_mid = st.cnt_lo + (st.cnt_hi - st.cnt_lo) / 2;
  atomicAdd(n_open, 1u);
  return true;
}

// mid := the key of rank r (1-based) among the sample's node keys, by the
// whole block.  The keys are grouped by their top byte (k_bucket); the rank's
// bucket is found from the bucket offsets and the key inside it by an 8-bit
// radix select over the remaining 56 bits.
__device__ u64 select_rank(const Group& g, u32 s, u32 r) {
  __shared__ u32 hist[256];
  __shared__ u32 bk_sh, rank_sh;
  __shared__ u64 pre_sh;
  const u32* nb = g.nbkt + (size_t)s * (NBKT + 1);
  const u64* K = g.nkey_b + (size_t)s * g.cap_nodes;
  if (threadIdx.x == 0) bk_sh = 0;
  __syncthreads();
  for (u32 b = threadIdx.x; b < NBKT; b += blockDim.x)
    if (nb[b] < r && r <= nb[b + 1]) bk_sh = b;
  __syncthreads();
  const u32 nn = min(g.st[s].n_nodes, g.cap_nodes);
  const u32 bk = bk_sh, k0 = min(nb[bk], nn), k1 = min(nb[bk + 1], nn);
  u64 pre = (u64)bk << 56, mask = 0xFFull << 56;
  u32 rank = r - k0;
  for (int shift = 48; shift >= 0; shift -= 8) {
    for (u32 i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    for (u32 i = k0 + threadIdx.x; i < k1; i += blockDim.x) {
      const u64 kk = K[i];
      if ((kk & mask) == pre) atomicAdd(&hist[(u32)(kk >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      u32 d = 0, below = 0;
      while (d < 255 && below + hist[d] < rank) below += hist[d++];
      rank_sh = rank - below;
      pre_sh = pre | ((u64)d << shift);
    }
    __syncthreads();
    rank = rank_sh;
    pre = pre_sh;
    mask |= 255ull << shift;
    __syncthreads();
  }
  return pre;
}

// After a probe: one block per sample takes the bisection step and, if the
// search goes on, selects the key of the next rank as the next threshold.
__global__ void __launch_bounds__(256) k_search_decide(Group g, u32 probe_cap, u32* n_open) {
  __shared__ u32 go;
  const u32 s = blockIdx.x;
  SampleState& st = g.st[s];
  if (st.sdone) return;
  if (threadIdx.x == 0) go = search_step(g, st, probe_cap, n_open) ? 1u : 0u;
  __syncthreads();
  if (!go) return;
  const u64 mid = select_rank(g, s, st.cnt_mid);
  if (threadIdx.x == 0) st.mid = mid;
}

}  // namespace rsak
