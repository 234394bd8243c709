// rsa_config.cuh -- the configuration of the first m accepted k-mers of a
// finished sample (m = n_c: the percolating state, m = n_j: the jamming
// state; Sec. III "Structure of the percolating and jamming states").
//
//   cluster sizes   number of clusters made of exactly s k-mers, s = 1 .. m
//                   (s k sites each; n_s of Eq. CSD is that count over L^2);
//   winding         whether some cluster winds round the torus along x, and
//                   along y (Sec. II.D "in one or both directions").
//
// The k-mers tried first are the ones with the smallest keys, so the first m
// accepted k-mers are the nodes with key <= T_m, the m-th smallest node key,
// and the lattice edges among them are the contact-graph edges with time
// (the larger key of their two ends) <= T_m:
//   k_key_bins, k_key_select   T_m: a histogram of the keys over all blocks,
//                  then the keys of one bin and a radix select among them;
//   k_cfg_init     identity union-find, zero sizes and histogram;
//   k_cfg_union    union the edges with time <= T_m; an edge that closes a
//                  cycle of non-zero winding adds its directions;
//   k_cfg_count    k-mers per root;  k_cfg_hist  roots per size.
// A closed cycle's mismatch is its winding (a, b) times L, modulo 2^16.  The
// cycles closed while the union-find grows generate the windings of every
// cycle of the clusters, so "some closed cycle has a != 0" is "the clusters
// wind along x", whatever order the edges are united in.
// Scratch (the sample's search state is no longer needed): union-find words
// in the first half of its uf slot; sizes (u32) in the third quarter and the
// histogram (u32, entry s - 1 for size s) in the fourth; for the select, before
// these, the keys of one bin in the second half.
// A sample of few edges goes through all of it in one block (k_cfg_block): a
// call is bound by its launches and copies then.  The line lies at CFG_EDGES
// edges, where the walks of one block take as long as the launches: cluster
// sizes of 0.9 n_j k-mers, one block and several launches, 60 and 84 us at
// L = 256, k = 12 (6717 edges), 73 and 76 at L = 64, k = 1 (8192), 85 and 77 at
// L = 72, k = 1 (10368), 152 and 132 at L = 256, k = 4 (27307).
#pragma once
#include "rsa_search.cuh"

namespace rsak {

constexpr u32 CFG_BINS = EHIST + 4;
constexpr u32 CFG_CAPPED = 1u << 31;  // wdirs bit: a union-find walk hit its cap

__host__ __device__ __forceinline__ u64* cfg_uf(const Group& g, u32 s) {
  return region_of(g, g.uf, s);
}
__host__ __device__ __forceinline__ u32* cfg_size(const Group& g, u32 s) {
  return reinterpret_cast<u32*>(region_of(g, g.uf, s) + g.cap_nodes);
}
__host__ __device__ __forceinline__ u32* cfg_hist(const Group& g, u32 s) {
  return cfg_size(g, s) + g.cap_nodes;
}

__device__ __forceinline__ void cfg_clear(const Group& g, u32 s, u32 nn) {
  u64* W = cfg_uf(g, s);
  u32* size = cfg_size(g, s);
  u32* hist = cfg_hist(g, s);
  for (u32 m = blockIdx.x * blockDim.x + threadIdx.x; m < nn; m += gridDim.x * blockDim.x) {
    W[m] = uf_pack(m, 0, 0);
    size[m] = 0;
    hist[m] = 0;
  }
}

// Keys per time_bin; the last block finds the bin that holds rank m.  bins:
// CFG_BINS words, zero before and, by k_key_select, after; bins[EHIST ..]:
// ticket, bin, rank in it, keys gathered.
__global__ void __launch_bounds__(256) k_key_bins(Group g, u32 s, u32 m, u32* bins) {
  __shared__ u32 h[EHIST];
  __shared__ u32 part[256];
  __shared__ u32 last_sh;
  const u32 tid = threadIdx.x;
  const u32 nn = min(g.st[s].n_nodes, g.cap_nodes);
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  for (u32 i = tid; i < EHIST; i += 256) h[i] = 0;
  __syncthreads();
  for (u32 i = blockIdx.x * 256 + tid; i < nn; i += gridDim.x * 256)
    atomicAdd(&h[time_bin(K[i])], 1u);
  __syncthreads();
  for (u32 i = tid; i < EHIST; i += 256)
    if (h[i]) atomicAdd(&bins[i], h[i]);
  __threadfence();
  __syncthreads();
  if (tid == 0) last_sh = atomicAdd(&bins[EHIST], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last_sh) return;
  __threadfence();
  constexpr u32 PER = EHIST / 256;
  u32 sum = 0;
  for (u32 i = 0; i < PER; ++i) sum += __ldcg(bins + tid * PER + i);
  part[tid] = sum;
  __syncthreads();
  for (u32 d = 1; d < 256; d <<= 1) {
    const u32 o = tid >= d ? part[tid - d] : 0u;
    __syncthreads();
    part[tid] += o;
    __syncthreads();
  }
  u32 a = part[tid] - sum;
  for (u32 i = 0; i < PER; ++i) {
    const u32 v = __ldcg(bins + tid * PER + i);
    if (a < m && m <= a + v) {
      bins[EHIST + 1] = tid * PER + i;
      bins[EHIST + 2] = m - a;
    }
    a += v;
  }
  if (tid == 0) {
    bins[EHIST] = 0;
    bins[EHIST + 3] = 0;
  }
}

// Rank selection among cnt keys by a block of 256 threads or more: eight
// passes, each fixing the next 8 bits of the answer from a histogram of the
// keys that share the bits fixed so far.  sh: 260 words (shared).
__device__ u64 select_key(const u64* keys, u32 cnt, u32 rank, u32* sh) {
  const u32 tid = threadIdx.x, nt = blockDim.x;
  u32* hist = sh;
  u64 pre = 0, mask = 0;
  for (int shift = 56; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    for (u32 i = tid; i < cnt; i += nt) {
      const u64 kk = keys[i];
      if ((kk & mask) == pre) atomicAdd(&hist[(u32)(kk >> shift) & 255u], 1u);
    }
    __syncthreads();
    // inclusive prefix of the 256 counts by the first warp
    if (tid < 32) {
      u32 v[8], sum = 0;
      for (u32 i = 0; i < 8; ++i) { v[i] = hist[tid * 8 + i]; sum += v[i]; }
      u32 inc = sum;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const u32 o = __shfl_up_sync(FULL, inc, d);
        if ((int)tid >= d) inc += o;
      }
      u32 a = inc - sum;
      for (u32 i = 0; i < 8; ++i) {
        if (a < rank && rank <= a + v[i]) {
          sh[256] = rank - a;
          sh[257] = tid * 8 + i;
        }
        a += v[i];
      }
    }
    __syncthreads();
    rank = sh[256];
    pre |= (u64)sh[257] << shift;
    mask |= 255ull << shift;
    __syncthreads();
  }
  return pre;
}

// The keys of that bin into the second half of the sample's uf slot (sizes and
// histogram afterwards), the m-th key of all, T_m, into st.sel by the last block.
constexpr u32 SEL_THREADS = 1024;
__global__ void __launch_bounds__(SEL_THREADS) k_key_select(Group g, u32 s, u32* bins) {
  __shared__ u32 sh[260];
  __shared__ u32 last_sh;
  const u32 tid = threadIdx.x;
  SampleState& st = g.st[s];
  const u32 nn = min(st.n_nodes, g.cap_nodes), bin = bins[EHIST + 1];
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  u64* out = reinterpret_cast<u64*>(cfg_size(g, s));
  for (u32 i = blockIdx.x * SEL_THREADS + tid; i < nn; i += gridDim.x * SEL_THREADS) {
    const u64 k = K[i];
    if (time_bin(k) == bin) out[atomicAdd(&bins[EHIST + 3], 1u)] = k;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last_sh = atomicAdd(&bins[EHIST], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last_sh) return;
  __threadfence();
  const u64 T = select_key(out, __ldcg(bins + EHIST + 3), bins[EHIST + 2], sh);
  if (tid == 0) st.sel = T;
  for (u32 i = tid; i < CFG_BINS; i += SEL_THREADS) bins[i] = 0;
}

// at_wrap: the configuration of the first wrap, T_m = T_c.
__global__ void __launch_bounds__(256) k_cfg_init(Group g, u32 s, bool at_wrap) {
  SampleState& st = g.st[s];
  cfg_clear(g, s, min(st.n_nodes, g.cap_nodes));
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st.wdirs = 0;
    if (at_wrap) st.sel = st.tc;
  }
}

__global__ void __launch_bounds__(256) k_cfg_union(Group g, u32 s) {
  SampleState& st = g.st[s];
  const u64 T = st.sel;
  const u32 ne = min(st.n_edges, g.edge_limit);
  const u64* E = region_of(g, g.etime, s);
  const uint4* K = region_of(g, g.elink, s);
  u64* W = cfg_uf(g, s);
  bool capped = false;
  u32 dirs = 0;
  __shared__ u32 queue[queue_words(256)];
  scan_packed(
      ne, Team{blockIdx.x, gridDim.x}, *reinterpret_cast<EdgeQueue*>(queue),
      [&](u32 i) { return E[i] <= T; },
      [&](u32 i) {
        const uint4 e = K[i];
        u32 mis = 0;
        if (uf_union(W, e.x, e.y, e.z, &capped, g.uf_cap, &mis))
          dirs |= ((mis & 0xFFFFu) ? 1u : 0u) | ((mis >> 16) ? 2u : 0u);
      });
  if (capped) dirs |= CFG_CAPPED;
  dirs = __reduce_or_sync(FULL, dirs);
  if ((threadIdx.x & 31) == 0 && dirs) atomicOr(&st.wdirs, dirs);
}

__global__ void __launch_bounds__(256) k_cfg_count(Group g, u32 s) {
  SampleState& st = g.st[s];
  const u64 T = st.sel;
  const u32 nn = min(st.n_nodes, g.cap_nodes);
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  u64* W = cfg_uf(g, s);
  u32* size = cfg_size(g, s);
  bool capped = false;
  for (u32 m = blockIdx.x * blockDim.x + threadIdx.x; m < nn; m += gridDim.x * blockDim.x) {
    if (K[m] > T) continue;
    u32 ox, oy;
    const u32 r = uf_find(W, m, &ox, &oy, &capped, g.uf_cap);
    atomicAdd(&size[r], 1u);
  }
  if (__any_sync(FULL, capped) && (threadIdx.x & 31) == 0) atomicOr(&st.wdirs, CFG_CAPPED);
}

__global__ void k_cfg_hist(Group g, u32 s) {
  const u32 nn = min(g.st[s].n_nodes, g.cap_nodes);
  const u32* size = cfg_size(g, s);
  u32* hist = cfg_hist(g, s);
  for (u32 m = blockIdx.x * blockDim.x + threadIdx.x; m < nn; m += gridDim.x * blockDim.x) {
    const u32 c = size[m];
    if (c) atomicAdd(&hist[c - 1], 1u);
  }
}

// The whole configuration of a sample of few k-mers in one block, union-find
// words and sizes in shared memory.  out (in the sample's uf half): the
// winding bits, then, with sizes, the number of clusters of 1 .. m k-mers.
constexpr u32 CFG_THREADS = 1024;
__host__ __device__ inline size_t cfg_block_smem(u32 cap_nodes) { return (size_t)cap_nodes * 12; }
constexpr u32 CFG_NODES = 18500;  // cap_nodes that fit beside the bins
constexpr u32 CFG_EDGES = 8192;

__global__ void __launch_bounds__(CFG_THREADS) k_cfg_block(Group g, u32 s, u32 m, bool at_wrap,
                                                           bool sizes) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ u32 bins[EHIST / 2];
  __shared__ u32 wsum[33];
  __shared__ u32 sh[260];
  __shared__ u32 bin_sh, rank_sh, cnt_sh, dirs_sh;
  u64* W = reinterpret_cast<u64*>(smem_raw);
  u32* size = reinterpret_cast<u32*>(W + g.cap_nodes);
  const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SampleState& st = g.st[s];
  const u32 nn = min(st.n_nodes, g.cap_nodes);
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  u32* out = cfg_size(g, s);
  if (tid == 0) dirs_sh = cnt_sh = 0;
  u64 T = st.tc;
  if (!at_wrap) {
    // bins of 16 per power of two; thread t owns bin t
    bins[tid] = 0;
    __syncthreads();
    for (u32 i = tid; i < nn; i += CFG_THREADS) atomicAdd(&bins[time_bin(K[i]) / 2], 1u);
    __syncthreads();
    const u32 mine = bins[tid];
    u32 inc = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 o = __shfl_up_sync(FULL, inc, d);
      if ((int)lane >= d) inc += o;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    u32 a = inc - mine;
    for (u32 q = 0; q < warp; ++q) a += wsum[q];
    if (a < m && m <= a + mine) {
      bin_sh = tid;
      rank_sh = m - a;
    }
    __syncthreads();
    const u32 bin = bin_sh;
    for (u32 i = tid; i < nn; i += CFG_THREADS) {
      const u64 k = K[i];
      if (time_bin(k) / 2 == bin) W[atomicAdd(&cnt_sh, 1u)] = k;
    }
    __syncthreads();
    T = select_key(W, cnt_sh, rank_sh, sh);
    __syncthreads();
  }
  for (u32 i = tid; i < nn; i += CFG_THREADS) {
    W[i] = uf_pack(i, 0, 0);
    size[i] = 0;
  }
  for (u32 i = tid; i <= m; i += CFG_THREADS) out[i] = 0;
  __syncthreads();
  const u32 ne = min(st.n_edges, g.edge_limit);
  const u64* E = region_of(g, g.etime, s);
  const uint4* L = region_of(g, g.elink, s);
  bool capped = false;
  u32 dirs = 0;
  for (u32 i = tid; i < ne; i += CFG_THREADS) {
    if (E[i] > T) continue;
    const uint4 e = L[i];
    u32 mis = 0;
    if (fin_union(W, e.x, e.y, e.z, &capped, g.uf_cap, &mis))
      dirs |= ((mis & 0xFFFFu) ? 1u : 0u) | ((mis >> 16) ? 2u : 0u);
  }
  __syncthreads();
  if (sizes) {
    for (u32 i = tid; i < nn; i += CFG_THREADS) {
      if (K[i] > T) continue;
      atomicAdd(&size[(u32)flat_word(W, i, g.uf_cap, &capped)], 1u);
    }
    __syncthreads();
    for (u32 i = tid; i < nn; i += CFG_THREADS)
      if (size[i]) atomicAdd(&out[size[i]], 1u);
  }
  if (capped) dirs |= CFG_CAPPED;
  dirs = __reduce_or_sync(FULL, dirs);
  if (lane == 0 && dirs) atomicOr(&dirs_sh, dirs);
  __syncthreads();
  if (tid == 0) out[0] = dirs_sh;
}

}  // namespace rsak
