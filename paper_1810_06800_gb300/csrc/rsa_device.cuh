// rsa_device.cuh -- device code of the GB300 RSA library (sm_103a).
//
// Exact parallel form of the RSA scan of arXiv:1810.06800 Sec. II.B: the
// viable-list deposition tries each (orientation, y, x) candidate once in
// uniformly random order and accepts it iff its k cells are free.  With the
// order fixed by distinct 64-bit priorities this is the lexicographically
// first maximal independent set of the candidate conflict graph.  The
// priorities are taken in slices, smallest first (rsa_rounds.cuh): of a
// slice's candidates those still live against the accepted k-mers are put in
// a list, and a listed candidate whose priority is the smallest of all listed
// ones sharing a cell with it is accepted, round by round, until the slice is
// empty.  rsa_search.cuh builds the contact graph and finds the first wrap,
// rsa_sample.cuh runs a whole sample in one block with the same bodies, and
// rsa_config.cuh answers for the configuration at m k-mers.
//
// Priorities are recomputed from (seed, idx) wherever they are needed
// instead of being stored: splitmix64 costs a few integer instructions,
// while storing 2 L^2 keys would cost 16 bytes per cell of HBM traffic per
// pass and 16 GiB per sample at L = 32768.
#pragma once
#include <cstdint>

namespace rsak {

typedef unsigned long long u64;
typedef uint32_t u32;
typedef uint16_t u16;
typedef uint8_t u8;

constexpr u64 KEY_NONE = 0xFFFFFFFFFFFFFFFFull;  // dead / no candidate
constexpr u64 SM_GAMMA = 0x9E3779B97F4A7C15ull;  // splitmix64 increment
constexpr u32 NONE32 = 0xFFFFFFFFu;
constexpr unsigned FULL = 0xFFFFFFFFu;
// Work counters are spread over WORK_SLOTS addresses (by block index), so that
// many blocks adding to one counter do not queue on a single L2 address.
constexpr u32 WORK_SLOTS = 32;
constexpr u32 EHIST = 2048;  // bins of time_bin

// status bits (per sample), mapped to RSA_E* codes by the host
constexpr u32 ST_NODE_OVF = 1u;     // more accepted k-mers than L^2/k (bug)
constexpr u32 ST_EDGE_OVF = 2u;     // contact-edge buffer too small
constexpr u32 ST_UF_CAP = 4u;       // union-find retry cap hit
constexpr u32 ST_NOWRAP = 8u;       // no wrap at jamming
constexpr u32 ST_SEARCH_CAP = 16u;  // search did not converge
constexpr u32 ST_ROUND_CAP = 32u;   // round loop cap hit

// splitmix64 output finaliser (Stafford "Mix13"), Steele/Lea/Flood 2014.
__device__ __forceinline__ u64 mix64(u64 z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

struct Window {        // state of the first-wrap search (rsa_search.cuh)
  u64 lo, hi, mid, next_mid;                // window (lo, hi], thresholds
  u32 cur, hi_ok, ready, first;             // union-find buffer of the state at lo; a probe
                                            // has wrapped at hi; the window is the last one;
                                            // no probe yet
  u32 probes, pad;
};

struct SampleState {   // one per sample
  u32 n_nodes, n_edges, rounds, status;
  u32 done, sdone, ticket, win_n;
  u32 ranked, nc, wdirs;                    // wdirs: configuration pass, winding bits
  u32 contacts_x, contacts_y, contacts_xy;  // lattice edges between different
                                            // k-mers: both H, both V, mixed
  u64 tc;                                   // priority of the k-mer that first wraps
  u64 sel;                                  // configuration pass: m-th key
  Window w;
};
static_assert(sizeof(SampleState) == 128, "SampleState is 128 bytes");

struct Team {          // the blocks that share a sample: this one's rank of size
  u32 rank, size;
};

struct WinEdge;

struct Group {         // one batch of samples sharing (L, k)
  u32 L, k, n;
  u32 cap_nodes, cap_edges;
  u32 uf_cap;          // steps of one union-find walk or link retry loop
  u32 edge_limit;      // contact edges stored per sample (<= cap_edges)
  u64 LL;
  u64 rstride;         // bytes between samples in the buffers marked (r): those of the
                       // rounds and those of the search share one region per sample
  u32* owner;          // [n][L][L]   node id of the k-mer anchored at the cell; only
                       //             anchors are written, the rest is never read
  u64* base;           // [n]         splitmix64 stream base per sample
  const u64* keys;     // caller priorities [2 L^2] (test path), else null
  u64* node_key;       // [n][cap_nodes]
  u32* node_idx;       // [n][cap_nodes]  accepted candidate idx
  u32* node_pos;       // [n][cap_nodes]  o << 31 | y0 << 15 | x0 of the anchor
  u64* uf;             // (r) [2][cap_nodes] union-find words
  u64* etime;          // (r) [cap_edges] contact edges: max of the two priorities,
  uint4* elink;        // (r) [cap_edges] and node ids, lifted anchor(m2) - anchor(m1)
                       //                as 16-bit dx, dy
  u32* ehist;          // (r) [SEARCH_WORDS] edges per time_bin, then the counts of a
                       //                probe; null where no graph can be large
  WinEdge* win;        // (r) [win_cap]
  SampleState* st;     // [n]
  u64* work;           // [4][WORK_SLOTS] work counters of the deposition: candidates
                       //     hashed by the first pass, list entries tested, active
                       //     candidates resolved, k-mers accepted
};

// Sample s's part of a buffer of the shared region.
template <typename T>
__host__ __device__ __forceinline__ T* region_of(const Group& g, T* first, u32 s) {
  return reinterpret_cast<T*>(reinterpret_cast<char*>(first) + (size_t)s * g.rstride);
}

// Slots from a counter for the lanes with ok, one atomic per warp.
__device__ __forceinline__ u32 warp_append(u32* counter, bool ok) {
  const u32 m = __ballot_sync(FULL, ok);
  if (!m) return 0;
  const u32 lane = threadIdx.x & 31, leader = __ffs(m) - 1;
  u32 at = 0;
  if (lane == leader) at = atomicAdd(counter, (u32)__popc(m));
  at = __shfl_sync(FULL, at, leader);
  return at + __popc(m & ((1u << lane) - 1u));
}

// Monotone bin of a priority: 32 bins per power of two.
__device__ __forceinline__ u32 time_bin(u64 t) {
  const u32 lz = (u32)__clzll((long long)(t | 1));
  return (63 - lz) * 32 + (lz == 63 ? 0u : (u32)((t << (lz + 1)) >> 59));
}

// Add v to work counter c (slot chosen by the block index).
__device__ __forceinline__ void work_add(const Group& g, u32 c, u64 v) {
  atomicAdd(g.work + c * WORK_SLOTS + (blockIdx.x & (WORK_SLOTS - 1)), v);
}

template <typename T> __device__ __forceinline__ T tmax(T a, T b) { return b > a ? b : a; }

__device__ __forceinline__ u64 uf_pack(u32 p, u32 dx, u32 dy) {
  return (u64)p | ((u64)(dx & 0xFFFFu) << 32) | ((u64)(dy & 0xFFFFu) << 48);
}

constexpr u32 UF_CAP = 1u << 20;  // default walk / retry cap (Group::uf_cap)

}  // namespace rsak
