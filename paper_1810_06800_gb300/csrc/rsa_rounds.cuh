// rsa_rounds.cuh -- deposition to jamming by slices of the priority range
// (any 2 <= k <= L), sm_103a.
//
// A candidate of priority key conflicts with about D = k^2 + 2k others, so
// the ones accepted first all have priorities near 2^64 / D and nearly every
// candidate dies before its turn comes.  The scan therefore goes through the
// priority range in slices [lo, hi] (each twice as wide as the one before)
// and only ever works on the candidates of the current slice that are still
// live:
//   k_dense    every candidate hashed once; the idx of those with priority
//              below 2^(64 - a) go to one list per slice (level = leading
//              zeros of the priority);
//   k_pick     the entries of the current slice whose k cells are free become
//              the active set, together with the undecided rest of the slice
//              before; each is linked into a square bin of its anchor;
//   k_resolve  an active candidate that conflicts with no active candidate of
//              smaller priority is accepted: node, anchor bits, cover bits.
//              The others stay for the next slice, whose k_pick drops the
//              dead ones;
//   k_refill   after the listed slices (2^-a of all candidates): the few
//              candidates still live, read off the cover bits of each line,
//              become the list of all remaining slices.
// Exactness: when a slice is resolved every undecided candidate of smaller
// priority is in the active set, so "no active conflicting candidate is
// smaller" is the sequential scan's condition for acceptance, and acceptance
// order is irrelevant otherwise.
//
// Measured share of candidates (L = 1024 .. 2048, k = 4 .. 256): the active
// sets of all slices add up to 1.4 n_j, two to four rounds decide a slice,
// and 1.5% of the candidates are still live at priority 2^64 * 4 / k.  The
// arithmetic is thus one splitmix64 per candidate plus work proportional to
// the k-mers, where a round over the whole lattice costs two window minima
// of 64-bit priorities for every cell, eight to ten times over.
//
// Lines are kept as bits with their first k cells repeated after the end, so
// a window of k cells never wraps.  Cover bits of orientation o (lines along
// o) mark the cells a candidate of o must avoid: the k-mers of o on their own
// line, and the crossing ones.  A crossing k-mer would set one bit on each of
// k lines; instead the blocks of 2^bs whole lines it crosses get one bit in a
// block line, and only the lines at its two ends their own: 2^bs + k / 2^bs
// updates in place of k, against reading two lines in each test.
#pragma once
#include "rsa_search.cuh"

namespace rsak {

constexpr u32 RD_LEVELS = 32;
constexpr u32 RD_THREADS = 256;
constexpr u32 DENSE_THREADS = 256;
constexpr u32 DENSE_PER = 16;                      // candidates per thread and tile
constexpr u32 REFILL_WORDS = 9472;                 // words of line staged per block: 8 lines of
                                                   // L = 32768, k = 4096; at least one of any shape

struct RoundCfg {
  u32 W;            // words of a cover line, (L + k) bits and one spare
  u32 WA;           // words of an anchor line, (L + 2k) bits and one spare
  u32 bs, nbl;      // block lines: 2^bs lines each, nbl of them (bs = 0: none)
  u32 b, nb;        // bins of 2^b x 2^b cells, nb per side
  u32 a;            // k_dense lists priorities below 2^(64 - a)
  u32 lzmax;        // slice 0 takes every priority of at least lzmax leading zeros
  u32 nlev;         // listed slices, lzmax - a + 1
  u32 cap_act;      // active candidates per sample
  u32 cap_flat;     // entries of the refilled list
  u32 round_cap;
  u64 inv_L;        // ceil(2^45 / L)
  u32 lvl_off[RD_LEVELS], lvl_cap[RD_LEVELS];
};

struct Act {        // an active candidate (16 bytes, one load)
  u64 key;
  u32 pos;          // o << 31 | y << 15 | x of its anchor
  u32 next;         // next active candidate of its bin
};

struct Slice {      // where the scan of a sample stands
  u64 lo, hi;       // current slice, both ends included
  u64 fill_hi;      // the refilled list holds priorities up to this one
  u32 t;            // number of the slice: 0 .. lzmax
  u32 open;         // 0: no slice, only undecided candidates go on
  u32 drain;        // the active set was full: one round without new entries
  u32 refill;       // the lists are used up: k_refill has to run, from lo on
  u32 finished;     // every slice has been entered
  u32 par;          // active buffer written by this round
};

struct RoundState { // per sample
  Slice sl;
  u32 act[2];       // active candidates per buffer
  u32 taken;        // accepted in this round
  u32 flat_n;
  u32 ticket, ticket2;
  u32 lvl_n[RD_LEVELS];
};

__device__ __forceinline__ u64 slice_top(const RoundCfg& c, u32 t) {
  const u32 lz = c.lzmax - t;
  return lz == 0 ? ~0ull : (1ull << (64 - lz)) - 1ull;
}

__device__ __forceinline__ Slice first_slice(const RoundCfg& c) {
  Slice z = {};
  z.open = 1;
  z.hi = slice_top(c, 0);
  z.fill_hi = ~0ull;
  return z;
}

// r / L for r < L^2 (L <= 2^15): the product with ceil(2^45 / L) is at most
// r / 2^45 < 1 / L above 2^45 r / L.
__device__ __forceinline__ u32 row_of(const RoundCfg& c, u32 r) {
  return (u32)(((u64)r * c.inv_L) >> 45);
}

struct RoundPtrs {
  u32* fine;        // (r) [2][L][W]
  u32* block;       // (r) [2][nbl][W]
  u32* anch;        // [n][4][L][WA]: type * 2 + layout
  u32* list;        // (r) [list_cap]
  u32* flat;        // (r) [cap_flat]
  Act* act;         // (r) [2][cap_act]
  u32* heads;       // (r) [2][2][nb * nb]
  RoundState* rs;   // [n]
};

__device__ __forceinline__ u32* cover_line(const Group& g, const RoundCfg& c, const RoundPtrs& p,
                                           u32 s, u32 o, u32 line) {
  return region_of(g, p.fine, s) + (o * g.L + line) * c.W;  // < 2^28 words
}
__device__ __forceinline__ u32* block_line(const Group& g, const RoundCfg& c, const RoundPtrs& p,
                                           u32 s, u32 o, u32 bl) {
  return region_of(g, p.block, s) + (o * c.nbl + bl) * c.W;
}
// Anchors of k-mers of orientation `type`, as lines along `layout`.
__device__ __forceinline__ u32* anchor_line(const Group& g, const RoundCfg& c, const RoundPtrs& p,
                                            u32 s, u32 type, u32 layout, u32 line) {
  return p.anch + (((size_t)s * 4 + type * 2 + layout) * g.L + line) * c.WA;
}

// Per-sample set-up: stream base from the seed, state cleared.
__global__ void k_init(Group g, const u64* seeds) {
  const u32 s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.n) return;
  g.base[s] = mix64(seeds[s] + SM_GAMMA);
  SampleState z = {};
  g.st[s] = z;
}

__global__ void k_round_init(Group g, RoundCfg c, RoundPtrs p) {
  const u32 s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.n) return;
  RoundState z = {};
  z.sl = first_slice(c);
  p.rs[s] = z;
}

// Every candidate hashed once: bound by integer issue (L = 1024, k = 32: issue
// slots 74% busy, ALU pipe 60%, 40 instructions per candidate with one in 8 to
// be staged; 1000 samples, 2.1 G candidates, in 2.9 ms.  L = 32768, k = 4096, 4
// samples, 8.6 G candidates, in 8.1 ms).  A block goes over tiles of 4096 consecutive
// candidates; a thread keeps its 16 hits of a tile as a bit mask, so the
// inner loop is the hash and one compare.  Hits are staged in shared memory
// and leave by level, one global counter update per level and flush.
// (the high word of mix64's last step z ^ (z >> 31) has at least a >= 1
// leading zeros iff that of z has, so the hit test needs neither that step
// nor the low word of the second product)
template <u32 NT, u32 PER>   // threads of the block, at most; candidates of each in a tile
struct DenseSmem {
  static constexpr u32 STAGE = 8192;
  u32 count, lcnt[RD_LEVELS], lbase[RD_LEVELS];
  u32 stage[STAGE];
  u8 lev[STAGE];
};

template <bool KEYS, u32 NT, u32 PER>
__device__ void dense_body(const Group& g, const RoundCfg& c, const RoundPtrs& p, u32 s, Team team,
                           RoundState& r, DenseSmem<NT, PER>& sm) {
  const u32 tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const u32 tile_n = PER * nt;
  const u64 N = 2 * g.LL, zb = g.base[s] + SM_GAMMA, zstep = SM_GAMMA * nt;
  const u64 ntile = (N + tile_n - 1) / tile_n;
  const u32 limit = 1u << (32 - c.a);
  if (tid == 0) sm.count = 0;
  __syncthreads();
  for (u64 tile = team.rank; tile < ntile; tile += team.size) {
    const u64 i0 = tile * tile_n + tid;
    u32 hits = 0;
    if (KEYS) {
      for (u32 j = 0; j < PER; ++j) {
        const u64 i = i0 + j * nt;
        if (i < N && (u32)(g.keys[i] >> 32) < limit) hits |= 1u << j;
      }
    } else {
      u64 z = zb + SM_GAMMA * i0;
#pragma unroll
      for (u32 j = 0; j < PER; ++j, z += zstep) {
        u64 h = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        h = (h ^ (h >> 27)) * 0x94D049BB133111EBull;
        if ((u32)(h >> 32) < limit) hits |= 1u << j;
      }
      if (i0 + (u64)(PER - 1) * nt >= N) {
        for (u32 j = 0; j < PER; ++j)
          if (i0 + (u64)j * nt >= N) hits &= ~(1u << j);
      }
    }
    // this warp's hits, packed
    const u32 nh = __popc(hits);
    u32 pre = nh;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 o = __shfl_up_sync(FULL, pre, d);
      if ((int)lane >= d) pre += o;
    }
    u32 at = 0;
    if (lane == 31 && pre) at = atomicAdd(&sm.count, pre);
    at = __shfl_sync(FULL, at, 31) + pre - nh;
    u32* list = region_of(g, p.list, s);
    auto level_of = [&](u32 idx) {
      const u64 key = KEYS ? g.keys[idx] : mix64(zb + SM_GAMMA * idx);
      return c.lzmax - min((u32)__clzll((long long)key), c.lzmax);
    };
    auto put = [&](u32 t, u32 at2, u32 idx) {
      if (at2 < c.lvl_cap[t]) list[c.lvl_off[t] + at2] = idx;
      else atomicOr(&g.st[s].status, ST_NODE_OVF);
    };
    for (u32 m = hits; m; m &= m - 1, ++at) {
      const u32 idx = (u32)(i0 + (u64)(__ffs(m) - 1) * nt);
      if (at < sm.STAGE) {
        sm.stage[at] = idx;
      } else {
        // more hits than the stage holds: one atomic per hit.  Hashed priorities
        // meet it where one block tiles 16384 candidates and half of them are
        // hits (rsa_sample.cuh, k = 2 and 3); a tile of k_dense has 4096
        const u32 t = level_of(idx);
        put(t, atomicAdd(&r.lvl_n[t], 1u), idx);
      }
    }
    __syncthreads();
    const u32 n = min(sm.count, sm.STAGE);
    const bool last = tile + team.size >= ntile;
    if (n > sm.STAGE / 2 || last) {
      if (tid < RD_LEVELS) sm.lcnt[tid] = 0;
      __syncthreads();
      for (u32 i = tid; i < n; i += nt) {
        const u32 t = level_of(sm.stage[i]);
        sm.lev[i] = (u8)t;
        atomicAdd(&sm.lcnt[t], 1u);
      }
      __syncthreads();
      if (tid < c.nlev) {
        sm.lbase[tid] = sm.lcnt[tid] ? atomicAdd(&r.lvl_n[tid], sm.lcnt[tid]) : 0u;
        sm.lcnt[tid] = 0;
      }
      __syncthreads();
      for (u32 i = tid; i < n; i += nt) {
        const u32 t = sm.lev[i];
        put(t, sm.lbase[t] + atomicAdd(&sm.lcnt[t], 1u), sm.stage[i]);
      }
      __syncthreads();
      if (tid == 0) sm.count = 0;
    }
    __syncthreads();
  }
}

template <bool KEYS>
__global__ void __launch_bounds__(DENSE_THREADS) k_dense(Group g,
                                                         const __grid_constant__ RoundCfg c,
                                                         RoundPtrs p) {
  __shared__ DenseSmem<DENSE_THREADS, DENSE_PER> sm;
  dense_body<KEYS>(g, c, p, blockIdx.y, Team{blockIdx.x, gridDim.x}, p.rs[blockIdx.y], sm);
  if (threadIdx.x == 0 && blockIdx.x == 0) work_add(g, 0, 2 * g.LL);
}

// Word w of the bits [pos, pos + k) of a line, masked to them.
__device__ __forceinline__ u32 window_word(const u32* line, u32 w, u32 pos, u32 end) {
  u32 v = line[w];
  if (w == pos >> 5) v &= 0xFFFFFFFFu << (pos & 31u);
  if (w == end >> 5) v &= 0xFFFFFFFFu >> (31u - (end & 31u));
  return v;
}

// The active set of this round.  Bound by the loads of the cover words, which
// lie anywhere on the lattice (issue slots 38 to 67% busy).  Windows of up to
// PICK_LONGK cells are tested word by word by the lane that holds the
// candidate, which stops at the first covered word; longer ones at three
// words, at seven more, and the few that pass by the whole warp.  The line:
// k_pick of L = 2048, k = 128, 32 samples 0.39 ms by lanes and 0.51 by warps,
// L = 8192, k = 512, 32 samples 2.56 and 2.66, k = 1024, 8 samples 0.83 and
// 0.72, L = 32768, k = 4096, 4 samples 4.87 and 3.72 (3.07 with the seven
// words).
constexpr u32 PICK_LONGK = 768;
template <bool LONG>
__device__ void pick_body(const Group& g, const RoundCfg& c, const RoundPtrs& p, u32 s, Team team,
                          const Slice& sl, u32 n1, u32 n2, u32* count) {
  const u32 L = g.L, k = g.k, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const u32 par = sl.par, t = sl.t;
  const u64 lo = sl.lo, hi = sl.hi;
  const bool flat = t >= c.nlev;
  const u32* list = flat ? region_of(g, p.flat, s) : region_of(g, p.list, s) + c.lvl_off[t];
  const Act* prev = region_of(g, p.act, s) + (size_t)(par ^ 1u) * c.cap_act;
  Act* cur = region_of(g, p.act, s) + (size_t)par * c.cap_act;
  u32* heads = region_of(g, p.heads, s) + (size_t)par * 2 * c.nb * c.nb;
  const u64 zb = g.base[s] + SM_GAMMA;
  auto key_of = [&](u32 idx) { return g.keys ? g.keys[idx] : mix64(zb + SM_GAMMA * idx); };
  const u32 total = n1 + n2;
  for (u32 i0 = team.rank * nt; i0 < total; i0 += team.size * nt) {
    const u32 i = i0 + tid;
    bool ok = i < total;
    u32 o = 0, y = 0, x = 0, idx = 0;
    u64 key = 0;
    if (ok) {
      if (i < n1) {
        // a refilled list holds all later slices: first whether the entry is of
        // this one; of a slice's own list most entries are dead: first whether
        // it is live, and its priority only then
        idx = list[i];
        if (flat) {
          key = key_of(idx);
          ok = key >= lo && key <= hi;
        }
        u32 rr = idx;
        if (rr >= (u32)g.LL) { o = 1; rr -= (u32)g.LL; }
        y = row_of(c, rr);
        x = rr - y * L;
      } else {
        const uint4 e = *reinterpret_cast<const uint4*>(prev + (i - n1));
        key = (u64)e.y << 32 | e.x;
        o = e.z >> 31;
        y = (e.z >> 15) & 0x7FFFu;
        x = e.z & 0x7FFFu;
      }
    }
    const u32 line = o ? x : y, pos = o ? y : x, end = pos + k - 1;
    const u32* fl = cover_line(g, c, p, s, o, line);
    const u32* bl = c.bs ? block_line(g, c, p, s, o, line >> c.bs) : fl;
    const u32 w0 = pos >> 5, w1 = end >> 5;
    if (!LONG) {
      if (ok) {
        u32 v = 0;
        for (u32 w = w0; w <= w1; ++w) {
          v |= window_word(fl, w, pos, end);
          if (c.bs) v |= window_word(bl, w, pos, end);
          if (v) break;
        }
        ok = v == 0;
      }
    } else {
      if (ok) {
        const u32 wm = (w0 + w1) >> 1;
        ok = (window_word(fl, w0, pos, end) | window_word(bl, w0, pos, end) |
              window_word(fl, w1, pos, end) | window_word(bl, w1, pos, end) | fl[wm] | bl[wm]) == 0;
      }
      if (ok) {
        const u32 step = (w1 - w0) >> 3;  // >= 3: whole words inside the window
        u32 v = 0;
#pragma unroll
        for (u32 i = 1; i < 8; ++i) v |= fl[w0 + i * step] | bl[w0 + i * step];
        ok = v == 0;
      }
      // the words between, 32 at a time, one candidate after another
      for (u32 m = __ballot_sync(FULL, ok); m; m &= m - 1) {
        const u32 src = __ffs(m) - 1;
        const u32 so = __shfl_sync(FULL, o, src), ln = __shfl_sync(FULL, line, src);
        const u32 a0 = __shfl_sync(FULL, w0, src) + 1, a1 = __shfl_sync(FULL, w1, src);
        const u32* f2 = cover_line(g, c, p, s, so, ln);
        const u32* b2 = block_line(g, c, p, s, so, ln >> c.bs);
        u32 v = 0;
        for (u32 w = a0 + lane; w < a1; w += 32) v |= f2[w] | b2[w];
        const bool hit = __any_sync(FULL, v != 0);
        if (lane == src && hit) ok = false;
      }
    }
    if (ok && i < n1 && !flat) {
      key = key_of(idx);
      ok = key >= lo && key <= hi;  // (a narrowed slice)
    }
    const u32 slot = warp_append(count, ok);
    if (ok && slot < c.cap_act) {
      Act e;
      e.key = key;
      e.pos = (o << 31) | (y << 15) | x;
      e.next = atomicExch(heads + ((size_t)o * c.nb + (y >> c.b)) * c.nb + (x >> c.b), slot);
      *reinterpret_cast<uint4*>(cur + slot) = *reinterpret_cast<uint4*>(&e);
    }
  }
}

// Entries of the current slice's list.
__device__ __forceinline__ u32 slice_entries(const RoundCfg& c, const RoundState& r,
                                             const Slice& sl) {
  return !sl.open || sl.drain ? 0u : sl.t >= c.nlev ? r.flat_n : min(r.lvl_n[sl.t], c.lvl_cap[sl.t]);
}

template <bool LONG>
__global__ void __launch_bounds__(RD_THREADS) k_pick(Group g, const __grid_constant__ RoundCfg c,
                                                     RoundPtrs p) {
  const u32 s = blockIdx.y;
  if (g.st[s].done) return;
  RoundState& r = p.rs[s];
  const Slice sl = r.sl;
  const u32 n1 = slice_entries(c, r, sl), n2 = r.act[sl.par ^ 1u];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    r.taken = 0;
    work_add(g, 1, n1 + n2);
  }
  pick_body<LONG>(g, c, p, s, Team{blockIdx.x, gridDim.x}, sl, n1, n2, &r.act[sl.par]);
}

// Bins that the cells [a, a + len) of a ring of L cells touch, as n1 bins
// from b0 on and n2 from bin 0 on.
struct BinRun {
  u32 b0, n1, n;
  __device__ __forceinline__ BinRun(u32 a, u32 len, u32 L, u32 b) {
    if (len > L) len = L;
    b0 = a >> b;
    const u32 e = a + len;
    if (e <= L) {
      n1 = n = ((e - 1) >> b) - b0 + 1;
    } else {
      n1 = ((L - 1) >> b) - b0 + 1;
      n = n1 + min(((e - L - 1) >> b) + 1, b0);
    }
  }
  __device__ __forceinline__ u32 bin(u32 i) const { return i < n1 ? b0 + i : i - n1; }
};

__device__ __forceinline__ u32 ring_sub(u32 a, u32 b, u32 L) { return a >= b ? a - b : a + L - b; }

// Set bit q of a line and its copies one and two turns on.
__device__ __forceinline__ void set_bit_copies(u32* line, u32 q, u32 L, u32 bits) {
  for (; q < bits; q += L) atomicOr(line + (q >> 5), 1u << (q & 31u));
}

// Bits [a, e) of a line that fall in word w.
__device__ __forceinline__ u32 range_word(u32 w, u32 a, u32 e) {
  const u32 w0 = w * 32;
  if (e <= w0 || a >= w0 + 32) return 0;
  u32 m = 0xFFFFFFFFu;
  if (a > w0) m &= 0xFFFFFFFFu << (a - w0);
  if (e < w0 + 32) m &= 0xFFFFFFFFu >> (w0 + 32 - e);
  return m;
}

// Cover bits of an accepted k-mer, by the G lanes of a group (lane j).
template <int G>
__device__ void cover_kmer(const Group& g, const RoundCfg& c, const RoundPtrs& p, u32 s, u32 o,
                           u32 line, u32 pos, u32 j) {
  const u32 L = g.L, k = g.k;
  // its own line: [pos, pos + k), the part past the end again at the start,
  // the part among the first k cells again past the end
  u32* own = cover_line(g, c, p, s, o, line);
  const u32 e = pos + k;
  for (u32 w = (pos >> 5) + j; w <= (e - 1) >> 5; w += G) atomicOr(own + w, range_word(w, pos, e));
  if (e > L)
    for (u32 w = j; w <= (e - L - 1) >> 5; w += G) atomicOr(own + w, range_word(w, 0, e - L));
  if (pos < k) {
    const u32 a2 = pos + L, e2 = min(e, k) + L;
    for (u32 w = (a2 >> 5) + j; w <= (e2 - 1) >> 5; w += G) atomicOr(own + w, range_word(w, a2, e2));
  }
  // the lines it crosses: cells [pos, pos + k) of the ring as one or two
  // stretches; whole blocks of lines by their block line
  const u32 bits = L + k;
  for (u32 h = 0; h < 2; ++h) {
    const u32 a = h ? 0u : pos, b = h ? (e > L ? e - L : 0u) : min(e, L);
    if (a >= b) continue;
    u32 f0 = b, f1 = b;  // whole blocks cover lines [f0, f1)
    if (c.bs) {
      const u32 j0 = (a + (1u << c.bs) - 1) >> c.bs, j1 = b == L ? c.nbl : b >> c.bs;
      if (j0 < j1) {
        f0 = j0 << c.bs;
        f1 = min(j1 << c.bs, L);
        for (u32 bl = j0 + j; bl < j1; bl += G)
          set_bit_copies(block_line(g, c, p, s, o ^ 1u, bl), line, L, bits);
      }
    }
    for (u32 q = a + j; q < f0; q += G)
      set_bit_copies(cover_line(g, c, p, s, o ^ 1u, q), line, L, bits);
    for (u32 q = f1 + j; q < b; q += G)
      set_bit_copies(cover_line(g, c, p, s, o ^ 1u, q), line, L, bits);
  }
}

// The step from one round of n active candidates, `left` of them undecided,
// to the next.  True if the sample is done.
__device__ bool round_step(const RoundCfg& c, Slice& r, u32 n, u32 left, u32& rounds,
                           u32& status) {
  if (n > c.cap_act) {
    // too many: this round decided nothing; the same undecided candidates
    // again, with a narrower slice, or with none if it is one key wide
    if (r.hi == r.lo) r.drain = 1;
    else r.hi = r.lo + (r.hi - r.lo) / 8;
    return false;
  }
  r.par ^= 1u;
  if (r.drain) {
    r.drain = 0;
  } else if (r.open) {
    const u64 top = slice_top(c, r.t), wide = r.hi - r.lo;
    const bool listed = r.t < c.nlev, used_up = r.hi == (listed ? slice_top(c, c.nlev - 1) : r.fill_hi);
    r.lo = r.hi + 1;
    if (r.lo == 0) {
      r.finished = 1;
      r.open = 0;
    } else {
      if (r.hi == top) {
        r.t += 1;
        r.hi = slice_top(c, r.t);
      } else {  // narrowed before: wider again
        const u64 room = top - r.lo, w = wide < (1ull << 61) ? wide * 4 + 3 : room;
        r.hi = r.lo + (w < room ? w : room);
      }
      if (used_up) {
        r.refill = 1;  // k_refill opens the next slice
        r.open = 0;
        r.fill_hi = ~0ull;
      } else if (!listed) {
        r.hi = r.hi < r.fill_hi ? r.hi : r.fill_hi;
      }
    }
  }
  if (n) rounds += 1;
  if (r.finished && left == 0) return true;
  if (rounds >= c.round_cap) {
    status |= ST_ROUND_CAP;
    return true;
  }
  return false;
}

// The step after k_refill listed flat_n candidates.
__device__ __forceinline__ void refill_step(const RoundCfg& c, Slice& r, u32 flat_n) {
  if (flat_n > c.cap_flat) {
    // more than the list holds: fewer priorities, next time
    r.fill_hi = r.lo + (r.fill_hi - r.lo) / 8;
  } else {
    r.refill = 0;
    r.open = 1;
    r.hi = r.hi < r.fill_hi ? r.hi : r.fill_hi;
  }
}

// Bins of the round after, emptied while this one is resolved.
__device__ __forceinline__ void clear_bins(const Group& g, const RoundCfg& c, const RoundPtrs& p,
                                           u32 s, Team team, u32 buf) {
  u32* nx = region_of(g, p.heads, s) + (size_t)buf * 2 * c.nb * c.nb;
  for (u32 i = team.rank * blockDim.x + threadIdx.x; i < 2 * c.nb * c.nb;
       i += team.size * blockDim.x)
    nx[i] = NONE32;
}

// G lanes per active candidate.  Bins are about 4 sqrt(k) cells wide, which
// leaves one or two active candidates in each and k / 16 bins to look at.
// Bound by the latency of the chain counter - bin head - candidate - its next
// (L = 1024, k = 32: 39 to 42 of 53 to 57 resident warps wait for a load, issue
// slots 23 to 36% busy; 1000 samples 7.5 ms in all rounds).
// Adds this thread's accepted candidates to taken.
template <int G>
__device__ void resolve_body(const Group& g, const RoundCfg& c, const RoundPtrs& p, u32 s,
                             Team team, u32 par, u32 n, u32* nodes, u32& taken) {
  SampleState& st = g.st[s];
  const u32 L = g.L, k = g.k, tid = threadIdx.x;
  const u32* heads = region_of(g, p.heads, s) + (size_t)par * 2 * c.nb * c.nb;
  const Act* cur = region_of(g, p.act, s) + (size_t)par * c.cap_act;
  const u32 j = tid & (G - 1);
  const u32 gmask = G == 32 ? FULL : ((1u << (G & 31)) - 1u) << ((tid & 31) & ~(G - 1));
  const u32 gpb = blockDim.x / G;
  for (u32 i0 = team.rank * gpb; i0 < n; i0 += team.size * gpb) {
    const u32 i = i0 + tid / G;
    const bool valid = i < n;
    const uint4 raw = valid ? *reinterpret_cast<const uint4*>(cur + i) : make_uint4(0, 0, 0, 0);
    const u64 key = (u64)raw.y << 32 | raw.x;
    const u32 o = raw.z >> 31, y = (raw.z >> 15) & 0x7FFFu, x = raw.z & 0x7FFFu;
    const u32 line = o ? x : y, pos = o ? y : x;
    // conflicting anchors: on its own line less than k away; crossing ones
    // on the k lines of its cells, from k - 1 cells before its line to it
    const BinRun same(ring_sub(pos, k - 1, L), 2 * k - 1, L, c.b);
    const BinRun cl(pos, k, L, c.b), cp(ring_sub(line, k - 1, L), k, L, c.b);
    const u32 nbin = same.n + cl.n * cp.n;
    // does the active candidate a beat this one?
    auto beats = [&](const uint4& a) -> bool {
      if (((u64)a.y << 32 | a.x) >= key) return false;
      const u32 ao = a.z >> 31, ay = (a.z >> 15) & 0x7FFFu, ax = a.z & 0x7FFFu;
      const u32 aline = ao ? ax : ay, apos = ao ? ay : ax;
      if (ao == o) {
        const u32 d = ring_sub(apos, pos, L);
        return aline == line && (d < k || d > L - k);
      }
      return ring_sub(o ? ay : ax, pos, L) < k && ring_sub(line, o ? ax : ay, L) < k;
    };
    auto rest = [&](u32 e) -> bool {  // the chain of a bin from e on
      for (u32 guard = 0; e != NONE32 && guard < n; ++guard) {
        const uint4 a = *reinterpret_cast<const uint4*>(cur + e);
        if (beats(a)) return true;
        e = a.w;
      }
      return false;
    };
    // bins are stored by (orientation, row, column)
    auto head = [&](u32 bo, u32 bl, u32 bp) -> u32 {
      const u32 by = bo ? bp : bl, bx = bo ? bl : bp;
      return heads[(bo * c.nb + by) * c.nb + bx];
    };
    bool beaten = !valid;
    if (G == 1) {
      for (u32 q = 0; q < same.n && !beaten; ++q) beaten = rest(head(o, line >> c.b, same.bin(q)));
      for (u32 q1 = 0; q1 < cl.n && !beaten; ++q1)
        for (u32 q2 = 0; q2 < cp.n && !beaten; ++q2)
          beaten = rest(head(o ^ 1u, cl.bin(q1), cp.bin(q2)));
    } else {
      for (u32 q0 = 0; q0 < nbin && !beaten; q0 += G) {
        const u32 q = q0 + j;
        if (q < same.n) {
          beaten = rest(head(o, line >> c.b, same.bin(q)));
        } else if (q < nbin) {
          const u32 qq = q - same.n, q1 = qq / cp.n;
          beaten = rest(head(o ^ 1u, cl.bin(q1), cp.bin(qq - q1 * cp.n)));
        }
        beaten = (__ballot_sync(gmask, beaten) & gmask) != 0;
      }
    }
    // the lanes of a warp go on together from here: their k-mers are placed side
    // by side, with one node counter update (L = 1024, k = 32, 1000 samples: 8.2 ms
    // by lanes that left the search one after another, 7.4 now; four bins read
    // ahead at a time 9.3, every lane at its own pace through bins and chains
    // 11.7)
    __syncwarp();
    u32 node = warp_append(nodes, !beaten && j == 0);
    if (G > 1) node = __shfl_sync(FULL, node, 0, G);
    if (beaten) continue;
    if (node >= g.cap_nodes) {
      if (j == 0) atomicOr(&st.status, ST_NODE_OVF);
      continue;
    }
    if (j == 0) {
      const size_t nd = (size_t)s * g.cap_nodes + node;
      const u32 cell = y * L + x;
      g.node_key[nd] = key;
      g.node_idx[nd] = o * (u32)g.LL + cell;
      g.node_pos[nd] = raw.z;
      g.owner[(size_t)s * g.LL + cell] = node;
      ++taken;
    }
    if (G == 1 || j < 2) {
      const u32 bits = L + 2 * k;
      for (u32 lay = G == 1 ? 0 : j; lay < (G == 1 ? 2 : j + 1); ++lay)
        set_bit_copies(anchor_line(g, c, p, s, o, lay, lay ? x : y), lay ? y : x, L, bits);
    }
    cover_kmer<G>(g, c, p, s, o, line, pos, j);
  }
}

// With 16 and 32 lanes eight blocks per SM (32 registers, 8 bytes spilled): the
// more candidates wait at once, the better (L = 8192, k = 512, 32 samples 4.5 ->
// 3.7 ms, L = 32768, k = 4096, 4 samples 4.7 -> 4.5).  One lane gains nothing (7.6
// and 7.6 ms at L = 1024, k = 32, 1000 samples) and eight lanes, used where the
// GPU is not full, lose (one such sample 0.19 -> 0.20 ms): the compiler's choice
// stays (0 sets no bound; 1 would let it take 72 and 88 registers, L = 777,
// k = 100, 16 samples 0.57 -> 0.63 ms in all).
template <int G>
__global__ void __launch_bounds__(RD_THREADS, G >= 16 ? 8 : 0)
k_resolve(Group g, const __grid_constant__ RoundCfg c, RoundPtrs p) {
  __shared__ u32 taken_sh;
  const u32 s = blockIdx.y;
  SampleState& st = g.st[s];
  if (st.done) return;
  RoundState& r = p.rs[s];
  const u32 tid = threadIdx.x, par = r.sl.par, n = r.act[par];
  const Team team{blockIdx.x, gridDim.x};
  const bool over = n > c.cap_act;
  clear_bins(g, c, p, s, team, over ? par : par ^ 1u);
  if (tid == 0) taken_sh = 0;
  __syncthreads();
  u32 taken = 0;
  if (!over) resolve_body<G>(g, c, p, s, team, par, n, &st.n_nodes, taken);
  taken = __reduce_add_sync(FULL, taken);
  if ((tid & 31) == 0 && taken) atomicAdd(&taken_sh, taken);
  __syncthreads();
  if (tid == 0) {
    if (taken_sh) {
      atomicAdd(&r.taken, taken_sh);
      work_add(g, 3, taken_sh);
    }
    if (blockIdx.x == 0) work_add(g, 2, over ? 0 : n);
    __threadfence();
    if (atomicAdd(&r.ticket, 1u) == gridDim.x - 1) {
      __threadfence();
      r.ticket = 0;
      Slice sl = r.sl;
      u32 rounds = st.rounds, status = __ldcg(&st.status);
      const bool was_refill = sl.refill;
      if (round_step(c, sl, n, n - __ldcg(&r.taken), rounds, status)) st.done = 1;
      r.act[sl.par] = 0;  // the next round's buffer (this one's, if it was overfull)
      if (sl.refill && !was_refill) r.flat_n = 0;
      r.sl = sl;
      st.rounds = rounds;
      st.status = status;
    }
  }
}

// The candidates of every line still live once the list is used up, those
// with priorities in [lo, fill_hi].  k <= 33: the window OR of a word and the
// next by doubling in registers, one word per lane.  Longer windows reach past
// every word's end, so the live anchors of a word are those after its last
// covered cell and at least k before the next covered cell beyond it: the
// first covered cells of all words, and a suffix minimum over them, in one
// pass over the staged line; one warp per line.  (Doubling windows over whole
// lines in shared memory took 5.5 ms at L = 32768, k = 4096, 4 samples, and
// 1.95 ms at L = 1024, k = 32, 1000 samples; now 1.2 and 1.3.)
__device__ void refill_body(const Group& g, const RoundCfg& c, const RoundPtrs& p, u32 s,
                            Team team, const Slice& sl, u32* flat_n, u32* stage, u32 stage_words) {
  const u32 L = g.L, k = g.k, W = c.W, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u64 lo = sl.lo, hi = sl.fill_hi, zb = g.base[s] + SM_GAMMA;
  u32* flat = region_of(g, p.flat, s);
  const u32 WL = (L + 31) / 32;
  // lists the live anchors of word i of line q (2 L lines), by a whole warp
  auto put = [&](u32 o, u32 line, u32 i, u32 live) {
    if (i == WL - 1 && (L & 31u)) live &= (1u << (L & 31u)) - 1u;
    const u32 idx0 = o ? (u32)(g.LL + (u64)i * 32 * L + line) : line * L + i * 32;
    const u32 step = o ? L : 1;
    for (u32 m = live; m; m &= m - 1) {
      const u32 bit = __ffs(m) - 1, idx = idx0 + step * bit;
      const u64 key = g.keys ? g.keys[idx] : mix64(zb + SM_GAMMA * idx);
      if (key < lo || key > hi) live &= ~(1u << bit);  // below lo: in the active set already
    }
    if (!__any_sync(FULL, live != 0)) return;
    const u32 nh = __popc(live);
    u32 pre = nh;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 v = __shfl_up_sync(FULL, pre, d);
      if ((int)lane >= d) pre += v;
    }
    u32 at = 0;
    if (lane == 31) at = atomicAdd(flat_n, pre);
    at = __shfl_sync(FULL, at, 31) + pre - nh;
    for (u32 m = live; m; m &= m - 1, ++at)
      if (at < c.cap_flat) flat[at] = idx0 + step * (__ffs(m) - 1);
  };
  if (k <= 33) {
    const u32 items = 2 * L * WL, nt = blockDim.x;
    for (u32 i0 = team.rank * nt; i0 < items; i0 += team.size * nt) {
      const u32 it = i0 + threadIdx.x;
      u32 live = 0, o = 0, line = 0, i = 0;
      if (it < items) {
        const u32 q = it / WL;
        i = it - q * WL;
        o = q >= L;
        line = o ? q - L : q;
        const u32* fl = cover_line(g, c, p, s, o, line) + i;
        u64 v = (u64)fl[1] << 32 | fl[0];
        if (c.bs) {
          const u32* bl = block_line(g, c, p, s, o, line >> c.bs) + i;
          v |= (u64)bl[1] << 32 | bl[0];
        }
        for (u32 m = 1; m < k;) {
          const u32 d = min(m, k - m);
          v |= v >> d;
          m += d;
        }
        live = ~(u32)v;
      }
      put(o, line, i, live);
    }
    return;
  }
  // warps that have room for a line of W words
  const u32 nwarp = min(blockDim.x / 32, stage_words / W);
  if (warp >= nwarp) return;
  u32* ln = stage + warp * W;
  for (u32 q = team.rank * nwarp + warp; q < 2 * L; q += team.size * nwarp) {
    const u32 o = q >= L, line = o ? q - L : q;
    const u32* fl = cover_line(g, c, p, s, o, line);
    const u32* bl = c.bs ? block_line(g, c, p, s, o, line >> c.bs) : fl;
    // lane l keeps words [l per, (l + 1) per); staged, the line is read in
    // coalesced order all the same
    const u32 per = ((W + 31) / 32) | 1u;
    for (u32 i = lane; i < W; i += 32) ln[i] = c.bs ? fl[i] | bl[i] : fl[i];
    __syncwarp();
    const u32 a = min(lane * per, W), b = min(a + per, W);
    u32 first = NONE32;
    for (u32 i = a; i < b && first == NONE32; ++i)
      if (ln[i]) first = i * 32 + __ffs(ln[i]) - 1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 v = __shfl_down_sync(FULL, first, d);
      if (lane + d < 32) first = min(first, v);
    }
    u32 nxt = __shfl_down_sync(FULL, first, 1);  // first covered cell after this lane's words
    if (lane == 31) nxt = NONE32;
    // this lane's words from the last to the first, all lanes in step
    for (u32 st = 0; st < per; ++st) {
      const u32 i = a + per - 1 - st;
      const u32 w = i < b ? ln[i] : 0u;
      u32 live = 0;
      if (i < b && i < WL) {
        const u32 from = w ? 32u - __clz(w) : 0u;  // past the last covered cell
        const u32 end = nxt == NONE32      ? 32u
                        : nxt >= k + i * 32 ? min(nxt - k - i * 32 + 1, 32u)
                                            : 0u;
        if (from < end) live = (0xFFFFFFFFu << from) & (0xFFFFFFFFu >> (32 - end));
      }
      if (w) nxt = i * 32 + __ffs(w) - 1;
      put(o, line, i, live);
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(RD_THREADS) k_refill(Group g, const __grid_constant__ RoundCfg c,
                                                       RoundPtrs p) {
  __shared__ u32 stage[REFILL_WORDS];
  const u32 s = blockIdx.y;
  if (g.st[s].done) return;
  RoundState& r = p.rs[s];
  if (!r.sl.refill) return;
  const Slice sl = r.sl;
  refill_body(g, c, p, s, Team{blockIdx.x, gridDim.x}, sl, &r.flat_n, stage, REFILL_WORDS);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&r.ticket2, 1u) == gridDim.x - 1) {
      __threadfence();
      r.ticket2 = 0;
      Slice nx = sl;
      refill_step(c, nx, __ldcg(&r.flat_n));
      if (nx.refill) r.flat_n = 0;
      r.sl = nx;
    }
  }
}

// Samples not jammed yet.
__global__ void k_round_check(Group g, u32* n_active) {
  const u32 s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < g.n && !g.st[s].done) atomicAdd(n_active, 1u);
}

// ---------------------------------------------------------------------
// k = 1: the two candidates of a cell conflict only with each other, so each
// cell takes the one of smaller priority, in one pass, as node y L + x; its
// contacts are its right and lower neighbour.
// ---------------------------------------------------------------------
__device__ void sites_body(const Group& g, u32 s, Team team) {
  const u32 L = g.L, nt = blockDim.x;
  const u64 zb = g.base[s] + SM_GAMMA;
  const size_t nb = (size_t)s * g.cap_nodes;
  for (u64 i = team.rank * nt + threadIdx.x; i < g.LL; i += team.size * nt) {
    const u64 h = g.keys ? g.keys[i] : mix64(zb + SM_GAMMA * i);
    const u64 v = g.keys ? g.keys[i + g.LL] : mix64(zb + SM_GAMMA * (i + g.LL));
    const u32 o = v < h, y = (u32)i / L, x = (u32)i - y * L;
    g.node_key[nb + i] = o ? v : h;
    g.node_idx[nb + i] = (u32)(i + (o ? g.LL : 0));
    g.node_pos[nb + i] = (o << 31) | (y << 15) | x;
  }
}

__global__ void __launch_bounds__(256) k_sites(Group g) {
  const u32 s = blockIdx.y;
  sites_body(g, s, Team{blockIdx.x, gridDim.x});
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    SampleState& st = g.st[s];
    st.n_nodes = (u32)g.LL;
    st.rounds = 1;
    st.done = 1;
    work_add(g, 0, 2 * g.LL);
    work_add(g, 3, g.LL);
  }
}

__device__ __forceinline__ void contact_counts(SampleState& st, const u32 cnt[3]) {
#pragma unroll
  for (u32 i = 0; i < 3; ++i) {
    const u32 t = __reduce_add_sync(FULL, cnt[i]);
    if ((threadIdx.x & 31) == 0 && t)
      atomicAdd(i == 0 ? &st.contacts_x : i == 1 ? &st.contacts_y : &st.contacts_xy, t);
  }
}

// Edge `at` of a sample: times and links apart, so that a probe reads 8 bytes
// of the edges it leaves out.
__device__ __forceinline__ void put_edge(const Group& g, u32 s, SampleState& st, u32 at, u64 time,
                                         u32 m1, u32 m2, u32 dx, u32 dy) {
  if (at >= g.edge_limit) {
    atomicOr(&st.status, ST_EDGE_OVF);
    return;
  }
  region_of(g, g.etime, s)[at] = time;
  region_of(g, g.elink, s)[at] = make_uint4(m1, m2, (dx & 0xFFFFu) | (dy << 16), 0);
}

// Histogram of a block's edge times, added to the sample's at the end.
struct TimeHist {
  u32* h;
  __device__ __forceinline__ TimeHist(const Group& g, u32* sh) : h(g.ehist ? sh : nullptr) {
    if (h)
      for (u32 i = threadIdx.x; i < EHIST; i += blockDim.x) h[i] = 0;
    __syncthreads();
  }
  __device__ __forceinline__ void add(u64 time, u32 copies) {
    if (h) atomicAdd(&h[time_bin(time)], copies);
  }
  __device__ __forceinline__ void flush(const Group& g, u32 s) {
    __syncthreads();
    if (h)
      for (u32 i = threadIdx.x; i < EHIST; i += blockDim.x)
        if (h[i]) atomicAdd(region_of(g, g.ehist, s) + i, h[i]);
  }
};

__device__ void site_contacts_body(const Group& g, u32 s, Team team, u32* hist_sh) {
  const u32 L = g.L, nt = blockDim.x;
  SampleState& st = g.st[s];
  const u64* K = g.node_key + (size_t)s * g.cap_nodes;
  const u32* P = g.node_pos + (size_t)s * g.cap_nodes;
  TimeHist hist(g, hist_sh);
  u32 cnt[3] = {0, 0, 0};
  for (u64 i = team.rank * nt + threadIdx.x; i < g.LL; i += team.size * nt) {
    const u32 m = (u32)i, y = m / L, x = m - y * L;
    const u32 right = x + 1 == L ? m + 1 - L : m + 1, down = y + 1 == L ? x : m + L;
    const u64 km = K[m];
    const u32 om = P[m] >> 31;
#pragma unroll
    for (u32 dir = 0; dir < 2; ++dir) {
      const u32 b = dir ? down : right;
      const u64 time = tmax(km, K[b]);
      put_edge(g, s, st, 2 * m + dir, time, m, b, dir == 0, dir);
      hist.add(time, 1);
      if (b != m) {
        const u32 kind = om != P[b] >> 31 ? 2u : om;
        cnt[0] += kind == 0;
        cnt[1] += kind == 1;
        cnt[2] += kind == 2;
      }
    }
  }
  contact_counts(st, cnt);
  hist.flush(g, s);
  if (team.rank == 0 && threadIdx.x == 0) st.n_edges = 2 * (u32)g.LL;
}

__global__ void __launch_bounds__(256) k_site_contacts(Group g) {
  __shared__ u32 hist_sh[EHIST];
  if (g.st[blockIdx.y].sdone) return;
  site_contacts_body(g, blockIdx.y, Team{blockIdx.x, gridDim.x}, hist_sh);
}

// ---------------------------------------------------------------------
// Contact graph of the jammed lattice, k >= 2, from the k-mers themselves.
// The lattice edges (a, a + e), e in {+x, +y}, that leave a k-mer of
// orientation o, line l, cells [pos, pos + k) are the one past its last cell
// and the ones from line l to line l + 1.  On line l + 1 lie the parallel
// k-mers anchored less than k away, and the perpendicular ones that start
// there (those that came from line l would cross this one); the cell past
// the end is the first of a parallel k-mer or some cell of a perpendicular
// one.  Each is read off the anchor bits, a word at a time: about k / 8 words
// per k-mer, where reading the owners of all cells costs 4 bytes per cell.
// One edge per pair of k-mers and displacement, its contacts counted by the
// length of the overlap; a parallel run that passes cell 0 counts as two
// (runs start anew there).  Only a ring (k = L) beside itself is a contact
// of a k-mer with itself.
// ---------------------------------------------------------------------
__device__ __forceinline__ u32 anchor_bits(const u32* line, u32 a, u32 n) {
  const u32 w = a >> 5;
  const u32 v = __funnelshift_r(line[w], line[w + 1], a & 31u);
  return n < 32 ? v & ((1u << n) - 1u) : v;
}

template <int G>
__device__ void contacts_body(const Group& g, const RoundCfg& c, const RoundPtrs& p, u32 s,
                              Team team, u32* edges, u32* hist_sh) {
  const u32 L = g.L, k = g.k, tid = threadIdx.x;
  SampleState& st = g.st[s];
  const u32 nn = min(st.n_nodes, g.cap_nodes);
  const size_t nb = (size_t)s * g.cap_nodes;
  const u32* anchor_node = g.owner + (size_t)s * g.LL;
  TimeHist hist(g, hist_sh);
  const u32 j = tid & (G - 1), gpb = blockDim.x / G;
  u32 cnt[3] = {0, 0, 0};
  for (u32 m = team.rank * gpb + tid / G; m < nn; m += team.size * gpb) {
    const u32 pk = g.node_pos[nb + m];
    const u64 key = g.node_key[nb + m];
    const u32 o = pk >> 31, y = (pk >> 15) & 0x7FFFu, x = pk & 0x7FFFu;
    const u32 line = o ? x : y, pos = o ? y : x, ln = line + 1 == L ? 0 : line + 1;
    // contact with the k-mer anchored at (line al, position ap) in the
    // layout of o, displaced by (along, across) lines of o
    auto emit = [&](u32 al, u32 ap, u32 along, u32 across, u32 run, bool mixed, u32 copies) {
      const u32 b = anchor_node[o ? ap * L + al : al * L + ap];
      const u64 kb = g.node_key[nb + b];
      if (b != m) cnt[mixed ? 2 : o] += run;
      const u32 at = atomicAdd(edges, copies);
      const u64 time = tmax(key, kb);
      hist.add(time, copies);
      for (u32 i = 0; i < copies; ++i)
        put_edge(g, s, st, at + i, time, m, b, o ? across : along, o ? along : across);
    };
    // parallel k-mers on the next line
    {
      const u32 a = ring_sub(pos, k - 1, L);
      const u32* al = anchor_line(g, c, p, s, o, o, ln);
      for (u32 w = j; w * 32 < 2 * k - 1; w += G)
        for (u32 v = anchor_bits(al, a + w * 32, 2 * k - 1 - w * 32); v; v &= v - 1) {
          const int d = (int)(w * 32 + __ffs(v) - 1) - (int)(k - 1);
          u32 ap = a + w * 32 + __ffs(v) - 1;
          while (ap >= L) ap -= L;
          // cells first .. last of this k-mer touch the other; is cell 0 of
          // the line among them, other than as the first?
          const u32 first = d > 0 ? d : 0, len = k - (d < 0 ? -d : d);
          const u32 to0 = ring_sub(0, pos + first >= L ? pos + first - L : pos + first, L);
          const bool again = to0 > 0 && to0 < len && !(k == L && d == 0);
          emit(ln, ap, (u32)d, 1, len, false, again ? 2 : 1);
        }
    }
    // perpendicular k-mers that start on the next line
    {
      const u32* al = anchor_line(g, c, p, s, o ^ 1u, o, ln);
      for (u32 w = j; w * 32 < k; w += G)
        for (u32 v = anchor_bits(al, pos + w * 32, k - w * 32); v; v &= v - 1) {
          const u32 i = w * 32 + __ffs(v) - 1;
          emit(ln, pos + i >= L ? pos + i - L : pos + i, i, 1, 1, true, 1);
        }
    }
    // the cell past the end
    if (j == G - 1) {
      const u32 q = pos + k >= L ? pos + k - L : pos + k;
      if (anchor_bits(anchor_line(g, c, p, s, o, o, line), q, 1)) {
        emit(line, q, k, 0, 1, false, 1);
      } else {
        const u32 a = ring_sub(line, k - 1, L);
        const u32* al = anchor_line(g, c, p, s, o ^ 1u, o ^ 1u, q);
        for (u32 w = 0; w * 32 < k; ++w) {
          const u32 v = anchor_bits(al, a + w * 32, k - w * 32);
          if (v) {
            const u32 tt = w * 32 + __ffs(v) - 1;
            const u32 first = a + tt >= L ? a + tt - L : a + tt;
            emit(first, q, k, tt - (k - 1), 1, true, 1);
            break;
          }
        }
      }
    }
  }
  contact_counts(st, cnt);
  hist.flush(g, s);
}

// Six blocks per SM: the pass waits for owner lookups in L2 (issue slots 16%
// busy), and the registers that six leave per thread suffice.  L = 32768,
// k = 4096, 4 samples 1.53 -> 1.26 ms; L = 1024, k = 32, 1000 samples 2.07 ->
// 2.03.
template <int G>
__global__ void __launch_bounds__(256, 6) k_contacts(Group g, const __grid_constant__ RoundCfg c,
                                                  RoundPtrs p) {
  __shared__ u32 hist_sh[EHIST];
  if (g.st[blockIdx.y].sdone) return;
  contacts_body<G>(g, c, p, blockIdx.y, Team{blockIdx.x, gridDim.x},
                   &g.st[blockIdx.y].n_edges, hist_sh);
}

}  // namespace rsak
