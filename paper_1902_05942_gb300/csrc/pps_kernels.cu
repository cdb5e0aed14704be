// Kernels of the hashed path space filter (sm_103a) and their launchers.
//
//  k_fused         the whole frame in one persistent cooperative launch: sweep
//                  of the slot table, key construction (Alg. 1) and probing
//                  insert, accumulation (Sec. 3.2, 3.3.1), temporal blend
//                  (Sec. 3.4.1), one lookup per vertex, separated by grid
//                  barriers; within a phase every warp works alone.
//  k_fused<NEIGH>, k_neighbors
//                  neighborhood-search frames: the persistent kernel lists its
//                  low-count vertices with the lookups, a separate launch
//                  searches them.
//  k_fused_multi   the same phases over the tiles of several views.
//  k_insert, k_add, k_blend_sweep, k_query, k_clear_sweep
//                  the same steps as launches of their own (the split path).
//  k_blend_lookup, k_blend_apply
//                  the blend of a history that follows changes of resolution.
//
// Vertex streams are read with streaming loads (ld.global.cs), a warp's 32
// lanes taking 32 consecutive vertices; table words are read at L2
// (ld.relaxed.gpu / ld.global.cg) because other CTAs write them.
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include "pps_internal.h"

namespace pps {

namespace {

constexpr int kBlock = 256;       // split kernels
constexpr int kTile = 256;        // vertices per warp tile of the split path, at least
constexpr int kTileIds = kTile + 32 * 5;  // cell ids of a unit, such a tile's range (tile_ids, widest batch)
constexpr int kFusedBlock = 512;  // persistent kernels
constexpr int kFusedTile = 256;   // vertices per warp tile, large frames

__device__ __forceinline__ float4 load4(const float* p, size_t j, size_t end, bool vec) {
  if (vec && j + 4 <= end) return __ldcs(reinterpret_cast<const float4*>(p + j));
  float4 v;
  v.x = j < end ? __ldcs(p + j) : 0.f;
  v.y = j + 1 < end ? __ldcs(p + j + 1) : 0.f;
  v.z = j + 2 < end ? __ldcs(p + j + 2) : 0.f;
  v.w = j + 3 < end ? __ldcs(p + j + 3) : 0.f;
  return v;
}

__device__ __forceinline__ float comp(const float4& v, int q) {
  return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w;
}

__device__ __forceinline__ uint32_t vertex_id(const VertexPtrs& v, size_t j) {
  return v.id ? __ldcs(v.id + j) : v.id_base + static_cast<uint32_t>(j);
}

template <typename T>
__device__ __forceinline__ T block_sum(T x) {
  __shared__ T s_part[32];
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) s_part[w] = x;
  __syncthreads();
  T tot = 0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (blockDim.x + 31) / 32; ++i) tot += s_part[i];
  return tot;  // valid in thread 0
}

struct Counters {
  uint32_t ovf = 0, cells = 0;  // per thread (summed to 64 bits per CTA)
};

// ------------------------------------------------------------------ insert
// The insert runs in two passes with a barrier between them.
//
// Pass one (insert_warp) finds or creates every vertex's cell and writes its id
// to the stash.  The vertex that creates a cell owns it and STORES its own
// contribution and a count of one as the cell's accumulator.  Pass two
// (add_warp) adds the other vertices' contributions.  So an accumulator needs
// no clearing, a new cell costs a coalesced store where an atomic on a cold
// line would first fetch it from DRAM (random red.v4: 180 G/s on lines in L2,
// 23 G/s otherwise), and only the vertices that met an existing cell (about
// half) need an atomic, on lines written just before.  HD frame (5.06 M
// vertices, 2^23 slots): insert and accumulation 191 us in one pass with an
// atomic per vertex, 120 + 28 us in two; fixed point 293 us, 130 + 71 us.
//
// A warp inserts alone: no barrier and no shared counter between warps, so a
// warp with long probe sequences holds up no other.  Every key's home slot
// is tried with one compare-and-swap (no load before it: a load followed by a
// compare-and-swap of the same line costs three times the compare-and-swap,
// 42 against 121 G/s on a 64 MB table).  About one key in seven meets another
// key there; finishing those on the spot would make the whole warp wait for
// four or five more memory round trips of a few lanes.  They go into a queue of
// the warp's own in shared memory instead, and while it holds more than a step's
// worth the warp advances 32 at once, each by one step of its probe sequence.
//
// A key that waits there loses its place: later keys fill the slots it would
// have had, and more keys run out of probes (5.06 M vertices, 2^22 slots, 16
// probes: 0.178 % of the vertices, 0.128 % where every key is finished at once).
// So a warp that has seen a key use up a sixth of its probes empties its queue
// after every step from then on: 0.122 % at 242 us instead of 196; the oldest
// entries first instead left 0.171 %.  With 8 probes 1.11 % become 0.95 % (at once
// 0.99 %).  With a quarter of the probes instead of a sixth, 2.94 M vertices in 2^22
// slots lost 253 vertices at 64 probes, 225 like this, 219 at once; with an eighth
// no fewer, but on 9 M vertices with few collisions (2^23 slots, 64 probes) 351 us
// instead of 337.  Where the limit is short such keys are common and the time is
// spent on tables that lose next to nothing, too: 2^23 slots, 16 probes 191 -> 216
// us, temporal 354 -> 372; with 64 probes 190 -> 193 and 354 -> 350.
//
// What bounds pass one now is the keys: without any table access it takes
// 84 us (about 330 instructions per vertex at 8 warps per scheduler, 64
// registers), the compare-and-swaps add 20 us, the queue 20 us.
//
// Queue entries per warp: a step's worth that may stay, and the keys of two rows.
constexpr int kQueue = 96;

// Tables of 2^24 and 2^25 slots, larger than L2 but not by much, read the home
// slot before they try to take it: a compare-and-swap that fails still costs the
// sector's way back to DRAM (random compare-and-swaps 23 G/s on a 1 GB table, loads
// 43 G/s).  Frames without history, without and with the read, us: 2^23 slots 328
// and 341 (9.0 M vertices); 2^24 362 and 354 (9.0 M), 594 and 580 (14.9 M), 1,022 and
// 967 (17.2 M, load 0.8); 2^25 413 and 400, 656 and 640, 2,260 and 2,124 (34.4 M, load
// 0.8); 2^26 1,874 and 2,037 (34.4 M), 3,840 and 4,050 (61 M).
constexpr uint32_t kLookFrom = (1u << 24) - 1u, kLookTo = (1u << 25) - 1u;  // slots - 1

// Tables from 2^25 slots on empty the queue after every step, while the sectors of
// the keys' home slots are still in L2.  Without and with that, us: 2^24 slots 362
// and 378 (9.0 M vertices), 594 and 627 (14.9 M); 2^25 414 and 413, 654 and 656, 2,322
// and 2,260 (34.4 M); 2^26 2,037 and 1,874 (34.4 M), 4,066 and 3,841 (61 M).
constexpr uint32_t kLargeTable = (1u << 25) - 1u;  // slots - 1

// Shared memory of one warp: its queue of keys, and the contributions of a row
// of 32 vertices while equal cells are merged.
struct WarpShared {
  union {
    struct {
      uint32_t h1[kQueue], f[kQueue], step[kQueue], members[kQueue], first[kQueue];
    };
    uint32_t list[kQueue * 5];  // the lookup's low-count vertices
  };
  float row[96];
};

constexpr uint32_t kDeferred = 0xFFFFFFFEu;  // cell id not known yet

// The most cell ids that a warp draws from the range of one tile of `v`
// vertices, W vertices per lane and step: one for each new cell made while it
// works on the tile (its own vertices and up to 32 queued ones), and those its
// lanes hold in reserve.
__host__ __device__ constexpr uint32_t tile_ids(uint32_t v, int batch) { return v + 32u * (batch + 1); }

// What a warp carries from one insert to the next.
template <int W>
struct WarpInsert {
  uint32_t my[W];    // ids reserved for the lane's next new cells (kOverflowSlot: none)
  uint32_t claims;   // ids handed out of the current tile's range (the same in every lane)
  uint32_t id_base;  // that range's first id
  uint32_t queued;   // entries in the queue (the same in every lane)
  uint32_t most;     // entries that may stay in it after a step (the same in every lane)
  Counters cnt;
  __device__ __forceinline__ WarpInsert() : claims(0u), id_base(0u), queued(0u), most(32u) {
#pragma unroll
    for (int q = 0; q < W; ++q) my[q] = kOverflowSlot;
  }
  // Mark the reserved ids that ended up unused, for the passes over t.info.
  __device__ __forceinline__ void retire(const TableDev& t, bool rec) {
#pragma unroll
    for (int q = 0; q < W; ++q) {
      if (rec && my[q] != kOverflowSlot)
        st_once_u4(t.info + my[q], make_uint4(kNoSlot, 0u, 0u, kOverflowSlot));
      my[q] = kOverflowSlot;
    }
  }
  // An id for every lane with `need` that has none in my[q].
  __device__ __forceinline__ void reserve(int q, bool need) {
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, need && my[q] == kOverflowSlot);
    if (m >> lane & 1u) my[q] = id_base + claims + __popc(m & ((1u << lane) - 1u));
    claims += __popc(m);
  }
};

// A new cell `id`: its creator's contribution is its first (own = 0: none is,
// pass two adds them all), and (`rec`) its record {slot, home hash,
// fingerprint}.
__device__ __forceinline__ void create_cell(const TableDev& t, uint32_t id, float r, float g, float b,
                                            uint32_t slot, uint32_t h1, uint32_t f, bool rec,
                                            uint32_t own) {
  if (!own) {
    __stcg(value_ptr(t, id), make_float4(0.f, 0.f, 0.f, 0.f));
    if (t.fixed) __stcg(value_ptr(t, id) + 1, make_float4(0.f, 0.f, 0.f, 0.f));
  } else if (!t.fixed) {
    __stcg(t.acc + id, make_float4(r, g, b, 1.0f));
  } else {
    ulonglong2* a = reinterpret_cast<ulonglong2*>(t.acc64 + 4 * static_cast<size_t>(id));
    __stcg(a, make_ulonglong2(static_cast<unsigned long long>(to_fixed(r)),
                              static_cast<unsigned long long>(to_fixed(g))));
    __stcg(a + 1, make_ulonglong2(static_cast<unsigned long long>(to_fixed(b)), 1ull));
  }
  if (rec) st_once_u4(t.info + id, make_uint4(slot, h1, f, kOverflowSlot));
}

// Advance the last min(32, queued) queue entries by one step of their probe
// sequences: read the rest of the sequence in the slot's sector (one 32-byte
// load, up to four slots), take an empty one with a compare-and-swap; entries
// that met other keys go back into the queue.  Slots are only ever filled
// within a frame, so reading several at once is as good as one after the other:
// the first slot of the sequence that holds the fingerprint or is empty
// decides, and an empty one is taken only by its compare-and-swap.  A step is
// two or three dependent round trips to L2 whatever it reads, so fewer steps
// count, most where the table is full or the frame small: with two slots at a
// time and the colours read after the compare-and-swap a 720p frame took 117.9
// us, like this 114.4.  All lanes.
template <int W, bool KREC = false>
__device__ __forceinline__ void queue_step(const TableDev& t, const VertexPtrs& v, WarpInsert<W>& s,
                                           WarpShared& sh, bool rec, uint32_t own, uint32_t* stash,
                                           uint4* qkw = nullptr) {
  const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
  const uint32_t take = min(32u, s.queued), at = s.queued - take, e = at + lane;
  const bool have = lane < take;
  uint32_t h1 = 0u, f = 0u, step = 0u, members = 0u, first = 0u;
  uint4 kr{};
  if (KREC && have) kr = qkw[e];
  if (have) {
    h1 = sh.h1[e];
    f = sh.f[e];
    step = sh.step[e];
    members = sh.members[e];
    first = sh.first[e];
  }
  s.reserve(0, have);
  __syncwarp();
  uint32_t id = kDeferred;
  if (have) {
    const uint32_t slot0 = (h1 + step) & t.mask, o = slot0 & 3u;
    unsigned long long w[4], a = ~0ull;
    ld_relaxed_u64x4_keep(t.slots + (slot0 - o), w);
    uint32_t hit = 4u;
#pragma unroll
    for (uint32_t k = 3; k < 4u; --k)
      if (k >= o && step + (k - o) < t.max_probes && (w[k] == 0ull || slot_fp(w[k]) == f)) {
        hit = k;
        a = w[k];
      }
    step += hit - o;
    const uint32_t slot = slot0 - o + hit;
    const uint32_t lead = first + __ffs(members) - 1;
    bool made = false;
    float r = 0.f, g = 0.f, b = 0.f;
    if (a == 0ull) {
      a = atomicCAS(t.slots + slot, 0ull, slot_word(f, s.my[0]));
      made = a == 0ull;
      r = __ldg(v.r + lead);
      g = __ldg(v.g + lead);
      b = __ldg(v.b + lead);
    }
    if (made) {
      id = s.my[0];
      create_cell(t, id, r, g, b, slot, h1, f, rec, own);
      if (KREC) __stcg(t.kw + id, kr);
      ++s.cnt.cells;
      s.my[0] = kOverflowSlot;
    } else if (hit < 4u && slot_fp(a) == f) {
      id = slot_id(a);
    } else {
      if (hit < 4u) ++step;  // another key took the slot meanwhile
      if (step >= t.max_probes) {
        id = kOverflowSlot;
        s.cnt.ovf += __popc(members);
      }
    }
    if (id != kDeferred) {
      st_once_u32(stash + lead, made ? id | own : id);
      for (uint32_t m = members & (members - 1u); m; m &= m - 1u)
        st_once_u32(stash + first + __ffs(m) - 1, id);
    }
  }
  const unsigned again = __ballot_sync(0xFFFFFFFFu, id == kDeferred && have);
  if (again >> lane & 1u) {
    const uint32_t o = at + __popc(again & lt);
    sh.h1[o] = h1;
    sh.f[o] = f;
    sh.step[o] = step;
    sh.members[o] = members;
    sh.first[o] = first;
    if (KREC) qkw[o] = kr;
  }
  s.queued = at + __popc(again);
  if (__any_sync(0xFFFFFFFFu, have && 6u * step >= t.max_probes)) s.most = 0u;  // crowded: no key may wait
  __syncwarp();
}

// Pass one for the 32 W vertices from j0 on (those below `end`), one warp:
// lane l takes vertices j0 + l, j0 + 32 + l, ...  Their cell ids go to
// stash[vertex]: the id, with kOwnerBit for the cell's creator, or
// kOverflowSlot on probe overflow; those of queued keys follow later.  New
// cells take ids of the tile's own range; an id that a lane reserved and did
// not need is used for its next new cell.
//
// Equal keys within a row of 32 vertices go through the table once when
// `merge` says so: 1 never; 2 when two neighbouring lanes hold equal keys,
// which one shuffle and a vote find (coherent primary hits repeat keys across
// neighbouring pixels, secondary bounces rarely repeat one within a warp, and
// there the match costs more than the probes it saves); 3 always.
//
// `rec`: write each new cell's record (t.info) for the later blend and clear;
// a frame that neither blends nor clears slot by slot never reads it.
// `own`: kOwnerBit, or 0 on frames whose contributions all wait for pass two.
// KV: the vertices may carry the key variants (distance, extra word).
// KREC: also keep each new cell's quantized key in t.kw; `qkw` holds those of the
// queued keys (finishing every key on the spot instead, a 1.6 M vertex frame with
// migrating history took 229.7 us, with the queue 215.2).
template <int W, bool KV, bool KREC>
__device__ __forceinline__ void insert_warp(const KeyConst& kc, const TableDev& t,
                                            const VertexPtrs& v, size_t j0, size_t end,
                                            WarpInsert<W>& s, WarpShared& sh, bool rec, uint32_t own,
                                            int merge, uint32_t* stash, uint4* qkw = nullptr) {
  const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
  uint32_t h1[W], f[W];
  uint4 kr[W];  // KREC: the quantized keys
  {
    float px[W], py[W], pz[W], nx[W], ny[W], nz[W];
#pragma unroll
    for (int q = 0; q < W; ++q) {
      const size_t j = j0 + 32 * q + lane;
      const bool ok = j < end;
      px[q] = ok ? __ldcs(v.px + j) : 0.f;
      py[q] = ok ? __ldcs(v.py + j) : 0.f;
      pz[q] = ok ? __ldcs(v.pz + j) : 0.f;
      nx[q] = ok ? __ldcs(v.nx + j) : 0.f;
      ny[q] = ok ? __ldcs(v.ny + j) : 0.f;
      nz[q] = ok ? __ldcs(v.nz + j) : 1.f;
    }
#pragma unroll
    for (int q = 0; q < W; ++q) {
      const size_t j = j0 + 32 * q + lane;
      const bool ok = j < end;
      const uint32_t vid = ok ? vertex_id(v, j) : 0u;
      Key k;
      if constexpr (KV || KREC) {
        KeyExtra ke{};
        if (KV && ok) ke = key_extra(v, j);
        const KeyWords kw = key_words(kc, px[q], py[q], pz[q], nx[q], ny[q], nz[q], vid, v.stream_id, ke);
        k = key_hash(kc, kw);
        kr[q] = make_uint4(kw.X, kw.Y, kw.Z, (kw.L & 0xFFu) | (kw.NQ << 8));
      } else {
        k = vertex_key(kc, px[q], py[q], pz[q], nx[q], ny[q], nz[q], vid, v.stream_id);
      }
      h1[q] = k.h1;
      f[q] = k.fp;
    }
  }
  unsigned grp[W];
  uint32_t lead = 0u;  // bit q: this lane leads its group in row q
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const bool ok = j0 + 32 * q + lane < end;
    const unsigned long long kk = (static_cast<unsigned long long>(h1[q]) << 32) | f[q];
    bool match = merge == 3;
    if (merge == 2) {
      const unsigned long long up = __shfl_up_sync(0xFFFFFFFFu, kk, 1);
      match = __ballot_sync(0xFFFFFFFFu, lane > 0 && ok && up == kk) != 0u;
    }
    grp[q] = 1u << lane;
    if (match) grp[q] = __match_any_sync(0xFFFFFFFFu, kk) & __ballot_sync(0xFFFFFFFFu, ok);
    if (ok && (grp[q] & lt) == 0u) lead |= 1u << q;
    s.reserve(q, lead >> q & 1u);
  }
  unsigned long long old[W];
  const bool look = t.mask >= kLookFrom && t.mask <= kLookTo;
#pragma unroll
  for (int q = 0; q < W; ++q) {
    old[q] = 0ull;
    if (look && (lead >> q & 1u)) old[q] = ld_relaxed_u64(t.slots + (h1[q] & t.mask));
  }
#pragma unroll
  for (int q = 0; q < W; ++q)
    if ((lead >> q & 1u) && old[q] == 0ull)
      old[q] = atomicCAS(t.slots + (h1[q] & t.mask), 0ull, slot_word(f[q], s.my[q]));
  float r[W], g[W], b[W];
#pragma unroll
  for (int q = 0; q < W; ++q)
    if (lead >> q & 1u) {
      const size_t j = j0 + 32 * q + lane;
      r[q] = __ldg(v.r + j);
      g[q] = __ldg(v.g + j);
      b[q] = __ldg(v.b + j);
    }
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const size_t j = j0 + 32 * q + lane;
    uint32_t id = kDeferred, owner = 0u;
    if (lead >> q & 1u) {
      const uint32_t slot = h1[q] & t.mask;
      const bool won = old[q] == 0ull;
      if (won)
        id = s.my[q];
      else if (slot_fp(old[q]) == f[q])
        id = slot_id(old[q]);
      else if (t.max_probes == 1u)
        id = kOverflowSlot;
      if (won) {
        if (KREC) __stcg(t.kw + id, kr[q]);
        create_cell(t, id, r[q], g[q], b[q], slot, h1[q], f[q], rec, own);
        owner = own;
        ++s.cnt.cells;
        s.my[q] = kOverflowSlot;
      }
      if (id == kOverflowSlot) s.cnt.ovf += __popc(grp[q]);
    }
    const uint32_t mine = __shfl_sync(0xFFFFFFFFu, id, __ffs(grp[q]) - 1);
    if (j < end && mine != kDeferred) st_once_u32(stash + j, mine | owner);
    const unsigned put = __ballot_sync(0xFFFFFFFFu, (lead >> q & 1u) && id == kDeferred);
    if (put) {
      if (put >> lane & 1u) {
        const uint32_t o = s.queued + __popc(put & lt);
        sh.h1[o] = h1[q];
        sh.f[o] = f[q];
        sh.step[o] = 1u;
        sh.members[o] = grp[q];
        sh.first[o] = static_cast<uint32_t>(j0 + 32 * q);
        if (KREC) qkw[o] = kr[q];
      }
      s.queued += __popc(put);
      __syncwarp();
      if (W > 2)  // (two rows find room)
        while (s.queued > 2u * s.most) queue_step<W, KREC>(t, v, s, sh, rec, own, stash, qkw);
    }
  }
  while (s.queued > (t.mask >= kLargeTable ? 0u : s.most))
    queue_step<W, KREC>(t, v, s, sh, rec, own, stash, qkw);
}

// Pass two for W rows of 32 vertices from j0 on, STEP apart (those below
// `end`), one warp: the contributions of the vertices that do not own their
// cells.  Neighbouring vertices of the same cell are added up first, as in pass
// one.
template <bool FIXED, int W = 4, int STEP = 32>
__device__ __forceinline__ void add_warp_as(const TableDev& t, const VertexPtrs& v, size_t j0, size_t end,
                                            const uint32_t* stash, int merge, WarpShared& sh) {
  const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
  uint32_t id[W];
  float r[W], g[W], b[W];
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const size_t j = j0 + STEP * q + lane;
    id[q] = j < end ? __ldcg(stash + j) : kOverflowSlot;
  }
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const size_t j = j0 + STEP * q + lane;
    if (!(id[q] & kOwnerBit)) {  // neither an owner nor overflowed
      r[q] = __ldcs(v.r + j);
      g[q] = __ldcs(v.g + j);
      b[q] = __ldcs(v.b + j);
    }
  }
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const bool ok = !(id[q] & kOwnerBit);
    long long fr = 0, fg = 0, fb = 0;
    if (FIXED && ok) {
      fr = to_fixed(r[q]);
      fg = to_fixed(g[q]);
      fb = to_fixed(b[q]);
    }
    unsigned grp = 1u << lane;
    if (merge != 1) {
      const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, id[q], 1);
      if (merge == 3 || __ballot_sync(0xFFFFFFFFu, lane > 0 && ok && up == id[q])) {
        grp = __match_any_sync(0xFFFFFFFFu, id[q]);
        if (ok) {
          sh.row[lane] = r[q];
          sh.row[32 + lane] = g[q];
          sh.row[64 + lane] = b[q];
        }
        __syncwarp();
        if (ok && (grp & lt) == 0u) {  // the group's lowest lane
          for (unsigned m = grp & (grp - 1u); m; m &= m - 1u) {
            const int l = __ffs(m) - 1;
            const float mr = sh.row[l], mg = sh.row[32 + l], mb = sh.row[64 + l];
            if (FIXED) {
              fr += to_fixed(mr);
              fg += to_fixed(mg);
              fb += to_fixed(mb);
            } else {
              r[q] = __fadd_rn(r[q], mr);
              g[q] = __fadd_rn(g[q], mg);
              b[q] = __fadd_rn(b[q], mb);
            }
          }
        }
        __syncwarp();
      }
    }
    if (ok && (grp & lt) == 0u) accumulate<FIXED>(t, id[q], r[q], g[q], b[q], fr, fg, fb, __popc(grp));
  }
}

__device__ __forceinline__ void add_warp(const TableDev& t, const VertexPtrs& v, size_t j0, size_t end,
                                         const uint32_t* stash, int merge, WarpShared& sh) {
  if (t.fixed)
    add_warp_as<true>(t, v, j0, end, stash, merge, sh);
  else
    add_warp_as<false>(t, v, j0, end, stash, merge, sh);
}

// Pass two for two neighbouring vertices per lane, j and j + 1 (those below
// `end`), on frames where nobody owns a cell (so that ids may take 32 bits):
// equal cells' contributions are added up first.
template <bool FIXED>
__device__ __forceinline__ void add_pairs(const TableDev& t, const VertexPtrs& v, size_t j, size_t end,
                                          const uint32_t* stash) {
  uint32_t id[2];
  float r[2], g[2], b[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) id[q] = j + q < end ? __ldcg(stash + j + q) : kOverflowSlot;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (id[q] == kOverflowSlot) continue;
    r[q] = __ldcs(v.r + j + q);
    g[q] = __ldcs(v.g + j + q);
    b[q] = __ldcs(v.b + j + q);
  }
  const bool both = id[0] != kOverflowSlot && id[0] == id[1];
  long long fr[2] = {0, 0}, fg[2] = {0, 0}, fb[2] = {0, 0};
  if (FIXED) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (id[q] != kOverflowSlot) {
        fr[q] = to_fixed(r[q]);
        fg[q] = to_fixed(g[q]);
        fb[q] = to_fixed(b[q]);
      }
  }
  if (both) {
    r[0] = __fadd_rn(r[0], r[1]);
    g[0] = __fadd_rn(g[0], g[1]);
    b[0] = __fadd_rn(b[0], b[1]);
    fr[0] += fr[1];
    fg[0] += fg[1];
    fb[0] += fb[1];
  }
  if (id[0] != kOverflowSlot)
    accumulate<FIXED>(t, id[0], r[0], g[0], b[0], fr[0], fg[0], fb[0], both ? 2u : 1u);
  if (id[1] != kOverflowSlot && !both)
    accumulate<FIXED>(t, id[1], r[1], g[1], b[1], fr[1], fg[1], fb[1], 1u);
}

// The cell id of a stash word (kOverflowSlot: probe overflow).
__device__ __forceinline__ uint32_t stash_id(uint32_t w) {
  return w == kOverflowSlot ? w : w & ~kOwnerBit;
}

// Neighborhood search (Sec. 3.3.1) for vertex j, whose own cell holds fewer
// than t.lowcount members: the pooled average of the 3 x 3 x 3 block of cells
// around its cell at the same level and with the same quantized normal.  A
// plain frame pools the cells' sums and counts (FP32 sums, or exact int64
// fixed-point sums with one rounding at the end); after a blend it pools the
// blended values weighted by their counts N.  Cells are visited in a fixed
// order (dx, dy, dz each -1, 0, +1, dz fastest), each found by a read-only
// probe.  Inlined into k_neighbors; the split lookup calls it out of line.
__device__ __forceinline__ Result neighbor_pool_inl(const KeyConst& kc, const TableDev& t,
                                             const VertexPtrs& v, size_t j, bool blended,
                                             Result own) {
  const KeyWords w0 =
      key_words(kc, __ldg(v.px + j), __ldg(v.py + j), __ldg(v.pz + j), __ldg(v.nx + j),
                __ldg(v.ny + j), __ldg(v.nz + j), vertex_id(v, j), v.stream_id, key_extra(v, j));
  float sr = 0.f, sg = 0.f, sb = 0.f;
  long long fr = 0, fg = 0, fb = 0;
  unsigned long long n = 0;
  // three cells (dz = -1, 0, +1) at a time: their first probes, then their
  // values, each as loads in flight together
#pragma unroll 1
  for (int o3 = 0; o3 < 9; ++o3) {
    uint32_t home[3], fp[3], id[3];
    unsigned long long w[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      KeyWords kw = w0;
      kw.X += static_cast<uint32_t>(o3 / 3 - 1);
      kw.Y += static_cast<uint32_t>(o3 % 3 - 1);
      kw.Z += static_cast<uint32_t>(q - 1);
      const Key k = key_hash(kc, kw);
      home[q] = k.h1 & t.mask;
      fp[q] = k.fp;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) w[q] = __ldcg(t.slots + home[q]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (w[q] == 0ull)
        id[q] = kOverflowSlot;
      else if (slot_fp(w[q]) == fp[q])
        id[q] = slot_id(w[q]);
      else  // the home slot holds another key: the rest of the probe sequence
        id[q] = probe_find_from(t, home[q], fp[q], 1u);
    }
    float4 c[3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (id[q] != kOverflowSlot && !(t.fixed && !blended)) c[q] = __ldcg(value_ptr(t, id[q]));
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (id[q] == kOverflowSlot) continue;
      if (blended) {
        const uint32_t N = __float_as_uint(c[q].w);
        const float fN = __uint2float_rn(N);
        sr = __fadd_rn(sr, __fmul_rn(fN, c[q].x));
        sg = __fadd_rn(sg, __fmul_rn(fN, c[q].y));
        sb = __fadd_rn(sb, __fmul_rn(fN, c[q].z));
        n += N;
      } else if (!t.fixed) {
        sr = __fadd_rn(sr, c[q].x);
        sg = __fadd_rn(sg, c[q].y);
        sb = __fadd_rn(sb, c[q].z);
        n += static_cast<unsigned long long>(c[q].w);
      } else {
        const unsigned long long* a = t.acc64 + 4 * static_cast<size_t>(id[q]);
        fr += static_cast<long long>(__ldcg(a + 0));
        fg += static_cast<long long>(__ldcg(a + 1));
        fb += static_cast<long long>(__ldcg(a + 2));
        n += __ldcg(a + 3);
      }
    }
  }
  if (n == 0) return own;  // the own cell is always found; kept as a guard
  Result r;
  const float fn = __ull2float_rn(n);
  if (t.fixed && !blended) {
    r.r = __fdiv_rn(__fmul_rn(__ll2float_rn(fr), 0x1p-24f), fn);
    r.g = __fdiv_rn(__fmul_rn(__ll2float_rn(fg), 0x1p-24f), fn);
    r.b = __fdiv_rn(__fmul_rn(__ll2float_rn(fb), 0x1p-24f), fn);
  } else {
    r.r = __fdiv_rn(sr, fn);
    r.g = __fdiv_rn(sg, fn);
    r.b = __fdiv_rn(sb, fn);
  }
  r.n = static_cast<uint32_t>(min(n, 0xFFFFFFFFull));
  r.status = 5;  // PPS_STATUS_NEIGHBORS
  return r;
}

// The same out of line, for the split lookup (k_query), whose other work
// should not pay the search's registers.
__device__ __noinline__ Result neighbor_pool(const KeyConst& kc, const TableDev& t,
                                             const VertexPtrs& v, size_t j, bool blended,
                                             Result own) {
  return neighbor_pool_inl(kc, t, v, j, blended, own);
}

// Searching similar normals by linear probing (Sec. 3.2.2) for a vertex whose
// cell is `id`: with the normal only in the fingerprint, every cell of the
// voxel has the voxel's home slot and lies within P slots of it, so the walk
// from the home slot to the first empty slot (at most P slots) passes all of
// them, between the entries of other voxels.  Each entry's cell record (its
// quantized key) says whether it is the same voxel (x~, l') with a quantized
// normal within r steps on every axis; those cells are pooled: FP32 sums, or
// exact int64 sums in fixed-point mode, or after a blend the blended values
// weighted by their N.  Kept out of line: only tables with the search pay.
__device__ __noinline__ Result similar_pool(const TableDev& t, uint32_t id, bool blended) {
  const uint4 rec = __ldcg(t.kw + id);
  const uint32_t home = __ldcg(&t.info[id].y) & t.mask;
  const int r = static_cast<int>(t.normal_search) - 1;
  const int qx = static_cast<int>((rec.w >> 8) & 0xFFu);
  const int qy = static_cast<int>((rec.w >> 16) & 0xFFu);
  const int qz = static_cast<int>(rec.w >> 24);
  float sr = 0.f, sg = 0.f, sb = 0.f;
  long long fr = 0, fg = 0, fb = 0;
  unsigned long long n = 0;
#pragma unroll 1
  for (uint32_t p = 0; p < t.max_probes; ++p) {
    const unsigned long long w = __ldcg(t.slots + ((home + p) & t.mask));
    if (w == 0ull) break;
    const uint32_t c = slot_id(w);
    const uint4 o = __ldcg(t.kw + c);
    if (o.x != rec.x || o.y != rec.y || o.z != rec.z || ((o.w ^ rec.w) & 0xFFu)) continue;
    const int dx = abs(static_cast<int>((o.w >> 8) & 0xFFu) - qx);
    const int dy = abs(static_cast<int>((o.w >> 16) & 0xFFu) - qy);
    const int dz = abs(static_cast<int>(o.w >> 24) - qz);
    if (max(dx, max(dy, dz)) > r) continue;
    if (blended) {
      const float4 v = __ldcg(value_ptr(t, c));
      const uint32_t N = __float_as_uint(v.w);
      const float fN = __uint2float_rn(N);
      sr = __fadd_rn(sr, __fmul_rn(fN, v.x));
      sg = __fadd_rn(sg, __fmul_rn(fN, v.y));
      sb = __fadd_rn(sb, __fmul_rn(fN, v.z));
      n += N;
    } else if (!t.fixed) {
      const float4 v = __ldcg(t.acc + c);
      if (v.w >= kExactCountLimit) atomicOr(&t.ctrl->error, kErrCountSaturated);
      sr = __fadd_rn(sr, v.x);
      sg = __fadd_rn(sg, v.y);
      sb = __fadd_rn(sb, v.z);
      n += static_cast<unsigned long long>(v.w);
    } else {
      const unsigned long long* a = t.acc64 + 4 * static_cast<size_t>(c);
      fr += static_cast<long long>(__ldcg(a + 0));
      fg += static_cast<long long>(__ldcg(a + 1));
      fb += static_cast<long long>(__ldcg(a + 2));
      n += __ldcg(a + 3);
    }
  }
  Result res;
  const float fn = __ull2float_rn(n);
  if (t.fixed && !blended) {
    res.r = __fdiv_rn(__fmul_rn(__ll2float_rn(fr), 0x1p-24f), fn);
    res.g = __fdiv_rn(__fmul_rn(__ll2float_rn(fg), 0x1p-24f), fn);
    res.b = __fdiv_rn(__fmul_rn(__ll2float_rn(fb), 0x1p-24f), fn);
  } else {
    res.r = __fdiv_rn(sr, fn);
    res.g = __fdiv_rn(sg, fn);
    res.b = __fdiv_rn(sb, fn);
  }
  res.n = static_cast<uint32_t>(min(n, 0xFFFFFFFFull));
  res.status = res.n < t.lowcount ? 1 : 0;
  return res;
}

// Vertex j with cell `id`: if its cell is low-count, replace its outputs by
// the neighborhood-search result.
__device__ __forceinline__ void neighbors_of_vertex(const KeyConst& kc, const TableDev& t,
                                                    const VertexPtrs& v, const OutPtrs& o,
                                                    size_t j, uint32_t id, bool blended) {
  if (id == kOverflowSlot) return;
  const CellMean m = value_of(t, load_value(t, id, blended), blended);
  if (m.n >= t.lowcount) return;
  const Result r = neighbor_pool(kc, t, v, j, blended, Result{m.r, m.g, m.b, m.n, 1});
  o.r[j] = r.r;
  o.g[j] = r.g;
  o.b[j] = r.b;
  if (o.count) o.count[j] = r.n;
  if (o.status) o.status[j] = r.status;
}

// A queued low-count vertex j: its neighborhood-search result into the
// outputs.  The vertex's own cell is among the 27, so the pooled count is at
// least its own.
__device__ __forceinline__ void neighbors_of_queued(const KeyConst& kc, const TableDev& t,
                                                    const VertexPtrs& v, const OutPtrs& o,
                                                    uint32_t j, bool blended) {
  const Result r = neighbor_pool_inl(kc, t, v, j, blended, Result{o.r[j], o.g[j], o.b[j], 0u, 1});
  o.r[j] = r.r;
  o.g[j] = r.g;
  o.b[j] = r.b;
  if (o.count) o.count[j] = r.n;
  if (o.status) o.status[j] = r.status;
}

// Look up the cells id[0..W-1] (loads issued together) and resolve each vertex:
// cell average / blended value, or its own contribution on overflow.
template <int W>
__device__ __forceinline__ void resolve_batch(const TableDev& t, const VertexPtrs& v, size_t j,
                                              size_t end, const uint32_t (&id)[W], bool blended,
                                              Result (&res)[W]) {
  AccRaw a[W];
#pragma unroll
  for (int q = 0; q < W; ++q)
    if (j + q < end && id[q] != kOverflowSlot) a[q] = load_value(t, id[q], blended);
#pragma unroll
  for (int q = 0; q < W; ++q) {
    res[q] = Result{0.f, 0.f, 0.f, 0u, 0};
    if (j + q >= end) continue;
    if (id[q] == kOverflowSlot) {
      // probe limit exceeded: the unfiltered contribution of the vertex itself
      res[q].r = __ldcs(v.r + j + q);
      res[q].g = __ldcs(v.g + j + q);
      res[q].b = __ldcs(v.b + j + q);
      res[q].status = 2;
    } else {
      const CellMean m = value_of(t, a[q], blended);
      res[q].r = m.r;
      res[q].g = m.g;
      res[q].b = m.b;
      res[q].n = m.n;
      res[q].status = m.n < t.lowcount ? 1 : 0;
    }
  }
}

// Blend the cells of tiles first, first + stride, ... below ntiles (tile_i ids
// each, bcount[tile] of them drawn), one warp.  Every lane carries one cell at a
// time through its probe sequence and takes the next cell as soon as its own
// is stored, so that a long probe holds up its lane only: a round reads one
// history entry per lane, value and fingerprint in one load; an empty entry is
// claimed with a compare-and-swap, an entry of another cell moves the lane's
// probe on.
template <bool EVICT>
__device__ __forceinline__ void blend_tiles(const TableDev& t, uint32_t first, uint32_t stride,
                                            uint32_t ntiles, uint32_t tile_i, float alpha,
                                            unsigned long long& n_hovf) {
  const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
  uint32_t tile = first, pos = 0u, count = tile < ntiles ? __ldcg(t.bcount + tile) : 0u;
  bool busy = false;
  uint32_t d = 0u, h = 0u, f = 0u, step = 0u;
  AccRaw a;
  for (;;) {
    const unsigned idle = __ballot_sync(0xFFFFFFFFu, !busy);
    if (idle && tile < ntiles) {
      const uint32_t k = pos + __popc(idle & lt);
      if (!busy && k < count) {
        d = tile * tile_i + k;
        const uint4 in = ld_once_u4(t.info + d);
        a = load_acc(t, d);
        if (in.x != kNoSlot) {
          busy = true;
          h = in.y & t.hmask;
          f = in.z;
          step = 0u;
        }
      }
      pos += __popc(idle);
      if (pos >= count) {
        tile += stride;
        pos = 0u;
        count = tile < ntiles ? __ldcg(t.bcount + tile) : 0u;
      }
    } else if (idle == 0xFFFFFFFFu) {
      break;  // no tile left, no lane busy
    }
    if (!busy) continue;
    if constexpr (EVICT) {
      bool fresh = true;
      const uint32_t e = hist_claim_evict(t, h, f, &fresh);
      const HistRaw old = e != kOverflowSlot && !fresh ? load_hist(t, e) : HistRaw{0.f, 0.f, 0.f, 0u};
      if (e == kOverflowSlot) ++n_hovf;
      blend_store(t, d, e, (t.hist_rank << 24) | (f & 0xFFFFFFu), mean_of(t, a), old, alpha);
      busy = false;
    } else {
      uint32_t fw;
      HistRaw old = load_hist_fp(t, h, &fw);
      if (fw == 0u) {
        fw = atomicCAS(hist_fp(t, h), 0u, f);
        // claimed, or taken meanwhile: by a cell whose value is this frame's
        if (fw == 0u) fw = f;
        old = HistRaw{0.f, 0.f, 0.f, 0u};
      }
      if (fw == f) {
        blend_store(t, d, h, f, mean_of(t, a), old, alpha);
        busy = false;
      } else if (++step >= t.max_probes) {
        ++n_hovf;
        blend_store(t, d, kOverflowSlot, f, mean_of(t, a), old, alpha);
        busy = false;
      } else {
        h = (h + 1u) & t.hmask;
      }
    }
  }
}

// Empty the slots of the cells [base, base + count).
__device__ __forceinline__ void clear_range(const TableDev& t, uint32_t base, uint32_t count,
                                            uint32_t first, uint32_t stride) {
  for (uint32_t k = first; k < count; k += stride) {
    const uint32_t slot = ld_once_u4(t.info + base + k).x;
    if (slot != kNoSlot) __stcg(t.slots + slot, 0ull);
  }
}

// Zero the whole slot table with 16-byte stores, `gthreads` threads from
// thread `gid`: cheaper than one scattered store per cell once a good share
// of the table is in use.
__device__ __forceinline__ void sweep_slots(const TableDev& t, size_t gid, size_t gthreads) {
  uint4* p = reinterpret_cast<uint4*>(t.slots);
  const size_t n16 = (static_cast<size_t>(t.mask) + 1) / 2;
  for (size_t i = gid; i < n16; i += gthreads) st_zero16_keep(p + i);
}

// ------------------------------------------------------------------ split path
// Pass one of the insert, one warp per tile of tile_v vertices; a tile's new
// cells get ids from the tile's own range, `units` ranges of kTileIds ids from
// unit_base on, whose counts (t.bcount) the later passes go by.
template <int W, bool KREC>
__global__ void __launch_bounds__(kBlock) k_insert(KeyConst kc, TableDev t, VertexPtrs v,
                                                   size_t n, uint32_t* stash, uint32_t unit_base,
                                                   uint32_t tile_v, uint32_t units, uint32_t own,
                                                   int merge) {
  __shared__ WarpShared s_warp[kBlock / 32];
  __shared__ uint4 s_kw[KREC ? kBlock / 32 : 1][kQueue];
  WarpShared& sh = s_warp[threadIdx.x >> 5];
  uint4* qkw = s_kw[KREC ? threadIdx.x >> 5 : 0];
  WarpInsert<W> s;
  const uint32_t tiles = static_cast<uint32_t>((n + tile_v - 1) / tile_v);
  for (uint32_t tile = grid_warp(); tile < tiles; tile += grid_warps()) {
    const uint32_t unit = unit_base + tile * units;
    const size_t t0 = static_cast<size_t>(tile) * tile_v, end = min(n, t0 + tile_v);
    s.claims = 0u;
    s.id_base = unit * kTileIds;
#pragma unroll 1
    for (size_t j0 = t0; j0 < end; j0 += 32 * W)
      insert_warp<W, true, KREC>(kc, t, v, j0, end, s, sh, true, own, merge, stash, qkw);
    if (tile + grid_warps() >= tiles)  // the warp's last
      while (s.queued) queue_step<W, KREC>(t, v, s, sh, true, own, stash, qkw);
    for (uint32_t u = threadIdx.x & 31u; u < units; u += 32)
      t.bcount[unit + u] = s.claims > u * kTileIds ? min(s.claims - u * kTileIds, static_cast<uint32_t>(kTileIds)) : 0u;
  }
  s.retire(t, true);
  const unsigned long long a = block_sum(static_cast<unsigned long long>(s.cnt.ovf));
  const unsigned long long b = block_sum(static_cast<unsigned long long>(s.cnt.cells));
  if (threadIdx.x == 0) {
    if (a) atomicAdd(&t.ctrl->overflow_vertices, a);
    if (b) atomicAdd(&t.ctrl->frame_cells, b);
    if (blockIdx.x == 0) atomicAdd(&t.ctrl->vertices, static_cast<unsigned long long>(n));
  }
}

// Pass two; id_out (nullable): the vertices' cell ids for the caller.
// `ordered`: nobody owns a cell, all contributions in the order of
// kPairsForwards, in tiles of 1,024 vertices, four to a thread.
__global__ void __launch_bounds__(kBlock) k_add(TableDev t, VertexPtrs v, size_t n, const uint32_t* stash,
                                                uint32_t* id_out, int ordered, int merge) {
  __shared__ WarpShared s_warp[kBlock / 32];
  const uint32_t lane = threadIdx.x & 31u;
  if (ordered) {
    for (size_t t0 = blockIdx.x * static_cast<size_t>(4 * kBlock); t0 < n; t0 += gridDim.x * static_cast<size_t>(4 * kBlock)) {
      const size_t j0 = t0 + 4 * threadIdx.x;
      for (size_t j = j0; j < j0 + 4; j += 2) {
        if (t.fixed)
          add_pairs<true>(t, v, j, n, stash);
        else
          add_pairs<false>(t, v, j, n, stash);
      }
      if (id_out)
        for (size_t j = j0; j < min(n, j0 + 4); ++j) id_out[j] = stash[j];
    }
    return;
  }
  for (size_t j0 = grid_warp() * static_cast<size_t>(128); j0 < n; j0 += grid_warps() * static_cast<size_t>(128)) {
    add_warp(t, v, j0, n, stash, merge, s_warp[threadIdx.x >> 5]);
    if (id_out)
      for (size_t j = j0 + lane; j < min(n, j0 + 128); j += 32) id_out[j] = stash_id(stash[j]);
  }
}

__global__ void __launch_bounds__(kBlock) k_query(KeyConst kc, TableDev t, VertexPtrs v, size_t n,
                                                  const uint32_t* id_in, OutPtrs o, int vec,
                                                  int ovec, int blended, uint32_t id_limit) {
  const size_t ngroups = (n + 3) / 4;
  for (size_t gi = blockIdx.x * (size_t)blockDim.x + threadIdx.x; gi < ngroups;
       gi += (size_t)gridDim.x * blockDim.x) {
    const size_t j = gi * 4;
    uint32_t id[4];
    if (id_in) {
#pragma unroll
      for (int q = 0; q < 4; ++q) id[q] = j + q < n ? __ldcs(id_in + j + q) : kOverflowSlot;
    } else {
      const float4 PX = load4(v.px, j, n, vec), PY = load4(v.py, j, n, vec),
                   PZ = load4(v.pz, j, n, vec);
      const float4 NX = load4(v.nx, j, n, vec), NY = load4(v.ny, j, n, vec),
                   NZ = load4(v.nz, j, n, vec);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        id[q] = kOverflowSlot;
        if (j + q < n) {
          const Key k = vertex_key(kc, comp(PX, q), comp(PY, q), comp(PZ, q), comp(NX, q),
                                   comp(NY, q), comp(NZ, q), vertex_id(v, j + q), v.stream_id,
                                   key_extra(v, j + q));
          id[q] = probe_find(t, k.h1 & t.mask, k.fp);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (id[q] != kOverflowSlot && id[q] >= id_limit) {  // not a cell of this frame
        atomicOr(&t.ctrl->error, kErrBadSlot);
        id[q] = kOverflowSlot;
      }
    }
    Result res[4];
    resolve_batch<4>(t, v, j, n, id, blended != 0, res);
    if (t.normal_search) {
#pragma unroll 1
      for (int q = 0; q < 4; ++q)
        if (j + q < n && id[q] != kOverflowSlot) res[q] = similar_pool(t, id[q], blended != 0);
    }
    store_batch(o, j, n, ovec != 0, res);
    if (t.neighbors) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (j + q < n) neighbors_of_vertex(kc, t, v, o, j + q, id[q], blended != 0);
    }
  }
}

__global__ void __launch_bounds__(kBlock) k_blend_sweep(TableDev t, uint32_t ntiles, float alpha) {
  unsigned long long n_hovf = 0;
  if (t.hist_evict)
    blend_tiles<true>(t, grid_warp(), grid_warps(), ntiles, kTileIds, alpha, n_hovf);
  else
    blend_tiles<false>(t, grid_warp(), grid_warps(), ntiles, kTileIds, alpha, n_hovf);
  const unsigned long long h = block_sum(n_hovf);
  if (threadIdx.x == 0 && h) atomicAdd(&t.ctrl->hist_overflow, h);
}

// Changes in resolution across frames (Sec. 3.4.2), for a cell whose history
// entry is new this frame; `rec` is the cell's quantized key.  Resolution
// decreased: the history of its eight finer children (2 x~ + {0,1}^3, level
// l' - 1, same quantized normal) is added up, sums and counts, giving
// sum(N_i c_i) / sum(N_i) with count sum(N_i) (FP32, children in the order
// dx, dy, dz, the last fastest).  Otherwise, resolution increased: its coarser
// parent (floor(x~ / 2), level l' + 1) passes on its average with count
// ceil(N / 8).  Read-only probes; an entry claimed during this frame holds
// N = 0 and counts as absent, so the result is the history as it was before
// the frame.  Kept out of line: only new entries pay for it.
__device__ __forceinline__ uint32_t hist_find(const TableDev& t, uint32_t home, uint32_t f) {
  for (uint32_t p = 0; p < t.max_probes; ++p) {
    const uint32_t h = (home + p) & t.hmask;
    const uint32_t w = __ldcg(hist_fp(t, h));
    if (w == 0u) return kOverflowSlot;
    if (w == f) return h;
  }
  return kOverflowSlot;
}

__device__ __noinline__ HistRaw migrate_history(const KeyConst& kc, const TableDev& t, uint4 rec) {
  KeyWords w;
  w.X = rec.x;
  w.Y = rec.y;
  w.Z = rec.z;
  w.L = static_cast<uint32_t>(static_cast<int32_t>(static_cast<int8_t>(rec.w & 0xFFu)));
  w.NQ = rec.w >> 8;
  w.EX = 0u;
  w.has_ex = false;
  float sr = 0.f, sg = 0.f, sb = 0.f;
  uint32_t sn = 0u;
  for (uint32_t d = 0; d < 8; ++d) {
    KeyWords c = w;
    c.X = 2u * w.X + (d >> 2);
    c.Y = 2u * w.Y + ((d >> 1) & 1u);
    c.Z = 2u * w.Z + (d & 1u);
    c.L = w.L - 1u;
    const Key k = key_hash(kc, c);
    const uint32_t h = hist_find(t, k.h1 & t.hmask, k.fp);
    if (h == kOverflowSlot) continue;
    const HistRaw o = load_hist(t, h);
    if (o.n == 0u) continue;
    const float fn = __uint2float_rn(o.n);
    sr = __fadd_rn(sr, __fmul_rn(fn, o.r));
    sg = __fadd_rn(sg, __fmul_rn(fn, o.g));
    sb = __fadd_rn(sb, __fmul_rn(fn, o.b));
    sn += o.n;
  }
  if (sn) {
    const float fn = __uint2float_rn(sn);
    return HistRaw{__fdiv_rn(sr, fn), __fdiv_rn(sg, fn), __fdiv_rn(sb, fn), sn};
  }
  KeyWords p = w;
  p.X = static_cast<uint32_t>(static_cast<int32_t>(w.X) >> 1);
  p.Y = static_cast<uint32_t>(static_cast<int32_t>(w.Y) >> 1);
  p.Z = static_cast<uint32_t>(static_cast<int32_t>(w.Z) >> 1);
  p.L = w.L + 1u;
  const Key k = key_hash(kc, p);
  const uint32_t h = hist_find(t, k.h1 & t.hmask, k.fp);
  if (h != kOverflowSlot) {
    HistRaw o = load_hist(t, h);
    if (o.n) {
      o.n = (o.n + 7u) / 8u;
      return o;
    }
  }
  return HistRaw{0.f, 0.f, 0.f, 0u};
}

// The blend of a table whose history follows changes of resolution, in two
// launches so that every migration reads the history as it was before the
// frame: k_blend_lookup finds or claims each cell's history entry and keeps
// the value its blend starts from (own, migrated, or none) in t.hold and the
// entry in info.w; k_blend_apply blends and stores.
__global__ void __launch_bounds__(kBlock) k_blend_lookup(KeyConst kc, TableDev t, uint32_t ntiles) {
  unsigned long long n_hovf = 0;
  for (uint32_t tile = grid_warp(); tile < ntiles; tile += grid_warps()) {
    const uint32_t base = tile * kTileIds, count = t.bcount[tile];
    for (uint32_t k = threadIdx.x & 31u; k < count; k += 32) {
      const uint32_t d = base + k;
      const uint4 in = __ldcg(t.info + d);
      if (in.x == kNoSlot) continue;
      const uint32_t home = in.y & t.hmask, f = in.z;
      const uint32_t old = atomicCAS(hist_fp(t, home), 0u, f);
      const uint32_t h = old == 0u || old == f ? home : hist_probe_rest(t, home, f, 1u);
      HistRaw hv{0.f, 0.f, 0.f, 0u};
      if (h == kOverflowSlot) {
        ++n_hovf;
      } else {
        hv = load_hist(t, h);
        if (hv.n == 0u) hv = migrate_history(kc, t, __ldcg(t.kw + d));
      }
      __stcg(t.hold + d, make_float4(hv.r, hv.g, hv.b, __uint_as_float(hv.n)));
      __stcg(&t.info[d].w, h);
    }
  }
  const unsigned long long s = block_sum(n_hovf);
  if (threadIdx.x == 0 && s) atomicAdd(&t.ctrl->hist_overflow, s);
}

__global__ void __launch_bounds__(kBlock) k_blend_apply(TableDev t, uint32_t ntiles, float alpha) {
  for (uint32_t tile = grid_warp(); tile < ntiles; tile += grid_warps()) {
    const uint32_t base = tile * kTileIds, count = t.bcount[tile];
    for (uint32_t k = threadIdx.x & 31u; k < count; k += 32) {
      const uint32_t d = base + k;
      const uint4 in = __ldcg(t.info + d);
      if (in.x == kNoSlot) continue;
      const AccRaw a = load_acc(t, d);
      const float4 o = __ldcg(t.hold + d);
      blend_store(t, d, in.w, in.z, mean_of(t, a), HistRaw{o.x, o.y, o.z, __float_as_uint(o.w)}, alpha);
    }
  }
}

// Neighborhood search of the low-count vertices that the persistent kernel
// queued, one per thread.
__global__ void __launch_bounds__(kBlock) k_neighbors(KeyConst kc, TableDev t, VertexPtrs v,
                                                      OutPtrs o, const uint32_t* nq, int blended) {
  const unsigned long long cnt = __ldcg(&t.ctrl->neigh_count);
  for (unsigned long long i = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x;
       i < cnt; i += static_cast<unsigned long long>(gridDim.x) * blockDim.x)
    neighbors_of_queued(kc, t, v, o, __ldcs(nq + i), blended != 0);
}

__global__ void __launch_bounds__(kBlock) k_clear_sweep(TableDev t, uint32_t ntiles, uint32_t tile_i,
                                                        int sweep) {
  if (sweep || __ldcg(&t.ctrl->left))
    sweep_slots(t, blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x,
                static_cast<size_t>(gridDim.x) * blockDim.x);
  else
    for (uint32_t tile = grid_warp(); tile < ntiles; tile += grid_warps())
      clear_range(t, tile * tile_i, t.bcount[tile], threadIdx.x & 31u, 32);
}

__global__ void __launch_bounds__(kBlock) k_keys(KeyConst kc, VertexPtrs v, size_t n,
                                                 uint32_t* h_out, uint32_t* f_out) {
  for (size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x; j < n;
       j += (size_t)gridDim.x * blockDim.x) {
    const Key k = vertex_key(kc, __ldcs(v.px + j), __ldcs(v.py + j), __ldcs(v.pz + j),
                             __ldcs(v.nx + j), __ldcs(v.ny + j), __ldcs(v.nz + j),
                             vertex_id(v, j), v.stream_id, key_extra(v, j));
    h_out[j] = k.h1;
    f_out[j] = k.fp;
  }
}

__global__ void __launch_bounds__(kBlock) k_count_nonzero(const unsigned char* base, uint32_t stride,
                                                          uint32_t off, uint32_t width, uint64_t n,
                                                          unsigned long long* out) {
  unsigned long long c = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const unsigned char* p = base + i * stride + off;
    c += width == 8 ? (*reinterpret_cast<const unsigned long long*>(p) != 0ull)
                    : (*reinterpret_cast<const uint32_t*>(p) != 0u);
  }
  const unsigned long long s = block_sum(c);
  if (threadIdx.x == 0 && s) atomicAdd(out, s);
}

// ------------------------------------------------------------------ fused path
struct FusedArgs {
  KeyConst kc;
  TableDev t;
  VertexPtrs v;
  OutPtrs o;
  size_t n;
  uint32_t tile_v;   // vertices (and cell ids) per warp tile
  uint32_t* stash;   // each vertex's cell id
  float alpha;
  int blend;
  int sweep;         // zero the whole slot table first, instead of the frame's slots at the end
  uint32_t* nq;      // neighborhood search: the queue of low-count vertices
  int merge;         // merging of equal keys within a warp (insert_warp)
  int backwards;     // insert from the end of the vertex stream
  int order;         // AddOrder of pass two
};

// The warp's list of low-count vertices (in its shared memory, the key queue's
// place) to the end of the frame's.
constexpr uint32_t kLowList = kQueue * 5;
__device__ __forceinline__ void flush_low(const TableDev& t, uint32_t* nq, WarpShared& sh, uint32_t& queued) {
  const uint32_t lane = threadIdx.x & 31u;
  __syncwarp();
  unsigned long long b = 0ull;
  if (lane == 0 && queued) b = atomicAdd(&t.ctrl->neigh_count, static_cast<unsigned long long>(queued));
  b = __shfl_sync(0xFFFFFFFFu, b, 0);
  for (uint32_t i = lane; i < queued; i += 32) nq[b + i] = sh.list[i];
  __syncwarp();
  queued = 0u;
}

// One lookup for each of the 128 vertices from j0 on (those below `end`), one
// warp, four rows of 32: the vertices of a row mostly have cells of
// neighbouring ids, so a row's loads fall on few lines.
template <bool NEIGH>
__device__ __forceinline__ void lookup_warp(const TableDev& t, const VertexPtrs& v, const OutPtrs& o,
                                            size_t j0, size_t end, const uint32_t* stash,
                                            bool blended, uint32_t* nq, WarpShared& sh, uint32_t& queued) {
  const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
  uint32_t id[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const size_t j = j0 + 32 * q + lane;
    id[q] = j < end ? stash_id(__ldcs(stash + j)) : kOverflowSlot;
  }
  AccRaw a[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (id[q] != kOverflowSlot) a[q] = load_value(t, id[q], blended);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const size_t j = j0 + 32 * q + lane;
    bool low = false;
    if (j < end) {
      CellMean m;
      uint32_t status;
      if (id[q] == kOverflowSlot) {
        // probe limit exceeded: the unfiltered contribution of the vertex itself
        m = CellMean{__ldcs(v.r + j), __ldcs(v.g + j), __ldcs(v.b + j), 0u};
        status = 2u;
      } else {
        m = value_of(t, a[q], blended);
        low = m.n < t.lowcount;
        status = low ? 1u : 0u;
      }
      __stcs(o.r + j, m.r);
      __stcs(o.g + j, m.g);
      __stcs(o.b + j, m.b);
      if (o.count) __stcs(o.count + j, m.n);
      if (o.status) __stcs(o.status + j, static_cast<uint8_t>(status));
    }
    // neighborhood search: list the low-count vertices, for k_neighbors, which
    // searches them at full occupancy (so the irregular searches neither
    // unbalance this kernel's warps nor cost it registers).  They gather in
    // shared memory first: one atomic on the list's counter per few hundred.
    if constexpr (NEIGH) {
      const unsigned m = __ballot_sync(0xFFFFFFFFu, low);
      if (low) sh.list[queued + __popc(m & lt)] = static_cast<uint32_t>(j);
      queued += __popc(m);
    }
  }
  if constexpr (NEIGH)
    if (queued > kLowList - 128u) flush_low(t, nq, sh, queued);
}

// Pass two of a frame whose half-precision history is blended (all threads):
// nobody owns a cell, and tiles of 2,048 vertices are handed out from a counter,
// in the order of FusedArgs::order and within a tile
//   kRowsBackwards  1,024 vertices at a time, the rows of 32 of a warp 512 apart;
//   kPairsForwards  1,024 vertices at a time, two neighbouring ones per lane,
// which is about the order that frames of this kind have always been added up in:
// one tile after the other, first or last part of the stream first.  An FP32 sum
// depends on the order of its additions in its last bit, and where the stored
// average lies next to the middle of two halves, that bit moves it by a unit of
// binary16, up to 9.8e-4 of the value, so for these histories a different
// order is a visible difference: with the creator's contribution first and the
// rest in any order, a frame of 1.66 M vertices had 33,300 cells with another
// sum than the insert in one pass gave, in this order 12,000, and 11,400 from
// one run of that insert to the next; of 61 M vertices (2^26 slots) 364,000,
// 74,000 and 44,000.  It costs 4 and 340 us there (of 116 and
// 8,200 us a frame).
__device__ __forceinline__ void add_ordered(const FusedArgs& a, WarpShared& sh) {
  constexpr uint32_t kHalf = 1024, kSpan = 2 * kHalf;
  static_assert(kFusedBlock == 512, "two rows, or one row of pairs, per warp and half tile");
  __shared__ uint32_t s_next;
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  const uint32_t ntiles = static_cast<uint32_t>((a.n + kSpan - 1) / kSpan);
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_next = static_cast<uint32_t>(atomicAdd(&a.t.ctrl->tile_next, 1ull));
    __syncthreads();
    const uint32_t k = s_next;
    if (k >= ntiles) return;
    const bool back = a.order == kRowsBackwards;
    const size_t t0 = static_cast<size_t>(back ? ntiles - 1u - k : k) * kSpan;
    for (uint32_t c = 0; c < kSpan; c += kHalf) {
      if (back) {
        add_warp_as<false, 2, kFusedBlock>(a.t, a.v, t0 + c + 32 * warp, a.n, a.stash, a.merge, sh);
        __syncthreads();
      } else {
        add_pairs<false>(a.t, a.v, t0 + c + 64 * warp + 2 * lane, a.n, a.stash);
      }
    }
  }
}

// The persistent kernel.  Every phase is a loop of independent warps:
//   0   the slot table is emptied (sweep), just before it is filled, so that
//       the compare-and-swaps meet it in L2; so is what another launch left;
//   A1  keys, probing insert, in tiles of a.tile_v vertices, every nw-th tile
//       to one warp (a counter that hands them out costs more than it
//       balances: its atomics serialize on one address, HD 146 us against 126),
//       from the end of the vertex stream on frames that have always been
//       inserted so (backwards: such a stream is bounce-major; its
//       secondary-bounce tiles, whose vertices nearly all create cells of their
//       own and cost the most, go first and let the cheap primary-hit tiles
//       balance the warps at the end) and from its start on the others, above
//       all on large tables: there the cells with many members, the primary
//       hits, have to come first, into an empty table, or a quarter more
//       vertices run out of probes (61 M vertices, 2^26 slots, 32 probes);
//       a tile's new cells take ids from the tile's own range, and each
//       vertex's cell id goes to the stash;
//   A2  accumulation (128 vertices at a time, or in order: add_ordered);
//   B   temporal blend of each tile's new cells;
//   C   one lookup per vertex (128 at a time); a frame that did not sweep
//       empties its slots,
// with a grid barrier between them.
template <bool TEMPORAL, int W, bool EVICT = false, bool NEIGH = false, bool KV = false>
__global__ void __launch_bounds__(kFusedBlock, W == 4 ? 1 : 2) k_fused(FusedArgs a) {
  __shared__ WarpShared s_warp[kFusedBlock / 32];
  WarpShared& sh = s_warp[threadIdx.x >> 5];
  const TableDev& t = a.t;
  const uint32_t tile_v = a.tile_v, tile_i = tile_ids(tile_v, W), lane = threadIdx.x & 31u;
  const uint32_t ntiles = static_cast<uint32_t>((a.n + tile_v - 1) / tile_v);
  const uint32_t gw = grid_warp(), nw = grid_warps();
  const bool blended = TEMPORAL && a.blend;
  if (blockIdx.x == 0 && threadIdx.x == 0) reset_counters(t.ctrl);
  if (a.sweep || __ldcg(&t.ctrl->left)) {  // (the same answer in every CTA: it changes after the next barrier)
    sweep_slots(t, blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x,
                static_cast<size_t>(gridDim.x) * blockDim.x);
    if (!grid_barrier(t.ctrl, gridDim.x)) return;
  }

  unsigned long long n_ovf, n_cells;
  {
    WarpInsert<W> s;
    const bool rec = blended || !a.sweep;
    const uint32_t own = TEMPORAL && a.order ? 0u : kOwnerBit;
    for (uint32_t k = gw; k < ntiles; k += nw) {
      const uint32_t tile = a.backwards ? ntiles - 1u - k : k;
      const size_t t0 = static_cast<size_t>(tile) * tile_v;
      const size_t end = min(a.n, t0 + tile_v);
      s.claims = 0u;
      s.id_base = tile * tile_i;
#pragma unroll 1
      for (size_t j0 = t0; j0 < end; j0 += 32 * W)
        insert_warp<W, KV, false>(a.kc, t, a.v, j0, end, s, sh, rec, own, a.merge, a.stash);
      if (k + nw >= ntiles)  // the warp's last tile
        while (s.queued) queue_step<W>(t, a.v, s, sh, rec, own, a.stash);
      if (lane == 0) __stcg(t.bcount + tile, s.claims);
    }
    s.retire(t, rec);
    n_ovf = block_sum(static_cast<unsigned long long>(s.cnt.ovf));
    n_cells = block_sum(static_cast<unsigned long long>(s.cnt.cells));
  }
  if (!grid_barrier(t.ctrl, gridDim.x)) return;
  if (threadIdx.x == 0) {
    if (n_ovf) atomicAdd(&t.ctrl->overflow_vertices, n_ovf);
    if (n_cells) atomicAdd(&t.ctrl->frame_cells, n_cells);
    if (blockIdx.x == 0) {
      atomicAdd(&t.ctrl->vertices, static_cast<unsigned long long>(a.n));
      t.ctrl->left = a.sweep ? 1ull : 0ull;
    }
  }

  if (TEMPORAL && a.order)
    add_ordered(a, sh);
  else
    for (size_t j = gw * static_cast<size_t>(128); j < a.n; j += nw * static_cast<size_t>(128))
      add_warp(t, a.v, j, a.n, a.stash, a.merge, sh);
  if (!grid_barrier(t.ctrl, gridDim.x)) return;

  if (blended) {
    unsigned long long n_hovf = 0;
    blend_tiles<EVICT>(t, gw, nw, ntiles, tile_i, a.alpha, n_hovf);
    const unsigned long long h = block_sum(n_hovf);
    if (threadIdx.x == 0 && h) atomicAdd(&t.ctrl->hist_overflow, h);
    if (!grid_barrier(t.ctrl, gridDim.x)) return;
  }

  uint32_t low = 0u;  // listed vertices not handed on yet
  for (size_t j = gw * static_cast<size_t>(128); j < a.n; j += nw * static_cast<size_t>(128))
    lookup_warp<NEIGH>(t, a.v, a.o, j, a.n, a.stash, blended, a.nq, sh, low);
  if (NEIGH) flush_low(t, a.nq, sh, low);
  if (!NEIGH && !a.sweep)  // (the neighborhood search still reads the slots)
    for (uint32_t tile = gw; tile < ntiles; tile += nw)
      clear_range(t, tile * tile_i, __ldcg(t.bcount + tile), lane, 32);
}

// The batched persistent kernel: the same phases over the tiles of several
// views, each with its own table.  Tiles are numbered across views (view v
// owns tiles [tile_base, tile_base + ntiles)); the insert and the blend give a
// warp every nw-th tile, the other phases a contiguous run.  A warp keeps the
// descriptor of the view it is working on in shared memory of its own.
struct MultiArgs {
  const ViewDesc* views;
  Ctrl* ctrl;  // grid barrier of the batch
  uint32_t* stash;  // indexed by tile, tile_v words each
  uint32_t nviews, total_tiles, tile_v;
  float alpha;
  int ordered;  // a view adds its contributions up in order
};

// The warp's copy of the descriptor of the view that tile gt belongs to;
// `cur` is the view it holds.  All lanes.
__device__ __forceinline__ void take_view(ViewDesc* mine, const MultiArgs& a, uint32_t gt,
                                          uint32_t& cur) {
  uint32_t v = cur == kOverflowSlot || gt < mine->tile_base ? 0u : cur;
  while (v + 1 < a.nviews && __ldg(&a.views[v + 1].tile_base) <= gt) ++v;
  if (v == cur) return;
  __syncwarp();
  const int words = static_cast<int>(sizeof(ViewDesc) / sizeof(uint32_t));
  for (int i = threadIdx.x & 31; i < words; i += 32)
    reinterpret_cast<uint32_t*>(mine)[i] = __ldg(reinterpret_cast<const uint32_t*>(a.views + v) + i);
  cur = v;
  __syncwarp();
}

template <bool TEMPORAL, int W, int BLOCK>
__global__ void __launch_bounds__(BLOCK, (W == 4 ? 1 : 2) * (kFusedBlock / BLOCK)) k_fused_multi(MultiArgs a) {
  __shared__ __align__(16) ViewDesc s_vd[BLOCK / 32];
  __shared__ WarpShared s_warp[BLOCK / 32];
  WarpShared& sh = s_warp[threadIdx.x >> 5];
  const uint32_t lane = threadIdx.x & 31u, tile_v = a.tile_v, tile_i = tile_ids(tile_v, W);
  ViewDesc& vd = s_vd[threadIdx.x >> 5];
  uint32_t cur = kOverflowSlot;  // the view in vd
  // this warp's run of tiles in the later phases
  const uint64_t gw = grid_warp(), nw = grid_warps();
  const uint32_t run0 = static_cast<uint32_t>(gw * a.total_tiles / nw);
  const uint32_t run1 = static_cast<uint32_t>((gw + 1) * a.total_tiles / nw);

  if (threadIdx.x == 0)
    for (uint32_t v = blockIdx.x; v < a.nviews; v += gridDim.x) reset_counters(a.views[v].t.ctrl);
  if (blockIdx.x == 0 && threadIdx.x == 0) reset_counters(a.ctrl);
  // empty the slot tables of the views that are swept, or were left full
  for (uint32_t v = 0; v < a.nviews; ++v) {
    take_view(&vd, a, __ldg(&a.views[v].tile_base), cur);
    if (cur == v && (vd.sweep || __ldcg(&vd.t.ctrl->left)))
      sweep_slots(vd.t, blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x,
                  static_cast<size_t>(gridDim.x) * blockDim.x);
  }
  cur = kOverflowSlot;
  if (!grid_barrier(a.ctrl, gridDim.x)) return;

  {
    WarpInsert<W> s;
    uint32_t last = 0u;  // the last tile worked on
    auto ids = [&]() { return a.stash + static_cast<size_t>(vd.tile_base) * tile_v; };
    auto own = [&]() { return TEMPORAL && vd.ordered ? 0u : kOwnerBit; };
    auto flush = [&]() {  // leave the view in vd
      while (s.queued) queue_step<W>(vd.t, vd.v, s, sh, true, own(), ids());
      if (lane == 0) __stcg(vd.t.bcount + last, s.claims);
      unsigned long long o = s.cnt.ovf, c = s.cnt.cells;
      for (int off = 16; off > 0; off >>= 1) {
        o += __shfl_xor_sync(0xFFFFFFFFu, o, off);
        c += __shfl_xor_sync(0xFFFFFFFFu, c, off);
      }
      if (lane == 0) {
        if (o) atomicAdd(&vd.t.ctrl->overflow_vertices, o);
        if (c) atomicAdd(&vd.t.ctrl->frame_cells, c);
      }
      s.cnt = Counters{};
      s.most = 32u;
      s.retire(vd.t, true);  // reserved ids belong to the view
    };
    for (uint32_t gt = gw; gt < a.total_tiles; gt += nw) {
      if (cur != kOverflowSlot && gt - vd.tile_base >= vd.ntiles) flush();
      take_view(&vd, a, gt, cur);
      last = gt - vd.tile_base;
      const size_t t0 = static_cast<size_t>(last) * tile_v;
      const size_t end = min(static_cast<size_t>(vd.n), t0 + tile_v);
      s.claims = 0u;
      s.id_base = last * tile_i;
#pragma unroll 1
      for (size_t j0 = t0; j0 < end; j0 += 32 * W)
        insert_warp<W, false, false>(vd.kc, vd.t, vd.v, j0, end, s, sh, true, own(), 2, ids());
      if (lane == 0) __stcg(vd.t.bcount + last, s.claims);
    }
    if (cur != kOverflowSlot) flush();
    for (uint32_t v = blockIdx.x; v < a.nviews; v += gridDim.x)
      if (threadIdx.x == 0)
        atomicAdd(&a.views[v].t.ctrl->vertices, static_cast<unsigned long long>(a.views[v].n));
  }
  if (!grid_barrier(a.ctrl, gridDim.x)) return;
  if (threadIdx.x == 0)
    for (uint32_t v = blockIdx.x; v < a.nviews; v += gridDim.x)
      if (a.views[v].ntiles) a.views[v].t.ctrl->left = a.views[v].sweep ? 1ull : 0ull;

  auto add_tile = [&](uint32_t gt) {
    take_view(&vd, a, gt, cur);
    const size_t t0 = static_cast<size_t>(gt - vd.tile_base) * tile_v;
    const size_t end = min(static_cast<size_t>(vd.n), t0 + tile_v);
    const uint32_t* ids = a.stash + static_cast<size_t>(vd.tile_base) * tile_v;
    if (TEMPORAL && vd.ordered)
      for (size_t j = t0; j < end; j += 64) add_pairs<false>(vd.t, vd.v, j + 2 * lane, end, ids);
    else
      for (size_t j = t0; j < end; j += 128) add_warp(vd.t, vd.v, j, end, ids, 2, sh);
  };
  if (TEMPORAL && a.ordered) {
    // as in add_ordered, forwards, a tile per warp
    __shared__ uint32_t s_next;
    for (;;) {
      __syncthreads();
      if (threadIdx.x == 0) s_next = static_cast<uint32_t>(atomicAdd(&a.ctrl->tile_next, 1ull));
      __syncthreads();
      const uint64_t first = static_cast<uint64_t>(s_next) * (BLOCK / 32);
      if (first >= a.total_tiles) break;
      const uint64_t gt = first + (threadIdx.x >> 5);
      if (gt < a.total_tiles) add_tile(static_cast<uint32_t>(gt));
    }
  } else {
    for (uint32_t gt = run0; gt < run1; ++gt) add_tile(gt);
  }
  if (!grid_barrier(a.ctrl, gridDim.x)) return;

  if (TEMPORAL) {
    // strided tiles: a view's costly (incoherent) tiles go to many warps
    for (uint64_t gt = gw; gt < a.total_tiles;) {
      take_view(&vd, a, static_cast<uint32_t>(gt), cur);
      if (vd.blended) {
        unsigned long long n_hovf = 0;
        blend_tiles<false>(vd.t, static_cast<uint32_t>(gt - vd.tile_base), static_cast<uint32_t>(nw), vd.ntiles, tile_i,
                           a.alpha, n_hovf);
        if (n_hovf) atomicAdd(&vd.t.ctrl->hist_overflow, n_hovf);
      }
      gt += (vd.tile_base + static_cast<uint64_t>(vd.ntiles) - gt + nw - 1) / nw * nw;  // past this view
    }
    if (!grid_barrier(a.ctrl, gridDim.x)) return;
  }

  for (uint32_t gt = run0; gt < run1; ++gt) {
    take_view(&vd, a, gt, cur);
    const size_t t0 = static_cast<size_t>(gt - vd.tile_base) * tile_v;
    const size_t end = min(static_cast<size_t>(vd.n), t0 + tile_v);
    uint32_t low = 0u;
    for (size_t j = t0; j < end; j += 128)
      lookup_warp<false>(vd.t, vd.v, vd.o, j, end, a.stash + static_cast<size_t>(vd.tile_base) * tile_v,
                         TEMPORAL && vd.blended, nullptr, sh, low);
  }
  for (uint32_t gt = run0; gt < run1; ++gt) {
    take_view(&vd, a, gt, cur);
    const uint32_t tile = gt - vd.tile_base;
    if (!vd.sweep) clear_range(vd.t, tile * tile_i, __ldcg(vd.t.bcount + tile), lane, 32);
  }
}

int split_grid(size_t work_items) {
  const size_t want = (work_items + kBlock - 1) / kBlock;
  const size_t cap = static_cast<size_t>(sm_count()) * 8;
  return static_cast<int>(std::max<size_t>(1, std::min(want, cap)));
}

}  // namespace

int sm_count() {
  static int cached = 0;
  if (!cached) {
    int dev = 0, c = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
    cached = c > 0 ? c : 1;
  }
  return cached;
}

int split_unit_ids() { return kTileIds; }

// Vertices per warp tile of the split path: 256, or more on frames so large that
// every warp still gets tiles enough; a larger tile wastes fewer ids on those its
// warp keeps in reserve (1.63 ids a vertex for 256 vertices, 1.22 for 1,024, 1.12 for
// 4,096, 1.02 for 16,384).
static uint32_t split_tile(size_t n) {
  uint32_t v = kTile;
  while (v < 16384u && n >= static_cast<size_t>(v) * 4 * 16384) v *= 4;
  return v;
}
static uint32_t tile_units(uint32_t tile_v) { return (tile_ids(tile_v, 4) + kTileIds - 1) / kTileIds; }

size_t split_units(size_t n) {
  const uint32_t v = split_tile(n);
  return (n + v - 1) / v * tile_units(v);
}
size_t fused_cells(size_t n, uint32_t tile, int batch) {
  return (n + tile - 1) / tile * tile_ids(tile, batch);
}

// Vertices per warp tile of the persistent kernels: 256, or fewer so that a
// small frame still gives every warp of the GPU work.
uint32_t fused_tile(size_t n, int batch) {
  const size_t warps = static_cast<size_t>(sm_count()) * 32;
  uint32_t v = kFusedTile;
  while (v > 32u * batch && n < 2 * warps * v) v /= 2;
  return v;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static bool vec_inputs(const VertexPtrs& v) {
  return aligned16(v.px) && aligned16(v.py) && aligned16(v.pz) && aligned16(v.nx) &&
         aligned16(v.ny) && aligned16(v.nz) && aligned16(v.r) && aligned16(v.g) &&
         aligned16(v.b);
}

static bool vec_outputs(const OutPtrs& o) {
  return aligned16(o.r) && aligned16(o.g) && aligned16(o.b) && (!o.count || aligned16(o.count)) &&
         (!o.status || (reinterpret_cast<uintptr_t>(o.status) & 3u) == 0);
}

cudaError_t launch_insert(const KeyConst& kc, const TableDev& t, const VertexPtrs& v, size_t n,
                          uint32_t* stash, uint32_t* id_out, uint32_t unit_base, bool wide, int batch,
                          int merge, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const uint32_t tile_v = split_tile(n), units = tile_units(tile_v);
  const int grid = split_grid((n + tile_v - 1) / tile_v * 32);
  const bool ordered = wide || add_order(t, false) != kAnyOrder;
  const uint32_t own = ordered ? 0u : kOwnerBit;
  if (t.hist_migrate || t.normal_search) {  // keep each new cell's quantized key
    if (batch == 2)
      k_insert<2, true><<<grid, kBlock, 0, st>>>(kc, t, v, n, stash, unit_base, tile_v, units, own, merge);
    else
      k_insert<4, true><<<grid, kBlock, 0, st>>>(kc, t, v, n, stash, unit_base, tile_v, units, own, merge);
  } else if (batch == 2) {
    k_insert<2, false><<<grid, kBlock, 0, st>>>(kc, t, v, n, stash, unit_base, tile_v, units, own, merge);
  } else {
    k_insert<4, false><<<grid, kBlock, 0, st>>>(kc, t, v, n, stash, unit_base, tile_v, units, own, merge);
  }
  k_add<<<split_grid((n + 127) / 128 * 32), kBlock, 0, st>>>(t, v, n, stash, id_out, ordered ? 1 : 0,
                                                            merge);
  return cudaGetLastError();
}

cudaError_t launch_query(const KeyConst& kc, const TableDev& t, const VertexPtrs& v, size_t n,
                         const uint32_t* id_in, const OutPtrs& o, bool blended, uint32_t id_limit,
                         cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_query<<<split_grid((n + 3) / 4), kBlock, 0, st>>>(kc, t, v, n, id_in, o,
                                                      vec_inputs(v) ? 1 : 0,
                                                      vec_outputs(o) ? 1 : 0, blended ? 1 : 0,
                                                      id_limit);
  return cudaGetLastError();
}

cudaError_t launch_keys(const KeyConst& kc, const VertexPtrs& v, size_t n, uint32_t* h_out,
                        uint32_t* f_out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_keys<<<split_grid(n), kBlock, 0, st>>>(kc, v, n, h_out, f_out);
  return cudaGetLastError();
}

cudaError_t launch_blend(const KeyConst& kc, const TableDev& t, uint32_t ntiles, float alpha,
                         cudaStream_t st) {
  if (ntiles == 0) return cudaSuccess;
  const int grid = split_grid(static_cast<size_t>(ntiles) * 32);
  if (t.hist_migrate) {
    k_blend_lookup<<<grid, kBlock, 0, st>>>(kc, t, ntiles);
    k_blend_apply<<<grid, kBlock, 0, st>>>(t, ntiles, alpha);
  } else {
    k_blend_sweep<<<grid, kBlock, 0, st>>>(t, ntiles, alpha);
  }
  return cudaGetLastError();
}

// Sweeping the slot table pays once the frame's vertices reach an eighth of it.
static bool sweep_pays(const TableDev& t, size_t vertices) {
  return vertices >= (static_cast<size_t>(t.mask) + 1) / 8;
}

cudaError_t launch_clear(const TableDev& t, uint32_t ntiles, cudaStream_t st) {
  const int sweep = sweep_pays(t, static_cast<size_t>(ntiles) * kTile) ? 1 : 0;
  // (a launch without tiles is there for slots that may have been left)
  const int grid = split_grid(sweep || !ntiles ? t.mask / 2 + size_t{1} : static_cast<size_t>(ntiles) * 32);
  k_clear_sweep<<<grid, kBlock, 0, st>>>(t, ntiles, kTileIds, sweep);
  return cudaGetLastError();
}

// Evicting history: when the per-table epoch runs out, every entry's
// priority drops by `by` (at least 1 remains), keeping the order of recent
// entries.
__global__ void __launch_bounds__(kBlock) k_hist_age(TableDev t, uint32_t by) {
  const size_t Th = static_cast<size_t>(t.hmask) + 1;
  for (size_t h = blockIdx.x * (size_t)blockDim.x + threadIdx.x; h < Th;
       h += (size_t)gridDim.x * blockDim.x) {
    uint32_t* fp = hist_fp(t, static_cast<uint32_t>(h));
    const uint32_t w = *fp;
    if (w == 0u) continue;
    const uint32_t r = w >> 24;
    *fp = ((r > by ? r - by : 1u) << 24) | (w & 0xFFFFFFu);
  }
}

cudaError_t launch_hist_age(const TableDev& t, uint32_t by, cudaStream_t st) {
  k_hist_age<<<sm_count() * 8, kBlock, 0, st>>>(t, by);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(kBlock) k_combine_coarse(size_t n, const uint8_t* fine_status,
                                                           OutPtrs c, OutPtrs o) {
  for (size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x; j < n;
       j += (size_t)gridDim.x * blockDim.x) {
    if (fine_status[j] != 1 || c.status[j] == 2) continue;
    o.r[j] = c.r[j];
    o.g[j] = c.g[j];
    o.b[j] = c.b[j];
    if (o.count) o.count[j] = c.count[j];
    if (o.status) o.status[j] = 4;  // PPS_STATUS_COARSE
  }
}

cudaError_t launch_combine_coarse(size_t n, const uint8_t* fine_status, const OutPtrs& coarse,
                                  const OutPtrs& o, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const size_t blocks = std::min<size_t>((n + kBlock - 1) / kBlock, static_cast<size_t>(sm_count()) * 8);
  k_combine_coarse<<<static_cast<unsigned>(blocks), kBlock, 0, st>>>(n, fine_status, coarse, o);
  return cudaGetLastError();
}

cudaError_t launch_count_nonzero(const void* base, uint32_t stride, uint32_t off, uint32_t width,
                                 uint64_t n, unsigned long long* out, cudaStream_t st) {
  k_count_nonzero<<<sm_count() * 4, kBlock, 0, st>>>(static_cast<const unsigned char*>(base),
                                                     stride, off, width, n, out);
  return cudaGetLastError();
}

template <bool TEMPORAL, bool EVICT, bool NEIGH>
static const void* fused_fn(int batch, bool kv) {
  if (kv)
    return batch == 2 ? reinterpret_cast<const void*>(k_fused<TEMPORAL, 2, EVICT, NEIGH, true>)
                      : reinterpret_cast<const void*>(k_fused<TEMPORAL, 4, EVICT, NEIGH, true>);
  return batch == 2 ? reinterpret_cast<const void*>(k_fused<TEMPORAL, 2, EVICT, NEIGH>)
                    : reinterpret_cast<const void*>(k_fused<TEMPORAL, 4, EVICT, NEIGH>);
}

// The kernel for a frame: with or without a history, an evicting one or not,
// with or without the neighborhood search, with or without key variants.
static const void* fused_kernel(const FusedPlan& p) {
  if (p.temporal && p.evict)
    return p.neigh ? fused_fn<true, true, true>(p.batch, p.kv) : fused_fn<true, true, false>(p.batch, p.kv);
  if (p.temporal)
    return p.neigh ? fused_fn<true, false, true>(p.batch, p.kv) : fused_fn<true, false, false>(p.batch, p.kv);
  return p.neigh ? fused_fn<false, false, true>(p.batch, p.kv) : fused_fn<false, false, false>(p.batch, p.kv);
}

// CTAs of `fn` that are resident at once on one multiprocessor (asked once per
// kernel).
static cudaError_t resident_ctas(const void* fn, int block, int* out) {
  static std::mutex mu;
  static std::vector<std::pair<const void*, int>> known;
  std::lock_guard<std::mutex> lock(mu);
  for (const auto& k : known)
    if (k.first == fn) {
      *out = k.second;
      return cudaSuccess;
    }
  int nb = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, block, 0);
  if (e != cudaSuccess) return e;
  if (nb < 1) return cudaErrorInvalidConfiguration;
  known.emplace_back(fn, nb);
  *out = nb;
  return cudaSuccess;
}

// CTAs of a persistent launch over `ntiles` warp tiles: all that are resident
// at once, or one per four tiles for a small frame (a tile per scheduler), so
// that its grid barriers wait for no idle CTAs; but one at least for 32,768 slots
// to be swept, or a few vertices on a large table would leave that to a few CTAs
// (pps_filter_noalloc on 2^20 slots: one vertex 139 us without this, 16.5 with it,
// 1,000 vertices 46 and 18.5).
static int fused_grid(const void* fn, int block, size_t ntiles, size_t swept, cudaError_t* err) {
  int nb = 0;
  *err = resident_ctas(fn, block, &nb);
  if (*err != cudaSuccess) return 0;
  const size_t most = static_cast<size_t>(sm_count()) * std::min(nb, 1024 / block);
  const size_t want = std::max((ntiles + 3) / 4, swept / 32768);
  return static_cast<int>(std::max<size_t>(1, std::min(most, want)));
}

cudaError_t plan_fused(size_t n, size_t max_cells, FusedPlan* plan) {
  cudaError_t e = cudaSuccess;
  plan->evict = plan->evict && plan->temporal;
  plan->block = kFusedBlock;
  plan->tile = fused_tile(n, plan->batch);
  while (plan->tile < kFusedTile && fused_cells(n, plan->tile, plan->batch) > max_cells) plan->tile *= 2;
  const size_t ntiles = (n + plan->tile - 1) / plan->tile;
  plan->grid = fused_grid(fused_kernel(*plan), kFusedBlock, ntiles, plan->swept, &e);
  return e;
}

cudaError_t launch_fused(const KeyConst& kc, const TableDev& t, const VertexPtrs& v, size_t n,
                         const OutPtrs& o, bool blend, float alpha, const FusedPlan& plan, uint32_t* stash, uint32_t* nq, cudaStream_t st) {
  FusedArgs a;
  a.kc = kc;
  a.t = t;
  a.v = v;
  a.o = o;
  a.n = n;
  a.tile_v = plan.tile;
  a.stash = stash;
  a.alpha = alpha;
  a.blend = blend ? 1 : 0;
  a.sweep = plan.sweep ? 1 : 0;
  a.nq = nq;
  a.merge = plan.merge;
  a.backwards = plan.backwards ? 1 : 0;
  a.order = plan.order;
  void* args[] = {&a};
  cudaError_t e = cudaLaunchCooperativeKernel(fused_kernel(plan), dim3(plan.grid), dim3(plan.block), args,
                                              0, st);
  if (e != cudaSuccess || !plan.neigh) return e;
  k_neighbors<<<sm_count() * 8, kBlock, 0, st>>>(kc, t, v, o, nq, blend ? 1 : 0);
  if (!plan.sweep) {
    const uint32_t ntiles = static_cast<uint32_t>((n + plan.tile - 1) / plan.tile);
    k_clear_sweep<<<split_grid(static_cast<size_t>(ntiles) * 32), kBlock, 0, st>>>(
        t, ntiles, tile_ids(plan.tile, plan.batch), 0);
  }
  return cudaGetLastError();
}

AddOrder add_order(const TableDev& t, bool backwards) {
  if (t.hist_mode != 2 || t.fixed) return kAnyOrder;
  return backwards ? kRowsBackwards : kPairsForwards;
}

bool sweep_pays_host(const TableDev& t, size_t vertices) { return sweep_pays(t, vertices); }

template <bool TEMPORAL, int W>
static const void* multi_fn(int block) {
  return block == 256 ? reinterpret_cast<const void*>(k_fused_multi<TEMPORAL, W, 256>)
                      : reinterpret_cast<const void*>(k_fused_multi<TEMPORAL, W, 512>);
}

static const void* multi_kernel(bool temporal, int batch, int block) {
  if (temporal) return batch == 2 ? multi_fn<true, 2>(block) : multi_fn<true, 4>(block);
  return batch == 2 ? multi_fn<false, 2>(block) : multi_fn<false, 4>(block);
}

cudaError_t plan_multi(size_t total_tiles, uint32_t tile, size_t swept, bool temporal, int batch,
                       int block, MultiPlan* plan) {
  cudaError_t e = cudaSuccess;
  plan->block = block == 256 ? 256 : kFusedBlock;
  plan->batch = batch;
  plan->tile = tile;
  plan->grid = fused_grid(multi_kernel(temporal, batch, plan->block), plan->block, total_tiles, swept,
                          &e);
  return e;
}

cudaError_t launch_multi(const ViewDesc* views, uint32_t nviews, uint32_t total_tiles, Ctrl* ctrl,
                         bool temporal, bool ordered, float alpha, const MultiPlan& plan,
                         uint32_t* stash, cudaStream_t st) {
  MultiArgs a;
  a.views = views;
  a.ctrl = ctrl;
  a.stash = stash;
  a.nviews = nviews;
  a.total_tiles = total_tiles;
  a.tile_v = plan.tile;
  a.alpha = alpha;
  a.ordered = ordered ? 1 : 0;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(multi_kernel(temporal, plan.batch, plan.block), dim3(plan.grid),
                                     dim3(plan.block), args, 0, st);
}

}  // namespace pps
