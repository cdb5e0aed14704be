// Device-side building blocks of the hashed path space filter (sm_103a).
//
// Key construction follows Algorithm 1; the table follows Sec. 3.2 (open
// addressing, linear probing with a step limit) and Sec. 3.2.1 (32-bit
// fingerprints, 0 = empty); accumulation is the scatter form of Sec. 3.2 (one
// atomic add per component plus a counter, Sec. 3.3.1); temporal blending is
// Sec. 3.4.1.
//
// Every floating-point step of key construction uses an explicitly rounded
// intrinsic (__fadd_rn, __fmul_rn, __fdiv_rn, __fsqrt_rn), so nothing is
// contracted into an FMA and the integer keys are reproducible bit for bit by
// any IEEE-754 implementation that performs the same operations in the same
// order.
#pragma once

#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace pps {

constexpr uint32_t kOverflowSlot = 0xFFFFFFFFu;  // slot_out value on probe overflow
constexpr uint32_t kOwnerBit = 0x80000000u;      // stash word: this vertex owns its cell

// ---------------------------------------------------------------- parameters
struct KeyConst {
  float cam[3];
  float k;  // fl32(voxel_scale * pixel_angle)
  uint32_t hseed_home, hseed_fp;
  uint32_t mask;  // T - 1
  uint32_t max_probes;
  int32_t lod_min, lod_max;
  uint32_t jitter, nih;  // jitter on/off, normal in home hash
  // Philox4x32-10 keys of the jitter draw's ten rounds, two words each (seed and
  // frame, bumped by the Weyl constants; set_round_keys).  They are the same for
  // every vertex of a frame, so the kernels read them from their parameters, in
  // the order of their use (an HD frame 196.0 us with the first and the second
  // words in arrays of their own, 190.6 us like this).
  uint32_t rk[20];
  uint32_t seed, frame;
};

// Fill kc.rk from kc.seed and kc.frame; call whenever either changes.
__host__ __device__ inline void set_round_keys(KeyConst& kc) {
  uint32_t k0 = kc.seed, k1 = kc.frame;
  for (int r = 0; r < 10; ++r) {
    kc.rk[2 * r] = k0;
    kc.rk[2 * r + 1] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

// Per-frame and lifetime counters plus the device error word and the state of
// the grid barrier used by the persistent filter kernel.
struct Ctrl {
  unsigned long long frame_cells;
  unsigned long long overflow_vertices;
  unsigned long long vertices;
  unsigned long long hist_overflow;
  unsigned long long neigh_count;  // persistent kernel: low-count vertices queued for the search
  unsigned long long tile_next;    // ordered additions: next tile to hand out
  // The slots still hold the frame of a launch that empties them before it uses
  // them: the next launch that does not do so of itself has to.  It is kept here
  // and not on the host, which does not see the launches of a replayed graph.
  unsigned long long left;
  unsigned int error;
  unsigned int bar_count;
  unsigned int pad[2];
};
constexpr size_t kCtrlEmptyBytes = 7 * sizeof(unsigned long long);  // counters and `left`: zero once the slots are empty
constexpr size_t kCtrlErrorBytes = 2 * sizeof(unsigned int);        // error word and barrier, from `error` on

enum : unsigned int {
  kErrBarrierTimeout = 1u,
  kErrBadSlot = 2u,
  // FP32 accumulation: a cell reached 2^24 members, past which adding 1.0f to
  // its FP32 count no longer changes it, so its count and average are not
  // exact (fixed-point accumulation counts in 64 bits and has no such limit)
  kErrCountSaturated = 4u,
};

constexpr float kExactCountLimit = 16777216.0f;  // 2^24

// Table layout.
//
// The hashed table of Sec. 3.2 holds, per slot, only the key's 32-bit
// fingerprint and the id of its cell: slot = (id + 1) << 32 | fingerprint, 0 =
// empty.  At 8 bytes a slot, a table of 2^23 slots (64 MB) stays in L2, where
// the probing compare-and-swaps run several times faster than on DRAM-backed
// lines.  The cells themselves live in dense arrays indexed by the cell id:
//   acc   {sum r, sum g, sum b, count} FP32 (16 B), or int64 sums (32 B, fixed)
//   info  {slot, home hash, fingerprint, history cell} (16 B)
//   kw    the cell's quantized key {x~x, x~y, x~z, l' & 0xFF | q(n) << 8}
//         (16 B, tables whose history follows changes of resolution)
//   hold  the old value {c r, c g, c b, N} the cell's blend starts from
//         (16 B, same tables)
// Ids are handed out per block of vertices: a CTA (or a tile of the split
// path) owns the id range [block * B, block * B + count[block]), where B is its
// vertex count, so a frame's cells occupy a few contiguous runs and the
// per-cell passes (blend, clear) are coalesced sweeps over them.
//
// History cell, FP32 (32 B): [0,16) {c r, c g, c b, N}, [16,20) fingerprint.
// History cell, FP16 (16 B): [0,8) {half r, half g, half b, uint16 N}, [8,12) fp.
// After the blend the cell's acc holds the blended value {c r, c g, c b, N}.
struct TableDev {
  unsigned long long* slots;  // [T] index of the hashed table
  float4* acc;                // [D] FP32 accumulators (FP32 mode)
  unsigned long long* acc64;  // [D][4] fixed-point accumulators (fixed mode)
  uint4* info;                // [D] {slot, h1, fingerprint, history cell}
  uint4* kw;                  // [D] quantized keys (hist_migrate)
  float4* hold;               // [D] old values of the blend (hist_migrate)
  uint32_t* bcount;           // [blocks] cells claimed per id block
  unsigned char* hcells;      // [Th] history cells (temporal tables)
  Ctrl* ctrl;
  uint32_t hstride;           // bytes per history cell: 32 or 16
  uint32_t hfp_off;           // fingerprint offset in a history cell: 16 or 8
  uint32_t mask;              // T - 1
  uint32_t hmask;             // Th - 1
  uint32_t max_probes;
  uint32_t lowcount;
  int fixed;                  // accumulation mode
  int hist_mode;              // 0 none, 1 FP32, 2 FP16
  int neighbors;              // low-count vertices take the 3x3x3 pooled average
  int hist_evict;             // history fingerprints carry a priority (evicting table)
  int hist_migrate;           // history follows changes of resolution (Sec. 3.4.2)
  uint32_t hist_rank;         // evicting table: this frame's priority (blend epoch)
  uint32_t normal_search;     // 0 off; r + 1: lookups pool the voxel's normals within r steps
};

constexpr uint32_t kNoSlot = 0xFFFFFFFFu;  // info.x of an id reserved but not used

struct VertexPtrs {
  const float *px, *py, *pz, *nx, *ny, *nz, *r, *g, *b;
  const uint32_t* id;
  uint32_t id_base;
  uint32_t stream_id;
  const float* dist;       // optional distance for the level of detail
  const uint32_t* extra;   // optional extra key word
};

struct OutPtrs {
  float *r, *g, *b;
  uint32_t* count;
  uint8_t* status;
};

// ---------------------------------------------------------------- Philox4x32-10
// Salmon et al., SC'11: ten rounds of two 32x32->64 multiplies; the key is
// bumped by the Weyl constants between rounds.
// The first two output words of one draw, the round keys taken from the key
// constants.
__device__ __forceinline__ uint2 philox_first2_rk(uint32_t c0, uint32_t c1, const KeyConst& kc) {
  uint32_t x0 = c0, x1 = c1, x2 = 0u, x3 = 0u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t k0 = kc.rk[2 * r], k1 = kc.rk[2 * r + 1];
    // 32 x 32 -> 64-bit products, one instruction each
    const unsigned long long p0 = 0xD2511F53ull * x0, p1 = 0xCD9E8D57ull * x2;
    const uint32_t lo0 = static_cast<uint32_t>(p0), hi0 = static_cast<uint32_t>(p0 >> 32);
    const uint32_t lo1 = static_cast<uint32_t>(p1), hi1 = static_cast<uint32_t>(p1 >> 32);
    const uint32_t n0 = hi1 ^ x1 ^ k0, n2 = hi0 ^ x3 ^ k1;
    x0 = n0;
    x1 = lo1;
    x2 = n2;
    x3 = lo0;
  }
  return make_uint2(x0, x1);
}

// ---------------------------------------------------------------- MurmurHash3_x86_32
__device__ __forceinline__ uint32_t mm_body(uint32_t h, uint32_t k) {
  k *= 0xCC9E2D51u;
  k = __funnelshift_l(k, k, 15);
  k *= 0x1B873593u;
  h ^= k;
  h = __funnelshift_l(h, h, 13);
  return h * 5u + 0xE6546B64u;
}

__device__ __forceinline__ uint32_t mm_final(uint32_t h, uint32_t nbytes) {
  h ^= nbytes;
  h ^= h >> 16;
  h *= 0x85EBCA6Bu;
  h ^= h >> 13;
  h *= 0xC2B2AE35u;
  h ^= h >> 16;
  return h;
}

// ---------------------------------------------------------------- Algorithm 1
__device__ __forceinline__ float pow2_int(int l) {
  return __uint_as_float(static_cast<uint32_t>(l + 127) << 23);
}

// |p_cam - x|^2 in FP32, one rounding per operation.
__device__ __forceinline__ float camera_distance2(const KeyConst& kc, float x, float y, float z) {
  const float dx = __fsub_rn(kc.cam[0], x);
  const float dy = __fsub_rn(kc.cam[1], y);
  const float dz = __fsub_rn(kc.cam[2], z);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// |p_cam - x| in FP32, one rounding per operation.
__device__ __forceinline__ float camera_distance(const KeyConst& kc, float x, float y, float z) {
  return __fsqrt_rn(camera_distance2(kc, x, y, z));
}

// floor(log2 F) of an FP32 product F = k * d, from its exponent bits.
__device__ __forceinline__ int level_of(const KeyConst& kc, float F) {
  const int e = static_cast<int>((__float_as_uint(F) >> 23) & 0xFFu) - 127;
  return min(max(e, kc.lod_min), kc.lod_max);
}

// floor(log2(k * d)) from the exponent bits of the FP32 product.
__device__ __forceinline__ int level_at(const KeyConst& kc, float d) { return level_of(kc, __fmul_rn(kc.k, d)); }

// Algorithm 1's level_of_detail(|p_cam - x|).
//
// Only the exponent of F = fl(k * fl(sqrt(d2))) counts.  sqrt.approx is within
// 2^-23 of the square root relatively, and sqrt.rn and the products round by
// 2^-24 each, so the product with the approximate root is within 4 units of
// the last place of F, and both have the same exponent unless the approximate
// one lies within 8 units of a power of two (0 and infinity among them; a
// subnormal d2 reads as 0): there, about once in half a million vertices, the
// correctly rounded root decides.  It costs some ten instructions and a branch
// each of the two times a key needs a level (keys alone, 4.2 M vertices: 309
// instructions a vertex and 51.6 us with it, 286 and 49.1 us without it and
// with the fused forms below).
__device__ __forceinline__ int level_of_detail(const KeyConst& kc, float x, float y, float z) {
  const float d2 = camera_distance2(kc, x, y, z);
  float d;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(d) : "f"(d2));
  float F = __fmul_rn(kc.k, d);
  if (((__float_as_uint(F) + 8u) & 0x7FFFFFu) < 16u) F = __fmul_rn(kc.k, __fsqrt_rn(d2));
  return level_of(kc, F);
}

// floor(v), v's product with a power of two, as int32: clamped to
// [-2^31, 2147483520] (the conversion rounds down).
__device__ __forceinline__ int32_t quantize_coord(float v, float inv) {
  const float q = __fmul_rn(v, inv);
  return __float2int_rd(fminf(fmaxf(q, -2147483648.0f), 2147483520.0f));
}

// clamp(floor((c + 1) * 128), 0, 255).  Scaling by 128 is exact, so the fused
// form rounds once, like c + 1; the conversion to 8 bits truncates and clamps.
__device__ __forceinline__ uint32_t quantize_normal(float c) {
  uint32_t q;
  asm("{\n .reg .u8 t;\n cvt.rzi.u8.f32 t, %1;\n cvt.u32.u8 %0, t;\n}" : "=r"(q) : "f"(__fmaf_rn(c, 128.0f, 128.0f)));
  return q;
}

struct Key {
  uint32_t h1;  // full 32-bit home hash; the home index is h1 & (T - 1)
  uint32_t fp;
};

// The words a key is hashed from: the quantized position x~ (three int32 as
// bits), the level l', the packed quantized normal and, if given, an extra
// word.
struct KeyWords {
  uint32_t X, Y, Z, L, NQ, EX;
  bool has_ex;
};

// Where the optional per-vertex inputs of the key variants are: a distance
// for the level of detail and an extra key word of vertex j (read where they
// are used, so that a frame without them carries nothing extra).
struct KeyExtra {
  const float* dist = nullptr;
  const uint32_t* extra = nullptr;
  size_t j = 0;
};

__device__ __forceinline__ KeyExtra key_extra(const VertexPtrs& v, size_t j) {
  KeyExtra e;
  e.dist = v.dist;
  e.extra = v.extra;
  e.j = j;
  return e;
}

__device__ __forceinline__ KeyWords key_words(const KeyConst& kc, float px, float py, float pz,
                                              float nx, float ny, float nz, uint32_t id,
                                              uint32_t stream_id, const KeyExtra& ke = KeyExtra{}) {
  const int l0 = ke.dist ? level_at(kc, __ldg(ke.dist + ke.j)) : level_of_detail(kc, px, py, pz);
  float xj = px, yj = py, zj = pz;
  int l1 = l0;
  if (kc.jitter) {
    // jitter(n): a point of the tangent plane, (u, w) uniform in [-0.5, 0.5)
    const uint2 rnd = philox_first2_rk(id, stream_id, kc);
    // (products of 24-bit integers with 2^-24, and with s = +-1, are exact: the
    // fused forms round once, like the separate operations)
    const float u = __fmaf_rn(__uint2float_rn(rnd.x >> 8), 0x1p-24f, -0.5f);
    const float w = __fmaf_rn(__uint2float_rn(rnd.y >> 8), 0x1p-24f, -0.5f);
    // tangent frame after Duff et al. (JCGT 2017)
    const float s = copysignf(1.0f, nz);
    const float a = -__frcp_rn(__fadd_rn(s, nz));  // = -1 / (s + nz), correctly rounded
    const float q = __fmul_rn(__fmul_rn(nx, ny), a);
    const float tx = __fmaf_rn(s, __fmul_rn(__fmul_rn(nx, nx), a), 1.0f);
    const float ty = __fmul_rn(s, q);
    const float tz = -__fmul_rn(s, nx);
    const float bx = q;
    const float by = __fadd_rn(s, __fmul_rn(__fmul_rn(ny, ny), a));
    const float bz = -ny;
    const float E = pow2_int(l0);  // voxel edge at the pre-jitter level
    // (not fused: the product with E is exact only between underflow and overflow)
    xj = __fadd_rn(px, __fmul_rn(__fadd_rn(__fmul_rn(u, tx), __fmul_rn(w, bx)), E));
    yj = __fadd_rn(py, __fmul_rn(__fadd_rn(__fmul_rn(u, ty), __fmul_rn(w, by)), E));
    zj = __fadd_rn(pz, __fmul_rn(__fadd_rn(__fmul_rn(u, tz), __fmul_rn(w, bz)), E));
    l1 = ke.dist ? level_at(kc, __fadd_rn(__fsub_rn(__ldg(ke.dist + ke.j),
                                                    camera_distance(kc, px, py, pz)),
                                          camera_distance(kc, xj, yj, zj)))
                 : level_of_detail(kc, xj, yj, zj);
  }
  const float inv = pow2_int(-l1);
  KeyWords kw;
  kw.X = static_cast<uint32_t>(quantize_coord(xj, inv));
  kw.Y = static_cast<uint32_t>(quantize_coord(yj, inv));
  kw.Z = static_cast<uint32_t>(quantize_coord(zj, inv));
  kw.L = static_cast<uint32_t>(l1);
  kw.NQ = quantize_normal(nx) | (quantize_normal(ny) << 8) | (quantize_normal(nz) << 16);
  kw.has_ex = ke.extra != nullptr;
  kw.EX = kw.has_ex ? __ldg(ke.extra + ke.j) : 0u;
  return kw;
}

// hash (home) and hash2 (fingerprint, 0 remapped to 1) of the key words.
__device__ __forceinline__ Key key_hash(const KeyConst& kc, const KeyWords& kw) {
  uint32_t h = kc.hseed_home;
  h = mm_body(h, kw.X);
  h = mm_body(h, kw.Y);
  h = mm_body(h, kw.Z);
  h = mm_body(h, kw.L);
  uint32_t hbytes = 16u;
  if (kc.nih) {
    h = mm_body(h, kw.NQ);
    hbytes = 20u;
  }
  uint32_t f = kc.hseed_fp;
  f = mm_body(f, kw.X);
  f = mm_body(f, kw.Y);
  f = mm_body(f, kw.Z);
  f = mm_body(f, kw.L);
  f = mm_body(f, kw.NQ);
  uint32_t fbytes = 20u;
  if (kw.has_ex) {
    h = mm_body(h, kw.EX);
    f = mm_body(f, kw.EX);
    hbytes += 4u;
    fbytes += 4u;
  }
  h = mm_final(h, hbytes);
  f = mm_final(f, fbytes);
  return Key{h, f ? f : 1u};
}

__device__ __forceinline__ Key vertex_key(const KeyConst& kc, float px, float py, float pz,
                                          float nx, float ny, float nz, uint32_t id,
                                          uint32_t stream_id, const KeyExtra& ke = KeyExtra{}) {
  return key_hash(kc, key_words(kc, px, py, pz, nx, ny, nz, id, stream_id, ke));
}

// ---------------------------------------------------------------- memory helpers
// L2 eviction priority "evict last" for the lines the next frame touches
// again (slot index, accumulators): the vertex streams and outputs pass
// through L2 with evict-first loads and stores (.cs), these stay behind them.
__device__ __forceinline__ unsigned long long l2_evict_last() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// L2 eviction priority "evict first" for data a frame touches once and the
// next frame does not need in L2 (cell records, history cells, the stash):
// they should not push the slot index and the accumulators out.  Loads of such
// data written by other CTAs of the same launch bypass L1 (.cg).
__device__ __forceinline__ unsigned long long l2_evict_first() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ uint4 ld_once_u4(const void* p) {
  uint4 v;
  asm volatile("ld.global.cg.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p), "l"(l2_evict_first())
               : "memory");
  return v;
}

__device__ __forceinline__ uint2 ld_once_u2(const void* p) {
  uint2 v;
  asm volatile("ld.global.cg.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
               : "=r"(v.x), "=r"(v.y)
               : "l"(p), "l"(l2_evict_first())
               : "memory");
  return v;
}

__device__ __forceinline__ void st_once_u4(void* p, uint4 v) {
  asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "r"(v.x),
               "r"(v.y), "r"(v.z), "r"(v.w), "l"(l2_evict_first())
               : "memory");
}

__device__ __forceinline__ void st_once_u2(void* p, uint2 v) {
  asm volatile("st.global.L2::cache_hint.v2.u32 [%0], {%1, %2}, %3;" ::"l"(p), "r"(v.x), "r"(v.y),
               "l"(l2_evict_first())
               : "memory");
}

__device__ __forceinline__ void st_once_u32(void* p, uint32_t v) {
  asm volatile("st.global.L2::cache_hint.u32 [%0], %1, %2;" ::"l"(p), "r"(v), "l"(l2_evict_first())
               : "memory");
}

// The four slots of a sector (p 32-byte aligned), each a relaxed read of its own.
__device__ __forceinline__ void ld_relaxed_u64x4_keep(const unsigned long long* p, unsigned long long (&w)[4]) {
  asm volatile("ld.relaxed.gpu.global.L2::cache_hint.v4.u64 {%0, %1, %2, %3}, [%4], %5;"
               : "=l"(w[0]), "=l"(w[1]), "=l"(w[2]), "=l"(w[3])
               : "l"(p), "l"(l2_evict_last())
               : "memory");
}

__device__ __forceinline__ void red_add_v4_keep(float4* p, float a, float b, float c, float d) {
  asm volatile("red.relaxed.gpu.global.add.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p),
               "f"(a), "f"(b), "f"(c), "f"(d), "l"(l2_evict_last())
               : "memory");
}

__device__ __forceinline__ void st_zero16_keep(void* p) {
  asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %1, %1, %1}, %2;" ::"l"(p), "r"(0u),
               "l"(l2_evict_last())
               : "memory");
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ long long to_fixed(float v) {
  return __float2ll_rn(__fmul_rn(v, 16777216.0f));  // round(v * 2^24), exact product
}

__device__ __forceinline__ unsigned long long slot_word(uint32_t f, uint32_t id) {
  return (static_cast<unsigned long long>(id + 1u) << 32) | f;
}
__device__ __forceinline__ uint32_t slot_fp(unsigned long long w) {
  return static_cast<uint32_t>(w);
}
__device__ __forceinline__ uint32_t slot_id(unsigned long long w) {
  return static_cast<uint32_t>(w >> 32) - 1u;
}

// Read-only lookup of a key's cell id (query without a stored id), from
// probe step p0 on.
__device__ __forceinline__ uint32_t probe_find_from(const TableDev& t, uint32_t home, uint32_t f,
                                                    uint32_t p0) {
  for (uint32_t p = p0; p < t.max_probes; ++p) {
    const unsigned long long w = __ldcg(t.slots + ((home + p) & t.mask));
    if (w == 0ull) return kOverflowSlot;
    if (slot_fp(w) == f) return slot_id(w);
  }
  return kOverflowSlot;
}

__device__ __forceinline__ uint32_t probe_find(const TableDev& t, uint32_t home, uint32_t f) {
  return probe_find_from(t, home, f, 0u);
}

// History table probing: 32-bit compare-and-swap on the history fingerprint.
__device__ __forceinline__ uint32_t* hist_fp(const TableDev& t, uint32_t h) {
  return reinterpret_cast<uint32_t*>(t.hcells + static_cast<size_t>(h) * t.hstride + t.hfp_off);
}

__device__ __forceinline__ uint32_t hist_probe_rest(const TableDev& t, uint32_t home, uint32_t f,
                                                    uint32_t p0) {
  for (uint32_t p = p0; p < t.max_probes; ++p) {
    const uint32_t h = (home + p) & t.hmask;
    const uint32_t old = atomicCAS(hist_fp(t, h), 0u, f);
    if (old == 0u || old == f) return h;
  }
  return kOverflowSlot;
}

// Evicting history table (Sec. 3.4.3): fingerprint word = priority << 24 |
// low 24 bits of the fingerprint, 0 = empty.  Find the cell's entry in its
// window (refreshing its priority to this frame's), or claim the first empty
// cell, or -- with the window full -- replace the smallest word if its
// priority is older than this frame's.  `fresh`: the entry holds no history
// of this cell.  Compare-and-swaps on the whole word keep a concurrent
// claim, refresh or replacement from being lost; a few retries, then none.
static __device__ __noinline__ uint32_t hist_claim_evict(const TableDev& t, uint32_t home,
                                                         uint32_t f, bool* fresh) {
  const uint32_t f24 = f & 0xFFFFFFu;
  const uint32_t nw = (t.hist_rank << 24) | f24;
  for (int attempt = 0; attempt < 4; ++attempt) {
    uint32_t victim = kOverflowSlot, vword = 0xFFFFFFFFu;
    bool retry = false;
    for (uint32_t p = 0; p < t.max_probes; ++p) {
      const uint32_t h = (home + p) & t.hmask;
      uint32_t* fp = hist_fp(t, h);
      uint32_t w = __ldcg(fp);
      if (w == 0u) {
        w = atomicCAS(fp, 0u, nw);
        if (w == 0u) {
          *fresh = true;
          return h;
        }
      }
      if ((w & 0xFFFFFFu) == f24) {
        if (w != nw) {
          const uint32_t o = atomicCAS(fp, w, nw);
          if (o != w && (o & 0xFFFFFFu) != f24) {
            retry = true;  // replaced under us: scan again
            break;
          }
        }
        *fresh = false;
        return h;
      }
      if (w < vword) {
        vword = w;
        victim = h;
      }
    }
    if (retry) continue;
    if ((vword >> 24) >= t.hist_rank) return kOverflowSlot;  // all entries are this frame's
    if (atomicCAS(hist_fp(t, victim), vword, nw) == vword) {
      *fresh = true;
      return victim;
    }
  }
  return kOverflowSlot;
}

// Accumulate a group of `cnt` contributions (sums r, g, b) into cell `id`.
template <bool FIXED>
__device__ __forceinline__ void accumulate(const TableDev& t, uint32_t id, float r, float g, float b,
                                           long long fr, long long fg, long long fb, uint32_t cnt) {
  if (!FIXED) {
    red_add_v4_keep(t.acc + id, r, g, b, static_cast<float>(cnt));
    return;
  }
  unsigned long long* a = t.acc64 + 4 * static_cast<size_t>(id);
  atomicAdd(a + 0, static_cast<unsigned long long>(fr));
  atomicAdd(a + 1, static_cast<unsigned long long>(fg));
  atomicAdd(a + 2, static_cast<unsigned long long>(fb));
  atomicAdd(a + 3, static_cast<unsigned long long>(cnt));
}

// Cell average of this frame: sum / count, one FP32 round-to-nearest division
// (fixed mode: fl32(sum) * 2^-24 / fl32(count)).
struct CellMean {
  float r, g, b;
  uint32_t n;
};

// The raw accumulator of a cell as loaded from memory (both modes).
struct AccRaw {
  float4 lo;  // FP32 sums, or int64 sums r, g as bits (fixed)
  float4 hi;  // fixed mode: int64 sum b and count as bits
};

__device__ __forceinline__ float4* value_ptr(const TableDev& t, uint32_t id) {
  return t.fixed ? reinterpret_cast<float4*>(t.acc64 + 4 * static_cast<size_t>(id)) : t.acc + id;
}

__device__ __forceinline__ AccRaw load_acc(const TableDev& t, uint32_t id) {
  AccRaw a;
  const float4* p = value_ptr(t, id);
  a.lo = __ldcg(p);
  a.hi = t.fixed ? __ldcg(p + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
  return a;
}

__device__ __forceinline__ long long bits64(float x, float y) {
  return static_cast<long long>((static_cast<unsigned long long>(__float_as_uint(y)) << 32) |
                                __float_as_uint(x));
}

__device__ __forceinline__ CellMean mean_of(const TableDev& t, const AccRaw& a) {
  CellMean m;
  if (!t.fixed) {
    if (a.lo.w >= kExactCountLimit) atomicOr(&t.ctrl->error, kErrCountSaturated);
    m.r = __fdiv_rn(a.lo.x, a.lo.w);
    m.g = __fdiv_rn(a.lo.y, a.lo.w);
    m.b = __fdiv_rn(a.lo.z, a.lo.w);
    m.n = static_cast<uint32_t>(a.lo.w);
  } else {
    const long long sr = bits64(a.lo.x, a.lo.y), sg = bits64(a.lo.z, a.lo.w);
    const long long sb = bits64(a.hi.x, a.hi.y);
    const unsigned long long n = static_cast<unsigned long long>(bits64(a.hi.z, a.hi.w));
    const float fn = __ull2float_rn(n);
    m.r = __fdiv_rn(__fmul_rn(__ll2float_rn(sr), 0x1p-24f), fn);
    m.g = __fdiv_rn(__fmul_rn(__ll2float_rn(sg), 0x1p-24f), fn);
    m.b = __fdiv_rn(__fmul_rn(__ll2float_rn(sb), 0x1p-24f), fn);
    m.n = static_cast<uint32_t>(n);
  }
  return m;
}

// History value as loaded from memory.
struct HistRaw {
  float r, g, b;
  uint32_t n;
};

__device__ __forceinline__ HistRaw load_hist(const TableDev& t, uint32_t h) {
  HistRaw o;
  const unsigned char* c = t.hcells + static_cast<size_t>(h) * t.hstride;
  if (t.hist_mode == 1) {
    const uint4 v = ld_once_u4(c);
    o.r = __uint_as_float(v.x);
    o.g = __uint_as_float(v.y);
    o.b = __uint_as_float(v.z);
    o.n = v.w;
  } else {
    const uint2 v = ld_once_u2(c);
    const float2 rg = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
    o.r = rg.x;
    o.g = rg.y;
    o.b = __half2float(__ushort_as_half(static_cast<unsigned short>(v.y & 0xFFFFu)));
    o.n = v.y >> 16;
  }
  return o;
}

// Write history entry h (fingerprint word fw): the whole 32-byte cell in FP32,
// so that the sector needs no read-back when it leaves L2 (random 16-byte
// stores run at 23 G/s on a table in DRAM, 32-byte ones at 42 G/s).
__device__ __forceinline__ void store_hist(const TableDev& t, uint32_t h, uint32_t fw, float cr,
                                           float cg, float cb, uint32_t N) {
  unsigned char* c = t.hcells + static_cast<size_t>(h) * 32;
  asm volatile("st.global.L2::cache_hint.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %6, %6}, %7;" ::"l"(c),
               "r"(__float_as_uint(cr)), "r"(__float_as_uint(cg)), "r"(__float_as_uint(cb)), "r"(N),
               "r"(fw), "r"(0u), "l"(l2_evict_first())
               : "memory");
}

// Temporal filtering / integration of one cell (Sec. 3.4.1):
// c = alpha c_old + (1 - alpha) c_new, alpha < 0 meaning alpha = N_old / (N_old +
// N_new); no history -> c = c_new.  The history cell h (fingerprint word fw)
// is updated (h == kOverflowSlot: the history window was full; the cell keeps
// c_new and N = N_new) and the result replaces m.
__device__ __forceinline__ void blend_value(const TableDev& t, uint32_t h, uint32_t fw, CellMean& m,
                                            const HistRaw& old, float alpha) {
  if (h == kOverflowSlot) return;
  if (old.n != 0u) {
    const float a =
        alpha >= 0.0f ? alpha
                      : __fdiv_rn(__uint2float_rn(old.n),
                                  __fadd_rn(__uint2float_rn(old.n), __uint2float_rn(m.n)));
    const float a1 = __fsub_rn(1.0f, a);
    m.r = __fadd_rn(__fmul_rn(a, old.r), __fmul_rn(a1, m.r));
    m.g = __fadd_rn(__fmul_rn(a, old.g), __fmul_rn(a1, m.g));
    m.b = __fadd_rn(__fmul_rn(a, old.b), __fmul_rn(a1, m.b));
  }
  if (t.hist_mode == 1) {
    m.n += old.n;
    store_hist(t, h, fw, m.r, m.g, m.b, m.n);
  } else {
    m.n = min(old.n + m.n, 65535u);
    const __half2 rg = __floats2half2_rn(m.r, m.g);
    const __half hb = __float2half_rn(m.b);
    const uint32_t lo = *reinterpret_cast<const uint32_t*>(&rg);
    const uint32_t hi = static_cast<uint32_t>(__half_as_ushort(hb)) | (m.n << 16);
    st_once_u2(t.hcells + static_cast<size_t>(h) * t.hstride, make_uint2(lo, hi));
    // lookups see what the history stores
    const float2 back = __half22float2(rg);
    m.r = back.x;
    m.g = back.y;
    m.b = __half2float(hb);
  }
}

// The same for a cell of the frame table: the result replaces the cell's
// accumulator for the lookups.
__device__ __forceinline__ void blend_store(const TableDev& t, uint32_t id, uint32_t h, uint32_t fw,
                                            CellMean m, const HistRaw& old, float alpha) {
  blend_value(t, h, fw, m, old, alpha);
  __stcg(value_ptr(t, id), make_float4(m.r, m.g, m.b, __uint_as_float(m.n)));
}

// A history cell in one load: its value and its fingerprint word.
__device__ __forceinline__ HistRaw load_hist_fp(const TableDev& t, uint32_t h, uint32_t* fw) {
  HistRaw o;
  const unsigned char* c = t.hcells + static_cast<size_t>(h) * t.hstride;
  if (t.hist_mode == 1) {
    uint32_t x, y, z, w, u0, u1, u2, u3;
    asm volatile("ld.relaxed.gpu.global.L2::cache_hint.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
                 : "=r"(x), "=r"(y), "=r"(z), "=r"(w), "=r"(u0), "=r"(u1), "=r"(u2), "=r"(u3)
                 : "l"(c), "l"(l2_evict_first())
                 : "memory");
    (void)u1, (void)u2, (void)u3;  // padding
    o.r = __uint_as_float(x);
    o.g = __uint_as_float(y);
    o.b = __uint_as_float(z);
    o.n = w;
    *fw = u0;
  } else {
    const uint4 v = ld_once_u4(c);
    const float2 rg = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
    o.r = rg.x;
    o.g = rg.y;
    o.b = __half2float(__ushort_as_half(static_cast<unsigned short>(v.y & 0xFFFFu)));
    o.n = v.y >> 16;
    *fw = v.z;
  }
  return o;
}

// Value returned for cell `id`: the cell average, or the blended value.
__device__ __forceinline__ CellMean value_of(const TableDev& t, const AccRaw& a, bool blended) {
  if (!blended) return mean_of(t, a);
  CellMean m;
  m.r = a.lo.x;
  m.g = a.lo.y;
  m.b = a.lo.z;
  m.n = __float_as_uint(a.lo.w);
  return m;
}

__device__ __forceinline__ AccRaw load_value(const TableDev& t, uint32_t id, bool blended) {
  if (!blended) return load_acc(t, id);
  AccRaw a;
  a.lo = __ldcg(value_ptr(t, id));
  a.hi = make_float4(0.f, 0.f, 0.f, 0.f);
  return a;
}

// ---------------------------------------------------------------- vertices in, results out
struct Result {
  float r, g, b;
  uint32_t n;
  uint8_t status;
};

// The results of the four vertices from j on (those below `end`).
__device__ __forceinline__ void store_batch(const OutPtrs& o, size_t j, size_t end, bool vec,
                                            const Result (&res)[4]) {
  if (vec && j + 4 <= end) {
    __stcs(reinterpret_cast<float4*>(o.r + j), make_float4(res[0].r, res[1].r, res[2].r, res[3].r));
    __stcs(reinterpret_cast<float4*>(o.g + j), make_float4(res[0].g, res[1].g, res[2].g, res[3].g));
    __stcs(reinterpret_cast<float4*>(o.b + j), make_float4(res[0].b, res[1].b, res[2].b, res[3].b));
    if (o.count)
      __stcs(reinterpret_cast<uint4*>(o.count + j),
             make_uint4(res[0].n, res[1].n, res[2].n, res[3].n));
    if (o.status) {
      const uint32_t w = res[0].status | (res[1].status << 8) | (res[2].status << 16) |
                         (static_cast<uint32_t>(res[3].status) << 24);
      __stcs(reinterpret_cast<unsigned int*>(o.status + j), w);
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (j + q < end) {
      o.r[j + q] = res[q].r;
      o.g[j + q] = res[q].g;
      o.b[j + q] = res[q].b;
      if (o.count) o.count[j + q] = res[q].n;
      if (o.status) o.status[j + q] = res[q].status;
    }
  }
}

// This warp's place among the grid's warps.
__device__ __forceinline__ uint32_t grid_warp() {
  return blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
}
__device__ __forceinline__ uint32_t grid_warps() { return gridDim.x * (blockDim.x >> 5); }

// ---------------------------------------------------------------- grid barrier
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// The frame's counters to zero, by one thread; a grid barrier has to come
// before the first one that adds to them.
__device__ __forceinline__ void reset_counters(Ctrl* c) {
  c->frame_cells = 0ull;
  c->overflow_vertices = 0ull;
  c->vertices = 0ull;
  c->hist_overflow = 0ull;
  c->neigh_count = 0ull;
  c->tile_next = 0ull;
}

// Barrier over all CTAs of a cooperative launch, sense-reversing (Mellor-Crummey
// and Scott, 1991) on one word: the arrivals of one barrier add up to 2^31 (CTA 0
// adds 2^31 less one per other CTA), so the word's top bit is the sense, flips
// with the last arrival, and the low bits are back where they were: nobody
// resets anything.  Thread 0 of each CTA reads the sense, arrives with one
// reduction (it returns nothing, so nobody waits for it) and polls the same
// word.  The reduction releases and the poll acquires what the CTA's threads
// wrote.  An arrival counter whose last arrival resets it and then moves a
// generation on is three dependent round trips.  Frames of 7,680 and 65,536
// vertices (three barriers): 27.3 -> 24.4 us and 28.8 -> 24.5 us, about half of it
// this, half the counters' reset moving into the launch.
//
// The wait is bounded (about two seconds of wall time): on timeout the CTA
// raises kErrBarrierTimeout in the device error word and every CTA returns
// false, so the launch ends.
__device__ __forceinline__ bool grid_barrier(Ctrl* c, unsigned int nblocks,
                                             unsigned long long limit_ns = 2000000000ull) {
  constexpr unsigned int kSense = 0x80000000u;
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    unsigned int before;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(before) : "l"(&c->bar_count) : "memory");
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&c->bar_count),
                 "r"(blockIdx.x == 0 ? kSense - (nblocks - 1u) : 1u)
                 : "memory");
    unsigned long long t0 = 0ull;
    for (uint32_t i = 1; !((ld_acquire_u32(&c->bar_count) ^ before) & kSense); ++i) {
      if (i % 32u) continue;  // the error word and the clock now and then only
      const unsigned long long now = globaltimer_ns();
      if (t0 == 0ull) t0 = now;
      if (ld_acquire_u32(&c->error) & kErrBarrierTimeout) {
        ok = 0;
        break;
      }
      if (now - t0 > limit_ns) {
        atomicOr(&c->error, kErrBarrierTimeout);
        ok = 0;
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

}  // namespace pps
