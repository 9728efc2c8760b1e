// Decode attention read directly from the AnchorKV compressed cache (Eq. 3 folded into
// Eq. 4: no key or value row is ever rebuilt in memory).  Two launches per call (three with a dense suffix, whose
// chunks take a launch of their own between them).  Each launch after the first is a programmatic dependent of the one
// before it: it may start once that one's CTAs have, and waits where it needs its results.  So the decode is set up and
// its first tiles are on their way beside the scores, and the suffix's chunks run beside them (six ragged requests, 8B
// shape: 87.5 -> 85.6 us; four with RoPE and a suffix: 179 -> 172).  The first launch is an ordinary one (as a dependent
// of the call before, its wait cost more than the gap: 18.4 -> 20.5 us a call at 8 units of 32768).
//
// 1. The anchor scores S_A[a][g] = q_g . k_a of every anchor of every unit, once per anchor (Eq. 2-3),
//    in log2 units with sm_scale folded in, into the workspace, with the largest score per query head of
//    each chunk of 64 anchors; also each unit's query header (the rotated query q' = H(s o q)/128 of
//    Appendix A.1 Eq. 12, its sums per head, and q' as tensor-core fragments for the key residuals) and
//    zeroed arrival counters behind it.  akv_scores_kernel: a short-lived CTA per chunk, tensor-core products.  (With
//    RoPE at decode akv_rope_logits_kernel takes its place.)
//
// 2. akv_decode_kernel.  Persistent: one CTA per SM.  The tile blocks of all units, in unit
//    order, are split into equal contiguous ranges, one per CTA (stream-K): a unit's tiles may
//    lie in several CTAs and a CTA's range may cross units (its segments).  A CTA has eight token warps
//    and eight product warps (four warps per SM sub-partition at 128 registers), coupled by mbarriers, which
//    work on neighbouring tiles at the same time:
//      copies         a lane of token warp 0 (small query groups and long ranges: of each token warp in
//                     turn) brings the tiles into a byte ring of shared memory: one bulk
//                     asynchronous copy of the tile block and one of the anchor-value rows of the value
//                     slots the tile covers (the tile table records the range); table entries are read
//                     one tile ahead;
//      key residuals  (product warps, one tile ahead of the values) q' . c of the tile's staged key records
//                     on tensor cores, the terms scale (q' . c) + min sum(q') written over the records' own
//                     codes;
//      tokens         (token warps) each lane 4 consecutive stored tokens, every head: logits
//                     gamma_i S_A[a(i)] + residual term, p = 2^(l - m), the normaliser, p
//                     rows of the value records, and the value weights w[a] = sum_i p_i
//                     gamma_i (Eq. 3): tokens are stored sorted by value anchor, so runs
//                     inside a lane are summed in registers and stored, and runs across
//                     lanes merged by a warp segmented scan, without shared atomics;
//      value side     (product warps) the value-residual sum (p scale) c over the records and the anchor-
//                     value product w^T V_A over the tile's slots, both on tensor cores
//                     (weights and p scale as bf16 high + low parts, built once per tile as operands in
//                     place; codes exact), accumulated in registers across the segment's tiles.
//    At the end of a segment a warp per query head applies the inverse rotation once (Appendix E.1), stores
//    the CTA's partial numerator and normaliser into its workspace slot for the unit, and counts it in
//    on the head's counter; the warp that completes the count sums the head's slots in a fixed
//    order and writes the output.  Tiles denser than the staged counts, and runs on value
//    slots beyond a tile's weight rows, take CUDA-core paths; where anchors are many, tiles have more
//    weight rows than staged anchor-value rows, and the rest are read from global memory.
//
// What bounds the decode (70B shape, 128K: 54 tiles per SM): shared-memory wavefronts (about 3100 per tile, the
// gathers of score rows by random slots a quarter of them) and issue slots (about 11000 warp instructions
// per tile), each about half used; the rest is the latency of the phases' dependent chains.  Two groups
// of four warps that took a tile through all phases (255 registers, two warps per sub-partition) spent
// 2.8 us per tile pair-wise; token and product warps side by side spend 2.7 us and leave each other's
// latencies covered where tiles are few (8B shape, 32K: 24.6 -> 18.4 us per call, the score launch's part included).
//
// The exponent reference m is the largest anchor score of each query row.  Anchors are
// tokens of the unit, so it is a lower bound of the largest logit (sums cannot overflow unless
// a logit exceeds m by more than 2^120, which is flagged); every CTA of a unit takes the same
// m, so partial sums combine by plain addition.  Every wait on an mbarrier is bounded; a wait
// that runs out marks the CTA failed and the outputs of its units NaN.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <type_traits>
#include <vector>

#include "akv_device.cuh"
#include "akv_internal.h"

namespace akv {

// The decode kernels with more weight rows than staged anchor-value rows, the table in global memory: in translation units
// of their own, so that they compile beside the others.
template <int GS>
const void* wide_decode_kernel(int codec, int rope);

namespace {

constexpr int NTW = 8;              // token warps
constexpr int NMW = 8;              // product warps
constexpr int NCW = NTW + NMW;      // four per SM sub-partition, so 128 registers each
constexpr int NT = NCW * 32;        // 512 threads
constexpr int T = kTile;            // tokens per tile block
constexpr int LCH = T / (NTW * 32); // consecutive stored tokens per lane
static_assert(LCH == 4, "a lane's tokens are half a byte of a bitmap word and 16 bytes of a stream");
constexpr int NSG = 6;              // tiles in flight at most (their descriptors)
constexpr int kEnds = 2 * NTW;       // a tile's runs that may go on in a neighbour warp: each warp's first and last
constexpr int kOvl = 32;            // a tile's entries per overflow list (value records, anchor-value runs)
constexpr int kOvlBytes = 16 + 2 * kOvl * 9 * 4;  // a tile's two lists: counts, then entries
constexpr int kRingSlack = 4096;    // shared memory after the ring: the masked rows of the last
                                    // 16-row block of staged anchor values are read from here
constexpr float kLog2e = 1.4426950408889634f;
constexpr uint32_t F_MAX = tile_fixed_bytes(T);  // streams, bitmaps, rank words of a full tile

constexpr int SCH = kSuffixChunk;  // dense suffix: tokens per chunk

struct ScoreParams {
  const uint8_t* arena;
  const __nv_bfloat16* q;
  uint8_t* uh;     // [units] query headers, uh_stride bytes apart
  int uh_stride, rotate;
  unsigned long long sign_lo, sign_hi;
  float* sa;      // [units][ka_stride][G] anchor scores (log2 units)
  float* cmax;    // [units][n_ch][G] largest score of each chunk of CHA anchors
  int n_kv_heads, n_q_heads, ka_stride, n_ch;
  float scale_log2;
  // dense suffix (null ksuf: none): rows [units][suf_cap][128], lengths per request, n_sch
  // chunks of SCH tokens per unit, each a partial slot of suf_floats(G) floats
  const __nv_bfloat16* ksuf;
  const __nv_bfloat16* vsuf;
  const int32_t* suf_len;
  float* suf_part;
  int suf_cap, n_sch;
  int units;
  long long arena_rows;  // 256-byte rows of the arena
  // RoPE at decode (the suffix launch): suffix token t of a unit sits at position S + t
  unsigned long long turn[64];  // theta_j / (2 pi) as a 64-bit binary fraction of a turn
};

// The RoPE logits launch (AKV_FLAG_ROPE): every stored token's logit per head.
struct RopeParams {
  const uint8_t* arena;
  const __nv_bfloat16* q;
  float* lg;      // [units][s_stride][G] logits (log2 units, sm_scale folded in), stored order
  float* cmax;    // [units][n_tch][G] largest logit of each chunk of 64 stored tokens
  const uint8_t* uh;  // query headers: only their arrival counters are used (zeroed here)
  int uh_stride;
  int n_kv_heads, n_q_heads, rotate, s_stride, n_tch;
  float scale_log2;
  unsigned long long sign_lo, sign_hi;
  unsigned long long turn[64];  // theta_j / (2 pi) as a 64-bit binary fraction of a turn
};

struct __align__(16) Meta {  // a staged tile: as it was copied, then its shape (product warp 0, before the key terms are announced)
  uint32_t ring_off, blk_off, staged, lo, nrows, j, bytes;  // nrows: anchor-value rows staged
  uint32_t nw;                      // WIDE: value slots with a weight row
  uint32_t sm_v, cd_k, cd_v, sm_k;  // byte offsets of scales and codes in the block
  int n, nKs, nVs;                  // tokens; key records with terms, value records on tensor cores
  uint32_t fast;                    // every record staged, every slot has a weight row: the token path without rare cases; bit 1: value records staged;
                                    // kNoShape: the wait for the tile ran out, the shape is another tile's
};
constexpr uint32_t kNoShape = 4u;
struct Seg {  // a CTA's tiles of one unit
  int u, jb, je, ib;  // unit, its tiles [jb, je), CTA-local index of tile jb
  long long t0;       // global index of the unit's tile 0
  int nt, first, nseg, pad;
};
// What the copying lane keeps (in shared memory: no register of the other threads waits for it).
struct Prod {
  Seg s;                      // segment of the next tile to copy
  const uint8_t *tiles, *av;  // its unit's tile blocks, anchor values,
  const uint32_t* table;      // tile table
  int end;                    // CTA-local index past the segment
  int ii;                     // CTA-local index of the next tile to copy: so many are issued
  int nrel;                   // tiles released
  uint32_t head, used;        // ring bytes: next free place, bytes in flight
};

constexpr int kTurnGroup = 2;   // copies in turn: query groups at most
constexpr int kTurnTiles = 12;  // and tiles per CTA at least

struct DecodeParams {
  const uint8_t* arena;
  __nv_bfloat16* out;
  float* out_f32;
  const float* sa;
  const float* cmax;
  float* part;
  const uint8_t* uh;  // query headers (score launch), each with its unit's arrival counters behind it
  int uh_stride;
  long long ttot;  // tiles of all units
  int grid, n_kv_heads, n_q_heads, rotate, ka_stride, n_ch;
  float scale_log2;
  unsigned long long sign_lo, sign_hi;
  int R;           // value records per tile handled on tensor cores (their p rows); sizes the staging cap
  int X;           // anchor-value rows per tile that are staged, and the weight table's rows (WIDE: XW)
  int cap;         // staged bytes of a tile block at most
  int ring_bytes, drop_last, smem_sa;  // smem_sa: score table in shared memory (1), half of it (2)
  int o_bar, o_meta, o_misc, o_sa, o_ovf, o_qp, o_rows, o_gsum, o_wb, o_vs, o_pv, o_ovl, o_prod, o_ring;
  const float* lg;         // RoPE at decode: logits [units][s_stride][G] in stored order (else null)
  int s_stride;
  const float* suf_part;   // dense suffix partials [units][n_sch][suf_floats] (null: no suffix)
  const int32_t* suf_len;  // suffix tokens per request
  int suf_cap, n_sch;
  int cta_unit[kMaxGrid];  // first unit of each CTA's range
  int cta_tile[kMaxGrid];  // its first tile inside that unit
  int XW;                  // WIDE: the weight table's rows, more than X (else X)
};

// ---- device helpers ---------------------------------------------------------------

// Reduction (no return value) into this CTA's shared memory.
__device__ __forceinline__ void red_local(float* p, float v) {
  asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(smem_u32(p)), "f"(v) : "memory");
}
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

// 16 bytes of read-only global data, not kept in L1 (streamed once)
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Two 2-bit codes, at bits 0-1 and 16-17 of x, as an fp16 pair of exact small integers: OR
// them into the mantissa of 1024.0 (0x6400, unit spacing), then subtract 1024.
__device__ __forceinline__ uint32_t codes2_to_h2(uint32_t x) {
  uint32_t t, r;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(t) : "r"(x), "r"(0x00030003u), "r"(0x64006400u));
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(t), "r"(0x64006400u));
  return r;
}
// Two 2-bit codes as the exact bf16 pair c: OR into the mantissa of 128.0 (0x4300, unit
// spacing), then t * 1 - 128.
__device__ __forceinline__ uint32_t codes2_to_b2(uint32_t x) {
  uint32_t t, r;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(t) : "r"(x), "r"(0x00030003u), "r"(0x43004300u));
  asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(t), "r"(0x3F803F80u), "r"(0xC300C300u));
  return r;
}
// The Lloyd-Max codec (AKV_FLAG_LLOYD): a code c stands for level L[c] of
// {-1.5078125, -0.453125, 0.453125, 1.5078125}.  Two codes (bits 0-1 and 16-17 of x) become a
// 16-bit pair by a byte permutation out of the four-entry table held in two registers: the
// selector nibbles 2c, 2c + 1 of both codes come from one integer multiply-add and one gather.
__device__ __forceinline__ uint32_t lm_selector(uint32_t x) {
  const uint32_t u = (x & 0x00030003u) * 0x22u + 0x00100010u;  // bytes 0 and 2: nibbles 2c, 2c + 1
  uint32_t sel;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(sel) : "r"(u), "r"(0u), "r"(0x00000020u));
  return sel;
}
__device__ __forceinline__ uint32_t lm_pair(uint32_t x, uint32_t tab_lo, uint32_t tab_hi) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(tab_lo), "r"(tab_hi), "r"(lm_selector(x)));
  return r;
}
// Code pair as the fp16 (key-residual A operand) or bf16 (value-residual B operand) pair of the
// codec's reconstruction values: the codes themselves, or their Lloyd-Max levels (exact in both).
template <int CODEC>
__device__ __forceinline__ uint32_t code_pair_h2(uint32_t x) {
  if constexpr (CODEC == 0) return codes2_to_h2(x);
  else return lm_pair(x, 0xB740BE08u, 0x3E083740u);
}
// Both pairs of a value word's records, codes at bits 0, 16 and 8, 24: with the Lloyd-Max codec the four selector bytes
// come from one multiply-add (6 instructions for the two pairs, not 9: 8 x 131072, G = 8, Lloyd-Max 203.6 -> 196.7 us, G = 4
// 162.4 -> 158.2; the product warps are the longer side there).
template <int CODEC>
__device__ __forceinline__ uint2 code_pairs_b2(uint32_t x) {
  if constexpr (CODEC == 0) {
    return make_uint2(codes2_to_b2(x), codes2_to_b2(x >> 8));
  } else {
    const uint32_t u = (x & 0x03030303u) * 0x22u + 0x10101010u;
    uint32_t s0, s1;
    uint2 r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(s0) : "r"(u), "r"(0u), "r"(0x00000020u));
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(s1) : "r"(u), "r"(0u), "r"(0x00000031u));
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r.x) : "r"(0xBEE8BFC1u), "r"(0x3FC13EE8u), "r"(s0));
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r.y) : "r"(0xBEE8BFC1u), "r"(0x3FC13EE8u), "r"(s1));
    return r;
  }
}
// One code's reconstruction value on CUDA cores (the rare paths).
__device__ __forceinline__ float code_level(uint32_t c, int lloyd) {
  if (!lloyd) return (float)c;
  return c == 0u ? -1.5078125f : (c == 1u ? -0.453125f : (c == 2u ? 0.453125f : 1.5078125f));
}
__device__ __forceinline__ uint32_t pack_h2(__half lo, __half hi) {
  return (uint32_t)__half_as_ushort(lo) | ((uint32_t)__half_as_ushort(hi) << 16);
}
__device__ __forceinline__ uint32_t pack_b2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}
// bf16 high part of x and the bf16 of what is left: x ~= hi + lo to about 2^-17 relative
__device__ __forceinline__ void split_b(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}
__device__ __forceinline__ float half_lo(uint32_t w) {
  return __half2float(__ushort_as_half((unsigned short)(w & 0xFFFFu)));
}
__device__ __forceinline__ float half_hi(uint32_t w) { return __half2float(__ushort_as_half((unsigned short)(w >> 16))); }

// 2^x with the hardware approximation (relative error near 2^-22; results below the
// smallest normal flush to 0, which only drops weights under 2^-126 of the reference).
__device__ __forceinline__ float exp2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Unnormalised 128-point Walsh-Hadamard transform of one row held by a warp, lane l holding
// elements 4 l .. 4 l + 3: two butterfly stages inside the lane, five across lanes.
__device__ __forceinline__ void warp_wht128(float (&x)[4], int lane) {
  const float a0 = x[0] + x[1], a1 = x[0] - x[1], a2 = x[2] + x[3], a3 = x[2] - x[3];
  x[0] = a0 + a2;
  x[1] = a1 + a3;
  x[2] = a0 - a2;
  x[3] = a1 - a3;
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {  // stage of distance 4 m: partner lane l ^ m
    const float sg = (lane & m) ? -1.f : 1.f;  // v - x (upper partner) or x + v, one exact fma each
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float v = __shfl_xor_sync(0xffffffffu, x[j], m);
      x[j] = fmaf(sg, x[j], v);
    }
  }
}
// The rotation's signs s_j of dims 4 l .. 4 l + 3 applied to x.
__device__ __forceinline__ void apply_signs(float (&x)[4], int lane, unsigned long long lo, unsigned long long hi) {
  const unsigned long long sb = lane < 16 ? lo : hi;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if ((sb >> ((4 * lane + j) & 63)) & 1ull) x[j] = -x[j];
}

__device__ __forceinline__ const akv_unit_desc* unit_desc(const uint8_t* A, int u) {
  return reinterpret_cast<const akv_unit_desc*>(A + 256) + u;
}
// first element of unit u's query (and output) rows
__device__ __forceinline__ size_t qrow_base(int u, int n_kv_heads, int n_q_heads) {
  const int b = u / n_kv_heads, h = u % n_kv_heads;
  const int G = n_q_heads / n_kv_heads;
  return ((size_t)b * n_q_heads + (size_t)h * G) * 128;
}

// Geometry of one staged tile block: the first `staged` bytes are in shared memory, the
// rest is read from global memory (a tile with more records than the stage holds).
struct TileView {
  const uint8_t* st;   // stage
  uint32_t blk_off;    // the block in global memory, from the unit's tiles
  uint32_t staged;
  int u;
  int n, nw, n64, nk, nv;
  uint32_t sm_k, sm_v, cd_k, cd_v;  // byte offsets of scales and codes in the block
  // (the descriptor is read again where a byte past the stage is wanted: rare, and no register waits for it)
  __device__ __forceinline__ const uint8_t* gb(const uint8_t* A) const { return A + unit_desc(A, u)->off_tiles + blk_off; }
  __device__ __forceinline__ const uint8_t* at(const uint8_t* A, uint32_t off) const { return off < staged ? st + off : gb(A) + off; }
  __device__ __forceinline__ uint64_t bm(int side, int w) const {
    return reinterpret_cast<const uint64_t*>(st + 8 * n64)[side * nw + w];
  }
  __device__ __forceinline__ int rk(int side, int w) const {
    return reinterpret_cast<const uint16_t*>(st + 8 * n64 + 16 * nw + side * round16(2u * nw))[w];
  }
};
// The shape of a tile from its bitmaps and rank words.
__device__ __forceinline__ TileView tile_view(const uint8_t* st, const Meta& mt, int u, int S) {
  TileView v;
  v.st = st;
  v.blk_off = mt.blk_off;
  v.staged = mt.staged;
  v.u = u;
  v.n = min(T, S - (int)mt.j * T);
  v.nw = (int)tile_words(v.n);
  v.n64 = 64 * v.nw;
  v.nk = v.rk(0, v.nw - 1) + __popcll(v.bm(0, v.nw - 1));
  v.nv = v.rk(1, v.nw - 1) + __popcll(v.bm(1, v.nw - 1));
  const uint32_t F = tile_fixed_bytes(v.n);
  v.sm_k = F;
  v.sm_v = F + round16(4u * (uint32_t)v.nk);
  v.cd_k = v.sm_v + round16(4u * (uint32_t)v.nv);
  v.cd_v = v.cd_k + 32u * (uint32_t)v.nk;
  return v;
}
// The same as product warp 0 left it in the tile's descriptor.
__device__ __forceinline__ TileView tile_view(const uint8_t* st, const Meta& mt, int u) {
  TileView v;
  v.st = st;
  v.blk_off = mt.blk_off;
  v.staged = mt.staged;
  v.u = u;
  v.n = mt.n;
  v.nw = (int)tile_words(v.n);
  v.n64 = 64 * v.nw;
  v.nk = v.nv = 0;  // (not kept)
  v.sm_k = mt.sm_k;
  v.sm_v = mt.sm_v;
  v.cd_k = mt.cd_k;
  v.cd_v = mt.cd_v;
  return v;
}

// Bytes of a tile block at offset `off`: shared memory for its first `staged` bytes, else the
// block in global memory.
__device__ __forceinline__ const uint8_t* blk_at(const uint8_t* st, const uint8_t* gb, uint32_t staged, uint32_t off) {
  return off < staged ? st + off : gb + off;
}
// Records beyond the staged ones (a locally dense tile whose codes did not fit the staging
// cap) take these rare paths on CUDA cores, kept out of line so that the token loop stays
// small.  Their arguments are plain pointers and offsets: a struct passed by value would be
// built in local memory at every call.
// Key residual term scale (q'_g . c) + min sum(q'_g) of the key record whose scale-min word
// is at `smn_off` and whose codes start at `cd_off`.
__device__ __noinline__ float key_record_term(const uint8_t* st, const uint8_t* gb, uint32_t staged, uint32_t smn_off,
                                              uint32_t cd_off, const float* qpg, float sqg, int lloyd) {
  const uint32_t smn = *reinterpret_cast<const uint32_t*>(blk_at(st, gb, staged, smn_off));
  float dot = 0.f;
  for (int bb = 0; bb < 32; ++bb) {
    const uint32_t byte = *blk_at(st, gb, staged, cd_off + (uint32_t)bb);
#pragma unroll
    for (int c = 0; c < 4; ++c) dot += qpg[4 * bb + c] * code_level((byte >> (2 * c)) & 3u, lloyd);
  }
  return half_hi(smn) * sqg + half_lo(smn) * dot;
}
// accg += p (min + scale c) of value record r, in the rotated domain (value codes are
// dimension-major groups of 16 records; the group of r starts at `grp_off`).
__device__ __noinline__ void value_record_add(const uint8_t* st, const uint8_t* gb, uint32_t staged, uint32_t smn_off,
                                              uint32_t grp_off, int r, float p, float* accg, int lloyd) {
  const uint32_t smn = *reinterpret_cast<const uint32_t*>(blk_at(st, gb, staged, smn_off));
  const float ps = p * half_lo(smn), pm = p * half_hi(smn);
  for (int d = 0; d < 128; ++d) {
    const uint32_t w = *reinterpret_cast<const uint32_t*>(blk_at(st, gb, staged, grp_off + 4u * value_code_word(d)));
    atomicAdd(&accg[d], fmaf(ps, code_level((w >> value_code_bit(r % 16)) & 3u, lloyd), pm));
  }
}
// acc[g] x the anchor's value row (global memory, swizzled by the slot), added into ov[g][:]:
// a run whose value slot lies beyond the tile's weight rows (rare).
template <int GS>
__device__ __noinline__ void anchor_value_add(const uint8_t* AV, int anchor, const float* acc, float* ov) {
  const uint8_t* row = AV + (size_t)anchor * 256;
  for (int d = 0; d < 128; ++d) {  // dim d: element d % 8 of chunk d / 8, stored at (d / 8) ^ (row % 8)
    const float x = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(row + 16 * ((d >> 3) ^ (anchor & 7)) + 2 * (d & 7)));
#pragma unroll
    for (int g = 0; g < GS; ++g) atomicAdd(&ov[g * 128 + d], acc[g] * x);
  }
}

// Anchor-score table of a unit, ka rows: [a][GS] floats, except at GS = 8, where heads 0-3 and
// 4-7 are two arrays [2][ka][4]: a gathered 16-byte half-row then lies in any of the eight
// 16-byte bank groups of shared memory (a 32-byte row would start in only four of them).
template <int GS>
__device__ __forceinline__ size_t sa_at(int a, int g, int ka) {
  if constexpr (GS == 8) return (size_t)(g >> 2) * ka * 4 + (size_t)a * 4 + (g & 3);
  else return (size_t)a * GS + g;
}
template <int GS>
__device__ __forceinline__ void load_sa_row(const float* t, int a, int ka, float (&out)[GS]) {
  if constexpr (GS == 8) {
    const float4 v = *reinterpret_cast<const float4*>(t + a * 4), w = *reinterpret_cast<const float4*>(t + (ka + a) * 4);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    out[4] = w.x; out[5] = w.y; out[6] = w.z; out[7] = w.w;
  } else {
    if constexpr (GS == 4) {
      const float4 v = *reinterpret_cast<const float4*>(t + a * 4);
      out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    } else if constexpr (GS == 2) {
      const float2 v = *reinterpret_cast<const float2*>(t + a * 2);
      out[0] = v.x; out[1] = v.y;
    } else {
      out[0] = t[a];
    }
  }
}

// N consecutive 32-bit words (4 N-byte aligned) from shared memory.
template <int N>
__device__ __forceinline__ void load_words(const uint8_t* p, uint32_t (&w)[N]) {
  if constexpr (N == 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
  } else {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    w[0] = v.x; w[1] = v.y;
  }
}

// A row of GS floats (16-byte aligned for GS >= 4, else 8 or 4) as GS probabilities (pairs).
template <int GS, int NP>
__device__ __forceinline__ void store_row(float* p, const float2 (&v)[NP]) {
  if constexpr (GS == 8) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    *reinterpret_cast<float4*>(p + 4) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
  } else if constexpr (GS == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  } else if constexpr (GS == 2) {
    *reinterpret_cast<float2*>(p) = v[0];
  } else {
    p[0] = v[0].x;
  }
}
// A row of GS consecutive floats (16-byte aligned for GS >= 4, else 8 or 4) into registers.
template <int GS>
__device__ __forceinline__ void load_row(const float* p, float (&out)[GS]) {
  if constexpr (GS == 8) {
    const float4 v = *reinterpret_cast<const float4*>(p), w = *reinterpret_cast<const float4*>(p + 4);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    out[4] = w.x; out[5] = w.y; out[6] = w.z; out[7] = w.w;
  } else if constexpr (GS == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
  } else if constexpr (GS == 2) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    out[0] = v.x; out[1] = v.y;
  } else {
    out[0] = p[0];
  }
}

// =============================== anchor scores =====================================
// CTA (unit u, chunk ch): anchors ch*64 .. ch*64 + 63, warp w rows 16 w .. 16 w + 15, straight
// from global memory into the mma A fragments (rows are stored swizzled in 16-byte chunks by
// slot % 8; the k order is permuted the same way in A and B so that a thread's dims are
// contiguous: thread (r8, c4) of k-pair step j holds dims 32 j + 8 c4 .. + 7 of rows r8, r8 + 8).
// Dense suffix chunk sc of unit u (Appendix E.1 and E.2): suffix tokens j0 .. j0 + 63 of its
// request, scored against the unit's GS query rows on tensor cores (rows plain [token][128] bf16;
// the same permuted k order as the anchor chunks), p = 2^(s - m_c) under the chunk's own maximum
// m_c, then o[g][d] = sum_t p_t[g] V[t][d] (thread d) and l[g] = sum_t p_t[g] into the chunk's
// partial slot.  Chunks at or past the request's length write nothing (the combine reads the
// chunks below it only).  ROPE: the keys are pre-RoPE and turn to positions S + t first.
template <int GS, bool ROPE>
__device__ __forceinline__ void suffix_chunk(const ScoreParams& P, int u, int sc, __nv_bfloat16 (*vsm)[128]) {
  __shared__ float ps[SCH][8];
  __shared__ float wm[4][8];
  __shared__ float mc[8];
  const int len = max(0, min(P.suf_len[u / P.n_kv_heads], P.suf_cap));
  const int j0 = sc * SCH;
  if (j0 >= len) return;
  const int nv = min(SCH, len - j0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r8 = lane >> 2, c4 = lane & 3;
  const uint8_t* Kr = reinterpret_cast<const uint8_t*>(P.ksuf) + (size_t)u * P.suf_cap * 256;
  const uint8_t* Vr = reinterpret_cast<const uint8_t*>(P.vsuf) + (size_t)u * P.suf_cap * 256;
  // the chunk's value rows, all in flight at once (row t / 16 + 8 i, 16-byte column t % 16),
  // while the keys are scored
  uint4 vrow[SCH / 8];
#pragma unroll
  for (int i = 0; i < SCH / 8; ++i) {
    const int row = tid / 16 + 8 * i;
    vrow[i] = row < nv ? ldg_stream(Vr + (size_t)(j0 + row) * 256 + 16 * (tid % 16)) : make_uint4(0u, 0u, 0u, 0u);
  }
  const size_t qb = qrow_base(u, P.n_kv_heads, P.n_q_heads);
  uint2 bq[8];
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
    bq[ks] = r8 < GS ? *reinterpret_cast<const uint2*>(P.q + qb + (size_t)r8 * 128 + 32 * (ks >> 1) + 8 * c4 + 4 * (ks & 1))
                     : make_uint2(0u, 0u);
  const int t0 = j0 + 16 * warp;
  const int ra = min(t0 + r8, len - 1), rb = min(t0 + r8 + 8, len - 1);
  uint4 lo[4], hi[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int cc = 4 * j + c4;
    lo[j] = ldg_stream(Kr + (size_t)ra * 256 + 16 * cc);
    hi[j] = ldg_stream(Kr + (size_t)rb * 256 + 16 * cc);
  }
  float dd[4] = {0.f, 0.f, 0.f, 0.f};
  if constexpr (ROPE) {
    // RoPE at positions S + t: a thread's chunks c4 + 4 j (j < 2) and c4 + 4 j + 8 hold the two
    // members of pairs (d, d + 64), so each row turns in registers; the turned keys enter the
    // products as bf16 high and low parts
    const uint32_t S_u = (uint32_t)unit_desc(P.arena, u)->len;
    uint4 kr[2][4];  // [row ra / rb][chunk j]: the loaded rows
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      kr[0][j] = lo[j];
      kr[1][j] = hi[j];
    }
    uint32_t khi[2][4][4], klo[2][4][4];  // [row][chunk][bf16 pair]
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const uint32_t p = S_u + (uint32_t)(rr ? rb : ra);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const uint32_t* wa = reinterpret_cast<const uint32_t*>(&kr[rr][j]);
        const uint32_t* wb = reinterpret_cast<const uint32_t*>(&kr[rr][j + 2]);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          float ya[2], yb[2];
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const int dim = 8 * (4 * j + c4) + 2 * w + hh;  // < 64; its partner is dim + 64
            const float xa = __bfloat162float(__ushort_as_bfloat16((unsigned short)(hh ? wa[w] >> 16 : wa[w] & 0xFFFFu)));
            const float xb = __bfloat162float(__ushort_as_bfloat16((unsigned short)(hh ? wb[w] >> 16 : wb[w] & 0xFFFFu)));
            float sn, cs;
            __sincosf((float)(uint32_t)(((unsigned long long)p * P.turn[dim]) >> 40) * (6.2831853071795865f / 16777216.0f), &sn, &cs);
            ya[hh] = fmaf(xa, cs, -xb * sn);
            yb[hh] = fmaf(xb, cs, xa * sn);
          }
          __nv_bfloat162 ha = __floats2bfloat162_rn(ya[0], ya[1]), hb = __floats2bfloat162_rn(yb[0], yb[1]);
          const float2 fa = __bfloat1622float2(ha), fb = __bfloat1622float2(hb);
          __nv_bfloat162 la = __floats2bfloat162_rn(ya[0] - fa.x, ya[1] - fa.y), lb = __floats2bfloat162_rn(yb[0] - fb.x, yb[1] - fb.y);
          khi[rr][j][w] = *reinterpret_cast<const uint32_t*>(&ha);
          khi[rr][j + 2][w] = *reinterpret_cast<const uint32_t*>(&hb);
          klo[rr][j][w] = *reinterpret_cast<const uint32_t*>(&la);
          klo[rr][j + 2][w] = *reinterpret_cast<const uint32_t*>(&lb);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      mma_bf16(dd, khi[0][j][0], khi[1][j][0], khi[0][j][1], khi[1][j][1], bq[2 * j].x, bq[2 * j].y);
      mma_bf16(dd, khi[0][j][2], khi[1][j][2], khi[0][j][3], khi[1][j][3], bq[2 * j + 1].x, bq[2 * j + 1].y);
      mma_bf16(dd, klo[0][j][0], klo[1][j][0], klo[0][j][1], klo[1][j][1], bq[2 * j].x, bq[2 * j].y);
      mma_bf16(dd, klo[0][j][2], klo[1][j][2], klo[0][j][3], klo[1][j][3], bq[2 * j + 1].x, bq[2 * j + 1].y);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      mma_bf16(dd, lo[j].x, hi[j].x, lo[j].y, hi[j].y, bq[2 * j].x, bq[2 * j].y);
      mma_bf16(dd, lo[j].z, hi[j].z, lo[j].w, hi[j].w, bq[2 * j + 1].x, bq[2 * j + 1].y);
    }
  }
  const int g0 = 2 * c4;
  float sv[2][2];
  float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool ok = t0 + r8 + 8 * h < len;
    sv[h][0] = ok && g0 < GS ? dd[2 * h] * P.scale_log2 : -INFINITY;
    sv[h][1] = ok && g0 + 1 < GS ? dd[2 * h + 1] * P.scale_log2 : -INFINITY;
    mx0 = fmaxf(mx0, sv[h][0]);
    mx1 = fmaxf(mx1, sv[h][1]);
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
  }
  if (lane < 4) {
    wm[warp][2 * lane] = mx0;
    wm[warp][2 * lane + 1] = mx1;
  }
#pragma unroll
  for (int i = 0; i < SCH / 8; ++i) *reinterpret_cast<uint4*>(&vsm[tid / 16 + 8 * i][8 * (tid % 16)]) = vrow[i];
  __syncthreads();
  if (tid < 8) mc[tid] = fmaxf(fmaxf(wm[0][tid], wm[1][tid]), fmaxf(wm[2][tid], wm[3][tid]));
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int row = 16 * warp + r8 + 8 * h;
    if (g0 < GS) ps[row][g0] = sv[h][0] > -INFINITY ? exp2_approx(sv[h][0] - mc[g0]) : 0.f;
    if (g0 + 1 < GS) ps[row][g0 + 1] = sv[h][1] > -INFINITY ? exp2_approx(sv[h][1] - mc[g0 + 1]) : 0.f;
  }
  __syncthreads();
  float o[GS];
#pragma unroll
  for (int g = 0; g < GS; ++g) o[g] = 0.f;
  for (int j = 0; j < nv; ++j) {  // thread tid: dimension tid of every row
    const float v = __bfloat162float(vsm[j][tid]);
#pragma unroll
    for (int g = 0; g < GS; ++g) o[g] = fmaf(ps[j][g], v, o[g]);
  }
  float* dst = P.suf_part + ((size_t)u * P.n_sch + sc) * suf_floats(GS);
#pragma unroll
  for (int g = 0; g < GS; ++g) dst[g * 128 + tid] = o[g];
  if (tid < GS) {
    float l = 0.f;
    for (int j = 0; j < nv; ++j) l += ps[j][tid];
    dst[suf_l(GS) + tid] = l;
    dst[suf_m(GS) + tid] = mc[tid];
  }
}

// The dense suffix's chunks (grid: units x n_sch), a launch of their own after the score or RoPE
// logits launch (ROPE: the keys are pre-RoPE).
template <int GS, bool ROPE>
__global__ void __launch_bounds__(128) akv_suffix_kernel(const ScoreParams P) {
  extern __shared__ __align__(16) uint8_t score_dyn[];  // the chunk's value rows
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (a decode that waits for it where it needs it)
  suffix_chunk<GS, ROPE>(P, blockIdx.x / P.n_sch, blockIdx.x % P.n_sch,
                         reinterpret_cast<__nv_bfloat16 (*)[128]>(score_dyn));
  // nothing above reads what the launch before this one (the scores) writes, so the two run beside each other; the
  // decode waits for this launch alone, which therefore ends after that one
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The arrival counters of unit u's query heads, behind its query header.
__device__ __forceinline__ unsigned* unit_counters(const uint8_t* uh, int uh_stride, int u, int GS) {
  return reinterpret_cast<unsigned*>(const_cast<uint8_t*>(uh) + (size_t)u * uh_stride + hdr_bytes(GS));
}

// The unit's query header, by one warp: the rotated query q' = H(s o q) / 128 scaled to log2 units
// (Appendix A.1, Eq. 12; warp-local Walsh-Hadamard transform), its sums, and the key-residual mma
// B fragments: column n = lane / 4 is head n as the fp16 high part (set 0) and low part (set 1) for
// GS = 8, else head n % 4 high (n < 4) or low (n >= 4); k pairs (2t, 2t+1) <-> dims
// (16 ks + 2t, 16 ks + 2t + 8), (2t+8, 2t+9) <-> (16 ks + 2t + 1, 16 ks + 2t + 9).  qs: 8 x 128
// floats of shared memory for the rotated rows.
template <int GS>
__device__ __noinline__ void unit_query_header_warp(const ScoreParams& P, int u, float* qs) {
  const int lane = threadIdx.x & 31;
  constexpr int NBF = GS == 8 ? 2 : 1;
  uint8_t* H = P.uh + (size_t)u * P.uh_stride;
  float* hq = reinterpret_cast<float*>(H);
  float* hs = hq + GS * 128;
  uint2* hf = reinterpret_cast<uint2*>(hs + 8);
  const size_t qb = qrow_base(u, P.n_kv_heads, P.n_q_heads);
  const float f = P.rotate ? P.scale_log2 * (1.0f / 128.0f) : P.scale_log2;
  uint2 raw[GS];  // every row's loads in flight at once
#pragma unroll
  for (int g = 0; g < GS; ++g) raw[g] = *reinterpret_cast<const uint2*>(P.q + qb + (size_t)g * 128 + 4 * lane);
#pragma unroll
  for (int g = 0; g < GS; ++g) {
    float x[4] = {__bfloat162float(__ushort_as_bfloat16((unsigned short)(raw[g].x & 0xFFFFu))),
                  __bfloat162float(__ushort_as_bfloat16((unsigned short)(raw[g].x >> 16))),
                  __bfloat162float(__ushort_as_bfloat16((unsigned short)(raw[g].y & 0xFFFFu))),
                  __bfloat162float(__ushort_as_bfloat16((unsigned short)(raw[g].y >> 16)))};
    if (P.rotate) {
      apply_signs(x, lane, P.sign_lo, P.sign_hi);
      warp_wht128(x, lane);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] *= f;
    const float4 v = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4*>(qs + g * 128 + 4 * lane) = v;
    *reinterpret_cast<float4*>(hq + g * 128 + 4 * lane) = v;
    const float sg = warp_sum((x[0] + x[1]) + (x[2] + x[3]));
    if (lane == 0) hs[g] = sg;
  }
  if (lane >= GS && lane < 8) hs[lane] = 0.f;
  __syncwarp();  // the rotated rows are in shared memory for every lane
  const int gcol = lane >> 2, cc = lane & 3;
#pragma unroll
  for (int idx = 0; idx < NBF * 8; ++idx) {
    const int hl = idx >> 3, ks = idx & 7;
    uint2 fk = make_uint2(0u, 0u);
    const int head = GS == 8 ? gcol : (gcol & 3);
    const bool low = GS == 8 ? hl == 1 : gcol >= 4;
    if (head < GS) {
      const float* x = qs + head * 128 + 16 * ks + 2 * cc;
      auto part = [&](float v) {
        const __half hi = __float2half_rn(v);
        return low ? __float2half_rn(v - __half2float(hi)) : hi;
      };
      fk.x = pack_h2(part(x[0]), part(x[8]));
      fk.y = pack_h2(part(x[1]), part(x[9]));
    }
    hf[(hl * 8 + ks) * 32 + lane] = fk;
  }
  __syncwarp();  // the next unit's rows may overwrite qs
}

// Anchor scores (Eq. 2-3: S_A = q . k_a once per anchor): CTA b < units writes unit b's query header and zeroes its
// counters; the others take 64 anchors of a unit each (warp w rows 16 w .. 16 w + 15), straight from global memory into
// bf16 mma A fragments (rows are stored swizzled in 16-byte chunks by slot % 8; the k order is permuted the same way
// in A and B, so that a thread's dims are contiguous).  Bound by the anchor rows' bytes and a CTA's load latency; many
// short CTAs keep enough loads in flight, hold no tensor memory and little else, so the decode, the programmatic
// dependent, sets itself up beside them.  A persistent CTA per SM with tensor copies, tcgen05 products and
// tensor-memory accumulators took 7 us whatever the size at 8 x 656 anchors, where this takes 3, and was slower at
// every size (whole calls, us, that and this: 8 units of 32768 tokens 20.8, 18.4; six ragged requests 85.0, 80.0;
// 64 x 2622 anchors 170.9, 163.5; 64 x 6554 198.7, 189.6; 128 x 5243 390, 373).
template <int GS>
__global__ void __launch_bounds__(128) akv_scores_kernel(const ScoreParams P) {
  __shared__ __align__(16) float hdr_q[8 * 128];
  __shared__ float wm[4][8];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r8 = lane >> 2, c4 = lane & 3;
  if ((int)blockIdx.x < P.units) {
    if (tid < 8) unit_counters(P.uh, P.uh_stride, blockIdx.x, GS)[tid] = 0u;
    if (warp == 0) unit_query_header_warp<GS>(P, blockIdx.x, hdr_q);
    return;
  }
  const int u = ((int)blockIdx.x - P.units) / P.n_ch, ch = ((int)blockIdx.x - P.units) % P.n_ch;
  const akv_unit_desc* d = unit_desc(P.arena, u);
  const int k = d->n_anchors;
  if (ch * CHA >= k) return;
  const uint64_t off = d->off_anchor_k;
  const bool inside = !(off & 255u) && (long long)(off >> 8) + k <= P.arena_rows;
  const uint8_t* AK = P.arena + off;
  const size_t qb = qrow_base(u, P.n_kv_heads, P.n_q_heads);
  uint2 bq[8];
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
    bq[ks] = r8 < GS ? *reinterpret_cast<const uint2*>(P.q + qb + (size_t)r8 * 128 + 32 * (ks >> 1) + 8 * c4 + 4 * (ks & 1))
                     : make_uint2(0u, 0u);
  const int g0 = 2 * c4, a0 = ch * CHA + 16 * warp + r8;
  const int ra = inside ? min(a0, k - 1) : 0, rb = inside ? min(a0 + 8, k - 1) : 0;
  uint4 lo[4] = {}, hi[4] = {};
  if (inside) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      lo[j] = ldg_stream(AK + (size_t)ra * 256 + 16 * ((4 * j + c4) ^ (ra & 7)));
      hi[j] = ldg_stream(AK + (size_t)rb * 256 + 16 * ((4 * j + c4) ^ (rb & 7)));
    }
  }
  float dd[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    mma_bf16(dd, lo[j].x, hi[j].x, lo[j].y, hi[j].y, bq[2 * j].x, bq[2 * j].y);
    mma_bf16(dd, lo[j].z, hi[j].z, lo[j].w, hi[j].w, bq[2 * j + 1].x, bq[2 * j + 1].y);
  }
  float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int a = a0 + 8 * h;
    if (a >= k || g0 >= GS) continue;
    const float v0 = dd[2 * h] * P.scale_log2, v1 = dd[2 * h + 1] * P.scale_log2;
    float* t = P.sa + (size_t)u * P.ka_stride * GS + sa_at<GS>(a, g0, P.ka_stride);
    if constexpr (GS == 1) t[0] = v0;
    else *reinterpret_cast<float2*>(t) = make_float2(v0, v1);
    mx0 = fmaxf(mx0, v0);
    mx1 = fmaxf(mx1, v1);
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
  }
  if (lane < 4) {
    wm[warp][2 * lane] = mx0;
    wm[warp][2 * lane + 1] = mx1;
  }
  __syncthreads();
  if (tid < GS)  // (rows outside the arena: the unit's outputs become NaN)
    P.cmax[((size_t)u * P.n_ch + ch) * GS + tid] =
        inside ? fmaxf(fmaxf(wm[0][tid], wm[1][tid]), fmaxf(wm[2][tid], wm[3][tid])) : INFINITY;
}

// ============================ the unit's output ====================================
// One query head of unit u, by a warp: the sum of its partial slots in a fixed order, the dense suffix's chunks
// (m: the unit's reference), the normalisation, bf16 RNE output.  A CTA that failed left a NaN normaliser.
template <int GS>
__device__ __noinline__ void combine_head(const DecodeParams& P, int u, int first, int nseg, int h, float m) {
  const int lane = threadIdx.x & 31;
  constexpr int PF = part_floats(GS);
  auto slot = [&](int s) { return P.part + (size_t)(first + s + u) * PF; };  // CTA first + s
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  float L = 0.f;
  for (int s0 = 0; s0 < nseg; s0 += 16) {  // sixteen slots' loads in flight at a time, their normalisers with them
    const float l = lane < 16 && s0 + lane < nseg ? __ldcg(slot(s0 + lane) + part_l(GS) + h) : 0.f;
    float4 xa[16];
#pragma unroll
    for (int j = 0; j < 16; ++j)
      xa[j] = s0 + j < nseg ? __ldcg(reinterpret_cast<const float4*>(slot(s0 + j) + h * 128 + 4 * lane))
                            : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      a.x += xa[j].x; a.y += xa[j].y; a.z += xa[j].z; a.w += xa[j].w;
    }
    L += warp_sum(l);
  }
  if (P.suf_part) {  // the dense suffix joins the same softmax (Appendix E.1 and E.2)
    const int len = max(0, min(P.suf_len[u / P.n_kv_heads], P.suf_cap));
    if (len > 0) {
      // the compressed part's reference m, the common maximum M over it and the chunks' maxima, and every
      // part rescaled to M
      const float* sp0 = P.suf_part + (size_t)u * P.n_sch * suf_floats(GS);
      const int nsc = (len + SCH - 1) / SCH;
      float M = m;
      for (int c = lane; c < nsc; c += 32) M = fmaxf(M, sp0[(size_t)c * suf_floats(GS) + suf_m(GS) + h]);
      M = warp_max(M);
      const float f0 = exp2_approx(m - M);
      a.x *= f0;
      a.y *= f0;
      a.z *= f0;
      a.w *= f0;
      L *= f0;
      for (int c = 0; c < nsc; ++c) {
        const float* sp = sp0 + (size_t)c * suf_floats(GS);
        const float f = exp2_approx(sp[suf_m(GS) + h] - M);
        const float4 o = *reinterpret_cast<const float4*>(sp + h * 128 + 4 * lane);
        a.x = fmaf(f, o.x, a.x);
        a.y = fmaf(f, o.y, a.y);
        a.z = fmaf(f, o.z, a.z);
        a.w = fmaf(f, o.w, a.w);
        L = fmaf(f, sp[suf_l(GS) + h], L);
      }
    }
  }
  const bool bad = !(L < INFINITY);  // a failure, or a logit so far above the reference that the sums overflowed
  const float yv[4] = {a.x, a.y, a.z, a.w};
  const size_t o = qrow_base(u, P.n_kv_heads, P.n_q_heads) + (size_t)h * 128 + 4 * lane;
  float y[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) y[e] = bad ? __int_as_float(0x7FC00000) : yv[e] / L;
  *reinterpret_cast<uint2*>(P.out + o) = make_uint2(pack_b2(__float2bfloat16_rn(y[0]), __float2bfloat16_rn(y[1])),
                                                    pack_b2(__float2bfloat16_rn(y[2]), __float2bfloat16_rn(y[3])));
  if (P.out_f32) *reinterpret_cast<float4*>(P.out_f32 + o) = make_float4(y[0], y[1], y[2], y[3]);
}

// Probabilities of one token for every head: p_g = 2^(gamma S_A[a][g] + rt_g) (rt: the key-residual
// term minus m, or -m), added into the normaliser sums.
template <int GS, int NP>
__device__ __forceinline__ void head_probs(float gk, const float (&sa)[GS], const float (&rt)[GS], float2 (&pe)[NP],
                                           float2 (&l2)[NP]) {
  if constexpr (GS == 1) {
    const float p = exp2_approx(fmaf(gk, sa[0], rt[0]));
    pe[0] = make_float2(p, 0.f);
    l2[0].x += p;
  } else {
    const float2 gk2 = make_float2(gk, gk);
#pragma unroll
    for (int i2 = 0; i2 < NP; ++i2) {
      const float2 x = __ffma2_rn(gk2, make_float2(sa[2 * i2], sa[2 * i2 + 1]), make_float2(rt[2 * i2], rt[2 * i2 + 1]));
      pe[i2] = make_float2(exp2_approx(x.x), exp2_approx(x.y));
      l2[i2] = __fadd2_rn(l2[i2], pe[i2]);
    }
  }
}

// ============================ RoPE at decode (AKV_FLAG_ROPE) ============================
// Keys are stored pre-RoPE, so a token's score no longer factors through its anchor's score:
// q . R(p_i) x^_i with x^_i = gamma_i x_a(i) + r~_i (Eq. 3) and R(p) the rotate-half RoPE turn
// of dimension pairs (j, j + 64) by p theta_j (Section 3.2; Appendix E.1's score kernel rebuilds
// keys and applies RoPE from the stored positions the same way).  A warp takes 64 consecutive stored tokens
// (a word of the bitmap), 16 at a time, in the layout of the products' A operand: lane (r8, c4) holds dimension
// pairs 16 c4 .. 16 c4 + 15 of tokens r8 and r8 + 8, so a key is rebuilt, turned and split into fp16 high and
// low parts in the registers that the products read (no shuffles, no shared memory; q exact).  The residuals of
// the few tokens that have one are inverse-rotated by the whole warp into shared memory first.  The angle
// of pair j at position p is taken as a binary fraction of a turn, p * turn_j mod 2^64 (exact integer
// arithmetic; its upper 32 bits are kept, as a signed fraction), so the sine and cosine are evaluated on [-pi, pi)
// whatever the position.
// Bound: issue slots (51-57 % of them used, about 80 warp instructions per token: 2 x 64 x (angle, sine, cosine,
// turn, split)) and the latencies between them at 3 blocks of 136 registers per SM; the special-function units are
// next.  8 KV heads, requests of 40960, 20011, 65536 and 9001 tokens (1.08 M tokens), G = 4: 138 us; a warp per
// token with four dimensions per lane, which traded angles and partners by shuffles and passed keys through shared
// memory, took 322 us (163 warp instructions per token).  Of the whole decode, 179 us: with records read two tokens
// ahead 198, with 96 registers and 5 blocks per SM 205 (spills).
constexpr int kRopeWarps = 4;
template <int GS, int CODEC>
__global__ void __launch_bounds__(kRopeWarps * 32) akv_rope_logits_kernel(const RopeParams P) {
  __shared__ __align__(16) float rs[kRopeWarps][17][132];  // a group's inverse-rotated residuals, and a row of zeros
  __shared__ uint2 turn[64];                               // low and high words
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r8 = lane >> 2, c4 = lane & 3;
  const int n_blk = (P.n_tch + kRopeWarps - 1) / kRopeWarps;
  const int u = blockIdx.x / n_blk, c = (blockIdx.x % n_blk) * kRopeWarps + warp;  // unit, 64-token chunk
  const akv_unit_desc* d = unit_desc(P.arena, u);
  const int S = d->len, k = d->n_anchors;
  if (blockIdx.x % n_blk == 0 && tid < 8) unit_counters(P.uh, P.uh_stride, u, GS)[tid] = 0u;
  if (tid < 64) turn[tid] = make_uint2((uint32_t)P.turn[tid], (uint32_t)(P.turn[tid] >> 32));
  *reinterpret_cast<float4*>(&rs[warp][16][4 * lane]) = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const int ts0 = 64 * c;
  if (ts0 >= S) return;  // past this unit's end (a shorter request)
  const size_t qb = qrow_base(u, P.n_kv_heads, P.n_q_heads);
  // B operand, head r8: k places (2 c4, 2 c4 + 1) of step ks are dims 16 c4 + 2 ks, + 1, those 8 on dims 64 higher
  uint32_t bq[8][2];
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float2 v = make_float2(0.f, 0.f);
      if (r8 < GS) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(P.q + qb + (size_t)r8 * 128 + 64 * h + 16 * c4 + 2 * ks);
        v = make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
      }
      const __half2 b = __float22half2_rn(v);
      bq[ks][h] = *reinterpret_cast<const uint32_t*>(&b);
    }
  // the chunk inside its tile block: one bitmap word (64 tokens) per side
  const int j = ts0 / T, tl0 = ts0 % T;
  const int n = min(T, S - j * T), nw = (int)tile_words(n), n64 = 64 * nw;
  const uint8_t* blk = P.arena + d->off_tiles + reinterpret_cast<const uint32_t*>(P.arena + d->off_tile_table)[j];
  const uint64_t* bm = reinterpret_cast<const uint64_t*>(blk + 8 * n64);
  const uint16_t* rkk = reinterpret_cast<const uint16_t*>(blk + 8 * n64 + 16 * nw);
  const uint16_t* rkv = reinterpret_cast<const uint16_t*>(blk + 8 * n64 + 16 * nw + round16(2u * nw));
  const int nk = rkk[nw - 1] + __popcll(bm[nw - 1]), nv = rkv[nw - 1] + __popcll(bm[nw + nw - 1]);
  const uint32_t F = tile_fixed_bytes(n);
  const uint32_t sm_k = F, cd_k = F + round16(4u * (uint32_t)nk) + round16(4u * (uint32_t)nv);
  const uint64_t word = bm[tl0 / 64];
  const int rbase = rkk[tl0 / 64];
  const uint8_t* AK = P.arena + d->off_anchor_k;
  const uint32_t* kst = reinterpret_cast<const uint32_t*>(blk) + tl0;
  const uint32_t* pos = reinterpret_cast<const uint32_t*>(P.arena + d->off_pos) + ts0;
  // rotation signs of dims 4 lane .. 4 lane + 3 with the 1/128 folded in (the residuals' layout)
  float sgn128[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const unsigned long long sb = lane < 16 ? P.sign_lo : P.sign_hi;
    sgn128[e] = (P.rotate ? (((sb >> ((4 * lane + e) & 63)) & 1ull) ? -1.f : 1.f) : 1.f) * (P.rotate ? 1.0f / 128.0f : 1.f);
  }
  const int n_tok = min(64, S - ts0);  // the chunk's tokens
  float mx[2] = {-INFINITY, -INFINITY};
  // stream words and positions of the lane's tokens r8 and r8 + 8 of a group, read one group ahead
  uint32_t ekn[2], psn[2];
  auto read_words = [&](int g) {
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int t = 16 * g + 8 * x + r8;
      ekn[x] = t < n_tok ? kst[t] : 0u;
      psn[x] = t < n_tok ? pos[t] : 0u;
    }
  };
  read_words(0);
#pragma unroll 1  // (unrolled, the four groups' code does not fit the instruction cache: 251 us, not 138)
  for (int g = 0; 16 * g < n_tok; ++g) {
    const uint32_t ek[2] = {ekn[0], ekn[1]}, ps[2] = {psn[0], psn[1]};
    read_words(g + 1);
    // the anchor rows' 16-byte chunks 2 c4, 2 c4 + 1 and 8 + 2 c4, 9 + 2 c4 (stored at chunk ^ (slot % 8))
    uint4 xr[2][4];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int a = min((int)(ek[x] & 0xFFFFu), k - 1);
      const uint8_t* row = AK + (size_t)a * 256;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int ch = (h >> 1) * 8 + 2 * c4 + (h & 1);
        xr[x][h] = *reinterpret_cast<const uint4*>(row + 16 * (ch ^ (a & 7)));
      }
    }
    // residuals of the group's tokens: r~ = s o H(c^) / 128, c^ = min + scale L[code], into shared memory
    const uint32_t wbits = (uint32_t)(word >> (16 * g)) & 0xFFFFu;
    if (wbits) {
      __syncwarp();  // the last group's rows are read
      for (uint32_t left = wbits; left; left &= left - 1u) {
        const int i = __ffs(left) - 1;
        const int r = rbase + __popcll(word & ((1ull << (16 * g + i)) - 1ull));
        const uint32_t smn = *reinterpret_cast<const uint32_t*>(blk + sm_k + 4u * (uint32_t)r);
        const uint32_t byte = blk[cd_k + 32u * (uint32_t)r + (uint32_t)lane];
        float cr[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) cr[e] = fmaf(half_lo(smn), code_level((byte >> (2 * e)) & 3u, CODEC), half_hi(smn));
        if (P.rotate) warp_wht128(cr, lane);
        *reinterpret_cast<float4*>(&rs[warp][i][4 * lane]) =
            make_float4(cr[0] * sgn128[0], cr[1] * sgn128[1], cr[2] * sgn128[2], cr[3] * sgn128[3]);
      }
      __syncwarp();
    }
    float d4[4] = {0.f, 0.f, 0.f, 0.f};
    const float gk[2] = {half_hi(ek[0]), half_hi(ek[1])};
    // a token's residual row, or the zeros
    const float* rrow[2] = {rs[warp][((wbits >> r8) & 1u) ? r8 : 16] + 16 * c4, rs[warp][((wbits >> (r8 + 8)) & 1u) ? r8 + 8 : 16] + 16 * c4};
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {  // pairs 16 c4 + 2 ks, + 1
      uint32_t hi[4], lo[4];          // A: token r8 lower dims, token r8 + 8 lower, r8 upper, r8 + 8 upper
      const uint2 tn0 = turn[16 * c4 + 2 * ks], tn1 = turn[16 * c4 + 2 * ks + 1];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const uint4 cl = xr[x][ks >> 2], cu = xr[x][2 + (ks >> 2)];
        const uint32_t wl = (ks & 3) == 0 ? cl.x : ((ks & 3) == 1 ? cl.y : ((ks & 3) == 2 ? cl.z : cl.w));
        const uint32_t wu = (ks & 3) == 0 ? cu.x : ((ks & 3) == 1 ? cu.y : ((ks & 3) == 2 ? cu.z : cu.w));
        const float2 rl = *reinterpret_cast<const float2*>(rrow[x] + 2 * ks), ru = *reinterpret_cast<const float2*>(rrow[x] + 64 + 2 * ks);
        const float a0 = fmaf(gk[x], __uint_as_float(wl << 16), rl.x), a1 = fmaf(gk[x], __uint_as_float(wl & 0xFFFF0000u), rl.y);
        const float b0 = fmaf(gk[x], __uint_as_float(wu << 16), ru.x), b1 = fmaf(gk[x], __uint_as_float(wu & 0xFFFF0000u), ru.y);
        const uint32_t p = ps[x];
        float s0, c0, s1, c1;
        __sincosf((float)(int)(__umulhi(p, tn0.x) + p * tn0.y) * (6.2831853071795865f / 4294967296.0f), &s0, &c0);
        __sincosf((float)(int)(__umulhi(p, tn1.x) + p * tn1.y) * (6.2831853071795865f / 4294967296.0f), &s1, &c1);
        const float2 yl = make_float2(fmaf(a0, c0, -b0 * s0), fmaf(a1, c1, -b1 * s1));
        const float2 yu = make_float2(fmaf(b0, c0, a0 * s0), fmaf(b1, c1, a1 * s1));
        const __half2 hl = __float22half2_rn(yl), hu = __float22half2_rn(yu);
        const float2 fl = __half22float2(hl), fu = __half22float2(hu);
        const __half2 ll = __float22half2_rn(make_float2(yl.x - fl.x, yl.y - fl.y));
        const __half2 lu = __float22half2_rn(make_float2(yu.x - fu.x, yu.y - fu.y));
        hi[x] = *reinterpret_cast<const uint32_t*>(&hl);
        hi[2 + x] = *reinterpret_cast<const uint32_t*>(&hu);
        lo[x] = *reinterpret_cast<const uint32_t*>(&ll);
        lo[2 + x] = *reinterpret_cast<const uint32_t*>(&lu);
      }
      mma_f16(d4, make_uint4(hi[0], hi[1], hi[2], hi[3]), bq[ks][0], bq[ks][1]);
      mma_f16(d4, make_uint4(lo[0], lo[1], lo[2], lo[3]), bq[ks][0], bq[ks][1]);
    }
    // D rows r8, r8 + 8 (tokens), columns 2 c4, 2 c4 + 1 (heads)
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      const int ts = ts0 + 16 * g + r8 + 8 * hr;
      const float l0 = d4[2 * hr] * P.scale_log2, l1 = d4[2 * hr + 1] * P.scale_log2;
      if (ts < S && 2 * c4 < GS) {
        float* o = P.lg + ((size_t)u * P.s_stride + ts) * GS + 2 * c4;
        if constexpr (GS == 1) o[0] = l0;
        else *reinterpret_cast<float2*>(o) = make_float2(l0, l1);
        mx[0] = fmaxf(mx[0], l0);
        mx[1] = fmaxf(mx[1], l1);
      }
    }
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    mx[0] = fmaxf(mx[0], __shfl_xor_sync(0xffffffffu, mx[0], o));
    mx[1] = fmaxf(mx[1], __shfl_xor_sync(0xffffffffu, mx[1], o));
  }
  if (lane < 4) {
    float* o = P.cmax + ((size_t)u * P.n_tch + c) * GS;
    if (2 * lane < GS) o[2 * lane] = mx[0];
    if (2 * lane + 1 < GS) o[2 * lane + 1] = mx[1];
  }
}

// A lane's tokens of a tile: bitmap bytes and first record indices.
struct TokLane {
  uint32_t kbits, vbits;
  int rk, rv, t0;
};
// What the general token path reads of its tile.
struct TokTile {
  TileView tv;
  const uint8_t* gb;  // the block in global memory
  uint32_t lo, nrows;
  const float* SAt;   // anchor scores [k][GS]
  const float* rows;  // [0,8): -m, [8,16): -inf, [16,24): sum q'
  const float* qp;    // [GS][128] rotated query
  float* pv;          // [R][GS] p rows of the value records
  float* W;           // [nrows][GS] the tile's value weights
  float* ovf;         // [2][GS][128] overflow sums
  const uint8_t* AV;  // the unit's anchor values (global)
  const float* lgt;   // RoPE at decode: the tile's logit rows [T][GS] (global), else null
  int* ovl_n;         // the tile's overflow lists: value records beyond the staged ones, and runs
  float* ovl;         // beyond the weight rows, applied by the whole group after the tokens
  int k, nKs, nVs, ka, lloyd;
};

// The general token path (kept out of line: a tile with records beyond the staged ones, or runs
// beyond its weight rows): the same arithmetic as
// the fast path, with the rare cases on CUDA cores; it returns the lane's share of the
// normaliser (a shared-memory sum would take every lane's addition on the same words).  The
// arguments arrive by value and are copied into locals first: the shared-memory reductions below clobber memory, so a field read
// through the argument itself would be reloaded from its local-memory copy (L2 latency, the
// L1 here being small) after every reduction.
template <int NP>
struct LShare {
  float2 v[NP];
};
template <int GS>
__device__ __noinline__ LShare<(GS >= 2 ? GS / 2 : 1)> token_chunk_general(const TokTile tt_arg, const TokLane tl_arg) {
  constexpr int NP = GS >= 2 ? GS / 2 : 1;
  const TokTile tt = tt_arg;
  const TokLane tl = tl_arg;
  const TileView tv = tt.tv;
  const uint8_t* st = tv.st;
  const uint8_t* gb = tt.gb;
  const uint32_t staged = tv.staged;
  const int t0 = tl.t0;
  const int nvalid = min(LCH, tv.n - t0);
  const float* rsb = reinterpret_cast<const float*>(st + tv.cd_k);
  const float* negrow = tt.rows;
  const float* ninfrow = tt.rows + 8;
  const float* qp = tt.qp;
  const float* SAt = tt.SAt;
  float* W = tt.W;
  float* pv = tt.pv;
  float* ovf = tt.ovf;
  const uint8_t* AV = tt.AV;
  const float* lgt = tt.lgt;
  int* ovl_n = tt.ovl_n;
  float* ovl = tt.ovl;
  const int k = tt.k, nKs = tt.nKs, nVs = tt.nVs, ka = tt.ka, lloyd = tt.lloyd;
  const uint32_t lo = tt.lo;
  const int nrows = (int)tt.nrows;
  int rkn = tl.rk, rvn = tl.rv;
  const uint32_t kbits = tl.kbits, vbits = tl.vbits;
  float2 l2[NP];
#pragma unroll
  for (int i2 = 0; i2 < NP; ++i2) l2[i2] = make_float2(0.f, 0.f);
  uint32_t key = *reinterpret_cast<const uint32_t*>(st + 4 * (tv.n64 + t0)) & 0xFFFFu;
  float2 acc[NP];
#pragma unroll
  for (int i2 = 0; i2 < NP; ++i2) acc[i2] = make_float2(0.f, 0.f);
  auto flush = [&](uint32_t kk, const float2 (&v)[NP]) {
    const int ix = (int)(kk - lo);
    float vv[GS];
#pragma unroll
    for (int g = 0; g < GS; ++g) vv[g] = (g & 1) ? v[g >> 1].y : v[g >> 1].x;
    if (ix < nrows) {
      float* w = W + ix * GS;
#pragma unroll
      for (int g = 0; g < GS; ++g) red_local(w + g, vv[g]);
    } else {  // beyond the weight rows: listed for the group (else on CUDA cores here)
      const int e = atomicAdd(ovl_n + 1, 1);
      if (e < kOvl) {
        float* en = ovl + (kOvl + e) * 9;
        en[0] = __int_as_float((int)kk);
#pragma unroll
        for (int g = 0; g < GS; ++g) en[1 + g] = vv[g];
      } else {
        anchor_value_add<GS>(AV, (int)kk, vv, ovf);
      }
    }
  };
  for (int e = 0; e < LCH; ++e) {
    const uint32_t ek = e < nvalid ? *reinterpret_cast<const uint32_t*>(st + 4 * (t0 + e)) : 0u;
    const uint32_t ev = e < nvalid ? *reinterpret_cast<const uint32_t*>(st + 4 * (tv.n64 + t0 + e)) : 0u;
    const int a = min((int)(ek & 0xFFFFu), k - 1);
    float sa[GS], rt[GS];
    if (lgt) {  // RoPE: the token's logits (no anchor-score table)
#pragma unroll
      for (int g = 0; g < GS; ++g) sa[g] = 0.f;
    } else {
      load_sa_row<GS>(SAt, a, ka, sa);
    }
    const bool kb = (kbits >> e) & 1u;
    const int r = rkn;
    rkn += (int)kb;
    if (lgt) {  // RoPE: the logits minus m, or -inf for a token past the tile's end
      load_row<GS>(e >= nvalid ? ninfrow : negrow, rt);
      if (e < nvalid) {
#pragma unroll
        for (int g = 0; g < GS; ++g) rt[g] += lgt[(t0 + e) * GS + g];
      }
    } else if (kb && r >= nKs && e < nvalid) {  // beyond the staged records
#pragma unroll
      for (int g = 0; g < GS; ++g)
        rt[g] = key_record_term(st, gb, staged, tv.sm_k + 4u * (uint32_t)r, tv.cd_k + 32u * (uint32_t)r, qp + g * 128,
                                qp[GS * 128 + g], lloyd) +
                negrow[g];
    } else {  // the key-residual terms minus m, -m, or -inf for a token past the tile's end
      load_row<GS>(e >= nvalid ? ninfrow : negrow, rt);
      if (kb && e < nvalid) {
        float rs[GS];
        load_row<GS>(rsb + r * 8, rs);
#pragma unroll
        for (int g = 0; g < GS; ++g) rt[g] += rs[g];
      }
    }
    const float gk = lgt ? 0.f : half_hi(ek), gv = half_hi(ev);
    float2 pe[NP];
    head_probs<GS, NP>(gk, sa, rt, pe, l2);
    const bool vb = (vbits >> e) & 1u;
    const int rv = rvn;
    rvn += (int)vb;
    if (vb && e < nvalid) {
      if (rv < nVs) {
        store_row<GS>(pv + rv * GS, pe);
      } else {  // beyond the staged records: listed for the group (else on CUDA cores here)
        const int en_i = atomicAdd(ovl_n, 1);
        if (en_i < kOvl) {
          float* en = ovl + en_i * 9;
          en[0] = __int_as_float(rv);
#pragma unroll
          for (int g = 0; g < GS; ++g) en[1 + g] = (g & 1) ? pe[g >> 1].y : pe[g >> 1].x;
        } else {
#pragma unroll
          for (int g = 0; g < GS; ++g)
            value_record_add(st, gb, staged, tv.sm_v + 4u * (uint32_t)rv, tv.cd_v + 512u * (uint32_t)(rv / 16), rv,
                             (g & 1) ? pe[g >> 1].y : pe[g >> 1].x, ovf + GS * 128 + g * 128, lloyd);
        }
      }
    }
    // tokens past the tile join the current run with zero weight
    const uint32_t av = e < nvalid ? (ev & 0xFFFFu) : key;
    if (av != key) {
      flush(key, acc);
      key = av;
#pragma unroll
      for (int i2 = 0; i2 < NP; ++i2) acc[i2] = make_float2(0.f, 0.f);
    }
    const float2 gv2 = make_float2(gv, gv);
#pragma unroll
    for (int i2 = 0; i2 < NP; ++i2) acc[i2] = __ffma2_rn(pe[i2], gv2, acc[i2]);
  }
  flush(key, acc);
  LShare<NP> ls;
#pragma unroll
  for (int i2 = 0; i2 < NP; ++i2) ls.v[i2] = l2[i2];
  return ls;
}

// w^T V_A over the value slots of a tile that have a weight row but no staged anchor-value row (slots nr .. nw - 1, and those
// among the token warps' first and last runs), their rows read from global memory, on CUDA cores, added into the overflow's
// sums ov[g][:]: product thread t takes dimension t % 128 of every other slot.  A tile has such slots where a unit's
// anchors are more than one token in five or so, and staging all their rows would leave the ring no room.
// W: the weights; ends: the runs' weights as the operand built from them; vs: their slots; AV: slot 0's row.
template <int GS>
__device__ __forceinline__ void unstaged_rows(const float* W, const uint32_t* ends, const int* vs, const uint8_t* AV, uint32_t lo, int nr, int nw,
                                          int t, float* ov) {
  const int dim = t & 127;
  float av[GS];
#pragma unroll
  for (int g = 0; g < GS; ++g) av[g] = 0.f;
  auto value = [&](int slot) {  // (rows are stored swizzled by the slot)
    return __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(AV + (size_t)slot * 256 + 16 * ((uint32_t)(dim >> 3) ^ ((lo + (uint32_t)slot) & 7u)) + 2 * (dim & 7)));
  };
#pragma unroll 4
  for (int slot = nr + (t >> 7); slot < nw; slot += 2) {
    float w[GS];
    load_row<GS>(W + slot * GS, w);
    const float x = value(slot);
#pragma unroll
    for (int g = 0; g < GS; ++g) av[g] = fmaf(w[g], x, av[g]);
  }
  for (int e = t >> 7; e < kEnds; e += 2) {
    if (vs[e] < nr) continue;
    const float x = value(vs[e]);
#pragma unroll
    for (int g = 0; g < GS; ++g) {  // head g's place e of the operand: bf16 high and low parts
      const uint32_t* f = ends + 4 * (4 * g + (e & 7) / 2) + 2 * (e >> 3);
      const int sh = 16 * (e & 1);
      av[g] = fmaf(__uint_as_float((f[0] >> sh) << 16) + __uint_as_float((f[1] >> sh) << 16), x, av[g]);
    }
  }
#pragma unroll
  for (int g = 0; g < GS; ++g) red_local(ov + g * 128 + dim, av[g]);
}

// ================================ decode ============================================
// CODEC: 0 = uniform codes (c^ = min + c scale), 1 = Lloyd-Max levels (c^ = scale L[c]).
// MODE: where a unit's anchor scores are.  kTableSmem: copied from the score launch into shared memory;
// kTableGlobal: read from global memory where the score launch left them; kTableHalf (GS = 8): heads 0-3 in shared, heads 4-7
// in global memory; kRope: pre-RoPE keys, every
// token's logit comes from the RoPE logits launch (P.lg) instead of gamma S_A plus its key-residual
// term, and the key-residual phase has nothing to do.
enum Mode { kTableSmem = 0, kTableGlobal = 1, kRope = 2, kTableHalf = 3 };
// TURN: the token warps copy the tiles in turn.  With small query groups and no residual records a tile's tokens and values
// take so little that copying the next one, some 1500 cycles of one lane, is what every other warp waits for: 4 requests of
// 131072, 8 KV heads, G = 1 and 2, 1 % anchors 59.8 -> 55.6 us and 61.8 -> 57.6, 2 % 63.6 -> 59.7 and 64.8 -> 61.7.  With
// records the product warps are the longer side, and the other lanes' looks at the state cost 0 to 3 % (1 % of records
// already); calls of a few tiles per CTA lose by its set-up (3 requests of 16001, 9000 and 4173, 5 % records, G = 1: 18.57 ->
// 18.88; no records, even at 7 and 9 tiles per CTA, 39.5 -> 38.4 at 13), hence kTurnTiles.
// WIDE: tiles may cover more value slots than have their anchor-value rows staged (P.XW > P.X); kernels of their own,
// since the same code as a branch, inline or called, made the others slower (8 x 131072, G = 8: 164 -> 178, 193 us).
template <int GS, int CODEC, int MODE, bool WIDE = false, bool TURN = false>
__global__ void __launch_bounds__(NT, 1) akv_decode_kernel(const DecodeParams P) {
  extern __shared__ __align__(128) uint8_t smem[];
  constexpr int NP = GS >= 2 ? GS / 2 : 1;      // pairs of heads for the packed arithmetic
  constexpr bool ROPE = MODE == kRope, TABLE = MODE == kTableSmem;
  constexpr int PF = part_floats(GS);
  constexpr int NBF = GS == 8 ? 2 : 1;  // key-residual fragment sets: GS = 8 keeps high and low parts apart
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c4 = lane & 3, r8 = lane >> 2;
  const int c = blockIdx.x;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + P.o_bar);
  Meta* meta = reinterpret_cast<Meta*>(smem + P.o_meta);
  volatile int* failed = reinterpret_cast<volatile int*>(smem + P.o_misc);
  Seg* sg = reinterpret_cast<Seg*>(smem + P.o_misc + 16);  // the segment in work
  float* SAs = reinterpret_cast<float*>(smem + P.o_sa);
  float* ovf = reinterpret_cast<float*>(smem + P.o_ovf);  // [2][GS][128]: anchor-value and value-residual overflow sums
  float* qp = reinterpret_cast<float*>(smem + P.o_qp);    // [GS][128] rotated query q'; at a segment's end its sums [2][GS][128]
  float* sq = qp + GS * 128;                              // [8] sums of q' per head
  uint2* qf = reinterpret_cast<uint2*>(sq + 8);           // [NBF][8][32] key-residual B fragments
  float* rows = reinterpret_cast<float*>(smem + P.o_rows);  // [0,8): -m, [8,16): -inf, [24,32): m
  float* gsum = reinterpret_cast<float*>(smem + P.o_gsum);  // [8][8] normaliser per token warp, then [8][8] sum of p min per product warp
  uint8_t* ring = smem + P.o_ring;
  // per slot: a tile block and its anchor-value rows landed, and its place is free again; per tile parity: its key
  // terms are written, its tokens are done; per unit: query header and score table landed
  auto bar_full = [&](int s) { return smem_u32(bars + s); };
  auto bar_empty = [&](int s) { return smem_u32(bars + NSG + s); };
  auto bar_kdone = [&](int b) { return smem_u32(bars + 2 * NSG + b); };
  auto bar_tdone = [&](int b) { return smem_u32(bars + 2 * NSG + 2 + b); };
  const uint32_t bar_hdr = smem_u32(bars + 2 * NSG + 4), bar_sa_full = smem_u32(bars + 2 * NSG + 5);

  // This CTA's range of the concatenated tiles, walked as segments (one per unit it touches).
  // (products of tile indexes and CTAs stay below 2^32 for all but the largest calls: 32-bit divisions)
  const bool small = (unsigned long long)P.ttot * (unsigned)P.grid < (1ull << 32);
  auto quot = [&](long long x, long long y) -> long long { return small ? (long long)((unsigned)x / (unsigned)y) : x / y; };
  const long long B0 = quot((long long)c * P.ttot, P.grid), B1 = quot((long long)(c + 1) * P.ttot, P.grid);
  const int n_cta_tiles = (int)(B1 - B0);
  auto seg_fill = [&](Seg& s) {
    s.nt = unit_desc(P.arena, s.u)->n_tiles;
    s.je = (int)min((long long)s.nt, B1 - s.t0);
    s.first = (int)quot((s.t0 + 1) * P.grid - 1, P.ttot);
    s.nseg = (int)quot((s.t0 + s.nt) * P.grid - 1, P.ttot) - s.first + 1;
  };
  auto seg_begin = [&](Seg& s) {
    s.u = P.cta_unit[c];
    s.jb = P.cta_tile[c];
    s.t0 = B0 - s.jb;
    s.ib = 0;
    seg_fill(s);
  };
  auto seg_next = [&](Seg& s) {  // (not past the last segment)
    s.ib += s.je - s.jb;
    s.t0 += s.nt;
    ++s.u;
    s.jb = 0;
    seg_fill(s);
  };
  // The unit's query header, and its anchor-score table where it comes from the score launch (one thread;
  // the sums kept where the header goes have been read).
  auto start_unit = [&](int u) {
    const int k = unit_desc(P.arena, u)->n_anchors;
    const bool ok = !*failed;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (ok && !ROPE) {  // (RoPE: no key-side header is needed)
      mbar_expect_tx(bar_hdr, (uint32_t)hdr_bytes(GS));
      bulk_g2s(smem_u32(qp), P.uh + (size_t)u * P.uh_stride, (uint32_t)hdr_bytes(GS), bar_hdr);
    } else {
      mbar_arrive(bar_hdr);
    }
    if (MODE == kTableHalf && ok) {
      mbar_expect_tx(bar_sa_full, 16u * (uint32_t)k);
      bulk_g2s(smem_u32(SAs), P.sa + (size_t)u * P.ka_stride * GS, 16u * (uint32_t)k, bar_sa_full);
    } else if (MODE == kTableSmem && ok) {
      const float* src = P.sa + (size_t)u * P.ka_stride * GS;
      if (GS == 8) {  // the two four-head arrays, k rows of each
        const uint32_t half = 16u * (uint32_t)k;
        mbar_expect_tx(bar_sa_full, 2 * half);
        bulk_g2s(smem_u32(SAs), src, half, bar_sa_full);
        bulk_g2s(smem_u32(SAs + (size_t)P.ka_stride * 4), src + (size_t)P.ka_stride * 4, half, bar_sa_full);
      } else {
        const uint32_t bytes = round16(4u * (uint32_t)(k * GS));
        mbar_expect_tx(bar_sa_full, bytes);
        bulk_g2s(smem_u32(SAs), src, bytes, bar_sa_full);
      }
    } else {
      mbar_arrive(bar_sa_full);  // the unit's start, for the warps that wait on it
    }
  };

  // ---- copies: lane 0 of token warp 0.  Each tile goes, with the anchor-value rows of the value slots it
  // covers, into the ring, oldest first, as places come free; the table entries of the next tile are read
  // one tile ahead ----
  // TURN: tile ii by lane 0 of token warp ii % 8, except that warp 0 copies the first three; each such lane has a segment
  // and table entries of its own (read a turn, eight tiles, ahead), the state common to all is warp 0's and is handed on by
  // its ii: whoever finds its own tile there sees what the turns before left.
  Prod* pr = reinterpret_cast<Prod*>(smem + P.o_prod);
  Prod* pw = TURN ? pr + (warp & (NTW - 1)) : pr;
  int mine = warp < 3 && warp > 0 ? warp + NTW : warp;  // TURN: this lane's next tile
  uint32_t pe0 = 0, pe1 = 0, pe2 = 0;  // table entries of the next tile to copy: block offset, next offset, slot range
  auto read_entry = [&](int ii) {
    if (ii >= n_cta_tiles) return;
    if (ii >= pw->end) {  // (and at the start)
      Seg s = pw->s;
      while (ii >= s.ib + (s.je - s.jb)) seg_next(s);
      const akv_unit_desc* d = unit_desc(P.arena, s.u);
      pw->s = s;
      pw->end = s.ib + (s.je - s.jb);
      pw->tiles = P.arena + d->off_tiles;
      pw->av = P.arena + d->off_anchor_v;
      pw->table = reinterpret_cast<const uint32_t*>(P.arena + d->off_tile_table);
    }
    const int pj = pw->s.jb + (ii - pw->s.ib);
    const uint32_t* table = pw->table;
    pe0 = table[pj];
    pe1 = table[pj + 1];
    pe2 = table[pw->s.nt + 1 + pj];
  };
  // (one tile a call: the entries read after it are not waited for)
  auto copy_more = [&]() {  // the next tile, if it fits now (never waits)
    const int ii = TURN ? *(volatile int*)&pr->ii : pr->ii;
    if (TURN && ii != mine) return;
    if (ii < n_cta_tiles && !*failed) {
      if constexpr (TURN) __threadfence_block();  // what the turns before left
      const uint32_t RB = (uint32_t)P.ring_bytes;
      const uint32_t lo = pe2 & 0xFFFFu, hi = pe2 >> 16;
      const uint32_t staged = min(pe1 - pe0, (uint32_t)P.cap);
      const uint32_t nrows = min(hi - lo + 1u, (uint32_t)P.X);
      const uint32_t sz = staged + 256u * nrows;
      int nrel = pr->nrel;
      uint32_t used = pr->used;
      while (nrel < ii && mbar_test(bar_empty(nrel % NSG), (uint32_t)(nrel / NSG) & 1u)) {
        used -= meta[nrel % NSG].bytes;
        ++nrel;
      }
      pr->nrel = nrel;
      pr->used = used;
      const uint32_t head = pr->head;
      uint32_t at = 0;
      bool fits = ii - nrel < NSG;
      if (used > 0) {
        const uint32_t tail = meta[nrel % NSG].ring_off;  // the oldest tile in flight
        if (head > tail) {
          if (head + sz <= RB) at = head;
          else fits = fits && sz <= tail;
        } else {
          at = head;
          fits = fits && head + sz <= tail;
        }
      }
      if (!fits) return;
      const int sl = ii % NSG;
      Meta& mt = meta[sl];
      mt.ring_off = at;
      mt.blk_off = pe0;
      mt.staged = staged;
      mt.lo = lo;
      mt.nrows = nrows;
      mt.j = (uint32_t)(pw->s.jb + (ii - pw->s.ib));
      mt.bytes = sz;
      if constexpr (WIDE) mt.nw = min(hi - lo + 1u, (uint32_t)P.XW);
      // (drop_last: a test withholds the last tile of the range)
      if (P.drop_last > 0 && ii == n_cta_tiles - P.drop_last) {
        mt.nrows |= 0x80000000u;  // withheld: nothing in flight
      } else {
        mbar_expect_tx(bar_full(sl), sz);
        bulk_g2s(smem_u32(ring + at), pw->tiles + pe0, staged, bar_full(sl));
        if (nrows) bulk_g2s(smem_u32(ring + at + staged), pw->av + (size_t)lo * 256, 256u * nrows, bar_full(sl));
      }
      pr->head = at + sz;
      pr->used = used + sz;
      if constexpr (TURN) {
        __threadfence_block();
        *(volatile int*)&pr->ii = ii + 1;
        mine += mine < 2 ? 1 : (mine == 2 ? NTW - 2 : NTW);
        read_entry(mine);
      } else {
        pr->ii = ii + 1;
        read_entry(ii + 1);
      }
    }
  };
  if (tid == 0) {  // the first tile's table entries are on their way while shared memory is set up
    Seg s;
    seg_begin(s);
    *sg = s;
    pr->s = s;
    pr->end = 0;
    pr->ii = pr->nrel = 0;
    pr->head = pr->used = 0;
    read_entry(0);
  }
  if (tid == 0) {
    for (int s = 0; s < NSG; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), NMW);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_kdone(b), NMW);
      mbar_init(bar_tdone(b), NTW);
    }
    mbar_init(bar_hdr, 1);
    mbar_init(bar_sa_full, 1);
    *failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int e = tid; e < 2 * GS * 128; e += NT) ovf[e] = 0.f;  // (the overflow's sums start at zero)
  __syncthreads();

  if (tid == 0)
    for (int i = 0; i < 3; ++i) copy_more();
  if constexpr (TURN) {
    if (warp > 0 && warp < NTW && lane == 0 && mine < n_cta_tiles) {
      Seg s;
      seg_begin(s);
      pw->s = s;
      pw->end = 0;
      read_entry(mine);
    }
  }

  // =========================== token warps, product warps ==========================
  const bool tok = warp < NTW;
  const int wi8 = tok ? warp : warp - NTW;  // index among the role's warps
  const int mt_ = tid - NTW * 32;           // thread among the product warps
  auto all_sync = [&]() { named_sync(1, NCW * 32); };
  auto tok_sync = [&]() { named_sync(2, NTW * 32); };
  auto prod_sync = [&]() { named_sync(3, NMW * 32); };
  // (the launch before this one, and everything before it, is complete past this point)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid == 0) start_unit(sg->u);

  int lt = 0;     // this CTA's tiles so far
  int sigma = 0;  // segments so far
  for (;; ++sigma) {
    const int u = sg->u, S = unit_desc(P.arena, u)->len, k = unit_desc(P.arena, u)->n_anchors;
    const int n_seg = sg->je - sg->jb;
    // a bounded wait of the whole warp; after a failure nothing is waited for any more
    auto wait_or_fail = [&](uint32_t bar, uint32_t parity) {
      uint32_t done = mbar_try(bar, parity);
      if (__all_sync(0xffffffffu, done)) return true;
      unsigned long long t_0 = 0;
      for (unsigned n = 0;; ++n) {
        if (!done) done = mbar_try(bar, parity);
        if (__all_sync(0xffffffffu, done)) return true;
        if (warp_failed(failed)) return false;
        if ((n & 63u) == 63u) {
          const unsigned long long now = __shfl_sync(0xffffffffu, global_ns(), 0);
          if (t_0 == 0) t_0 = now;
          else if (now - t_0 >= kWaitNs) {
            *failed = 1;
            return false;
          }
        }
      }
    };

    if (tok) {
      // ---- the reference m of each head: the largest anchor score (a lower bound of the largest logit), or
      // with RoPE the largest logit; from the chunk maxima ----
      for (int g = wi8; g < GS; g += NTW) {
        float m = -INFINITY;
        const int nch = ROPE ? (S + 63) / 64 : (k + CHA - 1) / CHA;
        for (int ch = lane; ch < nch; ch += 32) m = fmaxf(m, P.cmax[((size_t)u * P.n_ch + ch) * GS + g]);
        m = warp_max(m);
        if (lane == 0) {
          rows[g] = -m;
          rows[8 + g] = -INFINITY;
          rows[24 + g] = m;
        }
      }
      wait_or_fail(bar_hdr, (uint32_t)sigma & 1u);
      wait_or_fail(bar_sa_full, (uint32_t)sigma & 1u);
      tok_sync();  // m of every head written
      const float* SAt = TABLE ? SAs : P.sa + (size_t)u * P.ka_stride * GS;
      float2 l2[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) l2[i] = make_float2(0.f, 0.f);
      for (int i = 0; i < n_seg; ++i, ++lt) {
        const int b = lt & 1;
        // (the tile itself too: its bytes came through the asynchronous proxy)
        if (warp == 0 || (TURN && n_cta_tiles > 3)) {  // the copying lanes' warps: the ring is topped up, and this tile certainly on its way
          unsigned long long t_0 = 0;
          for (unsigned n = 0;; ++n) {
            if (lane == 0) copy_more();
            __syncwarp();
            if (__shfl_sync(0xffffffffu, TURN ? *(volatile int*)&pr->ii : pr->ii, 0) > lt || warp_failed(failed)) break;
            if ((n & 63u) == 63u) {  // (bounded; the clock is read now and then)
              const unsigned long long now = __shfl_sync(0xffffffffu, global_ns(), 0);
              if (t_0 == 0) t_0 = now;
              else if (now - t_0 >= kWaitNs) break;
            }
          }
        }
        // (its shape comes with the key terms; without one it has no tokens)
        const bool go = wait_or_fail(bar_kdone(b), (uint32_t)(lt >> 1) & 1u) && wait_or_fail(bar_full(lt % NSG), (uint32_t)(lt / NSG) & 1u);
        if (go) {
          const Meta mt = meta[lt % NSG];
          const uint8_t* st = ring + mt.ring_off;
          const TileView tv = tile_view(st, mt, u);
          const bool fast_tile = mt.fast & 1u;
          float* W = reinterpret_cast<float*>(smem + P.o_wb) + (lt % 3) * ((WIDE ? P.XW : P.X) + kEnds) * GS;
          int* vs = reinterpret_cast<int*>(smem + P.o_vs) + (lt % 3) * kEnds;
          float* pv = reinterpret_cast<float*>(smem + P.o_pv) + b * P.R * GS;
          // ---- tokens: lane -> stored tokens t0 .. t0 + 3, every head ----
          const int t0 = wi8 * (32 * LCH) + LCH * lane;
          TokLane tl;
          tl.kbits = tl.vbits = 0u;
          tl.rk = tl.rv = 0;
          tl.t0 = t0;
          if (t0 < tv.n) {
            const int wi = t0 >> 6, sh = t0 & 63;
            const uint64_t wk = tv.bm(0, wi), wv = tv.bm(1, wi);
            tl.kbits = (uint32_t)(wk >> sh) & ((1u << LCH) - 1u);
            tl.vbits = (uint32_t)(wv >> sh) & ((1u << LCH) - 1u);
            tl.rk = tv.rk(0, wi) + __popcll(wk & ((1ull << sh) - 1ull));
            tl.rv = tv.rk(1, wi) + __popcll(wv & ((1ull << sh) - 1ull));
          }
          if (fast_tile) {  // warp-uniform
            // Every record staged, every run with a weight row.  No shared atomics: a run
            // that starts and ends inside a lane's tokens is stored as it is (no other lane has its
            // slot); runs that cross lanes are merged by a segmented scan.  Places past the end of a unit's
            // last tile join its last run with weight 0.
            const int nval = min(LCH, max(0, tv.n - t0)), t0c = min(t0, tv.n64 - LCH);
            const uint32_t last_key = reinterpret_cast<const uint32_t*>(st + 4 * tv.n64)[tv.n - 1] & 0xFFFFu;
            const float* rsb = reinterpret_cast<const float*>(st + tv.cd_k);
            const uint32_t lo = mt.lo;
            const int km1 = k - 1;
            int rk = tl.rk, rv = tl.rv;
            uint32_t key = 0, hk = 0;  // the run in work; the lane's first run (its head), kept for the merge
            bool multi = false;        // the lane's tokens hold more than one run
            float2 acc[NP], hs[NP];
#pragma unroll
            for (int i2 = 0; i2 < NP; ++i2) acc[i2] = hs[i2] = make_float2(0.f, 0.f);
            // RoPE: the lane's tokens' logit rows (global, stored order)
            const float* lgt = ROPE ? P.lg + ((size_t)u * P.s_stride + (size_t)mt.j * T + t0c) * GS : nullptr;
            // the table as shared memory (32-bit addressing, shared loads) or global memory (RoPE: not read)
            const float* SAtab = TABLE ? SAs : P.sa + (size_t)u * P.ka_stride * GS;
            float2 negm2[NP];  // -m: the logit offset of every token
#pragma unroll
            for (int i2 = 0; i2 < NP; ++i2) negm2[i2] = make_float2(rows[2 * i2], GS >= 2 ? rows[2 * i2 + 1] : 0.f);
            auto token_loop = [&](auto tail_c) {
              constexpr bool TAIL = decltype(tail_c)::value;  // some places of the tile hold no token
              uint32_t ek[LCH], ev[LCH];
              load_words<LCH>(st + 4 * t0c, ek);
              load_words<LCH>(st + 4 * (tv.n64 + t0c), ev);
              hk = key = !TAIL || nval > 0 ? ev[0] & 0xFFFFu : last_key;
#pragma unroll
              for (int e = 0; e < LCH; ++e) {
                const bool valid = !TAIL || e < nval;
                const float gv = valid ? half_hi(ev[e]) : 0.f;
                float2 x[NP];
                if constexpr (ROPE) {  // the token's logits from the RoPE logits launch, minus m
                  float lr[GS];
                  load_row<GS>(lgt + e * GS, lr);
#pragma unroll
                  for (int i2 = 0; i2 < NP; ++i2)
                    x[i2] = __fadd2_rn(make_float2(lr[2 * i2], GS >= 2 ? lr[2 * i2 + 1] : 0.f), negm2[i2]);
                } else {
                  const int a = min((int)(ek[e] & 0xFFFFu), km1);  // indices are < k by construction
                  float sa[GS];
                  if constexpr (MODE == kTableHalf) {
                    const float4 v = *reinterpret_cast<const float4*>(SAs + a * 4), w = *reinterpret_cast<const float4*>(SAtab + (P.ka_stride + a) * 4);
                    sa[0] = v.x; sa[1] = v.y; sa[2] = v.z; sa[3] = v.w;
                    sa[4] = w.x; sa[5] = w.y; sa[6] = w.z; sa[7] = w.w;
                  } else {
                    load_sa_row<GS>(SAtab, a, P.ka_stride, sa);
                  }
                  const bool kb = (tl.kbits >> e) & 1u;
                  const float gk = half_hi(ek[e]);
                  // logits gamma S_A - m, plus the key-residual term for the lanes whose token has one
                  const float2 gk2 = make_float2(gk, gk);
#pragma unroll
                  for (int i2 = 0; i2 < NP; ++i2)
                    x[i2] = __ffma2_rn(gk2, make_float2(sa[2 * i2], GS >= 2 ? sa[2 * i2 + 1] : 0.f), negm2[i2]);
                  if (kb) {
                    float rs[GS];
                    load_row<GS>(rsb + rk * 8, rs);
#pragma unroll
                    for (int i2 = 0; i2 < NP; ++i2)
                      x[i2] = __fadd2_rn(x[i2], make_float2(rs[2 * i2], GS >= 2 ? rs[2 * i2 + 1] : 0.f));
                  }
                  rk += (int)kb;
                }
                if constexpr (TAIL) {
#pragma unroll
                  for (int i2 = 0; i2 < NP; ++i2) x[i2] = valid ? x[i2] : make_float2(-INFINITY, -INFINITY);
                }
                float2 pe[NP];
#pragma unroll
                for (int i2 = 0; i2 < NP; ++i2) {
                  pe[i2] = make_float2(exp2_approx(x[i2].x), GS >= 2 ? exp2_approx(x[i2].y) : 0.f);
                  l2[i2] = __fadd2_rn(l2[i2], pe[i2]);
                }
                const bool vb = (tl.vbits >> e) & 1u;
                if (vb) store_row<GS>(pv + rv * GS, pe);
                rv += (int)vb;
                // the run of `key` ends here when the slot changes (branch-free): the lane's first
                // run is kept as its head (it may continue the previous lane's); a later one started
                // and ended in this lane, so its slot is this lane's alone and is stored as it is
                const float2 gv2 = make_float2(gv, gv);
                if (e == 0) {
#pragma unroll
                  for (int i2 = 0; i2 < NP; ++i2) acc[i2] = __fmul2_rn(pe[i2], gv2);
                } else {
                  const uint32_t av = valid ? ev[e] & 0xFFFFu : last_key;
                  const bool chg = av != key;
                  if (e > 1 && chg && multi) store_row<GS>(W + (int)(key - lo) * GS, acc);
                  const float f_first = (chg && !multi) ? 1.f : 0.f, f_keep = chg ? 0.f : 1.f;
                  const float2 first2 = make_float2(f_first, f_first), keep2 = make_float2(f_keep, f_keep);
#pragma unroll
                  for (int i2 = 0; i2 < NP; ++i2) {
                    hs[i2] = __ffma2_rn(acc[i2], first2, hs[i2]);
                    acc[i2] = __ffma2_rn(pe[i2], gv2, __fmul2_rn(acc[i2], keep2));
                  }
                  multi |= chg;
                  key = av;
                }
              }
            };
            if (tv.n == T) token_loop(std::false_type{});
            else token_loop(std::true_type{});
            // merge across lanes: the next lane's head continues this lane's last run when their
            // slots match; a head that does not continue the previous lane's run is complete
            const uint32_t ptk = __shfl_up_sync(0xffffffffu, key, 1);
            const uint32_t nhk = __shfl_down_sync(0xffffffffu, hk, 1);
            const unsigned multis = __ballot_sync(0xffffffffu, multi);
            if (multis) {  // (warp-uniform)
              const bool nmulti = lane < 31 && ((multis >> (lane + 1)) & 1u);
              const float f_tn = (nmulti && nhk == key) ? 1.f : 0.f;
              const float2 tn2 = make_float2(f_tn, f_tn);
#pragma unroll
              for (int i2 = 0; i2 < NP; ++i2) {
                const float2 nh = make_float2(__shfl_down_sync(0xffffffffu, hs[i2].x, 1),
                                              __shfl_down_sync(0xffffffffu, hs[i2].y, 1));
                acc[i2] = __ffma2_rn(nh, tn2, acc[i2]);
              }
            }
            // the warp's first run may continue the previous warp's last one and its last run go on in the
            // next: both get rows of their own past the slots' (a shared-memory float addition is a
            // compare-and-swap loop, and would meet the neighbour's)
            float* w_ends = W + ((WIDE ? P.XW : P.X) + 2 * wi8) * GS;
            if (multi && !(lane > 0 && ptk == hk)) {
              if (lane == 0) vs[2 * wi8] = (int)(hk - lo);
              store_row<GS>(lane == 0 ? w_ends : W + (int)(hk - lo) * GS, hs);
            }
            // segmented inclusive scan of the last runs over lanes with equal slots
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
              const uint32_t kd = __shfl_up_sync(0xffffffffu, key, d);
              const float f_add = (lane >= d && kd == key) ? 1.f : 0.f;
              const float2 add2 = make_float2(f_add, f_add);
#pragma unroll
              for (int i2 = 0; i2 < NP; ++i2) {
                const float2 vd = make_float2(__shfl_up_sync(0xffffffffu, acc[i2].x, d),
                                              __shfl_up_sync(0xffffffffu, acc[i2].y, d));
                acc[i2] = __ffma2_rn(vd, add2, acc[i2]);
              }
            }
            const uint32_t nkey = __shfl_down_sync(0xffffffffu, key, 1);
            const uint32_t key0 = __shfl_sync(0xffffffffu, key, 0);
            if (lane == 31 || nkey != key) {  // the last lane of a segment holds its total
              // (a single run over the whole warp counts as its last)
              const bool first = !(multis & 1u) && key == key0, last = lane == 31;
              if (last) vs[2 * wi8 + 1] = (int)(key - lo);
              else if (first) vs[2 * wi8] = (int)(key - lo);
              store_row<GS>(last ? w_ends + GS : (first ? w_ends : W + (int)(key - lo) * GS), acc);
            }
          } else if (t0 < tv.n) {
            int* ovl_n = reinterpret_cast<int*>(smem + P.o_ovl + b * kOvlBytes);
            float* ovl = reinterpret_cast<float*>(ovl_n + 4);
            const auto ls = token_chunk_general<GS>(
                TokTile{tv, tv.gb(P.arena), mt.lo, WIDE ? mt.nw : mt.nrows, SAt, rows, qp, pv, W, ovf, P.arena + unit_desc(P.arena, u)->off_anchor_v,
                        ROPE ? P.lg + ((size_t)u * P.s_stride + (size_t)mt.j * T) * GS : nullptr, ovl_n, ovl, k, mt.nKs, mt.nVs, P.ka_stride,
                        CODEC}, tl);
#pragma unroll
            for (int i2 = 0; i2 < NP; ++i2) l2[i2] = __fadd2_rn(l2[i2], ls.v[i2]);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tdone(b));
      }
#pragma unroll
      for (int g = 0; g < GS; ++g) {
        const float sl = warp_sum((g & 1) ? l2[g >> 1].y : l2[g >> 1].x);
        if (lane == 0) gsum[wi8 * 8 + g] = sl;
      }
    } else {
      // ================================ products ==================================
      float accA[2][4] = {}, accR[2][4] = {};  // anchor-value and value-residual sums, dims 16 wi8 .. 16 wi8 + 15
      float pminv = 0.f;                       // sum of p min, head r8 (a quarter per c4)
      wait_or_fail(bar_hdr, (uint32_t)sigma & 1u);
      uint2 bq[NBF][8];  // the unit's key-residual B fragments
      float sqh[2];      // sums of q' of heads 2 c4, 2 c4 + 1
#pragma unroll
      for (int f = 0; f < NBF; ++f)
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) bq[f][ks] = qf[(f * 8 + ks) * 32 + lane];
      sqh[0] = sq[2 * c4];
      sqh[1] = sq[2 * c4 + 1];
      // ---- key residuals of tile t: q' . c of the staged key records, tensor cores; the terms
      // scale (q' . c) + min sum(q') are written over the records' codes; the tile's weight rows zeroed.
      // (Waits for the tile, unless `landed`.) ----
      auto key_phase = [&](int t, bool landed) {
        const int b = t & 1;
        const bool go = landed || wait_or_fail(bar_full(t % NSG), (uint32_t)(t / NSG) & 1u);
        if (go) {
          const Meta mt = meta[t % NSG];
          const uint8_t* st = ring + mt.ring_off;
          const TileView tv = tile_view(st, mt, u, S);
          const uint32_t codes_staged = tv.staged > tv.cd_k ? (tv.staged - tv.cd_k) / 32u : 0u;
          const int nKs = ROPE ? 0 : min(tv.nk, (int)codes_staged);  // their terms go over their own codes: no cap but staging
          if (wi8 == 0 && lane == 0) {
            const int nVs = min(tv.nv, P.R);
            const bool fast = (ROPE || nKs == tv.nk) && nVs == tv.nv &&
                              (int)(((reinterpret_cast<const uint32_t*>(st + 4 * tv.n64))[tv.n - 1] & 0xFFFFu) - mt.lo) < (int)(WIDE ? mt.nw : mt.nrows);
            Meta& w = meta[t % NSG];
            w.sm_v = tv.sm_v;
            w.cd_k = tv.cd_k;
            w.cd_v = tv.cd_v;
            w.sm_k = tv.sm_k;
            w.n = tv.n;
            w.nKs = nKs;
            w.nVs = nVs;
            w.fast = (fast ? 1u : 0u) | (tv.cd_v + 512u * (uint32_t)((nVs + 15) / 16) <= tv.staged ? 2u : 0u);
          }
          float* W = reinterpret_cast<float*>(smem + P.o_wb) + (t % 3) * ((WIDE ? P.XW : P.X) + kEnds) * GS;
          for (int e = 4 * mt_; e < ((WIDE ? P.XW : P.X) + kEnds) * GS; e += 4 * NMW * 32) *reinterpret_cast<float4*>(W + e) = make_float4(0.f, 0.f, 0.f, 0.f);
          if (mt_ < kEnds) reinterpret_cast<int*>(smem + P.o_vs)[(t % 3) * kEnds + mt_] = -1;
          if (mt_ < 2) reinterpret_cast<int*>(smem + P.o_ovl + b * kOvlBytes)[mt_] = 0;
          float* rsb = reinterpret_cast<float*>(const_cast<uint8_t*>(st) + tv.cd_k);
          for (int g16 = wi8; g16 * 16 < nKs; g16 += NMW) {
            uint32_t wd[2][8], smn[2];  // [record r8 / r8 + 8][16-dim step]; scale and min
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
              const int sl = g16 * 16 + r8 + 8 * hr;
              uint4 w0 = make_uint4(0u, 0u, 0u, 0u), w1 = w0;
              smn[hr] = 0u;
              if (sl < nKs) {
                w0 = *reinterpret_cast<const uint4*>(st + tv.cd_k + 32u * (uint32_t)sl);
                w1 = *reinterpret_cast<const uint4*>(st + tv.cd_k + 32u * (uint32_t)sl + 16u);
                smn[hr] = *reinterpret_cast<const uint32_t*>(st + tv.sm_k + 4u * (uint32_t)sl);
              }
              wd[hr][0] = w0.x; wd[hr][1] = w0.y; wd[hr][2] = w0.z; wd[hr][3] = w0.w;
              wd[hr][4] = w1.x; wd[hr][5] = w1.y; wd[hr][6] = w1.z; wd[hr][7] = w1.w;
            }
            float d[2][4] = {};
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              const uint32_t xa = wd[0][ks] >> (4 * c4), xb = wd[1][ks] >> (4 * c4);
              const uint4 a = make_uint4(code_pair_h2<CODEC>(xa), code_pair_h2<CODEC>(xb), code_pair_h2<CODEC>(xa >> 2),
                                         code_pair_h2<CODEC>(xb >> 2));
              if constexpr (GS == 8) {
                mma_f16(d[0], a, bq[0][ks].x, bq[0][ks].y);
                mma_f16(d[1], a, bq[NBF - 1][ks].x, bq[NBF - 1][ks].y);
              } else {
                mma_f16(d[ks & 1], a, bq[0][ks].x, bq[0][ks].y);
              }
            }
            __syncwarp();  // every lane has its codes before any term overwrites them
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              v[e] = d[0][e] + d[1][e];
              if constexpr (GS != 8) v[e] += __shfl_xor_sync(0xffffffffu, v[e], 2);
            }
            if (GS == 8 || c4 < 2) {
#pragma unroll
              for (int hr = 0; hr < 2; ++hr) {
                const int sl = g16 * 16 + r8 + 8 * hr;
                if (sl < nKs && 2 * c4 < GS) {  // (rows of eight floats; heads past GS are not read)
                  const float sc = half_lo(smn[hr]), mn = half_hi(smn[hr]);
                  *reinterpret_cast<float2*>(rsb + sl * 8 + 2 * c4) = make_float2(mn * sqh[0] + sc * v[2 * hr], mn * sqh[1] + sc * v[2 * hr + 1]);
                }
              }
            }
          }
        } else if (wi8 == 0 && lane == 0) {
          meta[t % NSG].fast = kNoShape;
          meta[t % NSG].n = 0;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_kdone(b));
      };
      if (n_seg > 0) key_phase(lt, false);
      for (int i = 0; i < n_seg; ++i, ++lt) {
        const int b = lt & 1;
        // the next tile's key terms first, if it is there, so that the token warps have work while this tile's
        // values are summed (else after them: its place may be this tile's)
        bool ahead = i + 1 >= n_seg;
        if (!ahead && !warp_failed(failed) &&
            __all_sync(0xffffffffu, mbar_test(bar_full((lt + 1) % NSG), (uint32_t)((lt + 1) / NSG) & 1u))) {
          key_phase(lt + 1, true);
          ahead = true;
        }
        const bool waited = wait_or_fail(bar_tdone(b), (uint32_t)(lt >> 1) & 1u);
        const Meta mt = meta[lt % NSG];
        const bool go = waited && !(mt.fast & kNoShape);
        const uint8_t* st = ring + mt.ring_off;
        float* W = reinterpret_cast<float*>(smem + P.o_wb) + (lt % 3) * ((WIDE ? P.XW : P.X) + kEnds) * GS;
        float* pv = reinterpret_cast<float*>(smem + P.o_pv) + b * P.R * GS;
        const int nVs = mt.nVs, nr = (int)mt.nrows, nb16 = (nr + 15) / 16;
        if (go) {
          if (!(mt.fast & 1u)) {  // the overflow lists: thread mt_ takes dimension mt_ % 128 of every entry of one list
            const TileView tv = tile_view(st, mt, u);
            const int* ovl_n = reinterpret_cast<const int*>(smem + P.o_ovl + b * kOvlBytes);
            const float* ovl = reinterpret_cast<const float*>(ovl_n + 4);
            const int dim = mt_ & 127;
            float av[GS];
#pragma unroll
            for (int g = 0; g < GS; ++g) av[g] = 0.f;
            if (mt_ < 128) {
              const int nv_o = min(ovl_n[0], kOvl);
              for (int e = 0; e < nv_o; ++e) {  // p (min + scale L(c)) of a value record, rotated domain
                const float* en = ovl + e * 9;
                const uint32_t r = (uint32_t)__float_as_int(en[0]);
                const uint32_t smn = *reinterpret_cast<const uint32_t*>(tv.at(P.arena, tv.sm_v + 4u * r));
                const uint32_t w = *reinterpret_cast<const uint32_t*>(tv.at(P.arena, tv.cd_v + 512u * (r / 16u) + 4u * value_code_word(dim)));
                const float val = fmaf(half_lo(smn), code_level((w >> value_code_bit((int)(r % 16u))) & 3u, CODEC), half_hi(smn));
#pragma unroll
                for (int g = 0; g < GS; ++g) av[g] = fmaf(en[1 + g], val, av[g]);
              }
              if (nv_o)
#pragma unroll
                for (int g = 0; g < GS; ++g) red_local(ovf + GS * 128 + g * 128 + dim, av[g]);
            } else {
              const int na_o = min(ovl_n[1], kOvl);
              for (int e = 0; e < na_o; ++e) {  // weight x the anchor's value row (global, swizzled by the slot)
                const float* en = ovl + (kOvl + e) * 9;
                const int kk = __float_as_int(en[0]);
                const uint8_t* row = P.arena + unit_desc(P.arena, u)->off_anchor_v + (size_t)kk * 256;
                const float x = __bfloat162float(
                    *reinterpret_cast<const __nv_bfloat16*>(row + 16 * ((dim >> 3) ^ (kk & 7)) + 2 * (dim & 7)));
#pragma unroll
                for (int g = 0; g < GS; ++g) av[g] = fmaf(en[1 + g], x, av[g]);
              }
              if (na_o)
#pragma unroll
                for (int g = 0; g < GS; ++g) red_local(ovf + g * 128 + dim, av[g]);
            }
          }
          // ---- operands of the value side, each built once by one warp, over the numbers it is made of, as the
          // mma A fragments (lane 4 g + c4: k places 2 c4, 2 c4 + 1, then those + 8; bf16 high part, then
          // low part): p scale of 16 value records (with the sum of p min per head), or 16 slots' weights ----
          const int n_vg = (nVs + 15) / 16;
          for (int x = wi8; x < n_vg + nb16 + 1; x += NMW) {
            const bool val = x < n_vg;
            const int blk = x - n_vg;  // block of slots; the last one: the token warps' first and last runs
            float* src = val ? pv + 16 * GS * x : (blk < nb16 ? W + 16 * GS * blk : W + (WIDE ? P.XW : P.X) * GS);
            const int lim = val ? nVs - 16 * x : (blk < nb16 ? nr - 16 * blk : kEnds);
            const int kk[4] = {2 * c4, 2 * c4 + 1, 2 * c4 + 8, 2 * c4 + 9};
            float f[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) f[e] = kk[e] < lim && r8 < GS ? src[kk[e] * GS + r8] : 0.f;
            if (val) {
              uint32_t smn[4];
              const uint32_t so = mt.sm_v + 64u * (uint32_t)x;  // (padded to 16 bytes: pairs may be read together)
              if (mt.fast & 2u) {
#pragma unroll
                for (int e = 0; e < 4; ++e) smn[e] = kk[e] < lim ? *reinterpret_cast<const uint32_t*>(st + so + 4u * (uint32_t)kk[e]) : 0u;
              } else {
                const TileView tv = tile_view(st, mt, u);
#pragma unroll
                for (int e = 0; e < 4; ++e) smn[e] = kk[e] < lim ? *reinterpret_cast<const uint32_t*>(tv.at(P.arena, so + 4u * (uint32_t)kk[e])) : 0u;
              }
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                pminv = fmaf(f[e], half_hi(smn[e]), pminv);
                f[e] *= half_lo(smn[e]);
              }
            }
            __nv_bfloat16 hi[4], lo_[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) split_b(f[e], hi[e], lo_[e]);
            __syncwarp();  // everything is read before it is overwritten
            if (r8 < GS)
              *reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(src) + 16 * lane) =
                  make_uint4(pack_b2(hi[0], hi[1]), pack_b2(lo_[0], lo_[1]), pack_b2(hi[2], hi[3]), pack_b2(lo_[2], lo_[3]));
          }
        }
        prod_sync();  // every operand is built
        if (go) {
          // ---- anchor values: w^T V_A over the tile's staged slots, then over the token warps' first and last
          // runs, whose rows are picked by their slots ----
          const uint8_t* Vr = st + mt.staged;
          const int mi = lane >> 3, ri = lane & 7;
          const int* vs = reinterpret_cast<const int*>(smem + P.o_vs) + (lt % 3) * kEnds;
          for (int blk = 0; blk <= nb16; ++blk) {
            const bool ends = blk == nb16;
            const int ka = (ends ? 0 : 16 * blk) + 2 * c4;
            const uint4 a = r8 < GS ? *reinterpret_cast<const uint4*>(reinterpret_cast<const uint8_t*>(ends ? W + (WIDE ? P.XW : P.X) * GS : W + 16 * GS * blk) + 16 * lane)
                                    : make_uint4(0u, 0u, 0u, 0u);
            // rows past the staged slots, or of runs that are not there, hold other bytes: their halves of B are cleared
            uint32_t m0, m1;
            int slot;
            if (ends) {
              const int2 v0 = *reinterpret_cast<const int2*>(vs + ka), v1 = *reinterpret_cast<const int2*>(vs + ka + 8);
              m0 = (v0.x >= 0 ? 0xFFFFu : 0u) | (v0.y >= 0 ? 0xFFFF0000u : 0u);
              m1 = (v1.x >= 0 ? 0xFFFFu : 0u) | (v1.y >= 0 ? 0xFFFF0000u : 0u);
              slot = max(vs[(mi & 1) * 8 + ri], 0);
              if constexpr (WIDE) {  // (those past the staged rows are taken below)
                m0 &= (v0.x < nr ? 0xFFFFu : 0u) | (v0.y < nr ? 0xFFFF0000u : 0u);
                m1 &= (v1.x < nr ? 0xFFFFu : 0u) | (v1.y < nr ? 0xFFFF0000u : 0u);
                slot = min(slot, nr - 1);
              }
            } else {
              m0 = (ka < nr ? 0xFFFFu : 0u) | (ka + 1 < nr ? 0xFFFF0000u : 0u);
              m1 = (ka + 8 < nr ? 0xFFFFu : 0u) | (ka + 9 < nr ? 0xFFFF0000u : 0u);
              slot = 16 * blk + (mi & 1) * 8 + ri;
            }
            const int cc = (2 * wi8 + (mi >> 1)) ^ (int)((mt.lo + (uint32_t)slot) & 7u);
            uint32_t b00, b01, b10, b11;
            ldsm_x4_trans(smem_u32(Vr + slot * 256 + 16 * cc), b00, b01, b10, b11);
            mma_bf16(accA[0], a.x, a.y, a.z, a.w, b00 & m0, b01 & m1);
            mma_bf16(accA[1], a.x, a.y, a.z, a.w, b10 & m0, b11 & m1);
          }
          // ---- value residuals: (p scale) c over the staged records, in the rotated domain;
          // this lane's two code words hold dimensions 16 wi8 + 8 nb + r8 of 16 records ----
          const uint32_t woff = mt.cd_v + 4u * (uint32_t)(32 * (wi8 >> 1) + 4 * r8 + 2 * (wi8 & 1));
          auto residual = [&](int g16, const uint2 w2) {
            const uint4 a = r8 < GS ? *reinterpret_cast<const uint4*>(reinterpret_cast<const uint8_t*>(pv) + g16 * 64 * GS + lane * 16)
                                    : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t wd[2] = {w2.x, w2.y};
#pragma unroll
            for (int nb = 0; nb < 2; ++nb) {
              // records 2c, 2c+1 at bits 2c and 2c + 16, records 2c+8, 2c+9 eight bits higher
              const uint32_t x = wd[nb] >> (2 * c4);
              const uint2 b = code_pairs_b2<CODEC>(x);
              mma_bf16(accR[nb], a.x, a.y, a.z, a.w, b.x, b.y);
            }
          };
          if (mt.fast & 2u) {
#pragma unroll 4
            for (int g16 = 0; g16 * 16 < nVs; ++g16) residual(g16, *reinterpret_cast<const uint2*>(st + woff + 512u * (uint32_t)g16));
          } else {
            const TileView tv = tile_view(st, mt, u);
            for (int g16 = 0; g16 * 16 < nVs; ++g16)
              residual(g16, *reinterpret_cast<const uint2*>(tv.at(P.arena, woff + 512u * (uint32_t)g16)));
          }
          if constexpr (WIDE) {
            if (mt.nw > mt.nrows)
              unstaged_rows<GS>(W, reinterpret_cast<const uint32_t*>(W + (WIDE ? P.XW : P.X) * GS), vs,
                                P.arena + unit_desc(P.arena, u)->off_anchor_v + (size_t)mt.lo * 256, mt.lo, nr, (int)mt.nw, mt_, ovf);
          }
        }
        // (the key terms were written over the tile's bytes: ordered before the copy that takes their place, which goes
        // through the asynchronous proxy)
        if constexpr (!ROPE) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_empty(lt % NSG));  // this warp is done with the tile
        if (!ahead) key_phase(lt + 1, false);
      }
      prod_sync();  // every warp is done with the header, where the segment's sums go
      static_assert(2 * GS * 512 <= hdr_bytes(GS), "a segment's sums fit its header's place");
      if (r8 < GS) {
#pragma unroll
        for (int nb = 0; nb < 2; ++nb) {
          const int col = 16 * wi8 + 8 * nb + 2 * c4;
          *reinterpret_cast<float2*>(qp + r8 * 128 + col) = make_float2(accA[nb][0] + accA[nb][2], accA[nb][1] + accA[nb][3]);
          *reinterpret_cast<float2*>(qp + (GS + r8) * 128 + col) = make_float2(accR[nb][0] + accR[nb][2], accR[nb][1] + accR[nb][3]);
        }
      }
      pminv += __shfl_xor_sync(0xffffffffu, pminv, 1);
      pminv += __shfl_xor_sync(0xffffffffu, pminv, 2);
      if (c4 == 0) gsum[64 + wi8 * 8 + r8] = pminv;
    }

    // ---- the segment's end: a token warp per query head turns the sums into the CTA's slot of the unit (the
    // value-residual part gets its sum of p min and the inverse rotation s o H(.) / 128, once per head and CTA;
    // the anchor-value part and the overflow's sums are added), counts it in on the head's counter, and
    // combines the head if that completes it ----
    all_sync();
    const bool has_next = sg->t0 + sg->je < B1;
    if (tok) {
      if (TURN ? lane == 0 && mine < n_cta_tiles : tid == 0) copy_more();
      const int first = sg->first, nseg = sg->nseg;
      float* dst = P.part + (size_t)(c + u) * PF;
      auto warp_sums = [&](int off, int g) {
        float v = 0.f;
#pragma unroll
        for (int x = 0; x < 8; ++x) v += gsum[off + x * 8 + g];
        return v;
      };
      static_assert(GS <= NTW, "a warp per query head");
      const int h = wi8;
      if (h < GS) {
        float4* oa = reinterpret_cast<float4*>(ovf + h * 128 + 4 * lane);
        float4* orr = reinterpret_cast<float4*>(ovf + GS * 128 + h * 128 + 4 * lane);
        const float4 a = *reinterpret_cast<const float4*>(qp + h * 128 + 4 * lane);
        const float4 r = *reinterpret_cast<const float4*>(qp + (GS + h) * 128 + 4 * lane);
        const float4 oav = *oa, orv = *orr;
        const float pm = warp_sums(64, h);
        float x[4] = {r.x + orv.x + pm, r.y + orv.y + pm, r.z + orv.z + pm, r.w + orv.w + pm};
        if (P.rotate) {
          warp_wht128(x, lane);
          apply_signs(x, lane, P.sign_lo, P.sign_hi);
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] *= (1.0f / 128.0f);
        }
        *reinterpret_cast<float4*>(dst + h * 128 + 4 * lane) =
            make_float4(a.x + oav.x + x[0], a.y + oav.y + x[1], a.z + oav.z + x[2], a.w + oav.w + x[3]);
        if (lane == 0) dst[part_l(GS) + h] = *failed ? __int_as_float(0x7FC00000) : warp_sums(0, h);
        *oa = make_float4(0.f, 0.f, 0.f, 0.f);
        *orr = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      const float m = rows[24 + (h & 7)];
      tok_sync();  // the sums are read
      if (tid == 0 && has_next) start_unit(u + 1);
      if (h < GS) {
        bool last = true;  // (a unit of one CTA: nothing to count)
        if (nseg > 1) {
          unsigned old = 0;
          if (lane == 0) {
            __threadfence();
            old = atomicAdd(unit_counters(P.uh, P.uh_stride, u, GS) + h, 1u);
          }
          last = __shfl_sync(0xffffffffu, old, 0) == (unsigned)(nseg - 1);
          if (last) __threadfence();
        }
        if (last) combine_head<GS>(P, u, first, nseg, h, m);
      }
    }
    if (!has_next) break;
    all_sync();
    if (tid == 0) {
      Seg s = *sg;
      seg_next(s);
      *sg = s;
    }
    all_sync();
  }
  // every copy has landed before the CTA may exit (bounded; they all have unless a wait ran out)
  if (tid == 0) {
    for (int t = max(0, pr->ii - NSG); t < pr->ii; ++t)
      if (!(meta[t % NSG].nrows >> 31)) mbar_wait(bar_full(t % NSG), (uint32_t)(t / NSG) & 1u);
    mbar_wait(bar_hdr, (uint32_t)sigma & 1u);
    mbar_wait(bar_sa_full, (uint32_t)sigma & 1u);
  }
}

struct DeviceInfo {
  int sms = 0;
  int smem_optin = 0;
};

DeviceInfo device_info() {
  static std::mutex mu;
  static DeviceInfo cache[64];
  static bool have[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  if (dev >= 0 && dev < 64 && have[dev]) return cache[dev];
  DeviceInfo d;
  cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&d.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (dev >= 0 && dev < 64) {
    cache[dev] = d;
    have[dev] = true;
  }
  return d;
}

size_t align128(size_t x) { return (x + 127) & ~(size_t)127; }

double max_density(const Layout& L) {
  double dens = 0.0;
  for (const auto& s : L.shape) dens = std::max(dens, (double)std::max(s.nk, s.nv) / (double)s.S);
  return dens;
}
double max_anchor_density(const Layout& L) {
  double dens = 0.0;
  for (const auto& s : L.shape) dens = std::max(dens, (double)s.k / (double)s.S);
  return dens;
}

double mean_density(const Layout& L) {
  double n = 0.0, t = 0.0;
  for (const auto& s : L.shape) {
    n += (double)std::max(s.nk, s.nv);
    t += (double)s.S;
  }
  return n / t;
}

// Value records per tile with p rows at least: 1.35x the densest unit's mean plus slack; records of a
// denser tile beyond the plan's count take the CUDA-core paths, which cost far more.  An encoder's tiles
// are uneven (tokens of a cluster lie together and their residuals are alike), so a plan takes as many
// more as shared memory has room for: a 32K layer of 656 anchors whose densest tile held more than 1.35x the mean
// plus slack took 42 us with that count and 19 us with all its records staged.
int full_r(const Layout& L) {
  const int R = (int)(T * max_density(L) * 1.35) + 32;
  return std::max(16, (R + 15) & ~15);
}
// Weight rows of a tile wanted: 2x the mean number of value slots it covers plus slack; runs on slots beyond a plan's
// take a CUDA-core path.
int full_w(const Layout& L) {
  const int X = (int)(2.0 * (T * max_anchor_density(L) + 1.0)) + 16;
  return std::min(T, std::max(16, (X + 15) & ~15));
}
// Anchor-value rows staged per tile: those slots', at most 256; the rest are read from global memory.
int full_x(const Layout& L) { return std::min(256, full_w(L)); }
// bytes of a full tile's block with r records per side, at most
long long block_bytes_at_most(int r) { return (long long)F_MAX + 2 * round16(4u * (uint32_t)r) + 64LL * r; }

struct Plan {
  DecodeParams P;
  bool turn = false;  // the token warps copy in turn
  size_t smem = 0;
  int grid = 0;
};

// Shared-memory carve-up for X staged anchor-value rows of XW weight rows, the table in shared memory or not, a ring of at
// least `ring_min` bytes that holds a block of Rmin records per side beside its anchor-value rows, and as many p rows as fit
// beside it, at least Rmin; false if they don't.
bool make_plan_rx(const Layout& L, int GS, int Rmin, int X, int XW, int smem_sa, int smem_optin, long long ring_min, Plan* out) {
  DecodeParams& P = out->P;
  P.X = X;
  P.XW = XW;
  P.ka_stride = (L.max_k + 3) & ~3;
  P.smem_sa = smem_sa;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align128(off + bytes);
    return (int)o;
  };
  P.o_bar = take((2 * NSG + 6) * 8);
  P.o_meta = take(NSG * sizeof(Meta));
  P.o_misc = take(16 + sizeof(Seg));  // failure flag; the segment in work
  P.o_sa = take(smem_sa == 1 ? (size_t)P.ka_stride * GS * 4 : (smem_sa == 2 ? (size_t)P.ka_stride * 16 : 0));
  P.o_ovf = take((size_t)2 * GS * 128 * 4);
  P.o_qp = take((size_t)hdr_bytes(GS));  // the unit's query header: q', its sums, B fragments
  P.o_rows = take(32 * 4);
  P.o_gsum = take(2 * 8 * 8 * 4);
  // three tiles' weights of their slots and of the warps' first and last runs, and the slots of those; two tiles'
  // p rows (then A operands) and overflow lists
  P.o_wb = take((size_t)3 * (XW + kEnds) * GS * 4);
  P.o_vs = take((size_t)3 * kEnds * 4);
  P.o_ovl = take((size_t)2 * kOvlBytes);
  P.o_prod = take((GS <= kTurnGroup ? NTW : 1) * sizeof(Prod));
  const long long room = (long long)smem_optin - (long long)off - kRingSlack - 128;
  const long long fit = (room - ring_min) / (2 * GS * 4) & ~15LL;
  if (fit < Rmin) return false;
  P.R = (int)std::min<long long>(fit, T);
  P.o_pv = take((size_t)2 * P.R * GS * 4);
  P.o_ring = (int)off;
  P.ring_bytes = (int)(((long long)smem_optin - (long long)off - kRingSlack) & ~127LL);
  // staged bytes of a tile block at most: all of one with R records per side, as far as the ring holds it
  // beside its anchor-value rows
  P.cap = (int)std::min<long long>(block_bytes_at_most(P.R), (P.ring_bytes - 256LL * X) & ~15LL);
  if (P.cap < block_bytes_at_most(Rmin)) return false;
  out->smem = (size_t)P.o_ring + (size_t)P.ring_bytes + kRingSlack;
  return true;
}

// Preference: the anchor-score table in shared memory (the token gathers' fast path), with a ring of five mean tiles
// (one in each role, two landing, and what wrapping around leaves unused) and p rows for tiles half again as dense as
// the R they need, then less, the least p rows and anchor-value rows trimmed towards 3/4 of their values with it; then
// the table in global memory (gathers through L1 and L2) the same way; then a ring of one such tile with ever fewer
// anchor-value rows staged; then anything that holds one tile.  4 requests
// of 131072, 8B shape, us per call with rings of 4.5, 3.5, 2.5 mean tiles alone and with these: 2 % anchors and 20 %
// residuals 115.3 -> 114.5, 4 % and 10 % 107.1 -> 105.4, 4 % and 20 % 135.1 -> 126.9; six ragged requests with 20 %
// residuals 80.0 -> 77.4.  Every choice but the last keeps the records of a mean tile, and some more, on the tensor-core paths
// (16 units of 60000 tokens, 2 % anchors and 35, 50, 90 % residuals, G = 8: 52, 64, 95 us; with p rows for 320 records at
// most 10283, 8568, 39697; 12 % and 10 %, G = 4, where the ring was too short for a mean tile's records: 533 -> 52).
// Where the slots of tiles near the mean (15 % and 16 over it: fa above 0.2) are more than the rows staged at most, tiles
// have more weight rows than those, 2x the mean (the WIDE kernels, table in global memory): 16 x 60000 tokens, 25 % anchors,
// G = 1, 2, 4, 8: 59, 62, 65, 77 us per
// call; with such tiles on the general token path 97, 147, 241, 428.  30 %: 81, 84, 88, 116 (1809, 3487, 5965, 11632).
// Half the table in shared memory (G = 8) where it does not fit and records are many, if the ring still holds two mean
// tiles: 4 requests of 131072, 8 KV heads, 4 % anchors, all in global memory and this: 20 % residuals 182.7, 171.9 us, 30 %
// 203, 193; with fewer records the ring's length is worth more: 10 % 136, 142, 5 % even; with a ring of 1.5 tiles (2
// requests, 5 % and 20 %) 99.9, 105.4.
// table false: no anchor-score table is read (RoPE at decode), so none is placed in shared memory.
bool make_plan(const Layout& L, int GS, int smem_optin, bool table, Plan* out, std::string* why) {
  const int R0 = full_r(L), X0 = full_x(L);
  const bool wide = 1.15 * (T * max_anchor_density(L) + 1.0) + 16.0 > 256.0;
  const int Rmin = std::min(T, std::max(16, ((R0 * 3 / 4) + 15) & ~15)), Xmin = std::max(16, ((X0 * 3 / 4) + 15) & ~15);
  const double rows = std::min(256.0, T * max_anchor_density(L) + 2.0);
  const double mean = (double)F_MAX + T * mean_density(L) * 72.0 + 256.0 + 256.0 * rows;
  for (const int sa : {1, 2, 0}) {
    if (sa && (!table || wide || (sa == 2 && GS != 8))) continue;
    for (const double tiles : {5.0, 4.5, 4.0, 3.5, 3.0, 2.5, 2.0, 1.5}) {
      if (sa == 2 && (tiles < 2.0 || mean_density(L) < 0.15)) break;
      const bool trim = tiles < 4.0;
      const int R = trim ? Rmin : std::min(T, tiles > 4.5 ? R0 * 3 / 2 : R0);
      for (int X = X0; X >= (trim ? Xmin : X0); X -= 16)
        if (make_plan_rx(L, GS, R, X, wide ? full_w(L) : X, sa, smem_optin, (long long)(tiles * mean), out)) return true;
    }
  }
  for (int X = X0; X >= 16; X -= 16)
    if (make_plan_rx(L, GS, Rmin, X, wide ? full_w(L) : X, 0, smem_optin, block_bytes_at_most(Rmin) + 256LL * X, out)) return true;
  for (int X = X0; X >= 16; X -= 16)
    if (make_plan_rx(L, GS, 16, X, X, 0, smem_optin, block_bytes_at_most(16) + 256LL * X, out)) return true;
  *why = "shared memory: no room for the decode pipeline";
  return false;
}

using ScoreFn = void (*)(const ScoreParams);
using RopeFn = void (*)(const RopeParams);
template <int GS, int MODE>
const void* decode_kernel_c(int codec) {
  return codec ? (const void*)akv_decode_kernel<GS, 1, MODE> : (const void*)akv_decode_kernel<GS, 0, MODE>;
}
template <int GS>
const void* decode_kernel(int codec, int rope, const Plan& pl) {
  const DecodeParams& P = pl.P;
  if constexpr (GS <= kTurnGroup)
    if (pl.turn) return codec ? (const void*)akv_decode_kernel<GS, 1, kTableSmem, false, true> : (const void*)akv_decode_kernel<GS, 0, kTableSmem, false, true>;
  if (P.XW > P.X) return wide_decode_kernel<GS>(codec, rope);
  if (rope) return decode_kernel_c<GS, kRope>(codec);
  if constexpr (GS == 8)
    if (P.smem_sa == 2) return decode_kernel_c<GS, kTableHalf>(codec);
  return P.smem_sa ? decode_kernel_c<GS, kTableSmem>(codec) : decode_kernel_c<GS, kTableGlobal>(codec);
}
template <int GS>
RopeFn rope_kernel(int codec) {
  return codec ? akv_rope_logits_kernel<GS, 1> : akv_rope_logits_kernel<GS, 0>;
}
template <int GS>
ScoreFn suffix_kernel(bool rope) {
  return rope ? akv_suffix_kernel<GS, true> : akv_suffix_kernel<GS, false>;
}

// Launch configuration per (device, G, layout shape): computed once, then reused, so that a
// call made during CUDA-graph capture only issues the launches.
struct LaunchKey {
  int dev, G, codec, rope, units, max_len, max_k, ctas;
  long long dens_key, adens_key, mdens_key, ttot;
  std::vector<int32_t> tiles;  // per unit: the CTAs' ranges depend on the order of the lengths
  bool operator<(const LaunchKey& o) const {
    return std::tie(dev, G, codec, rope, units, max_len, max_k, ctas, dens_key, adens_key, mdens_key, ttot, tiles) <
           std::tie(o.dev, o.G, o.codec, o.rope, o.units, o.max_len, o.max_k, o.ctas, o.dens_key, o.adens_key, o.mdens_key, o.ttot, o.tiles);
  }
};

}  // namespace

template <int GS>
int launch_g(const Layout& L, const akv_params& p, const void* arena, size_t arena_bytes, const void* q, void* out, float* out_f32,
             float sm_scale, const DecodeSuffix& sfx, void* ws, void* stream, std::string* why) {
  static std::mutex mu;
  static std::map<LaunchKey, Plan> cache;
  const int units = (int)L.shape.size();
  int dev = 0;
  cudaGetDevice(&dev);
  long long ttot = 0;
  std::vector<int32_t> tiles;
  tiles.reserve(L.shape.size());
  for (const auto& s : L.shape) {
    ttot += s.nt;
    tiles.push_back(s.nt);
  }
  // testing controls (akv_decode_set_debug): a requested number of CTAs, and the failure-detection
  // hook with which every CTA withholds the last tile of its range, so the waits on it run out
  // after their bound and the outputs of its units become NaN
  const int ctas = g_debug_cluster.load(std::memory_order_relaxed);
  const int drop = g_debug_withhold.load(std::memory_order_relaxed);
  const int codec = (p.flags & AKV_FLAG_LLOYD) ? 1 : 0;
  const int rope = (p.flags & AKV_FLAG_ROPE) ? 1 : 0;
  const LaunchKey key{dev, L.G, codec, rope, units, L.max_len, L.max_k, ctas, (long long)(max_density(L) * 1e6),
                      (long long)(max_anchor_density(L) * 1e6), (long long)(mean_density(L) * 1e6), ttot, std::move(tiles)};
  Plan pl;
  bool have = false;
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(key);
    if (it != cache.end()) {
      pl = it->second;
      have = true;
    }
  }
  if (!have) {
    const DeviceInfo di = device_info();
    if (!make_plan(L, GS, di.smem_optin, !rope, &pl, why)) return -1;
    int grid = (int)std::min<long long>(std::min(di.sms, kMaxGrid), ttot);
    if (ctas > 0) grid = (int)std::min<long long>(ctas, ttot);
    pl.grid = grid;
    pl.turn = GS <= kTurnGroup && !rope && max_density(L) == 0.0 && pl.P.smem_sa == 1 && pl.P.XW == pl.P.X && ttot >= (long long)kTurnTiles * grid;
    const cudaError_t e =
        cudaFuncSetAttribute(decode_kernel<GS>(codec, rope, pl), cudaFuncAttributeMaxDynamicSharedMemorySize, di.smem_optin);
    if (e != cudaSuccess) return (int)e;
    // first unit and tile of every CTA's range
    long long t0 = 0;
    int u = 0;
    for (int c = 0; c < grid; ++c) {
      const long long b = (long long)c * ttot / grid;
      while (t0 + L.shape[u].nt <= b) t0 += L.shape[u++].nt;
      pl.P.cta_unit[c] = u;
      pl.P.cta_tile[c] = (int)(b - t0);
    }
    pl.P.ttot = ttot;
    pl.P.grid = grid;
    // chunk maxima per unit: of 64 anchors, or with RoPE of 64 stored tokens
    pl.P.n_ch = rope ? (L.max_len + 63) / 64 : (L.max_k + CHA - 1) / CHA;
    std::lock_guard<std::mutex> lk(mu);
    if (cache.size() >= 64) cache.clear();  // (bounded: a server's calls come in many combinations of lengths)
    cache[key] = pl;
  }
  const DecodeWs W = decode_ws_layout(L, sfx.cap);
  const int n_sch = sfx.K ? (sfx.cap + SCH - 1) / SCH : 0;
  uint8_t* wsb = (uint8_t*)ws;
  DecodeParams& P = pl.P;
  P.arena = (const uint8_t*)arena;
  P.out = (__nv_bfloat16*)out;
  P.out_f32 = out_f32;
  P.sa = (const float*)(wsb + W.o_sa);
  P.cmax = (const float*)(wsb + W.o_cmax);
  P.part = (float*)(wsb + W.o_part);
  P.uh = wsb + W.o_uh;
  P.uh_stride = (hdr_bytes(GS) + 255) & ~255;
  P.n_kv_heads = p.n_kv_heads;
  P.n_q_heads = p.n_q_heads;
  P.rotate = (p.flags & AKV_FLAG_ROTATE) ? 1 : 0;
  P.scale_log2 = sm_scale * kLog2e;
  P.sign_lo = L.header.sign_bits[0];
  P.sign_hi = L.header.sign_bits[1];
  P.drop_last = drop;
  P.lg = rope ? (const float*)(wsb + W.o_lg) : nullptr;
  P.s_stride = (L.max_len + 63) & ~63;
  P.suf_part = n_sch ? (const float*)(wsb + W.o_suf) : nullptr;
  P.suf_len = sfx.len;
  P.suf_cap = sfx.cap;
  P.n_sch = n_sch;

  ScoreParams S;
  S.arena = P.arena;
  S.q = (const __nv_bfloat16*)q;
  S.sa = (float*)(wsb + W.o_sa);
  S.cmax = (float*)(wsb + W.o_cmax);
  S.n_kv_heads = p.n_kv_heads;
  S.n_q_heads = p.n_q_heads;
  S.ksuf = (const __nv_bfloat16*)sfx.K;
  S.vsuf = (const __nv_bfloat16*)sfx.V;
  S.suf_len = sfx.len;
  S.suf_part = (float*)(wsb + W.o_suf);
  S.suf_cap = sfx.cap;
  S.n_sch = n_sch;
  S.ka_stride = P.ka_stride;
  S.n_ch = P.n_ch;
  S.scale_log2 = P.scale_log2;
  S.uh = wsb + W.o_uh;
  S.uh_stride = P.uh_stride;
  S.rotate = P.rotate;
  S.sign_lo = P.sign_lo;
  S.sign_hi = P.sign_hi;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(units * P.n_ch), 1, 1);
  cfg.blockDim = dim3(128, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = (cudaStream_t)stream;
  void *ev_scores_p = nullptr, *ev_decode_p = nullptr;
  get_decode_events(&ev_scores_p, &ev_decode_p);
  const cudaEvent_t ev_scores = (cudaEvent_t)ev_scores_p, ev_decode = (cudaEvent_t)ev_decode_p;
  cudaError_t e;
  if (rope) {  // the logits of every stored token (no anchor scores)
    RopeParams R;
    R.arena = P.arena;
    R.q = S.q;
    R.lg = (float*)(wsb + W.o_lg);
    R.cmax = (float*)(wsb + W.o_cmax);
    R.uh = P.uh;
    R.uh_stride = P.uh_stride;
    R.n_kv_heads = p.n_kv_heads;
    R.n_q_heads = p.n_q_heads;
    R.rotate = P.rotate;
    R.s_stride = P.s_stride;
    R.n_tch = P.n_ch;
    R.scale_log2 = P.scale_log2;
    R.sign_lo = P.sign_lo;
    R.sign_hi = P.sign_hi;
    // theta_j / (2 pi) < 1 as a 64-bit binary fraction of a turn (truncated past 2^-64)
    for (int j = 0; j < 64; ++j)
      R.turn[j] = (unsigned long long)std::ldexp(
          std::pow((double)p.rope_theta, -2.0 * (double)j / 128.0) / 6.283185307179586476925, 64);
    cfg.gridDim = dim3((unsigned)(units * ((P.n_ch + kRopeWarps - 1) / kRopeWarps)), 1, 1);
    cfg.blockDim = dim3(kRopeWarps * 32, 1, 1);
    e = cudaLaunchKernelEx(&cfg, rope_kernel<GS>(codec), R);
    cfg.blockDim = dim3(128, 1, 1);
    for (int j = 0; j < 64; ++j) S.turn[j] = R.turn[j];
  } else {
    S.units = units;
    S.arena_rows = (long long)(arena_bytes / 256);
    cfg.gridDim = dim3((unsigned)(units + units * P.n_ch), 1, 1);
    e = cudaLaunchKernelEx(&cfg, akv_scores_kernel<GS>, S);
  }
  // the launches after the first may start beside the one before them and wait for it where they need it
  cudaLaunchAttribute pdl;
  pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &pdl;
  cfg.numAttrs = 1;
  if (e == cudaSuccess && n_sch) {  // the dense suffix's chunks (with RoPE: keys turned to positions S + t)
    cfg.gridDim = dim3((unsigned)(units * n_sch), 1, 1);
    cfg.dynamicSmemBytes = (size_t)SCH * 256;  // a chunk's value rows
    e = cudaLaunchKernelEx(&cfg, suffix_kernel<GS>(rope != 0), S);
    cfg.dynamicSmemBytes = 0;
  }
  if (e != cudaSuccess) return (int)e;
  if (ev_scores && (e = cudaEventRecord(ev_scores, cfg.stream)) != cudaSuccess) return (int)e;
  cfg.gridDim = dim3((unsigned)pl.grid, 1, 1);
  cfg.blockDim = dim3(NT, 1, 1);
  cfg.dynamicSmemBytes = pl.smem;
  void* args[] = {&P};
  e = cudaLaunchKernelExC(&cfg, decode_kernel<GS>(codec, rope, pl), args);
  if (e != cudaSuccess) {
    cudaFuncAttributes fa{};
    cudaFuncGetAttributes(&fa, decode_kernel<GS>(codec, rope, pl));
    *why = "(decode kernel: " + std::to_string(fa.numRegs) + " registers, max " + std::to_string(fa.maxThreadsPerBlock) +
           " threads, " + std::to_string(pl.smem) + " B dynamic shared memory of " +
           std::to_string(fa.maxDynamicSharedSizeBytes) + ", grid " + std::to_string(pl.grid) + ")";
    return (int)e;
  }
  if (ev_decode && (e = cudaEventRecord(ev_decode, cfg.stream)) != cudaSuccess) return (int)e;
  return (int)cudaGetLastError();
}

}  // namespace akv
