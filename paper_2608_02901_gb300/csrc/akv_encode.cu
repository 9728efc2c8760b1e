// GPU encoder of the AnchorKV compressed cache (Algorithm 1 with the anchor and slot rules of this build; the paper's
// full selection).  Every decision (assignment, gamma, residual energy ranking, rotation, codes) is the one that IEEE
// fp64 with a fixed operation order takes, so the packed bytes are reproducible bit for bit.  That arithmetic is done
// only where it decides: this GPU's fp64 unit takes a warp instruction per 64 cycles and scheduler, so each step is
// first taken on tensor cores, in fp32 or in pairs of fp32, with a bound of its error, and what the bound leaves open
// (about 1 % of positions and records) is repeated in fp64.  8 units of 32768 tokens: 82.9 ms with fp64 throughout,
// 0.40 ms.  Compiled with --fmad=false; where a fused multiply-add is used explicitly in fp64 its product is exact, so
// rounding once or twice gives the same result.
//
// Kernels, in launch order, each over all units of the batch:
//   enc_anchors    select the k - W smallest hashes, number anchor slots by position
//   enc_rows       copy anchor rows into the arena (16-byte chunks swizzled), squared norms
//   enc_assign_tc  Eq. 1: the one or two anchors that can be a position's nearest, on tensor cores
//   enc_finish     Eq. 2 gamma, residual energies (per position), as far as fp32 decides them
//   enc_undecided  the rest, in paired fp32 and fp64
//   enc_slots      top-N residual energies per side -> residual flags and slot list
//   enc_slots_exact the same from fp64 energies, where the fp32 ones cannot rank (else empty)
//   enc_order      stored order: stable counting sort of positions by value anchor slot
//   enc_tile_count residual records per tile and side
//   enc_tile_table tile block offsets
//   enc_tile_fill  streams, bitmaps and rank words of every tile block
//   enc_quant      Eq. 12 rotation and 2-bit quantization of every slot, into its tile
// The full selection adds the observation rows' attention and the scores before them (enc_obs_*_f, enc_score_*) and
// the utilities and pools in enc_slots' place (enc_util_f, enc_pool_f), each followed by its exact form, which runs
// only for units whose ranking the errors leave open.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "akv_device.cuh"
#include "akv_internal.h"

namespace akv {
namespace {

// The Lloyd-Max codec's outer decision threshold: the midpoint of its levels 0.453125 and
// 1.5078125 (the Gaussian four-level Lloyd-Max levels 0.4528, 1.5104 to 8 significant bits).
constexpr double kLloydT = 0.98046875;

// Per-unit scratch pointers, derived from the workspace table the host writes.
struct EncUnitWs {
  // [S] each: selector scores; then (plain encoder) the first half holds the residual energies per
  // side as fp32 bits + 1, anchors 0, or (full selection, and slots that need fp64 energies) the
  // whole the fp64 bits + 1; then the counting sort's rows
  uint64_t* key0;
  uint64_t* key1;
  int32_t* slot_of;   // [S] anchor slot or -1
  int32_t* res_pos;   // [N_K + N_V] residual positions (keys, then values)
  double* n2[2];      // [k] squared anchor norms per side
  // [side]: the side has a nonzero anchor; [2 + side]: full selection's residual counts; [4 + side]:
  // an anchor norm outside the filter's range; [6 + side]: an energy outside the fp32 range, or a
  // band too wide, so that the slots are chosen from fp64 energies; [8 + side]: positions left to fp64,
  // [10 + side]: positions where any anchor may be the nearest (lists behind the energies)
  uint32_t* ctrl;
  uint32_t* st[2];    // [S] stream word (slot | fp16 gamma << 16) per position and side
  uint8_t* flag[2];   // [S] residual flag per side (values: over slot_of, which is read no more by then)
  float* inv[2];      // [k to a multiple of 32] 1 / anchor norm, 0 for a zero anchor (over perm and inv)
  int32_t* perm;      // [S] position of stored token t (full selection, before that: errors of u^K, fp64, over perm and at)
  int32_t* at;        // [S] stored index of position i
  uint32_t* cursor;   // [k + 1] value-anchor counts, then start of each run
  uint32_t* tcnt;     // [2 * n_tiles] residual records per tile (keys, values)
  double* alpha;      // full selection: [m][S] observation rows' attention
  double* yobs;       // full selection: [m][128] their exact outputs
};

struct EncArgs {
  const uint8_t* arena_c;
  uint8_t* arena;
  const uint8_t* ws_base;
  const uint64_t* ws_off;  // [units] byte offsets of each unit's scratch
  const __nv_bfloat16* K;
  const __nv_bfloat16* V;
  int32_t s_max;
  int32_t n_kv_heads;
  int32_t window;
  int32_t rotate;
  int32_t lloyd;  // AKV_FLAG_LLOYD: the Lloyd-Max codec
  uint64_t seed;
  unsigned long long sign_lo, sign_hi;
  // full selection (m_obs > 0): observation rows Q [units][m_obs][128], pooling width,
  // scored share, retained fraction
  const __nv_bfloat16* Q;
  int32_t m_obs, kappa;
  float rho, theta;
};

__device__ __forceinline__ const akv_unit_desc* unit_desc(const EncArgs& A, int u) {
  return reinterpret_cast<const akv_unit_desc*>(A.arena_c + 256) + u;
}

__device__ __forceinline__ uint64_t au(uint64_t x, uint64_t a) { return (x + a - 1) / a * a; }

__device__ EncUnitWs unit_ws(const EncArgs& A, int u, const akv_unit_desc* d) {
  uint8_t* p = const_cast<uint8_t*>(A.ws_base) + A.ws_off[u];
  EncUnitWs w;
  const uint64_t S = (uint64_t)d->len, k = (uint64_t)d->n_anchors, n = (uint64_t)(d->n_res_k + d->n_res_v);
  w.key0 = (uint64_t*)p;
  p += au(S * 8, 256);
  w.key1 = (uint64_t*)p;
  p += au(S * 8, 256);
  w.slot_of = (int32_t*)p;
  p += au(S * 4, 256);
  w.res_pos = (int32_t*)p;
  p += au(n * 4 + 16, 256);
  for (int s = 0; s < 2; ++s) {
    w.n2[s] = (double*)p;
    p += 2 * au(k * 8, 256);
  }
  w.ctrl = (uint32_t*)p;
  p += 256;
  for (int s = 0; s < 2; ++s) {
    w.st[s] = (uint32_t*)p;
    p += au(S * 4, 256);
  }
  w.flag[0] = p;
  w.flag[1] = reinterpret_cast<uint8_t*>(w.slot_of);
  p += au(S, 256);
  w.perm = (int32_t*)p;
  w.inv[0] = (float*)p;
  p += au(S * 4, 256);
  w.at = (int32_t*)p;
  w.inv[1] = (float*)p;
  p += au(S * 4, 256);
  w.cursor = (uint32_t*)p;
  p += au((k + 1) * 4, 256);
  w.tcnt = (uint32_t*)p;
  p += au((uint64_t)d->n_tiles * 8, 256);
  w.alpha = (double*)p;
  p += au((uint64_t)A.m_obs * S * 8, 256);
  w.yobs = (double*)p;
  return w;
}

// Anchor row a of a side in the source K or V (the arena holds it swizzled).
__device__ __forceinline__ const __nv_bfloat16* anchor_src(const EncArgs& A, int u, int side, const int32_t* apos, int a) {
  return (side ? A.V : A.K) + ((size_t)u * A.s_max + (size_t)apos[a]) * 128;
}

__device__ __forceinline__ uint64_t splitmix64_dev(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ double bf16_to_f64(__nv_bfloat16 v) { return (double)__bfloat162float(v); }
__device__ __forceinline__ double fp16_bits_to_f64(uint32_t h) {
  return (double)__half2float(__ushort_as_half((unsigned short)(h & 0xFFFFu)));
}

// fp64 -> fp16 bits, round to nearest even on the integer significand,
// saturating at +-65504 (values are finite here; NaN maps to 0x7E00).
__device__ uint32_t f64_to_fp16_bits(double x) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const uint32_t sign = (uint32_t)(bits >> 63) << 15;
  const int ex = (int)((bits >> 52) & 0x7FF);
  const unsigned long long frac = bits & 0xFFFFFFFFFFFFFull;
  if (ex == 0x7FF) return frac ? 0x7E00u : (sign | 0x7BFFu);
  if (fabs(x) >= 65504.0) return sign | 0x7BFFu;
  if (ex == 0) return sign;  // fp64 subnormals are far below half an fp16 ulp
  const int e = ex - 1023;
  if (e < -25) return sign;
  const unsigned long long m = frac | (1ull << 52);  // 53-bit significand
  const int sh = (e >= -14) ? 42 : 42 + (-14 - e);   // bits dropped
  unsigned long long r = m >> sh;
  const unsigned long long rem = m & ((1ull << sh) - 1ull);
  const unsigned long long half = 1ull << (sh - 1);
  if (rem > half || (rem == half && (r & 1ull))) ++r;
  uint32_t out;
  if (e >= -14) out = (uint32_t)(((e + 14) << 10) + (int)r);  // r carries the implicit 1024
  else out = (uint32_t)r;                                      // subnormal (1024 -> smallest normal)
  if (out >= 0x7C00u) out = 0x7BFFu;
  return sign | out;
}

// r-th smallest (1-based) of the n 64-bit keys key_at(0 .. n-1) (optionally of their
// complements), MSB-first radix select by 8-bit digits; returns the key and the rank of
// the answer among keys equal to it (*rank_in_eq, 1-based).  Block-wide.
template <class KeyAt>
__device__ uint64_t block_select_f(KeyAt key_at, int64_t n, uint32_t r, bool complement, uint32_t* hist,
                                   uint32_t* bcast, uint32_t* rank_in_eq) {
  uint64_t prefix = 0, mask = 0;
  for (int shift = 56; shift >= 0; shift -= 8) {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
      uint64_t key = key_at(i);
      if (complement) key = ~key;
      if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t cum = 0, sel = 255;
      for (uint32_t bkt = 0; bkt < 256; ++bkt) {
        if (cum + hist[bkt] >= r) {
          sel = bkt;
          break;
        }
        cum += hist[bkt];
      }
      bcast[0] = sel;
      bcast[1] = r - cum;
    }
    __syncthreads();
    prefix |= (uint64_t)bcast[0] << shift;
    mask |= 0xFFull << shift;
    r = bcast[1];
    __syncthreads();
  }
  *rank_in_eq = r;
  return complement ? ~prefix : prefix;
}
__device__ uint64_t block_select(const uint64_t* keys, int n, uint32_t r, bool complement, uint32_t* hist,
                                 uint32_t* bcast, uint32_t* rank_in_eq) {
  return block_select_f([keys](int64_t i) { return keys[i]; }, n, r, complement, hist, bcast, rank_in_eq);
}

// Exclusive block scan of 0/1 flags for a block of 1024 threads; returns the
// prefix and writes the block total to *total.
__device__ int block_scan_flag(int flag, int* warp_tot, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned bal = __ballot_sync(0xffffffffu, flag);
  const int pre_lane = __popc(bal & ((1u << lane) - 1u));
  if (lane == 0) warp_tot[warp] = __popc(bal);
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    int v = lane < nw ? warp_tot[lane] : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane < nw) warp_tot[lane] = incl - v;
    if (lane == 31) warp_tot[32] = incl;
  }
  __syncthreads();
  const int pre = warp_tot[warp] + pre_lane;
  *total = warp_tot[32];
  __syncthreads();
  return pre;
}

// ---- kernels -----------------------------------------------------------------

// Anchors of the full selection picked by score: floor(rho (k - w)) (Section 3.2); none in
// the plain encoder.
__device__ __forceinline__ int n_scored(const EncArgs& A, int rest) {
  return (A.m_obs > 0 && rest > 0) ? (int)floor((double)A.rho * (double)rest) : 0;
}

// Clusters of kSelCtas CTAs take one unit (and side): they share out its positions and exchange
// counts through distributed shared memory.
constexpr int kSelCtas = 8, kSelThreads = 512, kSelBand = 512;

// The CTA's share [lo, hi) of n items, of a multiple of 4 items.
__device__ __forceinline__ void cluster_share(int n, int rank, int& lo, int& hi) {
  const int per = (int)((((long long)n + kSelCtas - 1) / kSelCtas + 3) & ~3ll);
  lo = (int)min((long long)n, (long long)rank * per);
  hi = (int)min((long long)n, (long long)lo + per);
}

// One digit of a radix select over the cluster, called by all its CTAs after the cluster barrier that
// ends the counting: of the 2048 digits counted in every CTA's `hist` (taken from the largest down,
// or from the smallest up) the one that holds the want-th key; want becomes the rank inside it.  The
// number of keys with that digit goes to *inside.
template <bool DOWN>
__device__ uint32_t cluster_digit(cooperative_groups::cluster_group cl, uint32_t* hist, uint32_t* wsum, uint32_t* found,
                                  uint32_t& want, uint32_t* inside) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t c[4] = {0u, 0u, 0u, 0u};  // four digits per thread, in order
  for (int r = 0; r < kSelCtas; ++r) {
    const uint4 v = *reinterpret_cast<const uint4*>(cl.map_shared_rank(hist, r) + (DOWN ? 2044 - 4 * tid : 4 * tid));
    c[0] += DOWN ? v.w : v.x;
    c[1] += DOWN ? v.z : v.y;
    c[2] += DOWN ? v.y : v.z;
    c[3] += DOWN ? v.x : v.w;
  }
  const uint32_t sum = c[0] + c[1] + c[2] + c[3];
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  uint32_t before = incl - sum;
  for (int x = 0; x < warp; ++x) before += wsum[x];
  if (before < want && want <= before + sum) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (before < want && want <= before + c[e]) {
        found[0] = (uint32_t)(DOWN ? 2047 - 4 * tid - e : 4 * tid + e);
        found[1] = want - before;
        found[2] = c[e];
      }
      before += c[e];
    }
  }
  __syncthreads();
  const uint32_t digit = found[0];
  want = found[1];
  *inside = found[2];
  __syncthreads();
  return digit;
}
static_assert(kSelThreads * 4 == 2048, "four digits per thread");

// The unit's anchors: the last min(W, S) positions, the positions the full selection scored, and the
// `rest` smallest hashes of the others; slots numbered by position.  A radix select over the cluster
// finds the hash that bounds the rest (hashes are distinct, so it ends at the first digit whose keys
// are all wanted: two or three digits); hashes are computed where they are needed.  (One CTA per unit
// and eight digits of stored hashes took 72 us for 8 x 32768 positions and 232 us for 2 x 131072.)
__global__ void __cluster_dims__(kSelCtas, 1, 1) __launch_bounds__(kSelThreads) enc_anchors(const EncArgs A) {
  namespace cg = cooperative_groups;
  __shared__ __align__(16) uint32_t hist[3][2048];
  __shared__ uint32_t wsum[kSelThreads / 32];
  __shared__ uint32_t found[3];
  __shared__ uint32_t total;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int u = blockIdx.x / kSelCtas;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, k = d->n_anchors;
  const EncUnitWs w = unit_ws(A, u, d);
  const int win = min(A.window, S), pool = S - win;
  const bool full = A.m_obs > 0;
  // the sampled share: all k - w non-window anchors, less those the full selection scored
  const uint32_t rest = (uint32_t)(k - win - n_scored(A, k - win));
  const uint64_t base = A.seed ^ ((uint64_t)d->b << 40) ^ ((uint64_t)d->h << 32);
  int lo, hi;
  cluster_share(S, rank, lo, hi);
  for (int i = tid; i < 3 * 2048; i += kSelThreads) (&hist[0][0])[i] = 0u;
  __syncthreads();
  int sh = 64;          // the keys taken are those with key >> sh <= prefix
  uint64_t prefix = 0;
  if (rest > 0) {
    uint32_t want = rest;
#pragma unroll 1
    for (int dg = 0;; ++dg) {
      const int ns = max(0, sh - 11), bits = sh - ns;
      uint32_t* h = hist[dg % 3];
      for (int p = lo + tid; p < min(hi, pool); p += kSelThreads) {
        if (full && w.slot_of[p] == -2) continue;  // already chosen by its score
        const uint64_t v = splitmix64_dev(base ^ (uint64_t)p);
        if (dg == 0 || (v >> sh) == prefix) atomicAdd(&h[(uint32_t)(v >> ns) & ((1u << bits) - 1u)], 1u);
      }
      cl.sync();
      // (the third buffer's last readers passed the barrier before this one)
      if (dg > 0)
        for (int i = tid; i < 2048; i += kSelThreads) hist[(dg + 2) % 3][i] = 0u;
      uint32_t inside;
      const uint32_t digit = cluster_digit<false>(cl, h, wsum, found, want, &inside);
      prefix = (prefix << bits) | digit;
      sh = ns;
      if (want == inside || sh == 0) break;
    }
  }
  auto is_anchor = [&](int p) {
    return p >= pool || (full && w.slot_of[p] == -2) || (rest > 0 && (splitmix64_dev(base ^ (uint64_t)p) >> sh) <= prefix);
  };
  // slots by position: a warp takes a contiguous share of the CTA's, 32 positions at a time
  const int per = (((hi - lo) + kSelThreads - 1) / kSelThreads) * 32;
  const int wlo = min(hi, lo + warp * per), whi = min(hi, wlo + per);
  uint32_t n = 0;
  for (int p0 = wlo; p0 < whi; p0 += 32) {
    const int p = p0 + lane;
    n += (uint32_t)__popc(__ballot_sync(0xffffffffu, p < whi && is_anchor(p)));
  }
  if (lane == 0) wsum[warp] = n;
  __syncthreads();
  if (tid == 0) {
    uint32_t t = 0;
    for (int x = 0; x < kSelThreads / 32; ++x) t += wsum[x];
    total = t;
  }
  cl.sync();
  uint32_t at = 0;
  for (int r = 0; r < rank; ++r) at += *cl.map_shared_rank(&total, r);
  for (int x = 0; x < warp; ++x) at += wsum[x];
  int32_t* apos = reinterpret_cast<int32_t*>(A.arena + d->off_anchor_pos);
  for (int p0 = wlo; p0 < whi; p0 += 32) {
    const int p = p0 + lane;
    const bool is = p < whi && is_anchor(p);
    const unsigned bal = __ballot_sync(0xffffffffu, is);
    const uint32_t slot = at + (uint32_t)__popc(bal & ((1u << lane) - 1u));
    if (p < whi) w.slot_of[p] = is ? (int32_t)slot : -1;
    if (is) apos[slot] = p;
    at += (uint32_t)__popc(bal);
  }
  if (rank == 0 && tid < 16) w.ctrl[tid] = 0;
  cl.sync();  // no CTA leaves while another may still read its counts
}

// Bytes of one bf16 pair as two floats.
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// A bf16 value, as the bits of a float, in fp64, on the integer pipe: the fp64 unit of an SM sub-partition
// takes 64 cycles for one warp instruction, conversions included.
__device__ __forceinline__ double bf_f64(uint32_t f) {
  const uint32_t mag = f & 0x7FFFFFFFu;
  if (mag - 0x00800000u >= 0x7F000000u) return (double)__uint_as_float(f);  // 0, subnormal, inf, NaN
  return __hiloint2double((int)((f & 0x80000000u) | ((mag >> 3) + 0x38000000u)), 0);
}

// fp16 bits of a float, round to nearest even, saturating like f64_to_fp16_bits.
__device__ __forceinline__ uint32_t f32_to_fp16_bits(float x) {
  const uint32_t b = __half_as_ushort(__float2half_rn(x));
  if ((b & 0x7FFFu) < 0x7C00u) return b;
  return (b & 0x3FFu) ? 0x7E00u : ((b & 0x8000u) | 0x7BFFu);
}

// Anchor norms the fp32 filter handles: every product and sum of enc_assign_tc and enc_finish then
// stays inside the fp32 range.
constexpr double kNormLo = 0x1p-60, kNormHi = 0x1p60;  // of squared norms

// 32 anchors of one side per block: rows copied into the arena, squared norms (sequential in j; the
// square of a bf16 is exact, so a fused multiply-add rounds like the separate steps).  The rows pass
// through shared memory so that one lane per anchor runs the serial fp64 chain: with one lane per
// warp reading its row from global memory the same sums took 289 us for 8 units of 656 anchors.
__global__ void __launch_bounds__(256) enc_rows(const EncArgs A) {
  __shared__ __align__(16) uint4 rows[32][17];
  const int u = blockIdx.y, side = blockIdx.z;
  const akv_unit_desc* d = unit_desc(A, u);
  const int k = d->n_anchors, a0 = blockIdx.x * 32, tid = threadIdx.x;
  if (a0 >= k) return;
  EncUnitWs w = unit_ws(A, u, d);
  const int32_t* apos = reinterpret_cast<const int32_t*>(A.arena_c + d->off_anchor_pos);
  uint8_t* dst = A.arena + (side ? d->off_anchor_v : d->off_anchor_k);
  for (int e = tid; e < 32 * 16; e += 256) {
    const int r = e >> 4, c = e & 15, a = a0 + r;
    if (a >= k) continue;
    const uint4 v = reinterpret_cast<const uint4*>(anchor_src(A, u, side, apos, a))[c];
    rows[r][c] = v;
    // chunk c (dims 8 c .. 8 c + 7) at chunk place c ^ (a % 8)
    *reinterpret_cast<uint4*>(dst + (size_t)a * 256 + 16 * (c ^ (a & 7))) = v;
  }
  __syncthreads();
  if (tid >= 32) return;
  const int a = a0 + tid;
  double n = 0.0;
  if (a < k) {
    for (int c = 0; c < 16; ++c) {
      const uint4 v = rows[tid][c];
      const uint32_t wd[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double lo = bf_f64(wd[e] << 16), hi = bf_f64(wd[e] & 0xFFFF0000u);
        n = __fma_rn(lo, lo, n);
        n = __fma_rn(hi, hi, n);
      }
    }
    w.n2[side][a] = n;
  }
  const bool safe = n >= kNormLo && n <= kNormHi;
  w.inv[side][a] = a < k && safe ? (float)__ddiv_rn(1.0, __dsqrt_rn(n)) : 0.0f;  // (a < k rounded up to 32)
  if (__any_sync(0xffffffffu, a < k && n != 0.0) && tid == 0) atomicOr(&w.ctrl[side], 1u);
  if (__any_sync(0xffffffffu, a < k && n != 0.0 && !safe) && tid == 0) atomicOr(&w.ctrl[4 + side], 1u);
}

// ---- Eq. 1 on tensor cores ------------------------------------------------------------
// The nearest anchor of a position is the one with the largest |x . x_a| / |x_a|, decided in fp64.
// As a GEMM (positions x anchors x 128) the fp64 units need 81 ms for a layer of 8 x 32768 positions
// and 656 anchors; the tensor cores' fp32 sums of the exact bf16 products take the same scores to
// within 2^-15 |x| (128 exact products, fp32 accumulation; 4 times the worst bound of eight truncated
// steps, the column bits below included: how the hardware adds the products of a step is not documented, so this is an
// assumption, with that factor of 4 to spare and the tests' near ties to support it), so only the anchors within 2 x 2^-15 |x| of a
// position's largest score can be its nearest.  That leaves one anchor for about 99 % of positions; enc_finish and
// enc_undecided decide the rest.  The candidate word of a position: first candidate in bits 0-15, second
// in bits 16-31 (0xFFFF: none; the first again: the anchors of its group of 32), or 0xFFFFFFFF: any
// anchor may be the nearest.
//
// One persistent CTA per SM takes items of 256 positions of one unit and side (two M = 128 tiles
// that share every anchor chunk, which halves the L2 reads of the anchors), anchor chunks of 128.
// Warp 16 copies (three position tiles and three anchor chunks in flight), warp 17 issues the products (two
// accumulators of 128 TMEM columns per tile, taken by alternate chunks), warps 18 and 19 take the positions' norms one
// item ahead, warps 0-15 are the epilogues, four per tile and accumulator: a thread owns one position and half of its
// chunks, and takes 32 columns at a time without branches on single columns (those diverge: in the first chunks
// nearly every column is some lane's new maximum, and the kernel took 293 us that way): scores with the column number
// in their lowest bits give the largest and its column, and a clamped sum how many come near it.  The halves' candidates are put together at the
// item's end.  Waits are bounded; after a failure every remaining position gets the word that lets
// enc_finish decide it alone, so the result stays right.
// Bound: the epilogues' latencies, some 190 instructions per 32 columns and warp (56 % of the issue slots, ALU pipe
// 48 %, tensor pipe 28 %).  8 units of 32768 positions, 656 anchors: 126 us; 2 of 131072, 2621: 405 us.  With one
// accumulator of 192 columns per tile and eight epilogue warps, loads a step ahead: 143 and 480 us; eight warps that
// each take both tiles (inverse norms read once for them): 136 us.
constexpr int kAtN = 128;
constexpr int kAtA = 3, kAtB = 3;  // stages
constexpr uint32_t kAtHalfA = 128 * 128, kAtHalfB = kAtN * 128;  // bytes of 64 of the 128 dimensions
constexpr int kAtI = 4;  // chunks of inverse norms in flight
constexpr uint32_t kAtSmem = kAtA * 2 * kAtHalfA + kAtB * 2 * kAtHalfB + kAtI * kAtN * 4 + 2 * 256 * 4 + 2 * 256 * 8 + 1024;
constexpr int kAtThreads = 640;
constexpr float kAtMargin = 0x1p-14f;  // 2 x 2^-15, relative to |x|

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// a b + c clamped to [0, 1] (NaN: 0)
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
  float r;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// a with its five lowest bits replaced by col, without the sign (one instruction: the mask is a register, since an
// instruction holds one immediate)
__device__ __forceinline__ float tagged(float a, uint32_t mask, uint32_t col) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(__float_as_uint(a)), "r"(mask), "r"(col));
  return __uint_as_float(r);
}
// 32 columns of the thread's TMEM lane.  One statement with its wait: registers that a load fills before a separate
// wait were copied, some 70 moves per 32 columns.
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float2 (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
      " tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x), "=f"(v[3].y), "=f"(v[4].x), "=f"(v[4].y), "=f"(v[5].x), "=f"(v[5].y), "=f"(v[6].x), "=f"(v[6].y), "=f"(v[7].x), "=f"(v[7].y), "=f"(v[8].x), "=f"(v[8].y), "=f"(v[9].x), "=f"(v[9].y), "=f"(v[10].x), "=f"(v[10].y), "=f"(v[11].x), "=f"(v[11].y), "=f"(v[12].x), "=f"(v[12].y), "=f"(v[13].x), "=f"(v[13].y), "=f"(v[14].x), "=f"(v[14].y), "=f"(v[15].x), "=f"(v[15].y)
      : "r"(taddr)
      : "memory");
}

__global__ void __launch_bounds__(kAtThreads, 1)
    enc_assign_tc(const __grid_constant__ EncArgs A, const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmA, long long items,
                  int max_t) {
  extern __shared__ __align__(1024) uint8_t as_dyn[];
  __shared__ __align__(8) uint64_t bars[2 * kAtA + 2 * kAtB + 12 + kAtI];
  __shared__ uint32_t tmem_sh;
  __shared__ int failed_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sA = (smem_u32(as_dyn) + 1023u) & ~1023u, sB = sA + kAtA * 2 * kAtHalfA;
  auto a_full = [&](int s) { return smem_u32(bars + s); };
  auto a_free = [&](int s) { return smem_u32(bars + kAtA + s); };
  auto b_full = [&](int s) { return smem_u32(bars + 2 * kAtA + s); };
  auto b_free = [&](int s) { return smem_u32(bars + 2 * kAtA + kAtB + s); };
  auto acc_full = [&](int a) { return smem_u32(bars + 2 * kAtA + 2 * kAtB + a); };  // a = 2 h + m
  auto acc_empty = [&](int a) { return smem_u32(bars + 2 * kAtA + 2 * kAtB + 4 + a); };
  auto nrm_full = [&](int b) { return smem_u32(bars + 2 * kAtA + 2 * kAtB + 8 + b); };
  auto nrm_free = [&](int b) { return smem_u32(bars + 2 * kAtA + 2 * kAtB + 10 + b); };
  auto inv_free = [&](int s) { return smem_u32(bars + 2 * kAtA + 2 * kAtB + 12 + s); };
  const uint32_t sI = sB + kAtB * 2 * kAtHalfB;
  float* inv_sm = reinterpret_cast<float*>(as_dyn + (sI - smem_u32(as_dyn)));  // [kAtI][kAtN]
  float* nrm_sm = inv_sm + kAtI * kAtN;                                        // [2][256] squared norms
  uint2* part_sm = reinterpret_cast<uint2*>(nrm_sm + 2 * 256);                 // [2][256] half 0's candidates
  volatile int* failed = &failed_sh;
  if (tid == 0) {
    for (int i = 0; i < 2 * kAtA + 2 * kAtB + 4; ++i) mbar_init(smem_u32(bars + i), 1);
    for (int a = 0; a < 4; ++a) mbar_init(acc_empty(a), 4);  // one arrival per epilogue warp
    for (int b = 0; b < 2; ++b) {
      mbar_init(nrm_full(b), 2);   // per norm warp
      mbar_init(nrm_free(b), 16);  // per epilogue warp
    }
    for (int s = 0; s < kAtI; ++s) mbar_init(inv_free(s), 8);
    *failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tc_alloc(smem_u32(&tmem_sh), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_sh;

  // item (unit u, side, tile t): positions 256 t .. of the unit; every role walks the same items
  struct Item {
    int u, side, t, S, k;
  };
  auto next_item = [&](long long& i, Item& it) {  // the item at or after i that holds positions
    for (; i < items; i += gridDim.x) {
      it.t = (int)(i % max_t);
      it.side = (int)((i / max_t) & 1);
      it.u = (int)(i / max_t / 2);
      const int2 sk = __ldg(reinterpret_cast<const int2*>(unit_desc(A, it.u)));
      it.S = sk.x;
      it.k = sk.y;
      if (it.t * 256 < it.S) return true;
    }
    return false;
  };
  auto n_tiles = [](const Item& it) { return it.S - it.t * 256 > 128 ? 2 : 1; };

  if (warp == 16) {
    if (lane == 0) {  // ---- copies
      int na = 0, nb = 0;
      auto load_a = [&](const Item& it, int m) {
        const int s = na % kAtA;
        if (!mbar_wait(a_free(s), (uint32_t)((na / kAtA) & 1) ^ 1u)) return false;
        const CUtensorMap* tm = it.side ? &tmV : &tmK;
        const int row = it.u * A.s_max + it.t * 256 + 128 * m;
        mbar_expect_tx(a_full(s), 2 * kAtHalfA);
        tma_load_2d(sA + s * 2 * kAtHalfA, tm, 0, row, a_full(s));
        tma_load_2d(sA + s * 2 * kAtHalfA + kAtHalfA, tm, 64, row, a_full(s));
        ++na;
        return true;
      };
      bool ok = true;
      Item it;
      for (long long i = blockIdx.x; ok && next_item(i, it); i += gridDim.x) {
        const akv_unit_desc* d = unit_desc(A, it.u);
        const EncUnitWs w = unit_ws(A, it.u, d);
        const float* inv = it.side ? w.inv[1] : w.inv[0];
        const int row0 = (int)((it.side ? d->off_anchor_v : d->off_anchor_k) >> 8);
        ok = load_a(it, 0);
        for (int c0 = 0; ok && c0 < it.k; c0 += kAtN) {
          const int s = nb % kAtB, nr = (min(kAtN, it.k - c0) + 63) / 64;  // boxes of 64 anchor rows
          if (*failed || !mbar_wait(b_free(s), (uint32_t)((nb / kAtB) & 1) ^ 1u) ||
              !mbar_wait(inv_free(nb % kAtI), (uint32_t)((nb / kAtI) & 1) ^ 1u)) {
            ok = false;
            break;
          }
          const uint32_t ib = (uint32_t)min(kAtN, (it.k - c0 + 31) & ~31) * 4u;
          mbar_expect_tx(b_full(s), (uint32_t)nr * 2 * 64 * 128 + ib);
          bulk_g2s(sI + (uint32_t)(nb % kAtI) * kAtN * 4u, inv + c0, ib, b_full(s));
          for (int r = 0; r < nr; ++r) {
            tma_load_2d(sB + s * 2 * kAtHalfB + r * 64 * 128, &tmA, 0, row0 + c0 + 64 * r, b_full(s));
            tma_load_2d(sB + s * 2 * kAtHalfB + kAtHalfB + r * 64 * 128, &tmA, 64, row0 + c0 + 64 * r, b_full(s));
          }
          ++nb;
          if (c0 == 0 && n_tiles(it) == 2) ok = load_a(it, 1);
        }
      }
      if (!ok) *failed = 1;
      // (bounded) every copy has landed before the CTA may exit
      for (int j = max(0, na - kAtA); j < na; ++j) mbar_wait(a_full(j % kAtA), (uint32_t)(j / kAtA) & 1u);
      for (int j = max(0, nb - kAtB); j < nb; ++j) mbar_wait(b_full(j % kAtB), (uint32_t)(j / kAtB) & 1u);
    }
    __syncwarp();
  } else if (warp == 17) {
    if (lane == 0) {  // ---- products
      int na = 0, nb = 0, ni = 0;
      uint32_t nacc[4] = {0u, 0u, 0u, 0u};
      bool ok = true;
      Item it;
      for (long long i = blockIdx.x; ok && next_item(i, it); i += gridDim.x, ++ni) {
        const int nm = n_tiles(it);
        for (int c = 0, c0 = 0; ok && c0 < it.k; c0 += kAtN, ++nb, ++c) {
          const int h = (c + ni) & 1;
          const int sb = nb % kAtB;
          const uint32_t n = (uint32_t)min(kAtN, (it.k - c0 + 15) & ~15);
          const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
          ok = !*failed && mbar_wait(b_full(sb), (uint32_t)(nb / kAtB) & 1u);
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            if (!ok || m >= nm) break;
            const int sa = (na + m) % kAtA;
            ok = (c0 > 0 || mbar_wait(a_full(sa), (uint32_t)((na + m) / kAtA) & 1u)) &&
                 mbar_wait(acc_empty(2 * h + m), ((h ? nacc[2 + m] : nacc[m]) & 1u) ^ 1u);
            if (!ok) break;
            tc_fence_after();
            const uint64_t da = sw128_desc(sA + sa * 2 * kAtHalfA), db = sw128_desc(sB + sb * 2 * kAtHalfB);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const uint32_t ka = (uint32_t)(kk >> 2) * kAtHalfA + (uint32_t)(kk & 3) * 32;
              const uint32_t kb = (uint32_t)(kk >> 2) * kAtHalfB + (uint32_t)(kk & 3) * 32;
              tc_mma(tmem + 128u * (uint32_t)(2 * h + m), da + (ka >> 4), db + (kb >> 4), idesc, kk > 0 ? 1u : 0u);
            }
            if (h) ++nacc[2 + m];
            else ++nacc[m];
            tc_commit(acc_full(2 * h + m));
            if (c0 + kAtN >= it.k) tc_commit(a_free(sa));
          }
          if (ok) tc_commit(b_free(sb));
        }
        na += nm;
      }
      if (!ok) *failed = 1;
      // (bounded) every product has completed before the CTA may exit: the last commits have arrived
#pragma unroll
      for (int a = 0; a < 4; ++a)
        if (nacc[a] > 0) mbar_wait(acc_full(a), (nacc[a] - 1u) & 1u);
    }
    __syncwarp();
  } else if (warp >= 18) {  // ---- squared norms of the item's 256 positions, four per thread
    int j = 0;
    Item it;
    for (long long i = blockIdx.x; next_item(i, it); i += gridDim.x, ++j) {
      const int t = tid - 576, b = j & 1;
      const uint4* X = reinterpret_cast<const uint4*>((it.side ? A.V : A.K) + ((size_t)it.u * A.s_max + it.t * 256) * 128);
      float nx2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (it.t * 256 + t + 64 * h >= it.S) continue;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const uint4 v = __ldg(X + (size_t)(t + 64 * h) * 16 + c);
          const uint32_t wd[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            nx2[h] = __fmaf_rn(bf_lo(wd[e]), bf_lo(wd[e]), nx2[h]);
            nx2[h] = __fmaf_rn(bf_hi(wd[e]), bf_hi(wd[e]), nx2[h]);
          }
        }
      }
      __syncwarp();
      if (__shfl_sync(0xffffffffu, *failed, 0) != 0 || !mbar_wait_w(nrm_free(b), (uint32_t)((j >> 1) & 1) ^ 1u)) {
        *failed = 1;
        break;
      }
#pragma unroll
      for (int h = 0; h < 4; ++h) nrm_sm[256 * b + 64 * h + t] = nx2[h];
      __syncwarp();
      if (lane == 0) mbar_arrive(nrm_full(b));
    }
  } else {  // ---- epilogue of tile m, half h of its chunks
    const int m = (warp >> 2) & 1, h = warp >> 3, q = warp & 3;
    uint32_t tag_mask;
    asm volatile("mov.b32 %0, 0x7FFFFFE0;" : "=r"(tag_mask));
    int nacc = 0, ni = 0, nc = 0;  // accumulators, items and anchor chunks so far
    bool ok = true;
    Item it;
    for (long long i = blockIdx.x; next_item(i, it); i += gridDim.x, ++ni) {
      const int p = it.t * 256 + 128 * m + 32 * q + lane;
      const EncUnitWs w = unit_ws(A, it.u, unit_desc(A, it.u));
      __syncwarp();
      ok = ok && __shfl_sync(0xffffffffu, *failed, 0) == 0 && mbar_wait_w(nrm_full(ni & 1), (uint32_t)(ni >> 1) & 1u);
      const float nx2 = ok ? nrm_sm[256 * (ni & 1) + 128 * m + 32 * q + lane] : 0.f;
      __syncwarp();
      if (lane == 0) mbar_arrive(nrm_free(ni & 1));
      if (m >= n_tiles(it)) {  // no positions of this tile: its chunks pass by
        for (int c = 0, c0 = 0; c0 < it.k; c0 += kAtN, ++nc, ++c) {
          if (((c + ni) & 1) != h) continue;
          if (ok && nc >= kAtI) ok = mbar_wait_w(inv_free(nc % kAtI), (uint32_t)(nc / kAtI - 1) & 1u);
          if (lane == 0) mbar_arrive(inv_free(nc % kAtI));
        }
        continue;
      }
      const bool usable = nx2 >= (float)kNormLo && nx2 <= (float)kNormHi && w.ctrl[4 + it.side] == 0u;
      const float marg = kAtMargin * 1.001f * __fsqrt_rn(nx2);
      const float rm = 1.f / marg;  // (an unusable row may give anything here: its word is not used)
      float m1 = 0.f;               // the largest score so far
      uint32_t i1 = 0xFFFFu, i2 = 0xFFFFu;  // its anchor; a second one within the margin, or i1: its group
      bool more = false;                    // candidates beyond these
      // 32 columns at a time: scores with the column in the five lowest bits (2^-18 relative), their
      // largest, and how many lie within the margin of it (s / margin, shifted so that 1 is reached
      // there, clamped to [0, 1])
      auto step = [&](const float2 (&s)[16], const float* iv, uint32_t a0) {
        float v[32];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float4 f = *reinterpret_cast<const float4*>(iv + 4 * e);
          const float2 x = __fmul2_rn(s[2 * e], make_float2(f.x, f.y)), y = __fmul2_rn(s[2 * e + 1], make_float2(f.z, f.w));
          v[4 * e] = tagged(x.x, tag_mask, (uint32_t)(4 * e));
          v[4 * e + 1] = tagged(x.y, tag_mask, (uint32_t)(4 * e + 1));
          v[4 * e + 2] = tagged(y.x, tag_mask, (uint32_t)(4 * e + 2));
          v[4 * e + 3] = tagged(y.y, tag_mask, (uint32_t)(4 * e + 3));
        }
        float mx[11];
#pragma unroll
        for (int e = 0; e < 10; ++e) mx[e] = max3(v[3 * e], v[3 * e + 1], v[3 * e + 2]);
        mx[10] = fmaxf(v[30], v[31]);
        const float c1 = max3(max3(max3(mx[0], mx[1], mx[2]), max3(mx[3], mx[4], mx[5]), max3(mx[6], mx[7], mx[8])), mx[9], mx[10]);
        const float top = fmaxf(m1, c1), off = __fmaf_rn(-top, rm, 2.f);
        float2 near2[4] = {};
#pragma unroll
        for (int e = 0; e < 32; e += 2)
          near2[(e / 2) & 3] = __fadd2_rn(near2[(e / 2) & 3], make_float2(fma_sat(v[e], rm, off), fma_sat(v[e + 1], rm, off)));
        const float2 nr = __fadd2_rn(__fadd2_rn(near2[0], near2[1]), __fadd2_rn(near2[2], near2[3]));
        const bool several = nr.x + nr.y > 1.004f;
        const bool here = c1 >= m1 - marg, alone = c1 > m1 + marg;  // alone: nothing before comes near
        const uint32_t idx = a0 + (__float_as_uint(c1) & 31u);
        more = here ? !alone && (more || several || i2 != 0xFFFFu) : more;
        i2 = here ? (alone ? (several ? idx : 0xFFFFu) : idx) : i2;
        i1 = alone ? idx : i1;
        m1 = top;
      };
      for (int c = 0, c0 = 0; c0 < it.k; c0 += kAtN, ++nc, ++c) {
        if (((c + ni) & 1) != h) continue;
        __syncwarp();
        ok = ok && __shfl_sync(0xffffffffu, *failed, 0) == 0 && mbar_wait_w(acc_full(2 * h + m), (uint32_t)nacc & 1u);
        if (!ok) continue;  // (the same for the whole warp)
        ++nacc;
        tc_fence_after();
        const int n = min(kAtN, it.k - c0);
        const uint32_t tcol = tmem + ((uint32_t)(32 * q) << 16) + 128u * (uint32_t)(2 * h + m);
        const float* iv = inv_sm + (nc % kAtI) * kAtN;
        for (int sc = 0; sc < n; sc += 32) {
          float2 s[16];
          tc_ld32(tcol + (uint32_t)sc, s);
          if (sc + 32 >= n) {  // the tile's last read of the accumulator has come back
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty(2 * h + m));
          }
          step(s, iv + sc, (uint32_t)(c0 + sc));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(inv_free(nc % kAtI));
      }
      // the two halves' candidates together (a barrier of the two warps that share these positions; half 0 writes
      // the other buffer for the next item)
      uint2* part = part_sm + 256 * (ni & 1) + 128 * m + 32 * q + lane;
      more = more || !ok;
      if (h == 0) *part = make_uint2(__float_as_uint(more ? -1.f : m1), i1 | (i2 << 16));
      asm volatile("bar.sync %0, 64;" ::"r"(1 + 4 * m + q) : "memory");
      if (h == 1 && p < it.S) {
        const uint2 o = *part;
        const float om = __uint_as_float(o.x);
        uint32_t word = 0xFFFFFFFFu;
        if (usable && !more && om >= 0.f) {
          if (m1 > om + marg) word = i1 | (i2 << 16);
          else if (om > m1 + marg) word = o.y;
          else if (i2 == 0xFFFFu && (o.y >> 16) == 0xFFFFu && fmaxf(m1, om) > marg) word = min(i1, o.y & 0xFFFFu) | (max(i1, o.y & 0xFFFFu) << 16);
        }
        (it.side ? w.st[1] : w.st[0])[p] = word;
      }
    }
    if (!ok) *failed = 1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tc_dealloc(tmem, 512);
}

// Exact x . x_a, summed j = 0 .. 127 in order (a product of two bf16 is exact, so the fused
// step rounds once, like a separate add).
__device__ double exact_dot(const uint4* x, const uint4* row, int a) {
  double s = 0.0;
  for (int c0 = 0; c0 < 16; c0 += 8) {
    uint4 xv[8], av[8];  // (loads in flight together)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      xv[c] = __ldg(x + c0 + c);
      av[c] = __ldg(row + ((c0 + c) ^ (a & 7)));
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t xw[4] = {xv[c].x, xv[c].y, xv[c].z, xv[c].w}, aw[4] = {av[c].x, av[c].y, av[c].z, av[c].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        s = __fma_rn(bf_f64(xw[e] << 16), bf_f64(aw[e] << 16), s);
        s = __fma_rn(bf_f64(xw[e] & 0xFFFF0000u), bf_f64(aw[e] & 0xFFFF0000u), s);
      }
    }
  }
  return s;
}

// Whether x == gamma x_a holds exactly in every dimension (a duplicate of its anchor): the
// fp32 products are exact when they are 0 or not below 2^-100.
__device__ bool exactly_zero_residual(const uint4* x, const uint4* row, int a, float g) {
  for (int c = 0; c < 16; ++c) {
    const uint4 xv = __ldg(x + c), av = __ldg(row + (c ^ (a & 7)));
    const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w}, aw[4] = {av.x, av.y, av.z, av.w};
    for (int e = 0; e < 8; ++e) {
      const float xe = (e & 1) ? bf_hi(xw[e >> 1]) : bf_lo(xw[e >> 1]);
      const float ae = (e & 1) ? bf_hi(aw[e >> 1]) : bf_lo(aw[e >> 1]);
      const float pe = __fmul_rn(g, ae);
      if (pe != xe || (fabsf(pe) < 0x1p-100f && g != 0.f && ae != 0.f)) return false;
    }
  }
  return true;
}

// Exact residual energy (Eq. 5's r in fp64, squares summed in order) of position row x under
// stream word st; the key that the slots are ranked by.
__device__ uint64_t exact_energy_key(const uint4* x, const uint4* row, uint32_t st, bool valid) {
  const int a = (int)(st & 0xFFFFu);
  const double g = fp16_bits_to_f64(st >> 16);
  double e = 0.0;
  for (int c = 0; c < 16; ++c) {
    const uint4 xv = __ldg(x + c), av = __ldg(row + (c ^ (a & 7)));
    const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w}, aw[4] = {av.x, av.y, av.z, av.w};
    for (int h = 0; h < 8; ++h) {
      const uint32_t xe = (h & 1) ? xw[h >> 1] & 0xFFFF0000u : xw[h >> 1] << 16;
      const uint32_t ae = (h & 1) ? aw[h >> 1] & 0xFFFF0000u : aw[h >> 1] << 16;
      const double pj = valid ? __dmul_rn(g, bf_f64(ae)) : 0.0;
      const double r = __dsub_rn(bf_f64(xe), pj);
      e = __dadd_rn(e, __dmul_rn(r, r));
    }
  }
  return (uint64_t)__double_as_longlong(e) + 1ull;
}

// Residual energy in fp32 as a key (bits + 1).  r = x - gamma x_a is one exactly rounded step and
// every square is positive, so the sum is within 2^-19 of the exact energy while it lies in
// [2^-90, 2^100]; an energy outside (and not exactly 0) sets the unit's fp64 flag.
constexpr float kEnLo = 0x1p-90f, kEnHi = 0x1p100f;
__device__ __forceinline__ uint32_t energy_key(float e, const uint4* x, const uint4* row, int a, float g, uint32_t* inexact) {
  if (!(e >= kEnLo && e <= kEnHi) && !(e == 0.f && exactly_zero_residual(x, row, a, g))) atomicOr(inexact, 1u);
  return __float_as_uint(e) + 1u;
}

// s + c += p with the rounding error kept in c (Knuth's two-sum): the sum of exact products in twice
// the precision of fp32.
__device__ __forceinline__ void two_sum_add(float& s, float& c, float p) {
  const float t = s + p, z = t - s;
  c += (s - (t - z)) + (p - z);
  s = t;
}

// gamma's fp16 bits where the fp32 quotient gq is within ge of one rounding boundary, the one between
// the neighbours gh and gh2 (at or below gq - ge and gq + ge): x . x_a = s + c against the boundary times
// |x_a|^2, both in twice the precision of fp32; false if even that does not decide.
__device__ bool gamma_at_edge(float s, float c, float ab, double n2, uint32_t gh2, uint32_t& gh) {
  const float nh = (float)n2, nl = (float)(n2 - (double)nh);
  const float mid = 0.5f * (__half2float(__ushort_as_half((unsigned short)gh)) + __half2float(__ushort_as_half((unsigned short)gh2)));
  const float pm = mid * nh, pe = __fmaf_rn(mid, nl, __fmaf_rn(mid, nh, -pm));
  const float diff = (s - pm) + (c - pe);
  // (errors of the sum, the product and the fp64 result that this stands for: below 2^-33 of each)
  if (!(fabsf(diff) > (ab + fabsf(pm)) * 0x1p-32f)) return false;
  if (diff > 0.f) gh = gh2;
  return true;
}

// Eq. 1 decided and Eq. 2: gamma = fp16(x . x_a / |x_a|^2), and the residual energy of every
// position.  Eight lanes take a position (16 dimensions each).  Two candidate anchors are told apart by
// their scores in fp32 unless those lie within their error (24 roundings of sum |x x_a|).  x . x_a in
// fp32 fixes gamma's fp16 rounding unless the quotient comes within its error of a rounding boundary;
// there the products are summed again in twice the precision and compared with the boundary times
// |x_a|^2.  What even that leaves (equal scores of duplicate anchors, mostly) and the positions with more
// candidates go to the unit's lists, which enc_undecided finishes in fp64.  fp64 for every position
// would be 335 M operations for the energies alone, 0.55 ms for 2 x 8 x 32768 positions, and a few fp64
// chains in every block (271 us for the kernel) cost as much as full warps of them.
constexpr int kFinPos = 256;  // positions per block
__global__ void __launch_bounds__(256) enc_finish(const EncArgs A) {
  __shared__ int todo[kFinPos], full[kFinPos];
  __shared__ int n_todo, n_full, at_todo, at_full;
  const int u = blockIdx.y, side = blockIdx.z;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, p0 = blockIdx.x * kFinPos;
  if (p0 >= S) return;
  const EncUnitWs w = unit_ws(A, u, d);
  const uint4* X = reinterpret_cast<const uint4*>((side ? A.V : A.K) + (size_t)u * A.s_max * 128);
  const uint4* AR = reinterpret_cast<const uint4*>(A.arena_c + (side ? d->off_anchor_v : d->off_anchor_k));
  uint32_t* stream = w.st[side];
  const float* inv = w.inv[side];
  const double* n2 = w.n2[side];
  uint32_t* key = reinterpret_cast<uint32_t*>(side ? w.key1 : w.key0);
  uint32_t* inexact = &w.ctrl[6 + side];
  const bool want_e = A.m_obs == 0;  // (the full selection ranks by its own utilities)
  const int tid = threadIdx.x, sub = tid & 7;
  if (tid == 0) n_todo = n_full = 0;
  __syncthreads();
  auto load16 = [](const uint4* lo, const uint4* hi, uint32_t (&o)[8]) {
    const uint4 v = __ldg(lo), t = __ldg(hi);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    o[4] = t.x; o[5] = t.y; o[6] = t.z; o[7] = t.w;
  };
  auto load_anchor = [&](int a, uint32_t (&o)[8]) {
    load16(AR + (size_t)a * 16 + ((2 * sub) ^ (a & 7)), AR + (size_t)a * 16 + ((2 * sub + 1) ^ (a & 7)), o);
  };
  auto dot = [](const uint32_t (&xw)[8], const uint32_t (&aw)[8], float& dd, float& ab) {  // and sum |x x_a|
    dd = ab = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      dd = __fmaf_rn(bf_lo(xw[c]), bf_lo(aw[c]), dd);
      dd = __fmaf_rn(bf_hi(xw[c]), bf_hi(aw[c]), dd);
      ab = __fmaf_rn(fabsf(bf_lo(xw[c])), fabsf(bf_lo(aw[c])), ab);
      ab = __fmaf_rn(fabsf(bf_hi(xw[c])), fabsf(bf_hi(aw[c])), ab);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      dd += __shfl_xor_sync(0xffffffffu, dd, o);
      ab += __shfl_xor_sync(0xffffffffu, ab, o);
    }
  };
  // a position's slot and candidate word are read one step ahead, so that its rows don't wait for them (8 units of
  // 32768 positions: 61 -> 55 us)
  int sl_n = 0;
  uint32_t word_n = 0u;
  auto read_word = [&](int q) {
    const bool in = q < kFinPos && p0 + q < S;
    sl_n = in ? w.slot_of[p0 + q] : 0;
    word_n = in ? stream[p0 + q] : 0u;
  };
  read_word(tid >> 3);
  for (int q = tid >> 3; q < kFinPos; q += 32) {
    const int p = p0 + q;
    const bool in = p < S;
    const int sl = sl_n;
    const uint32_t word = word_n;
    int a = (int)(word & 0xFFFFu);
    const int a2 = (int)(word >> 16);
    const bool some = in && sl < 0, lone = some && a2 != a;  // lone: one candidate, or two
    bool one = lone && a2 == 0xFFFF;
    uint32_t xw[8] = {}, aw[8] = {};
    if (lone) {
      load16(X + (size_t)p * 16 + 2 * sub, X + (size_t)p * 16 + 2 * sub + 1, xw);
      load_anchor(a, aw);
    }
    float iv = lone ? inv[a] : 0.f;
    read_word(q + 32);
    float dd, ab;
    dot(xw, aw, dd, ab);
    const bool two = lone && a2 != 0xFFFF;
    if (__any_sync(0xffffffffu, two)) {
      uint32_t bw[8] = {};
      if (two) load_anchor(a2, bw);
      const float iv2 = two ? inv[a2] : 0.f;
      float dd2, ab2;
      dot(xw, bw, dd2, ab2);
      // 19 roundings in a sum, two in its score
      const float gap = fabsf(dd) * iv - fabsf(dd2) * iv2, tol = (ab * iv + ab2 * iv2) * 0x1p-19f;
      if (two) {
        one = fabsf(gap) > tol;
        if (gap < 0.f) {
          a = a2;
          dd = dd2;
          ab = ab2;
          iv = iv2;
#pragma unroll
          for (int c = 0; c < 8; ++c) aw[c] = bw[c];
        }
      }
    }
    // gamma: 1 / |x_a|^2 from the inverse norm (dd 19 roundings, the quotient 5 more)
    const float i2 = iv * iv, gq = dd * i2, ge = ab * i2 * 0x1p-19f;
    uint32_t gh = f32_to_fp16_bits(gq - ge);
    const uint32_t gh2 = f32_to_fp16_bits(gq + ge);
    one = one && ab >= 0x1p-80f && ab <= 0x1p100f;
    bool fixed = one && gh == gh2;
    const bool edge = one && !fixed && (gq < 0.f ? gh == gh2 + 1u : gh2 == gh + 1u);  // one boundary in reach
    if (__any_sync(0xffffffffu, edge)) {
      float hs = 0.f, hc = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        two_sum_add(hs, hc, bf_lo(xw[c]) * bf_lo(aw[c]));  // (16-bit products: exact)
        two_sum_add(hs, hc, bf_hi(xw[c]) * bf_hi(aw[c]));
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const float os = __shfl_xor_sync(0xffffffffu, hs, o), oc = __shfl_xor_sync(0xffffffffu, hc, o);
        two_sum_add(hs, hc, os);
        hc += oc;
      }
      if (edge) {
        fixed = gamma_at_edge(hs, hc, ab, n2[a], gh2, gh);
      }
    }
    const float g = __half2float(__ushort_as_half((unsigned short)gh));
    float e = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float r0 = __fmaf_rn(-g, bf_lo(aw[c]), bf_lo(xw[c])), r1 = __fmaf_rn(-g, bf_hi(aw[c]), bf_hi(xw[c]));
      e = __fmaf_rn(r0, r0, e);
      e = __fmaf_rn(r1, r1, e);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (sub == 0 && in) {
      if (sl >= 0) {  // an anchor: its own slot, coefficient 1
        stream[p] = (uint32_t)sl | (0x3C00u << 16);
        if (want_e) key[p] = 0u;
      } else if (fixed) {
        stream[p] = (uint32_t)a | (gh << 16);
        if (want_e) key[p] = energy_key(e, X + (size_t)p * 16, AR + (size_t)a * 16, a, g, inexact);
      } else if (!lone) {
        full[atomicAdd(&n_full, 1)] = p;
      } else {
        todo[atomicAdd(&n_todo, 1)] = p;
      }
    }
  }
  __syncthreads();
  // the lists lie behind the energies: undecided positions from the front, the others from the back
  int* list = reinterpret_cast<int*>(key + S);
  if (tid == 0) {
    at_todo = n_todo ? (int)atomicAdd(&w.ctrl[8 + side], (uint32_t)n_todo) : 0;
    at_full = n_full ? (int)atomicAdd(&w.ctrl[10 + side], (uint32_t)n_full) : 0;
  }
  __syncthreads();
  for (int i = tid; i < n_todo; i += 256) list[at_todo + i] = todo[i];
  for (int i = tid; i < n_full; i += 256) list[S - 1 - (at_full + i)] = full[i];
}

// x . x_a by one thread in twice the precision of fp32 (s + c, within 128^2 2^-48 sum |x x_a|), and that sum.
__device__ void paired_dot(const uint4* x, const uint4* row, int a, float& s, float& c, float& ab) {
  s = c = ab = 0.f;
  for (int c0 = 0; c0 < 16; c0 += 8) {
    uint4 xv[8], av[8];  // (loads in flight together)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      xv[i] = __ldg(x + c0 + i);
      av[i] = __ldg(row + ((c0 + i) ^ (a & 7)));
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t xw[4] = {xv[i].x, xv[i].y, xv[i].z, xv[i].w}, aw[4] = {av[i].x, av[i].y, av[i].z, av[i].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float p0 = bf_lo(xw[e]) * bf_lo(aw[e]), p1 = bf_hi(xw[e]) * bf_hi(aw[e]);  // (exact)
        two_sum_add(s, c, p0);
        two_sum_add(s, c, p1);
        ab += fabsf(p0) + fabsf(p1);
      }
    }
  }
}

// |x . x_a| / |x_a| in fp32 for rows of any finite size, as enc_undecided's own score, within 2^-19 |x|: x comes scaled by
// a power of two to a largest component in [1, 2), and again by 2^64 and 2^-64 (xs[0 .. 2][128]) for anchors whose norm
// would take the products out of the range; the anchor's norm from the leading bits of its square.  0 for an anchor that
// cannot be the nearest (zero, or not finite).
__device__ __noinline__ float scaled_score(const float (*xs)[128], const uint4* row, int a, double n2) {
  const uint32_t hi = (uint32_t)__double2hiint(n2), lo = (uint32_t)__double2loint(n2);
  if (hi == 0u || hi >= 0x7FF00000u) return 0.f;
  const int e = (int)(hi >> 20) - 1023, h = e >> 1;  // |x_a| = sqrt(m) 2^h, m in [1, 4)
  const float m = __uint_as_float((uint32_t)(127 + (e & 1)) << 23 | (hi & 0xFFFFFu) << 3 | lo >> 29);
  const int cls = h < -60 ? 1 : (h > 60 ? 2 : 0), c = cls == 1 ? 64 : (cls == 2 ? -64 : 0);
  const float* x = xs[cls];
  float s = 0.f;
#pragma unroll 8
  for (int g = 0; g < 16; ++g) {
    const uint4 v = __ldg(row + (g ^ (a & 7)));
    const float* xc = x + 8 * g;
    float t = xc[0] * bf_lo(v.x);
    t = __fmaf_rn(xc[1], bf_hi(v.x), t);
    t = __fmaf_rn(xc[2], bf_lo(v.y), t);
    t = __fmaf_rn(xc[3], bf_hi(v.y), t);
    t = __fmaf_rn(xc[4], bf_lo(v.z), t);
    t = __fmaf_rn(xc[5], bf_hi(v.z), t);
    t = __fmaf_rn(xc[6], bf_lo(v.w), t);
    t = __fmaf_rn(xc[7], bf_hi(v.w), t);
    s += t;
  }
  return fabsf(s) * __frsqrt_rn(m) * __uint_as_float((uint32_t)(127 - h - c) << 23);
}

// The positions that enc_finish left.  First list: one or two candidate anchors, a thread each; second list: any
// anchor of a group of 32, or any at all, a block each.  Scores are told apart in fp32, then in twice its
// precision (as squares: dot^2 |other|^2), duplicates by their bytes; fp64 chains run only for what is
// left, since one of 128 steps takes about 10 us here.  Rows outside the filter's range are scaled first (8 units of 32768
// positions with one anchor of norm 2^-32 each, so that the filter is off: 11 ms; with fp64 scores for every
// position and anchor 160).
constexpr int kUndThreads = 128;
// Blocks per unit and side, a ninth of them for the first list: 72 in a large batch (24 units already start 3456),
// up to 576 for fewer than 8 units, whose lists are as long as their requests.  2 units of 131072 positions: 76 us with
// the 288 of this rule, 122 us with 72.
__host__ __device__ constexpr int und_first(int blocks) { return blocks / 9; }
inline int und_blocks(int units) { return 72 * std::min(8, std::max(1, 8 / std::max(1, units))); }
__global__ void __launch_bounds__(kUndThreads) enc_undecided(const EncArgs A) {
  __shared__ __align__(16) float xs[128], xs3[3][128];  // a position's row; scaled
  __shared__ float red[kUndThreads / 32];
  __shared__ int lowest;
  __shared__ double bcs[kUndThreads], bds[kUndThreads];
  __shared__ int bas[kUndThreads];
  const int u = blockIdx.y, side = blockIdx.z;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, k = d->n_anchors;
  const EncUnitWs w = unit_ws(A, u, d);
  const int n_todo = (int)w.ctrl[8 + side], n_full = (int)w.ctrl[10 + side];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_first = und_first((int)gridDim.x), b = (int)blockIdx.x;
  const bool second = b >= n_first;
  if (second ? n_full <= b - n_first : n_todo <= b * kUndThreads) return;
  const uint4* X = reinterpret_cast<const uint4*>((side ? A.V : A.K) + (size_t)u * A.s_max * 128);
  const uint4* AR = reinterpret_cast<const uint4*>(A.arena_c + (side ? d->off_anchor_v : d->off_anchor_k));
  uint32_t* stream = w.st[side];
  const double* n2 = w.n2[side];
  const float* inv = w.inv[side];
  uint32_t* key = reinterpret_cast<uint32_t*>(side ? w.key1 : w.key0);
  const int* list = reinterpret_cast<const int*>(key + S);
  uint32_t* inexact = &w.ctrl[6 + side];
  const bool want_e = A.m_obs == 0;

  auto store = [&](int p, int a, uint32_t gh) {  // nearest anchor a (-1: none) and gamma are known
    const int as = a >= 0 ? a : 0;
    stream[p] = (uint32_t)as | (gh << 16);
    if (!want_e) return;
    const float g = a >= 0 ? __half2float(__ushort_as_half((unsigned short)gh)) : 0.f;
    const uint4 *x = X + (size_t)p * 16, *row = AR + (size_t)as * 16;
    float e = 0.f;
#pragma unroll 4
    for (int c = 0; c < 16; ++c) {
      const uint4 xv = __ldg(x + c), av = __ldg(row + (c ^ (as & 7)));
      const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w}, aw[4] = {av.x, av.y, av.z, av.w};
      float ec = 0.f;  // (a sum per chunk keeps the rounding errors of the chain at 24)
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const float r0 = a >= 0 ? __fmaf_rn(-g, bf_lo(aw[h]), bf_lo(xw[h])) : bf_lo(xw[h]);
        const float r1 = a >= 0 ? __fmaf_rn(-g, bf_hi(aw[h]), bf_hi(xw[h])) : bf_hi(xw[h]);
        ec = __fmaf_rn(r0, r0, ec);
        ec = __fmaf_rn(r1, r1, ec);
      }
      e += ec;
    }
    key[p] = energy_key(e, x, row, as, g, inexact);
  };
  auto finish = [&](int p, int a, double dot) { store(p, a, a >= 0 ? f64_to_fp16_bits(__ddiv_rn(dot, n2[a])) : 0u); };
  auto in_range = [](float ab) { return ab >= 0x1p-80f && ab <= 0x1p100f; };
  // gamma and energy for nearest anchor a, x . x_a = hs + hc
  auto settle = [&](int p, int a, float hs, float hc, float ab) {
    const float iv = inv[a], i2 = iv * iv, gq = (hs + hc) * i2, ge = fabsf(gq) * 0x1p-20f + ab * i2 * 0x1p-33f;
    uint32_t gh = f32_to_fp16_bits(gq - ge);
    const uint32_t gh2 = f32_to_fp16_bits(gq + ge);
    bool fixed = in_range(ab) && iv > 0.f;
    if (fixed && gh != gh2) fixed = (gq < 0.f ? gh == gh2 + 1u : gh2 == gh + 1u) && gamma_at_edge(hs, hc, ab, n2[a], gh2, gh);
    if (fixed) store(p, a, gh);
    else finish(p, a, exact_dot(X + (size_t)p * 16, AR + (size_t)a * 16, a));
  };
  auto same_rows = [&](int a, int b) {
    bool same = true;
    for (int c = 0; c < 16; ++c) {
      const uint4 v = __ldg(AR + (size_t)a * 16 + (c ^ (a & 7))), o = __ldg(AR + (size_t)b * 16 + (c ^ (b & 7)));
      same = same && v.x == o.x && v.y == o.y && v.z == o.z && v.w == o.w;
    }
    return same;
  };
  if (!second) {
    for (int t = b * kUndThreads + tid; t < n_todo; t += n_first * kUndThreads) {
      const int p = list[t];
      const uint32_t word = stream[p];
      const int a1 = (int)(word & 0xFFFFu), a2 = (int)(word >> 16);
      const uint4* x = X + (size_t)p * 16;
      float s1, c1, ab1;
      paired_dot(x, AR + (size_t)a1 * 16, a1, s1, c1, ab1);
      if (a2 == 0xFFFF) {
        settle(p, a1, s1, c1, ab1);
        continue;
      }
      float s2, c2, ab2;
      paired_dot(x, AR + (size_t)a2 * 16, a2, s2, c2, ab2);
      const double d1 = (double)s1 + (double)c1, d2 = (double)s2 + (double)c2;
      const double q1 = d1 * d1 * n2[a2], q2 = d2 * d2 * n2[a1];
      // (a square is off by twice the dot's error times the dot)
      const bool told = in_range(ab1) && in_range(ab2) && fabs(q1 - q2) > 0x1p-31 * (fabs(d1) * (double)ab1 * n2[a2] + fabs(d2) * (double)ab2 * n2[a1]);
      if (told || same_rows(a1, a2)) {
        const bool first = told ? q1 > q2 : a1 < a2;
        settle(p, first ? a1 : a2, first ? s1 : s2, first ? c1 : c2, first ? ab1 : ab2);
        continue;
      }
      const double e1 = exact_dot(x, AR + (size_t)a1 * 16, a1), e2 = exact_dot(x, AR + (size_t)a2 * 16, a2);
      const double r1 = __ddiv_rn(fabs(e1), __dsqrt_rn(n2[a1])), r2 = __ddiv_rn(fabs(e2), __dsqrt_rn(n2[a2]));
      const bool first = r1 > r2 || (r1 == r2 && a1 < a2);
      finish(p, first ? a1 : a2, first ? e1 : e2);
    }
    return;
  }
  for (int t = b - n_first; t < n_full; t += (int)gridDim.x - n_first) {
    const int p = list[S - 1 - t];
    const uint32_t word = stream[p];
    const int a_lo = word == 0xFFFFFFFFu ? 0 : (int)(word & 0xFFE0u), a_hi = word == 0xFFFFFFFFu ? k : min(k, a_lo + 32);
    const uint4* x = X + (size_t)p * 16;
    __syncthreads();
    xs[tid] = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(x)[tid] << 16);
    if (tid == 0) lowest = 0x7FFFFFFF;
    float nx2 = xs[tid] * xs[tid];
    const bool zero = __syncthreads_and(xs[tid] == 0.f);
    for (int o = 16; o > 0; o >>= 1) nx2 += __shfl_xor_sync(0xffffffffu, nx2, o);
    if (lane == 0) red[warp] = nx2;
    __syncthreads();
    nx2 = (red[0] + red[1]) + (red[2] + red[3]);
    bool filter = !zero && nx2 >= (float)kNormLo && nx2 <= (float)kNormHi && w.ctrl[4 + side] == 0u;
    const bool scaled = !filter && !zero && __syncthreads_and(fabsf(xs[tid]) < INFINITY);
    if (scaled) {
      const uint32_t top = __reduce_max_sync(0xffffffffu, __float_as_uint(xs[tid]) & 0x7FFFFFFFu);
      __syncthreads();
      if (lane == 0) red[warp] = __uint_as_float(top);
      __syncthreads();
      int e;
      frexpf(fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3])), &e);
      const float v = ldexpf(xs[tid], 1 - e);  // (exact, or far below 2^-100)
      xs3[0][tid] = v;
      xs3[1][tid] = v * 0x1p64f;
      xs3[2][tid] = v * 0x1p-64f;
      nx2 = v * v;
      for (int o = 16; o > 0; o >>= 1) nx2 += __shfl_xor_sync(0xffffffffu, nx2, o);
      __syncthreads();
      if (lane == 0) red[warp] = nx2;
      __syncthreads();
      nx2 = (red[0] + red[1]) + (red[2] + red[3]);
      filter = true;
    }
    auto score = [&](int a) {  // fp32, within 2^-19 |x| of |x . x_a| / |x_a| (sums per chunk: 26 roundings)
      const uint4* row = AR + (size_t)a * 16;
      if (scaled) return scaled_score(xs3, row, a, n2[a]);
      float s = 0.f;
#pragma unroll 8
      for (int c = 0; c < 16; ++c) {
        const uint4 v = __ldg(row + (c ^ (a & 7)));
        const float* xc = xs + 8 * c;
        float e = xc[0] * bf_lo(v.x);
        e = __fmaf_rn(xc[1], bf_hi(v.x), e);
        e = __fmaf_rn(xc[2], bf_lo(v.y), e);
        e = __fmaf_rn(xc[3], bf_hi(v.y), e);
        e = __fmaf_rn(xc[4], bf_lo(v.z), e);
        e = __fmaf_rn(xc[5], bf_hi(v.z), e);
        e = __fmaf_rn(xc[6], bf_lo(v.w), e);
        e = __fmaf_rn(xc[7], bf_hi(v.w), e);
        s += e;
      }
      return fabsf(s) * inv[a];
    };
    // a thread's two largest scores, and its third; the block's largest and what comes near it
    float b1 = -1.f, b2 = -1.f, b3 = -1.f, near = 0.f;
    int j1 = -1, j2 = -1;
    if (filter) {
      for (int a = a_lo + tid; a < a_hi; a += kUndThreads) {
        const float v = score(a);
        if (v > b1) {
          b3 = b2; b2 = b1; b1 = v;
          j2 = j1; j1 = a;
        } else if (v > b2) {
          b3 = b2; b2 = v;
          j2 = a;
        } else {
          b3 = fmaxf(b3, v);
        }
      }
      float mx = b1;
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      __syncthreads();
      if (lane == 0) red[warp] = mx;
      __syncthreads();
      mx = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
      near = mx - 0x1p-17f * 1.001f * __fsqrt_rn(nx2);
      if (mx > 0x1p-14f * __fsqrt_rn(nx2)) {
        // a thread with three near the largest looks at all its anchors again, else at its two
        const bool crowd = b3 >= near;
        if (b1 < near) j1 = -1;
        if (b2 < near) j2 = -1;
        auto each = [&](auto&& f) {  // f(anchor) for the thread's near anchors
          if (crowd) {
            for (int a = a_lo + tid; a < a_hi; a += kUndThreads)
              if (score(a) >= near) f(a);
          } else {
            if (j1 >= 0) f(j1);
            if (j2 >= 0) f(j2);
          }
        };
        each([&](int a) { atomicMin(&lowest, a); });
        __syncthreads();
        const int a0 = lowest;
        bool same = true;  // one left, or copies of one row: the lowest slot is the nearest
        each([&](int a) { same = same && (a == a0 || same_rows(a, a0)); });
        if (__syncthreads_and(same)) {
          if (tid == 0) {
            float s, c, ab;
            paired_dot(x, AR + (size_t)a0 * 16, a0, s, c, ab);
            settle(p, a0, s, c, ab);
          }
          continue;
        }
        if (crowd) j1 = -3;
      } else {
        j1 = -2;  // every anchor of the thread
      }
    } else {
      j1 = -2;
    }
    double bc = -1.0, bd = 0.0;
    int ba = -1;
    auto try_anchor = [&](int a) {
      const double na = n2[a];
      if (na == 0.0) return;
      const double dot = exact_dot(x, AR + (size_t)a * 16, a);
      const double c = __ddiv_rn(fabs(dot), __dsqrt_rn(na));
      if (c > bc || (c == bc && a < ba)) {
        bc = c;
        bd = dot;
        ba = a;
      }
    };
    if (j1 == -3) {
      for (int a = a_lo + tid; a < a_hi; a += kUndThreads)
        if (score(a) >= near) try_anchor(a);
    } else if (j1 == -2) {
      // (every usable anchor scores 0 against a zero row: the thread's first one stands for it)
      for (int a = a_lo + tid; a < a_hi && !(zero && ba >= 0); a += kUndThreads) try_anchor(a);
    } else {
      if (j1 >= 0) try_anchor(j1);
      if (j2 >= 0) try_anchor(j2);
    }
    bcs[tid] = bc;
    bds[tid] = bd;
    bas[tid] = ba;
    __syncthreads();
    if (tid == 0) {  // the largest, ties to the lowest slot
      for (int i = 1; i < kUndThreads; ++i)
        if (bas[i] >= 0 && (ba < 0 || bcs[i] > bc || (bcs[i] == bc && bas[i] < ba))) {
          bc = bcs[i];
          bd = bds[i];
          ba = bas[i];
        }
      finish(p, ba, bd);
    }
  }
}

// ---- residual slots (plain encoder) ---------------------------------------------------
// Per unit and side the N positions with the largest energies (ties: lower position), by a cluster
// of kSelCtas CTAs that share out the positions and exchange counts through distributed shared
// memory.  A radix select (digits of 11, 11 and 10 bits) finds the N-th largest of the fp32 energies;
// those are within 2^-19 of the fp64 ones, so a position above (1 + 2^-16) of it is in, one below
// (1 - 2^-16) of it is out, and the few between are ranked by their exact fp64 energies.  (One CTA per
// unit over 64-bit keys took 84 + 99 us for the two sides of 8 x 32768 positions.)
__global__ void __cluster_dims__(kSelCtas, 1, 1) __launch_bounds__(kSelThreads) enc_slots(const EncArgs A) {
  namespace cg = cooperative_groups;
  __shared__ __align__(16) uint32_t hist[3][2048];
  __shared__ uint32_t wsum[kSelThreads / 32];
  __shared__ uint32_t found[3];
  __shared__ uint32_t cnt_hi, cnt_band;   // this CTA's positions above the band, and inside it
  __shared__ uint32_t n_app, n_list;      // slots written by this CTA; entries of the cluster's list (CTA 0)
  __shared__ int band[kSelBand];          // this CTA's positions inside the band
  __shared__ uint64_t lkey[kSelBand];     // CTA 0: every band position's exact key ...
  __shared__ int lpos[kSelBand];          // ... and position
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int u = blockIdx.x / kSelCtas, side = blockIdx.y;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, N = side ? d->n_res_v : d->n_res_k;
  const EncUnitWs w = unit_ws(A, u, d);
  const uint32_t* key = reinterpret_cast<const uint32_t*>(side ? w.key1 : w.key0);
  uint8_t* flag = w.flag[side];
  int32_t* rp = w.res_pos + (side ? d->n_res_k : 0);
  int lo, hi;
  cluster_share(S, rank, lo, hi);
  if (N == 0) {  // (the whole cluster)
    for (int p = lo + tid; p < hi; p += kSelThreads) flag[p] = 0;
    return;
  }
  if (w.ctrl[6 + side]) return;  // energies outside the fp32 range: enc_slots_exact
  for (int i = tid; i < 3 * 2048; i += kSelThreads) (&hist[0][0])[i] = 0u;
  if (tid == 0) cnt_hi = cnt_band = n_app = n_list = 0u;
  __syncthreads();
  // f(position, its key or 0 past the share), by whole warps; eight keys are read at a time (one at a time, the five
  // passes' reads took most of the kernel: 70 us, not 47, for 2 units of 131072 positions, 36, not 31, for 8 of 32768)
  auto each_key = [&](auto&& f) {
    for (int p0 = lo; p0 < hi; p0 += 8 * kSelThreads) {
      uint32_t v[8];
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const int p = p0 + x * kSelThreads + tid;
        v[x] = p < hi ? key[p] : 0u;
      }
#pragma unroll
      for (int x = 0; x < 8; ++x)
        if (p0 + x * kSelThreads < hi) f(p0 + x * kSelThreads + tid, v[x]);
    }
  };
  uint32_t prefix = 0, want = (uint32_t)N;
#pragma unroll 1
  for (int dg = 0; dg < 3; ++dg) {
    const int sh = dg == 0 ? 21 : (dg == 1 ? 10 : 0), bits = dg == 2 ? 10 : 11;
    each_key([&](int p, uint32_t v) {
      const bool in = p < hi && (dg == 0 || (v >> (sh + bits)) == prefix);
      const uint32_t digit = (v >> sh) & ((1u << bits) - 1u);
      if (dg == 0) {  // a few digits hold all the energies: equal ones of a warp are counted at once
        const unsigned peers = __match_any_sync(0xffffffffu, in ? digit : 0xFFFFFFFFu);
        if (in && (peers & ((1u << lane) - 1u)) == 0u) atomicAdd(&hist[dg][digit], (uint32_t)__popc(peers));
      } else if (in) {
        atomicAdd(&hist[dg][digit], 1u);
      }
    });
    cl.sync();
    uint32_t inside;
    prefix = (prefix << bits) | cluster_digit<true>(cl, hist[dg], wsum, found, want, &inside);
  }
  const uint32_t T = prefix;  // the N-th largest key; N <= S - k, so it is no anchor's (T >= 1)
  const float eT = __uint_as_float(T - 1u);
  const uint32_t k_lo = __float_as_uint(__fmul_rn(eT, 1.0f - 0x1p-16f)) + 1u;
  const uint32_t k_hi = __float_as_uint(__fmul_rn(eT, 1.0f + 0x1p-16f)) + 1u;
  each_key([&](int p, uint32_t v) {
    const unsigned above = __ballot_sync(0xffffffffu, v > k_hi);
    if (lane == 0 && above) atomicAdd(&cnt_hi, (uint32_t)__popc(above));
    if (v >= k_lo && v <= k_hi) {
      const uint32_t i = atomicAdd(&cnt_band, 1u);
      if (i < kSelBand) band[i] = p;
    }
  });
  cl.sync();
  uint32_t n_hi = 0, n_band = 0, hi_before = 0, band_before = 0;
  for (int r = 0; r < kSelCtas; ++r) {
    const uint32_t h = *cl.map_shared_rank(&cnt_hi, r), b = *cl.map_shared_rank(&cnt_band, r);
    if (r < rank) {
      hi_before += h;
      band_before += b;
    }
    n_hi += h;
    n_band += b;
  }
  const uint32_t need = (uint32_t)N - n_hi;  // of the band
  const bool all = need == n_band;           // the whole band is in
  const bool tied = eT == 0.f;               // every band energy is exactly 0: the lowest positions are in
  if (!all && !tied && n_band > kSelBand) {  // (the whole cluster) too many to rank here
    if (rank == 0 && tid == 0) atomicOr(&w.ctrl[6 + side], 1u);
    cl.sync();  // no CTA leaves while another may still read its counts
    return;
  }
  const uint32_t k_in = all ? k_lo : k_hi + 1u;
  const uint32_t at = all ? hi_before + band_before : hi_before;
  each_key([&](int p, uint32_t v) {
    const bool sel = p < hi && v >= k_in;
    const unsigned bal = __ballot_sync(0xffffffffu, sel);
    uint32_t i = 0;
    if (lane == 0 && bal) i = atomicAdd(&n_app, (uint32_t)__popc(bal));
    i = __shfl_sync(0xffffffffu, i, 0);
    if (p < hi) flag[p] = sel ? 1 : 0;
    if (sel) rp[at + i + __popc(bal & ((1u << lane) - 1u))] = p;
  });
  if (!all && tied) {  // in position order
    __syncthreads();
    if (tid == 0) {
      uint32_t i = band_before;
      for (int p = lo; p < hi && i < need; ++p)
        if (key[p] >= k_lo && key[p] <= k_hi) {
          flag[p] = 1;
          rp[n_hi + i++] = p;
        }
    }
  } else if (!all) {  // ranked by exact energies, ties to the lower position
    uint32_t* n0 = cl.map_shared_rank(&n_list, 0);
    uint64_t* k0 = cl.map_shared_rank(&lkey[0], 0);
    int* p0 = cl.map_shared_rank(&lpos[0], 0);
    const uint4* X = reinterpret_cast<const uint4*>((side ? A.V : A.K) + (size_t)u * A.s_max * 128);
    const uint4* AR = reinterpret_cast<const uint4*>(A.arena_c + (side ? d->off_anchor_v : d->off_anchor_k));
    const bool valid = w.ctrl[side] != 0u;
    const int mine = (int)cnt_band;  // (at most kSelBand = kSelThreads)
    uint64_t my_key = 0;
    const int my_pos = tid < mine ? band[tid] : -1;
    // 16 positions at a time: a warp squares a position's residual (four dimensions per lane), a lane sums
    // it in order, so that the serial part is 128 fp64 additions
    double* sq = reinterpret_cast<double*>(&hist[0][0]);  // [16][129]
    for (int b0 = 0; b0 < mine; b0 += kSelThreads / 32) {
      __syncthreads();
      if (b0 + warp < mine) {
        const int p = band[b0 + warp];
        const uint32_t st = w.st[side][p];
        const int a = (int)(st & 0xFFFFu);
        const double g = fp16_bits_to_f64(st >> 16);
        const uint2 xv = reinterpret_cast<const uint2*>(X + (size_t)p * 16)[lane];
        const uint2 av = reinterpret_cast<const uint2*>(AR + (size_t)a * 16 + ((lane >> 1) ^ (a & 7)))[lane & 1];
        const uint32_t xe[4] = {xv.x << 16, xv.x & 0xFFFF0000u, xv.y << 16, xv.y & 0xFFFF0000u};
        const uint32_t ae[4] = {av.x << 16, av.x & 0xFFFF0000u, av.y << 16, av.y & 0xFFFF0000u};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const double r = __dsub_rn(bf_f64(xe[e]), valid ? __dmul_rn(g, bf_f64(ae[e])) : 0.0);
          sq[warp * 129 + 4 * lane + e] = __dmul_rn(r, r);
        }
      }
      __syncthreads();
      if (tid >= b0 && tid < b0 + kSelThreads / 32 && tid < mine) {
        double e = 0.0;
        for (int j = 0; j < 128; ++j) e = __dadd_rn(e, sq[(tid - b0) * 129 + j]);
        my_key = (uint64_t)__double_as_longlong(e) + 1ull;
        const uint32_t i = atomicAdd(n0, 1u);
        k0[i] = my_key;
        p0[i] = my_pos;
      }
    }
    cl.sync();
    if (my_pos >= 0) {
      uint32_t before = 0;
      for (uint32_t i = 0; i < n_band; ++i) before += k0[i] > my_key || (k0[i] == my_key && p0[i] < my_pos);
      if (before < need) {
        flag[my_pos] = 1;
        rp[n_hi + before] = my_pos;
      }
    }
  }
  cl.sync();  // no CTA leaves while another may still read its shared memory
}
static_assert(kSelBand == kSelThreads, "a thread ranks one band position");

// The same from fp64 energies of every position, for the units and sides that enc_slots left (energies
// outside the fp32 range, or a band of more than kSelBand positions): one block each, else nothing.
__global__ void __launch_bounds__(1024) enc_slots_exact(const EncArgs A) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t bc[2];
  __shared__ int wt[33];
  const int u = blockIdx.x, side = blockIdx.y;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, N = side ? d->n_res_v : d->n_res_k;
  const EncUnitWs w = unit_ws(A, u, d);
  if (N == 0 || w.ctrl[6 + side] == 0u) return;
  uint64_t* key = side ? w.key1 : w.key0;
  // the fp32 keys lie where the first half of the fp64 ones go, so which positions are anchors (key 0;
  // the same for both sides) is taken from the stream words: an anchor's position is its slot's
  const int32_t* apos = reinterpret_cast<const int32_t*>(A.arena_c + d->off_anchor_pos);
  const uint4* X = reinterpret_cast<const uint4*>((side ? A.V : A.K) + (size_t)u * A.s_max * 128);
  const uint4* AR = reinterpret_cast<const uint4*>(A.arena_c + (side ? d->off_anchor_v : d->off_anchor_k));
  const bool valid = w.ctrl[side] != 0u;
  for (int p = threadIdx.x; p < S; p += blockDim.x) {
    const uint32_t st = w.st[side][p];
    key[p] = apos[st & 0xFFFFu] == p ? 0ull : exact_energy_key(X + (size_t)p * 16, AR + (size_t)(st & 0xFFFFu) * 16, st, valid);
  }
  __syncthreads();
  int32_t* rp = w.res_pos + (side ? d->n_res_k : 0);
  uint32_t need = 0;
  const uint64_t thr = block_select(key, S, (uint32_t)N, true, hist, bc, &need);
  int base = 0, eq_seen = 0;
  for (int c0 = 0; c0 < S; c0 += 1024) {
    const int p = c0 + threadIdx.x;
    const uint64_t kv = (p < S) ? key[p] : 0ull;
    const int is_eq = (p < S && kv == thr) ? 1 : 0;
    int eq_tot;
    const int eq_pre = block_scan_flag(is_eq, wt, &eq_tot);
    const int sel = p < S && (kv > thr || (is_eq && (uint32_t)(eq_seen + eq_pre) < need));
    eq_seen += eq_tot;
    int tot;
    const int pre = block_scan_flag(sel, wt, &tot);
    if (sel) rp[base + pre] = p;
    if (p < S) w.flag[side][p] = (uint8_t)sel;
    base += tot;
    __syncthreads();
  }
}

// Exclusive block scan of non-negative counts (1024 threads); returns the prefix and
// writes the block total to *total.
__device__ uint32_t block_scan_u32(uint32_t v, uint32_t* warp_tot, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t x = warp_tot[lane], xi = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, xi, o);
      if (lane >= o) xi += t;
    }
    warp_tot[lane] = xi - x;
    if (lane == 31) warp_tot[32] = xi;
  }
  __syncthreads();
  const uint32_t pre = warp_tot[warp] + incl - v;
  *total = warp_tot[32];
  __syncthreads();
  return pre;
}

// Stored order of one unit: positions sorted by value anchor slot, ties by position (a stable
// counting sort), by a cluster per unit.  Up to 128 warps take contiguous shares of the positions and
// count them by slot into a row of their own (rows [n_rows][k] over the energies, which are read no
// more; n_rows k 4 <= 16 S bytes); the rows' columns are then prefix-summed, and every warp scatters its share
// in order, 32 positions at a time, equal slots of a warp ranked by lane.  (One warp per unit doing
// the scatter took 357 us for 32768 positions and 1650 us for 131072.)
constexpr int kOrdWarps = kSelThreads / 32;  // per CTA
__global__ void __cluster_dims__(kSelCtas, 1, 1) __launch_bounds__(kSelThreads) enc_order(const EncArgs A) {
  namespace cg = cooperative_groups;
  __shared__ uint32_t part[8][64];
  __shared__ uint32_t cta_total;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int u = blockIdx.x / kSelCtas;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, k = d->n_anchors;
  const EncUnitWs w = unit_ws(A, u, d);
  const uint32_t* st = w.st[1];
  uint32_t* mat = reinterpret_cast<uint32_t*>(w.key0);
  const int n_rows = (int)min((long long)(kSelCtas * kOrdWarps), 4ll * S / k);
  const int row = rank * kOrdWarps + warp;
  const int per = (int)((((long long)S + n_rows - 1) / n_rows + 31) & ~31ll);
  const int lo = row < n_rows ? (int)min((long long)S, (long long)row * per) : S;
  const int hi = (int)min((long long)S, (long long)lo + per);
  uint32_t* mine = mat + (size_t)row * k;
  auto slot_at = [&](int p) { return p < hi ? (st[p] & 0xFFFFu) : 0xFFFFFFFFu; };  // of position p
  if (row < n_rows) {
    for (int a = lane; a < k; a += 32) mine[a] = 0u;
    __threadfence();
    __syncwarp();
    for (int p0 = lo; p0 < hi; p0 += 128) {
      uint32_t a[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) a[x] = slot_at(p0 + 32 * x + lane);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const unsigned peers = __match_any_sync(0xffffffffu, a[x]);
        if (a[x] != 0xFFFFFFFFu && (peers & ((1u << lane) - 1u)) == 0u) atomicAdd(&mine[a[x]], (uint32_t)__popc(peers));
      }
    }
  }
  cl.sync();
  // this CTA's slots [rank kper, ..): 64 at a time, eight threads per slot over the rows
  const int kper = (k + kSelCtas - 1) / kSelCtas, a_lo = min(k, rank * kper), a_hi = min(k, a_lo + kper);
  const int rper = (n_rows + 7) / 8;  // rows per thread, at most 16
  uint32_t base = 0;                  // tokens of the CTA's slots so far
  for (int a0 = a_lo; a0 < a_hi; a0 += 64) {
    const int a = a0 + (tid & 63), g = tid >> 6;
    uint32_t v[16], sum = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int r = g * rper + j;
      v[j] = j < rper && r < n_rows && a < a_hi ? __ldcg(mat + (size_t)r * k + a) : 0u;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) sum += v[j];
    part[g][tid & 63] = sum;
    __syncthreads();
    uint32_t before = 0, tot = 0;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const uint32_t c = part[x][tid & 63];
      before += x < g ? c : 0u;
      tot += c;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int r = g * rper + j;
      if (j < rper && r < n_rows && a < a_hi) __stcg(mat + (size_t)r * k + a, before);
      before += v[j];
    }
    // slot starts: the 64 totals scanned by the first two warps
    uint32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    __syncthreads();
    if (warp < 2 && lane == 31) part[0][warp] = incl;
    __syncthreads();
    if (warp < 2 && a < a_hi) __stcg(w.cursor + a, base + (warp == 1 ? part[0][0] : 0u) + incl - tot);
    base += part[0][0] + part[0][1];
    __syncthreads();
  }
  if (tid == 0) cta_total = base;
  cl.sync();
  if (tid == 0) {
    uint32_t t = 0;
    for (int r = 0; r < kSelCtas; ++r) {
      part[1][r] = t;
      t += *cl.map_shared_rank(&cta_total, r);
    }
  }
  __syncthreads();
  // 128 positions at a time, so that four updates are under way together: a row's updates of successive 32 positions
  // are ordered by the warp barrier between them, not by the values they return (2 units of 131072: 72 -> 65 us)
  for (int p0 = lo; p0 < hi; p0 += 128) {
    uint32_t a[4], at[4] = {0u, 0u, 0u, 0u};
    unsigned peers[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) a[x] = slot_at(p0 + 32 * x + lane);
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      peers[x] = __match_any_sync(0xffffffffu, a[x]);
      if (a[x] != 0xFFFFFFFFu && (peers[x] & ((1u << lane) - 1u)) == 0u) at[x] = atomicAdd(&mine[a[x]], (uint32_t)__popc(peers[x]));
      __syncwarp();
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int p = p0 + 32 * x + lane;
      at[x] = __shfl_sync(0xffffffffu, at[x], __ffs(peers[x]) - 1) + (uint32_t)__popc(peers[x] & ((1u << lane) - 1u));
      if (p < hi) {
        at[x] += __ldcg(w.cursor + a[x]) + part[1][a[x] / kper];
        w.perm[at[x]] = p;
        w.at[p] = (int32_t)at[x];
      }
    }
  }
  cl.sync();  // no CTA leaves while another may still read its total
}

__device__ __forceinline__ int tile_len(int S, int j) { return min(kTile, S - j * kTile); }

// Residual records of each tile and side (one thread per stored token).
__global__ void __launch_bounds__(kTile) enc_tile_count(const EncArgs A) {
  const int u = blockIdx.y, j = blockIdx.x;
  const akv_unit_desc* d = unit_desc(A, u);
  if (j >= d->n_tiles) return;
  EncUnitWs w = unit_ws(A, u, d);
  const int t = j * kTile + threadIdx.x;
  const int i = t < d->len ? w.perm[t] : -1;
  const uint32_t f = i >= 0 ? (w.flag[0][i] | (w.flag[1][i] << 1)) : 0u;
  const int nk = __syncthreads_count(f & 1u), nv = __syncthreads_count(f & 2u);
  if (threadIdx.x == 0) {
    w.tcnt[2 * j] = (uint32_t)nk;
    w.tcnt[2 * j + 1] = (uint32_t)nv;
  }
}

// Tile block offsets of every unit (one block per unit, a thread per tile).
__global__ void __launch_bounds__(1024) enc_tile_table(const EncArgs A) {
  __shared__ uint32_t wt[33];
  const int u = blockIdx.x;
  const akv_unit_desc* d = unit_desc(A, u);
  const EncUnitWs w = unit_ws(A, u, d);
  uint32_t* table = reinterpret_cast<uint32_t*>(A.arena + d->off_tile_table);
  uint32_t run = 0;
  for (int j0 = 0; j0 < d->n_tiles; j0 += 1024) {
    const int j = j0 + threadIdx.x;
    const bool in = j < d->n_tiles;
    const int n = in ? tile_len(d->len, j) : 0;
    const uint32_t bytes = in ? tile_block_bytes(n, (int)w.tcnt[2 * j], (int)w.tcnt[2 * j + 1]) : 0u;
    uint32_t tot;
    const uint32_t pre = block_scan_u32(bytes, wt, &tot);
    if (in) {
      table[j] = run + pre;
      // value slots of the tile's first and last stored tokens
      const int t0 = j * kTile, t1 = t0 + n - 1;
      table[d->n_tiles + 1 + j] = (w.st[1][w.perm[t0]] & 0xFFFFu) | ((w.st[1][w.perm[t1]] & 0xFFFFu) << 16);
    }
    run += tot;
  }
  if (threadIdx.x == 0) table[d->n_tiles] = run;
}

// Streams, bitmaps and rank words of one tile block (one thread per stored token).
__global__ void __launch_bounds__(kTile) enc_tile_fill(const EncArgs A) {
  __shared__ uint32_t halves[2][kTile / 32];
  const int u = blockIdx.y, j = blockIdx.x;
  const akv_unit_desc* d = unit_desc(A, u);
  if (j >= d->n_tiles) return;
  EncUnitWs w = unit_ws(A, u, d);
  const int n = tile_len(d->len, j), nw = (int)tile_words(n), n64 = 64 * nw;
  const uint32_t off = reinterpret_cast<const uint32_t*>(A.arena_c + d->off_tile_table)[j];
  uint8_t* blk = A.arena + d->off_tiles + off;
  uint32_t* kst = reinterpret_cast<uint32_t*>(blk);
  uint32_t* vst = kst + n64;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t f = 0;
  if (t < n) {
    const int i = w.perm[j * kTile + t];
    kst[t] = w.st[0][i];
    vst[t] = w.st[1][i];
    f = w.flag[0][i] | (w.flag[1][i] << 1);
    if (d->off_pos) reinterpret_cast<uint32_t*>(A.arena + d->off_pos)[j * kTile + t] = (uint32_t)i;  // RoPE positions
  }
  const unsigned bk = __ballot_sync(0xffffffffu, f & 1u), bv = __ballot_sync(0xffffffffu, f & 2u);
  if (lane == 0) {
    halves[0][warp] = bk;
    halves[1][warp] = bv;
  }
  __syncthreads();
  if (t < 2 * nw) {
    const int side = t / nw, wi = t % nw;
    uint64_t* bm = reinterpret_cast<uint64_t*>(blk + 8u * n64) + side * nw;
    uint16_t* rk = reinterpret_cast<uint16_t*>(blk + 8u * n64 + 16u * nw + side * round16(2u * nw));
    const uint64_t word = (uint64_t)halves[side][2 * wi] | ((uint64_t)halves[side][2 * wi + 1] << 32);
    bm[wi] = word;
    int before = 0;
    for (int x = 0; x < 2 * wi; ++x) before += __popc(halves[side][x]);
    rk[wi] = (uint16_t)before;
  }
}

// Scale, min and codes of one record, by a warp; lane l's four codes are those of dims 4 l .. 4 l + 3.
struct Quantized {
  uint32_t scale, min, byte;
};

// Quantized record in fp64: r = x - gamma x_a, v = H(s o r), quantize.  v: 128 doubles of shared memory.
__device__ Quantized quantize_exact(const EncArgs& A, const __nv_bfloat16* X, const __nv_bfloat16* XA, double g, bool valid,
                                    double* v) {
  const int lane = threadIdx.x & 31;
  for (int j = lane; j < 128; j += 32) {
    const double pj = valid ? __dmul_rn(g, bf16_to_f64(XA[j])) : 0.0;
    double r = __dsub_rn(bf16_to_f64(X[j]), pj);
    if (A.rotate) {
      const unsigned long long sb = j < 64 ? A.sign_lo : A.sign_hi;
      if ((sb >> (j & 63)) & 1ull) r = -r;
    }
    v[j] = r;
  }
  __syncwarp();
  if (A.rotate) {
    for (int hh = 1; hh < 128; hh <<= 1) {
      for (int pr = lane; pr < 64; pr += 32) {
        const int j = (pr / hh) * 2 * hh + (pr % hh);
        const double x = v[j], y = v[j + hh];
        v[j] = __dadd_rn(x, y);
        v[j + hh] = __dsub_rn(x, y);
      }
      __syncwarp();
    }
  }
  uint32_t mnh, sch, byte = 0;
  if (A.lloyd) {
    // Lloyd-Max codec (Section 3.1, Appendix A.1): per-token RMS scale fp16(sqrt(sum v^2 / 128)),
    // the sum in index order (lane 0), min 0, codes by the decision regions of v / scale
    double ss = 0.0;
    if (lane == 0)
      for (int j = 0; j < 128; ++j) ss = __dadd_rn(ss, __dmul_rn(v[j], v[j]));
    ss = __shfl_sync(0xffffffffu, ss, 0);
    sch = f64_to_fp16_bits(__dsqrt_rn(__ddiv_rn(ss, 128.0)));
    mnh = 0u;
    const double sc = fp16_bits_to_f64(sch);
    for (int c = 0; c < 4; ++c) {
      int code = 2;  // a zero scale: every level reconstructs 0
      if (sc != 0.0) {
        const double t = __ddiv_rn(v[4 * lane + c], sc);
        code = t < -kLloydT ? 0 : (t < 0.0 ? 1 : (t < kLloydT ? 2 : 3));
      }
      byte |= (uint32_t)code << (2 * c);
    }
  } else {
    // min / max with the first index winning ties (as a sequential scan does)
    double mnv = v[4 * lane], mxv = mnv;
    int mni = 4 * lane, mxi = mni;
    for (int c = 1; c < 4; ++c) {
      const double x = v[4 * lane + c];
      if (x < mnv) { mnv = x; mni = 4 * lane + c; }
      if (x > mxv) { mxv = x; mxi = 4 * lane + c; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double omn = __shfl_xor_sync(0xffffffffu, mnv, o);
      const int omi = __shfl_xor_sync(0xffffffffu, mni, o);
      const double omx = __shfl_xor_sync(0xffffffffu, mxv, o);
      const int oxi = __shfl_xor_sync(0xffffffffu, mxi, o);
      if (omn < mnv || (omn == mnv && omi < mni)) { mnv = omn; mni = omi; }
      if (omx > mxv || (omx == mxv && oxi < mxi)) { mxv = omx; mxi = oxi; }
    }
    mnh = f64_to_fp16_bits(mnv);
    const double mn = fp16_bits_to_f64(mnh);
    double t = __ddiv_rn(__dsub_rn(mxv, mn), 3.0);
    if (!(t > 0.0)) t = 0.0;
    sch = f64_to_fp16_bits(t);
    const double sc = fp16_bits_to_f64(sch);
    for (int c = 0; c < 4; ++c) {
      int code = 0;
      if (sc != 0.0) {
        double qv = rint(__ddiv_rn(__dsub_rn(v[4 * lane + c], mn), sc));
        qv = fmin(fmax(qv, 0.0), 3.0);
        code = (int)qv;
      }
      byte |= (uint32_t)code << (2 * c);
    }
  }
  return Quantized{sch, mnh, byte};
}

// The same in fp32, where its error bounds decide every rounding; false (for the whole warp) where one does
// not.  r is one exactly rounded step; each of the seven butterfly stages rounds values whose sum of
// magnitudes is at most L1 = sum |r|, so v is within 8 x 2^-24 L1 of the exact transform (err below: 2 % more).  A value
// within err of a rounding boundary (fp16 min and scale, code regions) leaves the record to quantize_exact, about one
// record in a hundred.  (fp64 for every record took 457 us for 52,000 records: the fp64 units issue one warp instruction
// in 64 cycles; this takes 58, Lloyd-Max records of 24 short units 31, not 36 with their scales from the rotated sums.)
__device__ bool quantize_fast(const EncArgs& A, const uint2 xr, const uint2 ar, float g, bool valid, Quantized* q) {
  const int lane = threadIdx.x & 31;
  const uint32_t xw[4] = {xr.x << 16, xr.x & 0xFFFF0000u, xr.y << 16, xr.y & 0xFFFF0000u};
  const uint32_t aw[4] = {ar.x << 16, ar.x & 0xFFFF0000u, ar.y << 16, ar.y & 0xFFFF0000u};
  float v[4], l1 = 0.f, rr = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    v[e] = __uint_as_float(xw[e]);
    if (valid) v[e] = __fmaf_rn(-g, __uint_as_float(aw[e]), v[e]);
    l1 += fabsf(v[e]);
    rr = __fmaf_rn(v[e], v[e], rr);
    if (A.rotate) {
      const unsigned long long sb = lane < 16 ? A.sign_lo : A.sign_hi;
      if ((sb >> ((4 * lane + e) & 63)) & 1ull) v[e] = -v[e];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  if (!(l1 >= 0x1p-40f && l1 <= 0x1p60f)) return false;  // (sums of squares stay normal)
  // one rounding of the residual and seven of the butterflies, each at most 2^-24 of the sum of magnitudes that it is
  // part of; the rest for l1's own and second-order terms
  const float err = l1 * (1.02f * 0x1p-21f);
  if (A.rotate) {
    const float b0 = v[0] + v[1], b1 = v[0] - v[1], b2 = v[2] + v[3], b3 = v[2] - v[3];
    v[0] = b0 + b2;
    v[1] = b1 + b3;
    v[2] = b0 - b2;
    v[3] = b1 - b3;
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
      const float sg = (lane & m) ? -1.f : 1.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = __fmaf_rn(sg, v[e], __shfl_xor_sync(0xffffffffu, v[e], m));
    }
  }
  bool sure = true;
  q->byte = 0;
  if (A.lloyd) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rr += __shfl_xor_sync(0xffffffffu, rr, o);
    // sum v^2 / 128 is sum r^2 (the transform keeps it, times 128; without it the mean is taken): each residual rounded
    // once, nine roundings of the sum, so off by 2^-20.4 of it; the root adds two more.  (Summed after the rotation, whose
    // errors are not each value's own, 10 % of the scales were left to fp64.)
    const float ms = A.rotate ? rr : rr * 0.0078125f, es = ms * 0x1p-20f;
    q->min = 0u;
    q->scale = f32_to_fp16_bits(__fsqrt_rn(ms - es) * (1.f - 0x1p-22f));
    sure = q->scale == f32_to_fp16_bits(__fsqrt_rn(ms + es) * (1.f + 0x1p-22f));
    const float sc = __half2float(__ushort_as_half((unsigned short)q->scale));
    const float T = (float)kLloydT;
    if (sc == 0.f) {
      q->byte = 0xAAu;  // a zero scale: code 2 everywhere
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float t = __fdiv_rn(v[e], sc), et = __fdiv_rn(err, sc) + fabsf(t) * 0x1p-22f;
        sure = sure && fabsf(fabsf(t) - T) > et && fabsf(t) > et;
        q->byte |= (t < -T ? 0u : (t < 0.f ? 1u : (t < T ? 2u : 3u))) << (2 * e);
      }
    }
  } else {
    float mn = fminf(fminf(v[0], v[1]), fminf(v[2], v[3])), mx = fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    q->min = f32_to_fp16_bits(mn - err);
    sure = q->min == f32_to_fp16_bits(mn + err);
    const float m16 = __half2float(__ushort_as_half((unsigned short)q->min));
    const float t = __fdiv_rn(mx - m16, 3.f), et = err + fabsf(t) * 0x1p-22f;  // (a third of err, rounded up)
    sure = sure && t > et;
    q->scale = f32_to_fp16_bits(t - et);
    sure = sure && q->scale == f32_to_fp16_bits(t + et);
    const float sc = __half2float(__ushort_as_half((unsigned short)q->scale));
    if (sc != 0.f) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float c = __fdiv_rn(v[e] - m16, sc), ec = __fdiv_rn(err, sc) + (fabsf(c) + fabsf(__fdiv_rn(m16, sc))) * 0x1p-22f;
        const float f = floorf(c);
        sure = sure && fabsf(c - f - 0.5f) > ec;
        q->byte |= (uint32_t)fminf(fmaxf(rintf(c), 0.f), 3.f) << (2 * e);
      }
    }
  }
  return __all_sync(0xffffffffu, sure);
}

// One warp per residual slot: its scale, min and codes into its tile.
__global__ void __launch_bounds__(256) enc_quant(const EncArgs A) {
  __shared__ double vbuf[8][128];
  const int u = blockIdx.y, side = blockIdx.z;
  const akv_unit_desc* d = unit_desc(A, u);
  EncUnitWs w = unit_ws(A, u, d);
  // slots of this unit: the parameters' count, or the count the full selection chose
  const int N = A.m_obs > 0 ? (int)w.ctrl[2 + side] : (side ? d->n_res_v : d->n_res_k);
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = blockIdx.x * 8 + wi;
  if (s >= N) return;
  const int p = w.res_pos[(side ? d->n_res_k : 0) + s];
  const uint32_t st = w.st[side][p];
  const int a = (int)(st & 0xFFFFu);
  const bool valid = w.ctrl[side] != 0u;
  const __nv_bfloat16* X = (side ? A.V : A.K) + ((size_t)u * A.s_max + p) * 128;
  const uint8_t* row = A.arena_c + (side ? d->off_anchor_v : d->off_anchor_k) + (size_t)a * 256;
  Quantized q;
  if (!quantize_fast(A, *reinterpret_cast<const uint2*>(X + 4 * lane),
                     *reinterpret_cast<const uint2*>(row + 16 * ((lane >> 1) ^ (a & 7)) + 8 * (lane & 1)),
                     __half2float(__ushort_as_half((unsigned short)(st >> 16))), valid, &q))
    q = quantize_exact(A, X, anchor_src(A, u, side, reinterpret_cast<const int32_t*>(A.arena_c + d->off_anchor_pos), a),
                       fp16_bits_to_f64(st >> 16), valid, vbuf[wi]);
  const uint32_t mnh = q.min, sch = q.scale, byte = q.byte;
  // record r of its tile: the rank of the token among the tile's tokens with this side's bit
  const int ts = w.at[p], j = ts / kTile, tl = ts % kTile;
  const int n = tile_len(d->len, j), nw = (int)tile_words(n), n64 = 64 * nw;
  const int nkj = (int)w.tcnt[2 * j], nvj = (int)w.tcnt[2 * j + 1];
  const uint8_t* blkc = A.arena_c + d->off_tiles + reinterpret_cast<const uint32_t*>(A.arena_c + d->off_tile_table)[j];
  const uint64_t word = reinterpret_cast<const uint64_t*>(blkc + 8u * n64)[side * nw + (tl >> 6)];
  const uint16_t* rk = reinterpret_cast<const uint16_t*>(blkc + 8u * n64 + 16u * nw + side * round16(2u * nw));
  const int r = (int)rk[tl >> 6] + __popcll(word & ((1ull << (tl & 63)) - 1ull));
  const uint32_t F = tile_fixed_bytes(n);
  const uint32_t sm_off = F + (side ? round16(4u * (uint32_t)nkj) : 0u) + 4u * (uint32_t)r;
  const uint32_t cd_off = F + round16(4u * (uint32_t)nkj) + round16(4u * (uint32_t)nvj) +
                          (side ? 32u * (uint32_t)nkj : 0u) + 32u * (uint32_t)r;
  uint8_t* blk = const_cast<uint8_t*>(blkc);
  if (side == 0) {
    blk[cd_off + lane] = (uint8_t)byte;
  } else {  // value codes: dimension-major groups of 16 records
    uint32_t* grp = reinterpret_cast<uint32_t*>(blk + cd_off - 32u * (uint32_t)r + 512u * (uint32_t)(r / 16));
    for (int c = 0; c < 4; ++c)
      atomicOr(&grp[value_code_word(4 * lane + c)], ((byte >> (2 * c)) & 3u) << value_code_bit(r % 16));
  }
  if (lane == 0) *reinterpret_cast<uint32_t*>(blk + sm_off) = sch | (mnh << 16);
}

// ---- the paper's full selection (Algorithm 1; Section 3.2-3.4, Appendix A.2) --------------
// Each fp64 sum runs in a fixed order (positions, then rows, then dimensions ascending, one
// thread per output), and the exponential is evaluated by fixed steps, so every decision
// (scored anchors, pooled residual slots) comes out the same on any IEEE machine.

// e^x for x <= 0: Cody-Waite argument reduction (ln 2 split into a 42-bit leading part,
// whose product with n is exact, and the remainder), a degree-22 Taylor series of e^r by
// Horner's rule, then the exact scaling by 2^n; about 1 ulp.  Arguments below -700 give 0.
__device__ double exp_neg_dev(double x) {
  if (!(x >= -700.0)) return 0.0;
  const double ln2_hi = 0.693147180559890330187045037746429443359375;
  const double ln2_lo = 5.4979230187083711552420206887987e-14;
  const double n = rint(__ddiv_rn(x, 0.6931471805599453094172321));
  const double r = __dsub_rn(__dsub_rn(x, __dmul_rn(n, ln2_hi)), __dmul_rn(n, ln2_lo));
  double y = 1.0;
  for (int j = 22; j >= 1; --j) y = __dadd_rn(1.0, __dmul_rn(__ddiv_rn(r, (double)j), y));
  return ldexp(y, (int)n);
}

// ---- the full selection's sums in paired fp32 -------------------------------------------
// Scores and utilities only rank positions, so they are first taken with known errors: the inner
// products over 128 dimensions in twice the precision of fp32 (two_sum_add: the fp64 unit would need 64
// cycles per warp instruction for 1.6 G of them per 8 heads x 4096 positions x 128 rows), the rest in
// fp64.  A chain of n paired steps is within n^2 2^-48 of the sum of the terms' magnitudes (2^-34 for
// n = 128).  A ranking stands if the lowest selected value less its error exceeds the largest unselected
// one plus its own; else the unit's or request's flag has the exact kernels below repeat it (equal
// values, in practice).  ctrl[16]: scores undecided, [17 .. 19]: the largest squared norm of the
// observation rows, keys and values (fp32 bits), [12 + side] of a request's first unit: utilities undecided.
constexpr int kObsRows = 32;  // rows per block of the logits

// the largest squared norms and the outputs' sums start at zero
__global__ void __launch_bounds__(256) enc_obs_init(const EncArgs A) {
  const int u = blockIdx.x;
  const EncUnitWs w = unit_ws(A, u, unit_desc(A, u));
  if (threadIdx.x < 16) w.ctrl[16 + threadIdx.x] = 0u;
  for (int e = threadIdx.x; e < A.m_obs * 128; e += 256) w.yobs[e] = 0.0;
}

__device__ __forceinline__ double pair_f64(float s, float c) { return (double)s + (double)c; }
// The relative error of the observation rows' attention: twice a logit's error, for numerator and sum.
__device__ __forceinline__ float alpha_error(const EncUnitWs& w) {
  return 4.f * 0x1p-34f * 0.0885f * __fsqrt_rn(__uint_as_float(w.ctrl[17])) * __fsqrt_rn(__uint_as_float(w.ctrl[18])) + 0x1p-34f;
}
// Squared norms that keep every fp32 product of the kernels below from overflowing; and a norm from its fp32 square,
// rounded up by what squares below the fp32 range (2^-149 each) may have lost.
__device__ __forceinline__ bool norm_ok(float n2) { return n2 <= 0x1p60f; }
__device__ __forceinline__ float norm_up(float n2) { return __fsqrt_rn(n2 + 0x1p-140f); }

// Logits q_w . K_t / sqrt(D): a thread takes one position and eight rows at a time.
__global__ void __launch_bounds__(128) enc_obs_logit_f(const EncArgs A) {
  __shared__ __align__(16) uint4 ks[128][17];
  __shared__ __align__(16) float qs[8][128];
  const int u = blockIdx.y;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, t0 = blockIdx.x * 128, tid = threadIdx.x, t = t0 + tid;
  if (t0 >= S) return;
  const EncUnitWs w = unit_ws(A, u, d);
  const uint4* K = reinterpret_cast<const uint4*>(A.K + (size_t)u * A.s_max * 128);
  for (int e = tid; e < 128 * 16; e += 128)
    ks[e >> 4][e & 15] = t0 + (e >> 4) < S ? __ldg(K + (size_t)t0 * 16 + e) : make_uint4(0u, 0u, 0u, 0u);
  const double rs = __ddiv_rn(1.0, __dsqrt_rn(128.0));
  const int w1 = min(A.m_obs, (int)(blockIdx.z + 1) * kObsRows);
  float kn = 0.f;
  for (int w0 = blockIdx.z * kObsRows; w0 < w1; w0 += 8) {
    __syncthreads();
    for (int e = tid; e < 8 * 128; e += 128)
      qs[e >> 7][e & 127] = w0 + (e >> 7) < w1 ? __bfloat162float(A.Q[((size_t)u * A.m_obs + w0) * 128 + e]) : 0.f;
    __syncthreads();
    float s[8] = {}, c[8] = {};
    kn = 0.f;
    for (int g = 0; g < 16; ++g) {
      const uint4 v = ks[tid][g];
      const float k[8] = {bf_lo(v.x), bf_hi(v.x), bf_lo(v.y), bf_hi(v.y), bf_lo(v.z), bf_hi(v.z), bf_lo(v.w), bf_hi(v.w)};
#pragma unroll
      for (int j = 0; j < 8; ++j) kn = __fmaf_rn(k[j], k[j], kn);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float4 a = *reinterpret_cast<const float4*>(&qs[r][8 * g]), b = *reinterpret_cast<const float4*>(&qs[r][8 * g + 4]);
        const float q[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) two_sum_add(s[r], c[r], q[j] * k[j]);
      }
    }
    if (t < S)
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (w0 + r < w1) w.alpha[(size_t)(w0 + r) * S + t] = pair_f64(s[r], c[r]) * rs;
    if (tid < 8) {
      float qn = 0.f;
      for (int j = 0; j < 128; ++j) qn = __fmaf_rn(qs[tid][j], qs[tid][j], qn);
      atomicMax(&w.ctrl[17], __float_as_uint(qn < INFINITY ? qn : INFINITY));
    }
  }
  if (blockIdx.z == 0) atomicMax(&w.ctrl[18], __float_as_uint(kn < INFINITY ? kn : INFINITY));
}

// e^x for x <= 0 to 2^-43.5 (largest error seen over [-700, 0]: 2^-43.7): 2^(n / 512) from a table times e^r, r = x - n ln 2 / 512, |r| < 0.0007: r itself in fp64, the
// rest of e^r - 1 (below 2.5e-7) in fp32.  The fp64 unit is what bounds the kernel below (a warp instruction per 64
// cycles and scheduler, 85 % busy): 137 us for 8 units of 128 rows and 4096 positions, 203 us with a degree-10 series on
// |r| < 0.35 (2^-41.6).
__constant__ double kExp32[32] = {  // 2^(i / 32)
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0,
    0x1.172b83c7d517bp+0, 0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0,
    0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0, 0x1.3dea64c123422p+0, 0x1.44e086061892dp+0,
    0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0, 0x1.6247eb03a5585p+0,
    0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0,
    0x1.ae89f995ad3adp+0, 0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0,
    0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0, 0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0,
};
__constant__ double kExp512[16] = {  // 2^(i / 512)
    0x1.0000000000000p+0, 0x1.0058c86da1c0ap+0, 0x1.00b1afa5abcbfp+0, 0x1.010ab5b2cbd11p+0,
    0x1.0163da9fb3335p+0, 0x1.01bd1e77170b4p+0, 0x1.02168143b0281p+0, 0x1.027003103b10ep+0,
    0x1.02c9a3e778061p+0, 0x1.032363d42b027p+0, 0x1.037d42e11bbccp+0, 0x1.03d7411915a8ap+0,
    0x1.04315e86e7f85p+0, 0x1.048b9b35659d8p+0, 0x1.04e5f72f654b1p+0, 0x1.0540727fc1762p+0,
};
__device__ __forceinline__ double exp_neg_f(double x, const double* tab) {
  const float xf = (float)x;
  if (!(xf >= -700.f)) return 0.0;
  const float nf = rintf(xf * 738.65988f);  // 512 / ln 2
  const int n = (int)nf;
  const double r = fma((double)nf, -0.69314718055994530942 / 512.0, x);
  const float rf = (float)r, c = rf * rf * __fmaf_rn(rf, __fmaf_rn(rf, 1.f / 24.f, 1.f / 6.f), 0.5f);
  const double y = tab[n & 511];
  const double e = fma(y, r + (double)c, y);
  return __hiloint2double(__double2hiint(e) + ((n >> 9) << 20), __double2loint(e));  // (2^-1010 and above: normal)
}

// Softmax of each observation row over all positions (one block per row, sums as a tree).
__global__ void __launch_bounds__(512) enc_obs_softmax_f(const EncArgs A) {
  __shared__ double red[16], tab[512];
  const int u = blockIdx.y, wr = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len;
  double* a = unit_ws(A, u, d).alpha + (size_t)wr * S;
  tab[threadIdx.x] = kExp32[threadIdx.x >> 4] * kExp512[threadIdx.x & 15];
  // (a maximum good to fp32 keeps e^(x - max) below e^1: the quotient does not depend on it)
  float mf = -INFINITY;
  for (int t = threadIdx.x; t < S; t += 512) mf = fmaxf(mf, (float)a[t]);
  for (int o = 16; o > 0; o >>= 1) mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
  if (lane == 0) red[warp] = (double)mf;
  __syncthreads();
  double mx = red[0];
  for (int i = 1; i < 16; ++i) mx = red[i] > mx ? red[i] : mx;
  __syncthreads();
  double sum = 0.0;
  for (int t = threadIdx.x; t < S; t += 512) {
    const double e = exp_neg_f(a[t] - mx, tab);
    a[t] = e;
    sum += e;
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) red[warp] = sum;
  __syncthreads();
  sum = 0.0;
  for (int i = 0; i < 16; ++i) sum += red[i];
  const double f = 1.0 / sum;
  for (int t = threadIdx.x; t < S; t += 512) a[t] *= f;
}

// Outputs y_w = sum_t alpha_wt V_t: a block takes 256 positions and eight rows, a thread one dimension.
constexpr int kObsChunk = 256;
__global__ void __launch_bounds__(128) enc_obs_y_f(const EncArgs A) {
  __shared__ __align__(16) float2 as[kObsChunk][8];
  __shared__ float vn[4];
  const int u = blockIdx.z, tid = threadIdx.x, t0 = blockIdx.x * kObsChunk, w0 = blockIdx.y * 8;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len;
  if (t0 >= S) return;
  const EncUnitWs w = unit_ws(A, u, d);
  const int n = min(kObsChunk, S - t0);
  for (int r = 0; r < 8; ++r)
    for (int t = tid; t < kObsChunk; t += 128) {
      const double a = t < n && w0 + r < A.m_obs ? w.alpha[(size_t)(w0 + r) * S + t0 + t] : 0.0;
      const float hi = (float)a;
      as[t][r] = make_float2(hi, (float)(a - (double)hi));
    }
  __syncthreads();
  const __nv_bfloat16* V = A.V + ((size_t)u * A.s_max + t0) * 128 + tid;
  float s[8] = {}, c[8] = {};
#pragma unroll 4
  for (int t = 0; t < n; ++t) {
    const float v = __bfloat162float(V[(size_t)t * 128]);
#pragma unroll
    for (int r = 0; r < 8; r += 2) {
      const float4 a = *reinterpret_cast<const float4*>(&as[t][r]);
      const float p0 = a.x * v, p1 = a.z * v;
      c[r] += __fmaf_rn(a.x, v, -p0);
      c[r + 1] += __fmaf_rn(a.z, v, -p1);
      two_sum_add(s[r], c[r], p0);
      two_sum_add(s[r + 1], c[r + 1], p1);
      c[r] = __fmaf_rn(a.y, v, c[r]);
      c[r + 1] = __fmaf_rn(a.w, v, c[r + 1]);
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r)
    if (w0 + r < A.m_obs) atomicAdd(&w.yobs[(w0 + r) * 128 + tid], pair_f64(s[r], c[r]));
  if (w0 == 0) {  // the largest squared norm of the values
    float mx = 0.f;
    for (int t = tid >> 5; t < n; t += 4) {
      const uint2 x = *reinterpret_cast<const uint2*>(A.V + ((size_t)u * A.s_max + t0 + t) * 128 + 4 * (tid & 31));
      float q = bf_lo(x.x) * bf_lo(x.x) + bf_hi(x.x) * bf_hi(x.x) + bf_lo(x.y) * bf_lo(x.y) + bf_hi(x.y) * bf_hi(x.y);
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      mx = fmaxf(mx, q < INFINITY ? q : INFINITY);
    }
    if ((tid & 31) == 0) vn[tid >> 5] = mx;
    __syncthreads();
    if (tid == 0) atomicMax(&w.ctrl[19], __float_as_uint(fmaxf(fmaxf(vn[0], vn[1]), fmaxf(vn[2], vn[3]))));
  }
}

// Eq. 6 utilities of 32 positions: key0 = bits(u^K) + 1, key1 = bits(u^V) + 1, anchors 0, and the error of u^K (fp64,
// over perm and at; absolute, since |V - y|^2 may come out at or below 0 where V is close to y; infinite: no bound for
// either utility).  Thread (position, group g of eight): rows g and g + 8 of every sixteen.  With r the key residual as
// an exact pair, u^K sums alpha^2 (q . r)^2 / D (|V|^2 - 2 V . y + |y|^2).
constexpr int kUtPos = 32, kUtRows = 16;
struct UtilSmem {
  float rh[128][kUtPos], rl[128][kUtPos], v[128][kUtPos];  // residual pairs and values, by dimension
  union {  // (72.5 KB in all, for three blocks per SM; with the sums in a place of their own two fit: 617 us, not 578, for 8 units of
  // 4096 positions and 128 rows)
    struct {
      float q[kUtRows][128], yh[kUtRows][128], yl[kUtRows][128];
    };
    double red[8][kUtPos][3];  // before the first rows and after the last
  };
  double y2[kUtRows];
  float qn[kUtRows], yn[kUtRows];
  float red_n[2][kUtPos];
};
__global__ void __launch_bounds__(256) enc_util_f(const EncArgs A) {
  extern __shared__ __align__(16) uint8_t ut_dyn[];
  UtilSmem& s = *reinterpret_cast<UtilSmem*>(ut_dyn);
  const int u = blockIdx.y;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, p0 = blockIdx.x * kUtPos, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (p0 >= S) return;
  const EncUnitWs w = unit_ws(A, u, d);
  const uint4* AK = reinterpret_cast<const uint4*>(A.arena_c + d->off_anchor_k);
  const uint4* AV = reinterpret_cast<const uint4*>(A.arena_c + d->off_anchor_v);
  // residuals: eight threads per position, 16 dimensions each
  const int lp = tid >> 3, sub = tid & 7, pl = p0 + lp;
  const bool in = pl < S && w.slot_of[pl] < 0;
  float rn = 0.f, vn = 0.f, es = 0.f, ec = 0.f, vs = 0.f, vc = 0.f;
  {
    const uint32_t sk = in ? w.st[0][pl] : 0u, sv = in ? w.st[1][pl] : 0u;
    const int ak = (int)(sk & 0xFFFFu), av = (int)(sv & 0xFFFFu);
    const float gk = __half2float(__ushort_as_half((unsigned short)(sk >> 16)));
    const float gv = __half2float(__ushort_as_half((unsigned short)(sv >> 16)));
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int ch = 2 * sub + c;
      const uint4 z = make_uint4(0u, 0u, 0u, 0u);
      const uint4 xk = in ? __ldg(reinterpret_cast<const uint4*>(A.K + ((size_t)u * A.s_max + pl) * 128) + ch) : z;
      const uint4 xv = in ? __ldg(reinterpret_cast<const uint4*>(A.V + ((size_t)u * A.s_max + pl) * 128) + ch) : z;
      const uint4 yk = in ? __ldg(AK + (size_t)ak * 16 + (ch ^ (ak & 7))) : z, yv = in ? __ldg(AV + (size_t)av * 16 + (ch ^ (av & 7))) : z;
      const uint32_t kw[4] = {xk.x, xk.y, xk.z, xk.w}, vw[4] = {xv.x, xv.y, xv.z, xv.w};
      const uint32_t ka[4] = {yk.x, yk.y, yk.z, yk.w}, va[4] = {yv.x, yv.y, yv.z, yv.w};
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float x = (e & 1) ? bf_hi(kw[e >> 1]) : bf_lo(kw[e >> 1]), a = (e & 1) ? bf_hi(ka[e >> 1]) : bf_lo(ka[e >> 1]);
        float h = x, l = 0.f;
        two_sum_add(h, l, -(gk * a));  // (the product is exact)
        s.rh[8 * ch + e][lp] = h;
        s.rl[8 * ch + e][lp] = l;
        rn = __fmaf_rn(h, h, rn);
        const float v = (e & 1) ? bf_hi(vw[e >> 1]) : bf_lo(vw[e >> 1]), b = (e & 1) ? bf_hi(va[e >> 1]) : bf_lo(va[e >> 1]);
        s.v[8 * ch + e][lp] = v;
        two_sum_add(vs, vc, v * v);
        float rvh = v, rvl = 0.f;
        two_sum_add(rvh, rvl, -(gv * b));
        const float pp = rvh * rvh;
        ec += __fmaf_rn(2.f * rvh, rvl, __fmaf_rn(rvh, rvh, -pp));
        two_sum_add(es, ec, pp);
      }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      rn += __shfl_xor_sync(0xffffffffu, rn, o);
      const float a = __shfl_xor_sync(0xffffffffu, vs, o), b = __shfl_xor_sync(0xffffffffu, vc, o);
      two_sum_add(vs, vc, a);
      vc += b;
      const float a2 = __shfl_xor_sync(0xffffffffu, es, o), b2 = __shfl_xor_sync(0xffffffffu, ec, o);
      two_sum_add(es, ec, a2);
      ec += b2;
    }
    vn = vs;
    if (sub == 0) {  // handed to the position's threads below through the sums' places
      s.red[0][lp][0] = pair_f64(vs, vc);
      s.red[1][lp][0] = pair_f64(es, ec);
      // u^V has no bound but that of its factors: the value residual's energy has to be exactly 0 or inside the fp32
      // range, or the norm that goes with it is handed on as infinite
      const bool ev_ok = (es >= 0x1p-100f && es <= 0x1p100f) ||
                         (es == 0.f && (!in || exactly_zero_residual(reinterpret_cast<const uint4*>(A.V + ((size_t)u * A.s_max + pl) * 128),
                                                                     AV + (size_t)av * 16, av, gv)));
      s.red_n[0][lp] = ev_ok ? rn : INFINITY;
      s.red_n[1][lp] = vn;
    }
  }
  __syncthreads();
  const int p = p0 + lane, g = warp;
  const double v2 = s.red[0][lane][0], ev = s.red[1][lane][0];
  const float rnorm2 = s.red_n[0][lane], vnorm2 = s.red_n[1][lane];
  __syncthreads();
  const float ea = alpha_error(w), vmax = norm_up(__uint_as_float(w.ctrl[19]));
  const float ey = (0x1p-29f + ea) * vmax;  // |error of y| (256 paired steps of three additions, and alpha's)
  const float rnorm = norm_up(rnorm2), vnorm = norm_up(vnorm2);
  double uk = 0.0, uv = 0.0, ek = 0.0;
  for (int w0 = 0; w0 < A.m_obs; w0 += kUtRows) {
    const int nr = min(kUtRows, A.m_obs - w0);
    __syncthreads();
    for (int r = warp; r < kUtRows; r += 8) {  // a warp loads a row, and takes its norms
      float ys = 0.f, yc = 0.f, qn = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = lane + 32 * e;
        const float q = r < nr ? __bfloat162float(A.Q[((size_t)u * A.m_obs + w0 + r) * 128 + j]) : 0.f;
        const double y = r < nr ? w.yobs[(w0 + r) * 128 + j] : 0.0;
        const float yh = (float)y, yl = (float)(y - (double)yh), pp = yh * yh;
        s.q[r][j] = q;
        s.yh[r][j] = yh;
        s.yl[r][j] = yl;
        qn = __fmaf_rn(q, q, qn);
        yc += __fmaf_rn(2.f * yh, yl, __fmaf_rn(yh, yh, -pp));
        two_sum_add(ys, yc, pp);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        qn += __shfl_xor_sync(0xffffffffu, qn, o);
        const float a = __shfl_xor_sync(0xffffffffu, ys, o), b = __shfl_xor_sync(0xffffffffu, yc, o);
        two_sum_add(ys, yc, a);
        yc += b;
      }
      if (lane == 0) {
        s.y2[r] = pair_f64(ys, yc);
        s.qn[r] = norm_up(qn);
        s.yn[r] = norm_up(ys);
      }
    }
    __syncthreads();
    float qs[2] = {}, qc[2] = {}, ys[2] = {}, yc[2] = {};  // q . r and V . y of the thread's two rows
#pragma unroll 2
    for (int j = 0; j < 128; j += 4) {
      float rh[4], rl[4], v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        rh[e] = s.rh[j + e][lane];
        rl[e] = s.rl[j + e][lane];
        v[e] = s.v[j + e][lane];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = g + 8 * i;
        const float4 q4 = *reinterpret_cast<const float4*>(&s.q[r][j]), h4 = *reinterpret_cast<const float4*>(&s.yh[r][j]),
                     l4 = *reinterpret_cast<const float4*>(&s.yl[r][j]);
        const float q[4] = {q4.x, q4.y, q4.z, q4.w}, yh[4] = {h4.x, h4.y, h4.z, h4.w}, yl[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float a = q[e] * rh[e], b = v[e] * yh[e];
          qc[i] += __fmaf_rn(q[e], rl[e], __fmaf_rn(q[e], rh[e], -a));
          two_sum_add(qs[i], qc[i], a);
          yc[i] += __fmaf_rn(v[e], yl[e], __fmaf_rn(v[e], yh[e], -b));
          two_sum_add(ys[i], yc[i], b);
        }
      }
    }
    if (p < S) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = g + 8 * i;
        if (r >= nr) continue;
        const double a = w.alpha[(size_t)(w0 + r) * S + p], a2 = a * a;
        const double dq = pair_f64(qs[i], qc[i]), dv = fma(-2.0, pair_f64(ys[i], yc[i]), v2 + s.y2[r]);
        const double aq = a2 * (dq * dq) * 0.0078125;
        uk = fma(aq, dv, uk);
        uv += a2;
        // errors of q . r and of dv: paired chains of 128 steps, and y's; products below the fp32 range (2^-149 each)
        // by their own terms
        const float hq = __fmaf_rn(0x1p-32f * s.qn[r], rnorm, 0x1p-138f), sum = vnorm + s.yn[r] + ey;
        const float hv = __fmaf_rn(sum, __fmaf_rn(0x1p-31f, sum, 2.f * ey), 0x1p-136f);
        const float sq = __fmaf_rn(__fmaf_rn(2.f, fabsf((float)dq), hq), 0.0078125f * hq, 0x1p-148f);  // of (q . r)^2 / D
        ek = fma(a2, (double)__fmaf_rn(sq, fabsf((float)dv) + hv, 0x1p-148f), fma(aq, (double)hv, ek));
      }
    }
  }
  __syncthreads();  // the rows are read
  s.red[g][lane][0] = uk;
  s.red[g][lane][1] = uv;
  s.red[g][lane][2] = ek;
  __syncthreads();
  if (g != 0 || p >= S) return;
  double* err = reinterpret_cast<double*>(w.perm);
  if (w.slot_of[p] >= 0) {
    w.key0[p] = w.key1[p] = 0ull;
    err[p] = 0.0;
    return;
  }
  for (int x = 1; x < 8; ++x) {
    uk += s.red[x][lane][0];
    uv += s.red[x][lane][1];
    ek += s.red[x][lane][2];
  }
  const double rm = 1.0 / (double)A.m_obs;
  uk *= rm;
  uv *= ev * rm;
  const bool bounded = norm_ok(rnorm2) && norm_ok(vnorm2);
  w.key0[p] = (uint64_t)__double_as_longlong(uk > 0.0 ? uk : 0.0) + 1ull;
  w.key1[p] = (uint64_t)__double_as_longlong(uv > 0.0 ? uv : 0.0) + 1ull;
  err[p] = bounded ? 1.001 * ek * rm : (double)INFINITY;
}

// Whether a ranking by values v with errors e stands: the lowest selected v - e above the largest
// unselected v + e.  Order-preserving 64-bit form of an fp64 value, for the maxima over the cluster.
__device__ __forceinline__ uint64_t f64_order(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Top `want` of n 64-bit keys over the cluster (each CTA holding keys i in [lo, hi) through key_at), from the
// largest down: selected are those with key >> sh >= prefix.  False if equal keys straddle the cut.
template <class KeyAt>
__device__ bool cluster_top(cooperative_groups::cluster_group cl, KeyAt key_at, int64_t lo, int64_t hi, uint32_t want,
                            uint32_t (*hist)[2048], uint32_t* wsum, uint32_t* found, int& sh, uint64_t& prefix) {
  const int tid = threadIdx.x;
  for (int i = tid; i < 3 * 2048; i += kSelThreads) (&hist[0][0])[i] = 0u;
  __syncthreads();
  sh = 64;
  prefix = 0;
#pragma unroll 1
  for (int dg = 0;; ++dg) {
    const int ns = max(0, sh - 11), bits = sh - ns;
    uint32_t* h = hist[dg % 3];
    for (int64_t i0 = lo; i0 < hi; i0 += kSelThreads) {
      const int64_t i = i0 + tid;
      const uint64_t v = i < hi ? key_at(i) : 0ull;
      const bool in = i < hi && (dg == 0 || (v >> sh) == prefix);
      const uint32_t digit = in ? (uint32_t)(v >> ns) & ((1u << bits) - 1u) : 0xFFFFFFFFu;
      const unsigned peers = __match_any_sync(0xffffffffu, digit);
      if (in && (peers & ((1u << (tid & 31)) - 1u)) == 0u) atomicAdd(&h[digit], (uint32_t)__popc(peers));
    }
    cl.sync();
    if (dg > 0)
      for (int i = tid; i < 2048; i += kSelThreads) hist[(dg + 2) % 3][i] = 0u;
    uint32_t inside;
    const uint32_t digit = cluster_digit<true>(cl, h, wsum, found, want, &inside);
    prefix = (prefix << bits) | digit;
    sh = ns;
    if (want == inside) return true;
    if (sh == 0) return false;
  }
}
// Largest of a 64-bit value over the cluster.
__device__ uint64_t cluster_max(cooperative_groups::cluster_group cl, uint64_t v, unsigned long long* slot) {
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t t = __shfl_xor_sync(0xffffffffu, v, o);
    v = t > v ? t : v;
  }
  __syncthreads();
  if (threadIdx.x == 0) *slot = 0ull;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) atomicMax(slot, (unsigned long long)v);
  cl.sync();
  for (int r = 0; r < kSelCtas; ++r) {
    const uint64_t t = *cl.map_shared_rank(slot, r);
    v = t > v ? t : v;
  }
  return v;
}

// The floor(rho (k - w)) highest scores (ties: lower position) become anchors: slot_of = -2 marks them for
// enc_anchors, every other position gets -1.
__global__ void __cluster_dims__(kSelCtas, 1, 1) __launch_bounds__(kSelThreads) enc_score_pick_f(const EncArgs A) {
  namespace cg = cooperative_groups;
  __shared__ __align__(16) uint32_t hist[3][2048];
  __shared__ uint32_t wsum[kSelThreads / 32], found[3];
  __shared__ unsigned long long slot[2];
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, u = blockIdx.x / kSelCtas;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, k = d->n_anchors, win = min(A.window, S), P = S - win;
  const EncUnitWs w = unit_ws(A, u, d);
  const int ns = n_scored(A, k - win);
  int lo, hi, sh = 0;
  cluster_share(S, (int)cl.block_rank(), lo, hi);
  uint64_t prefix = ~0ull;
  if (ns > 0) {
    const int hp = min(hi, P);
    bool ok = cluster_top(cl, [&](int64_t i) { return w.key0[i]; }, lo, hp, (uint32_t)ns, hist, wsum, found, sh, prefix);
    const double e = 2.0 * (double)alpha_error(w);
    uint64_t in_lo = 0, out_hi = 0;  // complement of the lowest selected bound; largest unselected one
    for (int p = lo + tid; p < hp; p += kSelThreads) {
      const uint64_t key = w.key0[p];
      const double v = __longlong_as_double((long long)key);
      if ((key >> sh) >= prefix) in_lo = max(in_lo, ~f64_order(v - e * v - 1e-290));
      else out_hi = max(out_hi, f64_order(v + e * v + 1e-290));
    }
    in_lo = cluster_max(cl, in_lo, &slot[0]);
    out_hi = cluster_max(cl, out_hi, &slot[1]);
    ok = ok && ~in_lo > out_hi && __uint_as_float(w.ctrl[17]) <= 0x1p60f && __uint_as_float(w.ctrl[18]) <= 0x1p60f;
    if (!ok && cl.block_rank() == 0 && tid == 0) w.ctrl[16] = 1u;
  }
  for (int p = lo + tid; p < hi; p += kSelThreads) w.slot_of[p] = ns > 0 && p < P && (w.key0[p] >> sh) >= prefix ? -2 : -1;
  cl.sync();  // no CTA leaves while another may still read its counts
}

// A cluster per request and side: the side's Eq. 9 share of the budget goes to the highest utilities over all
// KV heads of the request (ties: lower head, then lower position) -> per-unit flags, slot lists and counts
// (ctrl[2 + side]).
__global__ void __cluster_dims__(kSelCtas, 1, 1) __launch_bounds__(kSelThreads) enc_pool_f(const EncArgs A) {
  namespace cg = cooperative_groups;
  __shared__ __align__(16) uint32_t hist[3][2048];
  __shared__ uint32_t wsum[kSelThreads / 32], found[3];
  __shared__ unsigned long long slot[2];
  __shared__ const uint64_t* keys[256];
  __shared__ const double* errs[256];
  __shared__ float rel[256];
  __shared__ int32_t* lists[256];
  __shared__ uint32_t* ctrls[256];
  __shared__ uint8_t* flags[256];
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, side = blockIdx.y, H = A.n_kv_heads, u0 = (int)(blockIdx.x / kSelCtas) * H;
  const akv_unit_desc* d0 = unit_desc(A, u0);
  const int S = d0->len, k = d0->n_anchors;
  bool ok = true;
  for (int h = tid; h < H; h += kSelThreads) {
    const akv_unit_desc* d = unit_desc(A, u0 + h);
    const EncUnitWs w = unit_ws(A, u0 + h, d);
    keys[h] = side ? w.key1 : w.key0;
    errs[h] = reinterpret_cast<const double*>(w.perm);
    rel[h] = 2.5f * alpha_error(w) + 0x1p-30f;
    lists[h] = w.res_pos + (side ? d->n_res_k : 0);
    ctrls[h] = w.ctrl;
    flags[h] = w.flag[side];
    for (int i = 17; i < 20; ++i) ok = ok && __uint_as_float(w.ctrl[i]) <= 0x1p60f;
  }
  ok = __syncthreads_and(ok);
  const int64_t N = budget_residuals(A.theta, S, H, A.window, k), cand = (int64_t)H * (S - k), n = (int64_t)H * S;
  int64_t want = side ? N - N / 2 : N / 2;
  if (want > cand) want = cand;
  const int64_t per = (n + kSelCtas - 1) / kSelCtas, lo = min(n, (int64_t)cl.block_rank() * per), hi = min(n, lo + per);
  int sh = 0;
  uint64_t prefix = ~0ull;
  if (want > 0) {
    ok = cluster_top(cl, [&](int64_t i) { return keys[i / S][i % S]; }, lo, hi, (uint32_t)want, hist, wsum, found, sh, prefix) && ok;
    uint64_t in_lo = 0, out_hi = 0;
    for (int64_t i = lo + tid; i < hi; i += kSelThreads) {
      const int h = (int)(i / S), p = (int)(i % S);
      const uint64_t key = keys[h][p];
      if (key == 0ull) continue;  // an anchor
      const double v = __longlong_as_double((long long)(key - 1ull));
      const double ek = errs[h][p], e = v * (double)rel[h] + (side == 0 || !(ek < (double)INFINITY) ? ek : 0.0) + 1e-300;
      const bool known = v + e < (double)INFINITY;  // (an error without a bound, or a NaN, leaves the ranking open)
      if ((key >> sh) >= prefix) in_lo = max(in_lo, known ? ~f64_order(v - e) : ~(uint64_t)0);
      else out_hi = max(out_hi, known ? f64_order(v + e) : ~(uint64_t)0);
    }
    in_lo = cluster_max(cl, in_lo, &slot[0]);
    out_hi = cluster_max(cl, out_hi, &slot[1]);
    // (every candidate in, or the cut clear of both sides' errors)
    ok = want == cand || (ok && ~in_lo > out_hi);
  }
  if (!ok) {
    if (cl.block_rank() == 0 && tid == 0) ctrls[0][12 + side] = 1u;
    cl.sync();
    return;
  }
  for (int64_t i0 = lo; i0 < hi; i0 += kSelThreads) {
    const int64_t i = i0 + tid;
    if (i >= hi) continue;
    const int h = (int)(i / S), p = (int)(i % S);
    const uint64_t key = keys[h][p];
    const bool sel = want > 0 && (want == cand ? key != 0ull : (key >> sh) >= prefix);
    flags[h][p] = sel ? 1 : 0;
    if (sel) lists[h][atomicAdd(&ctrls[h][2 + side], 1u)] = p;
  }
  cl.sync();
}

// The exact forms, run only where the paired sums left a ranking undecided: GATE 1, of the unit's scores;
// GATE 2, of the request's utilities (either side).
template <int GATE>
__device__ __forceinline__ bool gated(const EncArgs& A, int u) {
  if (GATE == 1) return unit_ws(A, u, unit_desc(A, u)).ctrl[16] != 0u;
  const int u0 = u / A.n_kv_heads * A.n_kv_heads;
  const uint32_t* c = unit_ws(A, u0, unit_desc(A, u0)).ctrl;
  return (c[12] | c[13]) != 0u;
}

// The attention of unit u is taken in fp64: for its scores (GATE 1), or for its request's utilities (GATE 2) where that has
// not been done for the scores.
template <int GATE>
__device__ __forceinline__ bool gated_alpha(const EncArgs& A, int u) {
  return gated<GATE>(A, u) && (GATE == 1 || !gated<1>(A, u));
}

// Logits q_w . K_t / sqrt(D) of every observation row and position (Eq. 4), into alpha.
template <int GATE>
__global__ void __launch_bounds__(128) enc_obs_logit(const EncArgs A) {
  __shared__ double qs[128];
  const int u = blockIdx.y;
  if (!gated_alpha<GATE>(A, u)) return;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len;
  const int t = blockIdx.x * 128 + threadIdx.x;
  if (blockIdx.x * 128 >= S) return;
  EncUnitWs w = unit_ws(A, u, d);
  const __nv_bfloat16* X = A.K + ((size_t)u * A.s_max + min(t, S - 1)) * 128;
  for (int wr = 0; wr < A.m_obs; ++wr) {
    __syncthreads();
    qs[threadIdx.x] = bf16_to_f64(A.Q[((size_t)u * A.m_obs + wr) * 128 + threadIdx.x]);
    __syncthreads();
    double acc = 0.0;  // (a product of two bf16 is exact: the fused step rounds like a separate add)
    for (int j = 0; j < 128; ++j) acc = __fma_rn(qs[j], bf16_to_f64(X[j]), acc);
    if (t < S) w.alpha[(size_t)wr * S + t] = __dmul_rn(acc, __ddiv_rn(1.0, __dsqrt_rn(128.0)));
  }
}

// Softmax of each observation row's logits over all S positions.
template <int GATE>
__global__ void __launch_bounds__(1024) enc_obs_softmax(const EncArgs A) {
  __shared__ double red[32];
  __shared__ double den_s;
  const int u = blockIdx.y, wr = blockIdx.x;
  if (!gated_alpha<GATE>(A, u)) return;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len;
  EncUnitWs w = unit_ws(A, u, d);
  double* a = w.alpha + (size_t)wr * S;
  double mx = -INFINITY;
  for (int t = threadIdx.x; t < S; t += blockDim.x) mx = fmax(mx, a[t]);
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = red[0];
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = fmax(m, red[i]);
    red[0] = m;
  }
  __syncthreads();
  mx = red[0];
  for (int t = threadIdx.x; t < S; t += blockDim.x) a[t] = exp_neg_dev(__dsub_rn(a[t], mx));
  __syncthreads();
  if (threadIdx.x == 0) {  // the normaliser, summed in position order
    double den = 0.0;
    for (int t = 0; t < S; ++t) den = __dadd_rn(den, a[t]);
    den_s = den;
  }
  __syncthreads();
  const double den = den_s;
  for (int t = threadIdx.x; t < S; t += blockDim.x) a[t] = __ddiv_rn(a[t], den);
}

// Exact output y_w = sum_t alpha_wt V_t of each observation row (positions in order).
__global__ void __launch_bounds__(128) enc_obs_y(const EncArgs A) {
  const int u = blockIdx.y, wr = blockIdx.x, j = threadIdx.x;
  if (!gated<2>(A, u)) return;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len;
  EncUnitWs w = unit_ws(A, u, d);
  const double* a = w.alpha + (size_t)wr * S;
  const __nv_bfloat16* V = A.V + (size_t)u * A.s_max * 128;
  double acc = 0.0;
  for (int t = 0; t < S; ++t) acc = __dadd_rn(acc, __dmul_rn(a[t], bf16_to_f64(V[(size_t)t * 128 + j])));
  w.yobs[wr * 128 + j] = acc;
}

// Selector score, step 1: the rows' attention averaged over the m rows (into key1 as fp64).
template <int GATE>
__global__ void enc_score_mean(const EncArgs A) {
  const int u = blockIdx.y;
  if (GATE && !gated<GATE>(A, u)) return;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, P = S - min(A.window, S);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= P) return;
  EncUnitWs w = unit_ws(A, u, d);
  double acc = 0.0;
  for (int wr = 0; wr < A.m_obs; ++wr) acc = __dadd_rn(acc, w.alpha[(size_t)wr * S + t]);
  w.key1[t] = (uint64_t)__double_as_longlong(__ddiv_rn(acc, (double)A.m_obs));
}

// Selector score, step 2: average pooling of width kappa centred on t over [0, P), zero
// outside, divided by kappa (Appendix A.2); the score's bits into key0 (scores are >= 0,
// so their bit patterns order like the values).
template <int GATE>
__global__ void enc_score_pool(const EncArgs A) {
  const int u = blockIdx.y;
  if (GATE && !gated<GATE>(A, u)) return;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, P = S - min(A.window, S);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= P) return;
  EncUnitWs w = unit_ws(A, u, d);
  const int h = A.kappa / 2;
  double acc = 0.0;
  for (int j = t - h; j <= t + h; ++j)
    if (j >= 0 && j < P) acc = __dadd_rn(acc, __longlong_as_double((long long)w.key1[j]));
  w.key0[t] = (uint64_t)__double_as_longlong(__ddiv_rn(acc, (double)A.kappa));
}

// The floor(rho (k - w)) highest scores (ties: lower position) become anchors: slot_of = -2
// marks them for enc_anchors, every other position gets -1.
__global__ void __launch_bounds__(1024) enc_score_pick(const EncArgs A) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t bc[2];
  __shared__ int wt[33];
  const int u = blockIdx.x;
  if (!gated<1>(A, u)) return;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len, k = d->n_anchors, win = min(A.window, S), P = S - win;
  EncUnitWs w = unit_ws(A, u, d);
  const int ns = n_scored(A, k - win);
  uint64_t thr = ~0ull;
  uint32_t need = 0;
  if (ns > 0) thr = block_select(w.key0, P, (uint32_t)ns, true, hist, bc, &need);
  int eq_seen = 0;
  for (int c0 = 0; c0 < S; c0 += 1024) {
    const int p = c0 + threadIdx.x;
    const uint64_t kv = (p < P) ? w.key0[p] : 0ull;
    const int is_eq = (ns > 0 && p < P && kv == thr) ? 1 : 0;
    int eq_tot;
    const int eq_pre = block_scan_flag(is_eq, wt, &eq_tot);
    const int sel = (ns > 0 && p < P) && (kv > thr || (is_eq && (uint32_t)(eq_seen + eq_pre) < need));
    eq_seen += eq_tot;
    if (p < S) w.slot_of[p] = sel ? -2 : -1;
    __syncthreads();
  }
}

// Eq. 6 utilities of the non-anchor positions (one thread per position, rows and
// dimensions in order): key0 = bits(u^K) + 1, key1 = bits(u^V) + 1, anchors 0.
constexpr int UT_ROWS = 16;  // observation rows staged in shared memory at a time
__global__ void __launch_bounds__(128) enc_util(const EncArgs A) {
  __shared__ double qs[UT_ROWS][128];
  __shared__ double ys[UT_ROWS][128];
  const int u = blockIdx.y;
  if (!gated<2>(A, u)) return;
  const akv_unit_desc* d = unit_desc(A, u);
  const int S = d->len;
  if (blockIdx.x * 128 >= S) return;
  EncUnitWs w = unit_ws(A, u, d);
  const int p = blockIdx.x * 128 + threadIdx.x;
  const int32_t* apos = reinterpret_cast<const int32_t*>(A.arena_c + d->off_anchor_pos);
  const bool live = p < S && apos[w.st[0][p] & 0xFFFFu] != p;  // (an anchor's position is its slot's)
  const __nv_bfloat16 *xk = nullptr, *xv = nullptr, *ak = nullptr, *av = nullptr;
  double gk = 0.0, gv = 0.0, ev = 0.0;
  if (live) {
    xk = A.K + ((size_t)u * A.s_max + p) * 128;
    xv = A.V + ((size_t)u * A.s_max + p) * 128;
    const uint32_t sk = w.st[0][p], sv = w.st[1][p];
    ak = anchor_src(A, u, 0, apos, (int)(sk & 0xFFFFu));
    av = anchor_src(A, u, 1, apos, (int)(sv & 0xFFFFu));
    gk = fp16_bits_to_f64(sk >> 16);
    gv = fp16_bits_to_f64(sv >> 16);
    for (int j = 0; j < 128; ++j) {
      const double rv = __dsub_rn(bf16_to_f64(xv[j]), __dmul_rn(gv, bf16_to_f64(av[j])));
      ev = __dadd_rn(ev, __dmul_rn(rv, rv));
    }
  }
  double uk = 0.0, uv = 0.0;
  for (int w0 = 0; w0 < A.m_obs; w0 += UT_ROWS) {
    const int nr = min(UT_ROWS, A.m_obs - w0);
    __syncthreads();
    for (int e = threadIdx.x; e < nr * 128; e += 128) {
      qs[e >> 7][e & 127] = bf16_to_f64(A.Q[((size_t)u * A.m_obs + w0 + (e >> 7)) * 128 + (e & 127)]);
      ys[e >> 7][e & 127] = w.yobs[(w0 + (e >> 7)) * 128 + (e & 127)];
    }
    __syncthreads();
    if (!live) continue;
    for (int r = 0; r < nr; ++r) {
      const double a = w.alpha[(size_t)(w0 + r) * S + p];
      const double a2 = __dmul_rn(a, a);
      double dq = 0.0, dv = 0.0;
      for (int j = 0; j < 128; ++j) {
        const double rk = __dsub_rn(bf16_to_f64(xk[j]), __dmul_rn(gk, bf16_to_f64(ak[j])));
        dq = __dadd_rn(dq, __dmul_rn(qs[r][j], rk));
        const double c = __dsub_rn(bf16_to_f64(xv[j]), ys[r][j]);
        dv = __dadd_rn(dv, __dmul_rn(c, c));
      }
      uk = __dadd_rn(uk, __dmul_rn(__dmul_rn(a2, __ddiv_rn(__dmul_rn(dq, dq), 128.0)), dv));
      uv = __dadd_rn(uv, __dmul_rn(a2, ev));
    }
  }
  if (p >= S) return;
  if (!live) {
    w.key0[p] = 0ull;
    w.key1[p] = 0ull;
    return;
  }
  uk = __ddiv_rn(uk, (double)A.m_obs);
  uv = __ddiv_rn(uv, (double)A.m_obs);
  w.key0[p] = (uint64_t)__double_as_longlong(uk) + 1ull;
  w.key1[p] = (uint64_t)__double_as_longlong(uv) + 1ull;
}

// One block per request: the side's Eq. 9 share of the budget goes to the highest
// utilities over all KV heads of the request (ties: lower head, then lower position) ->
// per-unit flags, ascending slot lists and counts (ctrl[2 + side]).
__global__ void __launch_bounds__(1024) enc_pool(const EncArgs A, int side) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t bc[2];
  __shared__ int wt[33];
  __shared__ const uint64_t* keys[256];
  __shared__ int32_t* lists[256];
  __shared__ uint32_t* ctrls[256];
  __shared__ uint8_t* flags[256];
  const int H = A.n_kv_heads, u0 = blockIdx.x * H;
  if (unit_ws(A, u0, unit_desc(A, u0)).ctrl[12 + side] == 0u) return;
  const akv_unit_desc* d0 = unit_desc(A, u0);
  const int S = d0->len, k = d0->n_anchors;
  for (int h = threadIdx.x; h < H; h += blockDim.x) {
    const akv_unit_desc* d = unit_desc(A, u0 + h);
    EncUnitWs w = unit_ws(A, u0 + h, d);
    keys[h] = side ? w.key1 : w.key0;
    lists[h] = w.res_pos + (side ? d->n_res_k : 0);
    ctrls[h] = w.ctrl;
    flags[h] = w.flag[side];
  }
  __syncthreads();
  const int64_t N = budget_residuals(A.theta, S, H, A.window, k);
  const int64_t cand = (int64_t)H * (S - k);
  int64_t want = side ? N - N / 2 : N / 2;
  if (want > cand) want = cand;
  const int64_t n = (int64_t)H * S;
  auto key_at = [&](int64_t i) { return keys[i / S][i % S]; };
  uint64_t thr = ~0ull;
  uint32_t need = 0;
  if (want > 0) thr = block_select_f(key_at, n, (uint32_t)want, true, hist, bc, &need);
  int eq_seen = 0;
  for (int h = 0; h < H; ++h) {
    int base = 0;
    for (int c0 = 0; c0 < S; c0 += 1024) {
      const int p = c0 + threadIdx.x;
      const uint64_t kv = p < S ? keys[h][p] : 0ull;
      const int is_eq = (want > 0 && p < S && kv == thr) ? 1 : 0;
      int eq_tot;
      const int eq_pre = block_scan_flag(is_eq, wt, &eq_tot);
      const int sel = (want > 0 && p < S) && (kv > thr || (is_eq && (uint32_t)(eq_seen + eq_pre) < need));
      eq_seen += eq_tot;
      int tot;
      const int pre = block_scan_flag(sel, wt, &tot);
      if (sel) lists[h][base + pre] = p;
      if (p < S) flags[h][p] = (uint8_t)sel;
      base += tot;
      __syncthreads();
    }
    if (threadIdx.x == 0) ctrls[h][2 + side] = (uint32_t)base;
  }
}

// The arena descriptors take the residual counts the full selection chose (last launch:
// every earlier kernel sizes its scratch from the reserved counts).
__global__ void enc_set_counts(const EncArgs A, int units) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= units) return;
  const akv_unit_desc* d = unit_desc(A, u);
  EncUnitWs w = unit_ws(A, u, d);
  akv_unit_desc* dm = reinterpret_cast<akv_unit_desc*>(A.arena + 256) + u;
  const int32_t nk = (int32_t)w.ctrl[2], nv = (int32_t)w.ctrl[3];
  dm->n_res_k = nk;
  dm->n_res_v = nv;
}

}  // namespace

// Scratch of akv_encode_noalloc, for callers that cannot hand the library a
// device workspace.  It is part of the module image: no allocation call makes
// it, and each device that loads the library keeps it until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[AKV_NOALLOC_SCRATCH_BYTES];

int noalloc_scratch(void** ptr, size_t* bytes) {
  // Host code must not use g_noalloc_scratch's name as a device address: it is
  // a host-side stand-in.  The device address is looked up on every call, with
  // the caller's device current, rather than cached: after cudaDeviceReset the
  // module is loaded again and the array may move, and a context other than the
  // primary one holds its own copy, so a cached address could point at memory
  // this call does not own.  The lookup costs far less than the encode.  The
  // first lookup on a device loads the library's module there.
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess) return (int)e;
  *ptr = p;
  *bytes = AKV_NOALLOC_SCRATCH_BYTES;
  return 0;
}

int launch_encode(const Layout& L, const EncodeWs& W, const akv_params& p, const void* K, const void* V, int32_t s_max,
                  void* arena, void* ws, void* stream, const akv_select_params* sel, const void* Q, int32_t m_obs) {
  cudaStream_t st = (cudaStream_t)stream;
  const int units = (int)L.shape.size();
  cudaError_t e;
  // header + descriptors, then the per-unit workspace table at the start of ws
  std::vector<uint8_t> head(kHeaderBytes + kDescBytes * (size_t)units);
  std::memcpy(head.data(), &L.header, sizeof(L.header));
  std::memcpy(head.data() + kHeaderBytes, L.desc.data(), kDescBytes * (size_t)units);
  if ((e = cudaMemsetAsync(arena, 0, (size_t)L.total_bytes, st)) != cudaSuccess) return (int)e;
  if ((e = cudaMemcpyAsync(arena, head.data(), head.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess) return (int)e;
  std::vector<uint64_t> table(W.unit_off.begin(), W.unit_off.end());
  if ((e = cudaMemcpyAsync(ws, table.data(), (size_t)units * 8, cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return (int)e;

  EncArgs A;
  A.arena_c = (const uint8_t*)arena;
  A.arena = (uint8_t*)arena;
  A.ws_base = (const uint8_t*)ws;
  A.ws_off = (const uint64_t*)ws;
  A.K = (const __nv_bfloat16*)K;
  A.V = (const __nv_bfloat16*)V;
  A.s_max = s_max;
  A.n_kv_heads = p.n_kv_heads;
  A.window = p.window;
  A.rotate = (p.flags & AKV_FLAG_ROTATE) ? 1 : 0;
  A.lloyd = (p.flags & AKV_FLAG_LLOYD) ? 1 : 0;
  A.seed = p.seed;
  A.sign_lo = L.header.sign_bits[0];
  A.sign_hi = L.header.sign_bits[1];
  const bool full = sel != nullptr && Q != nullptr && m_obs > 0;
  A.Q = (const __nv_bfloat16*)Q;
  A.m_obs = full ? m_obs : 0;
  A.kappa = full ? sel->kappa : 1;
  A.rho = full ? sel->rho : 0.0f;
  A.theta = full ? sel->theta : 0.0f;

  const unsigned maxS = (unsigned)L.max_len;
  if (full) {  // observation rows' attention, selector scores, the scored anchors
    const unsigned m = (unsigned)m_obs;
    enc_obs_init<<<units, 256, 0, st>>>(A);
    enc_obs_logit_f<<<dim3((maxS + 127) / 128, units, (m + kObsRows - 1) / kObsRows), 128, 0, st>>>(A);
    enc_obs_softmax_f<<<dim3(m, units), 512, 0, st>>>(A);
    enc_obs_y_f<<<dim3((maxS + kObsChunk - 1) / kObsChunk, (m + 7) / 8, units), 128, 0, st>>>(A);
    enc_score_mean<0><<<dim3((maxS + 255) / 256, units), 256, 0, st>>>(A);
    enc_score_pool<0><<<dim3((maxS + 255) / 256, units), 256, 0, st>>>(A);
    enc_score_pick_f<<<kSelCtas * (unsigned)units, kSelThreads, 0, st>>>(A);
    // the units whose scores the errors leave undecided
    enc_obs_logit<1><<<dim3((maxS + 127) / 128, units), 128, 0, st>>>(A);
    enc_obs_softmax<1><<<dim3(m, units), 1024, 0, st>>>(A);
    enc_score_mean<1><<<dim3((maxS + 255) / 256, units), 256, 0, st>>>(A);
    enc_score_pool<1><<<dim3((maxS + 255) / 256, units), 256, 0, st>>>(A);
    enc_score_pick<<<units, 1024, 0, st>>>(A);
  }
  enc_anchors<<<kSelCtas * (unsigned)units, kSelThreads, 0, st>>>(A);
  enc_rows<<<dim3((unsigned)(L.max_k + 31) / 32, units, 2), 256, 0, st>>>(A);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return (int)e;
  if ((e = cudaFuncSetAttribute(enc_assign_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAtSmem)) !=
      cudaSuccess)
    return (int)e;
  CUtensorMap tmK, tmV, tmA;
  if (!encode_row_map(&tmK, K, (uint64_t)units * (uint64_t)s_max, 128, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !encode_row_map(&tmV, V, (uint64_t)units * (uint64_t)s_max, 128, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !encode_row_map(&tmA, arena, (uint64_t)L.total_bytes / 256, 64, CU_TENSOR_MAP_SWIZZLE_NONE))
    return (int)cudaErrorNotSupported;
  const int max_t = (int)((maxS + 255) / 256);
  const long long items = 2ll * units * max_t;
  enc_assign_tc<<<(unsigned)std::min<long long>(items, sms), kAtThreads, kAtSmem, st>>>(A, tmK, tmV, tmA, items, max_t);
  enc_finish<<<dim3((maxS + kFinPos - 1) / kFinPos, units, 2), 256, 0, st>>>(A);
  enc_undecided<<<dim3((unsigned)und_blocks((int)units), units, 2), kUndThreads, 0, st>>>(A);
  if (full) {  // Eq. 6 utilities, then each side's pooled top-N per request
    const unsigned m = (unsigned)m_obs;
    if ((e = cudaFuncSetAttribute(enc_util_f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(UtilSmem))) !=
        cudaSuccess)
      return (int)e;
    enc_util_f<<<dim3((maxS + kUtPos - 1) / kUtPos, units), 256, sizeof(UtilSmem), st>>>(A);
    enc_pool_f<<<dim3(kSelCtas * (unsigned)(units / p.n_kv_heads), 2), kSelThreads, 0, st>>>(A);
    // the requests whose utilities the errors leave undecided
    enc_obs_logit<2><<<dim3((maxS + 127) / 128, units), 128, 0, st>>>(A);
    enc_obs_softmax<2><<<dim3(m, units), 1024, 0, st>>>(A);
    enc_obs_y<<<dim3(m, units), 128, 0, st>>>(A);
    enc_util<<<dim3((maxS + 127) / 128, units), 128, 0, st>>>(A);
    enc_pool<<<units / p.n_kv_heads, 1024, 0, st>>>(A, 0);
    enc_pool<<<units / p.n_kv_heads, 1024, 0, st>>>(A, 1);
  } else {
    enc_slots<<<dim3(kSelCtas * (unsigned)units, 2), kSelThreads, 0, st>>>(A);
    enc_slots_exact<<<dim3(units, 2), 1024, 0, st>>>(A);
  }
  enc_order<<<kSelCtas * (unsigned)units, kSelThreads, 0, st>>>(A);
  enc_tile_count<<<dim3((unsigned)L.max_tiles, units), kTile, 0, st>>>(A);
  enc_tile_table<<<units, 1024, 0, st>>>(A);
  enc_tile_fill<<<dim3((unsigned)L.max_tiles, units), kTile, 0, st>>>(A);
  const int maxN = std::max(L.max_nk, L.max_nv);
  if (maxN > 0) enc_quant<<<dim3((unsigned)(maxN + 7) / 8, units, 2), 256, 0, st>>>(A);
  if (full) enc_set_counts<<<(units + 127) / 128, 128, 0, st>>>(A, units);
  return (int)cudaGetLastError();
}

}  // namespace akv
