// Decode attention: the dispatch by query-group size, the workspace layout, the append path.
// The kernels are in akv_decode.cuh, instantiated per group size in akv_decode_g*.cu (separate units so that
// they compile in parallel).
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>
#include <string>

#include "akv_internal.h"

namespace akv {

std::atomic<int> g_debug_cluster{0}, g_debug_withhold{0};
namespace {
std::mutex g_events_mu;
cudaEvent_t g_ev_scores = nullptr, g_ev_decode = nullptr;
}  // namespace
void set_decode_events(void* after_scores, void* after_decode) {
  std::lock_guard<std::mutex> lk(g_events_mu);
  g_ev_scores = (cudaEvent_t)after_scores;
  g_ev_decode = (cudaEvent_t)after_decode;
}
void get_decode_events(void** after_scores, void** after_decode) {
  std::lock_guard<std::mutex> lk(g_events_mu);
  *after_scores = (void*)g_ev_scores;
  *after_decode = (void*)g_ev_decode;
}

// Workspace of a decode call: anchor scores, query headers and arrival counters, chunk maxima, partial slots.
DecodeWs decode_ws_layout(const Layout& L, int32_t suffix_cap) {
  DecodeWs w;
  const size_t units = L.shape.size();
  const size_t ka = (size_t)((L.max_k + 3) & ~3);
  const size_t nch = (size_t)((L.max_k + CHA - 1) / CHA);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = (off + bytes + 255) & ~(size_t)255;
    return o;
  };
  const bool rope = (L.header.params.flags & AKV_FLAG_ROPE) != 0;
  const size_t s_stride = (size_t)((L.max_len + 63) & ~63);
  w.o_sa = take(rope ? 0 : units * ka * (size_t)L.G * 4);
  w.o_uh = take(units * (size_t)((hdr_bytes(L.G) + 255) & ~255));  // with the heads' arrival counters in the padding
  // chunk maxima: of 64 anchors, or with RoPE of 64 stored tokens
  w.o_cmax = take(units * (rope ? s_stride / 64 : nch) * (size_t)L.G * 4);
  w.o_lg = take(rope ? units * s_stride * (size_t)L.G * 4 : 0);  // RoPE: every token's logits
  w.o_part = take((size_t)(kMaxGrid + units) * (size_t)part_floats(L.G) * 4);
  w.o_suf = take(units * (size_t)((suffix_cap + kSuffixChunk - 1) / kSuffixChunk) * (size_t)suf_floats(L.G) * 4);
  w.total = off;
  return w;
}

template <int GS>
int launch_g(const Layout& L, const akv_params& p, const void* arena, size_t arena_bytes, const void* q, void* out, float* out_f32,
             float sm_scale, const DecodeSuffix& sfx, void* ws, void* stream, std::string* why);

int launch_decode(const Layout& L, const akv_params& p, const void* arena, size_t arena_bytes, const void* q, void* out, float* out_f32,
                  float sm_scale, const DecodeSuffix& sfx, void* ws, void* stream, std::string* why) {
  switch (L.G) {
    case 1: return launch_g<1>(L, p, arena, arena_bytes, q, out, out_f32, sm_scale, sfx, ws, stream, why);
    case 2: return launch_g<2>(L, p, arena, arena_bytes, q, out, out_f32, sm_scale, sfx, ws, stream, why);
    case 4: return launch_g<4>(L, p, arena, arena_bytes, q, out, out_f32, sm_scale, sfx, ws, stream, why);
    case 8: return launch_g<8>(L, p, arena, arena_bytes, q, out, out_f32, sm_scale, sfx, ws, stream, why);
  }
  *why = "unsupported group size";
  return -1;
}

// The append path of the dense suffix (Appendix E.2): CTA b copies the new key and value rows of
// request b's KV heads to row len[b] of their suffix blocks, then counts the token in.  Every
// thread reads len[b] before the barrier; thread 0 writes it after.
__global__ void __launch_bounds__(256) akv_suffix_append_kernel(int H, const uint4* K_new, const uint4* V_new,
                                                                 uint4* K_suf, uint4* V_suf, int32_t* len, int cap) {
  const int b = blockIdx.x;
  const int n = len[b];
  const bool room = n >= 0 && n < cap;
  if (room) {
    for (int e = threadIdx.x; e < H * 16; e += blockDim.x) {  // 16 x 16 bytes per row
      const size_t row = (size_t)b * H + e / 16;
      K_suf[(row * cap + n) * 16 + e % 16] = K_new[row * 16 + e % 16];
      V_suf[(row * cap + n) * 16 + e % 16] = V_new[row * 16 + e % 16];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && room) len[b] = n + 1;
}

int launch_suffix_append(int32_t B, int32_t H, const void* K_new, const void* V_new, void* K_suf, void* V_suf,
                         int32_t* len, int32_t cap, void* stream) {
  akv_suffix_append_kernel<<<B, 256, 0, (cudaStream_t)stream>>>(H, (const uint4*)K_new, (const uint4*)V_new,
                                                                (uint4*)K_suf, (uint4*)V_suf, len, cap);
  return (int)cudaGetLastError();
}

const char* cuda_error_string(int err) { return cudaGetErrorString((cudaError_t)err); }

}  // namespace akv
