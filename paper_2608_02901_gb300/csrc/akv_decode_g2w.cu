// The decode kernels for two query heads per KV head whose tiles have more weight rows than staged anchor-value rows.
#include "akv_decode.cuh"

namespace akv {
template <>
const void* wide_decode_kernel<2>(int codec, int rope) {
  if (rope) return codec ? (const void*)akv_decode_kernel<2, 1, kRope, true> : (const void*)akv_decode_kernel<2, 0, kRope, true>;
  return codec ? (const void*)akv_decode_kernel<2, 1, kTableGlobal, true> : (const void*)akv_decode_kernel<2, 0, kTableGlobal, true>;
}
}  // namespace akv
