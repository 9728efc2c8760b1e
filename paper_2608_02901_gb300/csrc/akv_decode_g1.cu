// The decode kernels for one query head per KV head.
#include "akv_decode.cuh"

namespace akv {
template int launch_g<1>(const Layout&, const akv_params&, const void*, size_t, const void*, void*, float*, float,
                         const DecodeSuffix&, void*, void*, std::string*);
}  // namespace akv
