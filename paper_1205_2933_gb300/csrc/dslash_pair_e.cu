// The paired FP32 Dslash for Ls = 48, 64 (see dslash_pair.cuh).
#include "dslash_pair.cuh"

namespace dwf {

template void dslash_pair_ls<48>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);
template void dslash_pair_ls<64>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);

}  // namespace dwf
