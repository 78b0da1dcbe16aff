// The paired FP32 Dslash for Ls = 4, 8 (see dslash_pair.cuh).
#include "dslash_pair.cuh"

namespace dwf {

template void dslash_pair_ls<4>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);
template void dslash_pair_ls<8>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);

}  // namespace dwf
