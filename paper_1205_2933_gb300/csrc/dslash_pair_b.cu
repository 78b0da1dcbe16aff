// The paired FP32 Dslash for Ls = 16 (see dslash_pair.cuh).
#include "dslash_pair.cuh"

namespace dwf {

template void dslash_pair_ls<16>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);

}  // namespace dwf
