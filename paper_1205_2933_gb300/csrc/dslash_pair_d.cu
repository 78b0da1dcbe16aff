// The paired FP32 Dslash for Ls = 20, 24, 32 (see dslash_pair.cuh).
#include "dslash_pair.cuh"

namespace dwf {

template void dslash_pair_ls<20>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);
template void dslash_pair_ls<24>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);
template void dslash_pair_ls<32>(dwf_ctx *, float2 *, const float2 *, bool, int, int, double *, int, const ZUpdate *);

}  // namespace dwf
