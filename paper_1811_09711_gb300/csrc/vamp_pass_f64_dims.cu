// FP64 pass kernels by range of d (any number of bins), three CTAs per SM: 80
// registers and some spilled ones against 118 to 128, for half as many warps
// again to hide the integer chains behind (d = 8, K = 6, 1e6 calls: 391 -> 371
// us; generation 436 -> 398; d = 14, K = 64, 1e7 calls: 54.1 -> 52.7 ms).
#include "vamp_pass.cuh"

namespace vamp {
void add_pass_variants_f64_dims(std::vector<PassVariant>& v)
{
    v.push_back(make_variant_dims<double, 1, 1, 4, 3>());
    v.push_back(make_variant_dims<double, 1, 5, 8, 3>());
    v.push_back(make_variant_dims<double, 1, 9, 12, 3>());
    v.push_back(make_variant_dims<double, 1, 13, 16, 3>());
}
}  // namespace vamp
