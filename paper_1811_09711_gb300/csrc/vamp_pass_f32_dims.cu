// FP32-eval pass kernels by range of d (any number of bins).
#include "vamp_pass.cuh"

namespace vamp {
void add_pass_variants_f32_dims(std::vector<PassVariant>& v)
{
    v.push_back(make_variant_dims<float, 2, 1, 4>());
    v.push_back(make_variant_dims<float, 2, 5, 8>());
    v.push_back(make_variant_dims<float, 2, 9, 12>());
    v.push_back(make_variant_dims<float, 2, 13, 16>());
    v.push_back(make_variant_dims<float, 1, 1, 4>());
    v.push_back(make_variant_dims<float, 1, 5, 8>());
    v.push_back(make_variant_dims<float, 1, 9, 12>());
    v.push_back(make_variant_dims<float, 1, 13, 16>());
    // one call per thread, four CTAs per SM (64 registers): the fastest at 1e6
    // calls of few channels (d = 8, K = 6: 114 us against 131 and 146)
    v.push_back(make_variant_dims<float, 1, 1, 4, 4>());
    v.push_back(make_variant_dims<float, 1, 5, 8, 4>());
    v.push_back(make_variant_dims<float, 1, 9, 12, 4>());
    v.push_back(make_variant_dims<float, 1, 13, 16, 4>());
}
}  // namespace vamp
