// FP64 pass kernels by range of d (any number of bins).
#include "vamp_pass.cuh"

namespace vamp {
void add_pass_variants_f64_dims(std::vector<PassVariant>& v)
{
    v.push_back(make_variant_dims<double, 1, 1, 4>());
    v.push_back(make_variant_dims<double, 1, 5, 8>());
    v.push_back(make_variant_dims<double, 1, 9, 12>());
    v.push_back(make_variant_dims<double, 1, 13, 16>());
}
}  // namespace vamp
