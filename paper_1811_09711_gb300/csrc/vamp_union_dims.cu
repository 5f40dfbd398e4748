// Union pass kernels by range of d (any number of bins).  For d of 13 to 16 the
// any-shape kernel is the faster one (d = 15, K = 30, 1e6 calls: 507 us against
// 584 with a kernel of that range).
#include "vamp_union.cuh"

namespace vamp {
void add_pass_variants_union_dims(std::vector<PassVariant>& v)
{
    v.push_back(make_union_variant_dims<1, 4>());
    v.push_back(make_union_variant_dims<5, 8>());
    v.push_back(make_union_variant_dims<9, 12>());
}
}  // namespace vamp
