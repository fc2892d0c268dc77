// sample_f32_wax.cu -- instantiations of the several-integral kernel with the wide CTA, FP32 peaks with the strata per axis (§3.2).
// (Split into several translation units so that they compile in parallel.)
#include "sample_impl.cuh"

namespace vp {

template <int DMAX> static const void *kptr_many_f32_wax_d(int kind) {
    switch (kind) {
        case VP_GAUSS: return (const void *)k_sample_many<DMAX, false, false, VP_GAUSS, true, true>;
        case VP_BALL: return (const void *)k_sample_many<DMAX, false, false, VP_BALL, true, true>;
        case VP_EXPNORM: return (const void *)k_sample_many<DMAX, false, false, VP_EXPNORM, true, true>;
    }
    return nullptr;
}
const void *kptr_many_f32_wax(int bucket, int kind) {
    switch (bucket) {
        case 0: return kptr_many_f32_wax_d<4>(kind);
        case 1: return kptr_many_f32_wax_d<8>(kind);
        case 2: return kptr_many_f32_wax_d<12>(kind);
    }
    return nullptr;
}

}  // namespace vp
