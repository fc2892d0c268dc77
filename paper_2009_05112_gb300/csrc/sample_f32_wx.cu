// sample_f32_wx.cu -- instantiations of the several-integral kernel with the wide CTA, FP32 peaks, dimension-exact buckets.
// (Split into several translation units so that they compile in parallel.)
#include "sample_impl.cuh"

namespace vp {

template <int DMAX> static const void *kptr_many_f32_wx_d(int kind) {
    switch (kind) {
        case VP_GAUSS: return (const void *)k_sample_many<DMAX, true, false, VP_GAUSS, false, true>;
        case VP_BALL: return (const void *)k_sample_many<DMAX, true, false, VP_BALL, false, true>;
        case VP_EXPNORM: return (const void *)k_sample_many<DMAX, true, false, VP_EXPNORM, false, true>;
    }
    return nullptr;
}
const void *kptr_many_f32_wx(int bucket, int kind) {
    switch (bucket) {
        case 0: return kptr_many_f32_wx_d<4>(kind);
        case 1: return kptr_many_f32_wx_d<8>(kind);
        case 2: return kptr_many_f32_wx_d<12>(kind);
    }
    return nullptr;
}

}  // namespace vp
