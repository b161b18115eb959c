// k_lean_c128.cu -- in-place slab passes of complex128 states in FP64.
#include "k_lean.cuh"

namespace qs {

int launch_lean_c128(const LaunchCtx &c, const LeanPassArgs &a, const DevPass &h, char *err, size_t errlen)
{
    constexpr int B = kStageBitsC128;
    if (a.stage_bits == B - 1)
        return small_slab(a, h, 512) ? launch_lean_t<double, B - 1, 512, 1, false, 0, true, true>(c, a, h, err, errlen)
                                     : launch_lean_t<double, B - 1, 512, 1, false, 0, true>(c, a, h, err, errlen);
    return small_slab(a, h, 256) ? launch_lean_t<double, B, 256, 2, false, 0, true, true>(c, a, h, err, errlen)
                                 : launch_lean_t<double, B, 256, 2, false, 0, true>(c, a, h, err, errlen);
}

}  // namespace qs
