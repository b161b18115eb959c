// k_lean_df.cu -- in-place slab passes of complex128 states in double-float form.
#include "k_lean.cuh"

namespace qs {

int launch_lean_df(const LaunchCtx &c, const LeanPassArgs &a, const DevPass &h, char *err, size_t errlen)
{
    constexpr int B = kStageBitsC128;
    if (a.stage_bits == B - 1)
        return small_slab(a, h, 512) ? launch_lean_t<double, B - 1, 512, 1, true, 0, true, true>(c, a, h, err, errlen)
                                     : launch_lean_t<double, B - 1, 512, 1, true, 0, true>(c, a, h, err, errlen);
    if (small_slab(a, h, 256)) return launch_lean_t<double, B, 256, 2, true, 0, true, true>(c, a, h, err, errlen);
    return a.full ? launch_lean_t<double, B, 256, 2, true, 0, true>(c, a, h, err, errlen)
                  : launch_lean_t<double, B, 256, 2, true, 0, false>(c, a, h, err, errlen);
}

}  // namespace qs
