// k_lean.cu -- in-place slab passes of complex64 states, and the choice between the arithmetics.
#include "k_lean.cuh"

namespace qs {

int launch_lean_pass(const LaunchCtx &c, const LeanPassArgs &a, const DevPass &h, char *err, size_t errlen)
{
    if (c.dt == QS_C128) return a.df ? launch_lean_df(c, a, h, err, errlen) : launch_lean_c128(c, a, h, err, errlen);
    constexpr int B = kStageBitsC64;
    if (a.stage_bits == B - 1) return launch_lean_t<float, B - 1, 512, 1, false, 0, true>(c, a, h, err, errlen);
    if (a.nwords > 2000) return launch_lean_t<float, B, 256, 2, false, 0, true>(c, a, h, err, errlen);
    if (a.full)
        return a.nwords <= 480 ? launch_lean_t<float, B, 256, 2, false, 480, true>(c, a, h, err, errlen)
                               : launch_lean_t<float, B, 256, 2, false, 2000, true>(c, a, h, err, errlen);
    return a.nwords <= 480 ? launch_lean_t<float, B, 256, 2, false, 480, false>(c, a, h, err, errlen)
                           : launch_lean_t<float, B, 256, 2, false, 2000, false>(c, a, h, err, errlen);
}

}  // namespace qs
