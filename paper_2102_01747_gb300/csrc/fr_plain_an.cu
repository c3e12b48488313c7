// fr_plain_an.cu -- the single-request kernel of fr_plain.cuh compiled with the
// Mandelbulb's analytic normal, for requests that ask for it (a translation
// unit of its own so that it compiles in parallel with the rest); requests of
// the power 8 take the instantiation compiled for that power.  Unroll depths as
// measured: Lambert, power 8, 0.70 ms rolled, 0.66 at depth 2 and 0.67 at 4 for
// the 1080p frame; n = 5 at 1283x723 0.66, 0.68, 0.70 ms; Phong as in fr_plain.cu.
#include "fr_plain.cuh"

namespace fr {

cudaError_t launch_plain_ban(const DevReq &R, int block, bool count, cudaStream_t s)
{
    if (R.shading) {
        if (count) return launch_plain_t<1, 1, true, true, true>(R, block, s);
        if (R.power == 8 && !R.bulb_alg) return launch_plain_t<3, 4, false, true, true>(R, block, s);
        return R.power == 8 ? launch_plain_t<2, 4, false, true, true>(R, block, s)
                            : launch_plain_t<1, 4, false, true, true>(R, block, s);
    }
    if (count) return launch_plain_t<1, 1, true, false, true>(R, block, s);
    if (R.power == 8 && !R.bulb_alg) return launch_plain_t<3, 2, false, false, true>(R, block, s);
    return R.power == 8 ? launch_plain_t<2, 2, false, false, true>(R, block, s)
                        : launch_plain_t<1, 1, false, false, true>(R, block, s);
}

}  // namespace fr
