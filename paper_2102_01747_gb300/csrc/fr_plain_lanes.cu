// fr_plain_lanes.cu -- the one-ray-per-thread kernels of fr_plain.cuh with a
// pixel's 2, 4 or 8 samples on adjacent lanes (LANES, render_pixel_lanes), for
// requests with R.spl > 1 (a translation unit of its own so that it compiles
// in parallel with the rest).  Phong requests take the Phong-capable
// instantiation, the Mandelbulb's analytic normal the BAN one, both at unroll depth 1,
// and Lambert Mandelbulb requests of the power 8 with a stencil one compiled for that
// power.  Depths of the stencil's Lambert Mandelbulbs: power 8 with 2 samples at 1080p
// 1.00 ms rolled, 0.96 at depth 2, 0.98 at 4 (4K with 4 samples 5.84, 5.66 ms), n = 4 with 4
// samples at 1283x723 1.64, 1.64, 1.56 ms.
#include "fr_plain.cuh"

namespace fr {

cudaError_t launch_plain_lanes(const DevReq &R, int block, bool count, cudaStream_t s)
{
    if (R.kind == 0) {
        if (R.shading)
            return count ? launch_plain_t<0, 1, true, true, false, true>(R, block, s)
                         : launch_plain_t<0, 1, false, true, false, true>(R, block, s);
        return count ? launch_plain_t<0, 1, true, false, false, true>(R, block, s)
                     : launch_plain_t<0, 1, false, false, false, true>(R, block, s);
    }
    if (R.normal_mode == 2) {
        if (R.shading)
            return count ? launch_plain_t<1, 1, true, true, true, true>(R, block, s)
                         : launch_plain_t<1, 1, false, true, true, true>(R, block, s);
        return count ? launch_plain_t<1, 1, true, false, true, true>(R, block, s)
                     : launch_plain_t<1, 1, false, false, true, true>(R, block, s);
    }
    if (R.shading)
        return count ? launch_plain_t<1, 1, true, true, false, true>(R, block, s)
                     : launch_plain_t<1, 1, false, true, false, true>(R, block, s);
    if (count) return launch_plain_t<1, 1, true, false, false, true>(R, block, s);
    if (R.power == 8 && !R.bulb_alg) return launch_plain_t<3, 2, false, false, false, true>(R, block, s);
    return R.power == 8 ? launch_plain_t<2, 2, false, false, false, true>(R, block, s)
                        : launch_plain_t<1, 4, false, false, false, true>(R, block, s);
}

cudaError_t launch_batch_plain_lanes(const BatchArgs &A, long long ctas, int block, bool count, bool phong,
                                     cudaStream_t s)
{
    if (phong) return count ? launch_batch_plain_t<1, true, true, true>(A, ctas, block, s)
                            : launch_batch_plain_t<1, false, true, true>(A, ctas, block, s);
    return count ? launch_batch_plain_t<1, true, false, true>(A, ctas, block, s)
                 : launch_batch_plain_t<1, false, false, true>(A, ctas, block, s);
}

cudaError_t launch_batch_refill_lanes(const BatchArgs &A, int block, bool count, bool phong, cudaStream_t s)
{
    if (phong) return count ? launch_batch_refill_t<1, true, true, true>(A, block, s)
                            : launch_batch_refill_t<1, false, true, true>(A, block, s);
    return count ? launch_batch_refill_t<1, true, false, true>(A, block, s)
                 : launch_batch_refill_t<1, false, false, true>(A, block, s);
}

}  // namespace fr
