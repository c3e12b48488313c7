// fr_plain_wild.cu -- the kernels of fr_plain.cuh for Mandelbulb requests whose
// iterates may overflow (R.wild), which take the general orbit step, and for batch
// launches with such requests (a translation unit of its own so that it compiles in
// parallel with the rest).
#include "fr_plain.cuh"

namespace fr {

// Single requests.  One unroll depth; at 1, 2 and 4 the 1080p frame of power 8 with
// bailout 300 takes 0.797, 0.788, 0.785 ms (on the counting kernel 0.801, on kernels of
// its own before the orbit step was split in two 0.834), Phong 1.17, 1.15, 1.15 (1.18, 1.25),
// the analytic normal 0.80, 0.79, 0.80 (0.81, 0.82), n = 5 with bailout 1e4 0.96, 0.93,
// 0.93 (0.99, 0.97), its 160x90 thumbnail 0.214, 0.206, 0.210 (0.216, 0.294).
template <bool PHONG, int BAN>
static cudaError_t single_t(const DevReq &R, int block, cudaStream_t s)
{
    return R.spl > 1 ? launch_plain_t<4, 2, false, PHONG, BAN, true>(R, block, s)
                     : launch_plain_t<4, 2, false, PHONG, BAN>(R, block, s);
}

cudaError_t launch_plain_wild(const DevReq &R, int block, cudaStream_t s)
{
    if (R.normal_mode == 2) return R.shading ? single_t<true, 1>(R, block, s) : single_t<false, 1>(R, block, s);
    return R.shading ? single_t<true, 0>(R, block, s) : single_t<false, 0>(R, block, s);
}

template <int BULB>
static cudaError_t grid_t(const BatchArgs &A, long long ctas, int block, bool phong, bool lanes, cudaStream_t s)
{
    if (lanes) return phong ? launch_batch_plain_t<1, false, true, true, BULB>(A, ctas, block, s)
                            : launch_batch_plain_t<1, false, false, true, BULB>(A, ctas, block, s);
    return phong ? launch_batch_plain_t<1, false, true, false, BULB>(A, ctas, block, s)
                 : launch_batch_plain_t<1, false, false, false, BULB>(A, ctas, block, s);
}

template <int BULB>
static cudaError_t refill_t(const BatchArgs &A, int block, bool phong, bool lanes, cudaStream_t s)
{
    if (lanes) return phong ? launch_batch_refill_t<1, false, true, true, BULB>(A, block, s)
                            : launch_batch_refill_t<1, false, false, true, BULB>(A, block, s);
    return phong ? launch_batch_refill_t<1, false, true, false, BULB>(A, block, s)
                 : launch_batch_refill_t<1, false, false, false, BULB>(A, block, s);
}

cudaError_t launch_batch_plain_wild(const BatchArgs &A, long long ctas, int block, bool phong, bool lanes, int bulb,
                                    cudaStream_t s)
{
    return bulb == 4 ? grid_t<4>(A, ctas, block, phong, lanes, s) : grid_t<5>(A, ctas, block, phong, lanes, s);
}

cudaError_t launch_batch_refill_wild(const BatchArgs &A, int block, bool phong, bool lanes, int bulb, cudaStream_t s)
{
    return bulb == 4 ? refill_t<4>(A, block, phong, lanes, s) : refill_t<5>(A, block, phong, lanes, s);
}

}  // namespace fr
