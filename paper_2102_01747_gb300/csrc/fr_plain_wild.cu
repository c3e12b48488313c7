// fr_plain_wild.cu -- the batch kernels of fr_plain.cuh for launches with Mandelbulb
// requests whose iterates may overflow (R.wild), which take the general orbit step
// (a translation unit of its own so that it compiles in parallel with the rest).
#include "fr_plain.cuh"

namespace fr {

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
