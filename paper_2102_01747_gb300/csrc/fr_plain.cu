// fr_plain.cu -- launches of the one-ray-per-thread kernels of fr_plain.cuh
// (single requests that ask for the Mandelbulb's analytic normal go to
// fr_plain_an.cu).
#include "fr_plain.cuh"

namespace fr {

// Of a batch launch: whether some request has its samples on adjacent lanes, and the
// Mandelbulb's KIND: 1, or with wild requests among them 5, which holds both steps,
// or 4 where the wild ones are at least half of the Mandelbulbs' work (pixels x
// samples x iteration cap), since the general step serves every request.  64 mixed
// requests with the Mandelbulbs' bailouts at 10^(22/n), as 4 and as 5: one wild request
// 21.5 and 20.6 ms, a quarter of them 21.2 and 20.8, half 20.4 and 20.8, 15 of 16 20.1 and
// 20.9 (none wild 20.2); on the counting kernels 22.3, 22.0, 21.1 and 20.7.
static void traits(const BatchArgs &A, bool &lanes, int &bulb)
{
    double wild = 0.0, all = 0.0;
    lanes = false;
    for (int i = 0; i < A.n_reqs; i++) {
        const DevReq &R = A.reqs[i];
        lanes = lanes || R.spl > 1;
        if (R.kind != 1) continue;
        const double work = (double)R.n_units * R.spp * R.max_iter;
        all += work;
        if (R.wild) wild += work;
    }
    bulb = wild == 0.0 ? 1 : wild < 0.5 * all ? 5 : 4;
}

// phong: some request of the launch uses Phong shading (the Phong-capable code
// then serves every request of the launch, at unroll 1)
cudaError_t launch_batch_plain(const BatchArgs &A, long long ctas, int block, int unroll, bool count,
                               bool phong, cudaStream_t s)
{
    bool lanes;
    int bulb;
    traits(A, lanes, bulb);
    if (bulb != 1 && !count) return launch_batch_plain_wild(A, ctas, block, phong, lanes, bulb, s);
    if (lanes) return launch_batch_plain_lanes(A, ctas, block, count, phong, s);
    if (phong) return count ? launch_batch_plain_t<1, true, true>(A, ctas, block, s)
                            : launch_batch_plain_t<1, false, true>(A, ctas, block, s);
    if (count) return launch_batch_plain_t<1, true, false>(A, ctas, block, s);
    if (unroll == 2) return launch_batch_plain_t<2, false, false>(A, ctas, block, s);
    return launch_batch_plain_t<1, false, false>(A, ctas, block, s);
}

cudaError_t launch_batch_refill(const BatchArgs &A, int block, int unroll, bool count, bool phong, cudaStream_t s)
{
    bool lanes;
    int bulb;
    traits(A, lanes, bulb);
    if (bulb != 1 && !count) return launch_batch_refill_wild(A, block, phong, lanes, bulb, s);
    if (lanes) return launch_batch_refill_lanes(A, block, count, phong, s);
    if (phong) return count ? launch_batch_refill_t<1, true, true>(A, block, s)
                            : launch_batch_refill_t<1, false, true>(A, block, s);
    if (count) return launch_batch_refill_t<1, true, false>(A, block, s);
    if (unroll == 2) return launch_batch_refill_t<2, false, false>(A, block, s);
    return launch_batch_refill_t<1, false, false>(A, block, s);
}

// Phong requests run the Phong-capable instantiation at one unroll depth;
// Mandelbulb requests of the paper's power 8 (not counting) an instantiation for
// that power.  The loops take at least two steps per trip, the
// Mandelbulb's Phong ones four: a step is long enough to leave the loop's own branch and
// counter waiting on its chain, and unrolled the next step's start overlaps them.
// Measured at depths 1, 2 and 4, the Mandelbulb: the 1080p frame 0.70, 0.64, 0.66 ms, n = 6 at
// 640x360 0.52, 0.47, 0.50 ms, n = 3 at 1283x723 0.95, 0.94, 0.92 ms; Phong at
// 1080p 1.06, 1.07, 1.02 ms, at 320x180 0.38, 0.39, 0.34 ms.  The Julia set's
// depth counts pairs of steps (julia_de): the 4K frame 1.335, 1.320, 1.329 ms.
cudaError_t launch_plain(const DevReq &R, int block, int unroll, bool count, cudaStream_t s)
{
    if (R.wild && !count) return launch_plain_wild(R, block, s);
    if (R.spl > 1) return launch_plain_lanes(R, block, count, s);
    if (R.kind == 1 && R.normal_mode == 2) return launch_plain_ban(R, block, count, s);
    if (R.shading) {
        if (R.kind == 0)
            return count ? launch_plain_t<0, 1, true, true>(R, block, s) : launch_plain_t<0, 2, false, true>(R, block, s);
        if (count) return launch_plain_t<1, 1, true, true>(R, block, s);
        if (R.power == 8 && !R.bulb_alg) return launch_plain_t<3, 4, false, true>(R, block, s);
        return R.power == 8 ? launch_plain_t<2, 4, false, true>(R, block, s) : launch_plain_t<1, 4, false, true>(R, block, s);
    }
    if (count) return R.kind == 0 ? launch_plain_t<0, 1, true>(R, block, s)
                                  : launch_plain_t<1, 1, true>(R, block, s);
    if (R.kind == 0) {
        // an image whose warps run almost alone (at most four per scheduler) is best
        // served by the fewest tests, unless the orbit ends before the four steps do: with
        // pairs and with quads, 256x256 of one iteration 43.1 and 53.3 us (49 with a test
        // after each step), of two 41.1 and 49.0, of three 55.5 and 55.4, of eleven 78 and 70
        if (plain_tiles(R) <= 2432 && R.max_iter > 2) return launch_plain_t<0, kJuliaQuads, false>(R, block, s);
        return unroll == 4 ? launch_plain_t<0, 4, false>(R, block, s) : launch_plain_t<0, 2, false>(R, block, s);
    }
    if (R.power == 8 && !R.bulb_alg)
        return unroll == 4 ? launch_plain_t<3, 4, false>(R, block, s) : launch_plain_t<3, 2, false>(R, block, s);
    if (R.power == 8)
        return unroll == 4 ? launch_plain_t<2, 4, false>(R, block, s) : launch_plain_t<2, 2, false>(R, block, s);
    return unroll == 4 ? launch_plain_t<1, 4, false>(R, block, s) : launch_plain_t<1, 2, false>(R, block, s);
}

}  // namespace fr
