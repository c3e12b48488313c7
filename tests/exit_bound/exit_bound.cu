// The ball outside which the kernels take no distances (set_exit) against the distance
// estimates themselves, on the host: random parameters, random points at and beyond a
// radius, plain double arithmetic.  Prints "points balls worst", worst the smallest
// ratio of a point's estimate to the bound at its radius.
#include "fr_api.cu"

#include <complex>
#include <random>

namespace {

double estimate(const fr::DevReq &R, const double x[3])
{
    const int p = R.power;
    double m, dz = 1.0;
    if (R.kind == FR_KIND_BULB) {
        double w[3] = {x[0], x[1], x[2]};
        for (int k = 0; k < R.max_iter; k++) {
            const double r = std::sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
            const double b = p * std::acos(w[1] / r), a = p * std::atan2(w[0], w[2]), rn = std::pow(r, p);
            dz = p * std::pow(r, p - 1) * dz + 1.0;
            w[0] = rn * std::sin(b) * std::sin(a) + x[0];
            w[1] = rn * std::cos(b) + x[1];
            w[2] = rn * std::sin(b) * std::cos(a) + x[2];
            if (w[0] * w[0] + w[1] * w[1] + w[2] * w[2] > R.esc2) break;
        }
        m = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    } else {
        double z[4] = {x[0], x[1], x[2], R.slice_w};
        const double c[4] = {R.c.x, R.c.y, R.c.z, R.c.w};
        for (int k = 0; k < R.max_iter; k++) {
            const double v2 = z[1] * z[1] + z[2] * z[2] + z[3] * z[3], n = std::sqrt(z[0] * z[0] + v2);
            dz *= p * std::pow(n, p - 1);
            // a power of a quaternion is one of the complex number a + i |v| in the plane of v
            const std::complex<double> q = std::pow(std::complex<double>(z[0], std::sqrt(v2)), p);
            const double f = v2 > 0.0 ? q.imag() / std::sqrt(v2) : 0.0;
            z[0] = q.real() + c[0];
            for (int j = 1; j < 4; j++) z[j] = f * z[j] + c[j];
            if (z[0] * z[0] + z[1] * z[1] + z[2] * z[2] + z[3] * z[3] > R.esc2) break;
        }
        m = z[0] * z[0] + z[1] * z[1] + z[2] * z[2] + z[3] * z[3];
    }
    return 0.25 * std::log(m) * std::sqrt(m) / dz;
}

}  // namespace

int main()
{
    std::mt19937_64 gen(2102);
    auto uniform = [&](double a, double b) { return a + (b - a) * (double)(gen() >> 11) * 0x1p-53; };
    long long points = 0, balls = 0;
    double worst = 1e30;
    for (int i = 0; i < 6000; i++) {
        fr::DevReq R{};
        R.kind = i & 1;
        R.power = R.kind == FR_KIND_BULB ? 2 + (int)uniform(0, 15) : 2 + (int)uniform(0, 2);
        const double k = std::pow(10.0, uniform(-2.0, 0.2));
        if (R.kind != FR_KIND_BULB)
            R.c = make_float4(uniform(-k, k), uniform(-k, k), uniform(-k, k), uniform(-k, k));
        R.max_iter = 1 + (int)std::pow(10.0, uniform(0.0, 2.0));
        R.esc2 = (float)std::pow(10.0, uniform(-0.3, 2.5));
        R.slice_w = R.kind == FR_KIND_BULB ? 0.0f : (float)uniform(-1.0, 1.0);
        R.bound_r2 = (float)std::pow(uniform(1.0, 3.0), 2.0);
        R.max_steps = 256;
        R.eps = 5e-4f;
        R.max_step = 0.2f;
        R.eye = make_float4(0.0f, 0.0f, 2.5f, 0.0f);
        set_exit(R);
        const bool ball = R.exit_r2 > 0.0f;
        balls += ball;
        for (int j = 0; j < 40; j++) {
            // half of the points on the ball's own radius
            const double r = ball && j % 2 ? std::sqrt((double)R.exit_r2) : uniform(1.0, 3.0);
            int n = 0;
            const double bound = distance_bound(R, r, &n);
            if (!(bound > 0.0)) continue;
            double x[3] = {uniform(-1, 1), uniform(-1, 1), uniform(-1, 1)};
            const double l = std::sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
            const double s = r * (j % 4 < 2 ? 1.0 : uniform(1.0, 1.5)) / l;
            for (double &v : x) v *= s;
            const double d = estimate(R, x);
            points++;
            if (!(d / bound >= worst)) worst = d / bound;
            if (ball && j % 2 && !(d > R.eps)) worst = -1.0;
        }
    }
    std::printf("%lld %lld %.6f\n", points, balls, worst);
    return 0;
}
