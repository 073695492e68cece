// Host checks of the library's host/device arithmetic (test_host_arithmetic.py compiles and runs this).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "geometry.cuh"

using namespace pncg;
typedef v3<double> D3;
typedef v3<float> F3;

static F3 tof(D3 a) { return mkv((float)a.x, (float)a.y, (float)a.z); }
static D3 tod(F3 a) { return mkv((double)a.x, (double)a.y, (double)a.z); }

// cand_bound over pairs in a random place and turn in a cell of size s, sin^2 of the angle in [s0, s1], the distance up to
// 0.98 dhat: prints how many bounds lie above the true distance (double), and the largest excess in dhat
static void bounds(int ee, double ratio, double s0, double s1, int n)
{
    std::mt19937_64 g(1);
    std::uniform_real_distribution<double> U(0, 1);
    std::normal_distribution<double> N;
    const double dhat = 1e-3, L = ratio * dhat, infl = 3 * dhat, s = L + (ee ? 1 : 2) * infl;
    int above = 0;
    double worst = 0;
    for (int t = 0; t < n; ++t) {
        const double th = std::sqrt(s0 * std::pow(s1 / s0, U(g))), d = (0.02 + 0.96 * U(g)) * dhat, l2 = L * std::pow(10.0, -2 * U(g));
        double q[4], nq = 0;
        for (double &v : q) { v = N(g); nq += v * v; }
        for (double &v : q) v /= std::sqrt(nq);
        auto rot = [&](double x, double y, double z) {
            const double w = q[0], a = q[1], b = q[2], c = q[3];
            return mkv((1 - 2 * (b * b + c * c)) * x + 2 * (a * b - w * c) * y + 2 * (a * c + w * b) * z,
                       2 * (a * b + w * c) * x + (1 - 2 * (a * a + c * c)) * y + 2 * (b * c - w * a) * z,
                       2 * (a * c - w * b) * x + 2 * (b * c + w * a) * y + (1 - 2 * (a * a + b * b)) * z);
        };
        const D3 o = mkv(U(g) * s, U(g) * s, U(g) * s);
        const double ux = l2 * std::cos(th), uy = l2 * std::sin(th);
        F3 p[4];
        float cf[4];
        F3 tf;
        double cd[4];
        D3 td;
        double lo, ref;
        if (ee) {   // edges p0 p1 and p2 p3
            const double c = U(g), c2 = U(g);
            p[0] = tof(o + rot(-c * L, 0, 0)); p[1] = tof(o + rot((1 - c) * L, 0, 0));
            p[2] = tof(o + rot(-c2 * ux, -c2 * uy, d)); p[3] = tof(o + rot((1 - c2) * ux, (1 - c2) * uy, d));
            const F3 e0 = p[1] - p[0], e1 = p[3] - p[2];
            lo = cand_bound(ee_coeffs<float>(p[0] - p[2], p[1] - p[2], e1, cf, tf), dot(e0, e0), dot(e0, e1), dot(e1, e1), (float)s);
            ref = ee_coeffs<double>(tod(p[0]) - tod(p[2]), tod(p[1]) - tod(p[2]), tod(p[3]) - tod(p[2]), cd, td);
        } else {    // point p0, triangle p1 p2 p3
            double a = U(g), b = U(g);
            if (a + b > 1) { a = 1 - a; b = 1 - b; }
            p[1] = tof(o); p[2] = tof(o + rot(L, 0, 0)); p[3] = tof(o + rot(ux, uy, 0));
            p[0] = tof(o + rot(a * L + b * ux, b * uy, d));
            const F3 e1 = p[2] - p[1], e2 = p[3] - p[1];
            lo = cand_bound(pt_coeffs<float>(p[0] - p[1], e1, e2, cf, tf), dot(e1, e1), dot(e1, e2), dot(e2, e2), (float)s);
            ref = pt_coeffs<double>(tod(p[0]) - tod(p[1]), tod(p[2]) - tod(p[1]), tod(p[3]) - tod(p[1]), cd, td);
        }
        if (!(lo <= ref)) ++above;
        worst = std::max(worst, (lo - ref) / dhat);
    }
    std::printf("%d %.3e\n", above, worst);
}

// Quot<true> against the division: prints how many of n quotients differ
static void quotients(int n)
{
    std::mt19937_64 g(2);
    std::uniform_real_distribution<double> U(1, 2), E(-60, 60);
    int differ = 0;
    for (int t = 0; t < n; ++t) {
        const double a = (g() & 1 ? -1 : 1) * std::ldexp(U(g), (int)E(g)), d = std::ldexp(U(g), (int)E(g));
        if (Quot<true, double>(d)(a) != a / d) ++differ;
    }
    std::printf("%d\n", differ);
}

// b' of the barrier at gaps d = dhat (1 - x), x in [x0, x1]: the rms error, in units of 2^-53, of the FP64 form (whose
// logarithm is the library's on the host) and of -2 r L - r^2 / d with one fused rounding
static void barrier(double x0, double x1, int n)
{
    std::mt19937_64 g(3);
    std::uniform_real_distribution<double> U(0, 1);
    const double dhat = 1e-3;
    long double e = 0, ref = 0;
    for (int t = 0; t < n; ++t) {
        const double d = dhat * (1 - x0 * std::pow(x1 / x0, U(g))), r = d - dhat;
        const long double b = -2.0L * r * log1pl((long double)r / dhat) - (long double)r * r / d;
        double b1, b2;
        barrier_d12r<double, true>(d, r, dhat, b1, b2);
        const double c1 = std::fma(-2.0 * r, std::log1p(r / dhat), -(r * r / d));
        e += (b1 / b - 1) * (b1 / b - 1);
        ref += (c1 / b - 1) * (c1 / b - 1);
    }
    std::printf("%.4f %.4f\n", (double)sqrtl(e / n) * 0x1p53, (double)sqrtl(ref / n) * 0x1p53);
}

int main(int argc, char **argv)
{
    if (argc == 7 && !std::strcmp(argv[1], "bounds"))
        bounds(std::atoi(argv[2]), std::atof(argv[3]), std::atof(argv[4]), std::atof(argv[5]), std::atoi(argv[6]));
    else if (argc == 3 && !std::strcmp(argv[1], "quotients"))
        quotients(std::atoi(argv[2]));
    else if (argc == 5 && !std::strcmp(argv[1], "barrier"))
        barrier(std::atof(argv[2]), std::atof(argv[3]), std::atoi(argv[4]));
    else return 2;
    return 0;
}
