// Host check of the cutoff bits of teno7_f64math.cuh over the magnitudes FP32 holds
// and next to the cutoff's thresholds, at both ends of the error of the approximate
// reciprocal.  Prints "<what> <cases> <differences>" per line.
#include <cstdio>
#include <random>

static float host_err = 1.f;  // the device's approximation is off by up to 2^-22
#define T7_HOST_ERR *host_err
#include "teno7_f64math.cuh"

using namespace t7;

static const float ERR[] = {1.f, 1.f + 2.4e-7f, 1.f - 2.4e-7f};

// a window of one of several forms: a jump, a spike, a kink, noise; unit size, on a
// base that is zero or not
static void shape(std::mt19937_64 &r, int i, double w[5]) {
    std::uniform_real_distribution<double> u(-1, 1);
    const double base = i % 3 == 0 ? 0.0 : u(r), d = u(r), e = pow(10, -6 * fabs(u(r)));
    for (int t = 0; t < 5; t++) {
        switch (i % 5) {
            case 0: w[t] = base + (t > 2 ? d : 0) + e * u(r); break;
            case 1: w[t] = base + (t > 1 ? d : 0) + e * u(r); break;
            case 2: w[t] = base + (t == 2 ? d : 0) + e * u(r); break;
            case 3: w[t] = base + (t > 2 ? d : e) * (t - 2); break;
            default: w[t] = base + u(r); break;
        }
    }
}

static bool differ(const double w[5], const Cut64 &K) {
    return cutoff_bits(w[0], w[1], w[2], w[3], w[4], K) !=
           cutoff_bits_f64(w[0], w[1], w[2], w[3], w[4], K.eps, K.CT, K.kt);
}

// magnitudes: from betas below FP32's least normal number to above its largest
static void check_scale() {
    std::mt19937_64 r(21);
    long n = 0, bad = 0;
    for (float err : ERR) {
        host_err = err;
        for (double CT : {1e-5, 1e-7, 1e-3, 0.2})
            for (double eps : {1e-60, 1e-40, 2.4e-7}) {
                const Cut64 K = cut64(eps, CT, keep_all_factor(CT));
                for (double scale : {1e-24, 1e-20, 3e-19, 1e-19, 1e-18, 1e-15, 1e-6, 1.0, 1e6, 1e15, 1e17, 3e17, 1e18,
                                     2e18, 3e18, 4e18, 6e18, 1e19, 1.4e19, 2e19, 1e20, 1e24})
                    for (int i = 0; i < 2000; i++) {
                        double w[5];
                        shape(r, i, w);
                        for (double &x : w) x *= scale;
                        n++;
                        bad += differ(w, K);
                    }
            }
    }
    printf("scale %ld %ld\n", n, bad);
}

// next to a threshold: the windows a + x (b - a) for the x between two windows at which
// the FP64 bits change, found by bisection, and x beside it
static void check_threshold() {
    std::mt19937_64 r(22);
    long n = 0, bad = 0;
    for (float err : ERR) {
        host_err = err;
        for (double CT : {1e-5, 1e-3})
            for (double eps : {1e-40, 2.4e-7}) {
                const Cut64 K = cut64(eps, CT, keep_all_factor(CT));
                for (int i = 0; i < 4000; i++) {
                    double a[5], b[5], w[5];
                    shape(r, i, a);
                    shape(r, i / 5, b);
                    auto at = [&](double x) {
                        for (int t = 0; t < 5; t++) w[t] = a[t] + x * (b[t] - a[t]);
                        return cutoff_bits_f64(w[0], w[1], w[2], w[3], w[4], eps, CT, K.kt);
                    };
                    const unsigned end = at(1.0);
                    if (at(0.0) == end) continue;
                    double lo = 0.0, hi = 1.0;
                    for (int k = 0; k < 60; k++) {
                        const double m = 0.5 * (lo + hi);
                        (at(m) == end ? hi : lo) = m;
                    }
                    for (double d : {0.0, 1e-15, 1e-12, 1e-9, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3, 1e-2, 2e-2})
                        for (double sgn : {1.0, -1.0}) {
                            at(hi * (1.0 + sgn * d));
                            n++;
                            bad += differ(w, K);
                        }
                }
            }
    }
    printf("threshold %ld %ld\n", n, bad);
}

int main() {
    check_scale();
    check_threshold();
    return 0;
}
