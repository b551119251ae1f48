// Host check of teno7_f64math.cuh: the FP32-decided cutoff bits against the
// FP64 evaluation.  Prints "<what> <cases> <differences>" per line.
#include <cstdio>
#include <random>

// the device's approximate reciprocal and root are off by up to 2^-22: check at
// both ends of that
static float host_err = 1.f;
#define T7_HOST_ERR *host_err
#include "teno7_f64math.cuh"

using namespace t7;

static void check_cutoff() {
    std::mt19937_64 r(3);
    std::uniform_real_distribution<double> u(-1, 1);
    long bad = 0, total = 0;
    for (double CT : {1e-5, 1e-7, 1e-3, 0.2, 0.5, 1e-300})
        for (double eps : {1e-60, 1e-40, 1e-18, 1e-12, 2.4e-7, 1e-3}) {
            const double kt = keep_all_factor(CT);
            const Cut64 K = cut64(eps, CT, kt);
            for (int i = 0; i < 40000; i++) {
                const double base = u(r) * pow(10, u(r) * 3), amp = pow(10, u(r) * 8 - 8 + (i % 3) * 4);
                const double d0 = u(r), d1 = u(r), d2 = u(r);
                double w[5];
                for (int t = 0; t < 5; t++) {
                    const double x = t - 2;
                    switch (i % 7) {
                        case 0: w[t] = base + amp * u(r); break;                                         // noise
                        case 1: w[t] = base + amp * (d0 * x + 0.1 * d1 * x * x + 0.01 * d2 * x * x * x); break;  // smooth
                        case 2: w[t] = base + (t > 2 ? amp * d0 : 0) + 1e-3 * amp * u(r); break;         // jumps
                        case 3: w[t] = base + (t > 1 ? amp * d0 : 0) + 1e-9 * amp * u(r); break;
                        case 4: w[t] = base; break;                                                      // constant
                        case 5: w[t] = base + amp * u(r) * (t == 2); break;                              // a spike
                        default: w[t] = amp * (t > 2 ? d0 * x * x : d1 * x) * (i % 2 ? 1 : 1e-20); break;  // a kink
                    }
                }
                total++;
                bad += cutoff_bits(w[0], w[1], w[2], w[3], w[4], K) !=
                       cutoff_bits_f64(w[0], w[1], w[2], w[3], w[4], eps, CT, kt);
            }
        }
    printf("cutoff %ld %ld\n", total, bad);
    // zeros, subnormals, magnitudes beyond FP32, infinities and NaN in every place
    const double s[] = {0.0, -0.0, 1e-310, 1e-40, 1e-20, 1.0, 1e20, 1e60, 1e300, INFINITY, NAN};
    const Cut64 K = cut64(2.4e-7, 1e-5, keep_all_factor(1e-5));
    total = bad = 0;
    for (double a : s)
        for (double b : s)
            for (double c : s)
                for (double d : s)
                    for (double e : s) {
                        total++;
                        bad += cutoff_bits(a, b, c, d, e, K) != cutoff_bits_f64(a, b, c, d, e, K.eps, K.CT, K.kt);
                    }
    printf("cutoff_special %ld %ld\n", total, bad);
}

static bool same(double x, double y) { return f64_bits(x) == f64_bits(y) || (x != x && y != y); }

// quotients and roots: random mantissas (short and long) and exponents, results
// around powers of two, operands next to exact results, and special values
static void check_div_sqrt() {
    std::mt19937_64 r(11);
    long nd = 0, bd = 0, ns = 0, bs = 0;
    auto mantissa = [&](int kind) {
        uint64_t m = r() & 0xfffffffffffffull;
        if (kind == 1) m &= ~0ull << (r() % 52);
        if (kind == 2) m = 0xfffffffffffffull - (m >> (20 + r() % 32));
        if (kind == 3) m >>= 20 + r() % 32;
        return m;
    };
    for (float err : {1.f, 1.f + 2.4e-7f, 1.f - 2.4e-7f}) {
        host_err = err;
        for (int i = 0; i < 3000000; i++) {
            const int spread = i % 16 == 0 ? 1000 : 40;
            auto draw = [&](int kind) {
                const uint64_t e = 1023 - spread + r() % (2 * spread + 1);
                return f64_of(((r() & 1) << 63) | (e << 52) | mantissa(kind));
            };
            double a = draw(i % 4), b = draw((i / 4) % 4);
            if (i % 5 == 1) a = b * f64_of(f64_bits(a));                      // a quotient near a double
            if (i % 5 == 2) a = f64_of(f64_bits(b * a) + r() % 3 - 1);        // and one beside it
            if (i % 5 == 3) a = f64_of(f64_bits(b) + r() % 5 - 2);            // near one
            nd++;
            bd += !same(div64(a, b), a / b);
            double x = fabs(a);
            if (i % 3 == 1) x = b * b;
            if (i % 3 == 2) x = f64_of(f64_bits(b * b) + r() % 5 - 2);
            ns++;
            bs += !same(sqrt64(x), sqrt(x));
        }
        const double s[] = {0.0, -0.0, 5e-324, 1e-310, 2.2250738585072014e-308, 1e-300, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0,
                            1e300, 1.7976931348623157e308, INFINITY, NAN, -1.0, -1e-310, -INFINITY};
        for (double a : s) {
            ns++;
            bs += !same(sqrt64(a), sqrt(a));
            for (double b : s) {
                nd++;
                bd += !same(div64(a, b), a / b);
            }
        }
    }
    printf("div %ld %ld\nsqrt %ld %ld\n", nd, bd, ns, bs);
}

// products, over the range mul64 takes: random, short mantissas (exact products
// and ties), and mantissas of ones
static void check_mul() {
    std::mt19937_64 r(5);
    long n = 0, bad = 0;
    for (int i = 0; i < 4000000; i++) {
        auto draw = [&](int kind) {
            uint64_t m = r() & 0xfffffffffffffull;
            if (kind == 1) m &= ~0ull << (20 + r() % 32);
            if (kind == 2) m = 0xfffffffffffffull - (m >> (20 + r() % 32));
            if (kind == 3) m &= ~0ull << (24 + r() % 4);
            return f64_of(((r() & 1) << 63) | ((623 + r() % 800) << 52) | m);
        };
        const double x = i % 1000 == 0 ? 0.0 : draw(i % 4), g = draw((i / 4) % 4);
        if (mul_unranged(g) || (x != 0.0 && mul_unranged(x))) bad++;
        n++;
        const double p = mul64(mul_op(x), g);
        bad += p != x * g;
    }
    for (double v : {0.0, 1e-130, 1e130, (double)INFINITY, (double)NAN, 5e-324}) bad += mul_unranged(v) != 1;
    printf("mul %ld %ld\n", n, bad);
}

int main() {
    check_cutoff();
    check_mul();
    check_div_sqrt();
    return 0;
}
