// Host check of csrc/pw_limb.cuh against exact integer arithmetic: splits of
// doubles over the whole window (and the refusals around it), sums of products
// with a scaled part as a stencil point forms them, their rounding to double.
// Prints "cases N bad M worst W" with W the largest error in units of 2^-53 of
// the sum of the magnitudes of the products.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <initializer_list>

#include "pw_limb.cuh"

typedef __int128 i128;

static uint64_t x64 = 88172645463325252ull;
static uint64_t rnd() {
    x64 ^= x64 << 13;
    x64 ^= x64 >> 7;
    x64 ^= x64 << 17;
    return x64;
}

// A nonzero double with exponent in [lo, hi) and a random or sparse significand.
static double value(int lo, int hi) {
    const int e = lo + (int)(rnd() % (uint64_t)(hi - lo));
    uint64_t f = rnd() & 0xFFFFFFFFFFFFFull;
    switch (rnd() % 6) {
        case 0: f = 0; break;
        case 1: f = 0xFFFFFFFFFFFFFull; break;
        case 2: f &= ~((1ull << (rnd() % 52)) - 1); break;
        default: break;
    }
    const uint64_t b = ((rnd() & 1) << 63) | ((uint64_t)(e + 1023) << 52) | f;
    double d;
    memcpy(&d, &b, 8);
    return d;
}

// An exact signed fixed-point number of 16 x 32 bits (two's complement), unit 2^-256.
struct Big {
    uint32_t w[16];
    Big() { memset(w, 0, sizeof w); }
    void add_shifted(i128 v, int bit) {  // += v 2^bit, 0 <= bit
        uint64_t carry = 0;
        for (int i = 0; i < 16; ++i) {
            const int lo = 32 * i - bit;  // bits lo .. lo + 31 of v (sign extended)
            uint32_t part;
            if (lo <= -32) part = 0;
            else if (lo < 0) part = (uint32_t)((unsigned __int128)v << (-lo));
            else if (lo >= 127) part = v < 0 ? 0xFFFFFFFFu : 0u;
            else part = (uint32_t)(v >> lo);
            const uint64_t t = (uint64_t)w[i] + part + carry;
            w[i] = (uint32_t)t;
            carry = t >> 32;
        }
    }
    void sub(const Big& o) {
        uint64_t borrow = 0;
        for (int i = 0; i < 16; ++i) {
            const uint64_t t = (uint64_t)w[i] - o.w[i] - borrow;
            w[i] = (uint32_t)t;
            borrow = (t >> 32) & 1;
        }
    }
    double to_double() const {  // approximate magnitude (about 1e-15 relative)
        Big a = *this;
        const bool neg = w[15] >> 31;
        if (neg) {
            Big z;
            z.sub(*this);
            a = z;
        }
        double r = 0;
        for (int i = 15; i >= 0; --i) r = r * 4294967296.0 + a.w[i];
        return (neg ? -r : r) * std::pow(2.0, -256);
    }
};

// += sign * a * b exactly (unit 2^-256)
static void add_product(Big& s, double a, double b, int sign) {
    int ea, eb;
    const i128 ma = (i128)(int64_t)std::ldexp(std::frexp(a, &ea), 53), mb = (i128)(int64_t)std::ldexp(std::frexp(b, &eb), 53);
    if (ma == 0 || mb == 0) return;
    s.add_shifted(sign * ma * mb, ea + eb - 106 + 256);
}

// += sign * a * b * c * 2^e exactly
static void add_triple(Big& s, double a, double b, double c, int sign, int e) {
    int ea, eb, ec;
    const int64_t ma = (int64_t)std::ldexp(std::frexp(a, &ea), 53), mb = (int64_t)std::ldexp(std::frexp(b, &eb), 53);
    const int64_t mc = (int64_t)std::ldexp(std::frexp(c, &ec), 53);
    const int bit = ea + eb + ec - 159 + e + 256;
    const int64_t h = 1ll << 27, b1 = mb / h, b0 = mb % h, c1 = mc / h, c0 = mc % h;
    s.add_shifted(sign * (i128)ma * b1 * c1, bit + 54);
    s.add_shifted(sign * (i128)ma * b1 * c0, bit + 27);
    s.add_shifted(sign * (i128)ma * b0 * c1, bit + 27);
    s.add_shifted(sign * (i128)ma * b0 * c0, bit);
}

static void add_double(Big& s, double a, int sign) {
    int ea;
    const i128 ma = (i128)(int64_t)std::ldexp(std::frexp(a, &ea), 53);
    const int bit = ea - 53 + 256;
    if (ma == 0) return;
    if (bit >= 0) s.add_shifted(sign * ma, bit);
    else s.add_shifted((sign * ma) >> -bit, 0);
}

int main() {
    long long cases = 0, bad = 0, small = 0;
    double worst = 0;
    const int E = pw::kLimbExp, EW = E - 3;
    // splits
    for (int n = 0; n < 400000; ++n) {
        const double x = n % 50 == 0 ? (n % 100 ? 0.0 : -0.0) : value(E - 36, E + 4);
        pw::Limb3 a;
        const bool ok = pw::limb_split(x, E, &a);
        const bool in = x == 0.0 || (std::fabs(x) < std::ldexp(1.0, E) && std::fabs(x) >= std::ldexp(1.0, E - 32));
        ++cases;
        if (ok != in) ++bad;
        if (!ok) continue;
        if (a.m < 0 || a.m > pw::kLimbMask || a.l < 0 || a.l > pw::kLimbMask) ++bad;
        const i128 v = ((i128)a.h << 58) + ((i128)a.m << 29) + a.l;
        int ea;
        const int64_t mx = (int64_t)std::ldexp(std::frexp(x, &ea), 53);
        const int up = ea - 53 - (E - 86);
        if (x != 0.0 && (up < 0 || v != ((i128)mx << up))) ++bad;
        if (x == 0.0 && v != 0) ++bad;
    }
    for (double x : {5e-324, 1e-310, -1e-310, (double)INFINITY, -(double)INFINITY, (double)NAN, 1e300, 2.0e-308}) {
        pw::Limb3 a;
        ++cases;
        if (pw::limb_split(x, E, &a)) ++bad;
    }
    for (int n = 0; n < 100000; ++n) {  // coefficients
        const double x = value(-30, 2);
        pw::Limb3 a;
        ++cases;
        if (!pw::limb_split<31>(x, 2, &a)) {
            ++bad;
            continue;
        }
        const i128 v = ((i128)a.h << 58) + ((i128)a.m << 29) + a.l;
        int ea;
        const int64_t mx = (int64_t)std::ldexp(std::frexp(x, &ea), 53);
        const int up = ea - 53 + 87;
        if (up >= 0 ? v != ((i128)mx << up) : v != ((i128)mx >> -up)) ++bad;
    }
    // points: x factorised, two y terms, one scaled pair, as the su sum is formed
    const int ranges[6][2] = {{2, 4}, {-2, E}, {E - 32, E - 12}, {E - 32, E}, {E - 1, E}, {-10, 3}};
    for (int n = 0; n < 600000; ++n) {
        const int* r = ranges[n % 6];
        double u[6], v[4], w[4];
        for (double& t : u) t = value(r[0], r[1]);
        for (double& t : v) t = value(r[0], r[1]);
        if (n % 7 == 0) u[1] = u[0] + (rnd() % 3 ? 0.0 : std::ldexp(u[0], -40)), v[2] = -v[0];  // near cancellation
        if (n % 11 == 0) u[3] = 0.0, v[1] = 0.0;
        pw::Limb3 U[6], V[4], W[4], C;
        bool in = true;
        for (int i = 0; i < 6; ++i) in &= pw::limb_split(u[i], E, &U[i]);
        for (int i = 0; i < 4; ++i) in &= pw::limb_split(v[i], E, &V[i]);
        for (int i = 0; i < 4; ++i) {
            w[i] = value(r[0] - 3, r[1] - 3);
            in &= pw::limb_split(w[i], EW, &W[i]);
        }
        const double c = std::ldexp(value(-8, 2), 0);
        in &= pw::limb_split<31>(c, 2, &C);
        if (!in) continue;
        ++cases;
        pw::LimbSum s = pw::limb_zero(), z = pw::limb_zero();
        pw::limb_mac(s, pw::limb_sub(U[0], U[1]), pw::limb_add(pw::limb_add(U[0], U[2]), U[1]));
        pw::limb_mac(s, U[3], pw::limb_add(V[0], V[1]));
        pw::limb_mac(s, U[4], pw::limb_neg_sum(V[2], V[3]));
        pw::limb_mac(z, U[2], pw::limb_add(W[0], W[1]));
        pw::limb_mac(z, U[5], pw::limb_neg_sum(W[2], W[3]));
        pw::limb_mac_scaled(s, z, C);
        const int scale = 2 * (E - 86);
        pw::limb_carry(s);
        bool large;
        const double got = pw::limb_to_double(s, scale, &large);
        // the least the magnitudes of the horizontal products can be, in units of g3
        auto mag = [](pw::Limb3 p, pw::Limb3 q) { return pw::limb_least(p.h, q.h); };
        const long long A = mag(pw::limb_sub(U[0], U[1]), pw::limb_add(pw::limb_add(U[0], U[2]), U[1])) +
                            mag(U[3], pw::limb_add(V[0], V[1])) + mag(U[4], pw::limb_neg_sum(V[2], V[3]));
        if (!large && A < (1ll << pw::kLimbEnough)) {
            ++small;
            continue;
        }
        // exact: the scaled pair's product with c in extended steps: c (u w) 2^(EH - EW)
        Big ex, zz;
        double M = 0;
        auto term = [&](double a, double b, int sg) {
            add_product(ex, a, b, sg);
            M += std::fabs(a) * std::fabs(b);
        };
        term(u[0], u[0], 1), term(u[0], u[2], 1), term(u[1], u[2], -1), term(u[1], u[1], -1);
        term(u[3], v[0], 1), term(u[3], v[1], 1), term(u[4], v[2], -1), term(u[4], v[3], -1);
        auto scaled = [&](double p, double q, int sg) {  // the limbs of w count 2^(EW - EH) of u's
            add_triple(ex, p, q, c, sg, E - EW);
            M += std::fabs(p * c * std::ldexp(1.0, E - EW)) * std::fabs(q);
        };
        scaled(u[2], w[0], 1), scaled(u[2], w[1], 1), scaled(u[5], w[2], -1), scaled(u[5], w[3], -1);
        const double exact = ex.to_double();
        add_double(ex, got, -1);
        const double err = std::fabs(ex.to_double());
        const double lim = 0.5 * std::ldexp(std::fabs(exact), -52) * 1.01;  // half a unit in the last place
        const double rel = err / (M * std::ldexp(1.0, -53));
        if (rel > worst) worst = rel;
        // one rounding of the result, plus the dropped limbs: 2^-24 of 2^28 units, two units of 2^-53 of M at most
        if (err > lim + 2.0 * M * std::ldexp(1.0, -53)) {
            if (bad < 5) std::printf("n %d range %d err/ulp %g rel %g got %.17g exact %.17g\n", n, n % 6, err / lim, rel, got, exact);
            ++bad;
        }
    }
    std::printf("cases %lld bad %lld small %lld worst %.3f\n", cases, bad, small, worst);
    return bad != 0;
}
