// pw_limb.cuh -- 87-bit fixed-point arithmetic for sums of products of
// doubles, in 32-bit integer instructions.
//
// GB300 retires about two FP64 lane operations per clock per SM but 26 (measured)
// multiply-adds of 32-bit integers into 64-bit sums, or 58 such products, and
// 128 integer additions. A stencil point of the PW scheme needs 18 products of
// doubles, added up; held as integers of one unit the sums need no alignment
// and the multiply-add no rounding, so products and sums together cost six
// integer multiply-adds per product, a third of the FP64 unit's time.
//
// A value x = (h 2^58 + m 2^29 + l) 2^lambda: h signed, m and l in [0, 2^29).
// With |x| < 2^E, lambda = E - 86, |h| < 2^28. The split of a double is
// exact for 0 and for every magnitude in the window [2^(E-32), 2^E); any other
// value (subnormals, infinities and NaN included) is refused, and the caller
// evaluates in FP64 wherever such a value takes part. Sums of up to three limb
// values need no carries: their limbs stay below 2^31.
//
// A product keeps the limb products down to h l and m m (six of the nine), in
// three 64-bit sums; m l and l l are dropped. A sum of six products with its
// scaling is then within 2^-24 units of its upper sum g3 (2^-26 in practice)
// of the exact one, and it is rounded to 53 bits once, at the end (to_double).
// So wherever the sum itself, or the sum of its products' magnitudes, reaches
// 2^28 units of g3 (kLimbEnough), the result is closer to the exact one than
// FP64 arithmetic, which rounds at every operation, would come. Products of
// values in the top 12 binades of the window are 2^32 .. 2^57 units; sums whose
// products are all smaller than 2^28 are left to the caller, who evaluates them
// in FP64.
//
// The same code compiles for the host, where a test compares it with exact
// integer arithmetic.
#pragma once

#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define PW_LHD __host__ __device__ __forceinline__
#else
#define PW_LHD inline
#endif

namespace pw {

constexpr int kLimb = 29;
constexpr int kLimbMask = (1 << kLimb) - 1;
// Exponent E of the window of u and v at scale z: 7 + 12 z. A level whose
// largest magnitude lies in [2^(E-12), 2^E) takes scale z, so that it keeps at
// least 20 binades below it; winds of 0.03 .. 128 m/s have z = 0. The scale
// depends on the level's own values only, and every arithmetic step on the
// scale only, never on the launch.
constexpr int kLimbExp = 7, kLimbStep = 12;
constexpr int kLimbWindow = 32;
constexpr int kLimbEnough = 28;

struct Limb3 {
    int h, m, l;
};

struct LimbSum {
    long long g3, g2, g1;  // value = g3 2^116 + g2 2^87 + g1 2^58 (units of l l)
};

PW_LHD uint32_t limb_hi(double x) {
#if defined(__CUDA_ARCH__)
    return static_cast<uint32_t>(__double2hiint(x));
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return static_cast<uint32_t>(b >> 32);
#endif
}

PW_LHD uint32_t limb_lo(double x) {
#if defined(__CUDA_ARCH__)
    return static_cast<uint32_t>(__double2loint(x));
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return static_cast<uint32_t>(b);
#endif
}

PW_LHD double limb_words(uint32_t h, uint32_t l) {
#if defined(__CUDA_ARCH__)
    return __hiloint2double(static_cast<int>(h), static_cast<int>(l));
#else
    const uint64_t b = (static_cast<uint64_t>(h) << 32) | l;
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}

// Low word of (hi:lo) >> (s mod 32), high word of (hi:lo) << (s mod 32).
PW_LHD uint32_t limb_shr(uint32_t lo, uint32_t hi, uint32_t s) {
#if defined(__CUDA_ARCH__)
    return __funnelshift_r(lo, hi, s);
#else
    s &= 31;
    return s ? (lo >> s) | (hi << (32 - s)) : lo;
#endif
}

PW_LHD uint32_t limb_shl(uint32_t lo, uint32_t hi, uint32_t s) {
#if defined(__CUDA_ARCH__)
    return __funnelshift_l(lo, hi, s);
#else
    s &= 31;
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}

PW_LHD long long limb_mul(int a, int b) { return static_cast<long long>(a) * b; }

// s += a b, one multiply-add into a 64-bit sum. (Written as the two halves with
// their carry, which become one instruction. mad.wide.s32 becomes a product and
// a 64-bit addition: more instructions, each at twice the rate; the forward
// kernel ran 580 us with those and 560 us with these at 512x512x64.)
PW_LHD void limb_fma(long long& s, int a, int b) {
#if defined(__CUDA_ARCH__)
    asm("{\n\t.reg .b32 l, h;\n\tmov.b64 {l, h}, %0;\n\t"
        "mad.lo.cc.u32 l, %1, %2, l;\n\tmadc.hi.s32 h, %1, %2, h;\n\tmov.b64 %0, {l, h};\n\t}"
        : "+l"(s)
        : "r"(a), "r"(b));
#else
    s += limb_mul(a, b);
#endif
}

// x as limbs of 2^(E - 86); false if x lies outside the window (*out is then
// not meaningful). kTop = 28: |h| < 2^28. The coefficients use kTop = 31 with
// E two larger (|c| < 4, h < 2^31). *depth: how many binades x lies below the
// window's top (negative above it, large for 0).
template <int kTop = 28>
PW_LHD bool limb_split(double x, int E, Limb3* out, int* depth = nullptr) {
    const uint32_t hi = limb_hi(x), lo = limb_lo(x);
    const uint32_t e = hi & 0x7FF00000u;
    // the implicit bit, absent from zero (and from subnormals, refused below)
    const uint32_t mh = (hi & 0x000FFFFFu) | (e < 0x00100000u ? e : 0x00100000u);
    // significand with its top bit at bit kTop - 1 of the upper word, then the shift that aligns it
    const uint32_t a1 = limb_shl(lo, mh, kTop - 21), a0 = lo << (kTop - 21);
    const int d = static_cast<int>((static_cast<uint32_t>(E - 1 + 1023) << 20) - e) >> 20;
    if (depth) *depth = d;
    const bool ok = static_cast<uint32_t>(d) < static_cast<uint32_t>(kLimbWindow) || (mh | lo) == 0;
    const uint32_t s = static_cast<uint32_t>(static_cast<int>(hi) >> 31);
    const uint64_t sn = (static_cast<uint64_t>(s) << 32) | s;
    const uint64_t n = (((static_cast<uint64_t>(a1) << 32) | a0) ^ sn) - sn;  // with the sign
    const uint32_t n0 = static_cast<uint32_t>(n), n1 = static_cast<uint32_t>(n >> 32);
    const uint32_t sh = static_cast<uint32_t>(d);
    const uint32_t w1 = limb_shr(n0, n1, sh), w0 = limb_shr(0u, n0, sh);
    out->h = static_cast<int>(n1) >> (sh & 31u);
    out->m = static_cast<int>(w1 >> 3);
    out->l = static_cast<int>(limb_shr(w0, w1, 6) & static_cast<uint32_t>(kLimbMask));
    return ok;
}

PW_LHD Limb3 limb_add(Limb3 a, Limb3 b) { return {a.h + b.h, a.m + b.m, a.l + b.l}; }
PW_LHD Limb3 limb_sub(Limb3 a, Limb3 b) { return {a.h - b.h, a.m - b.m, a.l - b.l}; }
PW_LHD Limb3 limb_neg_sum(Limb3 a, Limb3 b) { return {-a.h - b.h, -a.m - b.m, -a.l - b.l}; }

PW_LHD LimbSum limb_zero() { return {0, 0, 0}; }

// s += a b
PW_LHD void limb_mac(LimbSum& s, Limb3 a, Limb3 b) {
    limb_fma(s.g3, a.h, b.h);
    limb_fma(s.g2, a.h, b.m);
    limb_fma(s.g2, a.m, b.h);
    limb_fma(s.g1, a.h, b.l);
    limb_fma(s.g1, a.m, b.m);
    limb_fma(s.g1, a.l, b.h);
}

// Carries: g2 and g1 keep their meaning modulo 2^29 in their low bits.
PW_LHD void limb_carry(LimbSum& s) {
    s.g2 += s.g1 >> kLimb;
    s.g3 += s.g2 >> kLimb;
}

// s += z c, z a sum of products (|g3| < 2^58, carried here) and c a
// coefficient |c| < 4 split with kTop = 31, E = 2.
PW_LHD void limb_mac_scaled(LimbSum& s, LimbSum z, Limb3 c) {
    limb_carry(z);
    const int z3 = static_cast<int>(z.g3 >> kLimb), z2 = static_cast<int>(z.g3) & kLimbMask;
    const int z1 = static_cast<int>(z.g2) & kLimbMask;
    limb_fma(s.g3, z3, c.h);
    limb_fma(s.g2, z3, c.m);
    limb_fma(s.g2, z2, c.h);
    limb_fma(s.g1, z3, c.l);
    limb_fma(s.g1, z2, c.m);
    limb_fma(s.g1, z1, c.h);
}

PW_LHD int limb_clz(uint32_t x) {
#if defined(__CUDA_ARCH__)
    return __clz(static_cast<int>(x));
#else
    return x ? __builtin_clz(x) : 32;
#endif
}

// The carried sum as a double, rounded once to nearest (a tie away from zero):
// its value is (g3 2^116 + ...) 2^scale (scale: lambda + lambda). Integer
// operations only: the FP64 unit, slow as it is, would make every warp of a CTA
// queue for it at the same point. Of the sum's low bits 2^-29 units of g3
// remain, also where large products cancel to a sum below one unit. *large: the
// sum reaches 2^kLimbEnough units of g3; one that does not may have lost bits.
// 0 gives 0.
PW_LHD double limb_to_double(const LimbSum& s, int scale, bool* large) {
    const uint32_t t1 = static_cast<uint32_t>(s.g3 >> 32);
    const uint32_t sg = static_cast<uint32_t>(static_cast<int>(t1) >> 31);
    // the magnitude's words (one unit of the last one less, if negative)
    const uint32_t w2 = t1 ^ sg, w1 = static_cast<uint32_t>(s.g3) ^ sg, w0 = (static_cast<uint32_t>(s.g2) << 3) ^ sg;
    const bool up = w2 == 0;
    uint32_t a = up ? w1 : w2, b = up ? w0 : w1, c = up ? 0u : w0, base = static_cast<uint32_t>(scale + 116 + 63 + 1022);
    if (a == 0) {  // below one unit of g3: only w0 is left
        a = b;
        b = 0u;
        base -= 32u;
    }
    const uint32_t n = static_cast<uint32_t>(limb_clz(a));
    *large = !up || w1 >= 1u << kLimbEnough;
    const uint32_t m1 = limb_shl(b, a, n), m0 = limb_shl(c, b, n);  // top bit set
    // weight of the top bit: 2^(scale + 116 + 63 - n), 32 less if up; the bit itself adds one to the exponent field
    const uint32_t e = base - (up ? 32u : 0u) - n;
    const uint64_t v = (static_cast<uint64_t>(m1 >> 11) << 32 | limb_shr(m0, m1, 11)) + ((m0 >> 10) & 1u);
    const uint32_t h = static_cast<uint32_t>(v >> 32) + (e << 20);
    return limb_words(a == 0 ? 0u : h | (sg & 0x80000000u), a == 0 ? 0u : static_cast<uint32_t>(v));
}

// A lower bound of |a b| in units of g3 from the upper limbs of a and b, sums of
// up to three values: an upper limb is below its value by up to one per value.
PW_LHD long long limb_least(int a, int b) {
    const int x = (a < 0 ? -a : a) - 3, y = (b < 0 ? -b : b) - 3;
    return x > 0 && y > 0 ? limb_mul(x, y) : 0;
}

// Binades that |r| lies below 1 (|r| <= 1), rounded up; 63 for 0: products with
// the coefficient r count at least 2^-that of their magnitude.
PW_LHD int limb_binades(double r) {
    const int e = static_cast<int>(limb_hi(r) >> 20 & 0x7FFu);
    return e <= 1023 - 63 ? 63 : e >= 1023 ? 0 : 1023 - e;
}

// Whether horizontal products of magnitudes x and y (limb_least, before their
// coefficients, which lie sx and sy binades below 1) reach 2^kLimbEnough units.
PW_LHD bool limb_settled(long long x, long long y, int sx, int sy) {
    return (x >> sx) + (y >> sy) >= (1ll << kLimbEnough);
}

}  // namespace pw
