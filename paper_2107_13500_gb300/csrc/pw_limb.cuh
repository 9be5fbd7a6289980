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
// exact for 0 and for every magnitude in the window [2^(E-32), 2^E); smaller
// values are cut to the window's unit (limb_split_cut). Sums of up to three limb
// values need no carries: their limbs stay below 2^31.
//
// A product keeps the limb products down to h l and m m (six of the nine), in
// three 64-bit sums; m l and l l are dropped. A sum of six products with its
// scaling is then within 2^-24 units of its upper sum g3 (2^-26 in practice)
// of the exact one, cut values included, and it is rounded to 53 bits once, at
// the end (to_double).
// So wherever the sum itself, or the sum of its products' magnitudes, reaches
// 2^28 units of g3 (kLimbEnough), the result is closer to the exact one than
// FP64 arithmetic, which rounds at every operation, would come. Products of
// values in the top binade of the window are 2^54 .. 2^57 units; sums whose
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
// A window's exponent E is that of the largest magnitude it has to hold, so
// fields times a power of two give the same bits, scaled. kLimbExp: where there
// is none.
constexpr int kLimbExp = 7;
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
    const uint32_t hi = limb_hi(x), lo = limb_lo(x), mag = hi & 0x7FFFFFFFu;
    // the implicit bit, absent from zero (and from subnormals, refused below)
    const uint32_t one = mag < 0x00100000u ? mag : 0x00100000u;
    const uint32_t mh = (hi & 0x000FFFFFu) | (one & 0xFFF00000u);
    // significand with its top bit at bit kTop - 1 of the upper word, then the shift that aligns it
    const uint32_t a1 = limb_shl(lo, mh, kTop - 21), a0 = lo << (kTop - 21);
    const int d = static_cast<int>((static_cast<uint32_t>(E - 1 + 1023) << 20 | 0xFFFFFu) - mag) >> 20;
    if (depth) *depth = d;
    const bool ok = static_cast<uint32_t>(d) < static_cast<uint32_t>(kLimbWindow) || (mag | lo) == 0;
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

// Magnitude words x2 2^64 + x1 2^32 + x0, whose bit 6 is the limbs' unit, shifted
// down by s (0 .. 95; up by -s where s < 0, -95 at most) and cut there, as signed
// limbs. *cut: something was lost.
PW_LHD Limb3 limb_place(uint32_t x2, uint32_t x1, uint32_t x0, int s, bool negative, bool* cut) {
    uint32_t lost = 0;
    if (s < 0) {
        const uint32_t t = static_cast<uint32_t>(-s);
        if (t >= 64) x2 = x0, x1 = x0 = 0;
        else if (t >= 32) x2 = x1, x1 = x0, x0 = 0;
        x2 = limb_shl(x1, x2, t), x1 = limb_shl(x0, x1, t), x0 <<= t & 31u;
    } else {
        const uint32_t t = static_cast<uint32_t>(s);
        if (t >= 64) lost = x1 | x0, x0 = x2, x1 = x2 = 0;
        else if (t >= 32) lost = x0, x0 = x1, x1 = x2, x2 = 0;
        lost |= limb_shr(0u, x0, t);  // the bits below x0
        x0 = limb_shr(x0, x1, t), x1 = limb_shr(x1, x2, t), x2 >>= t & 31u;
    }
    *cut = (lost | (x0 & 63u)) != 0;
    uint64_t low = (static_cast<uint64_t>(x1) << 32 | x0) >> 6;  // m and l
    int h = static_cast<int>(x2);
    if (negative) {
        h = low != 0 ? ~h : -h;
        low = (0 - low) & ((1ull << 58) - 1);
    }
    return {h, static_cast<int>(low >> kLimb), static_cast<int>(low) & kLimbMask};
}

// The split for a value below the window (its top bit 32 binades or more under
// 2^E), cut towards zero to the unit, 2^(E - 86): off by less than that, which
// moves a product by less than 2^-28 units of g3. Returns whether anything was cut.
PW_LHD bool limb_split_low(double x, int E, Limb3* out) {
    const uint32_t hi = limb_hi(x), lo = limb_lo(x), e = hi >> 20 & 0x7FFu;
    const uint32_t mh = (hi & 0x000FFFFFu) | (e ? 0x00100000u : 0u);
    const uint32_t a1 = limb_shl(lo, mh, 7), a0 = lo << 7;  // as in limb_split
    const int d = E - 1 + 1023 - static_cast<int>(e ? e : 1u);
    const uint32_t s = static_cast<uint32_t>(d > 95 ? 95 : d), x1 = s < 64 ? a1 : 0u, x0 = s < 64 ? a0 : a1;
    const uint32_t y0 = limb_shr(x0, x1, s), y1 = x1 >> (s & 31u);
    const uint32_t lost = (s < 64 ? 0u : a0) | limb_shr(0u, x0, s) | (y0 & 63u);
    uint64_t low = (static_cast<uint64_t>(y1) << 32 | y0) >> 6;
    const bool minus = static_cast<int>(hi) < 0 && low != 0;
    if (minus) low = (1ull << 58) - low;
    *out = {minus ? -1 : 0, static_cast<int>(low >> kLimb), static_cast<int>(low) & kLimbMask};
    return lost != 0;
}

// The split for any |x| < 2^E, cut like that where it lies below the window; the
// unit is 2^-87 for kTop = 31, E = 2.
template <int kTop = 28>
PW_LHD bool limb_split_cut(double x, int E, Limb3* out) {
    const uint32_t hi = limb_hi(x), lo = limb_lo(x), e = hi >> 20 & 0x7FFu;
    const uint32_t mh = (hi & 0x000FFFFFu) | (e ? 0x00100000u : 0u);
    const int d = E - 1 + 1023 - static_cast<int>(e ? e : 1u);
    bool cut;
    *out = limb_place(limb_shl(lo, mh, kTop - 21), lo << (kTop - 21), 0u, d < 0 ? 0 : d > 95 ? 95 : d, hi >> 31 != 0, &cut);
    return cut;
}

// The limbs of a value in a window whose exponent is up larger (95 either way at
// most), as limb_split_cut would have them.
PW_LHD Limb3 limb_shift(Limb3 a, int up, bool* cut) {
    uint64_t low = static_cast<uint64_t>(a.m) << kLimb | static_cast<uint32_t>(a.l);
    if (up > -32 && up < 32) {  // where nothing is cut, the words shift with their sign
        const uint32_t x2 = static_cast<uint32_t>(a.h), x1 = static_cast<uint32_t>(low >> 26), x0 = static_cast<uint32_t>(low << 6);
        const uint32_t s = static_cast<uint32_t>(up < 0 ? -up : up);
        const uint32_t y0 = up < 0 ? x0 << s : limb_shr(x0, x1, s), y1 = up < 0 ? limb_shl(x0, x1, s) : limb_shr(x1, x2, s);
        const int h = up < 0 ? static_cast<int>(limb_shl(x1, x2, s)) : a.h >> s;
        *cut = false;
        if (up < 0 || (limb_shr(0u, x0, s) | (y0 & 63u)) == 0)
            return {h, static_cast<int>(y1 >> 3), static_cast<int>(limb_shr(y0, y1, 6) & static_cast<uint32_t>(kLimbMask))};
    }
    int h = a.h;
    if (h < 0) {
        h = low != 0 ? ~h : -h;
        low = (0 - low) & ((1ull << 58) - 1);
    }
    low <<= 6;
    return limb_place(static_cast<uint32_t>(h), static_cast<uint32_t>(low >> 32), static_cast<uint32_t>(low), up, a.h < 0, cut);
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
// queue for it at the same point. *mag: the upper word of the result's magnitude
// (limb_small). A sum below one unit of g3 gives 0: products that cancel that far
// are for limb_tiny.
PW_LHD double limb_to_double(const LimbSum& s, int scale, uint32_t* mag) {
    const uint32_t t1 = static_cast<uint32_t>(s.g3 >> 32);
    const uint32_t sg = static_cast<uint32_t>(static_cast<int>(t1) >> 31);
    // the magnitude's words (one unit of the last one less, if negative)
    const uint32_t w2 = t1 ^ sg, w1 = static_cast<uint32_t>(s.g3) ^ sg, w0 = (static_cast<uint32_t>(s.g2) << 3) ^ sg;
    const bool up = w2 == 0;
    const uint32_t a = up ? w1 : w2, b = up ? w0 : w1, c = up ? 0u : w0;
    const uint32_t n = static_cast<uint32_t>(limb_clz(a));
    const uint32_t m1 = limb_shl(b, a, n), m0 = limb_shl(c, b, n);  // top bit set
    // weight of the top bit: 2^(scale + 116 + 63 - n), 32 less if up; the bit itself adds one to the exponent field
    const uint32_t e = static_cast<uint32_t>(scale + 116 + 63 + 1022) - (up ? 32u : 0u) - n;
    const uint64_t v = (static_cast<uint64_t>(m1 >> 11) << 32 | limb_shr(m0, m1, 11)) + ((m0 >> 10) & 1u);
    const uint32_t h = a == 0 ? 0u : static_cast<uint32_t>(v >> 32) + (e << 20);
    *mag = h;
    return limb_words(h | (sg & 0x80000000u), a == 0 ? 0u : static_cast<uint32_t>(v));
}

// Whether a result of that upper word is less than 2^kLimbEnough units of g3: one
// that may have lost bits.
PW_LHD bool limb_small(uint32_t mag, int scale) {
    return mag < static_cast<uint32_t>(scale + 116 + kLimbEnough + 1023) << 20;
}

PW_LHD double limb_to_double(const LimbSum& s, int scale, bool* large) {
    uint32_t mag;
    const double x = limb_to_double(s, scale, &mag);
    *large = !limb_small(mag, scale);
    return x;
}

// A carried sum that limb_to_double gave as 0, from what is left of it: 2^-29
// units of g3.
PW_LHD double limb_tiny(const LimbSum& s, int scale) {
    const int t = static_cast<int>(static_cast<uint32_t>(s.g3) << kLimb | (static_cast<uint32_t>(s.g2) & kLimbMask));
    return static_cast<double>(t) * limb_words(static_cast<uint32_t>(scale + 116 - kLimb + 1023) << 20, 0u);
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
