// The sums of csrc/pw_limb.cuh on the host, for tests that know the exact value.
#include "pw_limb.cuh"

static double value_of(pw::LimbSum s, int scale, bool* large) {
    pw::limb_carry(s);
    uint32_t mag;
    const double x = pw::limb_to_double(s, scale, &mag);
    *large = !pw::limb_small(mag, scale);
    return mag == 0 ? pw::limb_tiny(s, scale) : x;
}

// su's horizontal products of n points, p = {uw, uc, ue, us, un, vs, vse, vc, ve}
// in a window of exponent E: the sum of q(i-1) Fx(i-1/2) - q(i+1) Fx(i+1/2) and
// the same in y as a double, and whether it reaches kLimbEnough.
extern "C" void limb_su_sums(int n, int E, const double* p, double* out, unsigned char* in, unsigned char* enough) {
    for (int q = 0; q < n; ++q, p += 9) {
        pw::Limb3 l[9];
        in[q] = 1;
        for (int k = 0; k < 9; ++k) in[q] &= pw::limb_split(p[k], E, &l[k]) ? 1 : 0;
        pw::LimbSum s = pw::limb_zero();
        pw::limb_mac(s, pw::limb_sub(l[0], l[2]), pw::limb_add(pw::limb_add(l[0], l[1]), l[2]));
        pw::limb_mac(s, l[3], pw::limb_add(l[5], l[6]));
        pw::limb_mac(s, l[4], pw::limb_neg_sum(l[7], l[8]));
        bool large;
        out[q] = value_of(s, 2 * (E - 86), &large);
        const long long m = pw::limb_least(l[0].h - l[2].h, l[0].h + l[1].h + l[2].h) +
                            pw::limb_least(l[3].h, l[5].h + l[6].h) + pw::limb_least(l[4].h, l[7].h + l[8].h);
        enough[q] = large || m >= (1ll << pw::kLimbEnough);
    }
}

// The same with coefficients of the x and y sums (|rx|, |ry| <= 1) as where tcx
// and tcy differ: rx X + ry Y, and whether the sum or the magnitudes of its
// products settle it.
extern "C" void limb_su_joined(int n, int E, double rx, double ry, const double* p, double* out, unsigned char* in,
                               unsigned char* enough) {
    pw::Limb3 cx, cy;
    (void)pw::limb_split<31>(rx, 2, &cx);
    (void)pw::limb_split<31>(ry, 2, &cy);
    for (int q = 0; q < n; ++q, p += 9) {
        pw::Limb3 l[9];
        in[q] = 1;
        for (int k = 0; k < 9; ++k) in[q] &= pw::limb_split(p[k], E, &l[k]) ? 1 : 0;
        pw::LimbSum x = pw::limb_zero(), y = pw::limb_zero(), s = pw::limb_zero();
        pw::limb_mac(x, pw::limb_sub(l[0], l[2]), pw::limb_add(pw::limb_add(l[0], l[1]), l[2]));
        pw::limb_mac(y, l[3], pw::limb_add(l[5], l[6]));
        pw::limb_mac(y, l[4], pw::limb_neg_sum(l[7], l[8]));
        pw::limb_mac_scaled(s, x, cx);
        pw::limb_mac_scaled(s, y, cy);
        bool large;
        out[q] = value_of(s, 2 * (E - 86), &large);
        const long long mx = pw::limb_least(l[0].h - l[2].h, l[0].h + l[1].h + l[2].h);
        const long long my = pw::limb_least(l[3].h, l[5].h + l[6].h) + pw::limb_least(l[4].h, l[7].h + l[8].h);
        enough[q] = large || pw::limb_settled(mx, my, pw::limb_binades(rx), pw::limb_binades(ry));
    }
}

// Limbs of n values in the window of exponent E, cut to its unit where they lie
// below it, and those of the window up binades larger; {h, m, l, cut} each.
extern "C" void limb_cut_and_shift(int n, int E, int up, const double* x, int* at_E, int* shifted) {
    for (int q = 0; q < n; ++q, at_E += 4, shifted += 4) {
        pw::Limb3 v;
        at_E[3] = pw::limb_split_cut(x[q], E, &v) ? 1 : 0;
        at_E[0] = v.h, at_E[1] = v.m, at_E[2] = v.l;
        bool cut;
        v = pw::limb_shift(v, up, &cut);
        shifted[0] = v.h, shifted[1] = v.m, shifted[2] = v.l, shifted[3] = cut ? 1 : 0;
    }
}

// The coefficient form: 2^-87 is the unit.
extern "C" void limb_cut_coef(int n, const double* x, int* out) {
    for (int q = 0; q < n; ++q, out += 4) {
        pw::Limb3 v;
        out[3] = pw::limb_split_cut<31>(x[q], 2, &v) ? 1 : 0;
        out[0] = v.h, out[1] = v.m, out[2] = v.l;
    }
}

// The cut form for values 32 binades and more below the window's top.
extern "C" void limb_cut_low(int n, int E, const double* x, int* out) {
    for (int q = 0; q < n; ++q, out += 4) {
        pw::Limb3 v;
        out[3] = pw::limb_split_low(x[q], E, &v) ? 1 : 0;
        out[0] = v.h, out[1] = v.m, out[2] = v.l;
    }
}
