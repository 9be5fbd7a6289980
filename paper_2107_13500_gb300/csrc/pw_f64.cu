// pw_f64.cu -- PW advection of FP64 fields to FP64 accuracy (PW_F64): the
// one-shot forward kernel and its persistent form over a batch plan.
//
// Every source term is a sum of six face terms c * q * (a + b) (Listing 1 and
// its two companions). GB300 retires about two FP64 lane operations per clock
// per SM, which capped this path at 19 GPt/s with 32.6 operations per point,
// the least its formulation allows (16.1 measured, 12 % of the HBM rate). So
// the sums of products run on the integer pipes instead (pw_limb.cuh): each
// level is split once, cooperatively, into 87-bit fixed-point values of three
// limbs, exact for every magnitude in a window of 32 binades; a product is six
// 32 x 32 multiply-adds into 64-bit sums, a face sum three additions, and each
// output is rounded to double once, by integer operations too. What stays on
// the FP64 pipe is one product per output.
//
// Factored per output, with T = tcx (or the larger of tcx and tcy):
//   s = T [ X + Y + rho(k) Z ],  rho = tz / T,
// X and Y the horizontal products (their own coefficients first where tcx and
// tcy differ), Z the vertical ones; rho as a limb number. Where tzc1(k) =
// tzc2(k) and tzd1(k) = tzd2(k) on every level (no density stratification,
// checked per domain on the device, bit for bit) the level's two vertical
// products share one scaling by rho.
//
// A level takes the scale of its window from its largest value in the tile
// (pw_limb.cuh), and the three levels of a step must share it. A level whose
// tile (halo included) holds a value outside the window (other than 0), an
// infinity or a NaN makes the steps that read it FP64 steps: the same six
// terms, term by term, in native FP64 from global memory. So does a
// domain whose coefficients the limbs cannot carry, and, point by point, an
// output whose products are too small for the limb sums (kLimbEnough). Which
// those are depends on the data of the tile and level only, not on the launch.
//
// Errors: an output is within about one rounding of the exact value of the
// sum and one of its product with T, against the several roundings of native
// FP64 arithmetic: relative to 64-bit evaluation 6.9e-16 where that had 8.2e-16
// (smooth winds, whose fluxes cancel), 1.4e-16 on i.i.d. winds for both.
//
// k-march: TMA brings each level of u, v, w (tile + halo, doubles) into one
// stage. Step k computes level k from the limbs of levels k-1, k and k+1 in a
// ring of three, two points per thread in turn; a barrier frees level k-1's
// slot, level k+2 is split into it, and a second barrier publishes it and frees
// the stage, so that the next level's copy has a step's products to arrive. Two
// points per thread halve the per-level work of a warp (waits, barriers, scale
// bookkeeping: about 130 of 650 instructions at one point) and a 32 x 16 tile
// splits 1.2 values per point and field (1.33 at 32 x 8).
//
// Bound: the integer pipes. 605 thread instructions per point (114 multiply-adds,
// a quarter of the FP32 rate each; about 90 for the split, 80 for the roundings,
// 70 for the scalings by rho), issue 48 %, 16 warps per SM at 128 registers;
// FP64 pipe 16 %, DRAM 19 %. Neither more warps (96 registers, 20 warps), nor
// shorter chains (separate sums of each limb product), nor the multiply-add as
// a product and an addition (half rate, one instruction more) moved it by more
// than 3 %. A tile's first three levels are copied at once, two of them into limb
// slots not yet in use, before the scan of the coefficients (one after another
// through the stage: 562 us at 512x512x64, 157 at 256x256x64 where it is now 150).
// 512x512x64 without density: 1043 -> 543 us (31 GPt/s); with density 1138 -> 571
// us; 1000x250x37 with density, tcx != tcy, unaligned: 658 -> 370 us; 128x128x64:
// 82 -> 45 us; a batch of 20 domains: 3879 -> 2078 us. Winds of 1e3 or 1e-3 times
// that size take 557 and 623 us. A field of FP64 steps only costs about 1700 us at
// 512x512x64, more than before; winds that cross zero to rounding on a few grid
// lines (2^-53 beside 1: those tiles fall to FP64) 1070, a Gaussian of 40 columns'
// width around one point 1340. Cutting values below the window instead of refusing
// them gained nothing there (their outputs are too small for the limb sums).
#include <cuda.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "pw.h"
#include "pw_common.cuh"
#include "pw_internal.h"
#include "pw_limb.cuh"
#include "pw_ring.cuh"

namespace pw {

namespace {

struct F64Cfg {
    // a thread owns PTS points of a column of the tile, ROWS rows apart
    static constexpr int TX = 32, TY = 16, S = 1, PTS = 2, ROWS = TY / PTS;
    using Shape = RingShape<double, TX, TY, S>;
    static constexpr int NT = TX * ROWS;
    static constexpr int MINB = 2;
    static constexpr int BX = Shape::BX;
    // limb cells {h, m, l, 0} of a field and level: rows 0..TY+1, columns 0..TX+1
    static constexpr int W = TX + 2, H = TY + 2, CELLS = W * H;
    static constexpr int SLOT = 3 * CELLS;
    static constexpr int SLOTS = 3;
    // Split work in chunks of 32 cells, warp w taking w, w + NT/32, ...: chunk
    // c < 3 H is columns 0..31 of row c % H of field c / H, the rest the last
    // two columns.
    static constexpr int ALL = 3 * H + (6 * H + 31) / 32, WARPS = NT / 32;
    static constexpr int CHUNKS = (ALL + WARPS - 1) / WARPS;
    // ring stages | ring barriers (64 B) | limbs [SLOTS][SLOT] | coefficients [4][4] | item, range, big | slack
    static constexpr int LIMB_OFFSET = S * Shape::STAGE_BYTES + 64;
    static constexpr int COEF_OFFSET = LIMB_OFFSET + SLOTS * SLOT * 16;
    static constexpr int ITEM_OFFSET = COEF_OFFSET + 4 * 4 * 16;
    static constexpr int SMEM_BYTES = ITEM_OFFSET + 32 + 128;
    static_assert((S + 2) * 8 <= 64, "ring and start barriers must fit before the limbs");
    static_assert(MINB * (SMEM_BYTES + 1024) <= 228 * 1024, "CTAs per SM");
    // While a tile starts, its first two levels arrive in limb slots 1 and 2 (not
    // yet in use), the third in the stage, so that the three copies overlap.
    static constexpr int RAW1 = round_up(LIMB_OFFSET + SLOT * 16, 128), RAW2 = round_up(LIMB_OFFSET + 2 * SLOT * 16, 128);
    static_assert(S == 1 && RAW1 + Shape::STAGE_BYTES <= LIMB_OFFSET + 2 * SLOT * 16 &&
                      RAW2 + Shape::STAGE_BYTES <= LIMB_OFFSET + 3 * SLOT * 16,
                  "a level's boxes fit a limb slot");
    static_assert(SLOT < 65536 && 3 * Shape::BOX_STRIDE / 8 < 65536, "offsets of a plan fit 16 bits");
};

template <class C>
struct F64K {
    using Shape = typename C::Shape;

    struct Smem {
        int4* limbs;      // [SLOTS][3][CELLS]
        int4* coef;       // [level & 3][4]: rho of tzc1, -tzc2, tzd1, -tzd2
        long long* item;  // work item handed from thread 0 to the CTA
        int* range;       // [2] exponents of the coefficients; [0] also of a level's values
        unsigned* big;    // [4]: the last load of this slot that held a value near its window's top
    };

    static __device__ __forceinline__ void setup(unsigned char* raw, Ring<Shape>& ring, Smem& sm) {
        ring.setup(raw);
        sm.limbs = reinterpret_cast<int4*>(ring.base + C::LIMB_OFFSET);
        sm.coef = reinterpret_cast<int4*>(ring.base + C::COEF_OFFSET);
        sm.item = reinterpret_cast<long long*>(ring.base + C::ITEM_OFFSET);
        sm.range = reinterpret_cast<int*>(ring.base + C::ITEM_OFFSET + 8);
        sm.big = reinterpret_cast<unsigned*>(ring.base + C::ITEM_OFFSET + 16);
    }

    // The ring's barrier, and one for each of a tile's first two levels.
    static __device__ __forceinline__ void init_barriers(Ring<Shape>& ring) {
        mbar_init(&ring.full[1], 1);
        mbar_init(&ring.full[2], 1);
        ring.init_barriers();
    }

    // Where a CTA stands: loads by level (tags of the limb slots), loads through
    // the ring, and the phases of the two start barriers.
    struct Counts {
        long long levels = 0, ring = 0;
        unsigned phase1 = 0, phase2 = 0;
    };

    // Levels read by a chunk kb..ke-1: one below, one above.
    static __device__ __forceinline__ int lowest(int kb) { return kb > 0 ? kb - 1 : 0; }
    static __device__ __forceinline__ int highest(const FwdArgs& a, int ke) { return ke < a.nz ? ke : a.nz - 1; }

    // Issue a tile's first three levels (one thread).
    static __device__ __forceinline__ void start_tile(Ring<Shape>& ring, const CUtensorMap* mu, const CUtensorMap* mv,
                                                      const CUtensorMap* mw, const FwdArgs& a, int bx, int by, int kb,
                                                      int ke, const Counts& n) {
        const int x0 = bx * C::TX, y0 = by * C::TY, lo = lowest(kb), nl = highest(a, ke) - lo + 1;
        fence_proxy_async_smem();
        for (int r = 0; r < 2 && r < nl; ++r) {
            uint64_t* bar = &ring.full[1 + r];
            unsigned char* dst = ring.base + (r == 0 ? C::RAW1 : C::RAW2);
            mbar_arrive_expect_tx(bar, 3 * Shape::BOX_BYTES);
            tma_load_3d(dst, mu, bar, x0, y0, lo + r);
            tma_load_3d(dst + Shape::BOX_STRIDE, mv, bar, x0, y0, lo + r);
            tma_load_3d(dst + 2 * Shape::BOX_STRIDE, mw, bar, x0, y0, lo + r);
        }
        if (nl > 2) ring.issue((long long)(unsigned)n.ring, lo + 2, mu, mv, mw, x0, y0);
    }

    // What the coefficient arrays of a domain allow: equal lower and upper
    // coefficients on every level, and how much lower w's window lies than u's
    // and v's (delta, at most -3), so that every rho 2^delta lies in [2^-30, 2)
    // or is 0.
    struct Domain {
        bool equal, limbs;
        int delta;
    };

    static __device__ __forceinline__ Domain scan_coefs(const FwdArgs& a, const Smem& sm, int tid) {
        if (tid == 0) {
            sm.range[0] = -4096;
            sm.range[1] = 4096;
        }
        __syncthreads();
        bool eq = true;
        int mx = -4096, mn = 4096;
        const int einv = (__double2hiint(a.tinv) >> 20) & 0x7FF;
        auto see = [&](double c) {
            const int h = __double2hiint(c) & 0x7FFFFFFF;
            if ((h | __double2loint(c)) == 0) return;
            const int e = (h >> 20) + einv - 2046;  // c / T in 2^e [1, 4)
            mx = max(mx, h >= 0x7FF00000 || h < 0x00100000 ? 4096 : e);
            mn = min(mn, e);
        };
        auto same = [](double x, double y) {
            return __double2hiint(x) == __double2hiint(y) && __double2loint(x) == __double2loint(y);
        };
        for (int k = 1 + tid; k < a.nz; k += C::NT) {
            const double t1 = __ldg(a.tzc1 + k);
            see(t1);
            if (k <= a.nz - 2) {
                const double t2 = __ldg(a.tzc2 + k), d1 = __ldg(a.tzd1 + k), d2 = __ldg(a.tzd2 + k);
                see(t2);
                see(d1);
                see(d2);
                eq &= same(t1, t2) && same(d1, d2);
            }
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        mn = __reduce_min_sync(0xffffffffu, mn);
        if ((tid & 31) == 0) {
            atomicMax(&sm.range[0], mx);
            atomicMin(&sm.range[1], mn);
        }
        Domain d;
        d.equal = __syncthreads_and(eq) != 0;
        mx = sm.range[0];
        mn = sm.range[1];
        d.delta = min(-3, -mx - 1);  // c / T < 2^(mx + 2)
        d.limbs = a.limbs && d.delta >= -40 && mn + d.delta >= -30;
        __syncthreads();  // the range is read before the next item writes it
        return d;
    }

    struct Plan {
        unsigned cell[C::CHUNKS];  // offset (doubles) in a stage at xoff = 0, << 16 | cell in a limb slot
    };

    static __device__ __forceinline__ Plan make_plan(int tid) {
        Plan p;
        const int warp = tid >> 5, lane = tid & 31;
#pragma unroll
        for (int q = 0; q < C::CHUNKS; ++q) {
            const int c = min(warp + q * C::WARPS, C::ALL - 1);
            int f = c / C::H, row = c % C::H, x = lane;
            if (c >= 3 * C::H) {
                // (the lanes past the last cell split it again, to the same limbs)
                const int n = min((c - 3 * C::H) * 32 + lane, 6 * C::H - 1);
                f = n / (2 * C::H);
                row = (n % (2 * C::H)) >> 1;
                x = 32 + (n & 1);
            }
            p.cell[q] = (unsigned)(f * (Shape::BOX_STRIDE / 8) + row * C::BX + x) << 16 |
                        (unsigned)(f * C::CELLS + row * C::W + x);
        }
        return p;
    }

    // Whether the warp has a chunk q.
    static __device__ __forceinline__ bool has_chunk(int tid, int q) {
        return (q + 1) * C::WARPS <= C::ALL || (tid >> 5) + q * C::WARPS < C::ALL;
    }

    // rho of level lev: lane n of warp 4 takes tzc1, -tzc2, tzd1, -tzd2 (loaded one split earlier).
    static __device__ __forceinline__ double coef_for(const FwdArgs& a, int lev, int tid) {
        const int n = tid - 128;
        if ((unsigned)n >= 4u) return 0.0;
        const double* arr = n == 0 ? a.tzc1 : n == 1 ? a.tzc2 : n == 2 ? a.tzd1 : a.tzd2;
        return __ldg(arr + lev);
    }

    // Split the staged boxes of level lev into limb slot `slot` at scale z (tag:
    // the level's number in the CTA's loads); false where a value is outside its
    // window. Tells the CTA where one lies in the scale's
    // own binades (the top kLimbStep of the window).
    static __device__ __forceinline__ bool split_level(const unsigned char* stage, const Smem& sm, unsigned tag, int lev,
                                                       int slot, int z, const FwdArgs& a, int delta, int tid,
                                                       const Plan& p, double coef) {
        const double* base = reinterpret_cast<const double*>(stage) + a.xoff;
        int4* out = sm.limbs + slot * C::SLOT;
        const int eh = kLimbExp + kLimbStep * z;
        bool ok = true;
        int top = kLimbWindow;
#pragma unroll
        for (int q = 0; q < C::CHUNKS; ++q) {
            if (!has_chunk(tid, q)) break;
            const int src = (int)(p.cell[q] >> 16), dst = (int)(p.cell[q] & 0xFFFFu);
            Limb3 v;
            int depth;
            ok &= limb_split(base[src], dst >= 2 * C::CELLS ? eh + delta : eh, &v, &depth);
            top = min(top, depth);
            out[dst] = make_int4(v.h, v.m, v.l, 0);
        }
        if (__any_sync(0xffffffffu, top < kLimbStep) && (tid & 31) == 0) sm.big[slot] = tag;
        const int n = tid - 128;
        if ((unsigned)n < 4u) {
            // w's limbs count 2^delta of u's
            const double two = __hiloint2double((1023 + delta) << 20, 0);
            const double r = __dmul_rn(__dmul_rn(coef, two), a.tinv);
            Limb3 v;
            (void)limb_split<31>(r, 2, &v);  // in range: see scan_coefs
            if (n & 1) v = Limb3{-v.h, -v.m, -v.l};
            sm.coef[(lev & 3) * 4 + n] = make_int4(v.h, v.m, v.l, 0);
        }
        return ok;
    }

    // The scale of a level that did not suit scale *z: from its largest
    // magnitude (w counted 2^-delta). Splits it again at that scale and returns
    // it (and in *z, for the next level), kZero for a level of zeros, or kNone
    // where no scale holds all its values. Every thread of the CTA calls it.
    static constexpr int kNone = 1 << 20, kZero = 1 << 21;
    static __device__ __noinline__ int rescale_level(const double* box, int4* limbs, int* range, int z, int delta, int tid) {
        const Plan p = make_plan(tid);
        int top = -8192;
        for (int q = 0; q < C::CHUNKS; ++q) {
            const int src = (int)(p.cell[q] >> 16), dst = (int)(p.cell[q] & 0xFFFFu);
            const int hi = __double2hiint(box[src]);
            const int e = ((hi >> 20) & 0x7FF) - 1023 - (dst >= 2 * C::CELLS ? delta : 0);
            if ((hi & 0x7FF00000) != 0) top = max(top, e);
        }
        if (tid == 0) *range = -8192;
        __syncthreads();
        top = __reduce_max_sync(0xffffffffu, top);
        if ((tid & 31) == 0) atomicMax(range, top);
        __syncthreads();
        top = *range;
        // z with 2^(E - kLimbStep) <= 2^top < 2^E (a level of zeros and subnormals: any)
        const int up = top - (kLimbExp - kLimbStep);
        const int zn = top == -8192 ? z : (up >= 0 ? up / kLimbStep : -((kLimbStep - 1 - up) / kLimbStep));
        bool ok = zn >= -25 && zn <= 25;  // (the results' exponents stay normal)
        const int eh = kLimbExp + kLimbStep * (ok ? zn : 0);
        for (int q = 0; q < C::CHUNKS; ++q) {
            const int src = (int)(p.cell[q] >> 16), dst = (int)(p.cell[q] & 0xFFFFu);
            Limb3 v;
            ok &= limb_split(box[src], dst >= 2 * C::CELLS ? eh + delta : eh, &v);
            limbs[dst] = make_int4(v.h, v.m, v.l, 0);
        }
        const bool none = __syncthreads_or(!ok) != 0;
        return none ? kNone : top == -8192 ? kZero : zn;
    }

    struct Slot {
        const int4* p;
        __device__ __forceinline__ Limb3 operator()(int c) const {
            const int4 t = p[c];
            return {t.x, t.y, t.z};
        }
    };

    static __device__ __forceinline__ Limb3 rho(const Smem& sm, int lev, int n) {
        const int4 t = sm.coef[(lev & 3) * 4 + n];
        return {t.x, t.y, t.z};
    }

    // rx X + ry Y (where tcx and tcy differ)
    static __device__ __forceinline__ LimbSum join_xy(LimbSum x, LimbSum y, const Limb3& rx, const Limb3& ry) {
        LimbSum s = limb_zero();
        limb_mac_scaled(s, x, rx);
        limb_mac_scaled(s, y, ry);
        return s;
    }

    // s + rho1 lo + rho2 hi: lo and hi the products through the lower and the
    // upper face (hi negated in kEq, where both take rho1; -rho2 is stored).
    template <bool kEq, bool kTop>
    static __device__ __forceinline__ void add_z(LimbSum& s, const Smem& sm, int lev, int n, Limb3 qlo, Limb3 flo,
                                                 Limb3 qhi, Limb3 fhi) {
        LimbSum z = limb_zero();
        limb_mac(z, qlo, flo);
        if (kEq) {
            if (!kTop) limb_mac(z, Limb3{-qhi.h, -qhi.m, -qhi.l}, fhi);
            limb_mac_scaled(s, z, rho(sm, lev, n));
        } else {
            limb_mac_scaled(s, z, rho(sm, lev, n));
            if (!kTop) {
                LimbSum y = limb_zero();
                limb_mac(y, qhi, fhi);
                limb_mac_scaled(s, y, rho(sm, lev, n + 1));
            }
        }
    }

    // Level k's three outputs on limbs: B, M and P the point in the slots of
    // levels k-1, k and k+1; su_scale of LimbSum's unit.
    template <bool kEq, bool kSameT, bool kTop>
    static __device__ __forceinline__ void limb_point(const Smem& sm, const int4* B, const int4* M, const int4* P, int lev,
                                                      const Limb3& rx, const Limb3& ry, double tref, int eh, int delta,
                                                      double* r_su, double* r_sv, double* r_sw, unsigned* small) {
        constexpr int W = C::W, N = C::CELLS;
        const Slot U{M}, V{M + N}, Z{M + 2 * N}, U1{P}, V1{P + N}, Z1{P + 2 * N}, Ub{B}, Vb{B + N}, Zb{B + 2 * N};
        const int su_scale = 2 * (eh - 86), sw_scale = su_scale + delta;
        const Limb3 uc = U(0), vc = V(0), wc = Z(0), wb = Zb(0);
        const Limb3 none = {0, 0, 0};
        {
            const Limb3 uw = U(-1), ue = U(1);
            LimbSum x = limb_zero(), y = limb_zero();
            // (u(i-1) - u(i+1)) (u(i-1) + u(i) + u(i+1)) is the two x terms in one product
            limb_mac(x, limb_sub(uw, ue), limb_add(limb_add(uw, uc), ue));
            LimbSum& yy = kSameT ? x : y;
            limb_mac(yy, U(-W), limb_add(V(-W), V(1 - W)));
            limb_mac(yy, U(W), limb_neg_sum(vc, V(1)));
            LimbSum s = kSameT ? x : join_xy(x, y, rx, ry);
            add_z<kEq, kTop>(s, sm, lev, 0, Ub(0), limb_add(wb, Zb(1)), kTop ? none : U1(0), limb_add(wc, Z(1)));
            limb_carry(s);
            bool large;
            *r_su = __dmul_rn(tref, limb_to_double(s, su_scale, &large));
            *small = large ? 0u : 1u;
        }
        {
            const Limb3 vs = V(-W), vn = V(W);
            LimbSum x = limb_zero(), y = limb_zero();
            limb_mac(y, limb_sub(vs, vn), limb_add(limb_add(vs, vc), vn));
            LimbSum& xx = kSameT ? y : x;
            limb_mac(xx, V(-1), limb_add(U(-1), U(W - 1)));
            limb_mac(xx, V(1), limb_neg_sum(uc, U(W)));
            LimbSum s = kSameT ? y : join_xy(x, y, rx, ry);
            add_z<kEq, kTop>(s, sm, lev, 0, Vb(0), limb_add(wb, Zb(W)), kTop ? none : V1(0), limb_add(wc, Z(W)));
            limb_carry(s);
            bool large;
            *r_sv = __dmul_rn(tref, limb_to_double(s, su_scale, &large));
            *small |= large ? 0u : 2u;
        }
        *r_sw = 0.0;
        if constexpr (!kTop) {
            const Limb3 wu = Z1(0);
            LimbSum x = limb_zero(), y = limb_zero();
            LimbSum& yy = kSameT ? x : y;
            limb_mac(x, Z(-1), limb_add(U(-1), U1(-1)));
            limb_mac(x, Z(1), limb_neg_sum(uc, U1(0)));
            limb_mac(yy, Z(-W), limb_add(V(-W), V1(-W)));
            limb_mac(yy, Z(W), limb_neg_sum(vc, V1(0)));
            LimbSum s = kSameT ? x : join_xy(x, y, rx, ry);
            add_z<kEq, false>(s, sm, lev, 2, wb, limb_add(wc, wb), wu, limb_add(wc, wu));
            limb_carry(s);
            bool large;
            *r_sw = __dmul_rn(tref, limb_to_double(s, sw_scale, &large));
            *small |= large ? 0u : 4u;
        }
    }

    // Of the outputs in `which`, whose limb sums came out small, those that the
    // limbs do not settle: neither do the magnitudes of their horizontal
    // products, with their coefficients, reach 2^28 units, nor are all their
    // advected values 0 (then the output is exactly 0). U, U1: the point in the slots of levels k and k+1; e: the point's
    // offset in the fields, on level k.
    static __device__ __noinline__ unsigned unsettled(const int4* U, const int4* U1, unsigned which, bool top,
                                                      const FwdArgs* a, size_t e) {
        constexpr int W = C::W, N = C::CELLS;
        const int4 *V = U + N, *Z = V + N, *V1 = U1 + N, *Z1 = V1 + N;
        auto zero = [](const int4& a) { return (a.x | a.y | a.z) == 0; };
        auto zero5 = [&](const int4* q, const int4* up) {
            return zero(q[-1]) && zero(q[1]) && zero(q[-W]) && zero(q[W]) && (top || zero(*up));
        };
        // (tcx and tcy over tref multiply the products before the sum is formed)
        const int sx = a->same_t ? 0 : limb_binades(__dmul_rn(a->tcx, a->tinv));
        const int sy = a->same_t ? 0 : limb_binades(__dmul_rn(a->tcy, a->tinv));
        unsigned left = 0;
        if ((which & 1u) && !(__ldg(static_cast<const double*>(a->u) + e - a->sz) == 0.0 && zero5(U, U1))) {
            const long long x = limb_least(U[-1].x - U[1].x, U[-1].x + U[0].x + U[1].x);
            const long long y = limb_least(U[-W].x, V[-W].x + V[1 - W].x) + limb_least(U[W].x, V[0].x + V[1].x);
            if (!limb_settled(x, y, sx, sy)) left |= 1u;
        }
        if ((which & 2u) && !(__ldg(static_cast<const double*>(a->v) + e - a->sz) == 0.0 && zero5(V, V1))) {
            const long long x = limb_least(V[-1].x, U[-1].x + U[W - 1].x) + limb_least(V[1].x, U[0].x + U[W].x);
            const long long y = limb_least(V[-W].x - V[W].x, V[-W].x + V[0].x + V[W].x);
            if (!limb_settled(x, y, sx, sy)) left |= 2u;
        }
        if ((which & 4u) && !(__ldg(static_cast<const double*>(a->w) + e - a->sz) == 0.0 && zero5(Z, Z1))) {
            const long long x = limb_least(Z[-1].x, U[-1].x + U1[-1].x) + limb_least(Z[1].x, U[0].x + U1[0].x);
            const long long y = limb_least(Z[-W].x, V[-W].x + V1[-W].x) + limb_least(Z[W].x, V[0].x + V1[0].x);
            if (!limb_settled(x, y, sx, sy)) left |= 4u;
        }
        return left;
    }

    // A point in native FP64, term by term, from global memory (e: its offset
    // in the fields, on level k).
    static __device__ __noinline__ double3 native_point(const FwdArgs* args, size_t e, int k) {
        const FwdArgs& a = *args;
        const size_t sy = (size_t)a.sy, sz = (size_t)a.sz;
        const double *U = static_cast<const double*>(a.u) + e, *V = static_cast<const double*>(a.v) + e;
        const double *Wl = static_cast<const double*>(a.w) + e;
        const double *Ub = U - sz, *Vb = V - sz, *Wb = Wl - sz;
        const bool top = k == a.nz - 1;
        const double t1 = __ldg(a.tzc1 + k);
        const double wc = __ldg(Wl), wx = wc + __ldg(Wl + 1), wy = wc + __ldg(Wl + sy), wb = __ldg(Wb);
        const double uc = __ldg(U), uw = __ldg(U - 1), ue = __ldg(U + 1), us = __ldg(U - sy), un = __ldg(U + sy);
        const double vc = __ldg(V), vw = __ldg(V - 1), ve = __ldg(V + 1), vs = __ldg(V - sy), vn = __ldg(V + sy);
        double su = a.tcx * (uw * (uc + uw) - ue * (uc + ue));
        su += a.tcy * (us * (vs + __ldg(V - sy + 1)) - un * (vc + ve));
        su += t1 * (__ldg(Ub) * (wb + __ldg(Wb + 1)));
        double sv = a.tcy * (vs * (vc + vs) - vn * (vc + vn));
        sv += a.tcx * (vw * (uw + __ldg(U + sy - 1)) - ve * (uc + un));
        sv += t1 * (__ldg(Vb) * (wb + __ldg(Wb + sy)));
        double sw = 0.0;
        if (!top) {
            const double *U1 = U + sz, *V1 = V + sz;
            const double t2 = __ldg(a.tzc2 + k), u1 = __ldg(U1), v1 = __ldg(V1), w1 = __ldg(Wl + sz);
            su -= t2 * (u1 * wx);
            sv -= t2 * (v1 * wy);
            sw = a.tcx * (__ldg(Wl - 1) * (uw + __ldg(U1 - 1)) - __ldg(Wl + 1) * (uc + u1));
            sw += a.tcy * (__ldg(Wl - sy) * (vs + __ldg(V1 - sy)) - __ldg(Wl + sy) * (vc + v1));
            sw += __ldg(a.tzd1 + k) * (wb * (wc + wb)) - __ldg(a.tzd2 + k) * (w1 * (wc + w1));
        }
        return make_double3(su, sv, sw);
    }

    // One tile (bx, by) of domain `a`, output levels kb..ke-1 (a chunk of the
    // column; it reads one level below and one above), its first levels issued by
    // start_tile. Loads are numbered relative to the lowest level read, lo: 0 and
    // 1 come through the start barriers, the others through the ring. Returns
    // false if a bounded wait expired (status set, copies drained). args: `a` in
    // memory.
    template <bool kEq, bool kSameT>
    static __device__ bool tile_impl(Ring<Shape>& ring, const Smem& sm, const CUtensorMap* mu, const CUtensorMap* mv,
                                     const CUtensorMap* mw, const FwdArgs& a, const FwdArgs* args, const Domain& dom,
                                     int bx, int by, int kb, int ke, Counts& count, int tid, const Plan& plan) {
        const int tx = tid % C::TX, ty = tid / C::TX;
        const int x0 = bx * C::TX, y0 = by * C::TY;
        const int i = x0 + 1 + tx, j = y0 + 1 + ty;  // the thread's first point; the others ROWS rows up each
        const int act = i <= a.nx && j <= a.ny ? min(C::PTS, (a.ny - j) / C::ROWS + 1) : 0;  // points inside the domain
        const int nz = a.nz;
        const int lo = lowest(kb), hi = highest(a, ke);
        const int nl = hi - lo + 1;  // levels read
        int issued = min(nl, 3);     // relative loads issued (thread 0)
        auto ring_load = [&](int r) { return (long long)(unsigned)(count.ring + (r - 2)); };
        auto wait = [&](int r) {
            return r == 0   ? mbar_wait_bounded(&ring.full[1], count.phase1 & 1)
                   : r == 1 ? mbar_wait_bounded(&ring.full[2], count.phase2 & 1)
                            : ring.wait(ring_load(r));
        };
        auto stage = [&](int r) { return ring.base + (r == 0 ? C::RAW1 : r == 1 ? C::RAW2 : 0); };
        double* __restrict__ su = static_cast<double*>(a.su);
        double* __restrict__ sv = static_cast<double*>(a.sv);
        double* __restrict__ sw = static_cast<double*>(a.sw);
        const size_t gsz = (size_t)a.sz;
        size_t g = (size_t)j * (size_t)a.sy + (size_t)i + (size_t)lo * gsz;
        const size_t grow = (size_t)C::ROWS * (size_t)a.sy;
        if (kb == 0) {  // level 1 of the paper is not computed
            for (int n = 0; n < act; ++n) {
                su[g + n * grow] = 0.0;
                sv[g + n * grow] = 0.0;
                sw[g + n * grow] = 0.0;
            }
        }
        Limb3 rx = {0, 0, 0}, ry = {0, 0, 0};
        if (!kSameT) {
            (void)limb_split<31>(__dmul_rn(a.tcx, a.tinv), 2, &rx);
            (void)limb_split<31>(__dmul_rn(a.tcy, a.tinv), 2, &ry);
        }

        const int c = (ty + 1) * C::W + tx + 1;  // the first point in a limb slot
        bool bad = false, abort = false;
        int z = 0;  // scale of the last level that had one
        // The level split at relative level r (ok: no value refused by this
        // thread), after the CTA's barrier: its scale, kZero or kNone.
        auto settle = [&](int r, bool refused) {
            if (!refused && sm.big[r % 3] == (unsigned)(count.levels + r)) return z;
            const int t = rescale_level(reinterpret_cast<const double*>(stage(r)) + a.xoff, sm.limbs + (r % 3) * C::SLOT,
                                        sm.range, z, dom.delta, tid);
            if (t < kNone) z = t;
            return t;
        };
        // relative levels 0..2 are split up front; the step at r splits r+2.
        // t0, t1, t2: scales of levels r-1, r, r+1 (CTA-uniform)
        double c_pre = coef_for(a, lo, tid);
        int t[3] = {kZero, kZero, kZero};
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            if (r < nl && !abort) {
                bad |= !wait(r);
                const bool ok = split_level(stage(r), sm, (unsigned)(count.levels + r), lo + r, r, z, a, dom.delta, tid,
                                            plan, c_pre);
                if (lo + r + 1 <= hi) c_pre = coef_for(a, lo + r + 1, tid);
                const bool refused = __syncthreads_or(bad || !ok) != 0;
                if (refused) abort = __syncthreads_or(bad);
                if (!abort) t[r] = settle(r, refused);
                if (r == 2 && !abort && tid == 0 && issued < nl) {  // the stage is free again
                    fence_proxy_async_smem();
                    ring.issue(ring_load(issued), lo + issued, mu, mv, mw, x0, y0);
                    ++issued;
                }
            }
        }
        int t0 = t[0], t1 = t[1], t2 = t[2];
        const int k1 = kb > 1 ? kb : 1;  // first computed level (lo = k1 - 1)
        g += (size_t)(k1 - lo) * gsz;

        // Level k = lo + r from the limb slots of r-1, r and r+1 (sl, sc, sp);
        // level k+2 then goes into slot sl.
        auto step = [&](auto top, int sl, int sc, int sp, int r) {
            constexpr bool kTop = decltype(top)::value;
            const int k = lo + r;
            // one scale for the three levels (zeros have any)
            const int zs = min(min(t0, t1), kTop ? kZero : t2);
            const bool limbs = dom.limbs && zs != kNone && (t0 == zs || t0 == kZero) && (t1 == zs || t1 == kZero) &&
                               (kTop || t2 == zs || t2 == kZero);
            const int eh = kLimbExp + kLimbStep * (zs == kZero ? 0 : zs);
            const int4* B = sm.limbs + sl * C::SLOT + c;
            const int4* M = sm.limbs + sc * C::SLOT + c;
            const int4* P = sm.limbs + sp * C::SLOT + c;
            size_t e = g;
#pragma unroll 1
            for (int n = 0; n < act; ++n) {
                double r_su, r_sv, r_sw;
                unsigned fp64 = 7u;  // outputs to evaluate in FP64
                if (limbs) {
                    unsigned small = 0;  // outputs whose limb sums are small
                    limb_point<kEq, kSameT, kTop>(sm, B, M, P, k, rx, ry, a.tref, eh, dom.delta, &r_su, &r_sv, &r_sw, &small);
                    fp64 = small != 0 ? unsettled(M, P, small, kTop, args, e) : 0u;
                }
                if (fp64 != 0) {
                    const double3 t = native_point(args, e, k);
                    if (fp64 & 1u) r_su = t.x;
                    if (fp64 & 2u) r_sv = t.y;
                    if (fp64 & 4u) r_sw = t.z;
                }
                su[e] = r_su;
                sv[e] = r_sv;
                sw[e] = r_sw;
                B += C::ROWS * C::W;
                M += C::ROWS * C::W;
                P += C::ROWS * C::W;
                e += grow;
            }
            g += gsz;
            t0 = t1;
            t1 = t2;
            if (kTop) return;
            t2 = kNone;
            __syncthreads();  // level k-1's limbs are free
            if (r + 2 < nl) {
                bad |= !ring.wait(ring_load(r + 2));
                bool ok = true;
                if (dom.limbs)
                    ok = split_level(ring.base, sm, (unsigned)(count.levels + r + 2), k + 2, sl, z, a, dom.delta, tid, plan,
                                     c_pre);
                if (k + 3 <= hi) c_pre = coef_for(a, k + 3, tid);
                // publishes level k+2's limbs, frees its stage
                const bool refused = __syncthreads_or(bad || !ok) != 0;
                if (refused) abort = __syncthreads_or(bad);
                if (!abort && dom.limbs) t2 = settle(r + 2, refused);
                if (!abort && tid == 0 && issued < nl) {
                    fence_proxy_async_smem();
                    ring.issue(ring_load(issued), lo + issued, mu, mv, mw, x0, y0);
                    ++issued;
                }
            }
        };
        const int rend = (ke < nz ? ke : nz - 1) - lo;
        int sl = 0, sc = 1, sp = 2;
#pragma unroll 1
        for (int r = 1; r < rend && !abort; ++r) {
            step(std::false_type(), sl, sc, sp, r);
            const int freed = sl;
            sl = sc;
            sc = sp;
            sp = freed;
        }
        if (ke == nz && k1 < ke && !abort) step(std::true_type(), sl, sc, sp, nz - 1 - lo);  // the domain's top level
        if (abort) {
            if (tid == 0) {
                atomicOr(&tu_status, kStatusTimeout);
                for (int q = 0; q < issued; ++q)
                    if (q < 2 || q == issued - 1) (void)wait(q);
            }
            return false;
        }
        __syncthreads();  // every read of this tile's stages and limbs is done before the next tile's
        count.levels += nl;
        count.ring += max(nl - 2, 0);
        count.phase1 += 1;
        count.phase2 += nl > 1 ? 1 : 0;
        return true;
    }

    template <bool kSameT>
    static __device__ bool tile(Ring<Shape>& ring, const Smem& sm, const CUtensorMap* mu, const CUtensorMap* mv,
                                const CUtensorMap* mw, const FwdArgs& a, const FwdArgs* args, int bx, int by, int kb,
                                int ke, Counts& count, int tid, const Plan& plan) {
        if (tid == 0) start_tile(ring, mu, mv, mw, a, bx, by, kb, ke, count);  // (the scan runs while they arrive)
        const Domain d = scan_coefs(a, sm, tid);
        if (d.equal) return tile_impl<true, kSameT>(ring, sm, mu, mv, mw, a, args, d, bx, by, kb, ke, count, tid, plan);
        return tile_impl<false, kSameT>(ring, sm, mu, mv, mw, a, args, d, bx, by, kb, ke, count, tid, plan);
    }
};

template <class C, bool kSameT>
__global__ void __launch_bounds__(C::NT, C::MINB) fwd_f64_kernel(const __grid_constant__ CUtensorMap mu,
                                                                 const __grid_constant__ CUtensorMap mv,
                                                                 const __grid_constant__ CUtensorMap mw,
                                                                 const __grid_constant__ FwdArgs a,
                                                                 const ItemSched sched) {
    using K = F64K<C>;
    extern __shared__ unsigned char smem_raw[];
    Ring<typename C::Shape> ring;
    typename K::Smem sm;
    K::setup(smem_raw, ring, sm);
    const int tid = threadIdx.x;
    if (tid == 0) {
        prefetch_tensormap(&mu);
        prefetch_tensormap(&mv);
        prefetch_tensormap(&mw);
        K::init_barriers(ring);
    }
    if (tid < 4) sm.big[tid] = ~0u;
    __syncthreads();
    typename K::Counts count;
    int bx, by, k0, k1;
    sched_item(sched, a.kend - a.kbeg, blockIdx.x, &bx, &by, &k0, &k1);
    const typename K::Plan plan = K::make_plan(tid);
    (void)K::template tile<kSameT>(ring, sm, &mu, &mv, &mw, a, &a, bx, by, a.kbeg + k0, a.kbeg + k1, count, tid,
                                 plan);
}

// Persistent form over a batch plan: work items (one tile column of one
// domain) come from the plan's counter, at most n_items iterations.
template <class C>
__global__ void __launch_bounds__(C::NT, C::MINB) fwd_f64_batched(BatchPlan* plan, int variant) {
    using K = F64K<C>;
    extern __shared__ unsigned char smem_raw[];
    Ring<typename C::Shape> ring;
    typename K::Smem sm;
    K::setup(smem_raw, ring, sm);
    const int tid = threadIdx.x;
    if (plan->variant != variant || plan->dtype != PW_F64) {
        if (tid == 0) atomicOr(&tu_status, kStatusBadPlan);
        return;
    }
    if (tid == 0) K::init_barriers(ring);
    if (tid < 4) sm.big[tid] = ~0u;
    __syncthreads();
    const long long n_items = plan->n_items;
    const typename K::Plan split = K::make_plan(tid);
    typename K::Counts count;
    for (long long it = 0; it < n_items; ++it) {
        if (tid == 0) *sm.item = (long long)atomicAdd(&plan->counter, 1ull);
        __syncthreads();
        const long long item = *sm.item;
        __syncthreads();  // every thread has read the slot before thread 0 rewrites it
        if (item >= n_items) break;
        const BatchDomain& d = plan->dom[find_domain(plan, item)];
        // private copy: the plan is global memory the compiler cannot prove
        // free of the output stores
        const FwdArgs args = d.args;
        const long long t = item - d.first_item;
        const int tiles_x = d.tiles_x, kchunks = d.kchunks;
        const long long tiles = (long long)tiles_x * d.tiles_y;
        const int ch = (int)(t / tiles), tt = (int)(t % tiles);
        const int kb = (int)((long long)args.nz * ch / kchunks);
        const int ke = (int)((long long)args.nz * (ch + 1) / kchunks);
        const int bx = tt % tiles_x, by = tt / tiles_x;
        const bool go = args.same_t
                            ? K::template tile<true>(ring, sm, &d.mu, &d.mv, &d.mw, args, &d.args, bx, by, kb, ke, count, tid, split)
                            : K::template tile<false>(ring, sm, &d.mu, &d.mv, &d.mw, args, &d.args, bx, by, kb, ke, count, tid, split);
        if (!go) break;
    }
}

template <class C>
TileShape f64_shape_of() {
    return TileShape{C::TX, C::TY, C::Shape::BX, C::Shape::BY, C::SMEM_BYTES, C::NT};
}

template <class C>
cudaError_t launch_one(const CUtensorMap& mu, const CUtensorMap& mv, const CUtensorMap& mw, const FwdArgs& a,
                       cudaStream_t st) {
    auto kern = a.same_t ? fwd_f64_kernel<C, true> : fwd_f64_kernel<C, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    ItemSched sched;
    if ((e = choose_sched(kern, C::NT, C::SMEM_BYTES, (a.nx + C::TX - 1) / C::TX, (a.ny + C::TY - 1) / C::TY,
                          a.kend - a.kbeg, &sched)) != cudaSuccess)
        return e;
    kern<<<(unsigned)sched.items, C::NT, C::SMEM_BYTES, st>>>(mu, mv, mw, a, sched);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_batched_cfg(int v, BatchPlan* plan, long long n_items, cudaStream_t st) {
    auto kern = fwd_f64_batched<C>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    long long grid = 0;
    if ((e = persistent_grid(kern, C::NT, C::SMEM_BYTES, n_items, &grid)) != cudaSuccess) return e;
    if (grid < 1) return cudaSuccess;
    kern<<<(unsigned)grid, C::NT, C::SMEM_BYTES, st>>>(plan, v);
    return cudaGetLastError();
}

}  // namespace

cudaError_t read_and_clear_status_f64(unsigned int* status, cudaStream_t st) {
    return read_and_clear_tu_status(status, st);
}

// Two variant numbers, one kernel.
int f64_variant_count() { return 2; }

TileShape fwd_f64_shape_variant(int) { return f64_shape_of<F64Cfg>(); }

TileShape fwd_f64_shape() { return f64_shape_of<F64Cfg>(); }

cudaError_t launch_fwd_f64(const CUtensorMap& mu, const CUtensorMap& mv, const CUtensorMap& mw, const FwdArgs& a,
                           cudaStream_t st) {
    return launch_one<F64Cfg>(mu, mv, mw, a, st);
}

cudaError_t launch_f64_batched(int v, BatchPlan* plan, long long n_items, cudaStream_t st) {
    return launch_batched_cfg<F64Cfg>(v, plan, n_items, st);
}

}  // namespace pw
