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
// A step's windows come from the largest magnitudes of the three levels that it
// reads, in the tile with its halo, and from the level's coefficients (scale_of):
// one window for u and v, which meet in X and Y, raised where rho w exceeds them,
// and one for w. Where u or v lies far below the other each has its own, and X
// and Y get coefficients as where tcx and tcy differ. (One window for all three,
// shared by twelve binades of magnitudes and widened by the domain's largest rho,
// left most points of winds over dx >= 20 dz to FP64.) Values below their window
// are cut to its unit; an output whose products are all too small for the limb
// sums (kLimbEnough) is evaluated in FP64, term by term, from a list that the CTA
// works off with whole warps beside the next step's points. Steps that read an infinity or a NaN, or a domain
// whose coefficients no limb number holds, are evaluated in FP64 throughout. All
// of that depends on the data of the tile and its levels only, not on the launch.
//
// Errors: an output is within about one rounding of the exact value of the
// sum and one of its product with T, against the several roundings of native
// FP64 arithmetic: relative to 64-bit evaluation 8.0e-16 where that had 1.0e-15
// (smooth winds, whose fluxes cancel), 1.4e-16 on i.i.d. winds for both.
//
// k-march: TMA brings each level of u, v, w (tile + halo, doubles) into one
// stage. Step k computes level k from the limbs of levels k-1, k and k+1 in a
// ring of three, two points per thread in turn; a barrier frees level k-1's
// slot, level k+2 is split into it, in the windows of step k, and a second barrier
// publishes it and frees the stage, so that the next level's copy has a step's
// products to arrive. If the next step needs other windows, its levels' limbs are
// shifted (rescale). Two points per thread halve the per-level work of a warp and
// a 32 x 16 tile splits 1.2 values per point and field (1.33 at 32 x 8).
//
// Bound: the integer pipes and their latency. 637 thread instructions per point
// (114 multiply-adds, a quarter of the FP32 rate each; about 100 for the split, 80
// for the roundings, 70 for the scalings by rho, 26 for the windows), issue 48 %,
// 16 warps per SM at 128 registers; FP64 pipe 15 %, DRAM 18 %. Neither more warps
// (96 registers, 20 warps), nor shorter chains (separate sums of each limb product),
// nor the multiply-add as a product and an addition (half rate, one instruction
// more) moved it by more than 3 %. A tile's first three levels are copied at once,
// two of them into limb slots not yet in use (one after another through the stage:
// 3 % more at 512x512x64). The windows' upkeep is kept out of the common path: the
// largest magnitudes found in a pass of their own ahead of the first barrier cost
// 6 % more, a decision by one warp 2 %, a top level compiled without its upper
// face's sums from zeros in their place 2 %.
// 512x512x64, native FP64 before -> now (us): smooth winds dx = 50 m 1066 -> 601,
// dx = 400 1060 -> 609, dx = 4000 1060 -> 611; with density 1157 -> 635; dx = 40,
// dy = 60 m 1062 -> 680; i.i.d. winds dx = 50 m 1062 -> 584, 1000 m 1062 -> 595;
// w = 0 1064 -> 603; v and w of 1e-8 beside u = 5 1059 -> 765; Taylor-Green 1064
// -> 790; sines that vanish on a grid of lines 1062 -> 980. Slower than native
// FP64: a bump of 20 columns' width on nothing (its outskirts vary by more binades
// in one tile than the sums hold) 1067 -> 1470, levels whose magnitudes differ by
// 8 from each to the next 1063 -> 1250, magnitudes random over 14 decades 1062 ->
// 1660, NaN throughout 1062 -> 1690. (The FP64 outputs of half the warps before
// their points and of half after them: 1400 for the bump, but 2 % on every call.)
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
    // limb cells {h, m, l, whether it was cut} of a field and level: rows 0..TY+1, columns 0..TX+1
    static constexpr int W = TX + 2, H = TY + 2, CELLS = W * H;
    static constexpr int SLOT = 3 * CELLS;
    static constexpr int SLOTS = 3;
    // Split work: of a field's cells a thread takes tid, tid + NT and, half the
    // CTA in turn for each field, one of the REST cells after those.
    static constexpr int REST = CELLS - 2 * NT, HALF = NT / 2;
    static_assert(REST > 0 && REST <= HALF, "three cells of a field per thread at most");
    // ring stages | ring barriers (64 B) | limbs [SLOTS][SLOT] | coefficients [4][4] + 2 as limbs | as doubles |
    // scale [4] | largest magnitudes [4] | coefficient exponents [4] | item | list counts [2], [2] | lists [2] | arguments | slack
    static constexpr int LIMB_OFFSET = S * Shape::STAGE_BYTES + 64;
    static constexpr int COEF_OFFSET = LIMB_OFFSET + SLOTS * SLOT * 16;
    static constexpr int RAW_OFFSET = COEF_OFFSET + (4 * 4 + 2) * 16;
    static constexpr int SCALE_OFFSET = RAW_OFFSET + 4 * 4 * 8;
    static constexpr int TOP_OFFSET = SCALE_OFFSET + 4 * 16;
    static constexpr int EXP_OFFSET = TOP_OFFSET + 4 * 16;
    static constexpr int ITEM_OFFSET = EXP_OFFSET + 4 * 4;
    static constexpr int LIST_OFFSET = ITEM_OFFSET + 32;
    static constexpr int ARGS_OFFSET = LIST_OFFSET + 4 * TX * TY * 2;
    static constexpr int SMEM_BYTES = ARGS_OFFSET + round_up((int)sizeof(FwdArgs), 16) + 128;
    static_assert(TX * TY <= 512, "a point of the tile fits 9 bits");
    static_assert((S + 2) * 8 <= 64, "ring and start barriers must fit before the limbs");
    static_assert(MINB * (SMEM_BYTES + 1024) <= 228 * 1024, "CTAs per SM");
    // While a tile starts, its first two levels arrive in limb slots 1 and 2 (not
    // yet in use), the third in the stage, so that the three copies overlap.
    static constexpr int RAW1 = round_up(LIMB_OFFSET + SLOT * 16, 128), RAW2 = round_up(LIMB_OFFSET + 2 * SLOT * 16, 128);
    static_assert(S == 1 && RAW1 + Shape::STAGE_BYTES <= LIMB_OFFSET + 2 * SLOT * 16 &&
                      RAW2 + Shape::STAGE_BYTES <= LIMB_OFFSET + 3 * SLOT * 16,
                  "a level's boxes fit a limb slot");
};

template <class C>
struct F64K {
    using Shape = typename C::Shape;

    struct Smem {
        unsigned char* base;
        template <typename T>
        __device__ __forceinline__ T* at(int offset) const {
            return reinterpret_cast<T*>(base + offset);
        }
        __device__ __forceinline__ int4* limbs() const { return at<int4>(C::LIMB_OFFSET); }  // [SLOTS][3][CELLS]
        // [level & 3][4]: rho of tzc1, -tzc2, tzd1, -tzd2 at the current scale; [16], [17]: of tcx, tcy
        __device__ __forceinline__ int4* coef() const { return at<int4>(C::COEF_OFFSET); }
        // [level & 3][4]: tzc1, tzc2, tzd1, tzd2 over tref
        __device__ __forceinline__ double* raw() const { return at<double>(C::RAW_OFFSET); }
        // [0]: the limbs' windows u, v, w, d; [1].w: flags of scale_of; the others: see holds
        __device__ __forceinline__ int4* scale() const { return at<int4>(C::SCALE_OFFSET); }
        // [level & 3]: exponents of the largest magnitudes of u, v, w in the tile
        __device__ __forceinline__ int4* top() const { return at<int4>(C::TOP_OFFSET); }
        // [level & 3]: |raw| < 2^(cexp + 1), -64 at least
        __device__ __forceinline__ int* cexp() const { return at<int>(C::EXP_OFFSET); }
        // work item handed from thread 0 to the CTA
        __device__ __forceinline__ long long* item() const { return at<long long>(C::ITEM_OFFSET); }
        // [2]: entries of the list, by the step's parity; [2], [3]: those of the second list
        __device__ __forceinline__ int* count() const { return at<int>(C::ITEM_OFFSET + 8); }
        // points with outputs whose sums are small: row TX + column | these << 9 | those below one unit << 12
        __device__ __forceinline__ unsigned short* list() const { return at<unsigned short>(C::LIST_OFFSET); }
        // outputs that FP64 evaluates: row TX + column | output << 9
        __device__ __forceinline__ unsigned short* list64() const { return list() + C::TX * C::TY; }
        // the work item's domain (persistent kernel)
        __device__ __forceinline__ int* args() const { return at<int>(C::ARGS_OFFSET); }
    };

    static __device__ __forceinline__ void setup(unsigned char* raw, Ring<Shape>& ring, Smem& sm) {
        ring.setup(raw);
        sm.base = ring.base;
    }

    // The same in functions of their own, found from the kernel's array so that the
    // compiler knows their accesses as shared ones.
    static __device__ __forceinline__ Smem here() {
        extern __shared__ unsigned char smem_raw[];
        Ring<Shape> ring;
        ring.setup(smem_raw);
        return Smem{ring.base};
    }

    // The ring's barrier, and one for each of a tile's first two levels.
    static __device__ __forceinline__ void init_barriers(Ring<Shape>& ring) {
        mbar_init(&ring.full[1], 1);
        mbar_init(&ring.full[2], 1);
        ring.init_barriers();
    }

    // Where a CTA stands: loads through the ring, and the phases of the two start
    // barriers.
    struct Counts {
        long long ring = 0;
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

    // Whether lower and upper coefficients are equal on every level.
    static __device__ __forceinline__ bool equal_coefs(const FwdArgs& a, int tid) {
        bool eq = true;
        auto same = [](double x, double y) {
            return __double2hiint(x) == __double2hiint(y) && __double2loint(x) == __double2loint(y);
        };
        for (int k = 1 + tid; k <= a.nz - 2; k += C::NT)
            eq &= same(__ldg(a.tzc1 + k), __ldg(a.tzc2 + k)) && same(__ldg(a.tzd1 + k), __ldg(a.tzd2 + k));
        return __syncthreads_and(eq) != 0;
    }

    // Offsets in a box of the thread's cells of a field, each of which is
    // row W + column, and whether it takes a third one of field f.
    struct Plan {
        int src[3];
    };

    static __device__ __forceinline__ int cell_of(int q, int tid) { return q < 2 ? tid + q * C::NT : 2 * C::NT + tid % C::HALF; }

    static __device__ __forceinline__ bool has_cell(int f, int q, int tid) {
        return q < 2 || ((f == 1) == (tid >= C::HALF) && tid % C::HALF < C::REST);
    }

    static __device__ __forceinline__ Plan make_plan(int tid) {
        Plan p;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int n = min(cell_of(q, tid), C::CELLS - 1);
            p.src[q] = n / C::W * C::BX + n % C::W;
        }
        return p;
    }

    // Coefficient n of level lev for lane n of warp 4 (the top level has no upper
    // ones).
    static __device__ __forceinline__ double coef_for(const FwdArgs& a, int lev, int tid) {
        const int n = tid - 128;
        if ((unsigned)n >= 4u || (n > 0 && lev == a.nz - 1)) return 0.0;
        const double* arr = n == 0 ? a.tzc1 : n == 1 ? a.tzc2 : n == 2 ? a.tzd1 : a.tzd2;
        return __ldg(arr + lev);
    }

    // Exponents of a step's windows, of the limbs of all three levels: u, v, w of
    // the advected fields, d of the advecting velocities times their coefficients
    // over tref.
    struct Scale {
        int u, v, w, d;
        __device__ __forceinline__ int field(int f) const { return f == 0 ? u : f == 1 ? v : w; }
    };
    static __device__ __forceinline__ Scale scale(Smem sm) {
        const int4 t = sm.scale()[0];
        return {t.x, t.y, t.z, t.w};
    }
    static constexpr int kNone = 1 << 20;      // d where no windows hold the values
    static constexpr int kMostExp = 307, kLeastExp = -289;  // (the results' exponents stay normal)
    static constexpr int kZero = -1022, kUnset = -5000;  // sm.top() of fields of zeros, or less; of levels not there
    // u and v take the window of d up to this many binades above their own. (Their
    // largest products are then still 2^38 units.)
    static constexpr int kSlack = 8;
    static constexpr unsigned kPlain = 8u;  // u = v = d and tcx = tcy: horizontal products are added as they are

    // c 2^up as a limb number, |c 2^up| < 4.
    static __device__ __forceinline__ int4 coef_limbs(double c, int up, bool negative) {
        const double x = __dmul_rn(c, __hiloint2double((1023 + up) << 20, 0));
        Limb3 v;
        if (!limb_split<31>(x, 2, &v)) (void)limb_split_cut<31>(x, 2, &v);
        return negative ? make_int4(-v.h, -v.m, -v.l, 0) : make_int4(v.h, v.m, v.l, 0);
    }

    // Lanes 0..3 of warp 4 hand level lev's coefficients to the CTA; kLimbs: as limbs
    // at the limbs' scale, too.
    template <bool kLimbs>
    static __device__ __forceinline__ void store_coefs(Smem sm, const FwdArgs& a, int lev, double coef, int tid) {
        const int n = tid - 128;
        if ((unsigned)n >= 4u) return;
        const double r = __dmul_rn(coef, a.tinv);
        const int hi = __double2hiint(r) & 0x7FFFFFFF;
        const int e = __reduce_max_sync(0xFu, (hi | __double2loint(r)) == 0 ? -4096 : (hi >> 20) - 1023);
        sm.raw()[(lev & 3) * 4 + n] = r;
        if (kLimbs) {
            const Scale z = scale(sm);
            sm.coef()[(lev & 3) * 4 + n] = coef_limbs(r, z.w - z.d, n & 1);
        }
        if (n == 0) sm.cexp()[lev & 3] = max(e, -64);
    }

    // Exponent of a field's largest magnitude in a box (|x| < 2^it), of the first
    // levels of a tile.
    static __device__ __forceinline__ void scan_level(const double* box, Smem sm, int lev, int tid, const Plan& p) {
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            int mag = 0;
            unsigned low = 0;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (!has_cell(f, q, tid)) continue;
                const double x = box[f * (Shape::BOX_STRIDE / 8) + p.src[q]];
                mag = max(mag, __double2hiint(x) & 0x7FFFFFFF);
                low |= (unsigned)__double2loint(x);
            }
            const bool lowest = __any_sync(0xffffffffu, low != 0u);
            mag = __reduce_max_sync(0xffffffffu, mag);
            const int e = mag >> 20;
            if ((tid & 31) == 0) atomicMax(&sm.top()[lev & 3].x + f, e == 0 && (mag != 0 || lowest) ? kZero + 1 : e - 1022);
        }
    }

    // A thread's cells of a box whose values lie below their window, cut to its
    // unit (the cell's last word: something was cut).
    static __device__ __noinline__ void split_cut(const double* box, int4* out, int* top, Scale z, int tid, int3 src) {
#pragma unroll 1
        for (int f = 0; f < 3; ++f) {
            const int E = z.field(f);
            double x[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) x[q] = has_cell(f, q, tid) ? box[f * (Shape::BOX_STRIDE / 8) + (q == 0 ? src.x : q == 1 ? src.y : src.z)] : 0.0;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int hi = __double2hiint(x[q]) & 0x7FFFFFFF;
                if (E + 1022 - (hi >> 20) < kLimbWindow || (hi | __double2loint(x[q])) == 0) continue;
                Limb3 v;
                const bool cut = limb_split_low(x[q], E, &v);
                out[f * C::CELLS + cell_of(q, tid)] = make_int4(v.h, v.m, v.l, cut ? 1 : 0);
                if (hi < 0x00100000) atomicMax(top + f, kZero + 1);  // (a subnormal is no zero)
            }
        }
    }

    // Split the staged boxes of level lev into limb slot `slot` at scale z; kTops:
    // and find the largest magnitude of each field.
    template <bool kTops>
    static __device__ __forceinline__ void split_level(const double* box, Smem sm, int lev, int slot, Scale z,
                                                       int tid, const Plan& p) {
        int4* out = sm.limbs() + slot * C::SLOT;
        int* top = &sm.top()[lev & 3].x;
        bool ok = true;
        int depth[3];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            depth[f] = 4096;  // of the largest magnitude, below the window's top
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (!has_cell(f, q, tid)) continue;
                Limb3 v;
                int d;
                ok &= limb_split(box[f * (Shape::BOX_STRIDE / 8) + p.src[q]], z.field(f), &v, &d);
                out[f * C::CELLS + cell_of(q, tid)] = make_int4(v.h, v.m, v.l, 0);
                depth[f] = min(depth[f], d);
            }
        }
        if (kTops) {  // lane f hands on field f's
            const int lane = tid & 31;
            int e = z.u - __reduce_min_sync(0xffffffffu, depth[0]);
            const int ev = z.v - __reduce_min_sync(0xffffffffu, depth[1]), ew = z.w - __reduce_min_sync(0xffffffffu, depth[2]);
            if (lane == 1) e = ev;
            if (lane == 2) e = ew;
            if (lane < 3) atomicMax(top + lane, e);
        }
        if (!ok) split_cut(box, out, top, z, tid, make_int3(p.src[0], p.src[1], p.src[2]));
    }

    // Exponents of the largest magnitudes of u, v, w on the levels that step k reads.
    static __device__ __forceinline__ int3 tops(Smem sm, int k, bool top) {
        const int4 a = sm.top()[(k - 1) & 3], b = sm.top()[k & 3];
        int3 t = make_int3(max(a.x, b.x), max(a.y, b.y), max(a.z, b.z));
        if (!top) {
            const int4 c = sm.top()[(k + 1) & 3];
            t = make_int3(max(t.x, c.x), max(t.y, c.y), max(t.z, c.z));
        }
        return t;
    }

    // The windows of step k, from the largest magnitudes t of the levels that it
    // reads and the level's coefficients, and nothing else: a point's arithmetic
    // does not depend on the launch. te: exponents of tcx and tcy over tref. b:
    // that of the horizontal velocities; every other exponent is a multiple of 4
    // above or below it, so that fields times a power of two give the same bits,
    // scaled, and a window lasts for more than a few levels.
    static __device__ __forceinline__ int over(int b, int e) { return b + ((e - b + 3) & ~3); }

    // Whether they are those of the limbs: the common case, decided by ranges of t
    // and of the coefficients' exponent that store_scale left with the scale (every
    // thread of a step comes through here: 45 instructions in place of 25 cost 2 % of
    // a call).
    static __device__ __forceinline__ bool holds(Smem sm, int k, bool top) {
        const int3 t = tops(sm, k, top);
        const int4 p = sm.scale()[2], q = sm.scale()[3], r = sm.scale()[1];
        auto in = [](int e, int least, int more) { return static_cast<unsigned>(e - least) <= static_cast<unsigned>(more); };
        return max(t.x + r.x, t.y + r.y) == p.w && in(t.x, p.x, q.x) && in(t.y, p.y, q.y) &&
               in(t.z, p.z, q.z) && sm.cexp()[k & 3] >= q.w && sm.cexp()[k & 3] <= r.z;
    }

    // Scale z and the ranges for which it holds (one thread; b, flags: of scale_of).
    static __device__ __forceinline__ void store_scale(Smem sm, Scale z, int b, unsigned flags, int2 te) {
        constexpr int kAny = 1 << 20;
        const unsigned zero = ~flags;
        const bool plain = (flags & kPlain) != 0;
        // what holds d up beside w (a field of zeros does not)
        const int other = max(plain || (zero & 1u) ? b : z.u + te.x, plain || (zero & 2u) ? b : z.v + te.y);
        const bool nw = (zero & 4u) == 0;
        // a field of zeros stays one; u and v of a plain scale reach its slack; others stay in their window
        auto least = [&](unsigned f, int e) { return zero & f ? -kAny : e; };
        auto more = [&](unsigned f, int n) { return zero & f ? kAny + kZero : n; };
        sm.scale()[0] = make_int4(z.u, z.v, z.w, z.d);
        sm.scale()[1] = make_int4(te.x, te.y, nw ? z.d - z.w : kAny, (int)flags);
        sm.scale()[2] = make_int4(least(1u, plain ? z.d - kSlack - 3 : z.u - 3), least(2u, plain ? z.d - kSlack - 3 : z.v - 3),
                                least(4u, z.w - 3), b);
        sm.scale()[3] = make_int4(more(1u, plain ? kAny : 3), more(2u, plain ? kAny : 3), more(4u, 3),
                                !nw || z.d == b || other > z.d - 4 ? -kAny : z.d - 3 - z.w);
    }

    // *flags: bits of the fields that are not 0 on these levels, and kPlain. *base: b.
    static __device__ __noinline__ Scale scale_of(int3 t, int cexp, int2 te, bool same_t, unsigned* flags, int* base) {
        const bool nu = t.x > kZero, nv = t.y > kZero, nw = t.z > kZero;
        *flags = (nu ? 1u : 0u) | (nv ? 2u : 0u) | (nw ? 4u : 0u);
        int b = max(nu ? t.x + te.x : kUnset, nv ? t.y + te.y : kUnset);
        if (b == kUnset) b = nw ? t.z + cexp : kLimbExp;
        Scale z = {over(b, t.x), over(b, t.y), over(b, t.z), b};
        if (nu) z.d = max(z.d, z.u + te.x);
        if (nv) z.d = max(z.d, z.v + te.y);
        if (nw) z.d = max(z.d, z.w + cexp);
        z.d = over(b, z.d);
        // (a field far below the rest is left low in its window)
        z.u = nu ? max(z.u, z.d - 200) : z.d;
        z.v = nv ? max(z.v, z.d - 200) : z.d;
        z.w = nw ? max(z.w, z.d - 200) : z.d;
        if (same_t && (!nu || z.u >= z.d - kSlack) && (!nv || z.v >= z.d - kSlack)) {
            z.u = z.v = z.d;
            *flags |= kPlain;
        }
        if (max(z.d, max(max(z.u, z.v), z.w)) > kMostExp || z.d < kLeastExp) z.d = kNone;
        *base = nu || nv ? b : kUnset - 64;  // (holds goes by u and v)
        return z;
    }

    // Scale z for the limbs: the coefficients of levels k and k + 1 and of x and y.
    static __device__ __forceinline__ void rescale_coefs(Smem sm, const FwdArgs& a, int k, Scale z, int tid) {
        if (tid < 8) {
            const int s = ((k + tid / 4) & 3) * 4 + tid % 4;
            sm.coef()[s] = coef_limbs(sm.raw()[s], z.w - z.d, tid & 1);
        } else if (tid < 10) {
            sm.coef()[16 + tid - 8] = tid == 8 ? coef_limbs(__dmul_rn(a.tcx, a.tinv), z.u - z.d, false)
                                        : coef_limbs(__dmul_rn(a.tcy, a.tinv), z.v - z.d, false);
        }
    }

    // Step k's scale z differs from that of the limbs (cur): its levels' limbs in
    // the new windows. Cells that were cut, and levels that exceeded their window,
    // are split again from global memory (their boxes are gone). Every thread of
    // the CTA calls it, with no limb being read.
    static __device__ __noinline__ void rescale(const FwdArgs* args, int x0, int y0, int k, bool top,
                                                int3 slots, Scale z, int tid) {
        const Smem sm = here();
        const FwdArgs& a = *args;
        const Scale cur = scale(sm);
        for (int f = 0; f < 3; ++f) {
            const int from = cur.field(f), to = z.field(f), up = to - from;
            if (up == 0) continue;
            const double* g = static_cast<const double*>(f == 0 ? a.u : f == 1 ? a.v : a.w);
            for (int l = -1; l <= (top ? 0 : 1); ++l) {
                int4* out = sm.limbs() + (l < 0 ? slots.x : l == 0 ? slots.y : slots.z) * C::SLOT + f * C::CELLS;
                const bool again = (&sm.top()[(k + l) & 3].x)[f] > from || up < -95 || up > 95;
                int4 cell[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) cell[q] = has_cell(f, q, tid) ? out[cell_of(q, tid)] : make_int4(0, 0, 0, 0);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if (!has_cell(f, q, tid)) continue;
                    const int n = cell_of(q, tid);
                    const int4 t = cell[q];
                    Limb3 v;
                    bool cut;
                    if (again || t.w != 0) {
                        const int i = x0 + n % C::W, j = y0 + n / C::W;
                        const bool in = i <= a.nx + 1 && j <= a.ny + 1;
                        cut = limb_split_cut(in ? __ldg(g + (size_t)(k + l) * (size_t)a.sz + (size_t)j * (size_t)a.sy + i) : 0.0,
                                             to, &v);
                    } else {
                        v = limb_shift(Limb3{t.x, t.y, t.z}, up, &cut);
                    }
                    out[n] = make_int4(v.h, v.m, v.l, cut ? 1 : 0);
                }
            }
        }
        rescale_coefs(sm, a, k, z, tid);
    }

    struct Slot {
        const int4* p;
        __device__ __forceinline__ Limb3 operator()(int c) const {
            const int4 t = p[c];
            return {t.x, t.y, t.z};
        }
    };

    static __device__ __forceinline__ Limb3 rho(Smem sm, int lev, int n) {
        const int4 t = sm.coef()[(lev & 3) * 4 + n];
        return {t.x, t.y, t.z};
    }

    // X and Y with their coefficients
    static __device__ __forceinline__ LimbSum join_xy(LimbSum x, LimbSum y, Smem sm) {
        const int4 p = sm.coef()[16], q = sm.coef()[17];
        LimbSum s = limb_zero();
        limb_mac_scaled(s, x, Limb3{p.x, p.y, p.z});
        limb_mac_scaled(s, y, Limb3{q.x, q.y, q.z});
        return s;
    }

    // s + rho1 lo + rho2 hi: lo and hi the products through the lower and the
    // upper face (hi negated in kEq, where both take rho1; -rho2 is stored).
    template <bool kEq, bool kTop>
    static __device__ __forceinline__ void add_z(LimbSum& s, Smem sm, int lev, int n, Limb3 qlo, Limb3 flo,
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
    // levels k-1, k and k+1, at scale z.
    template <bool kEq, bool kPlainSums, bool kTop>
    static __device__ __forceinline__ void limb_point(Smem sm, const int4* B, const int4* M, const int4* P, int lev,
                                                      double tref, double* r_su, double* r_sv, double* r_sw, uint3* mag) {
        constexpr int W = C::W, N = C::CELLS;
        const Slot U{M}, V{M + N}, Z{M + 2 * N}, U1{P}, V1{P + N}, Z1{P + 2 * N}, Ub{B}, Vb{B + N}, Zb{B + 2 * N};
        const Scale z = scale(sm);
        const int su_scale = z.d + z.u - 172, sv_scale = z.d + z.v - 172, sw_scale = z.d + z.w - 172;
        const Limb3 uc = U(0), vc = V(0), wc = Z(0), wb = Zb(0);
        const Limb3 none = {0, 0, 0};
        {
            const Limb3 uw = U(-1), ue = U(1);
            LimbSum x = limb_zero(), y = limb_zero();
            // (u(i-1) - u(i+1)) (u(i-1) + u(i) + u(i+1)) is the two x terms in one product
            limb_mac(x, limb_sub(uw, ue), limb_add(limb_add(uw, uc), ue));
            LimbSum& yy = kPlainSums ? x : y;
            limb_mac(yy, U(-W), limb_add(V(-W), V(1 - W)));
            limb_mac(yy, U(W), limb_neg_sum(vc, V(1)));
            LimbSum s = kPlainSums ? x : join_xy(x, y, sm);
            add_z<kEq, kTop>(s, sm, lev, 0, Ub(0), limb_add(wb, Zb(1)), kTop ? none : U1(0), limb_add(wc, Z(1)));
            limb_carry(s);
            *r_su = __dmul_rn(tref, limb_to_double(s, su_scale, &mag->x));
        }
        {
            const Limb3 vs = V(-W), vn = V(W);
            LimbSum x = limb_zero(), y = limb_zero();
            limb_mac(y, limb_sub(vs, vn), limb_add(limb_add(vs, vc), vn));
            LimbSum& xx = kPlainSums ? y : x;
            limb_mac(xx, V(-1), limb_add(U(-1), U(W - 1)));
            limb_mac(xx, V(1), limb_neg_sum(uc, U(W)));
            LimbSum s = kPlainSums ? y : join_xy(x, y, sm);
            add_z<kEq, kTop>(s, sm, lev, 0, Vb(0), limb_add(wb, Zb(W)), kTop ? none : V1(0), limb_add(wc, Z(W)));
            limb_carry(s);
            *r_sv = __dmul_rn(tref, limb_to_double(s, sv_scale, &mag->y));
        }
        *r_sw = 0.0;
        if constexpr (!kTop) {
            const Limb3 wu = Z1(0);
            LimbSum x = limb_zero(), y = limb_zero();
            LimbSum& yy = kPlainSums ? x : y;
            limb_mac(x, Z(-1), limb_add(U(-1), U1(-1)));
            limb_mac(x, Z(1), limb_neg_sum(uc, U1(0)));
            limb_mac(yy, Z(-W), limb_add(V(-W), V1(-W)));
            limb_mac(yy, Z(W), limb_neg_sum(vc, V1(0)));
            LimbSum s = kPlainSums ? x : join_xy(x, y, sm);
            add_z<kEq, false>(s, sm, lev, 2, wb, limb_add(wc, wb), wu, limb_add(wc, wu));
            limb_carry(s);
            *r_sw = __dmul_rn(tref, limb_to_double(s, sw_scale, &mag->z));
        }
    }

    // p a - q b in native FP64. (Products and sums of the native form are written
    // out, so that every kernel that it is compiled into rounds alike.)
    static __device__ __forceinline__ double diff(double p, double a, double q, double b) {
        return __fma_rn(p, a, -__dmul_rn(q, b));
    }

    // Output f of a point in native FP64, term by term, from global memory, and its
    // store (e: the point's offset in the fields, on level k).
    static __device__ __forceinline__ void native_inline(const FwdArgs& a, size_t e, int k, int f) {
        const size_t sy = (size_t)a.sy, sz = (size_t)a.sz;
        const double *U = static_cast<const double*>(a.u) + e, *V = static_cast<const double*>(a.v) + e;
        const double *Wl = static_cast<const double*>(a.w) + e;
        const bool top = k == a.nz - 1;
        const double wc = __ldg(Wl), wb = __ldg(Wl - sz), uc = __ldg(U), vc = __ldg(V);
        if (f == 2) {
            double sw = 0.0;
            if (!top) {
                const double *U1 = U + sz, *V1 = V + sz;
                const double w1 = __ldg(Wl + sz);
                sw = __dmul_rn(a.tcx, diff(__ldg(Wl - 1), __dadd_rn(__ldg(U - 1), __ldg(U1 - 1)), __ldg(Wl + 1),
                                           __dadd_rn(uc, __ldg(U1))));
                sw = __fma_rn(a.tcy, diff(__ldg(Wl - sy), __dadd_rn(__ldg(V - sy), __ldg(V1 - sy)), __ldg(Wl + sy),
                                          __dadd_rn(vc, __ldg(V1))), sw);
                sw = __fma_rn(__ldg(a.tzd1 + k), __dmul_rn(wb, __dadd_rn(wc, wb)), sw);
                sw = __fma_rn(-__ldg(a.tzd2 + k), __dmul_rn(w1, __dadd_rn(wc, w1)), sw);
            }
            static_cast<double*>(a.sw)[e] = sw;
            return;
        }
        // su and sv are mirror images: q along (o = 1 or sy) is its own velocity, p the other one across
        const bool x = f == 0;
        const double *q = x ? U : V, *p = x ? V : U;
        const size_t o = x ? 1 : sy, r = x ? sy : 1;  // strides along q's own direction and across
        const double qc = x ? uc : vc, pc = x ? vc : uc;
        const double ql = __ldg(q - o), qh = __ldg(q + o);
        double s = __dmul_rn(x ? a.tcx : a.tcy, diff(ql, __dadd_rn(qc, ql), qh, __dadd_rn(qc, qh)));
        s = __fma_rn(x ? a.tcy : a.tcx, diff(__ldg(q - r), __dadd_rn(__ldg(p - r), __ldg(p - r + o)), __ldg(q + r),
                                             __dadd_rn(pc, __ldg(p + o))), s);
        s = __fma_rn(__ldg(a.tzc1 + k), __dmul_rn(__ldg(q - sz), __dadd_rn(wb, __ldg(Wl - sz + o))), s);
        if (!top) s = __fma_rn(-__ldg(a.tzc2 + k), __dmul_rn(__ldg(q + sz), __dadd_rn(wc, __ldg(Wl + o))), s);
        static_cast<double*>(x ? a.su : a.sv)[e] = s;
    }

    static __device__ __noinline__ void native_output(const FwdArgs* args, size_t e, int k, int f) { native_inline(*args, e, k, f); }

    // Output f of a point in limbs once more, where the products cancel to less than
    // one unit: from the sum's lowest bits. (B, M, P: the point in the slots of levels
    // k-1, k and k+1. The general form serves all cases: on the top level the upper
    // coefficients are 0.)
    static __device__ __noinline__ double low_output(const int4* B, const int4* M, const int4* P, int lev, int f,
                                                     double tref) {
        const Smem sm = here();
        constexpr int W = C::W, N = C::CELLS;
        const Slot U{M}, V{M + N}, Z{M + 2 * N}, U1{P}, V1{P + N}, Q{M + f * N}, Q1{P + f * N}, Qb{B + f * N}, Zb{B + 2 * N};
        // twice the advecting velocities at the faces of the output's cell: lower and upper x, y, z
        const int ox = f == 0 ? 1 : 0, oy = f == 1 ? W : 0;  // the cell lies half a step along x or y
        LimbSum x = limb_zero(), y = limb_zero();
        if (f == 2) {
            limb_mac(x, Q(-1), limb_add(U(-1), U1(-1)));
            limb_mac(x, Q(1), limb_neg_sum(U(0), U1(0)));
            limb_mac(y, Q(-W), limb_add(V(-W), V1(-W)));
            limb_mac(y, Q(W), limb_neg_sum(V(0), V1(0)));
        } else {
            limb_mac(x, Q(-1), limb_add(U(-1), U(f == 0 ? 0 : W - 1)));
            limb_mac(x, Q(1), limb_neg_sum(U(0), U(f == 0 ? 1 : W)));
            limb_mac(y, Q(-W), limb_add(V(-W), V(f == 0 ? 1 - W : 0)));
            limb_mac(y, Q(W), limb_neg_sum(V(0), V(f == 0 ? 1 : W)));
        }
        LimbSum s = join_xy(x, y, sm);
        const Limb3 lower = f == 2 ? limb_add(Z(0), Zb(0)) : limb_add(Zb(0), Zb(ox + oy));
        const Limb3 upper = f == 2 ? limb_add(Z(0), Q1(0)) : limb_add(Z(0), Z(ox + oy));
        add_z<false, false>(s, sm, lev, f == 2 ? 2 : 0, Qb(0), lower, Q1(0), upper);
        limb_carry(s);
        const Scale z = scale(sm);
        const int unit = z.d + z.field(f) - 172;
        unsigned mag;
        const double r = limb_to_double(s, unit, &mag);
        return __dmul_rn(tref, mag == 0 ? limb_tiny(s, unit) : r);
    }

    // The listed outputs of step k: those whose limb sums came out small. Where the
    // magnitudes of their horizontal products, with their coefficients, reach 2^28
    // units, the sum stands, from its lowest bits where it is below one unit. It is
    // exactly 0 where all advected values are. The others are FP64's: if they are few,
    // at once, otherwise on a list of their own, for whole warps (late_outputs).
    // Returns whether there is one.
    static __device__ __noinline__ bool listed_outputs(const FwdArgs* args, int listed, int x0, int y0, int k, int* count,
                                                       int3 slots, int tid) {
        const Smem sm = here();
        constexpr int W = C::W, N = C::CELLS;
        const FwdArgs& a = *args;
        const bool top = k == a.nz - 1;
        const int4 z = sm.scale()[0], te = sm.scale()[1];
        const int sx = min(max(z.w - z.x - te.x, 0), 63), sy = min(max(z.w - z.y - te.y, 0), 63);
        const bool few = listed <= C::NT / 8;  // not worth another barrier
        // one output of a point each, neighbouring threads the same one
        for (int t = tid; t < 3 * listed; t += C::NT) {
            const int f = t < listed ? 0 : t < 2 * listed ? 1 : 2;
            const unsigned entry = sm.list()[t - f * listed], id = entry & 0x1FFu;
            if ((entry >> (9 + f) & 1u) == 0) continue;
            const int col = (int)(id % C::TX), row = (int)(id / C::TX), c = (row + 1) * W + col + 1;
            const int4 *B = sm.limbs() + slots.x * C::SLOT + c, *U = sm.limbs() + slots.y * C::SLOT + c, *V = U + N;
            const int4 *U1 = sm.limbs() + slots.z * C::SLOT + c, *V1 = U1 + N, *Q = U + f * N;
            long long x, y;
            if (f == 0) {
                x = limb_least(Q[-1].x, U[-1].x + U[0].x) + limb_least(Q[1].x, U[0].x + U[1].x);
                y = limb_least(Q[-W].x, V[-W].x + V[1 - W].x) + limb_least(Q[W].x, V[0].x + V[1].x);
            } else if (f == 1) {
                x = limb_least(Q[-1].x, U[-1].x + U[W - 1].x) + limb_least(Q[1].x, U[0].x + U[W].x);
                y = limb_least(Q[-W].x, V[-W].x + V[0].x) + limb_least(Q[W].x, V[0].x + V[W].x);
            } else {
                x = limb_least(Q[-1].x, U[-1].x + U1[-1].x) + limb_least(Q[1].x, U[0].x + U1[0].x);
                y = limb_least(Q[-W].x, V[-W].x + V1[-W].x) + limb_least(Q[W].x, V[0].x + V1[0].x);
            }
            auto zero = [](const int4& q) { return (q.x | q.y | q.z | q.w) == 0; };  // and nothing cut
            const size_t e = (size_t)k * (size_t)a.sz + (size_t)(y0 + 1 + row) * (size_t)a.sy + (size_t)(x0 + 1 + col);
            if (limb_settled(x, y, sx, sy)) {
                if (entry >> (12 + f) & 1u)
                    static_cast<double*>(f == 0 ? a.su : f == 1 ? a.sv : a.sw)[e] = low_output(B, U, U1, k, f, a.tref);
            } else if (!(zero(Q[-1]) && zero(Q[1]) && zero(Q[-W]) && zero(Q[W]) && zero(B[f * N]) && (top || zero(U1[f * N])))) {
                if (few) native_output(args, e, k, f);
                else sm.list64()[atomicAdd(count, 1)] = (unsigned short)(id | (unsigned)f << 9);
            }
        }
        __syncthreads();  // the limbs and the list are read
        return !few;
    }

    // The outputs of step k on the second list. They need no limbs, so they run with
    // the next step's points: the FP64 unit works beside the integer pipes of other
    // warps.
    static __device__ __noinline__ void late_outputs(const FwdArgs* args, int left, int x0, int y0, int k, int tid) {
        const Smem sm = here();
        const FwdArgs& a = *args;
#pragma unroll 2
        for (int q = tid; q < left; q += C::NT) {
            const int entry = sm.list64()[q], id = entry & 0x1FF;
            native_inline(a, (size_t)k * (size_t)a.sz + (size_t)(y0 + 1 + id / C::TX) * (size_t)a.sy +
                                 (size_t)(x0 + 1 + id % C::TX), k, entry >> 9);
        }
    }

    // Step k's windows where holds says that they are not those of the limbs: makes
    // them so. False where no windows hold the values. Every thread of the CTA calls
    // it.
    static __device__ __noinline__ bool change_scale(const FwdArgs* args, int x0, int y0, int k,
                                                         bool top, int3 slots, int tid) {
        const Smem sm = here();
        const int2 te = make_int2(sm.scale()[1].x, sm.scale()[1].y);
        unsigned flags;
        int base;
        const Scale z = scale_of(tops(sm, k, top), sm.cexp()[k & 3], te, args->same_t != 0, &flags, &base);
        if (z.d == kNone) return false;
        const Scale cur = scale(sm);
        const bool same = z.u == cur.u && z.v == cur.v && z.w == cur.w && z.d == cur.d;
        if (!same) rescale(args, x0, y0, k, top, slots, z, tid);
        __syncthreads();  // (every thread has read the scale)
        if (tid == 0) store_scale(sm, z, base, flags, te);
        __syncthreads();
        return true;
    }

    // One tile (bx, by) of domain `a`, output levels kb..ke-1 (a chunk of the
    // column; it reads one level below and one above), its first levels issued by
    // start_tile. Loads are numbered relative to the lowest level read, lo: 0 and
    // 1 come through the start barriers, the others through the ring. Returns
    // false if a bounded wait expired (status set, copies drained). args: `a` in
    // memory.
    template <bool kEq>
    static __device__ bool tile_impl(Ring<Shape>& ring, Smem sm, const CUtensorMap* mu, const CUtensorMap* mv,
                                     const CUtensorMap* mw, const FwdArgs& a, const FwdArgs* args, int bx, int by, int kb,
                                     int ke, Counts& count, int tid, const Plan& plan) {
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
        auto box = [&](int r) {
            return reinterpret_cast<const double*>(ring.base + (r == 0 ? C::RAW1 : r == 1 ? C::RAW2 : 0)) + a.xoff;
        };
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
        const int2 te = a.same_t ? make_int2(0, 0) : make_int2(-limb_binades(__dmul_rn(a.tcx, a.tinv)), -limb_binades(__dmul_rn(a.tcy, a.tinv)));

        const int c = (ty + 1) * C::W + tx + 1;  // the first point in a limb slot
        // relative levels 0..2 arrive together: their magnitudes give the first
        // step's scale, at which they are split; the step at r splits r+2
        bool bad = false;
        double coef[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) coef[r] = r < nl ? coef_for(a, lo + r, tid) : 0.0;
#pragma unroll
        for (int r = 0; r < 3; ++r)
            if (r < nl) store_coefs<false>(sm, a, lo + r, coef[r], tid);
        for (int r = 0; r < 3 && r < nl; ++r) bad |= !wait(r);
        if (tid < 4) sm.top()[tid] = make_int4(kUnset, kUnset, kUnset, 0);
        if (tid < 4) sm.count()[tid] = 0;
        bool abort = __syncthreads_or(bad);
        if (!abort && a.limbs && nl > 1) {
            for (int r = 0; r < 3 && r < nl; ++r) scan_level(box(r), sm, lo + r, tid, plan);
            __syncthreads();
            unsigned flags;
            int base;
            Scale z = scale_of(tops(sm, lo + 1, lo + 1 == nz - 1), sm.cexp()[(lo + 1) & 3], te, a.same_t != 0, &flags, &base);
            if (z.d == kNone) z = Scale{kLimbExp, kLimbExp, kLimbExp, kLimbExp}, base = kUnset - 64;
            if (tid == 0) store_scale(sm, z, base, flags, te);
            for (int r = 0; r < 3 && r < nl; ++r) {
                split_level<false>(box(r), sm, lo + r, r, z, tid, plan);
                if (r == 0) rescale_coefs(sm, a, lo + 1, z, tid);
                __syncthreads();
            }
        }
        if (!abort && tid == 0 && issued < nl) {  // the stage is free again
            fence_proxy_async_smem();
            ring.issue(ring_load(issued), lo + issued, mu, mv, mw, x0, y0);
            ++issued;
        }
        const int k1 = kb > 1 ? kb : 1;  // first computed level (lo = k1 - 1)
        g += (size_t)(k1 - lo) * gsz;

        // Level k = lo + r from the limb slots of r-1, r and r+1 (sl, sc, sp);
        // level k+2 then goes into slot sl.
        bool late = false;  // the step before left outputs to late_outputs
        auto step = [&](auto top, int sl, int sc, int sp, int r) {
            constexpr bool kTop = decltype(top)::value;
            const int k = lo + r;
            if (late) late_outputs(args, sm.count()[2 + ((r + 1) & 1)], x0, y0, k - 1, tid);
            late = false;
            if (!kTop && tid == 0) sm.count()[(r + 1) & 1] = 0;  // (read in the step before)
            bool limbs = a.limbs;
            if (limbs && !holds(sm, k, kTop)) {
                limbs = change_scale(args, x0, y0, k, kTop, make_int3(sl, sc, sp), tid);
            }
            const int4* B = sm.limbs() + sl * C::SLOT + c;
            const int4* M = sm.limbs() + sc * C::SLOT + c;
            const int4* P = sm.limbs() + sp * C::SLOT + c;
            size_t e = g;
            // (two loops, so that the common one has the registers to itself)
            auto points = [&](auto plain) {
#pragma unroll 1
                for (int n = 0; n < act; ++n) {
                    double r_su, r_sv, r_sw;
                    uint3 mag;
                    limb_point<kEq, decltype(plain)::value, kTop>(sm, B, M, P, k, a.tref, &r_su, &r_sv, &r_sw, &mag);
                    su[e] = r_su;
                    sv[e] = r_sv;
                    sw[e] = r_sw;
                    const Scale z = scale(sm);
                    unsigned small = (limb_small(mag.x, z.d + z.u - 172) ? 1u : 0u) | (limb_small(mag.y, z.d + z.v - 172) ? 2u : 0u);
                    if (!kTop) small |= limb_small(mag.z, z.d + z.w - 172) ? 4u : 0u;
                    // (a field of zeros has outputs of exactly 0)
                    if (small != 0 && (small &= (unsigned)sm.scale()[1].w) != 0) {
                        const unsigned none = (mag.x == 0 ? 1u : 0u) | (mag.y == 0 ? 2u : 0u) | (mag.z == 0 ? 4u : 0u);
                        sm.list()[atomicAdd(&sm.count()[r & 1], 1)] = (unsigned short)((unsigned)(n * C::NT + tid) | small << 9 | none << 12);
                    }
                    B += C::ROWS * C::W;
                    M += C::ROWS * C::W;
                    P += C::ROWS * C::W;
                    e += grow;
                }
            };
            if (!limbs) {
                for (int n = 0; n < 3 * act; ++n) native_output(args, e + n / 3 * grow, k, n % 3);
            } else if ((sm.scale()[1].w & kPlain) != 0) {
                points(std::true_type());
            } else {
                points(std::false_type());
            }
            g += gsz;
            __syncthreads();  // level k-1's limbs are free, the list is complete
            const int listed = sm.count()[r & 1];
            if (listed != 0) late = listed_outputs(args, listed, x0, y0, k, &sm.count()[2 + (r & 1)], make_int3(sl, sc, sp), tid);
            if (tid == 0) sm.count()[2 + ((r + 1) & 1)] = 0;  // (read at this step's start)
            if (kTop) return;
            if (r + 2 < nl) {
                if (tid == 0) sm.top()[(k + 3) & 3] = make_int4(kUnset, kUnset, kUnset, 0);  // (level k-1's: read no more)
                const double coef = coef_for(a, k + 2, tid);
                bad |= !ring.wait(ring_load(r + 2));
                if (a.limbs) {
                    const Scale z = scale(sm);
                    split_level<true>(box(r + 2), sm, k + 2, sl, z, tid, plan);
                    store_coefs<true>(sm, a, k + 2, coef, tid);
                }
                abort = __syncthreads_or(bad);  // publishes level k+2's limbs, frees its stage
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
        if (late) late_outputs(args, sm.count()[2 + ((ke - 1 - lo) & 1)], x0, y0, ke - 1, tid);
        if (abort) {
            if (tid == 0) {
                atomicOr(&tu_status, kStatusTimeout);
                for (int q = 0; q < issued; ++q)
                    if (q < 2 || q == issued - 1) (void)wait(q);
            }
            return false;
        }
        __syncthreads();  // every read of this tile's stages and limbs is done before the next tile's
        count.ring += max(nl - 2, 0);
        count.phase1 += 1;
        count.phase2 += nl > 1 ? 1 : 0;
        return true;
    }

    static __device__ bool tile(Ring<Shape>& ring, Smem sm, const CUtensorMap* mu, const CUtensorMap* mv,
                                const CUtensorMap* mw, const FwdArgs& a, const FwdArgs* args, int bx, int by, int kb,
                                int ke, Counts& count, int tid, const Plan& plan) {
        if (tid == 0) start_tile(ring, mu, mv, mw, a, bx, by, kb, ke, count);  // (the scan runs while they arrive)
        if (equal_coefs(a, tid)) return tile_impl<true>(ring, sm, mu, mv, mw, a, args, bx, by, kb, ke, count, tid, plan);
        return tile_impl<false>(ring, sm, mu, mv, mw, a, args, bx, by, kb, ke, count, tid, plan);
    }
};

template <class C>
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
    __syncthreads();
    typename K::Counts count;
    int bx, by, k0, k1;
    sched_item(sched, a.kend - a.kbeg, blockIdx.x, &bx, &by, &k0, &k1);
    const typename K::Plan plan = K::make_plan(tid);
    (void)K::tile(ring, sm, &mu, &mv, &mw, a, &a, bx, by, a.kbeg + k0, a.kbeg + k1, count, tid,
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
    __syncthreads();
    const long long n_items = plan->n_items;
    const typename K::Plan split = K::make_plan(tid);
    typename K::Counts count;
    for (long long it = 0; it < n_items; ++it) {
        if (tid == 0) *sm.item() = (long long)atomicAdd(&plan->counter, 1ull);
        __syncthreads();
        const long long item = *sm.item();
        __syncthreads();  // every thread has read the slot before thread 0 rewrites it
        if (item >= n_items) break;
        const BatchDomain& d = plan->dom[find_domain(plan, item)];
        // The arguments in shared memory: the plan is global memory that the compiler
        // cannot prove free of the output stores, and a private copy took registers
        // from the march.
        if (tid < (int)(sizeof(FwdArgs) / 4)) sm.args()[tid] = reinterpret_cast<const int*>(&d.args)[tid];
        __syncthreads();
        const FwdArgs& args = *reinterpret_cast<const FwdArgs*>(sm.args());
        const long long t = item - d.first_item;
        const int tiles_x = d.tiles_x, kchunks = d.kchunks;
        const long long tiles = (long long)tiles_x * d.tiles_y;
        const int ch = (int)(t / tiles), tt = (int)(t % tiles);
        const int kb = (int)((long long)args.nz * ch / kchunks);
        const int ke = (int)((long long)args.nz * (ch + 1) / kchunks);
        const int bx = tt % tiles_x, by = tt / tiles_x;
        const bool go = K::tile(ring, sm, &d.mu, &d.mv, &d.mw, args, &args, bx, by, kb, ke, count, tid, split);
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
    auto kern = fwd_f64_kernel<C>;
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
