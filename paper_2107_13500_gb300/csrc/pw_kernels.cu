// pw_kernels.cu -- helper kernels of the PW advection library: periodic halo
// fill, the per-level mean/perturbation split, the bounded-wait self-test
// and the device status word. The forward kernels live in pw_f64.cu (FP64, in
// fixed point), pw_paired.cu (paired FP32) and pw_split.cu (FP32); the adjoint in
// pw_adjoint.cu and pw_adjoint_f64.cu.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pw_common.cuh"
#include "pw_dadd.cuh"
#include "pw_internal.h"
#include "pw_pair.cuh"
#include "pw_ring.cuh"

namespace pw {


// ---------------------------------------------------------------------------
// Periodic halo fill: x halo on rows 1..ny, then the full rows 0 and ny+1.

template <typename T>
__global__ void fill_halo_x_kernel(T* f, int nx, int ny, int nz, long long sy, long long sz) {
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;  // row id over (k, j)
    if (r >= (long long)nz * ny) return;
    const int k = (int)(r / ny), j = 1 + (int)(r % ny);
    T* row = f + (size_t)k * (size_t)sz + (size_t)j * (size_t)sy;
    row[0] = row[nx];
    row[nx + 1] = row[1];
}

template <typename T>
__global__ void fill_halo_y_kernel(T* f, int nx, int ny, int nz, long long sy, long long sz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = blockIdx.y;
    if (i > nx + 1) return;
    T* lev = f + (size_t)k * (size_t)sz;
    lev[i] = lev[(size_t)ny * (size_t)sy + i];
    lev[(size_t)(ny + 1) * (size_t)sy + i] = lev[(size_t)sy + i];
}

cudaError_t launch_fill_halo(void* field, int elem_bytes, int nx, int ny, int nz, long long sy, long long sz,
                             cudaStream_t st) {
    const long long rows = (long long)nz * ny;
    const unsigned gx = (unsigned)((rows + 255) / 256);
    dim3 gy((nx + 2 + 255) / 256, nz);
    if (elem_bytes == 8) {
        fill_halo_x_kernel<double><<<gx, 256, 0, st>>>(static_cast<double*>(field), nx, ny, nz, sy, sz);
        fill_halo_y_kernel<double><<<gy, 256, 0, st>>>(static_cast<double*>(field), nx, ny, nz, sy, sz);
    } else {
        fill_halo_x_kernel<float><<<gx, 256, 0, st>>>(static_cast<float*>(field), nx, ny, nz, sy, sz);
        fill_halo_y_kernel<float><<<gy, 256, 0, st>>>(static_cast<float*>(field), nx, ny, nz, sy, sz);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// One forward-Euler update of three periodic fields, and its transpose.
//
// Both are one pass over HBM, out of place: update reads f and s and writes
// f + dt s with its periodic halo (24 B a cell in FP64); the transpose reads g
// and writes the folded gradient and dt times it (24 B). As separate
// operations (a product, a sum, a zero fill, a copy and two halo launches per
// field) the same values took 80 B a cell and more, and the copies ran between
// buffers 8 bytes apart modulo 16.
// A halo cell takes the value of the interior cell that it stands for, which
// its thread evaluates again: no cell depends on another thread's store, so
// one launch covers all three fields. A thread owns one column of kStepRows
// rows and keeps all their loads in flight. Bound by HBM: three 256x256x64
// FP64 fields (302 MB) take 60 us (update) and 62 us (transpose), 5 TB/s; the
// launches they replace took about 118 and 150 us, and the device copies
// between differently aligned buffers more than both. (Rows and columns numbered flat
// over the CTAs, without the partly empty CTAs at the ends of rows: 62 and 71
// us; warps that straddle rows store in more pieces.)

constexpr int kStepThreads = 128, kStepRows = 8;

struct StepArgs {
    const void* a[3];  // update: f; transpose: g
    const void* b[3];  // update: s
    void* o[3];        // update: f + dt s; transpose: folded g
    void* p[3];        // transpose: dt * folded g
};

__device__ __forceinline__ double step_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float step_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double step_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float step_add(float a, float b) { return __fadd_rn(a, b); }

// Interior index that the halo index n (0 or len + 1) stands for.
__device__ __forceinline__ int wrap_index(int n, int len) { return n == 0 ? len : n == len + 1 ? 1 : n; }

template <typename T>
__global__ void __launch_bounds__(kStepThreads)
    euler_update_kernel(const StepArgs q, T dt, int nx, int ny, int nz, int width, long long sy, long long sz) {
    const int i = blockIdx.x * kStepThreads + threadIdx.x;
    if (i >= width) return;
    const bool pad = i > nx + 1;  // row padding: copied as it is
    const int is = pad ? i : wrap_index(i, nx);
    for (long long m = blockIdx.z; m < 3ll * nz; m += gridDim.z) {
        const int n = (int)(m % 3), k = (int)(m / 3);
        const T* f = static_cast<const T*>(n == 0 ? q.a[0] : n == 1 ? q.a[1] : q.a[2]) + (size_t)k * (size_t)sz + is;
        const T* s = static_cast<const T*>(n == 0 ? q.b[0] : n == 1 ? q.b[1] : q.b[2]) + (size_t)k * (size_t)sz + is;
        T* o = static_cast<T*>(n == 0 ? q.o[0] : n == 1 ? q.o[1] : q.o[2]) + (size_t)k * (size_t)sz + i;
        for (int j0 = blockIdx.y * kStepRows; j0 < ny + 2; j0 += gridDim.y * kStepRows) {
            T x[kStepRows], y[kStepRows];
#pragma unroll
            for (int r = 0; r < kStepRows; ++r) {
                const int j = j0 + r;
                if (j >= ny + 2) continue;
                const size_t e = (size_t)(pad ? j : wrap_index(j, ny)) * (size_t)sy;
                x[r] = __ldg(f + e);
                y[r] = pad ? T(0) : __ldg(s + e);
            }
#pragma unroll
            for (int r = 0; r < kStepRows; ++r)
                if (j0 + r < ny + 2) o[(size_t)(j0 + r) * (size_t)sy] = pad ? x[r] : step_add(x[r], step_mul(dt, y[r]));
        }
    }
}

// Column i of row j after the halo rows are folded (1 <= j <= ny).
template <typename T>
__device__ __forceinline__ T fold_rows(const T* g, int j, int ny, long long sy) {
    T y = __ldg(g + (size_t)j * (size_t)sy);
    if (j == ny) y = step_add(y, __ldg(g));
    if (j == 1) y = step_add(y, __ldg(g + (size_t)(ny + 1) * (size_t)sy));
    return y;
}

template <typename T>
__global__ void __launch_bounds__(kStepThreads)
    euler_update_adjoint_kernel(const StepArgs q, T dt, int nx, int ny, int nz, int width, long long sy, long long sz) {
    const int i = blockIdx.x * kStepThreads + threadIdx.x;
    if (i >= width) return;
    const bool pad = i > nx + 1, halo = i == 0 || i == nx + 1;
    for (long long m = blockIdx.z; m < 3ll * nz; m += gridDim.z) {
        const int n = (int)(m % 3), k = (int)(m / 3);
        const size_t lev = (size_t)k * (size_t)sz;
        const T* g = static_cast<const T*>(n == 0 ? q.a[0] : n == 1 ? q.a[1] : q.a[2]) + lev;
        T* o = static_cast<T*>(n == 0 ? q.o[0] : n == 1 ? q.o[1] : q.o[2]) + lev + i;
        T* p = static_cast<T*>(n == 0 ? q.p[0] : n == 1 ? q.p[1] : q.p[2]) + lev + i;
        for (int j0 = blockIdx.y * kStepRows; j0 < ny + 2; j0 += gridDim.y * kStepRows) {
            T x[kStepRows];
#pragma unroll
            for (int r = 0; r < kStepRows; ++r) {
                const int j = j0 + r;
                x[r] = T(0);
                if (j >= ny + 2) continue;
                if (pad) x[r] = __ldg(g + (size_t)j * (size_t)sy + i);
                else if (!halo && j >= 1 && j <= ny) x[r] = fold_rows(g + i, j, ny, sy);
            }
            if (i == nx || i == 1) {  // the halo columns join, after their own rows were folded
#pragma unroll
                for (int r = 0; r < kStepRows; ++r) {
                    const int j = j0 + r;
                    if (j < 1 || j > ny) continue;
                    if (i == nx) x[r] = step_add(x[r], fold_rows(g, j, ny, sy));
                    if (i == 1) x[r] = step_add(x[r], fold_rows(g + nx + 1, j, ny, sy));
                }
            }
#pragma unroll
            for (int r = 0; r < kStepRows; ++r) {
                if (j0 + r >= ny + 2) continue;
                o[(size_t)(j0 + r) * (size_t)sy] = x[r];
                p[(size_t)(j0 + r) * (size_t)sy] = step_mul(x[r], dt);
            }
        }
    }
}

cudaError_t launch_euler_periodic(bool adjoint, int elem_bytes, const void* const* a3, const void* const* b3,
                                  double dt, int nx, int ny, int nz, int width, long long sy, long long sz,
                                  void* const* o3, void* const* p3, cudaStream_t st) {
    StepArgs q{};
    for (int n = 0; n < 3; ++n) {
        q.a[n] = a3[n];
        q.o[n] = o3[n];
        q.b[n] = adjoint ? nullptr : b3[n];
        q.p[n] = adjoint ? p3[n] : nullptr;
    }
    const int chunks = (ny + 2 + kStepRows - 1) / kStepRows;
    const long long planes = 3ll * nz;
    const dim3 grid((unsigned)((width + kStepThreads - 1) / kStepThreads), (unsigned)(chunks < 65535 ? chunks : 65535),
                    (unsigned)(planes < 65535 ? planes : 65535));
    if (elem_bytes == 8) {
        if (adjoint) euler_update_adjoint_kernel<double><<<grid, kStepThreads, 0, st>>>(q, dt, nx, ny, nz, width, sy, sz);
        else euler_update_kernel<double><<<grid, kStepThreads, 0, st>>>(q, dt, nx, ny, nz, width, sy, sz);
    } else {
        const float dtf = (float)dt;
        if (adjoint) euler_update_adjoint_kernel<float><<<grid, kStepThreads, 0, st>>>(q, dtf, nx, ny, nz, width, sy, sz);
        else euler_update_kernel<float><<<grid, kStepThreads, 0, st>>>(q, dtf, nx, ny, nz, width, sy, sz);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Per-level mean and float perturbation, in three launches that balance
// GB300's slow FP64 pipe (about two FP64 lane operations per clock per SM)
// against its FP32 and integer pipes.
//
// split_sum_kernel: a flat grid of CTAs, one per (row band, level): the
// interior of level k is cut into nbands bands of at most kSumRows rows.
// Each thread sums its share of a band (a fixed set of columns, rows in
// order): the first kSum64Rows rows of each column in FP64, the rest in
// paired FP32 -- each double split into a float pair by integer operations,
// pairs added with TwoSum, about 20 issue slots a value -- so that the FP64
// pipe and the FP32/integer pipes share the work; the FP64 part then joins
// the pair. A fixed shuffle tree per warp and the warps in order follow;
// thread 0 stores the band's pair and a flag (every pair-summed value and
// the FP64 part within the pairs' range) in three cells of the perturbation
// output's level k, which split_pert_kernel overwrites afterwards, so no
// scratch memory is needed.
//
// split_reduce_kernel: one CTA per level adds the band sums in a fixed
// order (lane l of the first warp the bands l, l+32, ... in turn, then a
// fixed shuffle tree), so the mean does not depend on scheduling. A level
// where a pair-summed value or an FP64 part lies outside [2^-60, 2^100)
// (zero excepted), or is infinite or NaN, is summed again wholly in FP64 by
// that CTA (a fixed order too), since float pairs cannot carry it.
//
// split_pert_kernel: a flat grid over every cell (halo included) writes
// float(f - mean[k]): one FP64 subtraction (one row in kPertRows by the
// exact integer adder of pw_dadd.cuh, so that the ALU shares the FP64
// pipe's load), then the round-to-nearest-even conversion to float by
// integer operations (the hardware conversion issues on the FP64 pipe too),
// which gives the hardware's result bit for bit; the values outside the
// normal float range take the hardware conversion. The
// levels are walked top down, the reverse of the mean pass, so the levels
// that pass read last are read again while they are still in L2.

#ifndef PW_SUM_THREADS
#define PW_SUM_THREADS 128
#endif
#ifndef PW_SUM_ROWS
#define PW_SUM_ROWS 16
#endif
#ifndef PW_SUM_F64_ROWS
#define PW_SUM_F64_ROWS 8
#endif
constexpr int kSumThreads = PW_SUM_THREADS, kSumRows = PW_SUM_ROWS;  // threads; rows per band at most (the loads in flight per column)
// Rows of each band summed in FP64 (the FP64 pipe is otherwise idle here)
// rather than in paired FP32 (about 20 issue slots per value).
constexpr int kSum64Rows = PW_SUM_F64_ROWS;
constexpr int kPertThreads = 128, kPertRows = 8;  // columns per CTA, rows per thread
// Rows of each kPertRows group whose subtraction runs on the integer ALU
// (exact binary64 addition of -mean) instead of the FP64 pipe: the two pipes
// then work side by side.
#ifndef PW_PERT_INT_ROWS
#define PW_PERT_INT_ROWS 1
#endif
constexpr int kPertIntRows = PW_PERT_INT_ROWS;

// Biased double exponents of the magnitudes the paired sum carries: [2^-60, 2^100).
constexpr unsigned kPairExpLo = 1023 - 60, kPairExpHi = 1023 + 100;

// The tests below read the two 32-bit words of a double and use integer
// operations only: written on the 64-bit pattern, the compiler may turn an
// exponent window or a zero test back into FP64 comparisons, which issue on
// the slow FP64 pipe.
__device__ __forceinline__ bool pair_summable(double x) {
    const unsigned hw = static_cast<unsigned>(__double2hiint(x)), lw = static_cast<unsigned>(__double2loint(x));
    const unsigned e = (hw >> 20) & 0x7FFu;
    return ((hw << 1) | lw) == 0 || (e - kPairExpLo < kPairExpHi - kPairExpLo);
}

// double -> float rounded to nearest even. Results in the normal float range
// and zeros by integer operations; everything else (float subnormals,
// overflow from below 2^128 excepted, infinities, NaN) by the hardware.
__device__ __forceinline__ float double_to_float_rn(double d) {
    const unsigned hi = static_cast<unsigned>(__double2hiint(d)), lo = static_cast<unsigned>(__double2loint(d));
    const unsigned e = (hi >> 20) & 0x7FFu;  // biased double exponent
    if (e - 897u < 254u) {                  // float exponent 1..254
        const unsigned m = __funnelshift_l(lo, hi, 3) & 0x7FFFFFu;  // the 23 fraction bits kept
        const unsigned rem = lo & 0x1FFFFFFFu;                       // the 29 dropped
        const unsigned inc = (rem > 0x10000000u) | ((rem == 0x10000000u) & (m & 1u));
        // a carry out of the fraction moves to the exponent (254 -> 255: infinity)
        return __uint_as_float((hi & 0x80000000u) | (((e - 896u) << 23) + m + inc));
    }
    if (((hi << 1) | lo) == 0) return __uint_as_float(hi & 0x80000000u);
    return __double2float_rn(d);
}

// Cell n (row-major over the (ny+2) x (nx+2) cells, halo included) of the
// perturbation output's level k: the band sums' scratch slots.
template <typename F>
__device__ __forceinline__ F* sum_slot(F* fp, long long psy, long long psz, int nx, int k, int n) {
    const int w = nx + 2, r = n / w, c = n - r * w;
    return fp + (size_t)k * (size_t)psz + (size_t)r * (size_t)psy + c;
}

// Programmatic dependent launch (see the comment above launch_split_field):
// pdl_trigger lets the next grid of the stream start once every CTA has called
// it, pdl_wait returns when the grid before has completed and its stores are
// visible.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__global__ void __launch_bounds__(kSumThreads)
    split_sum_kernel(const double* __restrict__ f, long long fsy, long long fsz, int nx, int ny, int nz, int nbands,
                     float* __restrict__ fp, long long psy, long long psz) {
    __shared__ float2 warp_part[kSumThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    pdl_trigger();
    // interior rows [r0, r1) of band b
    const int r0 = 1 + (int)((long long)ny * b / nbands);
    const int r1 = 1 + (int)((long long)ny * (b + 1) / nbands);
    for (int k = blockIdx.y; k < nz; k += gridDim.y) {
        const double* lev = f + (size_t)k * (size_t)fsz;
        pf s = {0.0f, 0.0f};
        double s64 = 0.0;  // the first kSum64Rows rows of each column, on the FP64 pipe
        bool ok = true;
        for (int i = 1 + tid; i <= nx; i += kSumThreads) {
            // rows advance by adding the stride: 64-bit integer products
            // would issue on the FP64 pipe
            // a band has at most kSumRows rows: all its loads in flight at once
            const double* p = lev + i + (size_t)r0 * (size_t)fsy;
            double x[kSumRows];
#pragma unroll
            for (int q = 0; q < kSumRows; ++q) {
                x[q] = (r0 + q < r1) ? __ldg(p) : 0.0;
                p += fsy;
            }
#pragma unroll
            for (int q = 0; q < kSumRows; ++q) {
                if (q < kSum64Rows) {
                    s64 = __dadd_rn(s64, x[q]);  // rows past the band add zeros
                } else if (r0 + q < r1) {
                    ok &= pair_summable(x[q]);
                    s = padd(s, split_double(x[q]));
                }
            }
        }
        // the FP64 part joins the pair sum (it must lie in the pairs' range)
        ok &= pair_summable(s64);
        s = padd(s, split_double(s64));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const pf t = {__shfl_xor_sync(0xffffffffu, s.h, o), __shfl_xor_sync(0xffffffffu, s.l, o)};
            s = padd(s, t);
        }
        if (lane == 0) warp_part[warp] = make_float2(s.h, s.l);
        const int all_ok = __syncthreads_and(ok);
        if (tid == 0) {
            pf t = {0.0f, 0.0f};
            for (int q = 0; q < kSumThreads / 32; ++q) t = padd(t, pf{warp_part[q].x, warp_part[q].y});
            *sum_slot(fp, psy, psz, nx, k, 3 * b) = t.h;
            *sum_slot(fp, psy, psz, nx, k, 3 * b + 1) = t.l;
            *sum_slot(fp, psy, psz, nx, k, 3 * b + 2) = __int_as_float(all_ok);
        }
        __syncthreads();  // warp_part is rewritten for the next level
    }
}

__global__ void __launch_bounds__(kSumThreads)
    split_reduce_kernel(const double* __restrict__ f, long long fsy, long long fsz, int nx, int ny, int nz, int nbands,
                        const float* __restrict__ fp, long long psy, long long psz, double* __restrict__ mean) {
    __shared__ double warp_part64[kSumThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_trigger();
    pdl_wait();
    // the slots were written while this grid was already starting: read from L2
    for (int k = blockIdx.x; k < nz; k += gridDim.x) {
        bool ok = true;
        for (int b = tid; b < nbands; b += kSumThreads) ok &= __float_as_int(__ldcg(sum_slot(fp, psy, psz, nx, k, 3 * b + 2))) != 0;
        if (__syncthreads_and(ok)) {
            if (warp == 0) {
                // lane l adds bands l, l+32, ... in order, then a fixed tree
                pf t = {0.0f, 0.0f};
                for (int b = lane; b < nbands; b += 32)
                    t = padd(t, pf{__ldcg(sum_slot(fp, psy, psz, nx, k, 3 * b)), __ldcg(sum_slot(fp, psy, psz, nx, k, 3 * b + 1))});
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const pf u = {__shfl_xor_sync(0xffffffffu, t.h, o), __shfl_xor_sync(0xffffffffu, t.l, o)};
                    t = padd(t, u);
                }
                if (lane == 0) mean[k] = ((double)t.h + (double)t.l) / ((double)nx * (double)ny);
            }
        } else {
            // values the pairs cannot carry: the level in FP64, columns
            // strided over the threads, rows in order, warps in order
            const double* lev = f + (size_t)k * (size_t)fsz;
            double s64 = 0.0;
            for (int i = 1 + tid; i <= nx; i += kSumThreads) {
                const double* p = lev + i + (size_t)fsy;
                for (int j = 1; j <= ny; ++j, p += fsy) s64 += __ldg(p);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s64 += __shfl_xor_sync(0xffffffffu, s64, o);
            if (lane == 0) warp_part64[warp] = s64;
            __syncthreads();
            if (tid == 0) {
                double t = 0.0;
                for (int q = 0; q < kSumThreads / 32; ++q) t += warp_part64[q];
                mean[k] = t / ((double)nx * (double)ny);
            }
        }
        __syncthreads();  // warp_part64 and the flags are read before the next level
    }
}

// The FP64 subtraction for lanes dadd_int refused, out of line so that the
// common path carries no FP64 instruction.
__device__ __noinline__ double dsub_refused(double x, double m, double d, bool ok) {
    return ok ? d : __dsub_rn(x, m);
}

// Thread x of CTA (bx, by, bz) converts column bx*kPertThreads + x of the
// row chunks by, by + gridDim.y, ... (kPertRows rows each) of levels
// nz-1-bz, nz-1-bz-gridDim.z, ... (top down).
__global__ void __launch_bounds__(kPertThreads)
    split_pert_kernel(const double* __restrict__ f, long long fsy, long long fsz, float* __restrict__ fp,
                      long long psy, long long psz, int nx, int ny, int nz, const double* __restrict__ mean) {
    const int i = blockIdx.x * kPertThreads + threadIdx.x;
    if (i > nx + 1) return;
    bool ready = false;  // the means are there, and the band sums read
    for (int k = nz - 1 - (int)blockIdx.z; k >= 0; k -= (int)gridDim.z) {
        for (int j0 = blockIdx.y * kPertRows; j0 < ny + 2; j0 += gridDim.y * kPertRows) {
            const double* col = f + (size_t)k * (size_t)fsz + (size_t)j0 * (size_t)fsy + i;
            float* ocol = fp + (size_t)k * (size_t)psz + (size_t)j0 * (size_t)psy + i;
            const int nr = min(kPertRows, ny + 2 - j0);
            if (nr == kPertRows) {
                double x[kPertRows];
#pragma unroll
                for (int q = 0; q < kPertRows; ++q) {
                    x[q] = __ldg(col);
                    col += fsy;
                }
                if (!ready) pdl_wait();
                ready = true;
                const double m = __ldcg(mean + k);
                const double neg_m = __hiloint2double(__double2hiint(m) ^ (int)0x80000000, __double2loint(m));
#pragma unroll
                for (int q = 0; q < kPertRows; ++q) {
                    double d;
                    if (q < kPertIntRows) {
                        // the same difference on the integer ALU; the FP64
                        // unit only for the lanes it refuses
                        const bool ok = dadd_int(x[q], neg_m, &d);
                        if (__any_sync(__activemask(), !ok)) d = dsub_refused(x[q], m, d, ok);
                    } else {
                        d = __dsub_rn(x[q], m);
                    }
                    *ocol = double_to_float_rn(d);
                    ocol += psy;
                }
            } else {
                if (!ready) pdl_wait();
                ready = true;
                const double m = __ldcg(mean + k);
                for (int q = 0; q < nr; ++q, col += fsy, ocol += psy) *ocol = double_to_float_rn(__dsub_rn(__ldg(col), m));
            }
        }
    }
}

// A launch that may start before the grid ahead of it in the stream ends.
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t st, A... args) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// The second and third launch start as soon as every CTA of the one before has
// started: the reduction's launch and the first loads of the perturbation pass
// (of f, which no kernel here writes) fall into the end of the sum pass.
// Everything that an earlier kernel wrote, and every store, comes after
// pdl_wait; each grid waits for the one before it, so the third has the first
// behind it too. What it hides is the reduction's latency (5 us of one CTA per
// level) and two launches. Per field: 512x512x64 72.2 -> 67.5 us, 1000x250x37
// 49.6 -> 44.4, 64x64x64 15.9 -> 12.4; 1024x1024x128, where DRAM is the bound,
// 424.6 and 425.4.
cudaError_t launch_split_field(const double* f, long long fsy, long long fsz, float* fp, long long psy,
                               long long psz, int nx, int ny, int nz, double* mean, cudaStream_t st) {
    const unsigned gz = (unsigned)(nz < 65535 ? nz : 65535);  // grid y/z limit; the kernels loop over levels
    // bands of at most kSumRows rows; their 3 scratch cells per band fit in
    // a level of the output (3 ceil(ny/kSumRows) <= 3 ny < (ny+2)(nx+2))
    const int nbands = (ny + kSumRows - 1) / kSumRows;
    split_sum_kernel<<<dim3((unsigned)nbands, gz), kSumThreads, 0, st>>>(f, fsy, fsz, nx, ny, nz, nbands, fp, psy, psz);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_pdl(split_reduce_kernel, dim3(gz), kSumThreads, st, f, fsy, fsz, nx, ny, nz, nbands, fp, psy, psz, mean);
    if (e != cudaSuccess) return e;
    const int chunks = (ny + 2 + kPertRows - 1) / kPertRows;
    const dim3 grid((unsigned)((nx + 2 + kPertThreads - 1) / kPertThreads), (unsigned)(chunks < 65535 ? chunks : 65535),
                    gz);
    return launch_pdl(split_pert_kernel, grid, kPertThreads, st, f, fsy, fsz, fp, psy, psz, nx, ny, nz, mean);
}

// ---------------------------------------------------------------------------
// Energy budget: per level, the interior sums of u su, v sv, w sw and of their
// absolute values, in FP64 and in a fixed order, so the result does not depend
// on scheduling. A cluster of kBudgetCluster CTAs sums one (level, field):
// CTA r the r-th equal band of rows, each thread its columns in row order,
// then a fixed shuffle tree, the warps in order and the CTAs in order (through
// distributed shared memory, so no scratch memory is needed). A second
// single-CTA launch weights the level sums by the cell masses and adds them
// level by level.
//
// Bound by the FP64 pipe (two lane operations per clock per SM): each element
// costs two of them, a sum and a sum of magnitudes, both as FMAs that round
// the exact product into the running sum (a product, a sum and a sum of
// magnitudes took three). Float inputs are widened by integer operations; the
// hardware conversion, which issues on the FP64 pipe, serves only subnormals,
// infinities and NaN. One CTA per (level, field) left 192 CTAs of a 64-level
// domain on 152 SMs, so some SMs had twice the work of others; with clusters
// of 8 there are 1536. 512x512x64 FP64: 203 us (3.97 TB/s, FP64 pipe 89 %
// busy), 476 us before; with the totals 210 us a call, 487 before.

constexpr int kBudgetThreads = 256, kBudgetCluster = 8, kBudgetRows = 4;

__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x);
    const unsigned e = (b >> 23) & 0xFFu;
    if (e - 1u < 254u || (b << 1) == 0) return float_bits_to_double(x);
    return (double)x;
}

template <typename TW, typename TS>
__global__ void __cluster_dims__(kBudgetCluster, 1, 1) __launch_bounds__(kBudgetThreads)
    energy_level_kernel(const TW* __restrict__ u, const TW* __restrict__ v, const TW* __restrict__ w, long long wsy,
                        long long wsz, const TS* __restrict__ su, const TS* __restrict__ sv,
                        const TS* __restrict__ sw, long long ssy, long long ssz, int nx, int ny, int nz,
                        double* __restrict__ level_sums) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double part[2][kBudgetThreads / 32];
    __shared__ double cta_sum[2];
    const int rank = (int)blockIdx.x, k = blockIdx.y, f = blockIdx.z;  // the cluster spans the grid's x
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = 1 + (int)((long long)ny * rank / kBudgetCluster);
    const int j1 = 1 + (int)((long long)ny * (rank + 1) / kBudgetCluster);
    const TW* a = (f == 0 ? u : f == 1 ? v : w) + (size_t)k * (size_t)wsz + (size_t)j0 * (size_t)wsy;
    const TS* b = (f == 0 ? su : f == 1 ? sv : sw) + (size_t)k * (size_t)ssz + (size_t)j0 * (size_t)ssy;
    double s = 0.0, t = 0.0;
    // rows in groups whose loads are all in flight; rows advance by adding the stride
    for (int j = j0; j < j1; j += kBudgetRows, a += kBudgetRows * wsy, b += kBudgetRows * ssy) {
        for (int i = 1 + tid; i <= nx; i += kBudgetThreads) {
            TW x[kBudgetRows];
            TS y[kBudgetRows];
            const TW* pa = a + i;
            const TS* pb = b + i;
#pragma unroll
            for (int q = 0; q < kBudgetRows; ++q) {
                x[q] = j + q < j1 ? __ldg(pa) : TW(0);
                y[q] = j + q < j1 ? __ldg(pb) : TS(0);
                pa += wsy;
                pb += ssy;
            }
#pragma unroll
            for (int q = 0; q < kBudgetRows; ++q) {
                const double xd = widen(x[q]), yd = widen(y[q]);
                s = __fma_rn(xd, yd, s);
                t = __fma_rn(fabs(xd), fabs(yd), t);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    if (lane == 0) {
        part[0][warp] = s;
        part[1][warp] = t;
    }
    __syncthreads();
    if (tid < 2) {
        double r = 0.0;
        for (int q = 0; q < kBudgetThreads / 32; ++q) r += part[tid][q];
        cta_sum[tid] = r;
    }
    cluster.sync();
    if (rank == 0 && tid < 2) {
        double r = 0.0;
        for (int q = 0; q < kBudgetCluster; ++q) r += *cluster.map_shared_rank(&cta_sum[tid], q);
        level_sums[(size_t)k * 6 + f + 3 * tid] = r;
    }
    cluster.sync();  // no CTA leaves while its sums may still be read
}

// Totals: warp n adds column n of the level sums. Lane l holds level 32 m + l
// of group m (its loads in flight together); the products are then added level
// by level, as the single-thread loop over nz did, whose dependent loads took
// most of its 12.7 us at 64 levels.
__global__ void __launch_bounds__(192)
    energy_total_kernel(const double* __restrict__ level_sums, const double* __restrict__ wu,
                        const double* __restrict__ ww, int nz, double* __restrict__ totals) {
    const int n = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double* wt = (n % 3 == 2) ? ww : wu;
    double r = 0.0;
    for (int k0 = 0; k0 < nz; k0 += 32) {
        const int k = k0 + lane;
        const double x = k < nz ? wt[k] : 0.0, y = k < nz ? level_sums[(size_t)k * 6 + n] : 0.0;
        const int m = min(32, nz - k0);
        for (int q = 0; q < m; ++q) r += __shfl_sync(0xffffffffu, x, q) * __shfl_sync(0xffffffffu, y, q);
    }
    if (lane == 0) totals[n] = r;
}

template <typename TW, typename TS>
static cudaError_t launch_energy_t(const void* u, const void* v, const void* w, long long wsy, long long wsz,
                                   const void* su, const void* sv, const void* sw, long long ssy, long long ssz,
                                   int nx, int ny, int nz, const double* wu, const double* ww, double* level_sums,
                                   double* totals, cudaStream_t st) {
    energy_level_kernel<TW, TS><<<dim3(kBudgetCluster, (unsigned)nz, 3), kBudgetThreads, 0, st>>>(
        static_cast<const TW*>(u), static_cast<const TW*>(v), static_cast<const TW*>(w), wsy, wsz,
        static_cast<const TS*>(su), static_cast<const TS*>(sv), static_cast<const TS*>(sw), ssy, ssz, nx, ny, nz,
        level_sums);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    energy_total_kernel<<<1, 192, 0, st>>>(level_sums, wu, ww, nz, totals);
    return cudaGetLastError();
}

cudaError_t launch_energy_budget(const void* u, const void* v, const void* w, int wind_bytes, long long wsy,
                                 long long wsz, const void* su, const void* sv, const void* sw, int tend_bytes,
                                 long long ssy, long long ssz, int nx, int ny, int nz, const double* wu,
                                 const double* ww, double* level_sums, double* totals, cudaStream_t st) {
    if (wind_bytes == 8 && tend_bytes == 8)
        return launch_energy_t<double, double>(u, v, w, wsy, wsz, su, sv, sw, ssy, ssz, nx, ny, nz, wu, ww,
                                               level_sums, totals, st);
    if (wind_bytes == 8)
        return launch_energy_t<double, float>(u, v, w, wsy, wsz, su, sv, sw, ssy, ssz, nx, ny, nz, wu, ww,
                                              level_sums, totals, st);
    if (tend_bytes == 8)
        return launch_energy_t<float, double>(u, v, w, wsy, wsz, su, sv, sw, ssy, ssz, nx, ny, nz, wu, ww,
                                              level_sums, totals, st);
    return launch_energy_t<float, float>(u, v, w, wsy, wsz, su, sv, sw, ssy, ssz, nx, ny, nz, wu, ww, level_sums,
                                         totals, st);
}

// ---------------------------------------------------------------------------
// Self-test of the bounded wait: one thread waits on an mbarrier that nothing
// ever completes and must give up after limit_ns, recording a timeout.

__global__ void selftest_wait_kernel(unsigned long long limit_ns) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        if (!mbar_wait_bounded(&bar, 0, limit_ns)) atomicOr(&tu_status, kStatusTimeout);
    }
}

cudaError_t launch_selftest_wait(unsigned long long limit_ns, cudaStream_t st) {
    selftest_wait_kernel<<<1, 32, 0, st>>>(limit_ns);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------

cudaError_t read_and_clear_status(unsigned int* status, cudaStream_t st) {
    unsigned int parts[6] = {0, 0, 0, 0, 0, 0};
    cudaError_t e = read_and_clear_tu_status(&parts[0], st);
    if (e == cudaSuccess) e = read_and_clear_status_paired(&parts[1], st);
    if (e == cudaSuccess) e = read_and_clear_status_split(&parts[2], st);
    if (e == cudaSuccess) e = read_and_clear_status_adjoint(&parts[3], st);
    if (e == cudaSuccess) e = read_and_clear_status_f64(&parts[4], st);
    if (e == cudaSuccess) e = read_and_clear_status_adjoint_f64(&parts[5], st);
    *status = parts[0] | parts[1] | parts[2] | parts[3] | parts[4] | parts[5];
    return e;
}

}  // namespace pw
