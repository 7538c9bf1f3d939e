// Reduction of the discrete energy of the leapfrog scheme.
//
// With M = 1/(V dt)^2 and L the 25-point Laplacian (zero outside the grid),
// the recurrence of Eq. 2 without source or damping is
// M (u^{n+1} - 2 u^n + u^{n-1}) = L u^n; multiplying by u^{n+1} - u^{n-1}
// and summing over the grid telescopes (L is symmetric), so
//     E^{n-1/2} = sum (u^n - u^{n-1})^2 / (V dt)^2 - sum u^n (L u^{n-1})
// is the same for every n. The kernels evaluate it from the float fields: each
// block sums a fixed set of rows into one partial, and one block adds the
// partials in a fixed order, so the result does not depend on scheduling.
//
// GB300 runs FP64 at a 64th of its FP32 rate, and evaluated in FP64 (some 90
// operations and conversions a cell) the kernel was bound by that pipe: 3.7 ms
// at 320 x 288 x 256. Instead the parts of a cell's term are formed exactly, or
// to more than 53 bits, from floats and integers:
//  - 5040 h^2 L p = 8064 s1 - 1008 s2 + 128 s3 - 9 s4 - 43050 p, s_m the sum of the
//    six neighbours at distance m: whole weights, none is rounded. Each value is
//    cut at two places below the largest of the 25 by adding a constant (error-free
//    extraction, Rump, Ogita and Oishi): the sum's low bits are a whole number of
//    22 bits, its remainder is exact. Whole numbers are added and weighted as
//    integers, without error; the rest, below 2^-44 of the largest value, in floats.
//    One conversion makes an FP64 number of the 64-bit sum.
//  - (u - p)^2 / w as three floats, through error-free sums and products (Dekker,
//    Knuth) and the remainders of two quotients.
// A thread adds the first in FP64 and the second in three floats. So the sum is
// as precise as one of FP64 terms, also on a single cell and where neighbouring
// values differ by any factor. (As pairs of floats throughout, 48 bits, single
// cells and fields with spikes were off by up to 1e-14 of their parts; FP64: 3e-16
// to 1e-15.) About 400 instructions a cell, 3 of them FP64, bound by issue (62 % of
// its slots): ws_energy of 320 x 288 x 256 in 0.43 ms, without allocation 0.49 (the
// pairs: 0.36, 0.39; FP64 3.8).
// Where the block's largest value is not within 2^-30 .. 2^40, values are scaled by
// a power of two that brings it to about 1, so no product underflows that matters.
// Blocks out of the scaled range, and threads that meet a value that is not finite
// or a model outside 2^-60 .. 2^30, take the FP64 form.
#include "ws_model.cuh"
#include "ws_ptx.cuh"

namespace ws {
namespace {

constexpr int kThreads = 256;   // 8 warps, each a row at a time

// Scratch of the allocation-free entry point: the per-block partial sums,
// one array per device that loads the library, held until the process exits.
static __device__ __align__(256) double g_noalloc_partials[kNoAllocMaxPartials];

// u^n / u^{n-1} / (V dt / h)^2 of the handle's padded layout (halo is zero).
struct PaddedFields {
    const float *u, *p, *w;
    Geom g;
    __device__ long long at(int i, int j, int k) const { return pidx(g, i, j, k); }
    __device__ long long row() const { return g.pnx; }
    __device__ long long plane() const { return g.plane; }
    // p at offset o from cell e of the array; in: whether that is in the grid
    __device__ float p_near(long long e, long long o, bool) const { return p[e + o]; }
    __device__ float w_at(long long e) const { return w[e]; }
    __device__ bool surely_positive(long long e) const { return w[e] > 0.0f; }   // w_at, if true
};

// Unpadded [nz][ny][nx] caller arrays; (V dt / h)^2 is formed from the
// velocity exactly as the stepper stores it (double, rounded once to float),
// and cells outside the grid read as zero, so every cell's term is the one
// the padded variant computes.
struct DenseFields {
    const float *u, *p, *v;
    int nx, ny, nz;
    ModelScale scale;
    __device__ long long at(int i, int j, int k) const { return ((long long)k * ny + j) * nx + i; }
    __device__ long long row() const { return nx; }
    __device__ long long plane() const { return (long long)nx * ny; }
    __device__ float p_near(long long e, long long o, bool in) const { return in ? p[e + o] : 0.0f; }
    __device__ float w_at(long long e) const { return to_model<FromVelocity>(v[e], scale); }
    __device__ bool surely_positive(long long e) const { return fabsf(v[e] * scale.hi) >= 0x1p-60f; }
};

// hi + lo, exactly: the rounded result of a float operation and its error.
struct Pair {
    float hi, lo;
};
__device__ __forceinline__ Pair two_sum(float a, float b) {   // a + b exactly
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return Pair{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair two_prod(float a, float b) {   // a b exactly
    const float p = __fmul_rn(a, b);
    return Pair{p, __fmaf_rn(a, b, -p)};
}

// The values that a cell's term needs.
struct Cell {
    float u, p, w;
    float2 n[4][3];   // p at distance 1 .. 4 on {x+, x-}, {y+, y-}, {z+, z-}
};

// kInside: the y and z neighbours lie in the grid.
template <bool kInside, class F>
__device__ __forceinline__ Cell load_cell(const F &f, int i, int j, int k, int nx, int ny, int nz) {
    Cell c;
    const long long e = f.at(i, j, k), sy = f.row(), sz = f.plane();
    c.u = f.u[e];
    c.p = f.p[e];
    c.w = f.w_at(e);
#pragma unroll
    for (int m = 1; m <= 4; ++m) {
        c.n[m - 1][0] = make_float2(f.p_near(e, m, i + m < nx), f.p_near(e, -m, i - m >= 0));
        c.n[m - 1][1] = make_float2(f.p_near(e, m * sy, kInside || j + m < ny),
                                    f.p_near(e, -m * sy, kInside || j - m >= 0));
        c.n[m - 1][2] = make_float2(f.p_near(e, m * sz, kInside || k + m < nz),
                                    f.p_near(e, -m * sz, kInside || k - m >= 0));
    }
    return c;
}

// x in FP64, by integer operations (a conversion takes the FP64 pipe). Values
// below 2^-126 count as zero; x is finite.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    return __hiloint2double((int)(m < 0x800000u ? 0u : ((m >> 3) + 0x38000000u) | (b & 0x80000000u)),
                            (int)(m < 0x800000u ? 0u : b << 29));
}

// 5040 h^2 L p of a cell's values times s (a power of two; kScaled false: 1), the
// exact sum rounded to FP64: see the head of this file. *finite: false if one of
// the values is not.
template <bool kScaled>
__device__ __forceinline__ double stencil_sum(const Cell &c, float s, bool *finite) {
    auto value = [&](int m, int a) {   // m = 0: p itself
        const float2 v = m ? c.n[m - 1][a] : make_float2(c.p, 0.0f);
        return kScaled ? mul2(v, splat(s)) : v;
    };
    float big = fabsf(value(0, 0).x);
#pragma unroll
    for (int m = 1; m <= 4; ++m)
#pragma unroll
        for (int a = 0; a < 3; ++a) big = fmaxf(big, fmaxf(fabsf(value(m, a).x), fabsf(value(m, a).y)));
    // the largest value's exponent; not below 2^-60 (what is smaller is summed in
    // the last part), and an infinite one makes both constants NaN
    const int ex = max(127 - 60, min(253, (int)(__float_as_uint(big) >> 23)));
    const unsigned c1 = ((unsigned)(ex + 2) << 23) | 0x400000u, c2 = ((unsigned)(ex - 20) << 23) | 0x400000u;
    const float2 s1 = splat(__uint_as_float(c1)), s2 = splat(__uint_as_float(c2));
    const float2 m1 = splat(-s1.x), m2 = splat(-s2.x), minus = splat(-1.0f);
    constexpr int kWeight[5] = {-43050, 8064, -1008, 128, -9};
    long long sum1 = 0, sum2 = 0;
    float rest = 0.0f;
#pragma unroll
    for (int m = 0; m <= 4; ++m) {
        unsigned bits1 = 0u, bits2 = 0u;
        float2 r3 = splat(0.0f);
#pragma unroll
        for (int a = 0; a < (m ? 3 : 1); ++a) {
            const float2 v = value(m, a);
            const float2 t1 = add2(s1, v), r1 = fma2(add2(t1, m1), minus, v);     // v - (t1 - s1)
            const float2 t2 = add2(s2, r1), r2 = fma2(add2(t2, m2), minus, r1);   // likewise
            bits1 += __float_as_uint(t1.x) + __float_as_uint(t1.y);
            bits2 += __float_as_uint(t2.x) + __float_as_uint(t2.y);
            r3 = a ? add2(r3, r2) : r2;
        }
        const unsigned n = m ? 6u : 2u;   // (m = 0: p, and a zero)
        sum1 += (long long)kWeight[m] * (int)(bits1 - n * c1);
        sum2 += (long long)kWeight[m] * (int)(bits2 - n * c2);
        rest = __fmaf_rn((float)kWeight[m], __fadd_rn(r3.x, r3.y), rest);
    }
    const long long sum = (sum1 << 22) + sum2;   // below 2^62, in units of 2^(ex - 170)
    const double d = __ll2double_rn(sum);
    const int up = sum ? (ex - 170) * (1 << 20) : 0;   // times 2^(ex - 170), in its exponent
    *finite = fabsf(rest) < 0x1p126f;
    return __dadd_rn(__hiloint2double(__double2hiint(d) + up, __double2loint(d)), widen(rest));
}

// The sums of a thread's cells: kin[0] + kin[1] + kin[2] of (u - p)^2 / w (three
// floats, more than 70 bits), pot of 5040 u h^2 L p.
struct Sums {
    float kin[3] = {0.0f, 0.0f, 0.0f};
    double pot = 0.0;
    __device__ double kinetic() const {
        return __dadd_rn((double)kin[0], __dadd_rn((double)kin[1], (double)kin[2]));
    }
};

// Adds a cell, of the values times s; false if a stencil value is not finite.
template <bool kScaled>
__device__ __forceinline__ bool add_cell(const Cell &c, float s, Sums *sum) {
    const float u = kScaled ? c.u * s : c.u, p = kScaled ? c.p * s : c.p;
    bool finite;
    const double lap = stencil_sum<kScaled>(c, s, &finite);
    sum->pot = __fma_rn(widen(u), lap, sum->pot);
    // u - p = d exactly; (u - p)^2 = q.hi + e.hi + f
    const Pair d = two_sum(u, -p), q = two_prod(d.hi, d.hi), x = two_prod(2.0f * d.hi, d.lo);
    const Pair e = two_sum(q.lo, x.hi);
    const float f = __fmaf_rn(d.lo, d.lo, __fadd_rn(x.lo, e.lo));
    // the nearest quotient by w, its exact remainder, that one's quotient, and again
    const float a0 = __fdiv_rn(q.hi, c.w);
    const Pair r = two_sum(__fmaf_rn(-a0, c.w, q.hi), e.hi);
    const float a1 = __fdividef(r.hi, c.w);
    const float a2 = __fdividef(__fadd_rn(__fmaf_rn(-a1, c.w, r.hi), __fadd_rn(r.lo, f)), c.w);
    const Pair k0 = two_sum(sum->kin[0], a0), k1 = two_sum(sum->kin[1], k0.lo), k2 = two_sum(k1.hi, a1);
    sum->kin[0] = k0.hi;
    sum->kin[1] = k2.hi;
    sum->kin[2] = __fadd_rn(sum->kin[2], __fadd_rn(a2, __fadd_rn(k1.lo, k2.lo)));
    return finite;
}

// The term of one cell in FP64: (u - p)^2 / (V dt)^2 - u (L p), every
// operation explicitly rounded (no contraction left to the compiler), so each
// field layout gives the same bits.
__device__ __noinline__ double cell_fp64(const Cell &c, const Coeffs64 &w, double h2) {
    const double pc = c.p;
    double l[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        l[a] = __dmul_rn(w.c0, pc);
#pragma unroll
        for (int m = 1; m <= 4; ++m) {
            const double cm = m == 1 ? w.c1 : m == 2 ? w.c2 : m == 3 ? w.c3 : w.c4;
            l[a] = __fma_rn(cm, __dadd_rn((double)c.n[m - 1][a].x, (double)c.n[m - 1][a].y), l[a]);
        }
    }
    const double lap = __ddiv_rn(__dadd_rn(__dadd_rn(l[0], l[1]), l[2]), h2);
    const double uc = c.u;
    const double d = __dsub_rn(uc, pc);
    const double vdt2 = __dmul_rn((double)c.w, h2);   // (V dt)^2
    return __fma_rn(-uc, lap, __ddiv_rn(__dmul_rn(d, d), vdt2));
}

// This thread's cells of rows [j0, j1) of plane k, a warp a row at a time;
// false if one of them has a model or a value out of range.
template <bool kScaled, bool kInside, class F>
__device__ __forceinline__ bool sum_rows(const F &f, int j0, int j1, int k, int nx, int ny, int nz,
                                         float s, Sums *sum) {
    bool good = true;
    for (int j = j0 + (threadIdx.x >> 5); j < j1; j += kThreads / 32)
        for (int i = threadIdx.x & 31; i < nx; i += 32) {
            const Cell q = load_cell<kInside>(f, i, j, k, nx, ny, nz);
            good = add_cell<kScaled>(q, s, sum) && good && q.w >= 0x1p-60f && q.w <= 0x1p30f;
        }
    return good;
}

// Block (x = row block jb, y = plane k) sums rows [jb*rows, jb*rows+rows) of
// plane k into partials[k * gridDim.x + jb]; a warp takes whole rows.
template <class F>
__global__ void __launch_bounds__(kThreads, 3)
    energy_partials_kernel(F f, int nx, int ny, int nz, int rows, double h2, Coeffs64 c,
                           double *__restrict__ partials) {
    const int k = blockIdx.y;
    const int j0 = blockIdx.x * rows;
    const int j1 = min(j0 + rows, ny);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the block's largest magnitude (bit patterns: NaN above infinity)
    unsigned big = 0u;
    for (int j = j0 + warp; j < j1; j += kThreads / 32)
        for (int i = lane; i < nx; i += 32) {
            const long long e = f.at(i, j, k);
            big = max(big, max(__float_as_uint(f.u[e]) & 0x7fffffffu,
                               __float_as_uint(f.p[e]) & 0x7fffffffu));
        }
    __shared__ unsigned s_big;
    __shared__ double warp_sum[kThreads / 32];
    if (threadIdx.x == 0) s_big = 0u;
    __syncthreads();
    big = __reduce_max_sync(0xffffffffu, big);
    if (lane == 0) atomicMax(&s_big, big);
    __syncthreads();
    big = s_big;
    double acc = 0.0;
    if (big == 0u) {   // every term is zero, or 0 / 0 where the model is bad
        bool good = true;
        for (int j = j0 + warp; j < j1; j += kThreads / 32) {
#pragma unroll 4
            for (int i = lane; i < nx; i += 32) good &= f.surely_positive(f.at(i, j, k));
        }
        for (int j = j0 + warp; !good && j < j1; j += kThreads / 32)
            for (int i = lane; i < nx; i += 32)
                if (!(f.w_at(f.at(i, j, k)) > 0.0f)) acc = nan("");
    } else {
        const int ex = (int)(big >> 23) - 127;
        // values near 1 need no scaling; else the block's largest is brought there
        const bool near1 = ex >= -30 && ex <= 40;
        const int se = near1 ? 0 : max(-60, min(60, -ex));
        const float s = __int_as_float((se + 127) << 23);
        const bool inside = j0 >= 4 && j1 + 4 <= ny && k >= 4 && k + 4 < nz;
        Sums sum;
        bool fast = near1 || abs(ex + se) <= 30;
        if (near1 && inside)
            fast = sum_rows<false, true>(f, j0, j1, k, nx, ny, nz, s, &sum);
        else if (fast)
            fast = sum_rows<true, false>(f, j0, j1, k, nx, ny, nz, s, &sum);
        const double kin = sum.kinetic();
        if (fast && isfinite(kin))
            acc = (kin - sum.pot / 5040.0) * scalbn(1.0, -2 * se) / h2;
        else
            for (int j = j0 + warp; j < j1; j += kThreads / 32)
                for (int i = lane; i < nx; i += 32)
                    acc = __dadd_rn(acc, cell_fp64(load_cell<false>(f, i, j, k, nx, ny, nz), c, h2));
    }
    // fixed-order block reduction: warp shuffles, then warp 0
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) warp_sum[warp] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = threadIdx.x < kThreads / 32 ? warp_sum[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) partials[(long long)k * gridDim.x + blockIdx.x] = acc;
    }
}

// One block: out[0] = sum of partials[0 .. n), in a fixed order.
__global__ void __launch_bounds__(kThreads) sum_partials_kernel(const double *__restrict__ partials,
                                                                int n, double *__restrict__ out) {
    double acc = 0.0;
    for (int q = threadIdx.x; q < n; q += blockDim.x) acc += partials[q];
    __shared__ double warp_sum[kThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = threadIdx.x < kThreads / 32 ? warp_sum[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) out[0] = acc;
    }
}

template <class F>
cudaError_t launch_energy(const F &f, int nx, int ny, int nz, double h, const Coeffs64 &c,
                          double *partials, double *out, cudaStream_t s) {
    const int rows = energy_rows_per_block();
    dim3 grid((ny + rows - 1) / rows, nz, 1);
    cudaError_t e = launch(energy_partials_kernel<F>, grid, kThreads, 0, s, f, nx, ny, nz, rows, h * h,
                           c, partials);
    if (e != cudaSuccess) return e;
    return launch(sum_partials_kernel, 1, kThreads, 0, s, partials, (int)(grid.x * grid.y), out);
}

}  // namespace

int energy_rows_per_block() { return 32; }

long long energy_partial_count(int ny, int nz) {
    const int rows = energy_rows_per_block();
    return (long long)((ny + rows - 1) / rows) * nz;
}

cudaError_t launch_energy_padded(const float *u, const float *p, const float *w, const Geom &g,
                                 double h, const Coeffs64 &c, double *partials, double *out,
                                 cudaStream_t s) {
    PaddedFields f{u, p, w, g};
    return launch_energy(f, g.nx, g.ny, g.nz, h, c, partials, out, s);
}

cudaError_t launch_energy_noalloc(const float *u, const float *p, const float *v, int nx, int ny,
                                  int nz, double h, double dt, const Coeffs64 &c, double *out,
                                  cudaStream_t s) {
    // Host code cannot pass g_noalloc_partials itself (in host code the name
    // is a stand-in, not a device address): look its address up on the
    // current device. This is done on every call, so an address never
    // outlives the context it belongs to (a device reset may move it).
    void *ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_partials);
    if (e != cudaSuccess) return e;
    double *partials = static_cast<double *>(ptr);
    DenseFields f{u, p, v, nx, ny, nz, model_scale(dt / h)};
    return launch_energy(f, nx, ny, nz, h, c, partials, out, s);
}

}  // namespace ws
