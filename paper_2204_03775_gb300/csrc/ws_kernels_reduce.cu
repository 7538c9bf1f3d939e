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
// at 320 x 288 x 256. Instead each cell is summed as pairs of floats, hi + lo,
// through error-free sums and products (Dekker, Knuth), about 280 FP32
// operations a cell, and only the threads' totals are FP64 (0.37 ms, issue-bound):
//  - 5040 h^2 L p = 8064 d1 - 1008 d2 + 128 d3 - 9 d4, d_m the six neighbours at
//    distance m less 6 p: whole weights, so none is rounded, and sums of floats
//    of like size leave lo words that are small multiples of one ulp.
//  - Where the block's largest value is not within 2^-30 .. 2^40, values are
//    scaled by a power of two that brings it to about 1, so no product underflows
//    that matters.
// The error of the sum against 80-bit arithmetic, both forms emulated on the
// CPU, on smooth fields of 40^3 to 96^3 cells: at most 1.6e-16, FP64 3.0e-16
// (whose weights are rounded); on white noise both 1 to 3e-16. Blocks out of the scaled range, and threads that meet a
// value that is not finite or a model below 2^-60, take the FP64 form.
#include "ws_model.cuh"

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

// hi + lo, lo below half an ulp of hi or so.
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
__device__ __forceinline__ Pair add(Pair a, Pair b) {
    const Pair s = two_sum(a.hi, b.hi);
    const float l = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    const float h = __fadd_rn(s.hi, l);
    return Pair{h, __fadd_rn(__fsub_rn(s.hi, h), l)};
}
__device__ __forceinline__ Pair mul(Pair a, float b) {
    const Pair p = two_prod(a.hi, b);
    return Pair{p.hi, __fmaf_rn(a.lo, b, p.lo)};
}

// a + b, lo not folded into hi (it may grow to a few ulps of it).
__device__ __forceinline__ Pair add_loose(Pair a, Pair b) {
    const Pair s = two_sum(a.hi, b.hi);
    return Pair{s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ Pair renormalize(Pair a) {
    const float h = __fadd_rn(a.hi, a.lo);
    return Pair{h, __fadd_rn(__fsub_rn(a.hi, h), a.lo)};
}

// The values that a cell's term needs.
struct Cell {
    float u, p, w;
    float n[4][6];   // p at distance 1 .. 4 on x+, x-, y+, y-, z+, z-
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
        c.n[m - 1][0] = f.p_near(e, m, i + m < nx);
        c.n[m - 1][1] = f.p_near(e, -m, i - m >= 0);
        c.n[m - 1][2] = f.p_near(e, m * sy, kInside || j + m < ny);
        c.n[m - 1][3] = f.p_near(e, -m * sy, kInside || j - m >= 0);
        c.n[m - 1][4] = f.p_near(e, m * sz, kInside || k + m < nz);
        c.n[m - 1][5] = f.p_near(e, -m * sz, kInside || k - m >= 0);
    }
    return c;
}

// Adds (u - p)^2 / w to *kin + *kin2 and 5040 u h^2 L p to *pot, of the values
// times s (a power of two; kScaled false: s = 1).
template <bool kScaled>
__device__ __forceinline__ void add_cell(const Cell &c, float s, Pair *kin, float *kin2, Pair *pot) {
    auto scaled = [&](float x) { return kScaled ? x * s : x; };
    const float u = scaled(c.u), p = scaled(c.p);
    const Pair p6 = two_prod(6.0f, p);
    Pair lap{0.0f, 0.0f};
#pragma unroll
    for (int m = 4; m >= 1; --m) {
        const float *n = c.n[m - 1];
        Pair d = two_sum(scaled(n[0]), scaled(n[1]));
        d = add_loose(d, two_sum(scaled(n[2]), scaled(n[3])));
        d = add_loose(d, two_sum(scaled(n[4]), scaled(n[5])));
        d = add_loose(d, Pair{-p6.hi, -p6.lo});
        const Pair t = mul(d, m == 1 ? 8064.0f : m == 2 ? -1008.0f : m == 3 ? 128.0f : -9.0f);
        lap = m == 4 ? t : add_loose(lap, t);
    }
    *pot = add(*pot, mul(renormalize(lap), u));
    // u - p = d exactly; (u - p)^2 = q + d.lo^2, the last below 2^-50 of q but
    // never negative, so it is summed apart
    const Pair d = two_sum(u, -p);
    Pair q = two_prod(d.hi, d.hi);
    q.lo = __fmaf_rn(2.0f * d.hi, d.lo, q.lo);
    // q / w: the nearest quotient, its exact remainder, that one's quotient
    const float a = __fdiv_rn(q.hi, c.w);
    const float r = __fadd_rn(__fmaf_rn(-a, c.w, q.hi), q.lo);
    *kin = add(*kin, Pair{a, __fdividef(r, c.w)});
    *kin2 = __fadd_rn(*kin2, __fdividef(__fmul_rn(d.lo, d.lo), c.w));
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
            l[a] = __fma_rn(cm, __dadd_rn((double)c.n[m - 1][2 * a], (double)c.n[m - 1][2 * a + 1]),
                            l[a]);
        }
    }
    const double lap = __ddiv_rn(__dadd_rn(__dadd_rn(l[0], l[1]), l[2]), h2);
    const double uc = c.u;
    const double d = __dsub_rn(uc, pc);
    const double vdt2 = __dmul_rn((double)c.w, h2);   // (V dt)^2
    return __fma_rn(-uc, lap, __ddiv_rn(__dmul_rn(d, d), vdt2));
}

// This thread's cells of rows [j0, j1) of plane k, a warp a row at a time;
// false if one of them has a model out of range.
template <bool kScaled, bool kInside, class F>
__device__ __forceinline__ bool sum_rows(const F &f, int j0, int j1, int k, int nx, int ny, int nz,
                                         float s, Pair *kin, float *kin2, Pair *pot) {
    bool good = true;
    for (int j = j0 + (threadIdx.x >> 5); j < j1; j += kThreads / 32)
        for (int i = threadIdx.x & 31; i < nx; i += 32) {
            const Cell q = load_cell<kInside>(f, i, j, k, nx, ny, nz);
            good = good && q.w >= 0x1p-60f;
            add_cell<kScaled>(q, s, kin, kin2, pot);
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
        Pair kin{0.0f, 0.0f}, pot{0.0f, 0.0f};
        float kin2 = 0.0f;
        bool fast = near1 || abs(ex + se) <= 30;
        if (near1 && inside)
            fast = sum_rows<false, true>(f, j0, j1, k, nx, ny, nz, s, &kin, &kin2, &pot);
        else if (fast)
            fast = sum_rows<true, false>(f, j0, j1, k, nx, ny, nz, s, &kin, &kin2, &pot);
        const double K = (double)kin.hi + ((double)kin.lo + (double)kin2), Q = (double)pot.hi + (double)pot.lo;
        if (fast && isfinite(K) && isfinite(Q))
            acc = (K - Q / 5040.0) * scalbn(1.0, -2 * se) / h2;
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
