// Copies between the caller's unpadded [nz][ny][nx] device arrays and the
// interiors of the padded fields, and the conversion of the caller's model.
//
// Copies: bound by HBM, 8 bytes a cell and field. One launch moves both time levels.
// (One 2D copy per plane and field, which this replaces, cost 4 to 8 us a
// plane whatever its size: 256^3 in and out 4.2 ms, 1024^3 35 ms.)
#include "ws_model.cuh"

namespace ws {

// Blocks of a launch: about two full loads of the GPU's 152 x 8 resident
// blocks; longer copies loop over their rows.
constexpr int kCopyBlocks = 2432;

// Threads a row: the widest of 32, 16, 8 that leaves the fewest idle, and more where
// long rows are too few to fill the GPU (65000 x 9 x 3, 27 rows: two fields in 18
// us, out 20; with 32 threads a row 91 and 95; 2D copies take 59 and 38).
unsigned row_grid(const Geom &g, dim3 *block) {
    const int nq = (g.nx + 3) / 4;
    int bx = 32;
    for (int b : {16, 8})
        if ((nq + b - 1) / b * b < (nq + bx - 1) / bx * bx) bx = b;
    const unsigned long long rows = (unsigned long long)g.ny * g.nz;
    while (bx >= 32 && bx < kRowThreads && nq >= 8 * bx && rows * bx < 608ull * kRowThreads) bx *= 2;
    *block = dim3(bx, kRowThreads / bx);
    const unsigned long long want = (rows + block->y - 1) / block->y;
    return (unsigned)(want < kCopyBlocks ? want : kCopyBlocks);
}

namespace {

// Vectors of one row that a thread keeps in flight per field: four in rows of
// whole vectors; one (two loads) in shifted rows, whose 60 registers leave
// fewer warps (755 x 994 x 400 in 863 us, with two of them 1007).
constexpr int kCopyDepth = 4, kShiftDepth = 1;

// One or two arrays on each side: in: user -> padded, out: padded -> user.
struct Fields {
    const float *src[2];
    float *dst[2];
};

// The caller's rows when they do not all start on 16 bytes: row r starts
// `shift` elements (0..3) behind the 16-byte boundary `base`; [lo, hi) are the
// elements of `base` that belong to the whole array.
struct Row {
    long long lo, hi;
    int shift;
};
__device__ __forceinline__ Row user_row(const float *array, long long start, long long cells) {
    const int shift = (int)((reinterpret_cast<uintptr_t>(array + start) >> 2) & 3u);
    return Row{shift - start, shift - start + cells, shift};
}

// The 16 bytes at element e of base, only those inside [lo, hi).
__device__ __forceinline__ float4 load_inside(const float *base, long long e, const Row &r) {
    if (e >= r.lo && e + 4 <= r.hi) return *reinterpret_cast<const float4 *>(base + e);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e + 0 >= r.lo && e + 0 < r.hi) v.x = base[e + 0];
    if (e + 1 >= r.lo && e + 1 < r.hi) v.y = base[e + 1];
    if (e + 2 >= r.lo && e + 2 < r.hi) v.z = base[e + 2];
    if (e + 3 >= r.lo && e + 3 < r.hi) v.w = base[e + 3];
    return v;
}

// Elements s .. s+3 of the 8 in (a, b).
__device__ __forceinline__ float4 window(const float4 &a, const float4 &b, int s) {
    switch (s) {
        case 0: return a;
        case 1: return make_float4(a.y, a.z, a.w, b.x);
        case 2: return make_float4(a.z, a.w, b.x, b.y);
        case 3: return make_float4(a.w, b.x, b.y, b.z);
        default: return b;
    }
}

// Elements [from, to) of v to p (16-byte aligned when all four go).
__device__ __forceinline__ void store_part(float *p, const float4 &v, int from, int to) {
    if (from <= 0 && to >= 4) {
        *reinterpret_cast<float4 *>(p) = v;
        return;
    }
    if (from <= 0 && to > 0) p[0] = v.x;
    if (from <= 1 && to > 1) p[1] = v.y;
    if (from <= 2 && to > 2) p[2] = v.z;
    if (from <= 3 && to > 3) p[3] = v.w;
}

// A group of blockDim.x threads copies a row; both fields of a row are in
// flight together. kAligned: every row is whole 16-byte vectors on both
// sides. Otherwise every access still is a 16-byte one on a 16-byte boundary:
// the shifted side is read as two neighbouring vectors, the second of which
// comes from L1, and a row's first and last vectors are written cell by cell,
// so nothing outside the row changes. Both fields of 755 x 994 x 400: in 863,
// out 754 us (5.6, 6.4 TB/s), against 1166, 1523 us with 4-byte accesses;
// 1024 x 512 x 512: in 650, out 641 us (6.6, 6.7 TB/s of the measured 6.78).
template <bool kAligned, bool kIn, int kFields>
__global__ void __launch_bounds__(kRowThreads)
    copy_rows_kernel(const Fields f, const int nx, const unsigned ny, const unsigned rows,
                     const int pitch, const long long plane, const long long cells) {
    const int step = blockDim.x;
    for (unsigned long long r = (unsigned long long)blockIdx.x * blockDim.y + threadIdx.y; r < rows;
         r += (unsigned long long)gridDim.x * blockDim.y) {
        const unsigned k = (unsigned)r / ny, j = (unsigned)r - k * ny;
        const long long uo = (long long)r * nx, po = k * plane + (long long)j * pitch;
        if constexpr (kAligned) {
            const int nq = nx / 4;
            for (int q = threadIdx.x; q < nq; q += kCopyDepth * step) {
                float4 x[kFields][kCopyDepth];
#pragma unroll
                for (int c = 0; c < kCopyDepth; ++c)
#pragma unroll
                    for (int m = 0; m < kFields; ++m)
                        if (q + c * step < nq)
                            x[m][c] = __ldcs(reinterpret_cast<const float4 *>(
                                                 f.src[m] + (kIn ? uo : po)) + q + c * step);
#pragma unroll
                for (int c = 0; c < kCopyDepth; ++c)
#pragma unroll
                    for (int m = 0; m < kFields; ++m)
                        if (q + c * step < nq)
                            reinterpret_cast<float4 *>(f.dst[m] + (kIn ? po : uo))[q + c * step] =
                                x[m][c];
            }
        } else {
            Row w[kFields];
            const float *ub[kFields];   // the caller's side, 16-byte aligned
            const float *pb[kFields];   // the padded side
            int nq = (nx + 3) / 4;      // in: padded vectors of the row
#pragma unroll
            for (int m = 0; m < kFields; ++m) {
                const float *user = kIn ? f.src[m] : f.dst[m];
                w[m] = user_row(user, uo, cells);
                ub[m] = user + uo - w[m].shift;
                pb[m] = (kIn ? f.dst[m] : f.src[m]) + po;
                // out: the most user vectors that either row touches
                if (!kIn) nq = max(nq, (nx + w[m].shift + 3) / 4);
            }
            // the row's vectors, and the one behind them, all lie in the array
            const bool inside = uo >= 4 && uo + nx + 8 <= cells;
            constexpr int D = kShiftDepth;
            for (int q = threadIdx.x; q < nq; q += D * step) {
                float4 a[kFields][D], b[kFields][D];
                if constexpr (kIn) {   // user cells 4v .. 4v+3 of the row
                    auto load = [&](auto &&vec) {
#pragma unroll
                        for (int c = 0; c < D; ++c)
#pragma unroll
                            for (int m = 0; m < kFields; ++m)
                                if (q + c * step < nq) {
                                    const long long e = 4ll * (q + c * step);
                                    a[m][c] = vec(m, e);
                                    b[m][c] = w[m].shift ? vec(m, e + 4) : a[m][c];
                                }
                    };
                    // all but the array's ends: plain loads, issued together
                    if (inside)
                        load([&](int m, long long e) {
                            return *reinterpret_cast<const float4 *>(ub[m] + e);
                        });
                    else
                        load([&](int m, long long e) { return load_inside(ub[m], e, w[m]); });
                } else {               // row cells 4v - shift .. + 3
#pragma unroll
                    for (int c = 0; c < D; ++c)
#pragma unroll
                        for (int m = 0; m < kFields; ++m) {
                            const int v = q + c * step;
                            if (v >= nq) continue;
                            b[m][c] = 4 * v < nx   // else beyond the row: not stored
                                          ? *reinterpret_cast<const float4 *>(pb[m] + 4 * v)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
                            a[m][c] = w[m].shift && v > 0
                                          ? *reinterpret_cast<const float4 *>(pb[m] + 4 * v - 4)
                                          : b[m][c];
                        }
                }
#pragma unroll
                for (int c = 0; c < D; ++c)
#pragma unroll
                    for (int m = 0; m < kFields; ++m) {
                        const int v = q + c * step;
                        if (v >= nq) continue;
                        if constexpr (kIn)
                            store_part(const_cast<float *>(pb[m]) + 4 * v,
                                       window(a[m][c], b[m][c], w[m].shift), 0, nx - 4 * v);
                        else
                            store_part(const_cast<float *>(ub[m]) + 4 * v,
                                       window(a[m][c], b[m][c], 4 - w[m].shift),
                                       w[m].shift - 4 * v, nx + w[m].shift - 4 * v);
                    }
            }
        }
    }
}

// Whole buffers (padding included) to zero: n floats of a, and of b if given.
// One launch for a pair of fields: a memset's call takes the host 11 us, which
// a run of a few hundred microseconds does not hide.
__global__ void __launch_bounds__(kRowThreads) zero_kernel(float4 *a, float4 *b, long long n4) {
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n4;
         t += (long long)gridDim.x * blockDim.x) {
        a[t] = z;
        if (b) b[t] = z;
    }
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <bool kIn>
cudaError_t launch_copy(const Fields &f, const Geom &g, cudaStream_t s) {
    // rows are whole vectors on both sides (the padded interiors always start
    // on 128 bytes)
    const float *const *user = kIn ? f.src : f.dst;
    const bool aligned = g.nx % 4 == 0 && aligned16(user[0]) && aligned16(user[1]);
    const unsigned rows = (unsigned)g.ny * (unsigned)g.nz;   // at most 65535^2
    dim3 block;
    const unsigned grid = row_grid(g, &block);
    const long long cells = (long long)rows * g.nx;
#define WS_COPY(AL, NF)                                                                   \
    launch(copy_rows_kernel<AL, kIn, NF>, grid, block, 0, s, f, g.nx, g.ny, rows, g.pnx, \
           g.plane, cells)
    if (aligned) return f.src[1] ? WS_COPY(true, 2) : WS_COPY(true, 1);
    return f.src[1] ? WS_COPY(false, 2) : WS_COPY(false, 1);
#undef WS_COPY
}

}  // namespace

cudaError_t launch_zero(float *a, float *b, size_t bytes, cudaStream_t s) {
    const long long n4 = (long long)(bytes / sizeof(float4));   // fields are whole 128-byte rows
    const long long want = (n4 + kRowThreads - 1) / kRowThreads;
    return launch(zero_kernel, (unsigned)(want < kCopyBlocks ? want : kCopyBlocks), kRowThreads, 0, s,
                  reinterpret_cast<float4 *>(a), reinterpret_cast<float4 *>(b), n4);
}

cudaError_t launch_copy_in(const float *a, const float *b, float *A, float *B, const Geom &g,
                           cudaStream_t s) {
    const long long o = pidx(g, 0, 0, 0);
    return launch_copy<true>(Fields{{a, b}, {A + o, b ? B + o : nullptr}}, g, s);
}

cudaError_t launch_copy_out(const float *A, const float *B, float *a, float *b, const Geom &g,
                            cudaStream_t s) {
    const long long o = pidx(g, 0, 0, 0);
    return launch_copy<false>(Fields{{A + o, B ? B + o : nullptr}, {a, b}}, g, s);
}

// ------------------------------------------------------------ model

namespace {

struct Extrema {
    unsigned hi, lo;
    // max and min as float bit patterns (their unsigned order is the float
    // order for x >= 0); a value that is not finite and > 0 counts as 0 in
    // the minimum, which the host rejects
    __device__ __forceinline__ void take(float x) {
        const bool good = x > 0.0f && isfinite(x);
        const unsigned b = __float_as_uint(x);
        hi = max(hi, good ? b : 0u);
        lo = min(lo, good ? b : 0u);
    }
};

template <class Conv>
__device__ __forceinline__ float convert(float x, const ModelScale &k, Extrema &e) {
    e.take(x);
    return to_model<Conv>(x, k);
}

// The model into the padded field w: from the caller's array (rows that are
// whole 16-byte vectors) or, src null, in place. Bound: HBM, 8 bytes a cell.
// Extrema meet in the block before its one atomic pair: one pair a warp, all
// on two words, took 0.67 ms at 256^3 and 44 ms at 1024^3; this takes 0.026
// and 1.43 ms from a velocity (6.0 TB/s), 0.035 and 1.73 from a slowness
// (one float division a cell); with the double products issued for every
// cell 7.8 ms at 1024^3.
template <class Conv>
__global__ void __launch_bounds__(kRowThreads)
    model_kernel(const float *src, float *w, const int nx, const unsigned ny, const unsigned rows,
                 const int pitch, const long long plane, const ModelScale scale,
                 unsigned *__restrict__ extrema) {
    Extrema e{0u, 0x7f800000u};
    const int step = blockDim.x;
    for (unsigned long long r = (unsigned long long)blockIdx.x * blockDim.y + threadIdx.y; r < rows;
         r += (unsigned long long)gridDim.x * blockDim.y) {
        const unsigned k = (unsigned)r / ny, j = (unsigned)r - k * ny;
        float *out = w + k * plane + (long long)j * pitch;
        const float *in = src ? src + (long long)r * nx : out;
        for (int i = 4 * threadIdx.x; i < nx; i += 8 * step) {
            // two vectors in flight (in place, the last one may reach into
            // the halo of its row)
            const int i2 = i + 4 * step;
            const float4 x = *reinterpret_cast<const float4 *>(in + i);
            const float4 y = i2 < nx ? *reinterpret_cast<const float4 *>(in + i2) : x;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int at = h ? i2 : i;
                const float4 v = h ? y : x;
                if (at + 4 <= nx) {
                    float4 o;
                    o.x = convert<Conv>(v.x, scale, e);
                    o.y = convert<Conv>(v.y, scale, e);
                    o.z = convert<Conv>(v.z, scale, e);
                    o.w = convert<Conv>(v.w, scale, e);
                    *reinterpret_cast<float4 *>(out + at) = o;
                } else if (at < nx) {
                    out[at] = convert<Conv>(v.x, scale, e);
                    if (at + 1 < nx) out[at + 1] = convert<Conv>(v.y, scale, e);
                    if (at + 2 < nx) out[at + 2] = convert<Conv>(v.z, scale, e);
                }
            }
        }
    }
    __shared__ unsigned hi, lo;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        hi = 0u;
        lo = 0x7f800000u;
    }
    __syncthreads();
    const unsigned whi = __reduce_max_sync(0xffffffffu, e.hi);
    const unsigned wlo = __reduce_min_sync(0xffffffffu, e.lo);
    if (((threadIdx.y * blockDim.x + threadIdx.x) & 31) == 0) {
        atomicMax(&hi, whi);
        atomicMin(&lo, wlo);
    }
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        atomicMax(&extrema[0], hi);
        atomicMin(&extrema[1], lo);
    }
}

// v may be null (the values are in w already). Rows that are not whole
// vectors are brought into the padded field first.
template <class Conv>
cudaError_t launch_model(const float *v, float *w, const Geom &g, double c, unsigned *extrema,
                         cudaStream_t s) {
    if (v && (g.nx % 4 != 0 || !aligned16(v))) {
        const cudaError_t e = launch_copy_in(v, nullptr, w, nullptr, g, s);
        if (e != cudaSuccess) return e;
        v = nullptr;
    }
    dim3 block;
    const unsigned grid = row_grid(g, &block);
    return launch(model_kernel<Conv>, grid, block, 0, s, v, w + pidx(g, 0, 0, 0), g.nx, g.ny,
                  (unsigned)g.ny * (unsigned)g.nz, g.pnx, g.plane, model_scale(c), extrema);
}

}  // namespace

cudaError_t launch_velocity_to_w(const float *v, float *w, const Geom &g, double dt_over_h,
                                 unsigned *extrema, cudaStream_t s) {
    return launch_model<FromVelocity>(v, w, g, dt_over_h, extrema, s);
}

cudaError_t launch_slowness2_to_w(const float *m, float *w, const Geom &g, double dt_over_h2,
                                  unsigned *extrema, cudaStream_t s) {
    return launch_model<FromSlowness2>(m, w, g, dt_over_h2, extrema, s);
}

}  // namespace ws
