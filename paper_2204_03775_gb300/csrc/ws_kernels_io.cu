// Copies between the caller's unpadded [nz][ny][nx] device arrays and the
// interiors of the padded fields.
//
// Bound: HBM, 8 bytes a cell and field. One launch moves both time levels.
// (One 2D copy per plane and field, which this replaces, cost 4 to 8 us a
// plane whatever its size: 256^3 in and out 4.2 ms, 1024^3 35 ms.)
#include "ws_internal.h"

namespace ws {
namespace {

constexpr int kCopyThreads = 256;
// Blocks of a launch: about two full loads of the GPU's 152 x 8 resident
// blocks; longer copies loop over their rows.
constexpr int kCopyBlocks = 2432;
// Loads of one row that a thread keeps in flight per field.
constexpr int kCopyDepth = 4;

template <int V>
struct VecOf;
template <>
struct VecOf<4> {
    using T = float4;
};
template <>
struct VecOf<1> {
    using T = float;
};

// A group of blockDim.x threads copies a row (nq vectors of V cells); both
// fields of a row are in flight together. kFields = 1 ignores s1 and d1.
template <int V, int kFields>
__global__ void __launch_bounds__(kCopyThreads)
    copy_rows_kernel(const float *__restrict__ s0, const float *__restrict__ s1,
                     float *__restrict__ d0, float *__restrict__ d1, const int nq,
                     const unsigned ny, const unsigned rows, const long long spitch,
                     const long long splane, const long long dpitch, const long long dplane) {
    using T = typename VecOf<V>::T;
    const int step = blockDim.x;
    for (unsigned long long r = (unsigned long long)blockIdx.x * blockDim.y + threadIdx.y; r < rows;
         r += (unsigned long long)gridDim.x * blockDim.y) {
        const unsigned k = (unsigned)r / ny, j = (unsigned)r - k * ny;
        const long long so = k * splane + j * spitch, dof = k * dplane + j * dpitch;
        const T *a0 = reinterpret_cast<const T *>(s0 + so);
        const T *a1 = reinterpret_cast<const T *>(s1 + so);
        T *b0 = reinterpret_cast<T *>(d0 + dof);
        T *b1 = reinterpret_cast<T *>(d1 + dof);
        for (int q = threadIdx.x; q < nq; q += kCopyDepth * step) {
            T x0[kCopyDepth], x1[kCopyDepth];
#pragma unroll
            for (int c = 0; c < kCopyDepth; ++c)
                if (q + c * step < nq) {
                    x0[c] = __ldcs(a0 + q + c * step);
                    if (kFields == 2) x1[c] = __ldcs(a1 + q + c * step);
                }
#pragma unroll
            for (int c = 0; c < kCopyDepth; ++c)
                if (q + c * step < nq) {
                    b0[q + c * step] = x0[c];
                    if (kFields == 2) b1[q + c * step] = x1[c];
                }
        }
    }
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <int V>
cudaError_t launch_copy(const float *s0, const float *s1, float *d0, float *d1, const Geom &g,
                        long long spitch, long long splane, long long dpitch, long long dplane,
                        cudaStream_t s) {
    const int nq = g.nx / V;
    // threads a row: the widest of 32, 16, 8 that leaves the fewest idle
    int bx = 32;
    for (int b : {16, 8})
        if ((nq + b - 1) / b * b < (nq + bx - 1) / bx * bx) bx = b;
    const dim3 block(bx, kCopyThreads / bx);
    const unsigned rows = (unsigned)g.ny * (unsigned)g.nz;   // at most 65535^2
    const unsigned want = (unsigned)(((unsigned long long)rows + block.y - 1) / block.y);
    const unsigned grid = want < (unsigned)kCopyBlocks ? want : (unsigned)kCopyBlocks;
    if (s1)
        copy_rows_kernel<V, 2><<<grid, block, 0, s>>>(s0, s1, d0, d1, nq, g.ny, rows, spitch, splane,
                                                      dpitch, dplane);
    else
        copy_rows_kernel<V, 1><<<grid, block, 0, s>>>(s0, nullptr, d0, nullptr, nq, g.ny, rows,
                                                      spitch, splane, dpitch, dplane);
    return cudaGetLastError();
}

}  // namespace

// 128-bit accesses need rows that are whole float4s on both sides: the padded
// interiors always start on 128 bytes, the caller's rows only when nx is a
// multiple of 4 and the arrays are 16-byte aligned; else one cell a thread
// (coalesced all the same).
cudaError_t launch_copy_in(const float *a, const float *b, float *A, float *B, const Geom &g,
                           cudaStream_t s) {
    const long long o = pidx(g, 0, 0, 0), plane = (long long)g.nx * g.ny;
    float *d1 = b ? B + o : nullptr;
    if (g.nx % 4 == 0 && aligned16(a) && aligned16(b))
        return launch_copy<4>(a, b, A + o, d1, g, g.nx, plane, g.pnx, g.plane, s);
    return launch_copy<1>(a, b, A + o, d1, g, g.nx, plane, g.pnx, g.plane, s);
}

cudaError_t launch_copy_out(const float *A, const float *B, float *a, float *b, const Geom &g,
                            cudaStream_t s) {
    const long long o = pidx(g, 0, 0, 0), plane = (long long)g.nx * g.ny;
    const float *s1 = B ? B + o : nullptr;
    if (g.nx % 4 == 0 && aligned16(a) && aligned16(b))
        return launch_copy<4>(A + o, s1, a, b, g, g.pnx, g.plane, g.nx, plane, s);
    return launch_copy<1>(A + o, s1, a, b, g, g.pnx, g.plane, g.nx, plane, s);
}

}  // namespace ws
