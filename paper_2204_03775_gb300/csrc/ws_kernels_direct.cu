// Direct step kernel (one thread per cell, neighbours read from global
// memory through L1/L2).
//
// The direct kernel is the plain form of the fused step: it is used for grids
// smaller than a streaming tile or so small that a step is all latency (every
// load of a cell is in flight at once, where the streaming kernel walks planes
// one after the other), and as a second, independent CUDA path in the parity
// tests. The hot path is the streaming kernel.
#include "ws_ptx.cuh"

namespace ws {

// One fused step at one cell: Laplacian (Section II, 25-point formula),
// leapfrog of Eq. 2, absorbing taper, source (right-hand side of Eq. 2).
// u: u^n, up: u^{n-1} on entry and u^{n+1} on exit (same cell only),
// w: (V dt / h)^2.
__device__ __forceinline__ void step_cell(const float *u, const float *up, float *out,
                                          const float *w, const StepArgs &a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    const Geom &g = a.g;
    if (i >= g.nx || j >= g.ny) return;
    const long long p = pidx(g, i, j, k);
    const long long sy = g.pnx, sz = g.plane;

    const float uc = u[p];
    float s[5];
#pragma unroll
    for (int m = 1; m <= 4; ++m) {
        s[m] = ((u[p + m] + u[p - m]) + (u[p + m * sy] + u[p - m * sy])) +
               (u[p + m * sz] + u[p - m * sz]);
    }
    // sum_m c_m (s_m - 6 u): exactly zero on constants (see Coeffs)
    float d[5];
#pragma unroll
    for (int m = 1; m <= 4; ++m) d[m] = fmaf(-6.0f, uc, s[m]);
    float lap = a.c.c4 * d[4];
    lap = fmaf(a.c.c3, d[3], lap);
    lap = fmaf(a.c.c2, d[2], lap);
    lap = fmaf(a.c.c1, d[1], lap);

    if (a.lap) a.lap[p] = lap;
    const float wc = w[p];
    const float gd = a.gx[i] * a.gy[j] * a.gz[k];
    float un = gd * fmaf(wc, lap, fmaf(2.0f, uc, -gd * up[p]));
    for (int q = 0; q < a.src.n; ++q) {
        const SourceSample &ss = a.src.s[q];
        if (ss.i == i && ss.j == j && ss.k == k) un = fmaf(wc, ss.amp, un);
    }
    out[p] = un;
}

// The first entry of rec[lo .. hi), sorted by k, on plane k or above, found by the
// whole block: 256 samples a round, so two rounds for 65536 entries.
__device__ __forceinline__ int block_first_entry(const RecEntry *rec, int lo, int hi, int k) {
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, n = blockDim.x * blockDim.y;
    while (lo < hi) {
        const int step = (hi - lo + n - 1) / n;
        const long long at = lo + (long long)tid * step;
        const int below = __syncthreads_count(at < hi && rec[at].k < k);
        if (below == 0) break;
        hi = min(hi, lo + below * step);   // the samples lo, lo + step, .. below it are smaller
        lo += (below - 1) * step + 1;
    }
    return lo;
}

// Receivers: the entries [lo, hi) of a block's tile, sorted by k, that lie on its
// plane k are sampled, or the residual is added to their cells (atomically:
// receivers may share one), once all its threads have stored. (As a launch of its
// own this cost 1 us a step on grids of a few microseconds.)
__device__ __forceinline__ void record_block(float *out, const float *w, const StepArgs &a, int k,
                                             int lo, int hi, const RecEntry *rec) {
    if (lo == hi) return;
    __syncthreads();
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    for (int e = lo + tid; e < hi; e += blockDim.x * blockDim.y) {
        if (rec[e].k > k) break;
        if (rec[e].k < k) continue;
        const int i = blockIdx.x * blockDim.x + rec[e].lane, j = blockIdx.y * blockDim.y + rec[e].owner;
        const long long p = pidx(a.g, i, j, k), t = (long long)rec[e].r * a.nt_max + a.trace_step;
        if (a.inject)
            atomicAdd(&out[p], __fmul_rn(__fmul_rn(w[p], a.gx[i] * a.gy[j] * a.gz[k]), a.inject[t]));
        else
            a.traces[t] = out[p];
    }
}

// Tables without ranges by plane: a tile's range up to a block's threads is scanned,
// a longer one searched for the block's plane first. With a receiver on each cell
// of a vertical plane (such a table, for comparison): 48 x 40 x 40 (320 entries a
// tile) searched 2.89 us a step, scanned 3.07; 11 x 11 x 1200 (9600) 7.98, 14.4; 20
// x 120 x 6000 (48000) 304, 1748 (every block reading its tile's whole range: 3182).
constexpr int kScanEntries = 256;

__global__ void __launch_bounds__(256) step_direct_kernel(const float *u,
                                                          const float *up, float *out,
                                                          const float *w,
                                                          const __grid_constant__ StepArgs a,
                                                          const int *rec_ptr, const int rec_planes,
                                                          const RecEntry *rec) {
    // no kernel writes the receiver table: its ranges are read before the
    // predecessor is waited for
    const int tile = blockIdx.y * gridDim.x + blockIdx.x;
    const int range = rec_planes ? tile * rec_planes + blockIdx.z : tile;
    int lo = rec_ptr ? rec_ptr[range] : 0, hi = rec_ptr ? rec_ptr[range + 1] : 0;
    if (!rec_planes && hi - lo > kScanEntries) lo = block_first_entry(rec, lo, hi, blockIdx.z);
    wait_predecessor();
    step_cell(u, up, out, w, a);
    record_block(out, w, a, blockIdx.z, lo, hi, rec);
}

cudaError_t launch_step_direct(const float *u, const float *up, float *out, const float *w,
                               const StepArgs &a, const int *rec_ptr, int rec_planes,
                               const RecEntry *rec, cudaStream_t s) {
    dim3 block(kDirectX, kDirectY, 1);
    dim3 grid((a.g.nx + kDirectX - 1) / kDirectX, (a.g.ny + kDirectY - 1) / kDirectY, a.g.nz);
    return launch_overlapped(step_direct_kernel, grid, block, 0, s, u, up, out, w, a, rec_ptr, rec_planes,
                             rec);
}

}  // namespace ws
