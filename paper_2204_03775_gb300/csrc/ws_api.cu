// Host side of the C ABI declared in include/wavestep.h: the handle, its
// buffers and tensor maps, and the entry points of the forward stepper.
#include "ws_host.h"

namespace wsh {

thread_local char g_err[512] = "";

int fail(int code, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
    return code;
}

int cuda_fail(cudaError_t e, const char *what) {
    cudaGetLastError();   // reported here: later calls, the caller's too, don't find it
    if (e == cudaErrorMemoryAllocation)
        return fail(WS_ERR_OOM, "%s: %s", what, cudaGetErrorString(e));
    return fail(WS_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// Leapfrog stability limit of V dt / h for the 3D 25-point Laplacian: the
// largest |eigenvalue| times h^2 is 3 (|w0| + 2 sum |wm|) (the checkerboard
// mode), and the recurrence needs (V dt / h)^2 * that <= 4.
double cfl_limit() {
    const double s = std::fabs(kW0) + 2.0 * (std::fabs(kW1) + std::fabs(kW2) + std::fabs(kW3) +
                                             std::fabs(kW4));
    return 2.0 / std::sqrt(3.0 * s);
}

double ricker(double t, double f0, double t0, double amp) {
    const double pi = 3.14159265358979323846;
    const double a = pi * f0 * (t - t0);
    const double a2 = a * a;
    return amp * (1.0 - 2.0 * a2) * std::exp(-a2);
}

// Cerjan factor of cell idx on an axis of n cells.
double taper(int idx, int n, int nb, double a) {
    const int d = std::min(idx, n - 1 - idx);
    if (nb <= 0 || d >= nb) return 1.0;
    const double x = a * double(nb - d);
    return std::exp(-x * x);
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (fn) return fn;
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
        return nullptr;
    fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    return fn;
}

cudaError_t HostTables::next(size_t n, char **p) {
    if (at == 0 && passed[group]) {
        const cudaError_t e = cudaEventSynchronize(passed[group]);
        if (e != cudaSuccess) return e;
    }
    table[group][at].resize(n);
    *p = table[group][at].data();
    return cudaSuccess;
}

cudaError_t HostTables::upload(void *dst, cudaStream_t stream) {
    const std::vector<char> &t = table[group][at];
    cudaError_t e = cudaMemcpyAsync(dst, t.data(), t.size(), cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return e;
    if (++at < kGroup && t.size() <= kLarge) return cudaSuccess;
    if (!passed[group]) e = cudaEventCreateWithFlags(&passed[group], cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(passed[group], stream);
    if (e != cudaSuccess) cudaStreamSynchronize(stream);   // no event guards the group
    group = 1 - group;
    at = 0;
    return e;
}

size_t field_bytes(const ws::Geom &g) {
    return size_t(g.pnx) * size_t(g.pny) * size_t(g.pnz) * sizeof(float);
}

// A tensor map of a padded field over its interior only: origin at interior
// cell (0, 0, 0) (a 128-byte aligned address), extent nx x ny x nz, the
// padded pitches. The kernels' boxes that reach past the interior (the 4-cell
// halo of the edge tiles, the ragged end of the last tiles) are filled with
// zeros by the copy engine without reading memory: exactly the zero halo,
// and no DRAM traffic for halo or row padding.
int encode_map(CUtensorMap *map, void *base, const ws::Geom &g, int bx, int by,
               int elem_bytes) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
    if (!enc) return fail(WS_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz};
    cuuint64_t strides[2] = {(cuuint64_t)g.pnx * elem_bytes, (cuuint64_t)g.plane * elem_bytes};
    cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)by, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    const CUtensorMapDataType dt =
        elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16;
    void *origin = static_cast<char *>(base) + ws::pidx(g, 0, 0, 0) * elem_bytes;
    CUresult r = enc(map, dt, 3, origin, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(WS_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return WS_OK;
}

int encode_maps(ws_t ws) {
    const ws::Geom &g = ws->g;
    const int tx = ws->tiling.tx, ty = ws->tiling.ty;
    int rc = WS_OK;
    for (int b = 0; b < 2 && rc == WS_OK; ++b) {
        rc = encode_map(&ws->tmap_halo[b], ws->buf[b], g, tx + 2 * ws::kHalo, ty + 2 * ws::kHalo);
        if (rc == WS_OK) rc = encode_map(&ws->tmap_tile[b], ws->buf[b], g, tx, ty);
    }
    if (rc == WS_OK) rc = encode_map(&ws->tmap_w, ws->w, g, tx, ty);
    ws->tmap_ok = rc == WS_OK;
    return rc;
}

bool stream_fits(const ws_t ws, const ws::StreamTiling &t) {
    return ws::stream_tiling_supported(t.tx, t.ty) && ws->g.nx >= t.tx && ws->g.ny >= t.ty;
}

// Planes per work item whatever the GPU: blocks of about 200, the last one about a
// quarter as long as the others, so that a launch, whose items run in block order,
// ends on short ones. A candidate of the tuners (a batch of 32 shots of 96 to 320
// cells a side, 64 x 16 tiles: 870 us a step, the rules for one to six waves of
// items 876 to 893), and what the estimates below fall back on.
int default_zblock(int nz) {
    const int blocks = std::max(1, (int)std::lround(nz / 200.0));
    if (blocks == 1) return nz;
    return (4 * nz + 4 * blocks - 4) / (4 * blocks - 3);   // ceil(nz / (blocks - 3/4))
}

// The default z block of a streaming kernel for a grid and tile: the one of the
// smallest estimated step, in units of one plane of a full SM (about 1 us for
// FP32 64 x 16 tiles). An item of p planes takes item + p on a full SM; a CTA
// alone on its SM walks a plane in `alone` of that, in between it is
// interpolated.
//  - Up to `waves` waves of resident CTAs: the waves one after the other, the
//    last one at the speed of its fewer CTAs. Small grids end up with one or
//    two nearly full waves: FP32 192 x 160 x 144 in 64 x 16 tiles, 10-plane
//    blocks (0.99 of a wave) 13.1 us, 8 (1.2 waves) 17.0, 5 (1.9) 14.2; 128^3
//    5-plane blocks 7.9 us, the former 8-plane minimum 10.5.
//  - More waves blur into one another: the work divided by the CTAs, and a
//    tail that grows with the length of the last items. Blocks are also tried
//    with a last one about a quarter as long, so that a launch ends on short
//    items (FP32 755 x 994 x 200: blocks of 160 and 40 planes 369 us, of 67
//    376; 384^3: 128 147 us, 96 195).
// The constants were fitted to step times over z blocks and tiles: FP32, 33
// grids of 16 thousand to 270 million cells, the choice within 2 % (geometric
// mean) of the best of any tile and block; 16-bit, 22 grids, within 1.3 % (a
// 200-plane default, shortened to two waves, was 37 % off: 512^3 359 us, now
// 302). At least 2 planes (fewer only repeat the prologue), at most 256.
struct BlockModel {
    double item, alone, waves;
};
constexpr BlockModel kModel32{2.5, 0.62, 3.0}, kModel16{3.0, 0.6, 4.0};

int best_zblock(int nz, long long tiles, int slots, int sms, const BlockModel &m, double *best_cost) {
    constexpr double kTail = 0.2;
    constexpr int kMin = 2, kMax = 256;
    const int ctas = slots / sms;
    auto cost = [&](int zb) {
        const long long blocks = (nz + zb - 1) / zb, n = tiles * blocks;
        const int last = nz - (int)(blocks - 1) * zb;
        if (n > m.waves * slots)
            return tiles * (blocks * m.item + nz) / slots +
                   kTail * (m.item + (tiles >= slots / 2 ? last : zb));
        const long long full = n / slots, rem = n % slots;
        if (rem == 0) return full * (m.item + zb) - (tiles >= slots ? zb - last : 0);
        const double share = ctas > 1 ? double((rem + sms - 1) / sms - 1) / (ctas - 1) : 1.0;
        return full * (m.item + zb) + m.item +
               (rem <= tiles ? last : zb) * (m.alone + (1.0 - m.alone) * share);
    };
    int best = 0;
    auto consider = [&](int zb) {
        if (zb < 1 || zb > kMax || zb > nz) return;
        const double c = cost(zb);
        if (best == 0 || c < *best_cost - 1e-9) {
            best = zb;
            *best_cost = c;
        }
    };
    for (int b = 1;; ++b) {
        const int zb = (nz + b - 1) / b;
        if (b > 1 && zb < kMin) break;
        if (b > 1) consider((4 * nz + 4 * b - 4) / (4 * b - 3));   // the last a quarter as long
        consider(zb);
        if (zb <= kMin) break;
    }
    return best;
}

int default_zblock(const ws::Geom &g, int tx, int ty) {
    int slots = 0, sms = 0;
    if (ws::stream_slots(tx, ty, false, &slots, &sms) != cudaSuccess) return default_zblock(g.nz);
    const long long tiles = (long long)((g.nx + tx - 1) / tx) * ((g.ny + ty - 1) / ty);
    double cost = 0.0;
    return best_zblock(g.nz, tiles, slots, sms, kModel32, &cost);
}

// The tile of a grid for which none was chosen: 64 x 16 is the fastest, 32 x 16
// takes about 1.2 times as long per cell of its tiles (256^3 52.3 against 47.7
// us), so it is taken where 64-wide tiles would be emptier than that (70 x 900
// x 300: 73 against 82 us; 221 x 293 x 338 stays at 64: 63 against 67). Low
// grids get 8-row tiles. False if no tile fits.
bool default_tile(const ws::Geom &g, ws::StreamTiling *t) {
    if (g.nx < 32 || g.ny < 8) return false;
    t->ty = g.ny >= 16 ? 16 : 8;
    const int w64 = (g.nx + 63) / 64 * 64, w32 = (g.nx + 31) / 32 * 32;
    t->tx = g.nx >= 64 && 5 * w64 <= 6 * w32 ? 64 : 32;
    return true;
}

// Choose the kernel for the next steps; fills *tiling for the streaming one.
// Grids of at most kDirectCells cells, left to choose by themselves, take the
// direct kernel (steps with receivers): 80 x 40 x 35 in 2.48 us against 2.87 in
// the best stream tile and block, 48 x 40 x 40 2.30 against 2.84; 218 x 37 x 20
// (161 thousand cells) 3.43 against 3.20, 101 x 37 x 45 3.44 against 3.27, 64^3
// 3.48 against 3.18, 138 x 55 x 138 9.2 against 7.1.
int pick_kernel(ws_t ws, ws::StreamTiling *tiling) {
    constexpr long long kDirectCells = 150000;
    if (ws->kernel == WS_KERNEL_DIRECT) return WS_KERNEL_DIRECT;
    const ws::Geom &g = ws->g;
    ws::StreamTiling t = ws->tiling;
    if (!ws->tile_chosen) {
        const bool automatic = ws->kernel == WS_KERNEL_AUTO;
        if (!default_tile(g, &t)) return WS_KERNEL_DIRECT;   // AUTO only: STREAM needs more
        if (automatic && !stream_fits(ws, ws->need)) ws->need = t;   // ws_set_kernel: STREAM
        if (automatic && t.zb <= 0 && (long long)g.nx * g.ny * g.nz <= kDirectCells)
            return WS_KERNEL_DIRECT;
    } else if (ws->kernel == WS_KERNEL_AUTO && !stream_fits(ws, t)) {
        const ws::StreamTiling cands[3] = {{32, 16, 0}, {32, 8, 0}, {64, 16, 0}};
        bool found = false;
        for (const auto &c : cands)
            if (stream_fits(ws, c)) {
                t.tx = c.tx;
                t.ty = c.ty;
                found = true;
                break;
            }
        if (!found) return WS_KERNEL_DIRECT;
    }
    if (t.zb <= 0) {
        if (ws->auto_zb.tx != t.tx || ws->auto_zb.ty != t.ty)
            ws->auto_zb = ws::StreamTiling{t.tx, t.ty, default_zblock(g, t.tx, t.ty)};
        t.zb = ws->auto_zb.zb;
    }
    *tiling = t;
    return WS_KERNEL_STREAM;
}

// The receiver table is of no tile any more (the buffer stays).
static void forget_rec_tiles(ws_t ws) {
    ws->rec_ptr = nullptr;
    ws->rec_entries = nullptr;
    ws->rec_tiling_tx = ws->rec_tiling_ty = 0;
}

void free_receivers(ws_t ws) {
    cudaFree(ws->traces);
    cudaFree(ws->rec_table);
    ws->traces = nullptr;
    ws->traces_cap = 0;
    ws->rec_table = nullptr;
    ws->rec_table_cap = 0;
    forget_rec_tiles(ws);
}

// cudaMalloc for a handle: where the memory runs out, its staging for host arrays,
// which can be made again, is given back first.
cudaError_t handle_malloc(ws_t ws, void **p, size_t n) {
    cudaError_t e = cudaMalloc(p, n);
    if (e != cudaErrorMemoryAllocation || !ws->stage) return e;
    cudaGetLastError();
    if ((e = cudaStreamSynchronize(ws->stream)) != cudaSuccess) return e;
    cudaFree(ws->stage);
    ws->stage = nullptr;
    return cudaMalloc(p, n);
}

// A device buffer of at least n bytes: *p as it is if it holds them and is not far
// too large (kept: up to four times n, or 16 MiB), else a new one (the stream
// drains first: the old one may still be in use).
static int keep_or_grow(ws_t ws, void **p, size_t *cap, size_t n, const char *what) {
    constexpr size_t kKeep = 16u << 20;
    if (n <= *cap && *cap <= std::max(4 * n, kKeep)) return WS_OK;
    WS_CUDA(cudaStreamSynchronize(ws->stream), what);
    cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    WS_CUDA(handle_malloc(ws, p, n), what);
    *cap = n;
    return WS_OK;
}

// An upload whose host memory the handle reuses must not be captured into a graph,
// which would read it again at each launch. A stream under capture fails here.
static int refuse_capture(ws_t ws, const char *what) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    WS_CUDA(cudaStreamIsCapturing(ws->stream, &st), what);
    if (st != cudaStreamCaptureStatusNone) WS_CUDA(cudaErrorStreamCaptureUnsupported, what);
    return WS_OK;
}

// Receiver table for tile t. Streaming kernels: per (tile, warp) a range of
// entries sorted by k; thread owner = (row pair) * tx/4 + x quad, lane = 4 *
// (row of the pair) + x cell. Direct kernel (direct): per tile and plane, or, where
// those are many more than the receivers, per tile, sorted by k (20 x 120 x 6000
// with a receiver on each cell of a vertical plane: 211 us a step, 304 from ranges
// by tile; without receivers 170); owner = row,
// lane = x cell. The upload is issued on `stream`, which the steps that read the
// table follow. It is from pageable memory, which the GPU may read in place and
// behind the work queued before (the driver need not stage it, least of all on a
// coherent CPU): the host table stays with the handle until its upload is through,
// which needs no wait for the queued steps.
int build_rec_tiles(ws_t ws, const ws::StreamTiling &t, bool direct, cudaStream_t stream) {
    if (ws->nrec == 0) return WS_OK;
    if (ws->rec_tiling_tx == t.tx && ws->rec_tiling_ty == t.ty && ws->rec_direct == direct)
        return WS_OK;
    const int tiles_x = (ws->g.nx + t.tx - 1) / t.tx;
    const int tiles_y = (ws->g.ny + t.ty - 1) / t.ty;
    const int nrec = ws->nrec, nz = ws->g.nz, *ijk = ws->rec_ijk.data();
    const bool planes = direct && (long long)tiles_x * tiles_y * nz <= std::max(16384LL, 4LL * nrec);
    const int threads = t.tx / 4 * (t.ty / 2), warps = direct ? 1 : threads / 32;
    const int ranges = tiles_x * tiles_y * (planes ? nz : warps);
    // counting sorts: the receivers in the order of their planes (unless ranges are
    // of one plane), then into their ranges
    std::vector<int> ptr(ranges + 1, 0), range(nrec), order;
    int sx = 0;   // tiles are 2^sx wide
    while (1 << sx < t.tx) ++sx;
    auto rows = [&](int j) { return direct ? j / ws::kDirectY : j / t.ty; };
    auto entry = [&](int r, int tile_row) {
        const int i = ijk[3 * r] & (t.tx - 1), j = ijk[3 * r + 1] - tile_row * t.ty;
        return direct ? ws::RecEntry{ijk[3 * r + 2], j, i, r}
                      : ws::RecEntry{ijk[3 * r + 2], (j >> 1) * (t.tx >> 2) + (i >> 2),
                                     (j & 1) * 4 + (i & 3), r};
    };
    for (int r = 0; r < nrec; ++r) {
        const int row = rows(ijk[3 * r + 1]), tile = row * tiles_x + (ijk[3 * r] >> sx);
        range[r] = planes ? tile * nz + ijk[3 * r + 2]
                          : direct ? tile : tile * warps + (entry(r, row).owner >> 5);
        ptr[range[r] + 1]++;
    }
    for (int q = 0; q < ranges; ++q) ptr[q + 1] += ptr[q];
    if (!planes) {
        std::vector<int> at(nz + 1, 0);
        for (int r = 0; r < nrec; ++r) at[ijk[3 * r + 2] + 1]++;
        for (int k = 0; k < nz; ++k) at[k + 1] += at[k];
        order.resize(nrec);
        for (int r = 0; r < nrec; ++r) order[at[ijk[3 * r + 2]]++] = r;
    }
    // one buffer and one upload: the ranges, then the entries
    const size_t head = (sizeof(int) * ptr.size() + 15) / 16 * 16;
    const size_t bytes = head + sizeof(ws::RecEntry) * nrec;
    int rc = refuse_capture(ws, "upload receiver table");
    if (rc != WS_OK) return rc;
    forget_rec_tiles(ws);   // until the upload is issued
    rc = keep_or_grow(ws, &ws->rec_table, &ws->rec_table_cap, bytes, "cudaMalloc receiver table");
    if (rc != WS_OK) return rc;
    char *table = nullptr;
    WS_CUDA(ws->rec_host.next(bytes, &table), "upload receiver table");
    std::memcpy(table, ptr.data(), sizeof(int) * ptr.size());
    ws::RecEntry *entries = reinterpret_cast<ws::RecEntry *>(table + head);
    for (int q = 0; q < nrec; ++q) {
        const int r = planes ? q : order[q];
        entries[ptr[range[r]]++] = entry(r, rows(ijk[3 * r + 1]));
    }
    WS_CUDA(ws->rec_host.upload(ws->rec_table, stream), "upload receiver table");
    ws->rec_ptr = static_cast<int *>(ws->rec_table);
    ws->rec_entries = reinterpret_cast<ws::RecEntry *>(static_cast<char *>(ws->rec_table) + head);
    ws->rec_tiling_tx = t.tx;
    ws->rec_tiling_ty = t.ty;
    ws->rec_direct = direct;
    ws->rec_planes = planes ? nz : 0;
    return WS_OK;
}

static bool on_this_device(const char *p) {
    cudaPointerAttributes a{};
    int dev = -1;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return (a.type == cudaMemoryTypeDevice && a.device == dev) || a.type == cudaMemoryTypeManaged;
}

// Whether kernels may take a caller's device array of an unpadded field (or no
// array): floats on their natural alignment, in this device's memory from the
// first byte to the last. A 2D copy takes any address, and returns an error where
// a kernel would fault. (Asking costs the host 0.5 us an array: two levels of 96^3
// in and out and a step between them 26.3 -> 28.2 us.)
static bool kernel_copyable(const ws_t ws, const void *p) {
    if (!p) return true;
    const char *c = static_cast<const char *>(p);
    const size_t bytes = sizeof(float) * size_t(ws->g.nx) * ws->g.ny * ws->g.nz;
    return (reinterpret_cast<uintptr_t>(p) & 3u) == 0 && on_this_device(c) &&
           on_this_device(c + bytes - 1);
}

// The handle's device staging for host arrays, made by the first of them and kept
// until ws_destroy or until the handle runs out of memory: planes of an unpadded
// field, at most kStageMax bytes (null: not even one plane, or no memory). *planes
// of them move by one contiguous copy and one kernel instead of a 2D copy per
// plane, at 9 us or more each from pageable memory: both levels of 101 x 37 x 45
// out 819 us, now 38; of 256 x 256 x 200 in 8.3 ms, now 0.65 (pinned 1.38, now 0.56).
static float *host_stage(ws_t ws, int *planes) {
    constexpr size_t kStageMax = 64u << 20;
    const ws::Geom &g = ws->g;
    const size_t plane = sizeof(float) * size_t(g.nx) * g.ny;
    *planes = (int)std::min<size_t>(g.nz, kStageMax / plane);
    if (*planes < 1) return nullptr;
    if (!ws->stage) {
        // another thread's capture must not see this allocation
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(ws->stream, &st) != cudaSuccess ||
            st != cudaStreamCaptureStatusNone || cudaMalloc(&ws->stage, plane * *planes) != cudaSuccess) {
            cudaGetLastError();
            ws->stage = nullptr;
        }
        cudaThreadExchangeStreamCaptureMode(&mode);
    }
    return ws->stage;
}

// Copy unpadded [nz][ny][nx] arrays into the interiors of padded buffers: device
// arrays by one kernel, host arrays through the staging buffer or plane by plane.
int copy_in(ws_t ws, float *dst, const float *src, int on_device, float *dst2, const float *src2) {
    const ws::Geom &g = ws->g;
    if (on_device && kernel_copyable(ws, src) && kernel_copyable(ws, src2)) {
        WS_CUDA(ws::launch_copy_in(src, src2, dst, dst2, g, ws->stream), "copy into the padded field");
        ws->launches++;
        return WS_OK;
    }
    int planes = 0;
    if (float *stage = on_device ? nullptr : host_stage(ws, &planes)) {
        const size_t plane = size_t(g.nx) * g.ny;
        for (int k = 0; k < g.nz; k += planes) {
            ws::Geom part = g;
            part.nz = std::min(planes, g.nz - k);
            WS_CUDA(cudaMemcpyAsync(stage, src + k * plane, sizeof(float) * plane * part.nz,
                                    cudaMemcpyHostToDevice, ws->stream),
                    "copy into the padded field");
            WS_CUDA(ws::launch_copy_in(stage, nullptr, dst + k * g.plane, nullptr, part, ws->stream),
                    "copy into the padded field");
            ws->launches++;
        }
        return src2 ? copy_in(ws, dst2, src2, on_device) : WS_OK;
    }
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    for (int k = 0; k < g.nz; ++k) {
        WS_CUDA(cudaMemcpy2DAsync(dst + ws::pidx(g, 0, 0, k), size_t(g.pnx) * 4,
                                  src + size_t(k) * g.ny * g.nx, size_t(g.nx) * 4,
                                  size_t(g.nx) * 4, g.ny, kind, ws->stream),
                "copy into the padded field");
    }
    return src2 ? copy_in(ws, dst2, src2, on_device) : WS_OK;
}

int copy_out(ws_t ws, float *dst, const float *src, int on_device, float *dst2, const float *src2) {
    const ws::Geom &g = ws->g;
    const size_t n = size_t(g.nx) * g.ny * g.nz;
    if (on_device && kernel_copyable(ws, dst) && kernel_copyable(ws, dst2)) {
        // outputs that overlap get their copies one after the other
        const bool both = src2 && (dst2 >= dst + n || dst >= dst2 + n);
        WS_CUDA(ws::launch_copy_out(src, both ? src2 : nullptr, dst, both ? dst2 : nullptr, g,
                                    ws->stream),
                "copy out of the padded field");
        ws->launches++;
        return src2 && !both ? copy_out(ws, dst2, src2, on_device) : WS_OK;
    }
    // one plane of long rows comes out in one 2D copy (512 x 512: 22 us, through the
    // staging 31; 30 x 60000: 268, 62)
    const bool direct = on_device || (g.nz == 1 && g.nx >= 256);
    int planes = 0;
    if (float *stage = direct ? nullptr : host_stage(ws, &planes)) {
        const size_t plane = size_t(g.nx) * g.ny;
        for (int k = 0; k < g.nz; k += planes) {
            ws::Geom part = g;
            part.nz = std::min(planes, g.nz - k);
            WS_CUDA(ws::launch_copy_out(src + k * g.plane, nullptr, stage, nullptr, part, ws->stream),
                    "copy out of the padded field");
            ws->launches++;
            WS_CUDA(cudaMemcpyAsync(dst + k * plane, stage, sizeof(float) * plane * part.nz,
                                    cudaMemcpyDeviceToHost, ws->stream),
                    "copy out of the padded field");
        }
        return src2 ? copy_out(ws, dst2, src2, on_device) : WS_OK;
    }
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    for (int k = 0; k < g.nz; ++k) {
        WS_CUDA(cudaMemcpy2DAsync(dst + size_t(k) * g.ny * g.nx, size_t(g.nx) * 4,
                                  src + ws::pidx(g, 0, 0, k), size_t(g.pnx) * 4,
                                  size_t(g.nx) * 4, g.ny, kind, ws->stream),
                "copy out of the padded field");
    }
    return src2 ? copy_out(ws, dst2, src2, on_device) : WS_OK;
}

// Whole fields (padding included) to zero: a, and b if not null, by one kernel, or
// large ones, which a memset writes faster, by memsets (two of 460 MB: 134 us, the
// kernel 144; of 100 MB: 41.4, 40.3).
int zero_fields(ws_t ws, float *a, float *b, size_t bytes, const char *what) {
    constexpr size_t kMemset = 128u << 20;
    if (bytes <= kMemset) {
        WS_CUDA(ws::launch_zero(a, b, bytes, ws->stream), what);
        ws->launches++;
        return WS_OK;
    }
    WS_CUDA(cudaMemsetAsync(a, 0, bytes, ws->stream), what);
    if (b) WS_CUDA(cudaMemsetAsync(b, 0, bytes, ws->stream), what);
    return WS_OK;
}

int upload_profiles(ws_t ws) {
    const ws::Geom &g = ws->g;
    std::vector<float> px(g.nx), py(g.ny), pz(g.nz);
    for (int i = 0; i < g.nx; ++i) px[i] = (float)taper(i, g.nx, ws->nb, ws->a);
    for (int j = 0; j < g.ny; ++j) py[j] = (float)taper(j, g.ny, ws->nb, ws->a);
    for (int k = 0; k < g.nz; ++k) pz[k] = (float)taper(k, g.nz, ws->nb, ws->a);
    // the cells of each axis whose factor is exactly 1 (a contiguous middle
    // range: the profile rises monotonically from both faces)
    auto ones = [](const std::vector<float> &p, int *lo, int *hi) {
        const int n = (int)p.size();
        int a = 0;
        while (a < n && p[a] != 1.0f) ++a;
        int b = a;
        while (b < n && p[b] == 1.0f) ++b;
        *lo = a;
        *hi = b;
    };
    ones(px, &ws->free_box.x0, &ws->free_box.x1);
    ones(py, &ws->free_box.y0, &ws->free_box.y1);
    ones(pz, &ws->free_box.z0, &ws->free_box.z1);
    WS_CUDA(cudaMemcpyAsync(ws->gx, px.data(), 4 * px.size(), cudaMemcpyHostToDevice, ws->stream),
            "upload taper");
    WS_CUDA(cudaMemcpyAsync(ws->gy, py.data(), 4 * py.size(), cudaMemcpyHostToDevice, ws->stream),
            "upload taper");
    WS_CUDA(cudaMemcpyAsync(ws->gz, pz.data(), 4 * pz.size(), cudaMemcpyHostToDevice, ws->stream),
            "upload taper");
    WS_CUDA(cudaStreamSynchronize(ws->stream), "upload taper");
    return WS_OK;
}

int encode_maps16(ws_t ws, int ty) {
    const ws::Geom &g = ws->g;
    int rc = WS_OK;
    for (int b = 0; b < 2 && rc == WS_OK; ++b)
        rc = encode_map(&ws->t16_halo[b], ws->buf16[b], g, kTile16X + 16, ty + 2 * ws::kHalo, 2);
    if (rc == WS_OK) rc = encode_map(&ws->t16_d, ws->d16, g, kTile16X, ty, 2);
    if (rc == WS_OK) rc = encode_map(&ws->t16_w, ws->w16, g, kTile16X, ty, 2);
    ws->t16_ty = rc == WS_OK ? ty : 0;
    return rc;
}

// A tile height of the 16-bit kernel for this grid: the one ws_set_kernel chose
// if the grid holds it, else the first of kTile16Ys that the grid holds (0:
// none).
int pick_tile16(const ws_t ws) {
    if (ws->tile16_y > 0 && ws->g.ny >= ws->tile16_y) return ws->tile16_y;
    for (int ty : kTile16Ys)
        if (ws->g.ny >= ty) return ty;
    return 0;
}

// Tile height and planes per work item of the 16-bit kernel's next steps: what
// was chosen, the rest of the smallest estimated step (an SM holds 48 rows of
// either height, so the estimates compare; see best_zblock).
ws::StreamTiling pick_tiling16(ws_t ws) {
    const int fixed = pick_tile16(ws);
    ws::StreamTiling t{kTile16X, fixed, ws->tiling.zb};
    if (t.zb > 0) return t;
    const bool chosen = ws->tile16_y == fixed;
    ws::StreamTiling &kept = ws->auto16;
    if (kept.zb > 0 && (kept.ty == fixed || !chosen) && ws->auto16_chosen == chosen) return kept;
    double best = 0.0;
    for (int ty : kTile16Ys) {
        if (chosen) ty = fixed;
        int slots = 0, sms = 0;
        if (ws->g.ny < ty || ws::stream16_slots(ty, &slots, &sms) != cudaSuccess) continue;
        const long long tiles =
            (long long)((ws->g.nx + kTile16X - 1) / kTile16X) * ((ws->g.ny + ty - 1) / ty);
        double cost = 0.0;
        const int zb = best_zblock(ws->g.nz, tiles, slots, sms, kModel16, &cost);
        if (t.zb <= 0 || cost < best) {
            best = cost;
            t.ty = ty;
            t.zb = zb;
        }
    }
    if (t.zb <= 0) t.zb = default_zblock(ws->g.nz);
    kept = t;
    ws->auto16_chosen = chosen;
    return t;
}

// FP32 levels (the handle's buffers, or device arrays) -> the 16-bit state
// (U = u^n, D = u^n - u^{n-1}), exponents in the step's slot.
int encode_state16(ws_t ws, const ws::Fp32Fields &f) {
    const int sn = (int)(ws->step & 3), so = (int)((ws->step + 1) & 3);
    WS_CUDA(ws::launch_encode16(ws->storage, f, ws->buf16[ws->cur], ws->d16, ws->g, ws->scale, sn,
                                ws->stream),
            "encode field");
    // the next step accumulates max |u^{n+1}| into slot (step + 1) & 3
    WS_CUDA(cudaMemsetAsync(&ws->scale->amax[so], 0, sizeof(unsigned), ws->stream), "encode field");
    ws->launches += 2;
    return WS_OK;
}

int encode_state16(ws_t ws) {
    const float *un = ws->buf[ws->cur], *um = ws->buf[1 - ws->cur];
    return encode_state16(ws, ws::padded_pair(un, um, ws->g));
}

// The 16-bit state -> FP32 levels.
int decode_state16(ws_t ws, const ws::Fp32Out &f) {
    const int sn = (int)(ws->step & 3);
    WS_CUDA(ws::launch_decode16(ws->storage, ws->buf16[ws->cur], ws->d16, f, ws->g, ws->scale, sn,
                                ws->stream),
            "decode field");
    ws->launches += 1;
    return WS_OK;
}

int decode_state16(ws_t ws) {
    return decode_state16(ws, ws::padded_pair(ws->buf[ws->cur], ws->buf[1 - ws->cur], ws->g));
}

// Point sources of step n: (V_s dt)^2 s(t_n) is added at each source cell,
// i.e. amp = h^2 s(t_n) times the stored (V dt / h)^2.
void sources_of_step(const ws_t ws, long long n, ws::Sources *out) {
    out->n = (int)ws->src.size();
    const double t = double(n) * ws->dt;
    for (int q = 0; q < out->n; ++q) {
        const SourceDef &d = ws->src[q];
        out->s[q] = ws::SourceSample{d.i, d.j, d.k,
                                     (float)(ws->h * ws->h * ricker(t, d.f0, d.t0, d.amp))};
    }
}

// Step arguments common to every step of the handle's model.
ws::StepArgs base_args(const ws_t ws) {
    ws::StepArgs a{};
    a.stall_item = -1;
    a.g = ws->g;
    a.c.c1 = (float)kW1;
    a.c.c2 = (float)kW2;
    a.c.c3 = (float)kW3;
    a.c.c4 = (float)kW4;
    a.gx = ws->gx;
    a.gy = ws->gy;
    a.gz = ws->gz;
    a.fr = ws->free_box;
    a.traces = ws->traces;
    a.nt_max = ws->nt_max;
    a.status = ws->status;
    return a;
}

// One FP32 step of the handle's model (Eq. 1 discretised): out = u^{n+1}
// from un = u^n (with its halo box map) and unm1 = u^{n-1} (with its tile box
// map); out may be unm1. Adds the sources of step n when `sources`, records
// the receivers' trace column n - trace_start when `record` (with a.inject: adds
// the residual of that column there instead).
int step_fp32(ws_t ws, ws::StepArgs &a, int kern, const ws::StreamTiling &tiling, const float *un,
              const CUtensorMap *un_halo, const float *unm1, const CUtensorMap *unm1_tile,
              float *out, long long n, bool sources, bool record) {
    if (sources)
        sources_of_step(ws, n, &a.src);
    else
        a.src.n = 0;
    a.trace_step = n - ws->trace_start;
    cudaError_t e;
    if (kern == WS_KERNEL_STREAM) {
        e = ws::launch_step_stream(un_halo, unm1_tile, &ws->tmap_w, un, out, a, tiling,
                                   record ? ws->rec_ptr : nullptr, ws->rec_entries, ws->stream);
        ws->launches++;
    } else {
        e = ws::launch_step_direct(un, unm1, out, ws->w, a, record ? ws->rec_ptr : nullptr,
                                   ws->rec_planes, ws->rec_entries, ws->stream);
        ws->launches++;
    }
    if (e != cudaSuccess) return cuda_fail(e, "step launch");
    return WS_OK;
}

// Select the FP32 kernel for the next steps and bring the tensor maps and
// the receiver table in line with its tiling.
int prepare_fp32(ws_t ws, int *kern, ws::StreamTiling *tiling) {
    *kern = pick_kernel(ws, tiling);
    if (*kern != WS_KERNEL_STREAM)
        return build_rec_tiles(ws, ws::StreamTiling{ws::kDirectX, ws::kDirectY, 0}, true, ws->stream);
    if (tiling->tx != ws->tiling.tx || tiling->ty != ws->tiling.ty) {
        ws->tiling.tx = tiling->tx;
        ws->tiling.ty = tiling->ty;
        int rc = encode_maps(ws);
        if (rc != WS_OK) return rc;
    }
    return build_rec_tiles(ws, *tiling, false, ws->stream);
}

void destroy(ws_t ws) {
    if (!ws) return;
    cudaStreamSynchronize(ws->stream);
    cudaFree(ws->buf[0]);
    cudaFree(ws->buf[1]);
    cudaFree(ws->w);
    cudaFree(ws->gx);
    cudaFree(ws->gy);
    cudaFree(ws->gz);
    cudaFree(ws->status);
    cudaFree(ws->energy);
    cudaFree(ws->buf16[0]);
    cudaFree(ws->buf16[1]);
    cudaFree(ws->d16);
    cudaFree(ws->w16);
    cudaFree(ws->scale);
    cudaFree(ws->stage);
    free_receivers(ws);
    delete ws->adj;
    delete ws;
}

}  // namespace wsh

using namespace wsh;

namespace {

// Padding canaries (test hooks). A padded field is the interior, the 4-cell
// zero halo around it, and the row padding beyond the halo in x; no kernel
// may write outside the interior, and nothing read beyond the halo may reach
// a result.
__device__ __forceinline__ int pad_class(const ws::Geom &g, long long idx) {
    const int x = (int)(idx % g.pnx);
    const long long r = idx / g.pnx;
    const int y = (int)(r % g.pny), z = (int)(r / g.pny);
    const bool ix = x >= ws::kXOff && x < ws::kXOff + g.nx;
    const bool iy = y >= ws::kHalo && y < g.ny + ws::kHalo;
    const bool iz = z >= ws::kHalo && z < g.nz + ws::kHalo;
    if (ix && iy && iz) return 0;                                     // interior
    const bool hx = x >= ws::kXOff - ws::kHalo && x < ws::kXOff + g.nx + ws::kHalo;
    return (hx && y < g.ny + 2 * ws::kHalo && z < g.nz + 2 * ws::kHalo) ? 1 : 2;   // halo : padding
}

template <class T>
__global__ void fill_pad_kernel(T *f, ws::Geom g, T canary) {
    const long long n = (long long)g.pnx * g.pny * g.pnz;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x)
        if (pad_class(g, idx) == 2) f[idx] = canary;
}

// Cells that differ from what they must hold: 0 in the halo, the canary in
// the padding (bit patterns).
template <class T>
__global__ void check_pad_kernel(const T *f, ws::Geom g, T canary, unsigned long long *bad) {
    const long long n = (long long)g.pnx * g.pny * g.pnz;
    unsigned long long c = 0;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int k = pad_class(g, idx);
        if ((k == 1 && f[idx] != T(0)) || (k == 2 && f[idx] != canary)) ++c;
    }
    if (c) atomicAdd(bad, c);
}

constexpr uint32_t kCanary32 = 0x7fc00000u;   // FP32 quiet NaN
constexpr uint16_t kCanaryF16 = 0x7e00u;      // FP16 quiet NaN
constexpr uint16_t kCanaryBf16 = 0x7fc0u;     // BF16 quiet NaN

// Every field buffer of the handle with its canary: the FP32 state and
// model, and with 16-bit storage the 16-bit state and model too.
template <class F>
int for_each_field(ws_t ws, F &&fn) {
    const uint16_t c16 = ws->storage == WS_STORAGE_BF16 ? kCanaryBf16 : kCanaryF16;
    for (float *f : {ws->buf[0], ws->buf[1], ws->w}) {
        int rc = fn(reinterpret_cast<uint32_t *>(f), kCanary32);
        if (rc != WS_OK) return rc;
    }
    if (ws->storage != WS_STORAGE_FP32) {
        for (uint16_t *f : {ws->buf16[0], ws->buf16[1], ws->d16}) {
            int rc = fn(f, c16);
            if (rc != WS_OK) return rc;
        }
        return fn(ws->w16, kCanaryF16);
    }
    return WS_OK;
}

constexpr int kPadGrid = 1216, kPadBlock = 256;

}  // namespace

extern "C" {

const char *ws_last_error(void) { return g_err; }

int ws_create(ws_t *out, int nx, int ny, int nz, double h, double dt) {
    if (!out) return fail(WS_ERR_BADARG, "ws_create: out is NULL");
    *out = nullptr;
    if (nx < 1 || ny < 1 || nz < 1 || nx > 65535 || ny > 65535 || nz > 65535)
        return fail(WS_ERR_BADARG, "ws_create: sizes must be in [1, 65535], got %d x %d x %d", nx,
                    ny, nz);
    if (!(h > 0.0) || !(dt > 0.0) || !std::isfinite(h) || !std::isfinite(dt))
        return fail(WS_ERR_BADARG, "ws_create: h and dt must be finite and > 0");
    ws_t ws = new (std::nothrow) ws_handle();
    if (!ws) return fail(WS_ERR_OOM, "ws_create: host allocation failed");
    ws::Geom &g = ws->g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.pnx = (ws::kXOff + nx + ws::kHalo + ws::kRowAlign - 1) / ws::kRowAlign * ws::kRowAlign;
    g.pny = ny + 2 * ws::kHalo;
    g.pnz = nz + 2 * ws::kHalo;
    g.plane = (long long)g.pnx * g.pny;
    ws->h = h;
    ws->dt = dt;
    const size_t fb = field_bytes(g);
    cudaError_t e = cudaSuccess;
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = cudaMalloc(&ws->buf[b], fb);
    if (e == cudaSuccess) e = cudaMalloc(&ws->w, fb);
    if (e == cudaSuccess) e = cudaMalloc(&ws->gx, sizeof(float) * nx);
    if (e == cudaSuccess) e = cudaMalloc(&ws->gy, sizeof(float) * ny);
    if (e == cudaSuccess) e = cudaMalloc(&ws->gz, sizeof(float) * nz);
    if (e == cudaSuccess) e = cudaMalloc(&ws->status, sizeof(unsigned) * 4);
    if (e == cudaSuccess)
        e = cudaMalloc(&ws->energy, sizeof(double) * (ws::energy_partial_count(ny, nz) + 1));
    for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = cudaMemsetAsync(ws->buf[b], 0, fb, ws->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws->w, 0, fb, ws->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws->status, 0, sizeof(unsigned) * 4, ws->stream);
    if (e != cudaSuccess) {
        destroy(ws);
        return cuda_fail(e, "ws_create");
    }
    int rc = upload_profiles(ws);
    if (rc == WS_OK) rc = encode_maps(ws);
    if (rc == WS_OK && (e = cudaStreamSynchronize(ws->stream)) != cudaSuccess)
        rc = cuda_fail(e, "ws_create");
    if (rc != WS_OK) {
        destroy(ws);
        return rc;
    }
    *out = ws;
    return WS_OK;
}

int ws_destroy(ws_t ws) {
    destroy(ws);
    return WS_OK;
}

int ws_set_stream(ws_t ws, void *cuda_stream) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_set_stream: NULL handle");
    WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_set_stream");
    ws->stream = static_cast<cudaStream_t>(cuda_stream);
    return WS_OK;
}

int ws_set_velocity(ws_t ws, const float *v, int on_device) {
    if (!ws || !v) return fail(WS_ERR_BADARG, "ws_set_velocity: NULL argument");
    ws->model_version++;
    ws->vel_ok = false;
    const bool direct = on_device && kernel_copyable(ws, v);
    if (!direct) {
        int rc = copy_in(ws, ws->w, v, on_device);
        if (rc != WS_OK) return rc;
    }
    static const unsigned init[2] = {0u, 0x7f800000u};
    WS_CUDA(cudaMemcpyAsync(ws->status + 1, init, sizeof init, cudaMemcpyHostToDevice, ws->stream),
            "ws_set_velocity");
    WS_CUDA(ws::launch_velocity_to_w(direct ? v : nullptr, ws->w, ws->g, ws->dt / ws->h,
                                     ws->status + 1, ws->stream),
            "velocity conversion kernel");
    ws->launches++;
    unsigned ext[2];
    WS_CUDA(cudaMemcpyAsync(ext, ws->status + 1, sizeof ext, cudaMemcpyDeviceToHost, ws->stream),
            "ws_set_velocity");
    WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_set_velocity");
    float vmax, vmin;
    std::memcpy(&vmax, &ext[0], 4);
    std::memcpy(&vmin, &ext[1], 4);
    if (ext[1] == 0u) return fail(WS_ERR_BADARG, "ws_set_velocity: every value must be finite and > 0");
    const double c = double(vmax) * ws->dt / ws->h;
    if (c > cfl_limit())
        return fail(WS_ERR_CFL, "ws_set_velocity: max(V) dt / h = %.6f exceeds the limit %.6f", c,
                    cfl_limit());
    ws->wmax = c * c;
    ws->vel_ok = true;
    ws->w16_ok = false;
    return WS_OK;
}

int ws_set_slowness2(ws_t ws, const float *m, int on_device) {
    if (!ws || !m) return fail(WS_ERR_BADARG, "ws_set_slowness2: NULL argument");
    ws->model_version++;
    ws->vel_ok = false;
    const bool direct = on_device && kernel_copyable(ws, m);
    if (!direct) {
        int rc = copy_in(ws, ws->w, m, on_device);
        if (rc != WS_OK) return rc;
    }
    static const unsigned init[2] = {0u, 0x7f800000u};
    WS_CUDA(cudaMemcpyAsync(ws->status + 1, init, sizeof init, cudaMemcpyHostToDevice, ws->stream),
            "ws_set_slowness2");
    const double r = ws->dt / ws->h;
    WS_CUDA(ws::launch_slowness2_to_w(direct ? m : nullptr, ws->w, ws->g, r * r, ws->status + 1,
                                      ws->stream),
            "slowness conversion kernel");
    ws->launches++;
    unsigned ext[2];
    WS_CUDA(cudaMemcpyAsync(ext, ws->status + 1, sizeof ext, cudaMemcpyDeviceToHost, ws->stream),
            "ws_set_slowness2");
    WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_set_slowness2");
    float mmin;
    std::memcpy(&mmin, &ext[1], 4);
    if (ext[1] == 0u)
        return fail(WS_ERR_BADARG, "ws_set_slowness2: every value must be finite and > 0");
    const double c = ws->dt / (ws->h * std::sqrt(double(mmin)));   // max V dt / h
    if (c > cfl_limit())
        return fail(WS_ERR_CFL, "ws_set_slowness2: max(V) dt / h = %.6f exceeds the limit %.6f", c,
                    cfl_limit());
    ws->wmax = c * c;
    ws->vel_ok = true;
    ws->w16_ok = false;
    return WS_OK;
}

int ws_set_sponge(ws_t ws, int nb, double a) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_set_sponge: NULL handle");
    if (nb < 0 || !(a >= 0.0) || !std::isfinite(a))
        return fail(WS_ERR_BADARG, "ws_set_sponge: need nb >= 0 and finite a >= 0");
    ws->nb = nb;
    ws->a = a;
    ws->model_version++;
    return upload_profiles(ws);
}

int ws_add_source(ws_t ws, int ix, int iy, int iz, double f0, double t0, double amp) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_add_source: NULL handle");
    const ws::Geom &g = ws->g;
    if (ix < 0 || ix >= g.nx || iy < 0 || iy >= g.ny || iz < 0 || iz >= g.nz)
        return fail(WS_ERR_BADARG, "ws_add_source: cell (%d, %d, %d) outside the grid", ix, iy, iz);
    if (!(f0 > 0.0) || !std::isfinite(f0) || !std::isfinite(t0) || !std::isfinite(amp))
        return fail(WS_ERR_BADARG, "ws_add_source: need finite t0, amp and f0 > 0");
    if ((int)ws->src.size() >= ws::kMaxSources)
        return fail(WS_ERR_BADARG, "ws_add_source: at most %d sources", ws::kMaxSources);
    ws->src.push_back({ix, iy, iz, f0, t0, amp});
    ws->model_version++;
    return WS_OK;
}

int ws_clear_sources(ws_t ws) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_clear_sources: NULL handle");
    ws->src.clear();
    ws->model_version++;
    return WS_OK;
}

int ws_set_receivers(ws_t ws, int nrec, const int *ijk, int nt_max) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_set_receivers: NULL handle");
    if (nrec < 0 || (nrec > 0 && (!ijk || nt_max < 1)))
        return fail(WS_ERR_BADARG, "ws_set_receivers: need nrec >= 0, ijk and nt_max >= 1");
    const ws::Geom &g = ws->g;
    for (int r = 0; r < nrec; ++r) {
        const int i = ijk[3 * r], j = ijk[3 * r + 1], k = ijk[3 * r + 2];
        if (i < 0 || i >= g.nx || j < 0 || j >= g.ny || k < 0 || k >= g.nz)
            return fail(WS_ERR_BADARG, "ws_set_receivers: receiver %d at (%d, %d, %d) outside the grid",
                        r, i, j, k);
    }
    if (nrec > 0 && (long long)nrec * nt_max > (1ll << 40))
        return fail(WS_ERR_BADARG, "ws_set_receivers: trace buffer too large");
    int rc = refuse_capture(ws, "ws_set_receivers");
    if (rc != WS_OK) return rc;
    ws->model_version++;
    ws->nrec = 0;
    ws->nt_max = 0;
    forget_rec_tiles(ws);   // the table is another one
    ws->rec_ijk.assign(ijk, ijk + 3 * size_t(nrec));
    ws->trace_start = ws->step;
    if (nrec == 0) {
        WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_set_receivers");
        free_receivers(ws);
        return WS_OK;
    }
    // buffers that are large enough stay: the clearing is ordered after the work
    // that still uses them
    const size_t bytes = sizeof(float) * size_t(nrec) * nt_max;
    void *traces = ws->traces;
    rc = keep_or_grow(ws, &traces, &ws->traces_cap, bytes, "cudaMalloc traces");
    ws->traces = static_cast<float *>(traces);
    if (rc != WS_OK) return rc;
    WS_CUDA(cudaMemsetAsync(ws->traces, 0, bytes, ws->stream), "zero traces");
    ws->nrec = nrec;
    ws->nt_max = nt_max;
    return WS_OK;
}

int ws_set_storage(ws_t ws, int storage) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_set_storage: NULL handle");
    if (storage != WS_STORAGE_FP32 && storage != WS_STORAGE_BF16 && storage != WS_STORAGE_FP16)
        return fail(WS_ERR_BADARG, "ws_set_storage: unknown storage %d", storage);
    if (storage == ws->storage) return WS_OK;
    ws->model_version++;
    if (storage != WS_STORAGE_FP32 && (ws->g.nx < kTile16X || pick_tile16(ws) == 0))
        return fail(WS_ERR_BADARG,
                    "ws_set_storage: 16-bit storage needs nx >= %d and ny >= %d (grid %d x %d)",
                    kTile16X, kTile16Ys[kNumTile16Ys - 1], ws->g.nx, ws->g.ny);
    // bring the state to FP32 first
    if (ws->storage != WS_STORAGE_FP32) {
        int rc = decode_state16(ws);
        if (rc != WS_OK) return rc;
    }
    if (storage != WS_STORAGE_FP32) {
        const size_t hb = size_t(ws->g.pnx) * ws->g.pny * ws->g.pnz * sizeof(uint16_t);
        for (uint16_t **f : {&ws->buf16[0], &ws->buf16[1], &ws->d16, &ws->w16})
            if (!*f) {
                void *q = nullptr;
                WS_CUDA(handle_malloc(ws, &q, hb), "cudaMalloc 16-bit field");
                *f = static_cast<uint16_t *>(q);
                WS_CUDA(cudaMemsetAsync(*f, 0, hb, ws->stream), "zero 16-bit field");
            }
        ws->w16_ok = false;
        if (!ws->scale) {
            WS_CUDA(cudaMalloc(&ws->scale, sizeof(ws::Scale16)), "cudaMalloc scales");
            WS_CUDA(cudaMemsetAsync(ws->scale, 0, sizeof(ws::Scale16), ws->stream), "zero scales");
        }
        int rc = encode_maps16(ws, pick_tile16(ws));
        if (rc != WS_OK) return rc;
        ws->storage = storage;
        rc = encode_state16(ws);
        if (rc != WS_OK) return rc;
    } else {
        ws->storage = storage;
    }
    return WS_OK;
}

int ws_set_kernel(ws_t ws, int kernel, int tile_x, int tile_y, int zblock) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_set_kernel: NULL handle");
    if (kernel != WS_KERNEL_AUTO && kernel != WS_KERNEL_DIRECT && kernel != WS_KERNEL_STREAM)
        return fail(WS_ERR_BADARG, "ws_set_kernel: unknown kernel %d", kernel);
    if (zblock < 0) return fail(WS_ERR_BADARG, "ws_set_kernel: zblock must be >= 0");
    // the streaming tile that must fit: the chosen one, else 64 x 8, or on a
    // narrower grid that AUTO has stepped the tile it took
    ws::StreamTiling t = ws->tile_chosen ? ws->tiling : ws->need;
    bool chosen = ws->tile_chosen;
    if (tile_x != 0 || tile_y != 0) {
        const bool fp32 = ws::stream_tiling_supported(tile_x, tile_y);
        const bool t16 = ws::stream16_tiling_supported(tile_x, tile_y);
        if (!fp32 && !t16)
            return fail(WS_ERR_BADARG, "ws_set_kernel: unsupported tile %d x %d", tile_x, tile_y);
        if (t16) {   // the 16-bit kernel's tile; the FP32 tile only if that kernel has it too
            if (ws->g.nx < tile_x || ws->g.ny < tile_y)
                return fail(WS_ERR_BADARG,
                            "ws_set_kernel: grid %d x %d is smaller than the tile %d x %d",
                            ws->g.nx, ws->g.ny, tile_x, tile_y);
            ws->tile16_y = tile_y;
        }
        if (fp32) {
            t.tx = tile_x;
            t.ty = tile_y;
            chosen = true;
        }
    }
    t.zb = zblock;
    if (kernel == WS_KERNEL_STREAM && !stream_fits(ws, t))
        return fail(WS_ERR_BADARG, "ws_set_kernel: grid %d x %d is smaller than the tile %d x %d",
                    ws->g.nx, ws->g.ny, t.tx, t.ty);
    ws->kernel = kernel;
    ws->tiling.zb = zblock;
    if (!chosen) return WS_OK;   // the step picks the tile
    const bool box_changed = t.tx != ws->tiling.tx || t.ty != ws->tiling.ty;
    ws->tiling = t;
    ws->tile_chosen = true;
    if (box_changed) return encode_maps(ws);
    return WS_OK;
}

int ws_step(ws_t ws, int nsteps) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_step: NULL handle");
    if (nsteps < 0) return fail(WS_ERR_BADARG, "ws_step: nsteps must be >= 0");
    if (!ws->vel_ok) return fail(WS_ERR_STATE, "ws_step: no valid velocity model");
    if (ws->nrec > 0) {
        const long long col = ws->step - ws->trace_start;
        if (col < 0 || col + nsteps > ws->nt_max)
            return fail(WS_ERR_STATE,
                        "ws_step: receivers hold %d steps from step %lld; cannot record steps "
                        "%lld..%lld",
                        ws->nt_max, ws->trace_start, ws->step, ws->step + nsteps - 1);
    }
    ws::StreamTiling tiling{};
    int kern = WS_KERNEL_STREAM;
    if (ws->storage != WS_STORAGE_FP32) {
        tiling = pick_tiling16(ws);
        if (tiling.ty != ws->t16_ty) {
            int rc = encode_maps16(ws, tiling.ty);
            if (rc != WS_OK) return rc;
        }
        int rc = build_rec_tiles(ws, tiling, false, ws->stream);
        if (rc != WS_OK) return rc;
        if (!ws->w16_ok) {
            WS_CUDA(ws::launch_model16(ws->w, ws->w16, ws->g, ws->stream), "16-bit model");
            ws->launches++;
            ws->w16_ok = true;
        }
    } else {
        int rc = prepare_fp32(ws, &kern, &tiling);
        if (rc != WS_OK) return rc;
    }
    ws::StepArgs a = base_args(ws);
    for (int s = 0; s < nsteps; ++s) {
        if (ws->storage != WS_STORAGE_FP32) {
            sources_of_step(ws, ws->step, &a.src);
            a.trace_step = ws->step - ws->trace_start;
            double hint = 0.0;
            for (int q = 0; q < a.src.n; ++q)
                hint = std::max(hint, std::fabs((double)a.src.s[q].amp) * ws->wmax);
            a.stall_item = ws->stall_item;
            ws->stall_item = -1;
            const ws::Maps16In maps{&ws->t16_halo[ws->cur], &ws->t16_d, &ws->t16_w,
                                    ws->buf16[1 - ws->cur], ws->d16};
            cudaError_t e = ws::launch_step_stream16(
                ws->storage, maps, a, ws->scale, ws->step, (float)hint, tiling,
                ws->nrec > 0 ? ws->rec_ptr : nullptr, ws->rec_entries, ws->stream);
            a.stall_item = -1;
            ws->launches++;
            if (e != cudaSuccess) return cuda_fail(e, "ws_step launch");
        } else {
            const int c = ws->cur;
            a.stall_item = kern == WS_KERNEL_STREAM ? ws->stall_item : -1;
            ws->stall_item = -1;
            int rc = step_fp32(ws, a, kern, tiling, ws->buf[c], &ws->tmap_halo[c], ws->buf[1 - c],
                               &ws->tmap_tile[1 - c], ws->buf[1 - c], ws->step, true,
                               ws->nrec > 0);
            a.stall_item = -1;
            if (rc != WS_OK) return rc;
        }
        ws->cur = 1 - ws->cur;
        ws->step++;
    }
    return WS_OK;
}

int ws_read_traces(ws_t ws, float *out, int on_device) {
    if (!ws || !out) return fail(WS_ERR_BADARG, "ws_read_traces: NULL argument");
    if (ws->nrec == 0) return WS_OK;
    WS_CUDA(cudaMemcpyAsync(out, ws->traces, sizeof(float) * size_t(ws->nrec) * ws->nt_max,
                            on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                            ws->stream),
            "ws_read_traces");
    if (!on_device) WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_read_traces");
    return WS_OK;
}

int ws_read_field(ws_t ws, float *u, float *u_prev, int on_device) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_read_field: NULL handle");
    int rc = WS_OK;
    if (ws->storage != WS_STORAGE_FP32) {
        if (on_device && kernel_copyable(ws, u) && kernel_copyable(ws, u_prev)) {
            // straight into the caller's arrays; outputs that overlap one
            // after the other
            const size_t n = size_t(ws->g.nx) * ws->g.ny * ws->g.nz;
            const bool both = !u || !u_prev || u_prev >= u + n || u >= u_prev + n;
            if (both) return decode_state16(ws, ws::dense_pair(u, u_prev, ws->g));
            rc = decode_state16(ws, ws::dense_pair<float>(u, nullptr, ws->g));
            if (rc == WS_OK) rc = decode_state16(ws, ws::dense_pair<float>(nullptr, u_prev, ws->g));
            return rc;
        }
        rc = decode_state16(ws);
        if (rc != WS_OK) return rc;
    }
    const float *un = ws->buf[ws->cur], *um = ws->buf[1 - ws->cur];
    if (u)
        rc = copy_out(ws, u, un, on_device, u_prev, u_prev ? um : nullptr);
    else if (u_prev)
        rc = copy_out(ws, u_prev, um, on_device);
    if (rc != WS_OK) return rc;
    if (!on_device) WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_read_field");
    return WS_OK;
}

int ws_write_field(ws_t ws, const float *u, const float *u_prev, long long step, int on_device) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_write_field: NULL handle");
    if (step < 0) return fail(WS_ERR_BADARG, "ws_write_field: step must be >= 0");
    if (ws->storage != WS_STORAGE_FP32 && on_device && (u || u_prev) && kernel_copyable(ws, u) &&
        kernel_copyable(ws, u_prev)) {
        ws->step = step;   // straight from the caller's arrays
        return encode_state16(ws, ws::dense_pair(u, u_prev, ws->g));
    }
    // everything outside the interior is zero from the start and stays so:
    // only a missing level needs its buffer cleared
    const size_t fb = field_bytes(ws->g);
    float *un = ws->buf[ws->cur], *um = ws->buf[1 - ws->cur];
    if (!u || !u_prev) {
        float *first = u ? um : un, *second = u || u_prev ? nullptr : um;
        const int zc = zero_fields(ws, first, second, fb, "ws_write_field");
        if (zc != WS_OK) return zc;
    }
    int rc = WS_OK;
    if (u)
        rc = copy_in(ws, un, u, on_device, u_prev ? um : nullptr, u_prev);
    else if (u_prev)
        rc = copy_in(ws, um, u_prev, on_device);
    if (rc != WS_OK) return rc;
    ws->step = step;
    if (ws->storage != WS_STORAGE_FP32) {
        rc = encode_state16(ws);
        if (rc != WS_OK) return rc;
    }
    if (!on_device) WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_write_field");
    return WS_OK;
}

int ws_get_step(ws_t ws, long long *step) {
    if (!ws || !step) return fail(WS_ERR_BADARG, "ws_get_step: NULL argument");
    *step = ws->step;
    return WS_OK;
}

int ws_synchronize(ws_t ws) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_synchronize: NULL handle");
    WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_synchronize");
    unsigned st = 0;
    WS_CUDA(cudaMemcpy(&st, ws->status, sizeof st, cudaMemcpyDeviceToHost), "ws_synchronize");
    if (st & ws::kStatusTimeout) {
        WS_CUDA(cudaMemset(ws->status, 0, sizeof(unsigned)), "ws_synchronize");
        return fail(WS_ERR_TIMEOUT, "a bounded device wait ran out in a step kernel");
    }
    return WS_OK;
}

int ws_energy(ws_t ws, double *e) {
    if (!ws || !e) return fail(WS_ERR_BADARG, "ws_energy: NULL argument");
    if (!ws->vel_ok) return fail(WS_ERR_STATE, "ws_energy: no valid velocity model");
    if (ws->storage != WS_STORAGE_FP32) {
        int rc = decode_state16(ws);
        if (rc != WS_OK) return rc;
    }
    const ws::Coeffs64 c{kW0, kW1, kW2, kW3, kW4};
    const long long np = ws::energy_partial_count(ws->g.ny, ws->g.nz);
    WS_CUDA(ws::launch_energy_padded(ws->buf[ws->cur], ws->buf[1 - ws->cur], ws->w, ws->g, ws->h, c,
                                     ws->energy, ws->energy + np, ws->stream),
            "energy kernels");
    ws->launches += 2;
    WS_CUDA(cudaMemcpyAsync(e, ws->energy + np, sizeof(double), cudaMemcpyDeviceToHost, ws->stream),
            "ws_energy");
    WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_energy");
    return WS_OK;
}

int ws_energy_noalloc(const float *u, const float *u_prev, const float *v, int nx, int ny, int nz,
                      double h, double dt, double *e, void *cuda_stream) {
    if (!u || !u_prev || !v || !e) return fail(WS_ERR_BADARG, "ws_energy_noalloc: NULL argument");
    if (nx < 1 || ny < 1 || nz < 1 || nx > 65535 || ny > 65535 || nz > 65535)
        return fail(WS_ERR_BADARG, "ws_energy_noalloc: sizes must be in [1, 65535], got %d x %d x %d",
                    nx, ny, nz);
    if (!(h > 0.0) || !(dt > 0.0) || !std::isfinite(h) || !std::isfinite(dt))
        return fail(WS_ERR_BADARG, "ws_energy_noalloc: h and dt must be finite and > 0");
    const long long np = ws::energy_partial_count(ny, nz);
    if (np > ws::kNoAllocMaxPartials)
        return fail(WS_ERR_BADARG,
                    "ws_energy_noalloc: %d x %d x %d needs %lld partial sums, ceil(ny/%d)*nz, but "
                    "the static scratch holds %d",
                    nx, ny, nz, np, ws::energy_rows_per_block(), ws::kNoAllocMaxPartials);
    const ws::Coeffs64 c{kW0, kW1, kW2, kW3, kW4};
    WS_CUDA(ws::launch_energy_noalloc(u, u_prev, v, nx, ny, nz, h, dt, c, e,
                                      static_cast<cudaStream_t>(cuda_stream)),
            "ws_energy_noalloc");
    return WS_OK;
}

int ws_test_stall(ws_t ws, int item) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_test_stall: NULL handle");
    if (item < -1) return fail(WS_ERR_BADARG, "ws_test_stall: item must be >= -1");
    ws->stall_item = item;
    return WS_OK;
}

long long ws_launch_count(ws_t ws) { return ws ? ws->launches : -1; }

int ws_test_fill_padding(ws_t ws) {
    if (!ws) return fail(WS_ERR_BADARG, "ws_test_fill_padding: NULL handle");
    int rc = for_each_field(ws, [&](auto *f, auto canary) {
        using T = std::remove_pointer_t<decltype(f)>;
        cudaError_t e = ws::launch(fill_pad_kernel<T>, kPadGrid, kPadBlock, 0, ws->stream, f, ws->g,
                                   canary);
        ws->launches++;
        return e == cudaSuccess ? WS_OK : cuda_fail(e, "ws_test_fill_padding");
    });
    if (rc != WS_OK) return rc;
    WS_CUDA(cudaStreamSynchronize(ws->stream), "ws_test_fill_padding");
    return WS_OK;
}

int ws_test_check_padding(ws_t ws, long long *bad) {
    if (!ws || !bad) return fail(WS_ERR_BADARG, "ws_test_check_padding: NULL argument");
    unsigned long long *d = nullptr;
    WS_CUDA(cudaMalloc(&d, sizeof *d), "ws_test_check_padding");
    cudaError_t e = cudaMemsetAsync(d, 0, sizeof *d, ws->stream);
    int rc = e == cudaSuccess ? WS_OK : cuda_fail(e, "ws_test_check_padding");
    if (rc == WS_OK)
        rc = for_each_field(ws, [&](auto *f, auto canary) {
            using T = std::remove_pointer_t<decltype(f)>;
            cudaError_t e2 = ws::launch(check_pad_kernel<T>, kPadGrid, kPadBlock, 0, ws->stream, f,
                                        ws->g, canary, d);
            ws->launches++;
            return e2 == cudaSuccess ? WS_OK : cuda_fail(e2, "ws_test_check_padding");
        });
    unsigned long long h = 0;
    if (rc == WS_OK) {
        e = cudaMemcpyAsync(&h, d, sizeof h, cudaMemcpyDeviceToHost, ws->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ws->stream);
        if (e != cudaSuccess) rc = cuda_fail(e, "ws_test_check_padding");
    }
    cudaFree(d);
    if (rc == WS_OK) *bad = (long long)h;
    return rc;
}

}  // extern "C"
