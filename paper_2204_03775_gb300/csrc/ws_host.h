// Host-side internals shared by the translation units of the C ABI
// (include/wavestep.h): the handle, the adjoint scratch and the helpers
// that the core entry points (ws_api.cu), the adjoint driver
// (ws_api_adjoint.cu) and the tuner and batches (ws_api_batch.cu) share.
#pragma once

#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <tuple>
#include <type_traits>
#include <vector>

#include "ws_internal.h"

namespace wsh {

int fail(int code, const char *fmt, ...);
int cuda_fail(cudaError_t e, const char *what);

#define WS_CUDA(call, what)                              \
    do {                                                 \
        cudaError_t e_ = (call);                         \
        if (e_ != cudaSuccess) return wsh::cuda_fail(e_, what); \
    } while (0)

// The 1D weights of the 8th-order second difference, offsets 0..4.
constexpr double kW0 = -205.0 / 72.0, kW1 = 8.0 / 5.0, kW2 = -1.0 / 5.0, kW3 = 8.0 / 315.0,
                 kW4 = -1.0 / 560.0;

// Leapfrog stability limit of V dt / h for the 3D 25-point Laplacian.
double cfl_limit();
// Ricker wavelet amp (1 - 2 a^2) exp(-a^2), a = pi f0 (t - t0).
double ricker(double t, double f0, double t0, double amp);
// Cerjan factor of cell idx on an axis of n cells.
double taper(int idx, int n, int nb, double a);

struct SourceDef {
    int i, j, k;
    double f0, t0, amp;
};

// Host memory of uploads that may run long after the call: two groups of buffers,
// each written again only once the event behind its last upload has passed. An
// event for each upload would cost 2 to 3 us on the way of a call of 27 (a state of
// 96^3 put back, receivers set, one step, the state out); large tables have one.
// All uploads are on streams that are ordered one behind the other.
struct HostTables {
    static constexpr int kGroup = 4;
    static constexpr size_t kLarge = 64 << 10;
    std::vector<char> table[2][kGroup];
    cudaEvent_t passed[2] = {nullptr, nullptr};
    int group = 0, at = 0;
    // The next buffer, of n bytes, free to be written.
    cudaError_t next(size_t n, char **p);
    // That buffer to dst, on `stream`.
    cudaError_t upload(void *dst, cudaStream_t stream);
    // (the uploads are through)
    ~HostTables() {
        for (cudaEvent_t e : passed)
            if (e) cudaEventDestroy(e);
    }
};

// The CUDA driver API's cuTensorMapEncodeTiled (null when unavailable).
PFN_cuTensorMapEncodeTiled_v12000 get_encode_fn();

}  // namespace wsh

struct ws_handle {
    ws::Geom g{};
    double h = 0, dt = 0;
    float *buf[2] = {nullptr, nullptr};  // the two wavefield levels
    int cur = 0;                         // buf[cur] = u^n, buf[1-cur] = u^{n-1}
    float *w = nullptr;                  // (V dt / h)^2, padded
    float *gx = nullptr, *gy = nullptr, *gz = nullptr;
    unsigned *status = nullptr;          // [0] status bits, [1] vmax bits, [2] vmin bits
    double *energy = nullptr;            // energy partial sums, then the total
    cudaStream_t stream = nullptr;
    bool vel_ok = false;
    int nb = 0;
    double a = 0;
    long long step = 0;
    std::vector<wsh::SourceDef> src;

    int nrec = 0, nt_max = 0;
    long long trace_start = 0;
    std::vector<int> rec_ijk;
    float *traces = nullptr;             // [nrec][nt_max] (kept while large enough)
    size_t traces_cap = 0;
    void *rec_table = nullptr;           // rec_ptr, then rec_entries (kept likewise)
    size_t rec_table_cap = 0;
    int *rec_ptr = nullptr;              // per-tile ranges of rec_entries
    ws::RecEntry *rec_entries = nullptr;
    wsh::HostTables rec_host;            // what the table's uploads read
    float *stage = nullptr;              // planes of an unpadded field, for host arrays
    int rec_tiling_tx = 0, rec_tiling_ty = 0;
    bool rec_direct = false;             // the table is the direct kernel's
    int rec_planes = 0;                  // and has this many ranges a tile (0: one)

    int kernel = WS_KERNEL_AUTO;
    ws::StreamTiling tiling{64, 16, 0};  // tile of the tensor maps; zb 0: default
    bool tile_chosen = false;            // by ws_set_kernel, ws_autotune or a batch
    ws::StreamTiling need{64, 8, 0};     // what STREAM must fit while none is chosen
    ws::StreamTiling auto_zb{0, 0, 0};   // default z block of the tile last used
    CUtensorMap tmap_halo[2];  // buf[b] with the (tx+8, ty+8, 1) box
    CUtensorMap tmap_tile[2];  // buf[b] with the (tx, ty, 1) box
    CUtensorMap tmap_w;        // w with the (tx, ty, 1) box
    bool tmap_ok = false;
    long long launches = 0;

    // 16-bit storage (WS_STORAGE_BF16 / WS_STORAGE_FP16): the state lives in
    // buf16[cur] (u^n) and d16 (u^n - u^{n-1}), the model in w16 as well as
    // w; buf then serves as FP32 scratch copies.
    int storage = WS_STORAGE_FP32;
    uint16_t *buf16[2] = {nullptr, nullptr};
    uint16_t *d16 = nullptr, *w16 = nullptr;
    bool w16_ok = false;       // w16 holds the current model
    ws::Scale16 *scale = nullptr;
    CUtensorMap t16_halo[2], t16_d, t16_w;
    double wmax = 0.0;         // max (V dt / h)^2 of the model
    ws::FreeBox free_box{};    // cells whose taper is exactly 1, per axis
    int tile16_y = 0;          // 16-bit tile height chosen by ws_set_kernel (0: default)
    ws::StreamTiling auto16{0, 0, 0};  // the 16-bit tiling a step chose last, and whether
    bool auto16_chosen = false;        // its height was given
    int t16_ty = 0;            // tile height the 16-bit tensor maps are encoded for

    // device scratch of ws_adjoint_gradient, kept for the next call
    struct AdjointCache *adj = nullptr;
    // bumped by every call that changes what a forward run from rest computes
    // (model, taper, sources, receivers, storage)
    unsigned long long model_version = 0;
    int stall_item = -1;       // test hook (ws_test_stall), consumed by the next FP32 step
};

// A padded FP32 field with the streaming kernel's two boxes on it.
struct MappedField {
    float *p = nullptr;
    CUtensorMap halo, tile;
};

// Scratch of ws_adjoint_gradient: checkpoint pairs, the stencil sums of one
// segment, four levels of rho and of recomputed states, the gradient accumulator
// and the trace arrays. Reused while the step count, receivers and tiling stay
// the same.
struct AdjointCache {
    int N = -1, nrec = -1, kern = -1, tx = 0, ty = 0;
    // the checkpoints hold the forward run of this model version (ws_forward)
    bool fwd_valid = false;
    unsigned long long fwd_version = 0;
    std::vector<void *> mem;        // everything below, for cudaFree
    std::vector<MappedField> ck;    // checkpoint j: (u^{jC}, u^{jC-1}), u^m in ck[2 (j-1) + (m & 1)]
    std::vector<float *> lap;       // L u^n of the segment's steps
    // rho^k in level[k % 4], so that four steps can be imaged together. Between
    // two segments only two levels are alive (rho^{n1+1}, rho^{n1+2}; n1 = the
    // next segment's end): the other two hold its recomputed u^n and u^{n-1}.
    MappedField level[ws::kMaxImagingSteps];
    MappedField &rho(int k) { return level[k % ws::kMaxImagingSteps]; }
    static_assert(ws::kMaxImagingSteps == 4, "the two idle levels below");
    MappedField &ring(int n1, int m) { return level[(n1 + 3 + (m & 1)) % ws::kMaxImagingSteps]; }
    float2 *acc = nullptr;          // compensated FP32 gradient sums, padded layout
    double *partials = nullptr;     // residual partial sums, then the misfit
    double *norm = nullptr;         // gradient-norm partial sums, then the norm
    float *r = nullptr, *dd = nullptr, *grad = nullptr;
    ~AdjointCache() {
        for (void *p : mem) cudaFree(p);
    }
};

namespace wsh {

size_t field_bytes(const ws::Geom &g);
// A tensor map of a padded field over its interior (cells outside read as
// zeros) with a (bx, by, 1) box.
int encode_map(CUtensorMap *map, void *base, const ws::Geom &g, int bx, int by,
               int elem_bytes = 4);
// The handle's maps for its current tiling.
int encode_maps(ws_t ws);
bool stream_fits(const ws_t ws, const ws::StreamTiling &t);
// Planes per work item: about 200, and the FP32 streaming kernel's default for a
// grid and tile.
int default_zblock(int nz);
int default_zblock(const ws::Geom &g, int tx, int ty);
// Choose the kernel for the next steps; fills *tiling for the streaming one.
int pick_kernel(ws_t ws, ws::StreamTiling *tiling);
void free_receivers(ws_t ws);
// cudaMalloc that gives back the handle's staging when memory runs out.
cudaError_t handle_malloc(ws_t ws, void **p, size_t n);
// Receiver table of the streaming kernels, or of the direct kernel, for tile t,
// uploaded on `stream` (ordered after the work on the handle's own that may
// still read the old table).
int build_rec_tiles(ws_t ws, const ws::StreamTiling &t, bool direct, cudaStream_t stream);
// Unpadded [nz][ny][nx] user arrays <-> interiors of padded fields, one or
// two fields a call (src2 / dst2 null: one).
int copy_in(ws_t ws, float *dst, const float *src, int on_device, float *dst2 = nullptr,
            const float *src2 = nullptr);
int copy_out(ws_t ws, float *dst, const float *src, int on_device, float *dst2 = nullptr,
             const float *src2 = nullptr);
// Whole fields to zero (b null: one).
int zero_fields(ws_t ws, float *a, float *b, size_t bytes, const char *what);
int upload_profiles(ws_t ws);
// The tiles of the 16-bit streaming kernel (64 x ty) that a step chooses from:
// 24 rows (two CTAs of 6 warps per SM) or 16 (three of 4 warps); 48 is
// selectable with ws_set_kernel (1024^3 about 17 % slower).
constexpr int kTile16X = 64;
constexpr int kTile16Ys[] = {24, 16};
constexpr int kNumTile16Ys = 2;
int pick_tile16(const ws_t ws);
ws::StreamTiling pick_tiling16(ws_t ws);
int encode_maps16(ws_t ws, int ty);
// FP32 levels (by default the handle's buffers) <-> the 16-bit state.
int encode_state16(ws_t ws, const ws::Fp32Fields &f);
int encode_state16(ws_t ws);
int decode_state16(ws_t ws, const ws::Fp32Out &f);
int decode_state16(ws_t ws);
// Point sources of step n (amp = h^2 s(t_n)).
void sources_of_step(const ws_t ws, long long n, ws::Sources *out);
// Step arguments common to every step of the handle's model.
ws::StepArgs base_args(const ws_t ws);
// One FP32 step: out = u^{n+1} from un = u^n and unm1 = u^{n-1} (out may be
// unm1); record: with the receivers (or a.inject at them).
int step_fp32(ws_t ws, ws::StepArgs &a, int kern, const ws::StreamTiling &tiling, const float *un,
              const CUtensorMap *un_halo, const float *unm1, const CUtensorMap *unm1_tile,
              float *out, long long n, bool sources, bool record);
// Select the FP32 kernel and bring maps and receiver table in line with it.
int prepare_fp32(ws_t ws, int *kern, ws::StreamTiling *tiling);
void destroy(ws_t ws);

// Device scratch of one call: freed, after the stream drains, on every return.
struct Scratch {
    ws_t ws;
    std::vector<void *> ptrs;
    explicit Scratch(ws_t w) : ws(w) {}
    ~Scratch() {
        cudaStreamSynchronize(ws->stream);
        for (void *p : ptrs) cudaFree(p);
    }
    template <class T>
    cudaError_t alloc(T **p, size_t bytes) {
        void *q = nullptr;
        cudaError_t e = handle_malloc(ws, &q, bytes);
        if (e != cudaSuccess) return e;
        ptrs.push_back(q);
        *p = static_cast<T *>(q);
        return cudaSuccess;
    }
};

}  // namespace wsh
