// Streaming step kernel for sm_103a: the hot path of the library.
//
// The grid is cut into work items: a TX x TY tile of (x, y) columns over a
// block of zb planes, walked in increasing z. The paper keeps a whole z
// column in a processing element's memory and receives x/y neighbours from 4
// PEs per direction over the fabric (Section III-B, III-C); here the column
// lives in a per-thread register queue of 9 planes (k-4 .. k+4), and the x/y
// neighbours come from a shared-memory copy of plane k with its 4-cell halo.
//
// One CTA per work item, dispatched by the hardware in item order as resident
// CTAs finish, so the tiles in flight are always a contiguous range of items
// and a tile's halo rows are still in L2 when its neighbour reads them.
//  - Every thread computes the 4 cells i .. i+3 of the two rows j and j+1: the
//    rows j-4 .. j-1 and j+2 .. j+5 serve both, and the waits, the ring
//    bookkeeping and the x loads of a plane are paid once for 8 cells.
//  - TMA copies (cp.async.bulk.tensor) fill two shared-memory rings: ring A
//    (u^n with halo, (TX+8) x (TY+8), P + 4 planes) and ring B (u^{n-1} and
//    (V dt/h)^2 tiles, P planes). Stage r carries what plane r needs new: the
//    u^n plane r+4 and ring B's plane r, on one "full" mbarrier. A warp that
//    has read plane r arrives on the stage's "empty" mbarrier; one lane of one
//    warp waits for it and issues stage r + P. There is no
//    producer warp (its registers would cost a third of the compute warps)
//    and no CTA-wide barrier in the loop.
//  - The four planes below the block, of which only the thread's own cells are
//    needed, are read from global memory straight into the queue.
// u^{n+1} is written in place of u^{n-1} with 128-bit stores (plain ones: with
// evict-first stores 1024 x 1024 x 512 ran at 415 instead of 422 Gcell/s).
// Taper, source injection and receiver sampling are fused into the pass.
// The z loop is unrolled by 3 with the queue indices rotated at compile time.
//
// Each thread's 4 cells of a row are processed as two pairs with the packed
// FP32x2 instructions of sm_100+ (add/mul/fma .rn .f32x2). Each lane is
// rounded exactly as the scalar instruction, so the arithmetic per cell is the
// same expression, in the same order, as the direct kernel, and the two CUDA
// paths agree bit for bit.
//
// Every wait is bounded (kWaitLimitNs); on a timeout the kernel records
// kStatusTimeout, all warps leave their loops, and the CTA waits (bounded)
// for its copies in flight before it exits.
//
// The same pipeline serves two sources of work items: one grid whose maps
// and arguments are kernel parameters (OneGrid), and a batch of independent
// shots on grids of different sizes (ShotBatch), whose per-shot tensor maps,
// geometry, sources and receivers sit in a descriptor table in global memory
// and whose items from every shot share one launch.
#include <climits>

#include "ws_ptx.cuh"

namespace ws {
namespace {

constexpr int kTrip = 3;   // planes per loop trip, and the stages in flight

// Tile geometry and ring sizes of one instantiation.
template <int TX, int TY>
struct StreamCfg {
    static constexpr int kCols = TX / 4;                 // threads across a row
    static constexpr int kThreads = kCols * (TY / 2);
    static constexpr int kWarps = kThreads / 32;
    static constexpr int P = kTrip;                      // stages (ring-B planes)
    static constexpr int NA = P + 4;                     // ring-A planes
    static constexpr int kRowW = TX + 2 * kHalo;         // floats per ring-A row
    static constexpr int kRows = TY + 2 * kHalo;
    static constexpr unsigned kRowBytes = kRowW * 4u;
    static constexpr unsigned kSlotABytes = kRowW * kRows * 4u;
    static constexpr unsigned kTileBytes = TX * TY * 4u;
    static constexpr unsigned kSlotBBytes = 2u * kTileBytes;   // u^{n-1} tile, then (V dt/h)^2
    static_assert(kThreads % 32 == 0, "whole warps");
    static_assert(kSlotABytes % 128 == 0 && kSlotBBytes % 128 == 0, "slots stay 128-byte aligned");
    static constexpr size_t kSmem = size_t(NA) * kSlotABytes + size_t(P) * kSlotBBytes;
};

// The tensor maps of one launch: u^n with the halo box, u^{n-1} and
// (V dt/h)^2 with the interior box.
struct StreamMaps {
    CUtensorMap u, up, w;
};

// What the copies of an item need: its extent and the three maps; stall (a
// test hook) withholds the item's first copies.
struct Job {
    Item it;
    const CUtensorMap *u, *up, *w;
    bool stall;
};

// What the threads need of an item's grid: fields read at the start of an
// item or on every plane, and accessors for what only source injection and
// receiver recording use.
struct View {
    Geom g;
    const float *gx, *gy, *gz;
    const float *u;            // u^n field (padded)
    float *out;                // u^{n+1} field (padded)
    long long lap_delta;       // L u^n goes to out + lap_delta (0: not stored)
    const int *rec_ptr;        // per-tile receiver ranges, or null
    const RecEntry *rec_;
    const SourceSample *src_;  // this step's source samples
    int nsrc_;
    float *traces_;            // [nrec][nt_max]
    const float *inject;       // residual [nrec][nt_max] (Mode::kInject)
    int nt_max_;
    long long trace_step_;
    __device__ __forceinline__ const SourceSample *src() const { return src_; }
    __device__ __forceinline__ int nsrc() const { return nsrc_; }
    __device__ __forceinline__ const RecEntry *rec() const { return rec_; }
    __device__ __forceinline__ float *traces() const { return traces_; }
    __device__ __forceinline__ int nt_max() const { return nt_max_; }
    __device__ __forceinline__ long long trace_step() const { return trace_step_; }
};

// What a launch does besides the step: records the receivers (if any), also
// stores the stencil sum L u^n (into a.lap), or adds W G r at the receivers
// (r = a.inject, the adjoint's residual) instead of recording them.
enum class Mode { kRecord, kLap, kInject };

// Items of one grid; everything comes from kernel parameters.
template <int TX, int TY, Mode M>
struct OneGrid {
    static constexpr Mode kMode = M;
    using V = View;
    const StreamMaps &mp;
    const StepArgs &a;
    const float *u;
    float *up;
    int zb, tiles_x, ntiles;
    const int *rec_ptr;
    const RecEntry *rec;

    __device__ __forceinline__ Job job(int item) const {
        return Job{item_of(item, tiles_x, ntiles, zb, a.g.nz, TX, TY), &mp.u, &mp.up, &mp.w,
                   item == a.stall_item};
    }
    __device__ __forceinline__ void view(int, View *v) const {
        v->g = a.g;
        v->gx = a.gx;
        v->gy = a.gy;
        v->gz = a.gz;
        v->src_ = a.src.s;
        v->nsrc_ = a.src.n;
        v->traces_ = a.traces;
        v->nt_max_ = a.nt_max;
        v->trace_step_ = a.trace_step;
        v->u = u;
        v->out = up;
        v->lap_delta = M == Mode::kLap ? a.lap - up : 0;
        v->inject = M == Mode::kInject ? a.inject : nullptr;
        v->rec_ptr = rec_ptr;
        v->rec_ = rec;
    }
};

// The view of a batch item: the fields of every plane in registers, the rest
// read from the shot's descriptor where they are used (held in registers for
// the whole item they would not fit the register budget).
struct BatchView {
    Geom g;
    const float *gx, *gy, *gz;
    const float *u;
    float *out;
    const int *rec_ptr;
    const BatchShot *shot;
    int t;
    __device__ __forceinline__ const SourceSample *src() const {
        return shot->src + (long long)t * shot->nsrc;
    }
    __device__ __forceinline__ int nsrc() const { return shot->nsrc; }
    __device__ __forceinline__ const RecEntry *rec() const { return shot->rec; }
    __device__ __forceinline__ float *traces() const { return shot->traces; }
    __device__ __forceinline__ int nt_max() const { return shot->nt_max; }
    __device__ __forceinline__ long long trace_step() const { return shot->trace_col0 + t; }
};

// Items of a batch of shots: items[q] = (shot, item of that shot), step t of
// the run; shot s reads u^n from buf[cur0 ^ (t & 1)].
template <int TX, int TY>
struct ShotBatch {
    static constexpr Mode kMode = Mode::kRecord;
    using V = BatchView;
    const BatchShot *shots;
    const int2 *items;
    int t;

    __device__ __forceinline__ Job job(int item) const {
        const int2 e = items[item];
        const BatchShot &s = shots[e.x];
        const int p = s.cur0 ^ (t & 1);
        return Job{item_of(e.y, s.tiles_x, s.ntiles, s.zb, s.g.nz, TX, TY), &s.halo[p],
                   &s.tile[1 - p], &s.w, t == 0 && e.y == s.stall_item};
    }
    __device__ __forceinline__ void view(int item, BatchView *v) const {
        const int2 e = items[item];
        const BatchShot &s = shots[e.x];
        const int p = s.cur0 ^ (t & 1);
        v->g = s.g;
        v->gx = s.gx;
        v->gy = s.gy;
        v->gz = s.gz;
        v->u = s.buf[p];
        v->out = s.buf[1 - p];
        v->rec_ptr = s.rec_ptr;
        v->shot = &s;
        v->t = t;
    }
};

// Barriers of one CTA.
template <int P>
struct Bars {
    uint64_t full[P], empty[P];   // stages
    uint64_t first;               // ring-A planes z0 .. z0+3
    int issued;                   // stages issued (for the drain)
    int first_issued;
    int abort;
};

// Per-thread state of the walk down an item.
struct Walk {
    float4 q[9][2];         // u^n of planes k-4 .. k+4, rows j and j+1 (rotated: see plane_step)
    float4 gxy[2];          // gx * gy of this thread's 4 columns per row
    float *out_k;           // u^{n+1} of (i, j, k)
    unsigned halo, own;     // byte offsets of the ring-A slots of planes k and k + 4
    int nvalid;             // cells of the 4 inside the grid (0 when the column is outside)
    bool row1;              // row j+1 inside the grid
    bool whole;             // all cells of the warp lie inside the grid
    int rcur, rend, rnext_k;
    unsigned src_mask;
    int next_event;         // the next plane with a source or a receiver
};

template <int TX, int TY>
struct Kern {
    using Cfg = StreamCfg<TX, TY>;
    static constexpr int P = Cfg::P, NA = Cfg::NA;
    using B = Bars<P>;

    // Stage r of the item into its slots (ring A at byte slotA): the u^n plane z0 + r + 4 with its
    // halo, and u^{n-1} and (V dt/h)^2 of plane z0 + r. The maps cover the
    // interior only (origin at interior cell 0): whatever of a box lies
    // outside the grid arrives as zeros without a memory read (the zero halo).
    // x is a multiple of 4 elements (16 bytes).
    static __device__ __forceinline__ void issue(B &br, unsigned ringA, unsigned ringB, const Job &jb,
                                                 int r, unsigned slotA, int stage) {
        uint64_t *bar = &br.full[stage];
        mbar_arrive_expect_tx(bar, Cfg::kSlotABytes + Cfg::kSlotBBytes);
        const unsigned b = ringB + stage * Cfg::kSlotBBytes;
        tma_load_3d_at(ringA + slotA, jb.u, bar, jb.it.i0 - kHalo,
                       jb.it.j0 - kHalo, jb.it.z0 + kHalo + r);
        tma_load_3d_at(b, jb.up, bar, jb.it.i0, jb.it.j0, jb.it.z0 + r);
        tma_load_3d_at(b + Cfg::kTileBytes, jb.w, bar, jb.it.i0, jb.it.j0, jb.it.z0 + r);
    }

    // The stencil sum of one row's 4 cells (two FP32x2 pairs). xl, xr: cells
    // x-4..x-1 and x+4..x+7 of the row; yp / ym: rows j+m / j-m of this row;
    // z from the register queue.
    template <int RQ>
    static __device__ __forceinline__ void stencil_row(const Walk &wk, const Coeffs &c, int r,
                                                       const float4 &xl, const float4 &xr,
                                                       const float4 (&yp)[4], const float4 (&ym)[4],
                                                       float2 (&lap)[2]) {
        const float4 xc = wk.q[(RQ + 4) % 9][r];
        // x pairs: offsets +-2 and +-4 are aligned float2 pairs of (xl, xc,
        // xr); offsets +-1 and +-3 straddle pairs and are summed per lane
        const float e[12] = {xl.x, xl.y, xl.z, xl.w, xc.x, xc.y, xc.z, xc.w,
                             xr.x, xr.y, xr.z, xr.w};
        float2 sx[2][5];
        sx[0][2] = add2(hi2(xc), hi2(xl));
        sx[1][2] = add2(lo2(xr), lo2(xc));
        sx[0][4] = add2(lo2(xr), lo2(xl));
        sx[1][4] = add2(hi2(xr), hi2(xl));
#pragma unroll
        for (int p = 0; p < 2; ++p) {
#pragma unroll
            for (int m = 1; m <= 3; m += 2) {
                const int l0 = 2 * p, l1 = 2 * p + 1;
                sx[p][m] = make_float2(e[4 + l0 + m] + e[4 + l0 - m], e[4 + l1 + m] + e[4 + l1 - m]);
            }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            float2 s[5];
#pragma unroll
            for (int m = 1; m <= 4; ++m) {
                const float2 sy = add2(pair(yp[m - 1], p), pair(ym[m - 1], p));
                const float2 sz = add2(pair(wk.q[(RQ + 4 + m) % 9][r], p),
                                       pair(wk.q[(RQ + 4 - m + 9) % 9][r], p));
                s[m] = add2(add2(sx[p][m], sy), sz);
            }
            const float2 uc = pair(xc, p);
            // sum_m c_m (s_m - 6 u): exactly zero on constants (see Coeffs)
            float2 l = mul2(splat(c.c4), fma2(splat(-6.0f), uc, s[4]));
            l = fma2(splat(c.c3), fma2(splat(-6.0f), uc, s[3]), l);
            l = fma2(splat(c.c2), fma2(splat(-6.0f), uc, s[2]), l);
            lap[p] = fma2(splat(c.c1), fma2(splat(-6.0f), uc, s[1]), l);
        }
    }

    // u^{n+1} = g (2 u - g u^{n-1} + W L) of one row's 4 cells.
    static __device__ __forceinline__ float4 update(const float2 (&lap)[2], const float4 &u,
                                                    const float4 &up, const float4 &w,
                                                    const float4 &gxy, float gzk) {
        float2 o[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float2 gd = mul2(pair(gxy, p), splat(gzk));
            const float2 ngd = mul2(pair(gxy, p), splat(-gzk));   // -gd, exactly
            const float2 t =
                fma2(pair(w, p), lap[p], fma2(splat(2.0f), pair(u, p), mul2(ngd, pair(up, p))));
            o[p] = mul2(gd, t);
        }
        return make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
    }

    // Rows j and j+1 of one plane: the common warp stores all 8 cells a thread.
    static __device__ __forceinline__ void store_rows(const Walk &wk, float *p, int pitch,
                                                      const float4 &a, const float4 &b) {
        if (wk.whole) {
            *reinterpret_cast<float4 *>(p) = a;
            *reinterpret_cast<float4 *>(p + pitch) = b;
            return;
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (r == 1 && !wk.row1) break;
            const float4 v = r ? b : a;
            float *q = p + r * pitch;
            if (wk.nvalid > 0) q[0] = v.x;
            if (wk.nvalid > 1) q[1] = v.y;
            if (wk.nvalid > 2) q[2] = v.z;
            if (wk.nvalid > 3) q[3] = v.w;
        }
    }

    // The first plane after k with a source or a receiver of this warp.
    template <class VT>
    static __device__ __forceinline__ int event_after(const Walk &wk, const VT &v, int k) {
        int next = wk.rnext_k;
        for (unsigned m = wk.src_mask; m; m &= m - 1) {
            const int sk = v.src()[__ffs(m) - 1].k;
            if (sk > k) next = min(next, sk);
        }
        return next;
    }

    // Adds W G r at the receivers of plane k: lane q takes entry cur + q and
    // reads its residual; each thread adds the entries of its cells one after
    // the other (receivers may share a cell), the threads side by side: entry by
    // entry for the whole warp took 256^3 gradients with 128 x 128 receivers 168
    // ms a shot, now 159; 128^3 with 24 x 24 receivers 1.78 ms, now 1.72. Where a
    // thread has more than 8 entries, so that some share a cell, the residuals of
    // each cell are summed first, pairwise: a gradient of 64^3 and 25 steps with 3000
    // receivers on one cell 11.8 ms, now 2.2. Entries and residuals are fetched 32
    // ahead: 128^3 with a plane of receivers 1.11 ms, now 0.99. (Entries of a plane
    // that is recorded are not: 32 uneven shots and 1024^3 ran 0.4 and 0.1 % slower.)
    template <class VT>
    static __device__ __forceinline__ void inject_plane(Walk &wk, const VT &v, int k,
                                                        float4 (&out)[2], const float4 &w0,
                                                        const float4 &w1, float gzk) {
        const int lane = threadIdx.x & 31;
        int cur = wk.rcur;
        // the next 32 entries and their residuals are fetched ahead
        auto entry = [&](int at) {
            RecEntry e{INT_MAX, 0, 0, 0};
            if (at + lane < wk.rend) e = v.rec()[at + lane];
            return e;
        };
        auto residual = [&](const RecEntry &e) {
            return e.k == k ? v.inject[(long long)e.r * v.nt_max() + v.trace_step()] : 0.0f;
        };
        RecEntry e = entry(cur), e1 = entry(cur + 32);
        float r = residual(e);
        for (;;) {
            const RecEntry e2 = entry(cur + 64);
            const float r1 = residual(e1);
            const bool take = e.k == k;
            const unsigned taken = __ballot_sync(0xffffffffu, take);
            unsigned mine = taken;   // the lanes whose entry is this thread's
#pragma unroll
            for (int b = 0; b < 5; ++b) {
                const unsigned set = __ballot_sync(0xffffffffu, (e.owner >> b) & 1);
                mine &= (lane >> b) & 1 ? set : ~set;
            }
            if (__any_sync(0xffffffffu, __popc(mine) > 8)) {
                const unsigned same =
                    __match_any_sync(0xffffffffu, take ? e.owner * 8 + e.lane : -1 - lane);
                unsigned above = same & (0xfffffffeu << lane);   // not yet added, of this cell
                int rank = __popc(same & ~(0xffffffffu << lane));
                const unsigned first = __ballot_sync(0xffffffffu, rank == 0);
                while (__any_sync(0xffffffffu, above != 0)) {   // odd ranks go to the even ones
                    const int q = above ? __ffs(above) - 1 : lane;
                    const float rq = __shfl_sync(0xffffffffu, r, q);
                    if (above) r = __fadd_rn(r, rq);
                    above &= __ballot_sync(0xffffffffu, (rank & 1) == 0);
                    rank >>= 1;
                }
                mine &= first;
            }
            for (; __any_sync(0xffffffffu, mine != 0); mine &= mine - 1) {
                const int q = mine ? __ffs(mine) - 1 : lane;
                const int cell = __shfl_sync(0xffffffffu, e.lane, q);
                const float rq = __shfl_sync(0xffffffffu, r, q);
                if (!mine) continue;
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (cell == c) {
                        const float gd = __fmul_rn(comp(wk.gxy[c / 4], c % 4), gzk);
                        const float wg = __fmul_rn(comp(c < 4 ? w0 : w1, c % 4), gd);
                        set_comp(out[c / 4], c % 4,
                                 __fadd_rn(comp(out[c / 4], c % 4), __fmul_rn(wg, rq)));
                    }
            }
            cur += __popc(taken);
            if (taken != 0xffffffffu) break;
            e = e1;
            e1 = e2;
            r = r1;
        }
        wk.rcur = cur;
        wk.rnext_k = cur < wk.rend ? v.rec()[cur].k : INT_MAX;
    }

    // Sources and receivers of plane k (few planes have any).
    template <Mode M, class VT>
    static __device__ __forceinline__ void events(Walk &wk, const VT &v, int k, int i, int j,
                                                  float4 (&out)[2], const float4 &w0,
                                                  const float4 &w1, float gzk) {
        for (unsigned m = wk.src_mask; m; m &= m - 1) {
            const SourceSample ss = v.src()[__ffs(m) - 1];
            if (ss.k != k) continue;
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                if (ss.i != i + l) continue;
                if (ss.j == j) set_comp(out[0], l, fmaf(comp(w0, l), ss.amp, comp(out[0], l)));
                if (ss.j == j + 1) set_comp(out[1], l, fmaf(comp(w1, l), ss.amp, comp(out[1], l)));
            }
        }
        if (k == wk.rnext_k) {
            if constexpr (M == Mode::kInject)
                inject_plane(wk, v, k, out, w0, w1, gzk);
            else
                record_plane2(out, k, &wk.rcur, wk.rend, &wk.rnext_k, v.rec(), v.traces(),
                              v.nt_max(), v.trace_step());
        }
        wk.next_event = event_after(wk, v, k);
    }

    // Plane k of the item, RQ = (k - z0) mod kTrip (also the stage); parity:
    // of the trip. Returns false when a bounded wait ran out.
    template <int RQ, Mode M, class VT>
    static __device__ __forceinline__ bool plane_step(Walk &wk, B &br, unsigned aOwn, unsigned bOwn,
                                                      unsigned ringA, unsigned ringB, const Job &jb,
                                                      const VT &v, const Coeffs &c, unsigned *status,
                                                      int k, int i, int j, unsigned parity,
                                                      bool issuer_warp) {
        constexpr int Q8 = (RQ + 8) % 9, Q4 = (RQ + 4) % 9;
        constexpr unsigned RS = Cfg::kRowBytes, TB = Cfg::kTileBytes;
        if (!__all_sync(0xffffffffu, mbar_try_wait(&br.full[RQ], parity))) {
            const bool ok = wait_phase(&br.full[RQ], parity, &br.abort, status);
            if (!__all_sync(0xffffffffu, ok)) return false;
        }
        // u^n of plane k + 4 into the queue
        wk.q[Q8][0] = lds4_at<0>(aOwn + wk.own);
        wk.q[Q8][1] = lds4_at<RS>(aOwn + wk.own);
        // u^n of plane k with its halo (in ring A for four planes already)
        const unsigned h = aOwn + wk.halo;
        const float4 xl0 = lds4_at<-16>(h), xr0 = lds4_at<16>(h);
        const float4 xl1 = lds4_at<(int)RS - 16>(h), xr1 = lds4_at<(int)RS + 16>(h);
        const float4 lm[4] = {lds4_at<-(int)RS>(h), lds4_at<-2 * (int)RS>(h),
                              lds4_at<-3 * (int)RS>(h), lds4_at<-4 * (int)RS>(h)};
        const float4 lp[4] = {lds4_at<2 * (int)RS>(h), lds4_at<3 * (int)RS>(h),
                              lds4_at<4 * (int)RS>(h), lds4_at<5 * (int)RS>(h)};
        // u^{n-1} and (V dt/h)^2 of plane k
        constexpr int OB = RQ * Cfg::kSlotBBytes;
        const float4 up0 = lds4_at<OB>(bOwn), up1 = lds4_at<OB + TX * 4>(bOwn);
        const float4 w0 = lds4_at<OB + (int)TB>(bOwn), w1 = lds4_at<OB + (int)TB + TX * 4>(bOwn);
        warp_arrive(&br.empty[RQ]);

        float2 lap0[2], lap1[2];
        {
            const float4 yp[4] = {wk.q[Q4][1], lp[0], lp[1], lp[2]};
            stencil_row<RQ>(wk, c, 0, xl0, xr0, yp, lm, lap0);
        }
        // Refill plane k's stage (and the ring-A slot of plane k) for plane
        // k + P as soon as every warp has read it. Half way through the
        // arithmetic the others usually have, so the lane does not wait, and
        // the copy has 2 1/2 planes of time: 384^3 at 381 Gcell/s, against 366
        // issued one plane later (the copy then has one), 358 right after the
        // arrive (the lane waits for its neighbours) and 371 after the
        // arithmetic. The vote that ends a failed walk is taken here, by this
        // warp alone: at the end of every plane, by all warps, the CTAs drifted
        // apart and it ran at 260.
        if (issuer_warp && k + P < jb.it.z1) {
            bool ok = true;
            if ((threadIdx.x & 31) == 0) {
                ok = wait_phase(&br.empty[RQ], parity, &br.abort, status);
                if (ok) {
                    br.issued++;
                    issue(br, ringA, ringB, jb, k + P - jb.it.z0, wk.halo, RQ);
                }
            }
            if (!__all_sync(0xffffffffu, ok)) return false;
        }
        {
            const float4 ym[4] = {wk.q[Q4][0], lm[0], lm[1], lm[2]};
            stencil_row<RQ>(wk, c, 1, xl1, xr1, lp, ym, lap1);
        }
        const float gzk = v.gz[k];
        float4 out[2] = {update(lap0, wk.q[Q4][0], up0, w0, wk.gxy[0], gzk),
                         update(lap1, wk.q[Q4][1], up1, w1, wk.gxy[1], gzk)};
        if (k == wk.next_event) events<M>(wk, v, k, i, j, out, w0, w1, gzk);
        store_rows(wk, wk.out_k, v.g.pnx, out[0], out[1]);
        if constexpr (M == Mode::kLap)   // the stencil sum, for the adjoint's imaging
            store_rows(wk, wk.out_k + v.lap_delta, v.g.pnx,
                       make_float4(lap0[0].x, lap0[0].y, lap0[1].x, lap0[1].y),
                       make_float4(lap1[0].x, lap1[0].y, lap1[1].x, lap1[1].y));
        wk.out_k += v.g.plane;
        wk.halo = wk.halo == (NA - 1) * Cfg::kSlotABytes ? 0u : wk.halo + Cfg::kSlotABytes;
        wk.own = wk.own == (NA - 1) * Cfg::kSlotABytes ? 0u : wk.own + Cfg::kSlotABytes;
        return true;
    }

    // After a trip of kTrip planes the queue is rotated by kTrip; rename it.
    static __device__ __forceinline__ void rotate_queue(Walk &wk) {
        float4 t[9][2];
#pragma unroll
        for (int m = 0; m < 9; ++m) {
            t[m][0] = wk.q[(m + kTrip) % 9][0];
            t[m][1] = wk.q[(m + kTrip) % 9][1];
        }
#pragma unroll
        for (int m = 0; m < 9; ++m) {
            wk.q[m][0] = t[m][0];
            wk.q[m][1] = t[m][1];
        }
    }
};

// The body of a launch: one CTA's item.
template <int TX, int TY, class S>
__device__ __forceinline__ void stream_body(const S &src, const Coeffs &c, unsigned *status) {
    using K = Kern<TX, TY>;
    using Cfg = typename K::Cfg;
    constexpr int P = Cfg::P;
    extern __shared__ __align__(128) float smem[];
    __shared__ Bars<P> br;
    const unsigned ringA = smem_addr(smem);
    const unsigned ringB = ringA + Cfg::NA * Cfg::kSlotABytes;
    const int tid = threadIdx.x;
    // the copies' lane: of a warp that differs between neighbouring CTAs, so
    // that the SM's sub-partitions share this work
    const bool issuer_warp = tid / 32 == (int)(blockIdx.x % Cfg::kWarps);
    const bool issuer = issuer_warp && (tid & 31) == 0;

    if (issuer) {
        for (int s = 0; s < P; ++s) {
            mbar_init(&br.full[s], 1);
            mbar_init(&br.empty[s], Cfg::kWarps);
        }
        mbar_init(&br.first, 1);
        br.issued = 0;
        br.first_issued = 0;
        br.abort = 0;
        fence_mbar_init();
    }
    __syncthreads();
    // Before the predecessor is waited for: what no kernel writes (descriptors,
    // tapers, receiver tables; their uploads are copies, which no kernel
    // overlaps). After the wait, these chains of loads took 0.3 to 0.9 us a step:
    // 64^3 with receivers 3.70 us, now 3.11, 128^3 8.46, now 7.54.
    const Job jb = src.job(blockIdx.x);
    const Item &it = jb.it;
    const int nb = it.z1 - it.z0;
    typename S::V v;
    src.view(blockIdx.x, &v);
    const Geom &g = v.g;
    const int tx = tid % Cfg::kCols, py = tid / Cfg::kCols;
    const int i = it.i0 + 4 * tx, j = it.j0 + 2 * py;
    const unsigned aOwn = ringA + 4u * ((kHalo + 2 * py) * Cfg::kRowW + kHalo + 4 * tx);
    const unsigned bOwn = ringB + 4u * (2 * py * TX + 4 * tx);
    const bool col_ok = (j < g.ny) && (i < g.nx);
    Walk wk;
    wk.nvalid = col_ok ? min(4, g.nx - i) : 0;
    wk.row1 = col_ok && j + 1 < g.ny;
    const long long at = pidx(g, col_ok ? i : 0, col_ok ? j : 0, it.z0);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        wk.gxy[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (col_ok && (r == 0 || wk.row1)) {
            const float gyj = v.gy[j + r];
            wk.gxy[r].x = v.gx[i] * gyj;
            if (wk.nvalid > 1) wk.gxy[r].y = v.gx[i + 1] * gyj;
            if (wk.nvalid > 2) wk.gxy[r].z = v.gx[i + 2] * gyj;
            if (wk.nvalid > 3) wk.gxy[r].w = v.gx[i + 3] * gyj;
        }
    }
    wk.src_mask = 0u;
    {
        const SourceSample *srcs = v.src();
        for (int qs = 0, ns = v.nsrc(); qs < ns; ++qs) {
            const SourceSample ss = srcs[qs];
            if (ss.i >= it.i0 && ss.i < it.i0 + TX && ss.j >= it.j0 && ss.j < it.j0 + TY &&
                ss.k >= it.z0 && ss.k < it.z1)
                wk.src_mask |= 1u << qs;
        }
    }
    wk.rcur = wk.rend = 0;
    if (v.rec_ptr != nullptr) {
        const int r = it.tile * Cfg::kWarps + (tid >> 5);
        wk.rend = v.rec_ptr[r + 1];
        wk.rcur = first_entry(v.rec(), v.rec_ptr[r], wk.rend, it.z0);
    }
    wk.rnext_k = wk.rcur < wk.rend ? v.rec()[wk.rcur].k : INT_MAX;
    wk.out_k = v.out + at;
    wk.whole = __all_sync(0xffffffffu, wk.nvalid == 4 && wk.row1);
    wk.next_event = K::event_after(wk, v, it.z0 - 1);
    wk.halo = 0u;
    wk.own = kHalo * Cfg::kSlotABytes;

    wait_predecessor();
    if (issuer) {
        if (!jb.stall) {   // else never filled: the bounded waits run out
            br.first_issued = 1;
            mbar_arrive_expect_tx(&br.first, kHalo * Cfg::kSlotABytes);
            for (int m = 0; m < kHalo; ++m)
                tma_load_3d_at(ringA + m * Cfg::kSlotABytes, jb.u, &br.first, it.i0 - kHalo,
                               it.j0 - kHalo, it.z0 + m);
        }
        const int n = min(P, nb);
        br.issued = n;
        for (int r = 0; r < n; ++r)
            K::issue(br, ringA, ringB, jb, r, (kHalo + r) * Cfg::kSlotABytes, r);
    }

    // the queue's planes z0-4 .. z0-1: this thread's own cells only, from
    // global memory (the planes below the grid are its zero halo)
#pragma unroll
    for (int m = 0; m < kHalo; ++m) {
        const float *p = v.u + at + (m - kHalo) * g.plane;
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        wk.q[m][0] = col_ok ? __ldcg(reinterpret_cast<const float4 *>(p)) : z;
        wk.q[m][1] = wk.row1 ? __ldcg(reinterpret_cast<const float4 *>(p + g.pnx)) : z;
    }

    bool ok = wait_phase(&br.first, 0u, &br.abort, status);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
#pragma unroll
        for (int m = 0; m < kHalo; ++m) {   // planes z0 .. z0+3
            wk.q[kHalo + m][0] = lds4_dyn(aOwn + m * Cfg::kSlotABytes);
            wk.q[kHalo + m][1] = lds4_dyn(aOwn + m * Cfg::kSlotABytes + Cfg::kRowBytes);
        }
        unsigned parity = 0;
        for (int kb = it.z0;; kb += kTrip, parity ^= 1u) {
#define WS_PLANE(RQ)                                                                              \
    if (kb + (RQ) >= it.z1 ||                                                                     \
        !K::template plane_step<RQ, S::kMode>(wk, br, aOwn, bOwn, ringA, ringB, jb, v, c,         \
                                              status, kb + (RQ), i, j, parity, issuer_warp))      \
        break;
            WS_PLANE(0)
            WS_PLANE(1)
            WS_PLANE(2)
#undef WS_PLANE
            K::rotate_queue(wk);
        }
    }

    // After an abort, wait (bounded) for the last copies issued into each
    // stage to land before the CTA exits.
    __syncthreads();
    if (br.abort && tid == 0) {
        for (int s = 0; s <= P; ++s) {
            // fills of stage s; the first planes as one more stage
            const int n = s < P ? (br.issued + P - 1 - s) / P : br.first_issued;
            uint64_t *bar = s < P ? &br.full[s] : &br.first;
            if (n == 0) continue;
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(bar, (unsigned)(n - 1) & 1u) && global_ns() - t0 < kWaitLimitNs) {
            }
        }
    }
}

template <int TX, int TY, int MINB, Mode M>
__global__ void __launch_bounds__(StreamCfg<TX, TY>::kThreads, MINB)
    step_stream_kernel(const __grid_constant__ StreamMaps maps, const float *u, float *up,
                       const __grid_constant__ StepArgs a, const int zb, const int tiles_x,
                       const int ntiles, const int *__restrict__ rec_ptr,
                       const RecEntry *__restrict__ rec) {
    const OneGrid<TX, TY, M> src{maps, a, u, up, zb, tiles_x, ntiles, rec_ptr, rec};
    stream_body<TX, TY>(src, a.c, a.status);
}

template <int TX, int TY, int MINB>
__global__ void __launch_bounds__(StreamCfg<TX, TY>::kThreads, MINB)
    step_batch_kernel(const BatchShot *__restrict__ shots, const int2 *__restrict__ items,
                      const int t, const Coeffs c, unsigned *status) {
    const ShotBatch<TX, TY> src{shots, items, t};
    stream_body<TX, TY>(src, c, status);
}

// Resident CTAs per SM and SM count of a kernel on the current device,
// looked up (and the kernel's shared-memory limit set) the first time the
// kernel runs on each device.
template <class KernFn>
cudaError_t occupancy(KernFn kern, int threads, size_t smem, LaunchFacts &lf, int *ctas_per_sm,
                      int *sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= LaunchFacts::kMaxDevices) return cudaErrorInvalidDevice;
    if (lf.ctas[dev] == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int n = 0, c = 0;
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, kern, threads, smem);
        if (e != cudaSuccess) return e;
        if (c < 1) return cudaErrorInvalidConfiguration;
        lf.sms[dev] = n;
        lf.ctas[dev] = c;
    }
    *ctas_per_sm = lf.ctas[dev];
    *sms = lf.sms[dev];
    return cudaSuccess;
}

// Calls fn with the configuration of tile tx x ty: (TX, TY, resident CTAs per
// SM that its registers and rings allow).
template <int TX, int TY, int MINB>
struct TileTag {
    static constexpr int kX = TX, kY = TY, kMin = MINB;
};
template <class F>
cudaError_t with_tile(int tx, int ty, F &&fn) {
    if (tx == 64 && ty == 32) return fn(TileTag<64, 32, 1>{});
    if (tx == 64 && ty == 16) return fn(TileTag<64, 16, 3>{});
    if (tx == 64 && ty == 8) return fn(TileTag<64, 8, 5>{});
    if (tx == 32 && ty == 16) return fn(TileTag<32, 16, 5>{});
    if (tx == 32 && ty == 8) return fn(TileTag<32, 8, 8>{});
    return cudaErrorInvalidValue;
}

template <class T, Mode M>
cudaError_t launch_grid(const StreamMaps &maps, const float *u, float *up, const StepArgs &a, int zb,
                        const int *rec_ptr, const RecEntry *rec, cudaStream_t s) {
    using Cfg = StreamCfg<T::kX, T::kY>;
    auto kern = step_stream_kernel<T::kX, T::kY, T::kMin, M>;
    static LaunchFacts lf;
    int ctas_per_sm = 0, sms = 0;
    cudaError_t e = occupancy(kern, Cfg::kThreads, Cfg::kSmem, lf, &ctas_per_sm, &sms);
    if (e != cudaSuccess) return e;
    const int tiles_x = (a.g.nx + T::kX - 1) / T::kX;
    const int ntiles = tiles_x * ((a.g.ny + T::kY - 1) / T::kY);
    const int nitems = ntiles * ((a.g.nz + zb - 1) / zb);
    return launch_overlapped(kern, nitems, Cfg::kThreads, Cfg::kSmem, s, maps, u, up, a, zb, tiles_x,
                             ntiles, rec_ptr, rec);
}

template <class T>
cudaError_t batch_facts(int *ctas_per_sm, int *sms) {
    static LaunchFacts lf;
    using Cfg = StreamCfg<T::kX, T::kY>;
    return occupancy(step_batch_kernel<T::kX, T::kY, T::kMin>, Cfg::kThreads, Cfg::kSmem, lf,
                     ctas_per_sm, sms);
}

}  // namespace

bool stream_tiling_supported(int tx, int ty) {
    return (tx == 64 && (ty == 8 || ty == 16 || ty == 32)) || (tx == 32 && (ty == 8 || ty == 16));
}

cudaError_t launch_step_stream(const CUtensorMap *tmap_u, const CUtensorMap *tmap_up,
                               const CUtensorMap *tmap_w, const float *u, float *up,
                               const StepArgs &a, const StreamTiling &t, const int *rec_ptr,
                               const RecEntry *rec, cudaStream_t s) {
    StreamMaps maps;
    maps.u = *tmap_u;
    maps.up = *tmap_up;
    maps.w = *tmap_w;
    return with_tile(t.tx, t.ty, [&](auto tag) {
        using T = decltype(tag);
        if (a.lap) return launch_grid<T, Mode::kLap>(maps, u, up, a, t.zb, rec_ptr, rec, s);
        if (a.inject) return launch_grid<T, Mode::kInject>(maps, u, up, a, t.zb, rec_ptr, rec, s);
        return launch_grid<T, Mode::kRecord>(maps, u, up, a, t.zb, rec_ptr, rec, s);
    });
}

cudaError_t stream_slots(int tx, int ty, bool batch, int *slots, int *sms) {
    return with_tile(tx, ty, [&](auto tag) {
        using T = decltype(tag);
        using Cfg = StreamCfg<T::kX, T::kY>;
        static LaunchFacts lf;
        int c = 0, n = 0;
        cudaError_t e = batch ? batch_facts<T>(&c, &n)
                              : occupancy(step_stream_kernel<T::kX, T::kY, T::kMin, Mode::kRecord>,
                                          Cfg::kThreads, Cfg::kSmem, lf, &c, &n);
        if (e == cudaSuccess) *slots = c * n;
        if (e == cudaSuccess && sms) *sms = n;
        return e;
    });
}

cudaError_t launch_step_batch(const BatchShot *shots, const int2 *items, int nitems, int t,
                              const Coeffs &c, unsigned *status, int tx, int ty, cudaStream_t s) {
    if (nitems <= 0) return cudaSuccess;
    return with_tile(tx, ty, [&](auto tag) {
        using T = decltype(tag);
        using Cfg = StreamCfg<T::kX, T::kY>;
        int ctas_per_sm = 0, sms = 0;
        cudaError_t e = batch_facts<T>(&ctas_per_sm, &sms);
        if (e != cudaSuccess) return e;
        return launch_overlapped(step_batch_kernel<T::kX, T::kY, T::kMin>, nitems, Cfg::kThreads,
                                 Cfg::kSmem, s, shots, items, t, c, status);
    });
}

}  // namespace ws
