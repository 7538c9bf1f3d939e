// Streaming step kernel with 16-bit field storage (BF16 or FP16), velocity form.
//
// The state is stored as
//     U = u^n   and   D = u^n - u^{n-1}   (16 bits each),
// and the model as FP16 of (V dt/h)^2 * 2^kW16Exp: 10 bytes per cell update
// (read U, D, W; write U', D'). All arithmetic is FP32: the step computes
// d~ = u^{n+1} - u^n of the tapered leapfrog update (Eq. 2 with the taper)
// and u~ = u^n + d~, and stores their 16-bit roundings.
//
// Why the velocity form: rounding u^{n+1} and keeping it as the next step's
// u^{n-1} makes every rounding error a kick to the discrete velocity
// u^n - u^{n-1}, and kicks integrate (relative error ~ N^1.5 eps over N
// steps). Storing D' = d~ (computed in FP32, not from the rounded U') leaves
// the rounding of U' in the displacement only, and the velocity carries just
// the rounding of D', which is an order of magnitude smaller than |u|.
//
// A 16-bit stencil is bound by instruction issue long before HBM, so the
// kernel is built to execute few instructions per cell:
//  - one CTA per work item (a 64 x TY tile over a block of planes; TY = 24:
//    6 warps, 16: 4 warps), every thread computes 4 x-cells of two rows; no
//    producer warp. Thread 0
//    (ring A: U with its halo) and thread 32 (ring B: the D and W tiles)
//    issue the TMA copies (cp.async.bulk.tensor) of later planes right after
//    each plane's barrier, which is the point where every thread is done with
//    the slots being refilled: no "empty" barriers, no polling producer. Each
//    slot has a "full" mbarrier (transaction bytes).
//  - ring A has 9 slots, ring B 3, and the z loop runs 3 planes per trip: the
//    indices of the 9-plane register queue and ring B's slots are compile-time
//    constants, ring A's slots and phases are carried from trip to trip, and
//    the queue is renamed by moves after each trip. (Nine planes per trip need
//    no renaming, but the body then leaves the instruction caches: 441 against
//    479 Gcell/s at 1024^3.)
//  - every value is decoded once: a thread decodes its own cells of plane
//    k+4 into its register queue and, at plane k, writes them as FP32 into a
//    double-buffered staging tile; the cells around the tile that the star
//    stencil reads (not the corners) are decoded into the same tile in units
//    of 4 cells, one unit per thread. One barrier per plane (which also ANDs
//    the threads' "no wait failed" flags, so a bounded wait that gives up
//    stops every warp at the same plane) separates the staging writes from the
//    neighbour reads (128-bit loads).
//  - the stencil sum is c0 u + sum_m c_m s_m with weights whose sum is exact
//    (zero_sum_weights16: no mass term), symmetric pairs first, two cells per
//    packed FP32x2 instruction.
//  - tiles whose cells all have taper 1 (the interior of the absorbing
//    layer) take d~ = W L + d on planes whose z taper is 1, without the taper
//    multiplies; the tapered form gives the same bits there.
//  - 158 registers (TY = 24): 12 warps per SM, as 2 CTAs of 24 rows or 3 of 16.
//
// One power-of-two scale per step for U' and D' (|d| <= |u^{n+1}| + |u^n|,
// so the same exponent bounds both): stored values are value * 2^e, with e
// chosen on the device from max |u^n| (accumulated by the previous step from
// the stored U', with packed 16-bit abs-max instructions) and a host bound
// on the source term, putting the field's largest value near 2^12, 16x below
// the FP16 maximum; exponents and maxima live in a 4-slot ring (Scale16)
// indexed by step, so no host synchronization is needed.
//
// Decoding is exact: both formats go through the hardware conversion, one
// instruction per value. The kernel computes on the stored values: every
// input of one field carries the same power-of-two factor, the model's factor
// 2^kW16Exp is folded into the stencil weights, and the factors meet in exact
// power-of-two multiplies. Results are rounded to 16 bits once, when stored.
#include <climits>
#include <cmath>

#include "ws_ptx.cuh"

namespace ws {
namespace {

// 64-bit shared load (4 x 16-bit), kept whole.
__device__ __forceinline__ uint2 lds2u(const uint16_t *p) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(smem_addr(p)));
    return v;
}

// FP16 -> FP32 of the two halves of a word (exact, subnormals included).
__device__ __forceinline__ float2 f16x2_to_f32(unsigned w) {
    float2 r;
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\t"
        "cvt.f32.f16 %0, l;\n\tcvt.f32.f16 %1, h;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "r"(w));
    return r;
}

struct Bf16Fmt {
    static __device__ __forceinline__ float2 two(unsigned w) {
        float2 r;
        asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\t"
            "cvt.f32.bf16 %0, l;\n\tcvt.f32.bf16 %1, h;\n\t}"
            : "=f"(r.x), "=f"(r.y)
            : "r"(w));
        return r;
    }
    static __device__ __forceinline__ float4 decode(uint2 v) {
        const float2 a = two(v.x), b = two(v.y);
        return make_float4(a.x, a.y, b.x, b.y);
    }
    static __device__ __forceinline__ uint2 encode(float4 f) {
        uint2 r;
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r.x) : "f"(f.y), "f"(f.x));
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r.y) : "f"(f.w), "f"(f.z));
        return r;
    }
    // running max of the magnitudes of two packed values (the sign bits of
    // the result are those of the operands' xor: meaningless, ignored)
    static __device__ __forceinline__ unsigned amax(unsigned acc, unsigned w) {
        unsigned r;
        asm("max.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(acc), "r"(w));
        return r;
    }
    static __device__ __forceinline__ float amax_value(unsigned acc) {
        const float2 v = two(acc);
        return fmaxf(fabsf(v.x), fabsf(v.y));
    }
};

struct Fp16Fmt {
    static __device__ __forceinline__ float4 decode(uint2 v) {
        const float2 a = f16x2_to_f32(v.x), b = f16x2_to_f32(v.y);
        return make_float4(a.x, a.y, b.x, b.y);
    }
    static __device__ __forceinline__ uint2 encode(float4 f) {
        uint2 r;
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r.x) : "f"(f.y), "f"(f.x));
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r.y) : "f"(f.w), "f"(f.z));
        return r;
    }
    static __device__ __forceinline__ unsigned amax(unsigned acc, unsigned w) {
        unsigned r;
        asm("max.xorsign.abs.f16x2 %0, %1, %2;" : "=r"(r) : "r"(acc), "r"(w));
        return r;
    }
    static __device__ __forceinline__ float amax_value(unsigned acc) {
        const float2 v = f16x2_to_f32(acc);
        return fmaxf(fabsf(v.x), fabsf(v.y));
    }
};

// Tile geometry of the 16-bit kernel. A thread computes the 4 x-cells
// i..i+3 of the rows j and j+1, so its per-plane costs (waits, the barrier,
// the loads of the x neighbours, bookkeeping) are spread over 8 cells and the
// y neighbours j-4..j-1 and j+2..j+5 serve both rows. Every thread computes:
// there is no producer warp. Ring A (U of a plane with its halo) holds NA
// planes, ring B (the D and W tiles of a plane) NB planes; a plane is
// processed per loop step and NU planes per loop trip (see WS16_TRIP), so
// the register-queue indices and ring-B slots are compile-time constants.
template <int TX, int TY, int NA, int NB>
struct Cfg16 {
    static constexpr int kCols = TX / 4;               // threads across a row
    static constexpr int kThreads = kCols * (TY / 2);
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kLead = 8;                    // halo box starts 8 cells left: 16-byte x
    static constexpr int kRowW = TX + 2 * kLead;       // elements per ring-A row
    static constexpr int kRows = TY + 2 * kHalo;
    static constexpr int kSlotA = kRowW * kRows;       // elements per ring-A slot
    static constexpr unsigned kSlotABytes = kSlotA * 2u;
    static constexpr int kTile = TX * TY;
    static constexpr int kSlotB = 2 * kTile;           // D tile, then W tile (16-bit elements)
    static constexpr unsigned kSlotBBytes = kSlotB * 2u;
    // FP32 staging tile: columns i0-4 .. i0+TX+3, rows j0-4 .. j0+TY+3 (the
    // four corner blocks are never read by the star stencil and stay unset)
    static constexpr int kSW = TX + 2 * kHalo;
    static constexpr int kStage = kSW * kRows;
    // halo cells decoded per plane, in units of 4 cells: 2*TX units in the 8
    // rows above and below the tile, 2*TY units beside it; thread t decodes
    // unit t and, when there are more units than threads, unit t + kThreads
    static constexpr int kBandUnits = 2 * TX;
    static constexpr int kUnits = kBandUnits + 2 * TY;
    static constexpr bool kAllFirst = kUnits >= kThreads;   // every thread has a first unit
    static constexpr bool kSecond = kUnits > kThreads;      // some threads have a second one
    // CTAs per SM that the register file holds at up to 168 registers a thread
    static constexpr int kMinBlocks = 384 / kThreads;
    static_assert(kThreads % 32 == 0 && kMinBlocks >= 1, "whole warps, 128 .. 384 threads");
    static_assert(TX == 64 && TY % 4 == 0 && kBandUnits <= kThreads && kUnits <= 2 * kThreads,
                  "64-wide tiles; one or two halo units per thread");
    static constexpr unsigned kStageBytes = kStage * 4u;
    static_assert(NA == 9 && NB == 3, "ring slots are compile-time constants of a 9-plane trip");
    static_assert(kSlotABytes % 128 == 0 && kSlotBBytes % 128 == 0 && kStageBytes % 128 == 0,
                  "slots stay 128-byte aligned");
    static constexpr size_t kSmem =
        size_t(2) * kStageBytes + size_t(NA) * kSlotABytes + size_t(NB) * kSlotBBytes;
};

struct Maps16 {
    CUtensorMap u, d, w;
};

// Shared-memory accesses at a 32-bit shared address plus a compile-time byte
// offset (negative offsets wrap modulo 2^32, which is the same address) from
// a per-thread base computed once per item (the sum is left to
// the compiler: measured 1 % faster than the offset as an immediate in the
// instruction text).
template <int OFF>
__device__ __forceinline__ uint2 lds2_at(unsigned a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                 : "=r"(v.x), "=r"(v.y)
                 : "r"(a + static_cast<unsigned>(OFF)));
    return v;
}
template <int OFF>
__device__ __forceinline__ void sts4_at(unsigned a, float4 v) {
    asm volatile("st.shared.v4.f32 [%0+%1], {%2, %3, %4, %5};" ::"r"(a), "n"(OFF), "f"(v.x),
                 "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// The stencil weights (zero_sum_weights16() times 2^-kW16Exp) as compile-time
// constants; the launcher checks them against the host computation.
constexpr float kW16C0 = -0x1.11555cp-9f, kW16C1 = 0x1.9999a4p-12f, kW16C2 = -0x1.9999ap-15f,
                kW16C3 = 0x1.a01ap-18f, kW16C4 = -0x1.d42p-22f;

// Barriers of one CTA: a "full" mbarrier per ring slot (transaction bytes);
// no "empty" barriers: a slot is refilled right after the plane barrier
// that follows its last read.
template <int NA, int NB>
struct Bars16 {
    uint64_t fullA[NA], fullB[NB];
    int issuedA[NA], issuedB[NB];   // copies issued into each slot (for the drain)
    int abort;
};

// 2^e as a float, e clamped to the normal range.
__device__ __forceinline__ float pow2f(int e) {
    e = max(-126, min(127, e));
    return __int_as_float((e + 127) << 23);
}

// x * 2^e for e beyond one float's exponent range, in two exact steps.
__device__ __forceinline__ float scale2(float x, int e) {
    const int h = e / 2;
    return x * pow2f(h) * pow2f(e - h);
}

// Exponent that puts a maximum magnitude a near 2^12 (a * 2^e in [2^11, 2^12)).
__device__ __forceinline__ int scale_exponent(float a) {
    if (!(a > 0.0f) || !isfinite(a)) return 0;
    int k;
    frexpf(a, &k);
    return max(-100, min(100, 12 - k));
}

// Rarely taken paths of a plane, kept as small inlined helpers.

// Sources of this plane inside the thread's 8 cells: d~ += W h^2 s in stored
// units (src_mask: the CTA's sources), i.e. (V_s dt)^2 s(t_n) added to
// u^{n+1} after the taper.
__device__ __forceinline__ void inject_sources(float4 *dn, const float4 *wr, unsigned src_mask,
                                               const Sources &src, int i, int j, int k,
                                               float wtrue, float amp2r) {
    for (int qs = 0; qs < src.n; ++qs) {
        const SourceSample &ss = src.s[qs];
        if (((src_mask >> qs) & 1u) && ss.k == k) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (ss.j != j + r) continue;
#pragma unroll
                for (int l = 0; l < 4; ++l)
                    if (ss.i == i + l)
                        set_comp(dn[r], l, fmaf(comp(wr[r], l) * wtrue, ss.amp * amp2r,
                                                comp(dn[r], l)));
            }
        }
    }
}

// Receivers of plane k, values u~ in stored units times 2^r2t (true units);
// returns the new (cursor, next plane).
__device__ __forceinline__ int2 record16(float4 u0, float4 u1, int r2t, int k, int rcur, int rend,
                                         const RecEntry *rec, float *traces, int nt_max,
                                         long long trace_step) {
    const float4 ut[2] = {make_float4(scale2(u0.x, r2t), scale2(u0.y, r2t), scale2(u0.z, r2t),
                                      scale2(u0.w, r2t)),
                          make_float4(scale2(u1.x, r2t), scale2(u1.y, r2t), scale2(u1.z, r2t),
                                      scale2(u1.w, r2t))};
    int next = INT_MAX;
    record_plane2(ut, k, &rcur, rend, &next, rec, traces, nt_max, trace_step);
    return make_int2(rcur, next);
}

// Per-thread state of the walk down an item.
struct Walk16 {
    float4 q[9][2];     // u^n (stored units) of planes k-4 .. k+4, rows j and j+1
    int rcur, rend, rnext_k;
    unsigned amax;      // running max |U'| (two 16-bit magnitudes, sign bits meaningless)
    bool ok;
};

// What a thread needs of its item, fixed over the walk. Shared addresses are
// 32-bit byte addresses of the thread's own place in ring slot 0 / staging
// buffer 0; the slot and buffer offsets are compile-time constants.
struct Ctx16 {
    unsigned aOwn, aUnit1, aUnit2; // ring A: own cells (row j), halo units
    unsigned bOwn;                 // ring B: own D cells (row j); W one tile on
    unsigned sOwn, sUnit1, sUnit2; // staging buffer 0: own cell (row j), halo units
    const float *gz;
    float4 gxy[2];         // gx * gy of the 4 columns per row (0 outside the grid)
    int i, j, z0, z1, nb, nplanes;
    bool unit1, unit2, xy_free, full;
    bool lean;             // xy_free, no source in the item, no change of scale this step
    int fz0, fz1;          // planes whose taper is exactly 1
    int nvalid, pitch;     // valid x cells; row pitch (elements)
    bool row1;             // row j+1 inside the grid
    long long d_delta, plane;
    unsigned src_mask;
};

// Stores of a thread with cells outside the grid (nvalid < 4 or no row j+1).
__device__ __forceinline__ void store_partial(uint16_t *p, long long d_delta, int pitch, uint2 su0,
                                              uint2 sd0, uint2 su1, uint2 sd1, int nvalid,
                                              bool row1) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (r == 1 && !row1) break;
        const uint2 su = r ? su1 : su0, sd = r ? sd1 : sd0;
        uint16_t *o = p + r * pitch;
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            if (l >= nvalid) break;
            const unsigned wu = l < 2 ? su.x : su.y, wd = l < 2 ? sd.x : sd.y;
            o[l] = (uint16_t)((l & 1) ? (wu >> 16) : (wu & 0xffffu));
            o[l + d_delta] = (uint16_t)((l & 1) ? (wd >> 16) : (wd & 0xffffu));
        }
    }
}

// u + d and x * f of 4 cells, as two FP32x2 operations each.
__device__ __forceinline__ float4 add4(const float4 &u, const float4 &d) {
    const float2 a = add2(lo2(u), lo2(d)), b = add2(hi2(u), hi2(d));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 mul4(const float4 &x, float f) {
    const float2 a = mul2(lo2(x), splat(f)), b = mul2(hi2(x), splat(f));
    return make_float4(a.x, a.y, b.x, b.y);
}

// 4 stored values (8 bytes), streaming store.
__device__ __forceinline__ void store16(uint16_t *p, const uint2 st) {
    asm volatile("st.global.cs.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(st.x), "r"(st.y) : "memory");
}

// Planes per loop trip: 9 (the ring depth: every ring slot and queue index
// is a compile-time constant) or 3 (a third of the code, with the queue
// renamed by moves after each trip and the ring-A slots computed). 3 is the
// default: the 9-plane loop body (~45 KB of code) does not stay in the
// instruction caches, and warps waited 1.40 cycles per issued instruction
// for instruction fetch against 0.25 with 3 planes (1024^3 FP16 441 -> 479
// Gcell/s, for 24 more moves per plane; 6-plane trips, 12 moves per plane,
// ran 471 against 497: fetch stalls again).
#ifndef WS16_TRIP
#define WS16_TRIP 3
#endif

template <class Fmt, int TX, int TY, int NA, int NB>
struct Kern16 {
    using Cfg = Cfg16<TX, TY, NA, NB>;
    using B = Bars16<NA, NB>;
    static constexpr int NU = WS16_TRIP;
    static_assert(NU == 9 || NU == 3, "9 or 3 planes per trip");

    // factors of one launch (uniform)
    struct Factors {
        float wtrue;    // stored W -> (V dt/h)^2
        float amp2r;    // source amplitude (h^2 s) -> stored U units
        float ro;       // stored U units -> the output units of U' and D'
        int r2t;        // stored U units -> true units: times 2^r2t
    };

    // U of relative plane pr (interior plane z0 - 4 + pr, with its halo) into
    // ring-A slot `slot`. The maps cover the interior only: box corner
    // (i0 - 8, j0 - 4, z0 - 4 + pr), cells outside the grid arrive as zeros
    // without a memory read; x is a multiple of 8 elements (16 bytes).
    static __device__ __forceinline__ void issue_a(B &br, uint16_t *ringA, const Maps16 &mp,
                                                   const Item &it, int slot, int pr) {
        br.issuedA[slot]++;
        mbar_arrive_expect_tx(&br.fullA[slot], Cfg::kSlotABytes);
        tma_load_3d(ringA + slot * Cfg::kSlotA, &mp.u, &br.fullA[slot], it.i0 - Cfg::kLead,
                    it.j0 - kHalo, it.z0 - kHalo + pr);
    }

    // D and W of interior plane z0 + b into ring-B slot `slot`.
    static __device__ __forceinline__ void issue_b(B &br, uint16_t *ringB, const Maps16 &mp,
                                                   const Item &it, int slot, int b) {
        br.issuedB[slot]++;
        uint16_t *dst = ringB + slot * Cfg::kSlotB;
        mbar_arrive_expect_tx(&br.fullB[slot], Cfg::kSlotBBytes);
        tma_load_3d(dst, &mp.d, &br.fullB[slot], it.i0, it.j0, it.z0 + b);
        tma_load_3d(dst + Cfg::kTile, &mp.w, &br.fullB[slot], it.i0, it.j0, it.z0 + b);
    }

    // The stencil sum of one row's 4 cells (two FP32x2 pairs): c0 u +
    // sum_m c_m s_m, s_m the six neighbours at distance m, each summed as
    // symmetric pairs first. xl, xr: cells x-4..x-1 and x+4..x+7 of the row;
    // yp/ym: rows j+m / j-m of this row; z from the register queue.
    template <int RQ>
    static __device__ __forceinline__ void stencil_row(const Walk16 &wk, int r, const float4 &xl,
                                                       const float4 &xr, const float4 (&yp)[4],
                                                       const float4 (&ym)[4], float2 (&lap)[2]) {
        const float4 xc = wk.q[(RQ + 4) % 9][r];
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
            float2 l = mul2(splat(kW16C0), pair(xc, p));
            l = fma2(splat(kW16C4), s[4], l);
            l = fma2(splat(kW16C3), s[3], l);
            l = fma2(splat(kW16C2), s[2], l);
            lap[p] = fma2(splat(kW16C1), s[1], l);
        }
    }

    // d~ = u~ - u of one row's 4 cells in velocity form, u^{n-1} = u - d:
    // u~ = g (2u - g u^{n-1} + W L) gives d~ = g (W L + g d) - (1 - g)^2 u.
    // With g = 1 (fast) this is W L + d, bit for bit the same value.
    static __device__ __forceinline__ float4 delta_fast(const float2 (&lap)[2], const float4 &d,
                                                        const float4 &w) {
        const float2 a = fma2(lo2(w), lap[0], lo2(d));
        const float2 b = fma2(hi2(w), lap[1], hi2(d));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    static __device__ __forceinline__ float4 delta_taper(const float2 (&lap)[2], const float4 &d,
                                                         const float4 &w, const float4 &u,
                                                         const float4 &gxy, float gzk) {
        float2 o[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float2 g = mul2(pair(gxy, p), splat(gzk));
            const float2 t = mul2(g, fma2(pair(w, p), lap[p], mul2(g, pair(d, p))));
            const float2 gm1 = fma2(pair(gxy, p), splat(gzk), splat(-1.0f));   // g - 1
            const float2 omg = fma2(pair(gxy, p), splat(-gzk), splat(1.0f));   // 1 - g, exactly -(g - 1)
            o[p] = fma2(omg, mul2(gm1, pair(u, p)), t);
        }
        return make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
    }

    // Plane k of the walk, RQ = (k - z0) mod NU; tp: parity of the trip;
    // so: byte offset of plane k's staging buffer; pk: U' of (i, j, k).
    template <int RQ>
    static __device__ __forceinline__ void plane_step(Walk16 &wk, const Ctx16 &cx, B &br,
                                                      uint16_t *ringA, uint16_t *ringB,
                                                      const Maps16 &mp, const Item &it,
                                                      const StepArgs &a, const Factors &fc,
                                                      unsigned so, uint16_t *pk, int k,
                                                      unsigned tp, int ts, unsigned wp,
                                                      const RecEntry *rec) {
        constexpr int Q8 = (RQ + 8) % 9, Q4 = (RQ + 4) % 9;
        constexpr int SB = RQ % NB;
        // plane r fills ring-B slot SB for the (NU trip / 3 + RQ / 3)-th time
        constexpr unsigned PB = (RQ / NB) & 1u;
        const unsigned pb = ((NU / NB) & 1 ? tp : 0u) ^ PB;
        constexpr int OB = SB * Cfg::kSlotBBytes;
        constexpr int RA = Cfg::kRowW * 2, RB = TX * 2, WB = Cfg::kTile * 2, RS = Cfg::kSW * 4;
        const int r = k - cx.z0;
        // ring-A slots of relative planes r + 8 (own cells) and r + 4 (halo),
        // and the parity of the fill the first is waited for: with the trip
        // starting at relative plane 9 w + ts, plane r + 8 fills its slot for
        // the (w + [ts + RQ + 8 >= 9])-th time (wp = w & 1)
        int sa_own, sa_halo;
        unsigned pa;
        if constexpr (NU == 9) {
            sa_own = (RQ + 8) % NA;
            sa_halo = (RQ + 4) % NA;
            pa = wp ^ (((RQ + 8) / NA) & 1u);
        } else {   // ts in {0, 3, 6}: ts + RQ + 8 < 18
            const bool wrap = ts + RQ + 8 >= NA;
            sa_own = wrap ? ts + RQ + 8 - NA : ts + RQ + 8;
            sa_halo = ts + RQ + 4 >= NA ? ts + RQ + 4 - NA : ts + RQ + 4;
            pa = wp ^ (unsigned)wrap;
        }
        const unsigned oa_own = sa_own * Cfg::kSlotABytes, oa_halo = sa_halo * Cfg::kSlotABytes;

        // U of plane k + 4 (ring A) and D, W of plane k (ring B): one test of
        // both barriers, the bounded waits only when either is not complete
        if (!(mbar_try_wait(&br.fullA[sa_own], pa) & mbar_try_wait(&br.fullB[SB], pb)))
            wk.ok = wait_phase(&br.fullA[sa_own], pa, &br.abort, a.status) &&
                    wait_phase(&br.fullB[SB], pb, &br.abort, a.status) && wk.ok;
        // this thread's two rows of plane k + 4 -> the queue (decoded once)
        wk.q[Q8][0] = Fmt::decode(lds2_at<0>(cx.aOwn + oa_own));
        wk.q[Q8][1] = Fmt::decode(lds2_at<RA>(cx.aOwn + oa_own));
        // D and W of plane k (raw; decoded where they are used)
        const uint2 dr0 = lds2_at<OB>(cx.bOwn), dr1 = lds2_at<OB + RB>(cx.bOwn);
        const uint2 wr0 = lds2_at<OB + WB>(cx.bOwn), wr1 = lds2_at<OB + WB + RB>(cx.bOwn);

        // staging tile of plane k: this thread's own two rows (decoded four
        // planes ago) and its halo unit; then every thread agrees before
        // anyone reads a neighbour
        const unsigned st = cx.sOwn + so;
        sts4_at<0>(st, wk.q[Q4][0]);
        sts4_at<RS>(st, wk.q[Q4][1]);
        if (Cfg::kAllFirst || cx.unit1)
            sts4_at<0>(cx.sUnit1 + so, Fmt::decode(lds2_at<0>(cx.aUnit1 + oa_halo)));
        if (Cfg::kSecond && cx.unit2)
            sts4_at<0>(cx.sUnit2 + so, Fmt::decode(lds2_at<0>(cx.aUnit2 + oa_halo)));
        wk.ok = __syncthreads_and(wk.ok) != 0;
        if (!wk.ok) return;
        // every thread is done with ring-A slot SA_HALO (plane k) and ring-B
        // slot SB: refill them with planes k + 9 (U, from warp 0) and k + 3
        // (D, W, from warp 1)
        if (threadIdx.x == 0 && r + 4 + NA < cx.nplanes)
            issue_a(br, ringA, mp, it, sa_halo, r + 4 + NA);
        if (threadIdx.x == 32 && r + NB < cx.nb) issue_b(br, ringB, mp, it, SB, r + NB);

        const float4 xl0 = lds4_at<-16>(st), xr0 = lds4_at<16>(st);
        const float4 xl1 = lds4_at<RS - 16>(st), xr1 = lds4_at<RS + 16>(st);
        // rows j-4..j-1 and j+2..j+5
        const float4 lm[4] = {lds4_at<-RS>(st), lds4_at<-2 * RS>(st), lds4_at<-3 * RS>(st),
                              lds4_at<-4 * RS>(st)};
        const float4 lp[4] = {lds4_at<2 * RS>(st), lds4_at<3 * RS>(st), lds4_at<4 * RS>(st),
                              lds4_at<5 * RS>(st)};
        float2 lap0[2], lap1[2];
        {
            const float4 yp[4] = {wk.q[Q4][1], lp[0], lp[1], lp[2]};
            stencil_row<RQ>(wk, 0, xl0, xr0, yp, lm, lap0);
        }
        {
            const float4 ym[4] = {wk.q[Q4][0], lm[0], lm[1], lm[2]};
            stencil_row<RQ>(wk, 1, xl1, xr1, lp, ym, lap1);
        }
        const float4 d0 = Fmt::decode(dr0), d1 = Fmt::decode(dr1);
        const float4 w0 = Fp16Fmt::decode(wr0), w1 = Fp16Fmt::decode(wr1);
        // the common plane: taper 1 everywhere in the tile, no source, no
        // receiver, no change of scale, every cell inside the grid
        if (cx.lean && (unsigned)(k - cx.fz0) < (unsigned)(cx.fz1 - cx.fz0) && k != wk.rnext_k) {
            const float4 dn0 = delta_fast(lap0, d0, w0), dn1 = delta_fast(lap1, d1, w1);
            const float4 un0 = add4(wk.q[Q4][0], dn0), un1 = add4(wk.q[Q4][1], dn1);
            const uint2 su0 = Fmt::encode(un0), su1 = Fmt::encode(un1);
            const uint2 sd0 = Fmt::encode(dn0), sd1 = Fmt::encode(dn1);
            uint16_t *pd = pk + cx.d_delta;
            store16(pk, su0);
            store16(pd, sd0);
            store16(pk + cx.pitch, su1);
            store16(pd + cx.pitch, sd1);
            wk.amax = Fmt::amax(Fmt::amax(wk.amax, su0.x), su0.y);
            wk.amax = Fmt::amax(Fmt::amax(wk.amax, su1.x), su1.y);
            return;
        }
        float4 dn[2];
        if (cx.xy_free && k >= cx.fz0 && k < cx.fz1) {
            dn[0] = delta_fast(lap0, d0, w0);
            dn[1] = delta_fast(lap1, d1, w1);
        } else {
            const float gzk = cx.gz[k];
            dn[0] = delta_taper(lap0, d0, w0, wk.q[Q4][0], cx.gxy[0], gzk);
            dn[1] = delta_taper(lap1, d1, w1, wk.q[Q4][1], cx.gxy[1], gzk);
        }
        if (cx.src_mask) {
            const float4 w[2] = {w0, w1};
            inject_sources(dn, w, cx.src_mask, a.src, cx.i, cx.j, k, fc.wtrue, fc.amp2r);
        }
        float4 un[2] = {add4(wk.q[Q4][0], dn[0]), add4(wk.q[Q4][1], dn[1])};
        if (k == wk.rnext_k) {
            const int2 rc = record16(un[0], un[1], fc.r2t, k, wk.rcur, wk.rend, rec, a.traces,
                                     a.nt_max, a.trace_step);
            wk.rcur = rc.x;
            wk.rnext_k = rc.y;
        }
        if (fc.ro != 1.0f) {   // the output exponent differs from the input's (rare)
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
                un[rr] = mul4(un[rr], fc.ro);
                dn[rr] = mul4(dn[rr], fc.ro);
            }
        }
        const uint2 su0 = Fmt::encode(un[0]), su1 = Fmt::encode(un[1]);
        const uint2 sd0 = Fmt::encode(dn[0]), sd1 = Fmt::encode(dn[1]);
        if (cx.full) {
            uint16_t *pd = pk + cx.d_delta;
            store16(pk, su0);
            store16(pd, sd0);
            store16(pk + cx.pitch, su1);
            store16(pd + cx.pitch, sd1);
        } else if (cx.nvalid > 0) {
            store_partial(pk, cx.d_delta, cx.pitch, su0, sd0, su1, sd1, cx.nvalid, cx.row1);
        }
        // cells outside the grid have zero taper, so zero u~ (NaN canaries in
        // the padding are ignored by the max)
        wk.amax = Fmt::amax(Fmt::amax(wk.amax, su0.x), su0.y);
        wk.amax = Fmt::amax(Fmt::amax(wk.amax, su1.x), su1.y);
    }

    // After a trip of NU planes starting at plane kb the queue holds planes
    // kb+NU-4 .. kb+NU+3 (the next trip's k-4 .. k+3) in slots rotated by
    // NU: rename them (the 9-plane trip needs no renaming).
    static __device__ __forceinline__ void rotate_queue(Walk16 &wk) {
        if constexpr (NU % 9 != 0) {
            float4 t[9][2];
#pragma unroll
            for (int m = 0; m < 9; ++m) {
                t[m][0] = wk.q[(m + NU) % 9][0];
                t[m][1] = wk.q[(m + NU) % 9][1];
            }
#pragma unroll
            for (int m = 0; m < 9; ++m) {
                wk.q[m][0] = t[m][0];
                wk.q[m][1] = t[m][1];
            }
        }
    }

    // planes kb + RQ .. kb + NU - 1 of a trip; false once the item ends.
    // se / so: staging byte offsets of even / odd RQ; pk: U' of (i, j, kb)
    template <int RQ>
    static __device__ __forceinline__ bool planes(Walk16 &wk, const Ctx16 &cx, B &br,
                                                  uint16_t *ringA, uint16_t *ringB,
                                                  const Maps16 &mp, const Item &it,
                                                  const StepArgs &a, const Factors &fc,
                                                  unsigned se, unsigned so, uint16_t *pk, int kb,
                                                  unsigned tp, int ts, unsigned wp,
                                                  const RecEntry *rec) {
        if constexpr (RQ < NU) {
            if (kb + RQ >= cx.z1) return false;
            plane_step<RQ>(wk, cx, br, ringA, ringB, mp, it, a, fc, (RQ & 1) ? so : se, pk,
                           kb + RQ, tp, ts, wp, rec);
            // wk.ok is the same in every thread after the plane barrier
            if (!wk.ok) return false;
            return planes<RQ + 1>(wk, cx, br, ringA, ringB, mp, it, a, fc, se, so,
                                  pk + cx.plane, kb, tp, ts, wp, rec);
        }
        return true;
    }
};

template <class Fmt, int TX, int TY, int NA, int NB>
__global__ void __launch_bounds__(Cfg16<TX, TY, NA, NB>::kThreads, Cfg16<TX, TY, NA, NB>::kMinBlocks)
    step_stream16_kernel(const __grid_constant__ Maps16 maps, uint16_t *u_out, uint16_t *d_io,
                         const __grid_constant__ StepArgs a,
                         Scale16 *sc, const long long step, const float src_hint,
                         const int zb, const int tiles_x, const int ntiles,
                         const int *__restrict__ rec_ptr, const RecEntry *__restrict__ rec) {
    using K = Kern16<Fmt, TX, TY, NA, NB>;
    using Cfg = typename K::Cfg;
    extern __shared__ __align__(128) float smem16[];
    __shared__ Bars16<NA, NB> br;
    float *stage = smem16;
    uint16_t *ringA = reinterpret_cast<uint16_t *>(smem16 + 2 * Cfg::kStage);
    uint16_t *ringB = ringA + NA * Cfg::kSlotA;
    const Geom &g = a.g;
    const FreeBox &fr = a.fr;
    const int tid = threadIdx.x;

    wait_predecessor();
    // scale of this step: U, D of step n have e; U', D' get e_o
    const int sn = (int)(step & 3), so = (int)((step + 1) & 3);
    const int e = sc->e[sn];
    const int e_o = scale_exponent(fmaxf(__uint_as_float(sc->amax[sn]), src_hint));
    typename K::Factors fc;
    fc.wtrue = pow2f(-kW16Exp);
    fc.amp2r = scale2(1.0f, e);
    fc.ro = pow2f(e_o - e);
    fc.r2t = -e;

    const Item it = item_of(blockIdx.x, tiles_x, ntiles, zb, g.nz, TX, TY);
    const int nb = it.z1 - it.z0, nplanes = nb + 2 * kHalo;
    const bool stall = (int)blockIdx.x == a.stall_item;

    if (tid == 0) {
        if (blockIdx.x == 0) {
            sc->e[so] = e_o;
            sc->amax[(step + 2) & 3] = 0u;  // accumulated by the next step
        }
        for (int s = 0; s < NA; ++s) {
            mbar_init(&br.fullA[s], 1);
            br.issuedA[s] = 0;
        }
        for (int s = 0; s < NB; ++s) {
            mbar_init(&br.fullB[s], 1);
            br.issuedB[s] = 0;
        }
        br.abort = 0;
        fence_mbar_init();
    }
    __syncthreads();
    // first fills: U planes 0 .. NA-1 of the item (z0-4 ..), D/W planes 0 .. NB-1
    if (tid == 0) {
        for (int pr = 0; pr < NA && pr < nplanes; ++pr)
            if (!(pr == 0 && stall))   // test hook: never filled, the bounded waits run out
                K::issue_a(br, ringA, maps, it, pr, pr);
        for (int b = 0; b < NB && b < nb; ++b) K::issue_b(br, ringB, maps, it, b, b);
    }

    Ctx16 cx;
    const int tx = tid % Cfg::kCols, py = tid / Cfg::kCols;
    cx.i = it.i0 + 4 * tx;
    cx.j = it.j0 + 2 * py;
    cx.z0 = it.z0;
    cx.z1 = it.z1;
    cx.nb = nb;
    cx.nplanes = nplanes;
    {
        const unsigned rA = smem_addr(ringA), rB = smem_addr(ringB), st0 = smem_addr(stage);
        cx.aOwn = rA + 2u * ((kHalo + 2 * py) * Cfg::kRowW + Cfg::kLead + 4 * tx);
        cx.bOwn = rB + 2u * (2 * py * TX + 4 * tx);
        cx.sOwn = st0 + 4u * ((kHalo + 2 * py) * Cfg::kSW + kHalo + 4 * tx);
        // halo unit u: u < 2 TX, 4 cells above/below the tile (rows 0..3,
        // TY+4..TY+7 of the staging tile); else 4 cells left/right of row
        // (u - 2 TX) / 2. Source and destination offsets of unit u:
        auto unit = [&](int u, unsigned *a, unsigned *s) {
            int y, c;
            if (u < Cfg::kBandUnits) {
                const int band = u / Cfg::kCols;
                y = band < kHalo ? band : TY + band;
                c = kHalo + 4 * (u - band * Cfg::kCols);
            } else {
                const int v = u - Cfg::kBandUnits;
                y = kHalo + (v >> 1);
                c = (v & 1) ? TX + kHalo : 0;
            }
            *a = rA + 2u * (y * Cfg::kRowW + c + (Cfg::kLead - kHalo));
            *s = st0 + 4u * (y * Cfg::kSW + c);
        };
        cx.unit1 = tid < Cfg::kUnits;
        cx.unit2 = tid + Cfg::kThreads < Cfg::kUnits;
        unit(cx.unit1 ? tid : 0, &cx.aUnit1, &cx.sUnit1);
        unit(cx.unit2 ? tid + Cfg::kThreads : 0, &cx.aUnit2, &cx.sUnit2);
    }
    const bool col_ok = (cx.j < g.ny) && (cx.i < g.nx);
    cx.nvalid = col_ok ? min(4, g.nx - cx.i) : 0;
    cx.row1 = cx.j + 1 < g.ny;
    cx.full = cx.nvalid == 4 && cx.row1;
    cx.pitch = g.pnx;
    cx.plane = g.plane;
    cx.d_delta = d_io - u_out;
    uint16_t *pu = u_out + pidx(g, col_ok ? cx.i : 0, col_ok ? cx.j : 0, it.z0);
    cx.gz = a.gz;
    cx.fz0 = fr.z0;
    cx.fz1 = fr.z1;
    cx.xy_free = it.i0 >= fr.x0 && it.i0 + TX <= fr.x1 && it.j0 >= fr.y0 && it.j0 + TY <= fr.y1;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
        cx.gxy[rr] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (col_ok && cx.j + rr < g.ny) {
            const float gyj = a.gy[cx.j + rr];
            cx.gxy[rr].x = a.gx[cx.i] * gyj;
            if (cx.nvalid > 1) cx.gxy[rr].y = a.gx[cx.i + 1] * gyj;
            if (cx.nvalid > 2) cx.gxy[rr].z = a.gx[cx.i + 2] * gyj;
            if (cx.nvalid > 3) cx.gxy[rr].w = a.gx[cx.i + 3] * gyj;
        }
    }
    cx.src_mask = 0u;
    for (int qs = 0; qs < a.src.n; ++qs) {
        const SourceSample &ss = a.src.s[qs];
        if (ss.i >= it.i0 && ss.i < it.i0 + TX && ss.j >= it.j0 && ss.j < it.j0 + TY &&
            ss.k >= it.z0 && ss.k < it.z1)
            cx.src_mask |= 1u << qs;
    }
    cx.lean = cx.xy_free && cx.src_mask == 0u && fc.ro == 1.0f;

    Walk16 wk;
    wk.ok = true;
    wk.amax = 0u;
    wk.rcur = wk.rend = 0;
    if (rec_ptr != nullptr) {
        const int rt = it.tile * Cfg::kWarps + (tid >> 5);
        wk.rend = rec_ptr[rt + 1];
        wk.rcur = first_entry(rec, rec_ptr[rt], wk.rend, it.z0);
    }
    wk.rnext_k = wk.rcur < wk.rend ? rec[wk.rcur].k : INT_MAX;

    // queue prologue: U planes z0-4 .. z0+3 (relative 0..7)
#pragma unroll
    for (int m = 0; m < 2 * kHalo; ++m) {
        wk.ok = wk.ok && wait_phase(&br.fullA[m], 0u, &br.abort, a.status);
        const uint16_t *p = ringA + m * Cfg::kSlotA + (cx.aOwn - smem_addr(ringA)) / 2;
        wk.q[m][0] = Fmt::decode(lds2u(p));
        wk.q[m][1] = Fmt::decode(lds2u(p + Cfg::kRowW));
    }
    wk.ok = __syncthreads_and(wk.ok) != 0;
    if (wk.ok) {
        // planes z0-4 .. z0-1 were needed only here: refill their slots
        if (tid == 0)
            for (int pr = NA; pr < NA + kHalo && pr < nplanes; ++pr)
                K::issue_a(br, ringA, maps, it, pr - NA, pr);
        // tp: trip parity; ts, wp: the trip's first relative plane mod 9 and
        // the parity of its quotient (the ring-A wrap count)
        unsigned tp = 0, wp = 0;
        int ts = 0;
        for (int kb = it.z0;; kb += K::NU, tp ^= 1u) {
            // staging buffer of plane k: k & 1
            const unsigned se = (kb & 1) * Cfg::kStageBytes, sodd = Cfg::kStageBytes - se;
            if (!K::template planes<0>(wk, cx, br, ringA, ringB, maps, it, a, fc, se, sodd,
                                       pu + (long long)(kb - it.z0) * cx.plane, kb, tp, ts, wp,
                                       rec))
                break;
            K::rotate_queue(wk);
            ts += K::NU;
            if (ts >= NA) {
                ts -= NA;
                wp ^= 1u;
            }
        }
    }

    // max |U'| of this warp, in true units, into the next step's slot
    float m = scale2(Fmt::amax_value(wk.amax), -e_o);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) atomicMax(&sc->amax[so], __float_as_uint(m));

    // after an abort, wait (bounded) for the last copy issued into each slot
    __syncthreads();
    if (br.abort && tid == 0) {
        for (int s = 0; s < NA + NB; ++s) {
            const int c = s < NA ? br.issuedA[s] : br.issuedB[s - NA];
            uint64_t *bar = s < NA ? &br.fullA[s] : &br.fullB[s - NA];
            if (c == 0) continue;
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(bar, (unsigned)(c - 1) & 1u) && global_ns() - t0 < kWaitLimitNs) {
            }
        }
    }
}

// Resident CTAs per SM and SM count of one instantiation on the current
// device, looked up (and its shared-memory limit set) the first time.
template <class Fmt, int TX, int TY, int NA, int NB>
cudaError_t facts16(int *ctas, int *sms) {
    using Cfg = Cfg16<TX, TY, NA, NB>;
    auto kern = step_stream16_kernel<Fmt, TX, TY, NA, NB>;
    static LaunchFacts lf;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= LaunchFacts::kMaxDevices) return cudaErrorInvalidDevice;
    if (lf.ctas[dev] == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)Cfg::kSmem);
        int c = 0, n = 0;
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, kern, Cfg::kThreads, Cfg::kSmem);
        if (e != cudaSuccess) return e;
        if (c < 1) return cudaErrorInvalidConfiguration;
        lf.sms[dev] = n;
        lf.ctas[dev] = c;
    }
    *ctas = lf.ctas[dev];
    *sms = lf.sms[dev];
    return cudaSuccess;
}

template <class Fmt, int TX, int TY, int NA, int NB>
cudaError_t launch16(const Maps16 &maps, uint16_t *u_out, uint16_t *d_io, const StepArgs &a,
                     Scale16 *sc, long long step, float src_hint, int zb,
                     const int *rec_ptr, const RecEntry *rec, cudaStream_t s) {
    using Cfg = Cfg16<TX, TY, NA, NB>;
    auto kern = step_stream16_kernel<Fmt, TX, TY, NA, NB>;
    int ctas = 0, sms = 0;
    cudaError_t e = facts16<Fmt, TX, TY, NA, NB>(&ctas, &sms);
    if (e != cudaSuccess) return e;
    const int tiles_x = (a.g.nx + TX - 1) / TX;
    const int ntiles = tiles_x * ((a.g.ny + TY - 1) / TY);
    const int nitems = ntiles * ((a.g.nz + zb - 1) / zb);
    return launch_overlapped(kern, nitems, Cfg::kThreads, Cfg::kSmem, s, maps, u_out, d_io, a, sc,
                             step, src_hint, zb, tiles_x, ntiles, rec_ptr, rec);
}

}  // namespace

bool stream16_tiling_supported(int tx, int ty) {
    return tx == 64 && (ty == 16 || ty == 24 || ty == 48);
}

cudaError_t stream16_slots(int ty, int *slots, int *sms) {
    int c = 0, n = 0;
    cudaError_t e = cudaErrorInvalidValue;
    if (ty == 16) e = facts16<Fp16Fmt, 64, 16, 9, 3>(&c, &n);
    if (ty == 24) e = facts16<Fp16Fmt, 64, 24, 9, 3>(&c, &n);
    if (ty == 48) e = facts16<Fp16Fmt, 64, 48, 9, 3>(&c, &n);
    if (e == cudaSuccess) *slots = c * n;
    if (e == cudaSuccess && sms) *sms = n;
    return e;
}

// Weights of the 16-bit kernel, times 2^-kW16Exp: floats within 7e-7 of the
// Taylor weights, chosen so that c0 = -6 (c1 + c2 + c3 + c4) holds exactly.
// The operator is then free of a mass term (it annihilates constants in
// exact arithmetic) while the centre weight is applied as one multiply
// instead of four FMAs. c2..c4 lie on a grid of 2^-23; S = c1 + ... + c4 is
// the multiple of 2^-21 (so 6 S is a float) nearest to the sum with the c1
// that keeps the second moment sum_m m^2 c_m = 1 exact, and
// c1 = S - (c2 + c3 + c4) (its second moment is then off by < 2.4e-7).
Weights16 zero_sum_weights16() {
    auto grid = [](double x, double q) { return std::nearbyint(x / q) * q; };
    const double q23 = std::ldexp(1.0, -23), q21 = std::ldexp(1.0, -21);
    const double c2 = grid(-1.0 / 5.0, q23), c3 = grid(8.0 / 315.0, q23), c4 = grid(-1.0 / 560.0, q23);
    const double t = c2 + c3 + c4;
    const double S = grid(1.0 - 4.0 * c2 - 9.0 * c3 - 16.0 * c4 + t, q21);
    const double c1 = S - t;
    const double c0 = -6.0 * S;
    const double f = std::ldexp(1.0, -kW16Exp);
    return Weights16{(float)(c0 * f), (float)(c1 * f), (float)(c2 * f), (float)(c3 * f),
                     (float)(c4 * f)};
}

cudaError_t launch_step_stream16(int storage, const Maps16In &m, const StepArgs &a, Scale16 *sc,
                                 long long step, float src_hint, const StreamTiling &t,
                                 const int *rec_ptr, const RecEntry *rec,
                                 cudaStream_t s) {
    // the kernel's compile-time weights must be those of zero_sum_weights16
    static const bool weights_ok = [] {
        const Weights16 w = zero_sum_weights16();
        return w.c0 == kW16C0 && w.c1 == kW16C1 && w.c2 == kW16C2 && w.c3 == kW16C3 &&
               w.c4 == kW16C4;
    }();
    if (!weights_ok) return cudaErrorInvalidValue;
    if (!stream16_tiling_supported(t.tx, t.ty)) return cudaErrorInvalidValue;
    Maps16 maps;
    maps.u = *m.u;
    maps.d = *m.d;
    maps.w = *m.w;
    // ring A 9 slots (the planes of one loop trip), ring B 3; 64 x 16 tiles
    // run 3 CTAs per SM, 64 x 24 two, 64 x 48 one (12 warps in all)
#define WS_LAUNCH16(FMT, TY)                                                                     \
    return launch16<FMT, 64, TY, 9, 3>(maps, m.u_out, m.d_io, a, sc, step, src_hint, t.zb, \
                                       rec_ptr, rec, s)
    if (storage == WS_STORAGE_BF16) {
        if (t.ty == 16) WS_LAUNCH16(Bf16Fmt, 16);
        if (t.ty == 24) WS_LAUNCH16(Bf16Fmt, 24);
        if (t.ty == 48) WS_LAUNCH16(Bf16Fmt, 48);
    }
    if (storage == WS_STORAGE_FP16) {
        if (t.ty == 16) WS_LAUNCH16(Fp16Fmt, 16);
        if (t.ty == 24) WS_LAUNCH16(Fp16Fmt, 24);
        if (t.ty == 48) WS_LAUNCH16(Fp16Fmt, 48);
    }
#undef WS_LAUNCH16
    return cudaErrorInvalidValue;
}

// ------------------------------------------------------------ conversions
//
// Bound: HBM. Every kernel walks the rows (row_grid) in vectors of 4 cells,
// one 8-byte access a 16-bit field and vector, and reads or writes the
// caller's unpadded arrays or the padded FP32 fields alike (Fp32Fields). One
// cell a thread, through the padded fields, with one atomic a warp for the
// maximum, a 1024^3 state took 32.9 ms in, 6.8 out and its model 4.2; now 1.19
// (amax2, 7.2 TB/s) + 1.91 (encode, 6.8), 2.10 (decode, 6.1), 0.96 ms.

namespace {

// Row j of plane k: 4 cells from cell i on, zeros beyond nx or without a field.
template <bool kVec>
__device__ __forceinline__ float4 row_load(const float *row, int i, int nx) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!row) return v;
    if constexpr (kVec) return *reinterpret_cast<const float4 *>(row + i);
    v.x = row[i];
    if (i + 1 < nx) v.y = row[i + 1];
    if (i + 2 < nx) v.z = row[i + 2];
    if (i + 3 < nx) v.w = row[i + 3];
    return v;
}

template <bool kVec>
__device__ __forceinline__ void row_store(float *row, int i, int nx, const float4 &v) {
    if (!row) return;
    if (kVec && i + 4 <= nx) {
        *reinterpret_cast<float4 *>(row + i) = v;
        return;
    }
    row[i] = v.x;
    if (i + 1 < nx) row[i + 1] = v.y;
    if (i + 2 < nx) row[i + 2] = v.z;
    if (i + 3 < nx) row[i + 3] = v.w;
}

// 4 packed 16-bit values to cells i .. of a padded row, none beyond nx.
__device__ __forceinline__ void row_store16(uint16_t *row, int i, int nx, uint2 v) {
    if (i + 4 <= nx) {
        *reinterpret_cast<uint2 *>(row + i) = v;
        return;
    }
    row[i] = (uint16_t)(v.x & 0xffffu);
    if (i + 1 < nx) row[i + 1] = (uint16_t)(v.x >> 16);
    if (i + 2 < nx) row[i + 2] = (uint16_t)(v.y & 0xffffu);
}

// This thread group's rows: calls fn(k, j) for each.
template <class F>
__device__ __forceinline__ void for_rows(unsigned ny, unsigned rows, F &&fn) {
    for (unsigned long long r = (unsigned long long)blockIdx.x * blockDim.y + threadIdx.y; r < rows;
         r += (unsigned long long)gridDim.x * blockDim.y) {
        const unsigned k = (unsigned)r / ny;
        fn(k, (unsigned)r - k * ny);
    }
}

__device__ __forceinline__ float amax_of(const float4 &u, const float4 &p) {
    const float a = fmaxf(fmaxf(fabsf(u.x), fabsf(u.y)), fmaxf(fabsf(u.z), fabsf(u.w)));
    const float d = fmaxf(fmaxf(fabsf(u.x - p.x), fabsf(u.y - p.y)),
                          fmaxf(fabsf(u.z - p.z), fabsf(u.w - p.w)));
    return fmaxf(a, d);
}

// max |u| and max |u - up| over the grid into *amax (float bits).
template <bool kVec>
__global__ void __launch_bounds__(kRowThreads)
    amax2_kernel(const Fp32Fields f, const int nx, const unsigned ny, const unsigned rows,
                 unsigned *__restrict__ amax) {
    float m = 0.0f;
    const int step = 4 * blockDim.x;
    for_rows(ny, rows, [&](unsigned k, unsigned j) {
        const long long o = k * f.plane + (long long)j * f.pitch;
        const float *u = f.u ? f.u + o : nullptr, *p = f.up ? f.up + o : nullptr;
        for (int i = 4 * threadIdx.x; i < nx; i += 2 * step) {
            const int i2 = i + step < nx ? i + step : i;   // two vectors in flight
            const float4 u0 = row_load<kVec>(u, i, nx), u1 = row_load<kVec>(u, i2, nx);
            const float4 p0 = row_load<kVec>(p, i, nx), p1 = row_load<kVec>(p, i2, nx);
            m = fmaxf(m, fmaxf(amax_of(u0, p0), amax_of(u1, p1)));
        }
    });
    __shared__ unsigned best;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    if (tid == 0) best = 0u;
    __syncthreads();
    const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));   // m >= 0
    if ((tid & 31) == 0) atomicMax(&best, w);
    __syncthreads();
    if (tid == 0) atomicMax(amax, best);
}

__device__ __forceinline__ float4 scale4(const float4 &x, float f0, float f1) {
    return make_float4(x.x * f0 * f1, x.y * f0 * f1, x.z * f0 * f1, x.w * f0 * f1);
}

// FP32 (u^n, u^{n-1}) -> U = u^n, D = u^n - u^{n-1} (16-bit, interior; U and D
// at interior cell 0), with the exponent from the maximum of slot `slot`;
// block 0 records it.
template <class Fmt, bool kVec>
__global__ void __launch_bounds__(kRowThreads)
    encode_kernel(const Fp32Fields f, uint16_t *__restrict__ U, uint16_t *__restrict__ D,
                  const int nx, const unsigned ny, const unsigned rows, const int pitch,
                  const long long plane, Scale16 *__restrict__ sc, int slot) {
    const int e = scale_exponent(__uint_as_float(sc->amax[slot]));
    const float f0 = pow2f(e / 2), f1 = pow2f(e - e / 2);   // the factors of scale2
    if (blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) sc->e[slot] = e;
    for_rows(ny, rows, [&](unsigned k, unsigned j) {
        const long long o = k * f.plane + (long long)j * f.pitch;
        const float *u = f.u ? f.u + o : nullptr, *p = f.up ? f.up + o : nullptr;
        const long long q = k * plane + (long long)j * pitch;
        for (int i = 4 * threadIdx.x; i < nx; i += 4 * blockDim.x) {
            const float4 a = row_load<kVec>(u, i, nx), b = row_load<kVec>(p, i, nx);
            const float4 d = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
            row_store16(U + q, i, nx, Fmt::encode(scale4(a, f0, f1)));
            row_store16(D + q, i, nx, Fmt::encode(scale4(d, f0, f1)));
        }
    });
}

// U, D (16-bit) -> FP32 u^n = U, u^{n-1} = U - D (interior).
template <class Fmt, bool kVec>
__global__ void __launch_bounds__(kRowThreads)
    decode_kernel(const uint16_t *__restrict__ U, const uint16_t *__restrict__ D, const Fp32Out f,
                  const int nx, const unsigned ny, const unsigned rows, const int pitch,
                  const long long plane, const Scale16 *__restrict__ sc, int slot) {
    const int e = -sc->e[slot];
    const float f0 = pow2f(e / 2), f1 = pow2f(e - e / 2);
    for_rows(ny, rows, [&](unsigned k, unsigned j) {
        const long long o = k * f.plane + (long long)j * f.pitch;
        float *u = f.u ? f.u + o : nullptr, *p = f.up ? f.up + o : nullptr;
        const long long q = k * plane + (long long)j * pitch;
        for (int i = 4 * threadIdx.x; i < nx; i += 4 * blockDim.x) {
            // a ragged row's last vector reaches into its halo
            const float4 a = scale4(Fmt::decode(*reinterpret_cast<const uint2 *>(U + q + i)), f0, f1);
            const float4 d = scale4(Fmt::decode(*reinterpret_cast<const uint2 *>(D + q + i)), f0, f1);
            row_store<kVec>(u, i, nx, a);
            row_store<kVec>(p, i, nx, make_float4(a.x - d.x, a.y - d.y, a.z - d.z, a.w - d.w));
        }
    });
}

// (V dt/h)^2 (FP32 padded) -> FP16 of value * 2^kW16Exp (interior; both at
// interior cell 0).
__global__ void __launch_bounds__(kRowThreads)
    model16_kernel(const float *__restrict__ w, uint16_t *__restrict__ w16, const int nx,
                   const unsigned ny, const unsigned rows, const int pitch, const long long plane) {
    for_rows(ny, rows, [&](unsigned k, unsigned j) {
        const long long q = k * plane + (long long)j * pitch;
        for (int i = 4 * threadIdx.x; i < nx; i += 4 * blockDim.x) {
            const float4 v = *reinterpret_cast<const float4 *>(w + q + i);
            row_store16(w16 + q, i, nx, Fp16Fmt::encode(mul4(v, (float)(1 << kW16Exp))));
        }
    });
}

}  // namespace

cudaError_t launch_encode16(int storage, const Fp32Fields &f, uint16_t *U, uint16_t *D,
                            const Geom &g, Scale16 *sc, int slot, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(&sc->amax[slot], 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const unsigned rows = (unsigned)g.ny * (unsigned)g.nz;
    const long long o = pidx(g, 0, 0, 0);
    dim3 block;
    const unsigned grid = row_grid(g, &block);
    e = launch(f.vec ? amax2_kernel<true> : amax2_kernel<false>, grid, block, 0, s, f, g.nx, g.ny, rows,
               &sc->amax[slot]);
    if (e != cudaSuccess) return e;
#define WS_ENCODE(FMT, V)                                                                         \
    launch(encode_kernel<FMT, V>, grid, block, 0, s, f, U + o, D + o, g.nx, g.ny, rows, g.pnx, \
           g.plane, sc, slot)
    if (storage == WS_STORAGE_BF16) return f.vec ? WS_ENCODE(Bf16Fmt, true) : WS_ENCODE(Bf16Fmt, false);
    return f.vec ? WS_ENCODE(Fp16Fmt, true) : WS_ENCODE(Fp16Fmt, false);
#undef WS_ENCODE
}

cudaError_t launch_decode16(int storage, const uint16_t *U, const uint16_t *D, const Fp32Out &f,
                            const Geom &g, const Scale16 *sc, int slot, cudaStream_t s) {
    const unsigned rows = (unsigned)g.ny * (unsigned)g.nz;
    const long long o = pidx(g, 0, 0, 0);
    dim3 block;
    const unsigned grid = row_grid(g, &block);
#define WS_DECODE(FMT, V)                                                                         \
    launch(decode_kernel<FMT, V>, grid, block, 0, s, U + o, D + o, f, g.nx, g.ny, rows, g.pnx, \
           g.plane, sc, slot)
    if (storage == WS_STORAGE_BF16) return f.vec ? WS_DECODE(Bf16Fmt, true) : WS_DECODE(Bf16Fmt, false);
    return f.vec ? WS_DECODE(Fp16Fmt, true) : WS_DECODE(Fp16Fmt, false);
#undef WS_DECODE
}

cudaError_t launch_model16(const float *w, uint16_t *w16, const Geom &g, cudaStream_t s) {
    const long long o = pidx(g, 0, 0, 0);
    dim3 block;
    const unsigned grid = row_grid(g, &block);
    return launch(model16_kernel, grid, block, 0, s, w + o, w16 + o, g.nx, g.ny,
                  (unsigned)g.ny * (unsigned)g.nz, g.pnx, g.plane);
}

}  // namespace ws
