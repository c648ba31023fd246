// ssvp_gather.cu - the fused scene-space gather + filter kernel (steps A3-A7).
//
// One thread per output pixel p of frame O, CTAs of 32 x 8 pixels.  For every window slot j
// (frame J = O - T + j) the thread projects its reference point into J, tests the k x k
// candidates around the projection against the radius (the back-projection test of Eq. 2,
// seeded by the output depth) and accumulates the Eq. 4 weighted colour (Eq. 3).
//
// Precision.  The radius is ~0.5 % of the scene depth, so the distance test needs the reference
// point in J's pixel grid to ~1e-9 relative, beyond FP32.  The per-(pixel, J) reference
// quantities (u', v' = projected position, z' = depth in J) are therefore carried as unevaluated
// FP32 pairs ("double-float", error-free transformations with FMA), computed from the FP64 camera
// composition the host splits into hi/lo pairs.  The per-candidate test then only forms small
// differences, all in plain FP32:
//     Y_q - y_ref = ((d_q - z') (q_x - c_x) + z' (q_x - u')) / f_x, ... , d_q - z'
// so the FP32 error of the distance is ~1e-7 of the radius rather than ~1e-7 of the depth.
//
// Two loops per (pixel, J).  The test loop runs over the k x k window two columns at a time (aligned
// 8-byte loads, packed FP32x2) and only decides which candidates can be samples: by the depth part of
// the distance alone, or, where the radius is small against the window, by all of it (see lateral).
// Its threshold is widened so that it keeps every sample; the sign of each result is shifted into a bit
// mask.  The filter loop takes the mask's bits, three (FP32 colour) or two at a time so that their
// loads overlap, decides membership by the exact test above and accumulates; a warp pays for it as
// often as its busiest lane has survivors.
//
// What bounds it (720p, +-15, k = 7, FP32; ncu): instruction issue, 0.70 of the slots, with the filter
// loop two thirds of the instructions (15 of 32 lanes active in it) and the loads' latency behind
// the rest; DRAM at 8 %.  Testing the depth first, the short projection and x/y-paired filter
// arithmetic took one 1080p +-30 frame from 5.47 to 3.97 ms, one 720p +-15 frame from 1.23 to 0.94 ms
// (k = 5: 0.81 to 0.61), and the mixed clips' plan, 640 x 360 to 720p with FP16 colour, from 14.1 to 13.2.
#include <cuda.h>  // CUtensorMap (the type only; the host encodes maps through the runtime's driver entry point)
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "../../include/ssvp.h"
#include "ssvp_df.cuh"
#include "ssvp_dispatch.h"
#include "ssvp_internal.h"

namespace ssvp {
namespace {

#ifndef SSVP_MIN_CTAS
#define SSVP_MIN_CTAS 4  // resident CTAs per SM the register allocation must allow
#endif
// The extraction gather of the learned filter keeps more values live than the plain one: at 64 registers (four CTAs
// per SM) it spills 96 bytes a thread, at 80 (three CTAs) none.  640 x 360 (two waves of three), +-10: 531 against 508
// us a learned frame; but where four CTAs an SM hold the whole launch in one wave and three do not, four are better:
// 480 x 270, +-6, +-10 and +-15, 245, 312 and 374 against 257, 333 and 402 us; 532 x 293, a little more than one wave
// of four, +-10, 394 against 383.
constexpr int kLearnCtas = 3;

#ifndef SSVP_TILE_Y
#define SSVP_TILE_Y 8  // output rows per CTA (a warp covers 32 pixels of one row)
#endif
constexpr int kTileX = 32, kTileY = SSVP_TILE_Y, kThreads = kTileX * kTileY;
// ---------------------------------------------------------------- TMA staging of the window frames
// SSVP_GATHER_WINDOW_TMA.  Each warp (32 output pixels of one row) stages, for every window frame J,
// the depth of a kBoxW x kBoxH box of J's padded depth plane into shared memory with one 3-D tensor
// copy (cp.async.bulk.tensor, completion counted on an mbarrier), in two buffers: the copy of frame
// j + 1 is issued before frame j is tested.  The box is placed around the window of the warp's first
// gathering lane, whose projection into J is recomputed in FP32 for the purpose (a box needs no
// more); on a smooth surface the other lanes' windows lie beside it.  A lane whose window is not
// inside the box (at depth edges neighbouring pixels reproject far apart) tests from the global
// plane, so membership and results are those of the global-load path.  The waits are bounded: on a
// time-out the warp raises bit 1 of the error word, returns to global loads for its remaining
// frames, and its issuing lane waits once more (bounded) for the copies it has in flight.
constexpr int kBoxW = 48, kBoxH = 12;               // floats; a box row is 192 bytes (a multiple of 16)
constexpr unsigned kBoxBytes = kBoxW * kBoxH * 4;   // 2,304 bytes, a multiple of 128
constexpr int kNoBox = 0x40000000;                  // origin of a buffer holding no box: no window fits
constexpr int kStageMaxK = 7;
constexpr unsigned kStgWaitHintNs = 100000, kStgWaitLimit = 10000;  // about 1 s per wait

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// bounded wait for the completion of the phase with parity `parity`; false on time-out
__device__ __forceinline__ bool stg_wait(unsigned bar, unsigned parity) {
    for (unsigned it = 0; it < kStgWaitLimit; ++it) {
        unsigned done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity), "r"(kStgWaitHintNs)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Per warp of a staging CTA: two mbarriers (one per box) and the origin (x, y) in J's padded plane
// of each box, or kNoBox.  The boxes themselves follow the slot geometry in dynamic shared memory,
// 128-byte aligned, two per warp.
constexpr int kStgWarps = kThreads / 32;
__shared__ unsigned long long g_stg_bar[kStgWarps][2];
__shared__ int2 g_stg_org[kStgWarps][2];

// shared-space address of buffer b of this warp's boxes (the slot geometry has n_slots entries)
__device__ __forceinline__ unsigned stg_box(const float4 *sgeom, int n_slots, int b) {
    const unsigned end = smem_addr(sgeom + kSlotVec * n_slots);
    return ((end + 127u) & ~127u) + ((threadIdx.x >> 5) * 2 + b) * kBoxBytes;
}
__device__ __forceinline__ unsigned stg_bar(int b) { return smem_addr(&g_stg_bar[threadIdx.x >> 5][b]); }

// Issue the copy of window slot s (frame J), the seq-th in the warp's order, into buffer seq & 1: called by the warp's first gathering
// lane, whose pixel offset in the tile is (du, dv), depth dref and lane index `lane`; tmap describes
// the clip's depth planes ({pitch, rows, F} floats, box {kBoxW, kBoxH, 1}).  skip (a test of the
// time-out path): the barrier is told to expect the box's bytes but no copy is issued, so the wait
// for it runs out.
template <int K>
__device__ __forceinline__ void stage_issue(const CUtensorMap *tmap, const float4 *sgeom, int n_slots, int s, int seq, float du,
                                            float dv, float dref, int lane, bool skip) {
    constexpr int h = (K - 1) / 2;
    const int b = seq & 1;
    const float4 *g = sgeom + kSlotVec * s;
    const int J = __float_as_int(g[5].w);
    int x0 = kNoBox, y0 = kNoBox;
    if (J >= 0) {
        const float4 q0 = g[0], q1 = g[1], q2 = g[2], q3 = g[3];
        const float w0 = fmaf(dref, q0.x + fmaf(q1.x, du, q1.z * dv), q2.x);
        const float w1 = fmaf(dref, q0.y + fmaf(q1.y, du, q1.w * dv), q2.y);
        const float w2 = fmaf(dref, q3.x + fmaf(q3.z, du, q3.w * dv), g[4].x);
        if (w2 > 1e-6f * dref) {
            const float rz = rcp_approx(w2), U = w0 * rz, V = w1 * rz;
            if (fabsf(U) < 1e6f && fabsf(V) < 1e6f) {
                const int ax = (int)floorf(U + 0.5f), ay = (int)floorf(V + 0.5f);
                // the warp's windows span columns [ax - lane - h, ax - lane + 31 + h]: centre them in
                // the box, x rounded down to a multiple of 4 floats (16 bytes, as tensor copies need)
                x0 = (ax - lane - h + kPad - (kBoxW - 34 - K) / 2) & ~3;
                y0 = ay - h + kPad - (kBoxH - K) / 2;
            }
        }
    }
    g_stg_org[threadIdx.x >> 5][b] = make_int2(x0, y0);
    const unsigned bar = stg_bar(b);
    if (x0 != kNoBox) {
        const unsigned dst = stg_box(sgeom, n_slots, b);
        // the warp's generic-proxy reads of this buffer (frame s - 2) precede the copy's writes
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(kBoxBytes) : "memory");
        if (!skip)
            asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
            "[%5];\n" ::"r"(dst),
            "l"(reinterpret_cast<unsigned long long>(tmap)), "r"(x0), "r"(y0), "r"(J), "r"(bar)
            : "memory");
    } else {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
    }
}

// The slot after jj in the order by groups ((group0 + jj) mod 4 rising, then jj); jj = -4: the first slot; -1
// after the last
__device__ __forceinline__ int next_slot(int jj, int group0, int n_slots) {
    if (jj >= 0 && jj + 4 < n_slots) return jj + 4;
    for (int g = jj < 0 ? 0 : ((group0 + jj) & 3) + 1; g < 4; ++g) {
        const int first = (g - group0) & 3;
        if (first < n_slots) return first;
    }
    return -1;
}

// The gather and filter of one output pixel (u, v) of frame O (steps A3-A7).  sgeom holds the
// per-slot geometry built for the tile whose first pixel is (u0, v0).  n_acc, n_exam and acc_w
// return the pixel's accepted and examined counts and sum of weights (they start at 0).
// K > 0: compile-time window width (k*k <= 64, one 64-bit accept mask per frame).
// K == 0: runtime k up to 31, one 32-bit accept mask per window row.
constexpr int kMaxSamples = 64;  // learned filter: capped sample set
constexpr float kLn2 = 0.6931471805599453f;

// One accepted sample of the learned filter's capped set, compactly: its FP32 colour with the
// BF16 pair (dist / r, (J - O) / T) in one 16-byte record and the pair (depth residual / r,
// log w) in one word; the other features are rebuilt by the MLP kernels.
__device__ __forceinline__ unsigned bf16_pair(float lo, float hi) {
    const __nv_bfloat162 b2 = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&b2);
}
// i = crop pixel * 64 + slot: the host keeps the sets of a crop below 2^32 samples, so one 32-bit
// index (widened in the address arithmetic) addresses both arrays
__device__ __forceinline__ void store_sample(const GatherArgs &a, unsigned i, const float4 c, unsigned f) {
    a.sets.col[i] = c;
    a.sets.f89[i] = f;
}
__device__ __forceinline__ void store_sample(const GatherArgs &a, unsigned i, float3 c, float dist_r, float dj_t,
                                             float dz_r, float logw) {
    store_sample(a, i, make_float4(c.x, c.y, c.z, __uint_as_float(bf16_pair(dist_r, dj_t))), bf16_pair(dz_r, logw));
}
// Two consecutive samples, i even: 32 + 8 bytes in two stores.  The samples of a warp's pixels lie 1 KB apart,
// so each store of a lane is a sector of its own whatever its size.
__device__ __forceinline__ void store_samples(const GatherArgs &a, unsigned i, const float4 c0, unsigned f0, const float4 c1,
                                              unsigned f1) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(a.sets.col + i), "f"(c0.x), "f"(c0.y), "f"(c0.z),
                 "f"(c0.w), "f"(c1.x), "f"(c1.y), "f"(c1.z), "f"(c1.w)
                 : "memory");
    *reinterpret_cast<uint2 *>(a.sets.f89 + i) = make_uint2(f0, f1);
}
// the distance feature is rounded to BF16 (8 significant bits): the approximate square root
// (a few FP32 ulp, exact at 0) is enough
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// How the test loop's survivors of a K x K window are kept: one bit per element of K rows of kC = K + 1
// columns (aligned pairs of columns cover the window and one column beside it), in window order from
// the top of the first word; kRows rows a word (7 x 8 bits need two words).
template <int K>
struct WindowBits {
    static constexpr int kC = K + 1, kRows = K == 7 ? 4 : K, kWords = K == 7 ? 2 : 1;
    static constexpr int kFill0 = 32 - kRows * kC, kFill1 = kWords == 2 ? 32 - (K - kRows) * kC : 0;
    static constexpr unsigned rows_mask(int n) {
        unsigned m = 0u;
        for (int r = 0; r < n; ++r)
            for (int c = 0; c < K; ++c) m |= 0x80000000u >> (r * kC + c);
        return m;
    }
    static constexpr unsigned kMask0 = rows_mask(kRows), kMask1 = kWords == 2 ? rows_mask(K - kRows) : 0u;
    // A bit's column and row, as exact floats and as the element offset row * pitch + col, from its index
    // im (with the exponent bits of 2^23 set, its float form).  The row comes times kRowUnit: where a row
    // has a power of two of bits, that is the index without its column bits.
    static constexpr float kRowUnit = K == 5 ? 1.0f : (float)kC;
    __device__ static __forceinline__ unsigned row5(unsigned im) { return ((im & 31u) * 43u) >> 8; }  // i / 6 for i < 32
    __device__ static __forceinline__ unsigned col(unsigned im) {
        return K == 5 ? im - 6u * row5(im) : (im & (kC - 1)) | kMagic;  // with the exponent bits too
    }
    __device__ static __forceinline__ f32x2 col_row(unsigned im) {
        const float fc = __uint_as_float(col(im));
        return f2_pack(fc - 8388608.0f, K == 5 ? small_float((int)row5(im)) : __uint_as_float(im) - fc);
    }
    __device__ static __forceinline__ unsigned offset(unsigned im, unsigned pitch) {
        if (K == 5) return row5(im) * pitch + (col(im) - kMagic);
        // index * (pitch / kC) + col * (1 - pitch / kC): the exponent bits enter once
        return im * (pitch / kC) + (col(im) * (1u - pitch / kC) - kMagic);
    }
};
template <>
struct WindowBits<0> {};
constexpr float kLateral = 4.0f;  // see lateral in gather_pixel

// x_ref of the pixel (u0 + du, v0 + dv) at depth dref in the frame of slot geometry g: Z its depth
// there and (U, V) its pixel position, as normalised double-float numbers; false when it lies behind
// (or at) the camera.  m = M (u, v, 1) = M (u0, v0, 1) + M (du, dv, 0): the base in double-float, the
// small offset exactly enough in FP32; w = dref m + e; U = w0 / w2, V = w1 / w2.  Only error-free
// transformations and one correction step of the quotient; intermediate pairs are left unnormalised
// (each low part is below 2^-22 of its high part), and x and y share packed operations.
__device__ __forceinline__ bool project_slot(const float4 *g, const float4 q4, float du, float dv, float dref, df &Z, df &U,
                                             df &V) {
    const float4 q3 = g[3];
    {
        const df m = two_sum(q3.x, __fmaf_rn(q3.z, du, __fmul_rn(q3.w, dv)));
        const df p = two_prod(m.hi, dref);
        const float pl = __fmaf_rn(__fadd_rn(m.lo, q3.y), dref, p.lo);
        const df s = two_sum(p.hi, q4.x);
        Z = fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(pl, q4.y)));
    }
    if (!(Z.hi > 1e-6f * dref)) return false;
    const float4 q0 = g[0], q1 = g[1], q2 = g[2];
    const f32x2 mh = f2_pack(q0.x, q0.y), ml = f2_pack(q0.z, q0.w), eh = f2_pack(q2.x, q2.y), el = f2_pack(q2.z, q2.w);
    const f32x2 t = f2_fma(f2_pack(q1.x, q1.y), f2_pack(du, du), f2_mul(f2_pack(q1.z, q1.w), f2_pack(dv, dv)));
    // m = mh + t (two-sum) + ml
    const f32x2 m = f2_add(mh, t), mb = f2_sub(m, mh);
    const f32x2 me = f2_add(f2_add(f2_sub(mh, f2_sub(m, mb)), f2_sub(t, mb)), ml);
    // w = m dref + e: -p is the rounded product's negative, so that the sum is a two-difference
    const f32x2 d2 = f2_pack(dref, dref), np = f2_mul(m, f2_pack(-dref, -dref));
    const f32x2 pl = f2_fma(me, d2, f2_fma(m, d2, np));
    const f32x2 w = f2_sub(eh, np), wb = f2_sub(w, eh);  // wb: what of -np went into w
    const f32x2 wl = f2_add(f2_sub(f2_sub(eh, f2_sub(w, wb)), f2_add(np, wb)), f2_add(pl, el));
    // q = w / Z: first quotient -nq, remainder, correction
    const float r = rcp_approx(Z.hi);
    const f32x2 zh2 = f2_pack(Z.hi, Z.hi), nq = f2_mul(w, f2_pack(-r, -r));
    const f32x2 rem = f2_fma(nq, f2_pack(Z.lo, Z.lo), f2_add(f2_fma(nq, zh2, w), wl));
    const f32x2 c = f2_mul(rem, f2_pack(r, r));
    const f32x2 hi = f2_sub(c, nq), lo = f2_sub(c, f2_add(hi, nq));
    f2_unpack(hi, U.hi, V.hi);
    f2_unpack(lo, U.lo, V.lo);
    return true;
}

// The test loops of a K x K window whose even-column rows start at dtest (pitch tpitch): one bit per
// element of K rows of K + 1 columns, the sign of the tested quantity shifted in, window order from
// the top of the words (not yet top-aligned, the spare column not yet masked).
// By depth: e^2 - thr, e = d - zh; nthr = -thr.
template <int K, bool STG>
__device__ __forceinline__ void test_depth(const float *dtest, long long tpitch, float zh, float nthr, unsigned (&m)[2]) {
    const f32x2 zh2 = f2_pack(zh, zh), nthr2 = f2_pack(nthr, nthr);
    m[0] = m[1] = 0u;
#pragma unroll
    for (int dy = 0; dy < K; ++dy) {
        const f32x2 *drow = reinterpret_cast<const f32x2 *>(dtest + (long long)dy * tpitch);
        unsigned &mw = m[dy / WindowBits<K>::kRows];
#pragma unroll
        for (int q = 0; q < (K + 1) / 2; ++q) {
            // staged: a generic load (shared memory, or the global plane outside the box)
            const f32x2 e = f2_sub(STG ? drow[q] : __ldg(drow + q), zh2);
            float ta, tb;
            f2_unpack(f2_fma(e, e, nthr2), ta, tb);
            mw = __funnelshift_l(__float_as_uint(ta), mw, 1);
            mw = __funnelshift_l(__float_as_uint(tb), mw, 1);
        }
    }
}

// By the whole distance: e^2 + X^2 + Y^2 - r^2 with (ax, ifx), (bx, zix), (ay, ify), (by, ziy) giving X
// and Y as in the exact test, ax and bx at the even column; lim bounds |By| of the rows that can hold a
// sample.  ROWS rows at a time, those that no lane of the warp needs left out: all seven at once take
// more registers than the kernel has (112 bytes spilled), and so do two with the three records in flight
// of the FP32 filter loop (1080p +-30: 3.97 against 4.11 ms).  Two where they fit hide more of the loads'
// latency: the mixed clips' plan 13.2 against 13.9 ms.
template <int K, int ROWS, bool STG>
__device__ __forceinline__ void test_distance(const float *dtest, long long tpitch, float zh, float r, float lim, float ax,
                                              float ifx, float bx, float zix, float ay, float ify, float by, float ziy,
                                              unsigned (&m)[2]) {
    using WB = WindowBits<K>;
    constexpr int KP = (K + 1) / 2;
    const float nthr = -(r * r);
    const f32x2 zh2 = f2_pack(zh, zh), nthr2 = f2_pack(nthr, nthr);
    f32x2 Ax[KP], Bx[KP];
#pragma unroll
    for (int q = 0; q < KP; ++q) {
        Ax[q] = f2_pack(__fmaf_rn((float)(2 * q), ifx, ax), __fmaf_rn((float)(2 * q + 1), ifx, ax));
        Bx[q] = f2_pack(__fmaf_rn((float)(2 * q), zix, bx), __fmaf_rn((float)(2 * q + 1), zix, bx));
    }
    auto rows = [&](int dy, auto n_rows, unsigned &mw) {
        constexpr int N = decltype(n_rows)::value;
        const float By0 = __fmaf_rn((float)dy, ziy, by), By1 = __fmaf_rn((float)(dy + N - 1), ziy, by);
        if (!__any_sync(__activemask(), By0 <= lim && By1 >= -lim)) {
            mw <<= N * WB::kC;
            return;
        }
        f32x2 e[N][KP];
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int q = 0; q < KP; ++q) {
                const f32x2 *p = reinterpret_cast<const f32x2 *>(dtest + (long long)(dy + i) * tpitch) + q;
                e[i][q] = f2_sub(STG ? *p : __ldg(p), zh2);
            }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float Ay = __fmaf_rn((float)(dy + i), ify, ay), By = i == 0 ? By0 : By1;
#pragma unroll
            for (int q = 0; q < KP; ++q) {
                const f32x2 X = f2_fma(e[i][q], Ax[q], Bx[q]), Y = f2_fma(e[i][q], f2_pack(Ay, Ay), f2_pack(By, By));
                float ta, tb;
                f2_unpack(f2_fma(X, X, f2_fma(Y, Y, f2_fma(e[i][q], e[i][q], nthr2))), ta, tb);
                mw = __funnelshift_l(__float_as_uint(ta), mw, 1);
                mw = __funnelshift_l(__float_as_uint(tb), mw, 1);
            }
        }
    };
    using One = std::integral_constant<int, 1>;
    using Two = std::integral_constant<int, 2>;
    m[0] = m[1] = 0u;
    if (ROWS == 1) {
#pragma unroll 1
        for (int dy = 0; dy < WB::kRows; ++dy) rows(dy, One{}, m[0]);
#pragma unroll 1
        for (int dy = WB::kRows; dy < K; ++dy) rows(dy, One{}, m[1]);
    } else {
#pragma unroll 1
        for (int dy = 0; dy + 1 < WB::kRows; dy += 2) rows(dy, Two{}, m[0]);
        if (WB::kRows & 1) rows(WB::kRows - 1, One{}, m[0]);
        if (K == 7) {
            rows(4, Two{}, m[1]);
            rows(6, One{}, m[1]);
        }
    }
}

// window centre floor(u' + 0.5) and the exact offset u' - centre in [-0.5, 0.5)
__device__ __forceinline__ void window_centre(const df U, const df V, float &cxf, float &cyf, float &ou, float &ov) {
    cxf = floorf(U.hi + 0.5f);
    cyf = floorf(V.hi + 0.5f);
    ou = __fadd_rn(__fsub_rn(U.hi, cxf), U.lo);
    ov = __fadd_rn(__fsub_rn(V.hi, cyf), V.lo);
    if (!(fabsf(ou) < 0.5f && fabsf(ov) < 0.5f)) {
        if (ou < -0.5f) { cxf -= 1.0f; ou += 1.0f; } else if (ou >= 0.5f) { cxf += 1.0f; ou -= 1.0f; }
        if (ov < -0.5f) { cyf -= 1.0f; ov += 1.0f; } else if (ov >= 0.5f) { cyf += 1.0f; ov -= 1.0f; }
    }
}

// LEARN: visit the frames in canonical order (O, O-1, O+1, ...) and store the features of the
// first kMaxSamples accepted samples (learned filter), one by one (1) or in pairs (2); the Eq. 3/4 result
// goes to a.sets.plain.
// STG: the candidate depths of the test loop come from the warp's staged boxes (K > 0, not LEARN);
// tmap describes the clip's depth planes
// a_rgb and a_xyz: -log2(e) / (2 sigma^2) of Eq. 4's colour and position terms
// The window's frames are summed in four groups, by J modulo 4 whatever the window, each from zero and in
// order, and the groups' sums are added in order (LEARN: in one group, canonical order).  S = 1: this thread
// goes through all four; S = 4: the pixel has four threads of the CTA, this one taking group `split`.  The
// result is the same to the bit.  s_sum: 4 x NT floats of shared memory for the groups' sums; NT threads a CTA.
// NS: survivors per iteration of the filter loop of a compile-time window.  Each is one more record in
// flight and up to NS - 1 idle slots at the end of a frame's list: 2 -> 3 takes a 1080p +-30 FP32 frame
// from 4.15 to 3.99 ms, but with FP16 colour, whose samples take two loads and conversions, and in the
// batched kernel the registers run out (a 720p FP16 frame 1.03 -> 1.06 ms, the mixed clips' plan 13.5 -> 14.0)
template <int K, int CFMT, int NS, int NT, bool DEBUG, int LEARN = 0, bool STG = false, int S = 1>
__device__ __forceinline__ void gather_pixel(const GatherArgs &a, const Planes &P, const int O, const int u0,
                                             const int v0, const int u, const int v, const bool active,
                                             const long long crop_idx, const float4 *sgeom, const int n_slots,
                                             const float r2, const float a_rgb, const float a_xyz, const bool weighted,
                                             float &n_acc, int &n_exam, float &acc_w, float *s_sum, const int split = 0,
                                             const CUtensorMap *tmap = nullptr) {
    static_assert(!STG || (K > 0 && K <= kStageMaxK && !LEARN), "staging: compile-time k <= 7, plain gather");
    using WB = WindowBits<K>;
    constexpr int kTestRows = K == 7 && (NS == 2 || LEARN) ? 2 : 1;  // see test_distance
    const int k = K > 0 ? K : a.k;
    const int h = (k - 1) >> 1;
    const int rec_words = 3 + (k * k + 31) / 32;
    float acc_r = 0.0f, acc_g = 0.0f, acc_b = 0.0f;
    int n_feat = 0;
    float4 held_c = make_float4(0.f, 0.f, 0.f, 0.f);  // LEARN 2: an even sample waits for the odd one after it
    unsigned held_f = 0u;
    const int Tw = (n_slots - 1) >> 1;
    const float inv_r = LEARN ? rsqrtf(r2) : 0.0f, inv_T = LEARN ? 1.0f / (float)max(Tw, 1) : 0.0f;
    const unsigned set0 = LEARN ? (unsigned)crop_idx * (unsigned)kMaxSamples : 0u;
    float3 cref = make_float3(0.f, 0.f, 0.f);
    float dref = 0.0f;
    if (active) {
        const long long pix = (long long)O * P.fstride + (long long)(v + kPad) * P.pitch + (u + kPad);
        dref = __ldg(P.depth + pix);
        cref = load_colour<CFMT>(P.colour, pix);
    }
    const bool gather = active && dref > 0.0f;  // false for NaN (invalid) depth
    const float r_up = __fsqrt_rn(r2) * 1.000001f;
    // Which test the warp's windows get.  Depth alone costs 2 packed operations per pair of columns and
    // lets through candidates inside the depth slab but off to the side; the whole distance costs 6.
    // The first is better unless the window's corners lie well outside the radius: at (corner distance)^2
    // = 4 r^2 (r = 2.5 pixels with k = 7) the two tie (640 x 360 +-15, 8 frames: 1.83 ms with the line at
    // 3, 4 or 6); 160 x 90 with k = 5 (r = 0.6 pixels) takes 0.100 with the whole distance and 0.152 ms by
    // depth, 1080p (r = 7 pixels) 5.03 and 4.16 ms.
    bool lateral = false;
    {
        const float4 qc = sgeom[kSlotVec * ((n_slots - 1) >> 1) + 4];
        const float bx = (0.5f * (float)k) * dref * qc.z, by = (0.5f * (float)k) * dref * qc.w;
        lateral = __any_sync(0xffffffffu, gather && fmaf(bx, bx, by * by) > kLateral * r2);
    }
    // staging: the warp's gathering lanes, the first of them issues the copies
    const unsigned G = STG ? __ballot_sync(0xffffffffu, gather) : 0u;
    int stg_fail = -1;  // staging: the slot whose wait gave up (-1: staging on)
    if (DEBUG && active && !gather && a.membership) {
        for (int j = 0; j < n_slots; ++j) a.membership[(crop_idx * n_slots + j) * rec_words] = -2;
    }

    if (gather) {
        const float du = (float)(u - u0), dv = (float)(v - v0);
        const int group0 = O - Tw;  // slot jj belongs to group (group0 + jj) mod 4
        int n_seen = 0;                         // STG: slots so far (slot n_seen is in buffer n_seen & 1)
        if (STG && (int)(threadIdx.x & 31) == __ffs(G) - 1)
            stage_issue<K>(tmap, sgeom, n_slots, next_slot(-4, group0, n_slots), 0, du, dv, dref, threadIdx.x & 31, a.stage == 2);
        // S = 1: a finished group's sums join those before it, in shared memory (in registers they spill)
        float *sum = LEARN ? nullptr : s_sum + (S > 1 ? split * NT + threadIdx.x % (NT / S) : threadIdx.x);
        constexpr int kStride = NT / S;
        if (!LEARN && S == 1) sum[0] = sum[kStride] = sum[2 * kStride] = sum[3 * kStride] = 0.0f;
        auto following = [&](int jj) {
            if (LEARN) return jj + 1;
            if (S > 1 || jj + 4 < n_slots) return jj + 4;
            sum[0] += acc_r;
            sum[kStride] += acc_g;
            sum[2 * kStride] += acc_b;
            sum[3 * kStride] += acc_w;
            acc_r = acc_g = acc_b = acc_w = 0.0f;
            const int nx = next_slot(jj, group0, n_slots);
            return nx < 0 ? n_slots : nx;
        };
        for (int jj = LEARN ? 0 : S > 1 ? (split - group0) & 3 : next_slot(-4, group0, n_slots); jj < n_slots;
             jj = following(jj), ++n_seen) {
            int2 org = make_int2(kNoBox, kNoBox);
            if (STG) {
                // every lane of G is done with the other buffer (the slot before): refill it with the next
                // slot, then wait for this one
                __syncwarp(G);
                const bool leader = (int)(threadIdx.x & 31) == __ffs(G) - 1;
                if (stg_fail < 0 && leader && n_seen + 1 < n_slots)
                    stage_issue<K>(tmap, sgeom, n_slots, next_slot(jj, group0, n_slots), n_seen + 1, du, dv, dref,
                                   threadIdx.x & 31, a.stage == 2);
                const bool ok = stg_fail >= 0 || stg_wait(stg_bar(n_seen & 1), (unsigned)(n_seen >> 1) & 1u);
                if (__all_sync(G, ok)) {
                    if (stg_fail < 0) org = g_stg_org[threadIdx.x >> 5][n_seen & 1];
                } else if (stg_fail < 0) {
                    stg_fail = n_seen;  // the rest of this warp's frames test from the global plane
                    if (leader) atomicOr(a.err, 2);
                }
            }
            // canonical order for the learned filter: O, O-1, O+1, O-2, O+2, ...
            const int j = LEARN ? Tw + (jj == 0 ? 0 : ((jj & 1) ? -((jj + 1) >> 1) : (jj >> 1))) : jj;
            const float4 *g = sgeom + kSlotVec * j;
            const float4 q5 = g[5];
            const int J = __float_as_int(q5.w);
            int32_t *rec = DEBUG && a.membership ? a.membership + (crop_idx * n_slots + j) * rec_words : nullptr;
            if (J < 0) {
                if (DEBUG && rec) rec[0] = -1;
                continue;
            }
            const float4 q4 = g[4];
            df Z, U, V;
            if (!project_slot(g, q4, du, dv, dref, Z, U, V)) {  // behind (or at) camera J
                if (DEBUG && rec) rec[0] = 0;
                continue;
            }
            float cxf, cyf, ou, ov;
            window_centre(U, V, cxf, cyf, ou, ov);
            if (!(cxf >= (float)-h && cxf <= (float)(P.W - 1 + h) && cyf >= (float)-h && cyf <= (float)(P.H - 1 + h))) {
                if (DEBUG && rec) { rec[0] = 2; }
                continue;  // no window pixel inside the image
            }
            const int cx = (int)cxf, cy = (int)cyf;
            if ((unsigned)(cx - h) < (unsigned)max(P.W - k + 1, 0) && (unsigned)(cy - h) < (unsigned)max(P.H - k + 1, 0)) {
                n_exam += k * k;
            } else {
                int nx = min(cx + h, P.W - 1) - max(cx - h, 0) + 1;
                int ny = min(cy + h, P.H - 1) - max(cy - h, 0) + 1;
                n_exam += nx * ny;
            }
            const float ifx = q4.z, ify = q4.w;
            const float zh = Z.hi, zl = Z.lo;
            // ray_x(q) = (q_x - cx_J) / fx and z' (q_x - u') / fx as affine functions of dx
            const float Ax0 = (cxf - (float)h - q5.x) * ifx, zix = zh * ifx, Bx0 = (-(float)h - ou) * zix;
            const float Ay0 = (cyf - (float)h - q5.y) * ify, ziy = zh * ify, By0 = (-(float)h - ov) * ziy;
            // the window's first element, and the even column at or before it (xw - par): the test
            // loop's loads are aligned pairs of columns
            const int xw = cx - h + kPad, yw = cy - h + kPad, par = xw & 1;
            const long long fbase = (long long)J * P.fstride;
            const int woff = yw * P.pitch + xw;
            const float *dwin = P.depth + fbase + woff;
            const void *cwin = CFMT == 0 ? (const void *)(reinterpret_cast<const float4 *>(P.colour) + fbase + woff)
                                         : (const void *)(reinterpret_cast<const uint2 *>(P.colour) + fbase + woff);
            const float beta = -q5.z;
            const float dj_t = LEARN ? (float)(j - Tw) * inv_T : 0.0f;  // the frame-offset feature
            if (DEBUG && rec) {
                rec[0] = 1; rec[1] = cx; rec[2] = cy;
                if (K == 0)
                    for (int wd = 3; wd < rec_words; ++wd) rec[wd] = 0;
            }
            // The depth test |d_q - z'| < r is necessary for the radius test (d^2 >= dz^2 in FP32 too: the
            // other terms are added to it).  It is evaluated as e^2 < thr, e = d_q - zh without the low
            // part of z': thr = (r + |zl|)^2 with its roundings covered.
            const float rc = fmaf(fabsf(zl), 1.000001f, r_up), nthr = -(rc * rc) * 1.000001f;
            // the whole distance with e for dz: the difference, |zl| times the slopes of X and Y, and the
            // roundings, which grow with the slopes, widen the radius; |Y| < r bounds |By| by r + |e Ay|
            const float sl = 1.0f + fabsf(Ax0) + fabsf(Ay0) + (float)k * (ifx + ify);
            const float rl = fmaf(fabsf(zl), sl, r_up) * fmaf(sl, 2e-6f, 1.0f), lim = rl * (sl - fabsf(Ax0)) * 1.0001f;
            if constexpr (K > 0) {
                // the test loop's depths: this lane's window in the staged box if it lies inside it
                const float *dtest = dwin - par;
                long long tpitch = P.pitch;
                if (STG) {
                    const int ox = xw - org.x, oy = yw - org.y;
                    if ((unsigned)ox <= (unsigned)(kBoxW - K) && (unsigned)oy <= (unsigned)(kBoxH - K)) {
                        // box columns start at a multiple of four, so ox has the parity of xw
                        dtest = reinterpret_cast<const float *>(reinterpret_cast<const char *>(sgeom) +
                                                                (stg_box(sgeom, n_slots, n_seen & 1) - smem_addr(sgeom))) +
                                oy * kBoxW + (ox - par);
                        tpitch = kBoxW;
                    }
                }
                unsigned m[2];
                if (lateral)
                    test_distance<K, kTestRows, STG>(dtest, tpitch, zh, rl, lim, fmaf(-(float)par, ifx, Ax0), ifx,
                                          fmaf(-(float)par, zix, Bx0), zix, Ay0, ify, By0, ziy, m);
                else
                    test_depth<K, STG>(dtest, tpitch, zh, nthr, m);
                // top-aligned, the spare column (the last one, or the first if the window starts at an odd
                // element) out: bit i of the words, from the top, is window element (i / (K + 1), i % (K + 1))
                m[0] = ((m[0] << WB::kFill0) << par) & WB::kMask0;
                m[1] = ((m[1] << WB::kFill1) << par) & WB::kMask1;
                unsigned acc_bits[2] = {0u, 0u};  // DEBUG: the accepted ones of m
                // LEARN keeps the sums of a frame's even and odd accepted samples apart, folded after the
                // frame, in whatever pairs the survivors come (the stored features and the plain result
                // do not depend on how the test loop selects them)
                float s_r[2] = {0.f, 0.f}, s_g[2] = {0.f, 0.f}, s_b[2] = {0.f, 0.f}, s_w[2] = {0.f, 0.f};
                bool odd = false;
                // The survivors, NS per iteration so that their loads overlap: the exact radius test, then
                // the filter.  x and y of a sample share packed operations, and so do the halves of its
                // 16-byte record, (r, g) and (b, depth), as they are loaded.
                constexpr float kRowScale = 1.0f / WB::kRowUnit;
                const f32x2 step_a = f2_pack(ifx, ify * kRowScale), step_b = f2_pack(zix, ziy * kRowScale);
                const f32x2 a0 = f2_pack(Ax0, Ay0), b0 = f2_pack(Bx0, By0);
                const f32x2 ref_rg = f2_pack(cref.x, cref.y), ref_bz = f2_pack(cref.z, zh);
                int pos = 0;
#pragma unroll 1
                while (WB::kWords == 2 ? (m[0] | m[1]) != 0u : m[0] != 0u) {
                    unsigned im[NS];
                    bool ok[NS];
                    f32x2 rg[NS], bz[NS];
#pragma unroll
                    for (int t = 0; t < NS; ++t) {
                        // the next bit goes to the top; a step over 32 zeros finds none (ok false)
                        const int c = __clz((int)m[0]);
                        pos += c;
                        const unsigned top = __funnelshift_lc(WB::kWords == 2 ? m[1] : 0u, m[0], c);
                        if (WB::kWords == 2) m[1] = __funnelshift_lc(0u, m[1], c);
                        m[0] = top & 0x7fffffffu;
                        ok[t] = (int)top < 0;
                        im[t] = ((unsigned)pos & (WB::kWords * 32 - 1)) | kMagic;  // any value stays inside the padded plane
                        load_record<CFMT>(dwin, cwin, (int)WB::offset(im[t], P.pitch), rg[t], bz[t]);
                    }
#pragma unroll
                    for (int t = 0; t < NS; ++t) {
                        const f32x2 xy = WB::col_row(im[t]);
                        const f32x2 erg = f2_sub(rg[t], ref_rg), ebz = f2_sub(bz[t], ref_bz);
                        float er, eg, eb, dz, X, Y;
                        f2_unpack(erg, er, eg);
                        f2_unpack(ebz, eb, dz);
                        dz = dz - zl;
                        const f32x2 XY = f2_fma(f2_pack(dz, dz), f2_fma(xy, step_a, a0), f2_fma(xy, step_b, b0));
                        f2_unpack(XY, X, Y);
                        const float d2 = fmaf(X, X, fmaf(Y, Y, dz * dz));
                        // log2 of the weight (a_rgb and a_xyz are negative, beta is minus the frame term)
                        const float e = fmaf(a_rgb, fmaf(er, er, fmaf(eg, eg, eb * eb)), fmaf(a_xyz, d2, beta));
                        const float w = weighted ? ex2(e) : 1.0f;
                        if (ok[t] && d2 < r2) {
                            n_acc += 1.0f;
                            if (DEBUG) {
                                const unsigned bit = 0x80000000u >> (im[t] & 31);
                                if (WB::kWords == 2 && (im[t] & 32u)) acc_bits[1] |= bit;
                                else acc_bits[0] |= bit;
                            }
                            if (!LEARN) {
                                acc_r = fmaf(w, er, acc_r);
                                acc_g = fmaf(w, eg, acc_g);
                                acc_b = fmaf(w, eb, acc_b);
                                acc_w += w;
                            } else {
                                if (n_feat < kMaxSamples) {
                                    float cr, cg, cb, cd;
                                    f2_unpack(rg[t], cr, cg);
                                    f2_unpack(bz[t], cb, cd);
                                    const float4 sc = make_float4(cr, cg, cb, __uint_as_float(bf16_pair(sqrt_approx(d2) * inv_r, dj_t)));
                                    const unsigned sf = bf16_pair(dz * inv_r, e * kLn2);
                                    if (LEARN == 1) {
                                        store_sample(a, set0 + n_feat, sc, sf);
                                    } else if (n_feat & 1) {
                                        store_samples(a, set0 + n_feat - 1, held_c, held_f, sc, sf);
                                    } else {
                                        held_c = sc;
                                        held_f = sf;
                                    }
                                    ++n_feat;
                                }
                                s_r[0] = odd ? s_r[0] : fmaf(w, er, s_r[0]);
                                s_r[1] = odd ? fmaf(w, er, s_r[1]) : s_r[1];
                                s_g[0] = odd ? s_g[0] : fmaf(w, eg, s_g[0]);
                                s_g[1] = odd ? fmaf(w, eg, s_g[1]) : s_g[1];
                                s_b[0] = odd ? s_b[0] : fmaf(w, eb, s_b[0]);
                                s_b[1] = odd ? fmaf(w, eb, s_b[1]) : s_b[1];
                                s_w[0] += odd ? 0.0f : w;
                                s_w[1] += odd ? w : 0.0f;
                                odd = !odd;
                            }
                        }
                    }
                }
                if (LEARN) {
                    acc_r += s_r[0] + s_r[1];
                    acc_g += s_g[0] + s_g[1];
                    acc_b += s_b[0] + s_b[1];
                    acc_w += s_w[0] + s_w[1];
                }
                if (DEBUG && rec) {
                    // record layout: bit dy * k + dx from the bottom
                    unsigned words[2] = {0u, 0u};
#pragma unroll
                    for (int dy = 0; dy < K; ++dy) {
                        const int first = dy % WB::kRows * WB::kC, at = dy * K;
                        const unsigned row = __brev(acc_bits[dy / WB::kRows] << first) & ((1u << K) - 1u);
                        words[at / 32] |= row << at % 32;
                        if (at % 32 + K > 32) words[1] |= row >> (32 - at % 32);
                    }
                    rec[3] = (int32_t)words[0];
                    if (K * K > 32) rec[4] = (int32_t)words[1];
                }
            } else {
                for (int dy = 0; dy < k; ++dy) {
                    const float Ay = __fmaf_rn((float)dy, ify, Ay0), By = __fmaf_rn((float)dy, ziy, By0);
                    // k + 1 columns (at most 32) from the even one, one bit each, top-aligned
                    const f32x2 *drow = reinterpret_cast<const f32x2 *>(dwin - par + (long long)dy * P.pitch);
                    const f32x2 zh2 = f2_pack(zh, zh);
                    unsigned int mask = 0u;
                    if (lateral) {
                        if (!__any_sync(__activemask(), fabsf(By) <= lim)) continue;
                        const f32x2 nthr2 = f2_pack(-(rl * rl), -(rl * rl)), Ay2 = f2_pack(Ay, Ay), By2 = f2_pack(By, By);
                        const float axe = fmaf(-(float)par, ifx, Ax0), bxe = fmaf(-(float)par, zix, Bx0);
                        for (int q = 0; q < (k + 1) >> 1; ++q) {
                            const f32x2 e = f2_sub(__ldg(drow + q), zh2), c = f2_pack((float)(2 * q), (float)(2 * q + 1));
                            const f32x2 X = f2_fma(e, f2_fma(c, f2_pack(ifx, ifx), f2_pack(axe, axe)),
                                                   f2_fma(c, f2_pack(zix, zix), f2_pack(bxe, bxe)));
                            const f32x2 Y = f2_fma(e, Ay2, By2);
                            float ta, tb;
                            f2_unpack(f2_fma(X, X, f2_fma(Y, Y, f2_fma(e, e, nthr2))), ta, tb);
                            mask = __funnelshift_l(__float_as_uint(ta), mask, 1);
                            mask = __funnelshift_l(__float_as_uint(tb), mask, 1);
                        }
                    } else {
                        const f32x2 nthr2 = f2_pack(nthr, nthr);
                        for (int q = 0; q < (k + 1) >> 1; ++q) {
                            const f32x2 e = f2_sub(__ldg(drow + q), zh2);
                            float ta, tb;
                            f2_unpack(f2_fma(e, e, nthr2), ta, tb);
                            mask = __funnelshift_l(__float_as_uint(ta), mask, 1);
                            mask = __funnelshift_l(__float_as_uint(tb), mask, 1);
                        }
                    }
                    mask = ((mask << (31 - k)) << par) & (0xffffffffu << (32 - k));
                    while (mask) {
                        const int dx = __clz((int)mask);
                        mask &= 0x7fffffffu >> dx;
                        float dq;
                        float3 c;
                        load_sample<CFMT>(dwin, cwin, dy * P.pitch + dx, dq, c);
                        const float dz = (dq - zh) - zl;
                        const float X = fmaf(dz, __fmaf_rn((float)dx, ifx, Ax0), __fmaf_rn((float)dx, zix, Bx0));
                        const float Y = fmaf(dz, Ay, By);
                        const float d2 = fmaf(X, X, fmaf(Y, Y, dz * dz));
                        if (!(d2 < r2)) continue;
                        if (DEBUG && rec) {
                            const int bit = dy * k + dx;
                            rec[3 + (bit >> 5)] |= (int32_t)(1u << (bit & 31));
                        }
                        const float er = c.x - cref.x, eg = c.y - cref.y, eb = c.z - cref.z;
                        const float e = fmaf(a_rgb, fmaf(er, er, fmaf(eg, eg, eb * eb)), fmaf(a_xyz, d2, beta));
                        float w = 1.0f;
                        if (weighted) w = ex2(e);
                        if (LEARN && n_feat < kMaxSamples) {
                            store_sample(a, set0 + n_feat, c, sqrt_approx(d2) * inv_r, dj_t, dz * inv_r, e * kLn2);
                            ++n_feat;
                        }
                        acc_r = fmaf(w, er, acc_r);
                        acc_g = fmaf(w, eg, acc_g);
                        acc_b = fmaf(w, eb, acc_b);
                        acc_w += w;
                        n_acc += 1.0f;
                    }
                }
            }
        }
        if (!LEARN && S > 1) {
            sum[0] = acc_r;
            sum[kStride] = acc_g;
            sum[2 * kStride] = acc_b;
            sum[3 * kStride] = acc_w;
        }
        if (STG && stg_fail >= 0 && (int)(threadIdx.x & 31) == __ffs(G) - 1) {
            // after a time-out: wait once more (bounded) for the copies that may still be in flight,
            // slot stg_fail and the slot issued before its wait
            stg_wait(stg_bar(stg_fail & 1), (unsigned)(stg_fail >> 1) & 1u);
            if (stg_fail + 1 < n_slots) stg_wait(stg_bar((stg_fail + 1) & 1), (unsigned)((stg_fail + 1) >> 1) & 1u);
        }
    }

    if (!LEARN && S == 1 && gather) {
        acc_r = s_sum[threadIdx.x];
        acc_g = s_sum[NT + threadIdx.x];
        acc_b = s_sum[2 * NT + threadIdx.x];
        acc_w = s_sum[3 * NT + threadIdx.x];
    }
    if constexpr (S > 1) {
        __syncthreads();
        if (split != 0) {
            acc_w = 0.0f;  // counted with the first thread's in the launch statistics
            return;
        }
        if (gather) {
            constexpr int kStride = NT / S;
            const float *sum = s_sum + threadIdx.x % kStride;
            acc_r = sum[0];
            acc_g = sum[kStride];
            acc_b = sum[2 * kStride];
            acc_w = sum[3 * kStride];
#pragma unroll
            for (int s = 1; s < S; ++s) {
                acc_r = sum[s * NT] + acc_r;
                acc_g = sum[s * NT + kStride] + acc_g;
                acc_b = sum[s * NT + 2 * kStride] + acc_b;
                acc_w = sum[s * NT + 3 * kStride] + acc_w;
            }
        }
    }
    if (active) {
        // Eq. 3 written around the reference colour: c_ref + sum w (c - c_ref) / sum w
        float o_r = cref.x, o_g = cref.y, o_b = cref.z;
        if (acc_w > 0.0f) {
            const float inv = 1.0f / acc_w;
            o_r = fmaf(acc_r, inv, o_r);
            o_g = fmaf(acc_g, inv, o_g);
            o_b = fmaf(acc_b, inv, o_b);
        }
        float *o = LEARN ? a.sets.plain + crop_idx * 3 : P.out + (((long long)O * P.H + v) * P.W + u) * 3;
        o[0] = o_r;
        o[1] = o_g;
        o[2] = o_b;
        if (LEARN) {
            if (K > 0 && LEARN == 2 && (n_feat & 1)) {
                a.sets.col[set0 + n_feat - 1] = held_c;
                a.sets.f89[set0 + n_feat - 1] = held_f;
            }
            // per pixel: the count kept, c_ref and the size of the whole set / 64 (what the plain
            // fallback averages)
            a.sets.n[crop_idx] = n_feat;
            a.sets.info[crop_idx] = make_float4(cref.x, cref.y, cref.z, n_acc * (1.0f / 64.0f));
        }
        if (DEBUG && a.pixel_stats) {
            int32_t *ps = a.pixel_stats + crop_idx * 3;
            ps[0] = (int)n_acc;
            ps[1] = n_exam;
            ps[2] = __float_as_int(acc_w);
        }
    }

}

// One CTA per 32 x kTileY output tile of one output frame (grid: tiles x output frames).
// STG: the staged gather; dynamic shared memory then holds, after the slot geometry (aligned up to
// 128 bytes), two boxes per warp, and tmap describes the clip's depth planes.
template <int K, int CFMT, bool DEBUG, int LEARN = 0, int MINB = SSVP_MIN_CTAS, bool STG = false, int S = 1>
__global__ void __launch_bounds__(kThreads, MINB) gather_kernel(const GatherArgs a, const __grid_constant__ CUtensorMap tmap) {
    extern __shared__ float4 sgeom[];
    __shared__ float s_const[4];
    __shared__ unsigned long long s_cnt[2][kThreads / 32];
    __shared__ float s_w[kThreads / 32];
    if (STG && (threadIdx.x & 31) == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(stg_bar(0)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(stg_bar(1)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }

    const int oi = blockIdx.z;
    const int O = a.frame_begin + oi;
    constexpr int kRows = kTileY / S;
    // the geometry is that of the kTileY-row tile the rows lie in, whatever S (its rounding decides ties)
    const int u0 = a.x0 + blockIdx.x * kTileX, vt = blockIdx.y * kRows, v0 = a.y0 + vt / kTileY * kTileY;
    for (int j = threadIdx.x; j < a.n_slots; j += kThreads) {
        float4 *g = sgeom + kSlotVec * j;
        build_slot(a.geom[(long long)oi * a.n_slots + j], (float)u0, (float)v0, g);
        // per-frame weights (Eq. 5, Eq. 10) join the frame term of the exponent
        const int J = __float_as_int(g[5].w);
        if (J >= 0 && a.frame_log2w) g[5].z -= a.frame_log2w[J];
        if (J >= 0 && a.slot_log2w) g[5].z -= a.slot_log2w[j];
    }
    if (threadIdx.x == 0) {
        float r = a.radius > 0.0f ? a.radius : -a.radius * *a.clip.median;
        float sx = a.sigma_xyz > 0.0f ? a.sigma_xyz : r;
        // the shutter weight of Eq. 10 replaces Eq. 4: no colour and no position term
        const bool shutter = a.mode == SSVP_MODE_SHUTTER;
        s_const[0] = r * r;
        s_const[1] = shutter ? 0.0f : -kLog2e / (2.0f * a.sigma_rgb * a.sigma_rgb);
        s_const[2] = shutter ? 0.0f : -kLog2e / (2.0f * sx * sx);
        s_const[3] = a.mode == SSVP_MODE_MEAN ? 0.0f : 1.0f;
    }
    __syncthreads();

    const int tx = threadIdx.x % kTileX, ty = threadIdx.x / kTileX % kRows, split = threadIdx.x / (kTileX * kRows);
    const int u = u0 + tx, v = a.y0 + vt + ty;
    const bool active = u < a.x0 + a.cw && v < a.y0 + a.ch;
    const long long crop_idx = (long long)(v - a.y0) * a.cw + (u - a.x0);
    int n_exam = 0;
    float n_acc = 0.0f, acc_w = 0.0f;
    __shared__ float s_sum[LEARN ? 1 : 4 * kThreads];
    gather_pixel<K, CFMT, CFMT == 0 || LEARN ? 3 : 2, kThreads, DEBUG, LEARN, STG, S>(
        a, a.clip, O, u0, v0, u, v, active, crop_idx, sgeom, a.n_slots, s_const[0], s_const[1], s_const[2], s_const[3] != 0.0f,
        n_acc, n_exam, acc_w, s_sum, split, &tmap);

    // launch statistics: warp, then block, then one atomic per CTA
    unsigned long long ce = (unsigned long long)n_exam, ca = (unsigned long long)n_acc;
    float sw = acc_w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ce += __shfl_xor_sync(0xffffffffu, ce, o);
        ca += __shfl_xor_sync(0xffffffffu, ca, o);
        sw += __shfl_xor_sync(0xffffffffu, sw, o);
    }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { s_cnt[0][warp] = ce; s_cnt[1][warp] = ca; s_w[warp] = sw; }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long te = 0, ta = 0;
        double tw = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) { te += s_cnt[0][i]; ta += s_cnt[1][i]; tw += s_w[i]; }
        atomicAdd(a.stat_counts, te);
        atomicAdd(a.stat_counts + 1, ta);
        atomicAdd(a.stat_sumw, tw);
    }
}


// Persistent batched gather (A10): CTAs of 32 x TY threads pull work items (clip, output-frame
// chunk, tile) from a device counter until the list is exhausted, so clips of uneven size share
// one launch without tail effects per clip.  The clip table is read from the kernel's parameter
// space (constant bank), so the per-clip plane pointers and strides need no registers.
template <int K, int CFMT, int TY>
__global__ void __launch_bounds__(32 * TY, 32 / TY) batch_kernel(const GatherArgs a, const BatchArgs b) {
    constexpr int NT = 32 * TY;
    extern __shared__ float4 sgeom[];
    __shared__ float s_const[4];
    // the work unit (one output frame of one item), kept in shared memory by thread 0 so that no
    // loop state stays live in registers across the gather
    __shared__ int s_c, s_u0, s_v0, s_oi, s_olast, s_done;
    __shared__ unsigned long long s_cnt[2][NT / 32];
    __shared__ double s_w[NT / 32];
    __shared__ float s_sum[4 * NT];
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { s_cnt[0][warp] = 0ull; s_cnt[1][warp] = 0ull; s_w[warp] = 0.0; }
    if (threadIdx.x == 0) { s_oi = 0; s_olast = 0; s_done = 0; }
    __syncthreads();
    for (;;) {
        if (threadIdx.x == 0) {
            // the next output frame of the current item, else the next item
            int c = -1;
            if (s_oi + 1 < s_olast) {
                ++s_oi;
                c = s_c;
            } else {
                const long long item = (long long)atomicAdd(b.counter, 1ull);
                if (item >= b.n_items) {
                    s_done = 1;
                } else {
                    c = 0;
                    while (c + 1 < b.n_clips && b.clip[c + 1].item_begin <= item) ++c;
                    s_c = c;
                    const BatchClip &bc = b.clip[c];
                    const long long local = item - bc.item_begin;
                    const int ntile = bc.tiles_x * bc.tiles_y;
                    const int tile = (int)(local % ntile), chunk = (int)(local / ntile);
                    s_u0 = (tile % bc.tiles_x) * 32;
                    s_v0 = (tile / bc.tiles_x) * TY;
                    s_oi = chunk * b.frame_chunk;
                    s_olast = min(s_oi + b.frame_chunk, bc.n_out);
                }
            }
            if (c >= 0) {
                const float r = a.radius > 0.0f ? a.radius : -a.radius * *b.clip[c].p.median;
                const float sx = a.sigma_xyz > 0.0f ? a.sigma_xyz : r;
                s_const[0] = r * r;
                s_const[1] = -kLog2e / (2.0f * a.sigma_rgb * a.sigma_rgb);
                s_const[2] = -kLog2e / (2.0f * sx * sx);
                s_const[3] = a.mode == 3 ? 0.0f : 1.0f;
            }
        }
        __syncthreads();
        if (s_done) break;
        const int c = s_c, oi = s_oi, u0 = s_u0, v0 = s_v0;
        const BatchClip &bc = b.clip[c];
        const PairGeom *geom = bc.geom + (long long)oi * a.n_slots;
        for (int j = threadIdx.x; j < a.n_slots; j += NT)
            build_slot(geom[j], (float)u0, (float)v0, sgeom + kSlotVec * j);
        __syncthreads();
        const int u = u0 + (threadIdx.x & 31), v = v0 + (threadIdx.x >> 5);
        const bool active = u < bc.p.W && v < bc.p.H;
        int n_exam = 0;
        float n_acc = 0.0f, acc_w = 0.0f;
        gather_pixel<K, CFMT, 2, NT, false>(a, bc.p, bc.frame_begin + oi, u0, v0, u, v, active, 0, sgeom, a.n_slots,
                                            s_const[0], s_const[1], s_const[2], s_const[3] != 0.0f, n_acc, n_exam, acc_w,
                                            s_sum);
        // launch statistics go to per-warp shared slots after every tile
        unsigned ce = (unsigned)n_exam, ca = (unsigned)n_acc;
        float sw = acc_w;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ce += __shfl_xor_sync(0xffffffffu, ce, o);
            ca += __shfl_xor_sync(0xffffffffu, ca, o);
            sw += __shfl_xor_sync(0xffffffffu, sw, o);
        }
        if ((threadIdx.x & 31) == 0) { s_cnt[0][warp] += ce; s_cnt[1][warp] += ca; s_w[warp] += sw; }
        __syncthreads();  // the shared geometry and the work unit are rebuilt next
    }
    if (threadIdx.x == 0) {
        unsigned long long te = 0, ta = 0;
        double tw = 0.0;
        for (int i = 0; i < NT / 32; ++i) { te += s_cnt[0][i]; ta += s_cnt[1][i]; tw += s_w[i]; }
        atomicAdd(a.stat_counts, te);
        atomicAdd(a.stat_counts + 1, ta);
        atomicAdd(a.stat_sumw, tw);
    }
}

// Capped sample sets of a list of pixels of one frame (training batches): one warp a pixel, so that no
// pixel outside the list is gathered.  The lanes first project the pixel into 32 window frames at once,
// then take each frame's window together, lane = candidate (rows 0-3, then 4-6 of an 8-column grid); the
// accepted ones, in canonical order, queue up and are filtered 32 at a time.  The geometry is that of the tiles
// of gather_kernel, so the sets are the same; the plain result's sums are per lane and differ in rounding.
// Bound by instruction issue (0.71 of the slots, ncu): 4,200 warp instructions a pixel at +-15 (5,000 and 131
// instead of 105 us for 16,384 pixels with each window's few samples filtered at once).  Extracting the whole
// 640 x 360 frame takes 385 us; the gradient of the batch went from 0.60 to 0.25 ms, with the training
// kernel's operand layout.
constexpr int kListThreads = 256, kListCtas = 4, kListGeomStride = 33;  // words a slot: an odd stride, no bank conflicts
constexpr int kListQueue = 128;  // samples a warp can hold: 31 waiting and one window's 49, rounded up

template <int CFMT>
__global__ void __launch_bounds__(kListThreads, kListCtas) extract_list_kernel(const GatherArgs a, const int32_t *list, int n_list) {
    extern __shared__ float4 s_dyn[];
    float4 *s_ctx = s_dyn + (threadIdx.x >> 5) * 32 * 4;                  // this warp's 32 frames x 4
    float4 *s_queue = s_dyn + kListThreads * 4 + (threadIdx.x >> 5) * kListQueue;  // this warp's samples
    float *s_geom = reinterpret_cast<float *>(s_dyn + kListThreads * 4 + kListThreads / 32 * kListQueue);  // n_slots x kListGeomStride
    const int lane = threadIdx.x & 31;
    const float *gsrc = reinterpret_cast<const float *>(a.geom);
    for (int i = threadIdx.x; i < a.n_slots * 32; i += kListThreads)
        s_geom[(i >> 5) * kListGeomStride + (i & 31)] = __ldg(gsrc + i);
    __syncthreads();
    const Planes &P = a.clip;
    const int k = a.k, h = (k - 1) >> 1, O = a.frame_begin, Tw = a.T;
    const float r = a.radius > 0.0f ? a.radius : -a.radius * *P.median;
    const float sx = a.sigma_xyz > 0.0f ? a.sigma_xyz : r;
    const float r2 = r * r, a_rgb = -kLog2e / (2.0f * a.sigma_rgb * a.sigma_rgb), a_xyz = -kLog2e / (2.0f * sx * sx);
    const float inv_r = rsqrtf(r2), inv_T = 1.0f / (float)max(Tw, 1);
    const int col = lane & 7, row0 = lane >> 3;
    const float dxf = (float)col;
    const unsigned below = (1u << lane) - 1u;

    for (int i = blockIdx.x * (kListThreads / 32) + (threadIdx.x >> 5); i < n_list; i += gridDim.x * (kListThreads / 32)) {
        const int px = __ldg(list + i), v = px / P.W, u = px - v * P.W;
        const long long pix = (long long)O * P.fstride + (long long)(v + kPad) * P.pitch + (u + kPad);
        const float dref = __ldg(P.depth + pix);
        const float3 cref = load_colour<CFMT>(P.colour, pix);
        float acc_r = 0.0f, acc_g = 0.0f, acc_b = 0.0f, acc_w = 0.0f;
        int n_acc = 0, n_done = 0;  // samples found, filtered
        // sample idx of the queue: its weight joins this lane's sums, the first 64 are stored
        auto filter = [&](int idx) {
            const float4 e = s_queue[idx & (kListQueue - 1)];
            const int id = __float_as_int(e.x), t = id & 255;
            const float4 c0 = s_ctx[t * 4], c3 = s_ctx[t * 4 + 3];
            const long long at = (long long)__float_as_int(c0.x) * P.fstride + (__float_as_int(c0.y) + (id >> 8 & 255) * P.pitch + (id >> 16));
            float dq;
            float3 c;
            load_sample<CFMT>(P.depth, P.colour, at, dq, c);
            const float er = c.x - cref.x, eg = c.y - cref.y, eb = c.z - cref.z;
            const float x = fmaf(a_rgb, fmaf(er, er, fmaf(eg, eg, eb * eb)), fmaf(a_xyz, e.y, c3.z));
            const float w = ex2(x);
            if (idx < kMaxSamples)
                store_sample(a, (unsigned)i * (unsigned)kMaxSamples + idx, c, sqrt_approx(e.y) * inv_r, c3.w, e.z * inv_r, x * kLn2);
            acc_r = fmaf(w, er, acc_r);
            acc_g = fmaf(w, eg, acc_g);
            acc_b = fmaf(w, eb, acc_b);
            acc_w += w;
        };
        if (dref > 0.0f) {
            for (int base = 0; base < a.n_slots; base += 32) {
                const int jj = base + lane;
                int J = -1, woff = 0;
                if (jj < a.n_slots) {
                    const int j = Tw + (jj == 0 ? 0 : ((jj & 1) ? -((jj + 1) >> 1) : (jj >> 1)));
                    PairGeom pg;
                    float *w = reinterpret_cast<float *>(&pg);
#pragma unroll
                    for (int q = 0; q < 32; ++q) w[q] = s_geom[j * kListGeomStride + q];
                    if (pg.J >= 0) {
                        const int u0 = u / kTileX * kTileX, v0 = v / kTileY * kTileY;
                        float4 g[kSlotVec];
                        build_slot(pg, (float)u0, (float)v0, g);
                        df Z, U, V;
                        if (project_slot(g, g[4], (float)(u - u0), (float)(v - v0), dref, Z, U, V)) {
                            float cxf, cyf, ou, ov;
                            window_centre(U, V, cxf, cyf, ou, ov);
                            if (cxf >= (float)-h && cxf <= (float)(P.W - 1 + h) && cyf >= (float)-h && cyf <= (float)(P.H - 1 + h)) {
                                J = pg.J;
                                const float ifx = pg.ifx, ify = pg.ify, zix = Z.hi * ifx, ziy = Z.hi * ify;
                                woff = ((int)cyf - h + kPad) * P.pitch + ((int)cxf - h + kPad);
                                s_ctx[lane * 4 + 1] = make_float4(Z.hi, Z.lo, (cxf - (float)h - pg.cx) * ifx, (cyf - (float)h - pg.cy) * ify);
                                s_ctx[lane * 4 + 2] = make_float4((-(float)h - ou) * zix, (-(float)h - ov) * ziy, ifx, ify);
                                s_ctx[lane * 4 + 3] = make_float4(zix, ziy, -(pg.beta * kLog2e), (float)(j - Tw) * inv_T);
                            }
                        }
                    }
                }
                s_ctx[lane * 4] = make_float4(__int_as_float(J), __int_as_float(woff), 0.f, 0.f);
                __syncwarp();
                // the frames whose window meets the image, in order; the next one's depths are loaded before
                // this one's are tested
                unsigned live = __ballot_sync(0xffffffffu, J >= 0);
                float dn[2];
                const float *dwin = nullptr;
                auto fetch = [&](int t) {
                    const float4 c0 = s_ctx[t * 4];
                    dwin = P.depth + (long long)__float_as_int(c0.x) * P.fstride + __float_as_int(c0.y);
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const int row = 4 * half + row0;
                        dn[half] = col < k && row < k ? __ldg(dwin + row * P.pitch + col) : __int_as_float(0x7fffffff);
                    }
                };
                if (live) fetch(__ffs((int)live) - 1);
                while (live) {
                    const int t = __ffs((int)live) - 1;
                    live &= live - 1u;
                    const float4 c1 = s_ctx[t * 4 + 1], c2 = s_ctx[t * 4 + 2], c3 = s_ctx[t * 4 + 3];
                    const float d[2] = {dn[0], dn[1]};
                    if (live) fetch(__ffs((int)live) - 1);
                    float d2[2], dz[2];
                    unsigned hits[2];
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const float dyf = (float)(4 * half + row0);
                        dz[half] = (d[half] - c1.x) - c1.y;
                        const float X = fmaf(dz[half], __fmaf_rn(dxf, c2.z, c1.z), __fmaf_rn(dxf, c3.x, c2.x));
                        const float Y = fmaf(dz[half], __fmaf_rn(dyf, c2.w, c1.w), __fmaf_rn(dyf, c3.y, c2.y));
                        d2[half] = fmaf(X, X, fmaf(Y, Y, dz[half] * dz[half]));
                        hits[half] = __ballot_sync(0xffffffffu, d2[half] < r2);
                    }
                    // the samples queue up in canonical order; every 32 are filtered together
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const int at = n_acc + (half ? __popc(hits[0]) : 0) + __popc(hits[half] & below);
                        if (hits[half] >> lane & 1u)
                            s_queue[at & (kListQueue - 1)] = make_float4(
                                __int_as_float(t | (4 * half + row0) << 8 | col << 16), d2[half], dz[half], 0.0f);
                    }
                    n_acc += __popc(hits[0]) + __popc(hits[1]);
                    for (; n_acc - n_done >= 32; n_done += 32) {
                        __syncwarp();
                        filter(n_done + lane);
                        __syncwarp();
                    }
                }
                __syncwarp();
                if (n_done + lane < n_acc) filter(n_done + lane);
                n_done = n_acc;
                __syncwarp();  // the next 32 frames overwrite s_ctx
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            acc_r += __shfl_xor_sync(0xffffffffu, acc_r, o);
            acc_g += __shfl_xor_sync(0xffffffffu, acc_g, o);
            acc_b += __shfl_xor_sync(0xffffffffu, acc_b, o);
            acc_w += __shfl_xor_sync(0xffffffffu, acc_w, o);
        }
        if (lane == 0) {
            const float inv = acc_w > 0.0f ? 1.0f / acc_w : 0.0f;
            float *o = a.sets.plain + 3 * (long long)i;
            o[0] = acc_w > 0.0f ? fmaf(acc_r, inv, cref.x) : cref.x;
            o[1] = acc_w > 0.0f ? fmaf(acc_g, inv, cref.y) : cref.y;
            o[2] = acc_w > 0.0f ? fmaf(acc_b, inv, cref.z) : cref.z;
            a.sets.n[i] = min(n_acc, kMaxSamples);
            a.sets.info[i] = make_float4(cref.x, cref.y, cref.z, (float)n_acc * (1.0f / 64.0f));
        }
    }
}

template <int K, int CFMT, int TY>
void *batch_fn() { return (void *)batch_kernel<K, CFMT, TY>; }

template <int CFMT, int TY>
void *batch_fn_k(int k) {
    switch (k) {
        case 1: return batch_fn<1, CFMT, TY>();
        case 3: return batch_fn<3, CFMT, TY>();
        case 5: return batch_fn<5, CFMT, TY>();
        case 7: return batch_fn<7, CFMT, TY>();
        default: return batch_fn<0, CFMT, TY>();
    }
}

void *batch_fn_any(int k, int tile_rows, int cfmt) {
    if (tile_rows == 4) return cfmt == 0 ? batch_fn_k<0, 4>(k) : batch_fn_k<1, 4>(k);
    if (tile_rows == 8) return cfmt == 0 ? batch_fn_k<0, 8>(k) : batch_fn_k<1, 8>(k);
    return nullptr;
}

// cuTensorMapEncodeTiled, from the driver through the runtime (no link against the driver library)
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeTiledFn) nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// The clip's depth planes as a 3-D FP32 tensor {pitch, rows, F} (row and frame strides in bytes are
// multiples of 16: the pitch is a multiple of 32 floats), read in boxes of kBoxW x kBoxH x 1; reads
// outside the tensor return NaN, which fails the radius test as the padding does.
cudaError_t encode_depth_map(const Planes &P, CUtensorMap *m) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return cudaErrorSymbolNotFound;
    const cuuint64_t dims[3] = {(cuuint64_t)P.pitch, (cuuint64_t)P.rows, (cuuint64_t)P.F};
    const cuuint64_t strides[2] = {(cuuint64_t)P.pitch * sizeof(float), (cuuint64_t)P.fstride * sizeof(float)};
    const cuuint32_t box[3] = {(cuuint32_t)kBoxW, (cuuint32_t)kBoxH, 1u}, elem[3] = {1u, 1u, 1u};
    const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, P.depth, dims, strides, box, elem,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NAN_REQUEST_ZERO_FMA);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int K, int CFMT>
cudaError_t launch_k(const GatherArgs &a, cudaStream_t s) {
    dim3 grid((a.cw + kTileX - 1) / kTileX, (a.ch + kTileY - 1) / kTileY, a.n_out);
    size_t smem = sizeof(float4) * kSlotVec * (size_t)a.n_slots;
    const bool dbg = a.membership || a.pixel_stats;
    CUtensorMap tmap;
    memset(&tmap, 0, sizeof(tmap));
    if (a.stage) {
        if constexpr (K > 0 && K <= kStageMaxK) {
            if (a.sets.col) return cudaErrorInvalidValue;
            cudaError_t e = encode_depth_map(a.clip, &tmap);
            if (e != cudaSuccess) return e;
            smem += 128 + (size_t)(kThreads / 32) * 2 * kBoxBytes;
            void (*fn)(const GatherArgs, const CUtensorMap) =
                dbg ? gather_kernel<K, CFMT, true, false, SSVP_MIN_CTAS, true>
                    : gather_kernel<K, CFMT, false, false, SSVP_MIN_CTAS, true>;
            // 48 KB without it, of which the kernel's own arrays take less than 8
            if (smem > 40 * 1024 &&
                (e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
                return e;
            fn<<<grid, kThreads, smem, s>>>(a, tmap);
            return cudaGetLastError();
        } else {
            return cudaErrorInvalidValue;
        }
    }
    // Sets stored in pairs halve the stores, which hold large crops back (every store of a lane is a sector of its
    // own), for some instructions more: +-6, two frames, 1080p 7.84 -> 6.99 ms, 960 x 540 1.90 -> 1.80, 800 x 450
    // 1.30 -> 1.27, 640 x 360 0.80 -> 0.82, 480 x 270 0.51 -> 0.52
    if (a.sets.col && (long long)a.cw * a.ch >= 300000)
        gather_kernel<K, CFMT, false, 2, kLearnCtas><<<grid, kThreads, smem, s>>>(a, tmap);
    else if (a.sets.col) {
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if (extract_four_ctas((long long)grid.x * grid.y * grid.z, sms)) gather_kernel<K, CFMT, false, 1, kLearnCtas + 1><<<grid, kThreads, smem, s>>>(a, tmap);
        else gather_kernel<K, CFMT, false, 1, kLearnCtas><<<grid, kThreads, smem, s>>>(a, tmap);
    } else if (dbg) gather_kernel<K, CFMT, true><<<grid, kThreads, smem, s>>>(a, tmap);
    else {
        // Few CTAs leave SMs idle or end in a nearly empty wave: then each pixel's frames are shared out to four
        // threads (CTAs of 32 x 2 pixels)
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if (window_shares((long long)grid.x * grid.y * grid.z, (long long)SSVP_MIN_CTAS * sms, a.n_slots, a.k)) {
            grid.y = (a.ch + kTileY / 4 - 1) / (kTileY / 4);
            gather_kernel<K, CFMT, false, false, SSVP_MIN_CTAS, false, 4><<<grid, kThreads, smem, s>>>(a, tmap);
        } else gather_kernel<K, CFMT, false><<<grid, kThreads, smem, s>>>(a, tmap);
    }
    return cudaGetLastError();
}

template <int CFMT>
cudaError_t launch_c(const GatherArgs &a, cudaStream_t s) {
    switch (a.k) {
        case 1: return launch_k<1, CFMT>(a, s);
        case 3: return launch_k<3, CFMT>(a, s);
        case 5: return launch_k<5, CFMT>(a, s);
        case 7: return launch_k<7, CFMT>(a, s);
        default: return launch_k<0, CFMT>(a, s);
    }
}

}  // namespace

cudaError_t launch_gather(const GatherArgs &a, cudaStream_t s) {
    if (a.n_out <= 0 || a.cw <= 0 || a.ch <= 0) return cudaSuccess;
    return a.clip.colour_fmt == 0 ? launch_c<0>(a, s) : launch_c<1>(a, s);
}

cudaError_t launch_extract_list(const GatherArgs &a, const int32_t *list, int n_list, cudaStream_t s) {
    if (n_list <= 0) return cudaSuccess;
    if (a.k > 7 || a.x0 != 0 || a.y0 != 0 || a.cw != a.clip.W || a.ch != a.clip.H) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const size_t smem = sizeof(float4) * (4 * kListThreads + kListThreads / 32 * kListQueue) + sizeof(float) * kListGeomStride * (size_t)a.n_slots;
    void (*fn)(const GatherArgs, const int32_t *, int) = a.clip.colour_fmt == 0 ? extract_list_kernel<0> : extract_list_kernel<1>;
    if (smem > 48 * 1024 && (e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    const int warps = kListThreads / 32, grid = std::min((n_list + warps - 1) / warps, sms * kListCtas);
    fn<<<grid, kListThreads, smem, s>>>(a, list, n_list);
    return cudaGetLastError();
}

int batch_grid(int k, int tile_rows, int colour_fmt, int n_slots) {
    void *fn = batch_fn_any(k, tile_rows, colour_fmt);
    if (!fn) return 0;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    size_t smem = sizeof(float4) * kSlotVec * (size_t)n_slots;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * tile_rows, smem) != cudaSuccess) return 0;
    return sms * (per_sm > 0 ? per_sm : 1);
}

cudaError_t launch_batch(const GatherArgs &a, const BatchArgs &b, int tile_rows, int colour_fmt, int grid,
                         cudaStream_t s) {
    void *fn = batch_fn_any(a.k, tile_rows, colour_fmt);
    if (!fn || grid <= 0) return cudaErrorInvalidValue;
    size_t smem = sizeof(float4) * kSlotVec * (size_t)a.n_slots;
    void *args[] = {(void *)&a, (void *)&b};
    return cudaLaunchKernel(fn, dim3(grid), dim3(32 * tile_rows), args, smem, s);
}

}  // namespace ssvp
