// ssvp_frustum.cu - the paper's frustum gather (Sec. "Sample Gathering", Eq. 1-2) fused with the
// Eq. 3/4 filter.  One thread per output pixel, or four that share its window frames.
//
// Per (pixel p, frame J):
//   1. The frustum V of Eq. 1 (the l x l square around p swept over O depths [near, far]) is
//      clipped to frame J's valid-depth slab [zlo_J, zhi_J] (no pixel of J has a depth outside
//      it, so nothing is lost) and projected into J: the 12 edges of V are clipped in O depth
//      and their end points projected.  A parallelogram along the projected central ray bounds
//      that hull (grown by a rounding margin); only its pixels are tested.
//   2. Each pixel q in it with depth d is back-projected into O through the homogeneous map
//      h = M_{O<-J} (q_x d, q_y d, d) + e_{O<-J}; it is a sample when near < h_3 < far and
//      |h_1 - u h_3| + |h_2 - v h_3| < (l / 2) h_3, which is Eq. 2's L1 test multiplied by the
//      positive O depth h_3.
//      Short hulls are walked row by row with this test.  In long ones most candidates lie at depths whose
//      back-projection is far from p along the projected ray: first whole blocks of 8 positions along the
//      hull are dropped by the depth range of the 8 x 8 pixel tiles they touch (computed with the frames'
//      depth ranges), then single candidates by a slightly wider form of the test, four across the hull
//      per position; what is left takes the exact test.
//   3. Samples are weighted by Eq. 4 around s_ref (times the per-frame factors of Eq. 5, or by
//      Eq. 10's shutter function alone) and reduced by Eq. 3, as in the window gather.
//
// What bounds it: instruction issue (720p, +-15, ncu: 0.70 of the slots, 3.10e9 warp instructions, ALU pipe 50 %; DRAM
// 524 MB).  Of that frame's 3.2 ms the candidates' tests take about a third, taking the samples (4.4 of 104 candidates
// a pixel and frame, a third of a warp's lanes at a time) a third, the bound of the hull 0.4 ms, the block checks 0.5
// ms.  Against one walk of every row: 720p +-15 3.76 -> 3.22 ms, 1080p +-30 36.9 -> 20.5, super-resolution 640 x 360 to
// 1080p 7.70 -> 6.89 (short hulls: the geometry read from shared memory); with four threads a pixel a 320 x 180
// frame 221 -> 146 us, inpainting of a 720p frame, one small box 1.06 -> 0.28 ms, a fifth of the frame 3.28 -> 3.11.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "../../include/ssvp.h"
#include "ssvp_df.cuh"
#include "ssvp_dispatch.h"
#include "ssvp_internal.h"

namespace ssvp {
namespace {

constexpr int kFrTileX = 32, kFrTileY = 8, kFrThreads = kFrTileX * kFrTileY;

// SplitMix64 output function (Steele, Lea and Flood, OOPSLA 2014); debug records sum it over the
// linear indices qy * W + qx + 1 of a sample set, an order-independent membership checksum.
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// Bound of the projected hull: minor = b * major + [lo, hi], major in [mlo, mhi].
struct HullBound {
    float b, lo, hi, mlo, mhi;
    bool xmajor, any;
};

__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ void bound_add(HullBound &hb, float px, float py) {
    const float maj = hb.xmajor ? px : py, mnr = hb.xmajor ? py : px;
    const float ic = fmaf(-hb.b, maj, mnr);
    hb.lo = fminf(hb.lo, ic);
    hb.hi = fmaxf(hb.hi, ic);
    hb.mlo = fminf(hb.mlo, maj);
    hb.mhi = fmaxf(hb.mhi, maj);
    hb.any = true;
}

// Interval of t in [t0, t1] where w(t) = w0 + t dw lies in [zlo, zhi]; false when empty.
__device__ __forceinline__ bool slab_interval(float w0, float dw, float zlo, float zhi, float t0, float t1, float &ta,
                                              float &tb) {
    if (dw != 0.0f) {
        const float sa = (zlo - w0) / dw, sb = (zhi - w0) / dw;
        ta = fmaxf(t0, fminf(sa, sb));
        tb = fminf(t1, fmaxf(sa, sb));
    } else {
        if (!(w0 >= zlo && w0 <= zhi)) return false;
        ta = t0;
        tb = t1;
    }
    return ta <= tb;
}

// Lateral edge of V through the O pixel point (cu, cv): h(z) = z A + e for O depth z.
__device__ __forceinline__ void lateral_edge(const float *M, const float *e, float cu, float cv, float nearp,
                                             float farp, float zlo, float zhi, HullBound &hb) {
    const float A0 = fmaf(M[0], cu, fmaf(M[1], cv, M[2]));
    const float A1 = fmaf(M[3], cu, fmaf(M[4], cv, M[5]));
    const float A2 = fmaf(M[6], cu, fmaf(M[7], cv, M[8]));
    float za, zb;
    // J depth along the edge: A2 z + e2
    if (!slab_interval(e[2], A2, zlo, zhi, nearp, farp, za, zb)) return;
    // the interval above is in units of z (w0 = e2 at z = 0), clipped to [near, far]
    const float wa = fmaf(A2, za, e[2]), wb = fmaf(A2, zb, e[2]);
    if (wa > 0.0f) bound_add(hb, fmaf(A0, za, e[0]) / wa, fmaf(A1, za, e[1]) / wa);
    if (wb > 0.0f) bound_add(hb, fmaf(A0, zb, e[0]) / wb, fmaf(A1, zb, e[1]) / wb);
}

// Edge of the near or far face of V at O depth z0, from O pixel point (cu, cv) to (cu', cv').
__device__ __forceinline__ void face_edge(const float *M, const float *e, float z0, float cu, float cv, float du,
                                          float dv, float zlo, float zhi, HullBound &hb) {
    // h(s) = z0 M (cu + s du, cv + s dv, 1) + e, s in [0, 1]
    const float P0 = fmaf(z0, fmaf(M[0], cu, fmaf(M[1], cv, M[2])), e[0]);
    const float P1 = fmaf(z0, fmaf(M[3], cu, fmaf(M[4], cv, M[5])), e[1]);
    const float P2 = fmaf(z0, fmaf(M[6], cu, fmaf(M[7], cv, M[8])), e[2]);
    const float D0 = z0 * fmaf(M[0], du, M[1] * dv), D1 = z0 * fmaf(M[3], du, M[4] * dv),
                D2 = z0 * fmaf(M[6], du, M[7] * dv);
    float sa, sb;
    if (!slab_interval(P2, D2, zlo, zhi, 0.0f, 1.0f, sa, sb)) return;
    const float wa = fmaf(D2, sa, P2), wb = fmaf(D2, sb, P2);
    if (wa > 0.0f) bound_add(hb, fmaf(D0, sa, P0) / wa, fmaf(D1, sa, P1) / wa);
    if (wb > 0.0f) bound_add(hb, fmaf(D0, sb, P0) / wb, fmaf(D1, sb, P1) / wb);
}

// SR: super-resolution (Sec. "Super resolution", Eq. 6-7) on the a.sr_scale-times output grid;
// the maps use the output-grid camera of O, s_ref is bilinear in the input frame, and the
// exponent gains Eq. 7's area term.
// INP: inpainting (Sec. "Inpainting and semi-transparency", Eq. 8-9): only pixels with a mask
// gather; three passes over S(p): the mean of all samples (Eq. 8), then two steps of the
// colour-weighted mean over unmasked samples (Eq. 9), each around the previous result.
// INP == 2: semi-transparency (the same section, after Eq. 9): in the last pass every sample,
// masked or not, also weighs the Eq. 4 weight around the pixel's own sample (I(p), x_ref, O),
// so the object's samples near x_ref blend with the background's mean-shift estimate.
// Fast path of the hull: the 4 lateral rays of the frustum, h(z) = z A + e, clipped to the slab
// alone.  Valid (returns true) when every ray's depth in J grows (or every one falls) with z and
// every clipped interval lies strictly inside (near, far): then no face of V touches the slab,
// every point of V in the slab has its O depth inside (near, far), and the hull is that of the
// 8 end points, which are projected here with approximate reciprocals (the bound's margin
// covers their error).
// corner c = 0..3 of the l x l square around (u, v), counter-clockwise from (u - L, v - L)
__device__ __forceinline__ float corner_u(int c, float u, float L) { return (c == 1 || c == 2) ? u + L : u - L; }
__device__ __forceinline__ float corner_v(int c, float v, float L) { return c >= 2 ? v + L : v - L; }

// rows of the map in the order major, minor, depth (Ma, ea: major; Mi, ei: minor)
__device__ __forceinline__ bool lateral_fast(const float (&Ma)[3], const float (&Mi)[3], const float (&Mz)[3], float ea, float ei,
                                             float ez, float u, float v, float L, float nearp, float farp, float zlo,
                                             float zhi, HullBound &hb) {
    float sgn = 0.0f;
    bool ok = true;
    auto add = [&](float maj, float mnr) {
        const float ic = fmaf(-hb.b, maj, mnr);
        hb.lo = fminf(hb.lo, ic);
        hb.hi = fmaxf(hb.hi, ic);
        hb.mlo = fminf(hb.mlo, maj);
        hb.mhi = fmaxf(hb.mhi, maj);
    };
    hb.any = true;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float cu = corner_u(c, u, L), cv = corner_v(c, v, L);
        const float A0 = fmaf(Ma[0], cu, fmaf(Ma[1], cv, Ma[2]));
        const float A1 = fmaf(Mi[0], cu, fmaf(Mi[1], cv, Mi[2]));
        const float A2 = fmaf(Mz[0], cu, fmaf(Mz[1], cv, Mz[2]));
        const float s = A2 > 0.0f ? 1.0f : (A2 < 0.0f ? -1.0f : 0.0f);
        ok = ok && s != 0.0f && (c == 0 || s == sgn);
        sgn = s;
        const float r = rcp_approx(A2);
        const float sa = (zlo - ez) * r, sb = (zhi - ez) * r;
        const float za = fminf(sa, sb), zb = fmaxf(sa, sb);
        ok = ok && za > nearp * 1.0001f && zb < farp * 0.9999f;
        const float wa = fmaf(A2, za, ez), wb = fmaf(A2, zb, ez);
        const float ra = rcp_approx(wa), rb = rcp_approx(wb);
        ok = ok && wa > 0.0f && wb > 0.0f;
        add(fmaf(A0, za, ea) * ra, fmaf(A1, za, ei) * ra);
        add(fmaf(A0, zb, ea) * rb, fmaf(A1, zb, ei) * rb);
    }
    return ok;
}

// Registers: 80 (three CTAs per SM), with some spilled in the form that can drop blocks.  For inpainting that form has 128
// (two CTAs) instead: 720p, +-15, one small box, 275 against 354 us.  The other is better off with
// three CTAs, which spill nothing: 640 x 360, +-5, two fifths of the frame masked, 262 against 335 us.
template <int INP, bool LONG> constexpr int kFrCtas = INP && LONG ? 2 : 3;
constexpr int kFrSlotVec = 8;  // float4 words of a window slot in shared memory:
//  0-2 = forward map M (9), e (3); 3 = zlo zhi (J's valid depth range), log2 weight of the frame (negated), J
//  4-6 = back map M (9), e (3); 7.x = 1 / fx of J, 7.y = whether hulls are long
constexpr int kTile = 8;       // side of the depth range tiles
// LONG instances: length of a window frame's hulls, in pixels, from which their blocks are checked by their depth range
// (see the slot loop).  The check costs about as much as 25 candidates, which a short hull does not save.  One choice
// for all pixels of a frame: the two walks sum in different orders, and a warp would pay for both (chosen pixel by
// pixel 720p, +-15, takes 3.37 ms).  720p, +-15: 3.25, 3.21, 3.39, 3.44 ms with the line at 24, 32, 48 and never; 640 x
// 360, +-30: 1.81, 1.80, 1.88, 1.94; 1080p, +-30: 20.6, 20.5, 20.7, 33.6.
constexpr int kLongHull = 32;
constexpr float kRound = 12582912.0f;  // 1.5 * 2^23: x + kRound holds x rounded to an integer in its low bits

// A pixel's sums over one group of its window frames, or over all: the colours and the weight, times 2^-m
struct FrSums { float r, g, b, w, m; };

// The sums of the next group join those before it, at the larger of the two powers; the roundings are spelled out,
// so that they are the same whichever thread joins
__device__ __forceinline__ void join_sums(FrSums &a, const FrSums &b) {
    const float m = fmaxf(a.m, b.m), sa = ex2(__fsub_rn(a.m, m)), sb = ex2(__fsub_rn(b.m, m));
    a.r = __fmaf_rn(sb, b.r, __fmul_rn(sa, a.r));
    a.g = __fmaf_rn(sb, b.g, __fmul_rn(sa, a.g));
    a.b = __fmaf_rn(sb, b.b, __fmul_rn(sa, a.b));
    a.w = __fmaf_rn(sb, b.w, __fmul_rn(sa, a.w));
    a.m = m;
}

// A pixel's window frames are summed in four groups, by J modulo 4 whatever the window, each in order, and the
// groups are joined in order.  S = 1: one thread a pixel goes through all four; S = 4: each pixel has four threads
// of the CTA (which takes 32 x 2 pixels), one a group; S = 0: one or the other, by how many pixels the mask has
// gather.  The result is the same to the bit, and every choice within it is the pixel's own: it depends neither on the
// crop nor on how many frames a launch has.
template <int CFMT, bool DEBUG, bool SR, int INP, int S, bool LONG>
__global__ void __launch_bounds__(kFrThreads, (kFrCtas<INP, LONG>)) frustum_kernel(const GatherArgs a) {
    static_assert(S == 1 || S == 4 || (S == 0 && INP), "one thread a pixel, one a group, or (inpainting) as the mask has it");
    extern __shared__ float4 s_slot[];
    __shared__ float s_const[8];
    __shared__ unsigned long long s_cnt[2][kFrThreads / 32];
    __shared__ float s_w[kFrThreads / 32];
    __shared__ FrSums s_red[kFrThreads];  // one thread a pixel: the sums of the groups so far (in registers they spill)
    __shared__ int s_dbg[DEBUG && S != 1 ? kFrThreads : 1][2];
    const Planes &P = a.clip;
    const int oi = blockIdx.z;
    const int O = a.frame_begin + oi;
    const int ns = a.n_slots;
    const int u = a.x0 + blockIdx.x * kFrTileX + threadIdx.x % kFrTileX;
    int shares = S;  // threads a pixel
    bool masked = false;
    if (S == 0) {
        // The mask at 16 x 16 places of the crop tells how many pixels gather.  The grid has a CTA for every 32 x 2
        // pixels; with one thread a pixel the first quarter of them take 32 x 8.
        const int su = a.x0 + (int)((2 * (threadIdx.x & 15) + 1) * (long long)a.cw / 32);
        const int sv = a.y0 + (int)((2 * (threadIdx.x >> 4) + 1) * (long long)a.ch / 32);
        const unsigned char *mp = P.mask + (long long)O * P.fstride + (long long)kPad * P.pitch + kPad;
        const bool here = __ldg(mp + (long long)sv * P.pitch + su) != 0;
        const int v4 = a.y0 + blockIdx.y * 2 + threadIdx.x / 32 % 2;
        if (u < a.x0 + a.cw && v4 < a.y0 + a.ch) masked = __ldg(mp + (long long)v4 * P.pitch + u) != 0;
        const long long n = (long long)__syncthreads_count(here) * a.cw * a.ch / 65536 * a.n_out;  // CTAs' worth of pixels
        shares = frustum_shares(n, (long long)kFrCtas<INP, LONG> * a.sms, ns) ? 4 : 1;
        if (shares == 1 && (int)blockIdx.y >= (a.ch + kFrTileY - 1) / kFrTileY) return;
    }
    const int rows = kFrTileY / shares;
    const int Wo = SR ? P.W * a.sr_scale : P.W;
    const int Ho = SR ? P.H * a.sr_scale : P.H;

    const int lane = threadIdx.x % kFrTileX, row = threadIdx.x / kFrTileX % rows, split = threadIdx.x / (kFrTileX * rows);
    const int v = a.y0 + blockIdx.y * rows + row;
    const bool active = u < a.x0 + a.cw && v < a.y0 + a.ch;
    const long long crop_idx = (long long)(v - a.y0) * a.cw + (u - a.x0);
    const float L = 0.5f * a.frustum_l, nearp = a.near_plane, farp = a.far_plane;
    const float zmid = 0.5f * (nearp + farp), zhalf = 0.5f * (farp - nearp);

    float3 cref = make_float3(0.f, 0.f, 0.f);
    float dref = 0.0f;
    if (active && !SR) {
        const long long pix = (long long)O * P.fstride + (long long)(v + kPad) * P.pitch + (u + kPad);
        dref = __ldg(P.depth + pix);
        cref = load_colour<CFMT>(P.colour, pix);
    }
    if (active && SR) {
        // bilinear s_ref at input coordinates ((u, v) + 0.5) / scale - 0.5, clamped to the image; an
        // invalid (NaN) depth among the four propagates and invalidates the reference
        const float is = 1.0f / (float)a.sr_scale;
        const float xc = fminf(fmaxf(((float)u + 0.5f) * is - 0.5f, 0.0f), (float)(P.W - 1));
        const float yc = fminf(fmaxf(((float)v + 0.5f) * is - 0.5f, 0.0f), (float)(P.H - 1));
        const int x0 = (int)floorf(xc), y0 = (int)floorf(yc);
        const int x1 = min(x0 + 1, P.W - 1), y1 = min(y0 + 1, P.H - 1);
        const float fx = xc - (float)x0, fy = yc - (float)y0;
        const long long fb = (long long)O * P.fstride;
        const long long p00 = fb + (long long)(y0 + kPad) * P.pitch + (x0 + kPad), p10 = p00 + (x1 - x0);
        const long long p01 = fb + (long long)(y1 + kPad) * P.pitch + (x0 + kPad), p11 = p01 + (x1 - x0);
        const float3 c00 = load_colour<CFMT>(P.colour, p00), c10 = load_colour<CFMT>(P.colour, p10);
        const float3 c01 = load_colour<CFMT>(P.colour, p01), c11 = load_colour<CFMT>(P.colour, p11);
        const float d00 = __ldg(P.depth + p00), d10 = __ldg(P.depth + p10), d01 = __ldg(P.depth + p01),
                    d11 = __ldg(P.depth + p11);
        const float gx = 1.0f - fx, gy = 1.0f - fy;
        cref.x = gy * (gx * c00.x + fx * c10.x) + fy * (gx * c01.x + fx * c11.x);
        cref.y = gy * (gx * c00.y + fx * c10.y) + fy * (gx * c01.y + fx * c11.y);
        cref.z = gy * (gx * c00.z + fx * c10.z) + fy * (gx * c01.z + fx * c11.z);
        dref = gy * (gx * d00 + fx * d10) + fy * (gx * d01 + fx * d11);
    }
    // inpainting gathers for masked pixels only and does not need their depth; the others need
    // a valid reference depth (NaN fails)
    const long long pix_o = (long long)O * P.fstride + (long long)(v + kPad) * P.pitch + (u + kPad);
    if (INP && shares == 1) masked = active && __ldg(P.mask + pix_o) != 0;
    const bool gather = INP ? masked : active && dref > 0.0f;
    if (INP && active) cref = load_colour<CFMT>(P.colour, pix_o);
    if (INP && !DEBUG && !__syncthreads_or(gather)) {
        // no pixel of the CTA gathers: the output is the input
        if (active && split == 0) {
            float *o = P.out + (((long long)O * P.H + v) * P.W + u) * 3;
            o[0] = cref.x;
            o[1] = cref.y;
            o[2] = cref.z;
        }
        return;
    }
    for (int j = threadIdx.x; j < ns; j += kFrThreads) {
        const PairGeom &gf = a.geom[(long long)oi * ns + j], &gb = a.geom_back[(long long)oi * ns + j];
        float4 *d = s_slot + kFrSlotVec * j;
        const int J = gf.J;
        float zlo = 0.0f, zhi = 0.0f, beta = 0.0f;
        if (J >= 0) {
            // J's valid depth range (order-preserving bit patterns; 0 words: no valid depth)
            const unsigned int zmin_w = __ldg(P.zrange + 2 * J), zmax_w = __ldg(P.zrange + 2 * J + 1);
            zlo = zmin_w ? __uint_as_float(~zmin_w) : __int_as_float(0x7f800000);
            zhi = __uint_as_float(zmax_w);
            // frame term of Eq. 4 plus the per-frame weights of Eq. 5 / Eq. 10, in log2 units
            beta = gf.beta * kLog2e;
            if (a.frame_log2w) beta -= __ldg(a.frame_log2w + J);
            if (a.slot_log2w) beta -= __ldg(a.slot_log2w + j);
        }
        d[0] = make_float4(gf.M_hi[0], gf.M_hi[1], gf.M_hi[2], gf.M_hi[3]);
        d[1] = make_float4(gf.M_hi[4], gf.M_hi[5], gf.M_hi[6], gf.M_hi[7]);
        d[2] = make_float4(gf.M_hi[8], gf.e_hi[0], gf.e_hi[1], gf.e_hi[2]);
        d[3] = make_float4(zlo, zhi, beta, __int_as_float(J));
        d[4] = make_float4(gb.M_hi[0], gb.M_hi[1], gb.M_hi[2], gb.M_hi[3]);
        d[5] = make_float4(gb.M_hi[4], gb.M_hi[5], gb.M_hi[6], gb.M_hi[7]);
        d[6] = make_float4(gb.M_hi[8], gb.e_hi[0], gb.e_hi[1], gb.e_hi[2]);
        // LONG: whether the blocks of J's hulls are checked, by the length that the ray of the image's centre projects to
        bool lng = false;
        if (LONG && J >= 0) {
            const float sc = SR ? 0.5f * (float)a.sr_scale : 0.5f, cu = sc * (float)P.W, cv = sc * (float)P.H;
            const float A0 = fmaf(gf.M_hi[0], cu, fmaf(gf.M_hi[1], cv, gf.M_hi[2]));
            const float A1 = fmaf(gf.M_hi[3], cu, fmaf(gf.M_hi[4], cv, gf.M_hi[5]));
            const float A2 = fmaf(gf.M_hi[6], cu, fmaf(gf.M_hi[7], cv, gf.M_hi[8]));
            float za, zb;
            if (zlo <= zhi && slab_interval(gf.e_hi[2], A2, zlo, zhi, a.near_plane, a.far_plane, za, zb)) {
                const float wa = fmaf(A2, za, gf.e_hi[2]), wb = fmaf(A2, zb, gf.e_hi[2]);
                const float dx = fmaf(A0, zb, gf.e_hi[0]) / wb - fmaf(A0, za, gf.e_hi[0]) / wa;
                const float dy = fmaf(A1, zb, gf.e_hi[1]) / wb - fmaf(A1, za, gf.e_hi[1]) / wa;
                lng = fmaxf(fabsf(dx), fabsf(dy)) >= (float)kLongHull;
            }
        }
        d[7] = make_float4(gf.ifx, __int_as_float(lng), 0.f, 0.f);
    }
    if (threadIdx.x == 0) {
        const float r = a.radius > 0.0f ? a.radius : -a.radius * *P.median;
        const float sx = a.sigma_xyz > 0.0f ? a.sigma_xyz : r;
        // the shutter weight of Eq. 10 replaces Eq. 4: no colour and no position term
        const bool shutter = a.mode == SSVP_MODE_SHUTTER;
        s_const[0] = shutter ? 0.0f : kLog2e / (2.0f * a.sigma_rgb * a.sigma_rgb);
        s_const[1] = shutter || INP == 1 ? 0.0f : kLog2e / (2.0f * sx * sx);
        s_const[2] = a.mode == SSVP_MODE_MEAN ? 0.0f : 1.0f;
        // the back maps' target camera, O's (slot T is J = O)
        const PairGeom &gO = a.geom_back[(long long)oi * ns + a.T];
        if (SR) {
            // sigma_area <= 0: one input-pixel footprint at the median depth (median / fx_O); the
            // back map of slot T (J = O) carries the output-grid 1 / fx of O
            const float sa = a.sigma_area > 0.0f ? a.sigma_area : *P.median * gO.ifx * (float)a.sr_scale;
            s_const[3] = kLog2e / (2.0f * sa * sa);
        }
        s_const[4] = gO.ifx;
        s_const[5] = gO.ify;
        s_const[6] = gO.cx;
        s_const[7] = gO.cy;
    }
    if (DEBUG && S != 1) s_dbg[threadIdx.x][0] = s_dbg[threadIdx.x][1] = 0;
    __syncthreads();
    const float a_rgb = s_const[0], a_xyz = s_const[1], a_area = SR ? s_const[3] : 0.0f;
    const bool weighted = s_const[2] != 0.0f;
    // semi-transparency: the pixel's own sample (I(p), x_ref, O) needs a valid depth (NaN fails)
    const float3 c_in = cref;
    const bool own = INP == 2 && dref > 0.0f;
    // Accumulators carry the common factor 2^-m, m the largest log2 weight so far: without the
    // reference sample (outside near / far) every weight can be far below FP32's range while
    // Eq. 3 is still well defined.  The start, -1e30, is below every finite exponent, and a
    // weight of exactly 0 (an exponent of -inf) stays 0.
    constexpr float kNoWeight = -1e30f;
    float acc_r = 0.0f, acc_g = 0.0f, acc_b = 0.0f, acc_w = 0.0f, m_log2 = 0.0f, sw_true = 0.0f;
    long long n_exam = 0;
    int n_acc = 0;
    if (DEBUG && active && !gather && a.membership)
        for (int j = split; j < ns; j += shares) {
            int32_t *rec = a.membership + (crop_idx * ns + j) * 4;
            rec[0] = -2; rec[1] = 0; rec[2] = 0; rec[3] = 0;
        }

    constexpr int kPasses = INP ? 3 : 1;
    for (int pass = 0; pass < kPasses; ++pass) {
    const bool wpass = INP ? pass > 0 : weighted;
    acc_r = acc_g = acc_b = acc_w = 0.0f;
    m_log2 = wpass ? kNoWeight : 0.0f;
    if (gather) {
      bool first = true;
      for (int grp = split; grp < 4; grp += shares) {
        const int j0 = (grp - (O - a.T)) & 3;
        if (j0 >= ns) continue;  // joining an empty group's zeros changes nothing
        for (int j = j0; j < ns; j += 4) {
            const float4 *sl = s_slot + kFrSlotVec * j;
            const float4 q3 = sl[3];
            const int J = __float_as_int(q3.w);
            int32_t *rec = DEBUG && a.membership && pass == 0 ? a.membership + (crop_idx * ns + j) * 4 : nullptr;
            if (J < 0) {
                if (DEBUG && rec) { rec[0] = -1; rec[1] = 0; rec[2] = 0; rec[3] = 0; }
                continue;
            }
            const float zlo = q3.x, zhi = q3.y;
            const float fu = (float)u, fv = (float)v;
            // ---- 1. bound of the projected frustum, clipped to the slab
            HullBound hb;
            hb.any = false;
            hb.xmajor = true;
            hb.b = 0.0f;
            bool check_nf = true;  // near / far test of every sample needed
            {
                const float4 q0 = sl[0], q1 = sl[1], q2 = sl[2];
                const float Mf[9] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x}, ef[3] = {q2.y, q2.z, q2.w};
                {
                    // direction of the projected central ray (its clipped end points), for the slope
                    const float A0 = fmaf(Mf[0], fu, fmaf(Mf[1], fv, Mf[2]));
                    const float A1 = fmaf(Mf[3], fu, fmaf(Mf[4], fv, Mf[5]));
                    const float A2 = fmaf(Mf[6], fu, fmaf(Mf[7], fv, Mf[8]));
                    float za, zb;
                    if (zlo <= zhi && slab_interval(ef[2], A2, zlo, zhi, nearp, farp, za, zb)) {
                        const float wa = fmaf(A2, za, ef[2]), wb = fmaf(A2, zb, ef[2]);
                        const float xa = fmaf(A0, za, ef[0]) / wa, ya = fmaf(A1, za, ef[1]) / wa;
                        const float xb = fmaf(A0, zb, ef[0]) / wb, yb = fmaf(A1, zb, ef[1]) / wb;
                        const float dx = xb - xa, dy = yb - ya;
                        if (isfinite(dx) && isfinite(dy)) {
                            hb.xmajor = fabsf(dx) >= fabsf(dy);
                            const float den = hb.xmajor ? dx : dy;
                            if (fabsf(den) > 1e-6f) hb.b = (hb.xmajor ? dy : dx) / den;
                        }
                    }
                }
                hb.lo = hb.mlo = __int_as_float(0x7f800000);
                hb.hi = hb.mhi = -__int_as_float(0x7f800000);
                if (zlo <= zhi) {
                    float Ma[3], Mi[3];
                    const float Mz[3] = {Mf[6], Mf[7], Mf[8]};
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        Ma[i] = hb.xmajor ? Mf[i] : Mf[3 + i];
                        Mi[i] = hb.xmajor ? Mf[3 + i] : Mf[i];
                    }
                    if (lateral_fast(Ma, Mi, Mz, hb.xmajor ? ef[0] : ef[1], hb.xmajor ? ef[1] : ef[0], ef[2], fu, fv, L, nearp,
                                     farp, zlo, zhi, hb)) {
                        check_nf = false;
                    } else {
                        // general case: all 12 edges of V clipped to the slab and to [near, far]
                        hb.any = false;
                        hb.lo = hb.mlo = __int_as_float(0x7f800000);
                        hb.hi = hb.mhi = -__int_as_float(0x7f800000);
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            const float cu = corner_u(c, fu, L), cv = corner_v(c, fv, L);
                            const int c2 = (c + 1) & 3;
                            const float du = corner_u(c2, fu, L) - cu, dv = corner_v(c2, fv, L) - cv;
                            lateral_edge(Mf, ef, cu, cv, nearp, farp, zlo, zhi, hb);
                            face_edge(Mf, ef, nearp, cu, cv, du, dv, zlo, zhi, hb);
                            face_edge(Mf, ef, farp, cu, cv, du, dv, zlo, zhi, hb);
                        }
                    }
                }
            }
            if (DEBUG && rec) { rec[0] = 0; rec[1] = 0; rec[2] = 0; rec[3] = 0; }
            if (!hb.any) continue;
            // rounding margin: FP32 end points are off by far less than 0.02 px + 1e-5 relative
            const float mg = 0.02f;
            float lo = hb.lo - (mg + 1e-5f * fabsf(hb.lo)), hi = hb.hi + (mg + 1e-5f * fabsf(hb.hi));
            const float mlo = hb.mlo - (mg + 1e-5f * fabsf(hb.mlo)), mhi = hb.mhi + (mg + 1e-5f * fabsf(hb.mhi));
            const int nmaj = hb.xmajor ? P.W : P.H, nmin = hb.xmajor ? P.H : P.W;
            // NaN bounds (degenerate projections) scan the whole image: fmaxf/fminf drop NaN; the
            // clamps on both sides keep every float -> int conversion in range
            const int m0 = (int)fminf(fmaxf(ceilf(mlo), 0.0f), (float)nmaj);
            const int m1 = (int)fmaxf(fminf(floorf(mhi), (float)(nmaj - 1)), -1.0f);
            if (m0 > m1) continue;
            if (DEBUG && rec) rec[0] = 1;
            // ---- 2. back-projection test rows, centred on p: h = d (R q~) + E; along the major axis sm, along
            // the minor one sn, and the constant
            float sm1, sm2, sm3, sn1, sn2, sn3, r1c, r2c, r3c, E1, E2, E3;
            {
                const float4 q4 = sl[4], q5 = sl[5], q6 = sl[6];
                const float R1[3] = {fmaf(-fu, q5.z, q4.x), fmaf(-fu, q5.w, q4.y), fmaf(-fu, q6.x, q4.z)};
                const float R2[3] = {fmaf(-fv, q5.z, q4.w), fmaf(-fv, q5.w, q5.x), fmaf(-fv, q6.x, q5.y)};
                E1 = fmaf(-fu, q6.w, q6.y);
                E2 = fmaf(-fv, q6.w, q6.z);
                E3 = q6.w;
                sm1 = hb.xmajor ? R1[0] : R1[1]; sm2 = hb.xmajor ? R2[0] : R2[1]; sm3 = hb.xmajor ? q5.z : q5.w;
                sn1 = hb.xmajor ? R1[1] : R1[0]; sn2 = hb.xmajor ? R2[1] : R2[0]; sn3 = hb.xmajor ? q5.w : q5.z;
                r1c = R1[2]; r2c = R2[2]; r3c = q6.x;
            }
            const float ifxO = s_const[4], ifyO = s_const[5], ux = fu - s_const[6], vy = fv - s_const[7];
            const float ifxJ = SR ? sl[7].x : 0.0f;  // 1 / fx of J for Eq. 7's area term
            const float beta = q3.z;
            const long long fbase = (long long)J * P.fstride + (long long)kPad * P.pitch + kPad;
            const int mstep = hb.xmajor ? 1 : P.pitch, nstep = hb.xmajor ? P.pitch : 1;
            const float *plane = P.depth + fbase;
            int mc = 0;
            unsigned long long mh = 0ull;
            // the pixel at (m, n) by the exact test of Eq. 2 (unless `tested` already); a sample joins the sums
            auto take = [&](int m, int n, auto tested) {
                const int pos = m * mstep + n * nstep;
                float d;
                float3 c;
                load_sample<CFMT>(plane, CFMT == 0 ? (const void *)(reinterpret_cast<const float4 *>(P.colour) + fbase)
                                                   : (const void *)(reinterpret_cast<const uint2 *>(P.colour) + fbase),
                                  pos, d, c);
                // Eq. 2: |h1| + |h2| < L h3 as |h1 + h2| < L h3 and |h1 - h2| < L h3
                const float fm = (float)m, fn = (float)n;
                const float b1 = fmaf(sn1, fn, r1c), b2 = fmaf(sn2, fn, r2c), b3 = fmaf(sn3, fn, r3c);
                const float hs = fmaf(d, fmaf(sm1 + sm2, fm, b1 + b2), E1 + E2);
                const float hd = fmaf(d, fmaf(sm1 - sm2, fm, b1 - b2), E1 - E2);
                const float h3 = fmaf(d, fmaf(sm3, fm, b3), E3);
                if (!decltype(tested)::value && !(fabsf(hs) < L * h3 && fabsf(hd) < L * h3)) return;
                if (check_nf && !(fabsf(h3 - zmid) < zhalf)) return;
                const float h1 = fmaf(d, fmaf(sm1, fm, b1), E1), h2 = fmaf(d, fmaf(sm2, fm, b2), E2);
                // Eq. 9: masked samples weigh 0 in the mean-shift steps (semi-transparency:
                // except for their Eq. 4 term in the last pass)
                const bool masked = INP && pass > 0 && __ldg(P.mask + fbase + pos) != 0;
                const bool add4 = INP == 2 && pass == 2 && own;
                if (masked && !add4) return;
                const float er = c.x - cref.x, eg = c.y - cref.y, eb = c.z - cref.z;
                float w = 1.0f;
                if (wpass) {
                    const float dz = h3 - dref;
                    const float ex = fmaf(ux, dz, h1) * ifxO, ey = fmaf(vy, dz, h2) * ifyO;
                    const float d2 = fmaf(ex, ex, fmaf(ey, ey, dz * dz));
                    // inpainting's colour term has no position or frame term
                    float x = INP ? -a_rgb * fmaf(er, er, fmaf(eg, eg, eb * eb))
                                  : -fmaf(a_rgb, fmaf(er, er, fmaf(eg, eg, eb * eb)), fmaf(a_xyz, d2, beta));
                    float w_rel = 1.0f;  // the sample's weight relative to 2^x
                    if (add4) {
                        // the two weights of the semi-transparency step, relative to the larger
                        const float fr = c.x - c_in.x, fg = c.y - c_in.y, fb = c.z - c_in.z;
                        const float x4 = -fmaf(a_rgb, fmaf(fr, fr, fmaf(fg, fg, fb * fb)), fmaf(a_xyz, d2, beta));
                        const float xi = masked ? -__int_as_float(0x7f800000) : x;
                        x = fmaxf(xi, x4);
                        w_rel = ex2(xi - x) + ex2(x4 - x);
                    }
                    if (SR) {  // Eq. 7: s_area = (d / fx_J)^2, the sample's pixel edge squared
                        const float edge = d * ifxJ;
                        x = fmaf(-a_area, edge * edge, x);
                    }
                    if (x > m_log2) {  // new largest weight: rescale what was summed so far
                        const float sc = ex2(m_log2 - x);
                        acc_r *= sc;
                        acc_g *= sc;
                        acc_b *= sc;
                        acc_w *= sc;
                        m_log2 = x;
                    }
                    w = w_rel * ex2(x - m_log2);
                }
                acc_r = fmaf(w, er, acc_r);
                acc_g = fmaf(w, eg, acc_g);
                acc_b = fmaf(w, eb, acc_b);
                acc_w += w;
                if (pass == 0) ++n_acc;
                if (DEBUG && pass == 0) {
                    const int qx = hb.xmajor ? m : n, qy = hb.xmajor ? n : m;
                    ++mc;
                    mh += mix64((unsigned long long)qy * (unsigned long long)P.W + (unsigned long long)qx + 1ull);
                }
            };
            if (!LONG || __float_as_int(sl[7].y) == 0) {
                // Short hulls: row by row of the minor axis, each row a run along the major axis, every candidate
                // b m + lo <= n <= b m + hi, m in [m0, m1] by the packed exact test (two candidates an operation;
                // |h1| + |h2| is the larger of |h1 + h2| and |h1 - h2|), up to 32 into a hit mask
                const float fb0 = fmaf(hb.b, (float)m0, 0.0f), fb1 = fmaf(hb.b, (float)m1, 0.0f);
                const int r0 = (int)fminf(fmaxf(ceilf(fminf(fb0, fb1) + lo), 0.0f), (float)nmin);
                const int r1 = (int)fmaxf(fminf(floorf(fmaxf(fb0, fb1) + hi), (float)(nmin - 1)), -1.0f);
                const bool flat = fabsf(hb.b) < 1e-6f;
                const float ib = flat ? 0.0f : 1.0f / hb.b;
                const f32x2 sp2 = f2_pack(sm1 + sm2, sm1 + sm2), sq2 = f2_pack(sm1 - sm2, sm1 - sm2), s32 = f2_pack(sm3, sm3);
                const f32x2 Ep2 = f2_pack(E1 + E2, E1 + E2), Eq2 = f2_pack(E1 - E2, E1 - E2), E32 = f2_pack(E3, E3);
                const f32x2 L2 = f2_pack(L, L), off01 = f2_pack(0.0f, 1.0f), off23 = f2_pack(2.0f, 3.0f);
                for (int n = r0; n <= r1; ++n) {
                    const float fn = (float)n;
                    int ma = m0, mb = m1;
                    if (!flat) {
                        // rounding of ta, tb is far below the 0.02 px margin already in lo and hi
                        const float ta = (fn - hi) * ib, tb = (fn - lo) * ib;
                        ma = max(m0, (int)fminf(fmaxf(ceilf(fminf(ta, tb) - 1e-3f), -1.0f), (float)nmaj));
                        mb = min(m1, (int)fmaxf(fminf(floorf(fmaxf(ta, tb) + 1e-3f), (float)nmaj), -1.0f));
                    }
                    if (ma > mb) continue;
                    if (pass == 0) n_exam += mb - ma + 1;
                    const float b1 = fmaf(sn1, fn, r1c), b2 = fmaf(sn2, fn, r2c), b3 = fmaf(sn3, fn, r3c);
                    const f32x2 bp2 = f2_pack(b1 + b2, b1 + b2), bq2 = f2_pack(b1 - b2, b1 - b2), b32 = f2_pack(b3, b3);
                    const float *rowp = plane + (long long)n * nstep;
                    for (int mc0 = ma; mc0 <= mb; mc0 += 32) {
                        const int cnt = min(mb - mc0, 31);
                        const float *dp = rowp + (long long)mc0 * mstep;
                        float fm = (float)mc0;
                        unsigned int hit = 0u;
                        // four candidates per step, their loads in flight together; the last step may read up to 3
                        // pixels past the run, inside the image or its 32-pixel padding, and their bits are dropped
                        for (int k = 0; k <= cnt; k += 4, dp += 4 * mstep, fm += 4.0f) {
                            float dq[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) dq[i] = __ldg(dp + i * mstep);
                            unsigned int bits = 0u;
                            const f32x2 fm2 = f2_pack(fm, fm);
#pragma unroll
                            for (int pr = 0; pr < 2; ++pr) {
                                const f32x2 fmp = f2_add(fm2, pr == 0 ? off01 : off23);
                                const f32x2 d2 = f2_pack(dq[2 * pr], dq[2 * pr + 1]);
                                const f32x2 sv = f2_fma(d2, f2_fma(sp2, fmp, bp2), Ep2);  // h1 + h2
                                const f32x2 tv = f2_fma(d2, f2_fma(sq2, fmp, bq2), Eq2);  // h1 - h2
                                const f32x2 cv = f2_mul(L2, f2_fma(d2, f2_fma(s32, fmp, b32), E32));
                                float sa, sb, ta, tb, ca, cb;
                                f2_unpack(sv, sa, sb);
                                f2_unpack(tv, ta, tb);
                                f2_unpack(cv, ca, cb);
                                // NaN depth fails the comparisons
                                const bool h0 = fabsf(sa) < ca && fabsf(ta) < ca, h1 = fabsf(sb) < cb && fabsf(tb) < cb;
                                bits |= ((unsigned int)h0 << (2 * pr)) | ((unsigned int)h1 << (2 * pr + 1));
                            }
                            // keep the bits of candidates inside the run (k + i <= cnt)
                            bits &= (2u << min(cnt - k, 3)) - 1u;
                            hit |= bits << k;
                        }
                        while (hit) {
                            const int k = __ffs((int)hit) - 1;
                            hit &= hit - 1u;
                            take(mc0 + k, n, std::true_type{});
                        }
                    }
                }
            } else {
                // examined candidates: the pixels of the parallelogram b m + lo <= n <= b m + hi, m in [m0, m1],
                // counted along the rows of its minor axis (|b| <= 1), whichever way they are decided below
                if (pass == 0) {
                    const float fb0 = fmaf(hb.b, (float)m0, 0.0f), fb1 = fmaf(hb.b, (float)m1, 0.0f);
                    const int r0 = (int)fminf(fmaxf(ceilf(fminf(fb0, fb1) + lo), 0.0f), (float)nmin);
                    const int r1 = (int)fmaxf(fminf(floorf(fmaxf(fb0, fb1) + hi), (float)(nmin - 1)), -1.0f);
                    if (fabsf(hb.b) < 1e-6f) {
                        if (r0 <= r1) n_exam += (long long)(r1 - r0 + 1) * (m1 - m0 + 1);
                    } else {
                        // rounding of the ends is far below the 0.02 px margin already in lo and hi
                        const float ib = 1.0f / hb.b, first = ib > 0.0f ? hi : lo, last = ib > 0.0f ? lo : hi;
                        int cnt = 0;
                        float fn = (float)r0;
                        for (int n = r0; n <= r1; ++n, fn += 1.0f) {
                            const float ta = __fsub_rn(__fmul_rn(fn - first, ib), 1e-3f), tb = __fadd_rn(__fmul_rn(fn - last, ib), 1e-3f);
                            const int ma = min(max(m0, __float2int_ru(ta)), nmaj), mb = tb == tb ? max(min(m1, __float2int_rd(tb)), -1) : m1;
                            cnt += max(mb - ma + 1, 0);
                        }
                        n_exam += cnt;
                    }
                }
                // a band wider than the image, or undefined: the whole image
                if (!(hi - lo < (float)(nmin + 64))) {
                    hb.b = lo = 0.0f;
                    hi = (float)(nmin - 1);
                }

                // Each of Eq. 2's two bounds, |h1 + h2| < L h3 and |h1 - h2| < L h3, as two quantities that are both
                // negative (packed): s - Lm h3 and -s - Lm h3 with s = h1 + h2, and the same with t = h1 - h2; Lm
                // is a rounding margin above L.  Each is d (cm m + cn n + c0) + cE.
                const float Lm = L + 0.01f + 2e-6f * (float)(P.W + P.H);
                auto form = [&](float x, float x3) { return f2_pack(fmaf(-Lm, x3, x), fmaf(-Lm, x3, -x)); };
                const f32x2 sm = form(sm1 + sm2, sm3), sn = form(sn1 + sn2, sn3), sc = form(r1c + r2c, r3c), sE = form(E1 + E2, E3);
                const f32x2 tm_ = form(sm1 - sm2, sm3), tn_ = form(sn1 - sn2, sn3), tc = form(r1c - r2c, r3c), tE = form(E1 - E2, E3);
                // For whole blocks one bound: along the direction (x1, x2) in which O positions move with depth, |x1|,
                // |x2| <= 1, a sample has |x1 h1 + x2 h2| <= |h1| + |h2| < L h3
                f32x2 cm, cn, c0, cE;
                {
                    const float ae = fmaxf(fabsf(E1), fabsf(E2)), ra = ae > 1e-30f ? rcp_approx(ae) : 0.0f;
                    const float x1 = ae > 1e-30f ? E1 * ra : 1.0f, x2 = E2 * ra;
                    cm = form(fmaf(x1, sm1, x2 * sm2), sm3);
                    cn = form(fmaf(x1, sn1, x2 * sn2), sn3);
                    c0 = form(fmaf(x1, r1c, x2 * r2c), r3c);
                    cE = form(fmaf(x1, E1, x2 * E2), E3);
                }
                // The band as columns: position m holds the minor pixels from ceil(b m + lo) on, at most nc; their
                // first is found by rounding b m + lo + 0.49, which may start one pixel early
                const float bb = hb.b, start = lo + 0.49f;
                const int nc = (int)(hi - lo + 0.02f) + 1, nch = (nc + 3) >> 2;  // in chunks of four, or two where that holds them
                const bool narrow = nc <= 2;
                // on the band's centre line, less what half the band's width can change: a lower bound of the
                // factor of d in P and Q
                const float hw = 0.5f * (hi - lo) + 0.02f, nmid = 0.5f * (lo + hi);
                const f32x2 am = f2_fma(cn, f2_pack(bb, bb), cm);
                const f32x2 a0 = f2_sub(f2_fma(cn, f2_pack(nmid, nmid), c0), f2_mul(f2_abs(cn), f2_pack(hw, hw)));
                const int TX = (P.W + kTile - 1) / kTile, TY = (P.H + kTile - 1) / kTile;
                const float2 *tiles = P.tiles + (long long)J * TX * TY;
                const int tm = hb.xmajor ? 1 : TX, tn = hb.xmajor ? TX : 1, ntn = hb.xmajor ? TY : TX;
                for (int blk0 = m0 / kTile; blk0 <= m1 / kTile; blk0 += 32) {
                    // the blocks of this group of 32 that may hold a sample
                    unsigned todo = 0u;
                    const int nb = min(m1 / kTile - blk0, 31);
#pragma unroll 2
                    for (int i = 0; i <= nb; ++i) {
                        const float fm = (float)((blk0 + i) * kTile);
                        const float e0 = fmaf(bb, fm, lo), e1 = fmaf(bb, fm + (float)(kTile - 1), lo);
                        // the tiles that the band touches over the block: one or two, more only for wide bands
                        const int t0 = max(__float2int_rd((fminf(e0, e1) - 0.02f) * (1.0f / kTile)), 0);
                        const int t1 = min(__float2int_rd((fmaxf(e0, e1) + (hi - lo) + 0.02f) * (1.0f / kTile)), ntn - 1);
                        const float2 *tp = tiles + (blk0 + i) * tm;
                        const int ta = min(t0, ntn - 1), tb = max(min(t0 + 1, t1), 0);
                        const float2 ra = __ldg(tp + ta * tn), rb = __ldg(tp + tb * tn);
                        float dlo = fminf(ra.x, rb.x), dhi = fmaxf(ra.y, rb.y);
                        for (int t = t0 + 2; t <= t1; ++t) {
                            const float2 r = __ldg(tp + t * tn);
                            dlo = fminf(dlo, r.x);
                            dhi = fmaxf(dhi, r.y);
                        }
                        const f32x2 dd = f2_pack(dlo, dhi);
                        const f32x2 g0 = f2_fma(am, f2_pack(fm, fm), a0), g1 = f2_fma(am, f2_pack((float)(kTile - 1), (float)(kTile - 1)), g0);
                        float p0, q0, p1, q1, pe, qe;
                        f2_unpack(g0, p0, q0);
                        f2_unpack(g1, p1, q1);
                        f2_unpack(cE, pe, qe);
                        // both quantities at the ends of the depth range and of the block: one that is nowhere negative
                        // there is nowhere negative between (linear in each)
                        const f32x2 pp = f2_fma(dd, f2_pack(p0, p0), f2_pack(pe, pe)) | f2_fma(dd, f2_pack(p1, p1), f2_pack(pe, pe));
                        const f32x2 qq = f2_fma(dd, f2_pack(q0, q0), f2_pack(qe, qe)) | f2_fma(dd, f2_pack(q1, q1), f2_pack(qe, qe));
                        const unsigned sp = (unsigned)(pp >> 32) | (unsigned)pp, sq = (unsigned)(qq >> 32) | (unsigned)qq;
                        // t0 > t1: outside the image; dlo > dhi: no valid depth
                        todo |= t0 <= t1 && dlo <= dhi ? ((sp & sq) >> 31) << i : 0u;
                    }
                    while (todo) {
                        const int i = __ffs((int)todo) - 1;
                        todo &= todo - 1u;
                        const int mb = (blk0 + i) * kTile;
                        for (int ch = 0; ch < nch; ++ch) {
                            // 8 positions x 2 or 4 pixels across the band, the first in the top bit.  Pixels beyond the
                            // band or the hull are never samples; the reads stay inside the image or its 32-pixel padding
                            unsigned hit = 0u;
                            auto columns = [&](auto per) {
                                constexpr int N = decltype(per)::value;
#pragma unroll
                                for (int c = 0; c < kTile; ++c) {
                                    const float fm = (float)(mb + c);
                                    const float t = fmaf(bb, fm, start) + kRound;
                                    const int n = min(max(__float_as_int(t) - __float_as_int(kRound) + 4 * ch, -4), nmin);
                                    const float fn = (t - kRound) + (float)(4 * ch);
                                    const f32x2 fm2 = f2_pack(fm, fm), fn2 = f2_pack(fn, fn);
                                    f32x2 As = f2_fma(sn, fn2, f2_fma(sm, fm2, sc)), At = f2_fma(tn_, fn2, f2_fma(tm_, fm2, tc));
                                    const float *dp = plane + (mb + c) * mstep + n * nstep;
                                    float d[N];
#pragma unroll
                                    for (int r = 0; r < N; ++r) d[r] = __ldg(dp + r * nstep);
#pragma unroll
                                    for (int r = 0; r < N; ++r) {
                                        float p, q, x, y;
                                        f2_unpack(f2_fma(f2_pack(d[r], d[r]), As, sE), p, q);
                                        f2_unpack(f2_fma(f2_pack(d[r], d[r]), At, tE), x, y);
                                        hit = __funnelshift_l(__float_as_uint(fmaxf(max3(p, q, x), y)), hit, 1);
                                        if (r < N - 1) {
                                            As = f2_add(As, sn);
                                            At = f2_add(At, tn_);
                                        }
                                    }
                                }
                            };
                            if (narrow) {
                                columns(std::integral_constant<int, 2>{});
                                hit <<= 16;
                            } else {
                                columns(std::integral_constant<int, 4>{});
                            }
                            while (hit) {
                                const int k = __clz((int)hit);
                                hit &= 0x7fffffffu >> k;
                                const int m = mb + (narrow ? k >> 1 : k >> 2);
                                const float t = fmaf(bb, (float)m, start) + kRound;
                                const int n = min(max(__float_as_int(t) - __float_as_int(kRound) + 4 * ch, -4), nmin) + (narrow ? k & 1 : k & 3);
                                take(m, n, std::false_type{});
                            }
                        }
                    }
                }
            }
            if (DEBUG && rec) {
                rec[1] = mc;
                rec[2] = (int32_t)(unsigned int)(mh & 0xffffffffull);
                rec[3] = (int32_t)(unsigned int)(mh >> 32);
            }
        }
        if (shares == 1 && ns > 1) {
            FrSums part = {acc_r, acc_g, acc_b, acc_w, m_log2}, &sum = s_red[threadIdx.x];
            if (!first) {
                FrSums all = sum;
                join_sums(all, part);
                part = all;
            }
            first = false;
            sum = part;
            acc_r = acc_g = acc_b = acc_w = 0.0f;
            m_log2 = wpass ? kNoWeight : 0.0f;
        }
      }
      if (shares == 1 && ns > 1) {
          const FrSums sum = s_red[threadIdx.x];
          acc_r = sum.r;
          acc_g = sum.g;
          acc_b = sum.b;
          acc_w = sum.w;
          m_log2 = sum.m;
      }
    }
    if (shares > 1) {
        // join the four threads' sums; every thread takes the result
        const int px = row * 32 + lane;
        s_red[threadIdx.x] = {acc_r, acc_g, acc_b, acc_w, m_log2};
        __syncthreads();
        FrSums sum = s_red[px];
#pragma unroll
        for (int s = 1; s < 4; ++s) join_sums(sum, s_red[s * (kFrThreads / 4) + px]);
        acc_r = sum.r;
        acc_g = sum.g;
        acc_b = sum.b;
        acc_w = sum.w;
        m_log2 = sum.m;
        __syncthreads();
    }
    sw_true = acc_w > 0.0f ? acc_w * exp2f(m_log2) : 0.0f;  // the true sum of weights of this pass
    if (INP && acc_w > 0.0f) {
        // this pass's weighted mean is the next pass's reference (and, after the last, the output)
        const float inv = 1.0f / acc_w;
        cref.x = fmaf(acc_r, inv, cref.x);
        cref.y = fmaf(acc_g, inv, cref.y);
        cref.z = fmaf(acc_b, inv, cref.z);
        acc_r = acc_g = acc_b = acc_w = 0.0f;
    }
    }  // passes

    if (DEBUG && S != 1) {
        atomicAdd(&s_dbg[row * 32 + lane][0], n_acc);
        atomicAdd(&s_dbg[row * 32 + lane][1], (int)min(n_exam, 0x7fffffffll));
        __syncthreads();
    }
    if (active && split == 0) {
        float o_r = cref.x, o_g = cref.y, o_b = cref.z;
        if (acc_w > 0.0f) {
            const float inv = 1.0f / acc_w;
            o_r = fmaf(acc_r, inv, o_r);
            o_g = fmaf(acc_g, inv, o_g);
            o_b = fmaf(acc_b, inv, o_b);
        }
        float *o = SR ? a.sr_out + (((long long)oi * Ho + v) * Wo + u) * 3 : P.out + (((long long)O * P.H + v) * P.W + u) * 3;
        o[0] = o_r;
        o[1] = o_g;
        o[2] = o_b;
        if (DEBUG && a.pixel_stats) {
            int32_t *ps = a.pixel_stats + crop_idx * 3;
            ps[0] = S != 1 ? s_dbg[row * 32 + lane][0] : n_acc;
            ps[1] = S != 1 ? s_dbg[row * 32 + lane][1] : (int32_t)min(n_exam, 0x7fffffffll);
            ps[2] = __float_as_int(sw_true);
        }
    }

    unsigned long long ce = (unsigned long long)n_exam, ca = (unsigned long long)n_acc;
    float sw = split == 0 ? sw_true : 0.0f;
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
        for (int i = 0; i < kFrThreads / 32; ++i) { te += s_cnt[0][i]; ta += s_cnt[1][i]; tw += s_w[i]; }
        atomicAdd(a.stat_counts, te);
        atomicAdd(a.stat_counts + 1, ta);
        atomicAdd(a.stat_sumw, tw);
    }
}

// Valid depth ranges of every frame and of its 8 x 8 pixel tiles: one warp per four tiles (32 columns,
// coalesced), grid (groups of four, tile rows in steps of 8, frames).  Positive floats order like their
// bit patterns, so a frame's range is kept as atomicMax of the bits (max) and of their complement (min);
// zero words mean "no valid depth".  A tile without one holds (inf, 0).
__global__ void __launch_bounds__(256) zrange_kernel(Planes P, unsigned int *zr, float2 *tiles) {
    const int f = blockIdx.z, lane = threadIdx.x & 31;
    const int TX = (P.W + kTile - 1) / kTile, TY = (P.H + kTile - 1) / kTile;
    const int ty = blockIdx.y * 8 + (threadIdx.x >> 5), x = blockIdx.x * 32 + lane;
    if (ty >= TY) return;
    // columns past the image lie in the padding (NaN), and so do rows
    const float *p = P.depth + (long long)f * P.fstride + (long long)(ty * kTile + kPad) * P.pitch + kPad + min(x, P.W);
    unsigned int mx = 0u, mn = 0u;
#pragma unroll
    for (int i = 0; i < kTile; ++i) {
        const unsigned int bits = __float_as_uint(__ldg(p + (long long)i * P.pitch));
        if (bits > 0u && bits < 0x7f800000u) {  // finite and > 0 (NaN pads fail)
            mx = max(mx, bits);
            mn = max(mn, ~bits);
        }
    }
#pragma unroll
    for (int o = 1; o < kTile; o <<= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        mn = max(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    }
    if ((lane & (kTile - 1)) == 0 && x < P.W)
        tiles[((long long)f * TY + ty) * TX + x / kTile] =
            mx ? make_float2(__uint_as_float(~mn), __uint_as_float(mx)) : make_float2(__int_as_float(0x7f800000), 0.0f);
#pragma unroll
    for (int o = kTile; o < 32; o <<= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        mn = max(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    }
    if (lane == 0 && mx) {
        atomicMax(zr + 2 * f, mn);
        atomicMax(zr + 2 * f + 1, mx);
    }
}

template <bool SR, int INP, int S, bool LONG>
cudaError_t launch_frustum_t(const GatherArgs &a, cudaStream_t s) {
    constexpr int kRows = kFrTileY / (S == 1 ? 1 : 4);
    const dim3 grid((a.cw + kFrTileX - 1) / kFrTileX, (a.ch + kRows - 1) / kRows, a.n_out);
    const bool dbg = a.membership || a.pixel_stats;
    const size_t smem = sizeof(float4) * kFrSlotVec * (size_t)a.n_slots;  // at most 32 KB
    void (*fn)(const GatherArgs) = a.clip.colour_fmt == 0
                                       ? (dbg ? frustum_kernel<0, true, SR, INP, S, LONG> : frustum_kernel<0, false, SR, INP, S, LONG>)
                                       : (dbg ? frustum_kernel<1, true, SR, INP, S, LONG> : frustum_kernel<1, false, SR, INP, S, LONG>);
    fn<<<grid, kFrThreads, smem, s>>>(a);
    return cudaGetLastError();
}

template <bool SR, int INP, int S>
cudaError_t launch_frustum_s(const GatherArgs &a, cudaStream_t s) {
    const float band = SR ? a.frustum_l / (float)a.sr_scale : a.frustum_l;
    return frustum_long_hulls(a.n_slots, std::max(a.clip.W, a.clip.H), band) ? launch_frustum_t<SR, INP, S, true>(a, s)
                                                                             : launch_frustum_t<SR, INP, S, false>(a, s);
}

// Eq. 8-9's mask from a scene-space box: per pixel of every frame, the world point of its depth
// (unprojected with K_J^-1 and the pose of J, in FP64 with every operation rounded on its own)
// inside the inclusive box -> 1.  cam: per frame K^-1 (9), R (9), t (3).  Pads stay 0.
__global__ void __launch_bounds__(256) mask_box_kernel(Planes P, const double *cam, double bx0, double by0, double bz0,
                                                       double bx1, double by1, double bz1) {
    const long long npx = (long long)P.W * P.H * P.F;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < npx; i += (long long)gridDim.x * blockDim.x) {
        const long long f = i / ((long long)P.W * P.H);
        const int rem = (int)(i - f * (long long)P.W * P.H);
        const int y = rem / P.W, x = rem - y * P.W;
        const long long o = f * P.fstride + (long long)(y + kPad) * P.pitch + (x + kPad);
        const float d = P.depth[o];
        unsigned char m = 0;
        if (d > 0.0f && d < __int_as_float(0x7f800000)) {  // NaN (invalid) fails
            const double *Ki = cam + 21 * f, *R = Ki + 9, *t = Ki + 18;
            const double q[3] = {(double)x, (double)y, 1.0};
            double Xc[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const double ray = __dadd_rn(__dadd_rn(__dmul_rn(Ki[3 * r], q[0]), __dmul_rn(Ki[3 * r + 1], q[1])),
                                             __dmul_rn(Ki[3 * r + 2], q[2]));
                Xc[r] = __dsub_rn(__dmul_rn((double)d, ray), t[r]);
            }
            double Xw[3];
#pragma unroll
            for (int c = 0; c < 3; ++c)
                Xw[c] = __dadd_rn(__dadd_rn(__dmul_rn(R[c], Xc[0]), __dmul_rn(R[3 + c], Xc[1])), __dmul_rn(R[6 + c], Xc[2]));
            m = Xw[0] >= bx0 && Xw[1] >= by0 && Xw[2] >= bz0 && Xw[0] <= bx1 && Xw[1] <= by1 && Xw[2] <= bz1;
        }
        P.mask[o] = m;
    }
}

}  // namespace

// Inpainting and semi-transparency gather for the masked pixels alone, in three passes; how many there are is known on
// the device only, so that a CTA decides itself.
cudaError_t launch_frustum(const GatherArgs &args, cudaStream_t s) {
    GatherArgs a = args;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    a.sms = sms;
    if (a.mode == SSVP_MODE_INPAINT && !a.sr_out) return launch_frustum_s<false, 1, 0>(a, s);
    if (a.mode == SSVP_MODE_SEMI && !a.sr_out) return launch_frustum_s<false, 2, 0>(a, s);
    const long long ctas = (long long)((a.cw + kFrTileX - 1) / kFrTileX) * ((a.ch + kFrTileY - 1) / kFrTileY) * a.n_out;
    const bool shared = frustum_shares(ctas, 3ll * sms, a.n_slots);
    if (a.sr_out) return shared ? launch_frustum_s<true, 0, 4>(a, s) : launch_frustum_s<true, 0, 1>(a, s);
    return shared ? launch_frustum_s<false, 0, 4>(a, s) : launch_frustum_s<false, 0, 1>(a, s);
}

cudaError_t launch_mask_box(const Planes &p, const double *cam, const double *box, cudaStream_t s) {
    const long long n = (long long)p.W * p.H * p.F;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 152 * 16);
    mask_box_kernel<<<blocks, 256, 0, s>>>(p, cam, box[0], box[1], box[2], box[3], box[4], box[5]);
    return cudaGetLastError();
}

cudaError_t launch_zrange(const Planes &p, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(p.zrange, 0, 2 * sizeof(unsigned int) * (size_t)p.F, s);
    if (e != cudaSuccess) return e;
    const int TY = (p.H + kTile - 1) / kTile;
    const dim3 grid((unsigned)((p.W + 31) / 32), (unsigned)((TY + 7) / 8), (unsigned)p.F);
    zrange_kernel<<<grid, 256, 0, s>>>(p, p.zrange, p.tiles);
    return cudaGetLastError();
}

}  // namespace ssvp
