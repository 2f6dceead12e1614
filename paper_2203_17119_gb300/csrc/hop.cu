// Wilson hop over all fifth-dimension (and right-hand-side) lanes.
//
//   (Dh psi)(x, l) = sum_mu (1 - g_mu) U_mu(x) psi(x+mu, l) + (1 + g_mu) U_mu(x-mu)^+ psi(x-mu, l)
//
// (the hopping term of D_W = (4 - M5) - Dh/2; the dagger swaps the two
// projectors).  The operator is identical on every lane l = r * Ls + s, so a
// CTA takes a tile of 4D sites of one parity and all of their lanes: the
// 8 links and 8 neighbour indices of every site of the tile are copied once
// into shared memory by one bulk (TMA) copy and reused by all lanes.  Each
// thread owns VL consecutive lanes of one site; spinor loads and stores are
// VL-wide vectors of the [site][12][lanes] layout, so a warp reads whole
// contiguous lane rows.  The spin projection to a half spinor uses the
// chiral-basis structure of (1 -+ g_mu): two colour vectors are transported
// per direction and the lower spins are rebuilt from them.
//
// Epilogues: PLAIN   out = scale * Dh in
//            MOO     out = M_oo x + scale * Dh in  (+ per-tile |out|^2),
//            the last step of the Schur operator M_pc = M_oo - M_oe M_ee^-1 M_eo.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <type_traits>
#include <map>
#include <utility>

#include "dev_common.cuh"
#include "dwf_internal.cuh"

namespace dwf {

struct HopArgs {
    const void* in;
    void* out;
    const void* xmoo;
    const void* links;   // parity table [site][8][9] complex (site-major)
    const double* links64;   // fixed-point hop: the FP64 table, for lanes the fixed point does not cover
    const int* fx_info;      // fixed-point hop: {link exponent, links covered by the fixed point}
                             // in device memory, so that a captured launch follows a new gauge field
    const int* nbr;      // [site][8]
    const int4* tiles;
    int T, N5, Ls, nrhs, ntiles;
    int lane_chunk;      // lanes of a site a CTA takes at a time (N5, or whole right-hand sides dividing it)
    int deal;            // sites are dealt to the site groups in turn across tiles
    int chunk;           // consecutive tiles a CTA takes before striding: neighbouring rows of
                         // the lattice on one SM, so y-neighbours are re-read from L1
    double scale, d, e, mf, b5, c5;
    double fa, inv_d, inv_den;   // EPI_BMINV: a = -e/d, 1/d, 1/(d (1 + mf a^Ls))
    double* partial;
    int* err;
    // EPI_POST: CG vectors (FP32) and per-system scalars
    void* cg_x;
    void* cg_r;
    const void* cg_p;
    const double* alpha;
    const int* run;
};

// Scans across the lanes of one right-hand side (Ls lanes held by Ls / VL
// consecutive threads of a warp) for the fifth-dimension factor between the
// hops of M_pc, B M^-1 = (b5 + c5 S)(d + e S)^-1 per chirality, S the
// twisted shift S_- (reads lane s - 1, wall -mf) or S_+ (s + 1).  With
// a = -e/d, S_-^Ls = -mf and (1 - a S)^-1 = sum_{k<Ls} (a S)^k / (1 + mf a^Ls):
//   (d + e S_-)^-1 x |_s = P_s / d - mf a^(s+1) P_(Ls-1) / (d (1 + mf a^Ls)),
//   P_s = sum_{t<=s} a^(s-t) x_t,
// a decayed prefix sum (in-thread, then across threads by shuffles); S_+ is
// the mirror image with suffix sums Q_s = sum_{t>=s} a^(t-s) x_t and
// a^(Ls-s) Q_0.
template <int VL>
struct ScanCtx {
    unsigned mask;          // the site group's threads
    int j, nthr, seg0;      // thread index in the rhs segment, threads per segment, its first lane
    float a, inv_d, wc;     // a, 1/d, mf / (d (1 + mf a^Ls))
    float mf, b5, c5;
    float astep[5];         // a^(VL o) for scan strides o = 1, 2, 4, 8, 16
    float pdn[VL], pup[VL]; // a^(s+1), a^(Ls-s) per lane
    float cdn[VL], cup[VL]; // carry factors a^(v+1), a^(VL-v)
};

template <int VL, bool DN>
__device__ __forceinline__ void scan_bminv(const ScanCtx<VL>& k, float (&x)[VL]) {
    float p[VL];
    if (DN) {
        p[0] = x[0];
#pragma unroll
        for (int v = 1; v < VL; ++v) p[v] = fmaf(k.a, p[v - 1], x[v]);
    } else {
        p[VL - 1] = x[VL - 1];
#pragma unroll
        for (int v = VL - 2; v >= 0; --v) p[v] = fmaf(k.a, p[v + 1], x[v]);
    }
    // inclusive scan of the thread totals over the segment (Hillis-Steele)
    const int me = k.seg0 + k.j;
    float tot = DN ? p[VL - 1] : p[0];
    // unrolled over the five possible strides (compile-time index into astep:
    // the context stays in registers); strides beyond the segment are skipped
#pragma unroll
    for (int lvl = 0; lvl < 5; ++lvl) {
        const int o = 1 << lvl;
        if (o < k.nthr) {
            const bool has = DN ? k.j >= o : k.j + o < k.nthr;
            const float v = __shfl_sync(k.mask, tot, has ? (DN ? me - o : me + o) : me);
            if (has) tot = fmaf(k.astep[lvl], v, tot);
        }
    }
    // carry in from the neighbouring thread's inclusive total
    const bool hc = DN ? k.j > 0 : k.j + 1 < k.nthr;
    const float carry = __shfl_sync(k.mask, tot, hc ? (DN ? me - 1 : me + 1) : me);
    if (hc) {
#pragma unroll
        for (int v = 0; v < VL; ++v) p[v] = fmaf(DN ? k.cdn[v] : k.cup[v], carry, p[v]);
    }
    // the wall term: P at the segment's last lane (Q at its first)
    const float T = __shfl_sync(k.mask, DN ? p[VL - 1] : p[0], DN ? k.seg0 + k.nthr - 1 : k.seg0);
    float y[VL];
#pragma unroll
    for (int v = 0; v < VL; ++v) y[v] = fmaf(-k.wc * (DN ? k.pdn[v] : k.pup[v]), T, p[v] * k.inv_d);
    // (b5 + c5 S) y
    float nb;
    if (DN) {
        const bool in = k.j > 0;
        nb = __shfl_sync(k.mask, y[VL - 1], in ? me - 1 : k.seg0 + k.nthr - 1) * (in ? 1.f : -k.mf);
    } else {
        const bool in = k.j + 1 < k.nthr;
        nb = __shfl_sync(k.mask, y[0], in ? me + 1 : k.seg0) * (in ? 1.f : -k.mf);
    }
#pragma unroll
    for (int v = 0; v < VL; ++v) {
        const float sv = DN ? (v > 0 ? y[(v + VL - 1) % VL] : nb) : (v < VL - 1 ? y[(v + 1) % VL] : nb);
        x[v] = fmaf(k.c5, sv, k.b5 * y[v]);
    }
}

// Lanes next to the first and last lane of this thread within its site
// group, for S5 across threads: the thread holding the lane above the last
// one (as its first lane) and the one holding the lane below the first one
// (as its last lane), with the wall factor -mf where the shift wraps.
struct LaneNbrs {
    int src_up, src_dn;
    unsigned mask;     // the site group's threads in the warp
    float f_up, f_dn;
};

// One direction K (0..3: +mu, 4..7: -mu) for the VL lanes of one site; src
// points at lane0 of the neighbour's spinor ([12][N5] complex), in global or
// shared memory.
template <int K, bool DAG, class Sin, class SL, class R, int VL>
__device__ __forceinline__ void hop_dir_src(const Sin* __restrict__ src, const SL* s_link, int N5,
                                            R (&ar)[12][VL], R (&ai)[12][VL]) {
    constexpr int MU = K & 3;
    constexpr bool FWD = K < 4;
    constexpr int SGI = (FWD != DAG) ? 1 : -1;   // (1 - SG g_mu) projector
    const R SG = (R)SGI;
    R ur[2][3][VL], ui[2][3][VL], lr[2][3][VL], li[2][3][VL];
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            load_lanes<Sin, VL, R>(src + (int64_t)((sp * 3 + c) * N5) * 2, ur[sp][c], ui[sp][c]);
            load_lanes<Sin, VL, R>(src + (int64_t)(((sp + 2) * 3 + c) * N5) * 2, lr[sp][c],
                                   li[sp][c]);
        }
    // half spinor h = u - SG A_mu l
    R hr[2][3][VL], hi[2][3][VL];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int v = 0; v < VL; ++v) {
            if (MU == 0) {
                hr[0][c][v] = ur[0][c][v] - SG * li[1][c][v];
                hi[0][c][v] = ui[0][c][v] + SG * lr[1][c][v];
                hr[1][c][v] = ur[1][c][v] - SG * li[0][c][v];
                hi[1][c][v] = ui[1][c][v] + SG * lr[0][c][v];
            } else if (MU == 1) {
                hr[0][c][v] = ur[0][c][v] + SG * lr[1][c][v];
                hi[0][c][v] = ui[0][c][v] + SG * li[1][c][v];
                hr[1][c][v] = ur[1][c][v] - SG * lr[0][c][v];
                hi[1][c][v] = ui[1][c][v] - SG * li[0][c][v];
            } else if (MU == 2) {
                hr[0][c][v] = ur[0][c][v] - SG * li[0][c][v];
                hi[0][c][v] = ui[0][c][v] + SG * lr[0][c][v];
                hr[1][c][v] = ur[1][c][v] + SG * li[1][c][v];
                hi[1][c][v] = ui[1][c][v] - SG * lr[1][c][v];
            } else {
                hr[0][c][v] = ur[0][c][v] - SG * lr[0][c][v];
                hi[0][c][v] = ui[0][c][v] - SG * li[0][c][v];
                hr[1][c][v] = ur[1][c][v] - SG * lr[1][c][v];
                hi[1][c][v] = ui[1][c][v] - SG * li[1][c][v];
            }
        }
    // g = W h (two colour vectors)
    const SL* w = s_link + K * 18;
    R gr[2][3][VL], gi[2][3][VL];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        R wr[3], wi[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) link_c<SL, R>(w, a * 3 + b, wr[b], wi[b]);
#pragma unroll
        for (int sp = 0; sp < 2; ++sp)
#pragma unroll
            for (int v = 0; v < VL; ++v) {
                R sr = wr[0] * hr[sp][0][v] - wi[0] * hi[sp][0][v];
                R si = wr[0] * hi[sp][0][v] + wi[0] * hr[sp][0][v];
                sr = fma(wr[1], hr[sp][1][v], sr); sr = fma(-wi[1], hi[sp][1][v], sr);
                si = fma(wr[1], hi[sp][1][v], si); si = fma(wi[1], hr[sp][1][v], si);
                sr = fma(wr[2], hr[sp][2][v], sr); sr = fma(-wi[2], hi[sp][2][v], sr);
                si = fma(wr[2], hi[sp][2][v], si); si = fma(wi[2], hr[sp][2][v], si);
                gr[sp][a][v] = sr;
                gi[sp][a][v] = si;
            }
    }
    // reconstruct: upper += g, lower += -SG A_mu^+ g
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int v = 0; v < VL; ++v) {
            ar[c][v] += gr[0][c][v];
            ai[c][v] += gi[0][c][v];
            ar[3 + c][v] += gr[1][c][v];
            ai[3 + c][v] += gi[1][c][v];
            if (MU == 0) {
                ar[6 + c][v] += SG * gi[1][c][v];
                ai[6 + c][v] -= SG * gr[1][c][v];
                ar[9 + c][v] += SG * gi[0][c][v];
                ai[9 + c][v] -= SG * gr[0][c][v];
            } else if (MU == 1) {
                ar[6 + c][v] -= SG * gr[1][c][v];
                ai[6 + c][v] -= SG * gi[1][c][v];
                ar[9 + c][v] += SG * gr[0][c][v];
                ai[9 + c][v] += SG * gi[0][c][v];
            } else if (MU == 2) {
                ar[6 + c][v] += SG * gi[0][c][v];
                ai[6 + c][v] -= SG * gr[0][c][v];
                ar[9 + c][v] -= SG * gi[1][c][v];
                ai[9 + c][v] += SG * gr[1][c][v];
            } else {
                ar[6 + c][v] -= SG * gr[0][c][v];
                ai[6 + c][v] -= SG * gi[0][c][v];
                ar[9 + c][v] -= SG * gr[1][c][v];
                ai[9 + c][v] -= SG * gi[1][c][v];
            }
        }
}

// The same direction for two lanes in FP32 with paired-FP32 instructions
// (fma/mul .f32x2 on sm_100 and later): each float2 holds one real or
// imaginary component of both lanes, so every operation of the scalar form
// above is one instruction for the pair.  Same formulas, same order.  Used
// for BF16 operands, whose conversion already yields separate components
// (15% faster at 32^4 x 16); for FP32 operands the regrouping of the loaded
// (re, im, re, im) quads and the extra register pressure made it slower.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

template <int K, bool DAG, class Sin, class SL>
__device__ __forceinline__ void hop_dir_x2(const Sin* __restrict__ src, const SL* s_link, int N5,
                                           float2 (&ar)[12], float2 (&ai)[12]) {
    constexpr int MU = K & 3;
    constexpr bool FWD = K < 4;
    constexpr float SG = (FWD != DAG) ? 1.f : -1.f;   // (1 - SG g_mu) projector
    const float2 P = f2(SG), M = f2(-SG);
    float2 ur[2][3], ui[2][3], lr[2][3], li[2][3];
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float re[2], im[2];
            load_lanes<Sin, 2, float>(src + (int64_t)((sp * 3 + c) * N5) * 2, re, im);
            ur[sp][c] = make_float2(re[0], re[1]);
            ui[sp][c] = make_float2(im[0], im[1]);
            load_lanes<Sin, 2, float>(src + (int64_t)(((sp + 2) * 3 + c) * N5) * 2, re, im);
            lr[sp][c] = make_float2(re[0], re[1]);
            li[sp][c] = make_float2(im[0], im[1]);
        }
    // half spinor h = u - SG A_mu l
    float2 hr[2][3], hi[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (MU == 0) {
            hr[0][c] = fma2(M, li[1][c], ur[0][c]);
            hi[0][c] = fma2(P, lr[1][c], ui[0][c]);
            hr[1][c] = fma2(M, li[0][c], ur[1][c]);
            hi[1][c] = fma2(P, lr[0][c], ui[1][c]);
        } else if (MU == 1) {
            hr[0][c] = fma2(P, lr[1][c], ur[0][c]);
            hi[0][c] = fma2(P, li[1][c], ui[0][c]);
            hr[1][c] = fma2(M, lr[0][c], ur[1][c]);
            hi[1][c] = fma2(M, li[0][c], ui[1][c]);
        } else if (MU == 2) {
            hr[0][c] = fma2(M, li[0][c], ur[0][c]);
            hi[0][c] = fma2(P, lr[0][c], ui[0][c]);
            hr[1][c] = fma2(P, li[1][c], ur[1][c]);
            hi[1][c] = fma2(M, lr[1][c], ui[1][c]);
        } else {
            hr[0][c] = fma2(M, lr[0][c], ur[0][c]);
            hi[0][c] = fma2(M, li[0][c], ui[0][c]);
            hr[1][c] = fma2(M, lr[1][c], ur[1][c]);
            hi[1][c] = fma2(M, li[1][c], ui[1][c]);
        }
    }
    // g = W h (two colour vectors)
    const SL* w = s_link + K * 18;
    float2 gr[2][3], gi[2][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float wr[3], wi[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) link_c<SL, float>(w, a * 3 + b, wr[b], wi[b]);
#pragma unroll
        for (int sp = 0; sp < 2; ++sp) {
            float2 sr = __fmul2_rn(f2(wr[0]), hr[sp][0]);
            float2 si = __fmul2_rn(f2(wr[0]), hi[sp][0]);
            sr = fma2(f2(-wi[0]), hi[sp][0], sr);
            si = fma2(f2(wi[0]), hr[sp][0], si);
            sr = fma2(f2(wr[1]), hr[sp][1], sr); sr = fma2(f2(-wi[1]), hi[sp][1], sr);
            si = fma2(f2(wr[1]), hi[sp][1], si); si = fma2(f2(wi[1]), hr[sp][1], si);
            sr = fma2(f2(wr[2]), hr[sp][2], sr); sr = fma2(f2(-wi[2]), hi[sp][2], sr);
            si = fma2(f2(wr[2]), hi[sp][2], si); si = fma2(f2(wi[2]), hr[sp][2], si);
            gr[sp][a] = sr;
            gi[sp][a] = si;
        }
    }
    // reconstruct: upper += g, lower += -SG A_mu^+ g
    const float2 one = f2(1.f);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        ar[c] = fma2(one, gr[0][c], ar[c]);
        ai[c] = fma2(one, gi[0][c], ai[c]);
        ar[3 + c] = fma2(one, gr[1][c], ar[3 + c]);
        ai[3 + c] = fma2(one, gi[1][c], ai[3 + c]);
        if (MU == 0) {
            ar[6 + c] = fma2(P, gi[1][c], ar[6 + c]);
            ai[6 + c] = fma2(M, gr[1][c], ai[6 + c]);
            ar[9 + c] = fma2(P, gi[0][c], ar[9 + c]);
            ai[9 + c] = fma2(M, gr[0][c], ai[9 + c]);
        } else if (MU == 1) {
            ar[6 + c] = fma2(M, gr[1][c], ar[6 + c]);
            ai[6 + c] = fma2(M, gi[1][c], ai[6 + c]);
            ar[9 + c] = fma2(P, gr[0][c], ar[9 + c]);
            ai[9 + c] = fma2(P, gi[0][c], ai[9 + c]);
        } else if (MU == 2) {
            ar[6 + c] = fma2(P, gi[0][c], ar[6 + c]);
            ai[6 + c] = fma2(M, gr[0][c], ai[6 + c]);
            ar[9 + c] = fma2(M, gi[1][c], ar[9 + c]);
            ai[9 + c] = fma2(P, gr[1][c], ai[9 + c]);
        } else {
            ar[6 + c] = fma2(M, gr[0][c], ar[6 + c]);
            ai[6 + c] = fma2(M, gi[0][c], ai[6 + c]);
            ar[9 + c] = fma2(M, gr[1][c], ar[9 + c]);
            ai[9 + c] = fma2(M, gi[1][c], ai[9 + c]);
        }
    }
}

template <int K, bool DAG, class Sin, class SL>
__device__ __forceinline__ void hop_dir2(const Sin* __restrict__ in, const int* s_nbr,
                                         const SL* s_link, int N5, int lane0, float2 (&ar)[12],
                                         float2 (&ai)[12]) {
    const int n = s_nbr[K];
    if (n < 0) return;   // link cut by a Dirichlet boundary
    hop_dir_x2<K, DAG, Sin, SL>(in + ((int64_t)n * 12 * N5 + lane0) * 2, s_link, N5, ar, ai);
}

template <int K, bool DAG, class Sin, class SL, class R, int VL>
__device__ __forceinline__ void hop_dir(const Sin* __restrict__ in, const int* s_nbr,
                                        const SL* s_link, int N5, int lane0, R (&ar)[12][VL],
                                        R (&ai)[12][VL]) {
    const int n = s_nbr[K];
    if (n < 0) return;   // link cut by a Dirichlet boundary
    hop_dir_src<K, DAG, Sin, SL, R, VL>(in + ((int64_t)n * 12 * N5 + lane0) * 2, s_link, N5, ar, ai);
}

// ------------------------------------------------ FP64 hop in fixed point
// GB300 has 2 FP64 lanes per clock and SM against 32 for the 32 x 32 -> 64-bit
// integer multiply-add, and the hop's 1320 flops per lane are what bounds the
// FP64 form (91% of the FP64 pipe).  So the FP64 hop transports in 64-bit
// fixed point: links as w = (w1 2^32 + w0) 2^(exp - 61), |w| < 1.125 2^exp, w0
// a signed word (set_gauge); the projected half spinors h as integers in units
// of 2^(E - 1080), E one above the largest biased exponent of any component
// met so far for this site and lane -- so |h| < 2^58 units, and when a larger
// one arrives the accumulators are shifted to the new unit.  With h = h1 2^32
// + h0 a real product is three multiply-adds,
//   w h 2^-64 = w1 h1 + (w1 h0 + w0 h1) 2^-32 + O(2^-2),
// the second sum enters the first by its high word (rounded: it starts at
// 2^31), and the colour sum and the sum over directions are integer adds.
// Bounds: the two product sums stay below 6 1.125 2^55 and 6 (1.125 2^60 +
// 2^57) < 2^63, the sum over directions below 2^62.
//
// Every number keeps FP64's precision, not only the largest.  A result is off
// by at most 25 of its units u (2.8 a direction: 2^-2 for each of six dropped
// w0 h0, 1/2 for the rounded high word, the rest for w and h; 2 for changes of
// the unit), about one u rms; the FP64 form by up to 16 2^-53 of the sum of
// the moduli of its terms.  So a lane keeps the fixed-point sums only where
// the terms of every one of its numbers reach 1.25 2^52 u: M adds, colour by
// colour and over the directions, the smaller |g| (larger of its parts) of the
// two transported spins, and each number takes one g from every direction.
// None of 2.4 M Gaussian lanes failed that (the median of M is 2^54.9 u, their
// least 2^52.6), and the error is 0.58 of the FP64 form's; where a third of the lanes are just
// covered it comes to about twice the FP64 form's (rms).  Lanes that fail run
// the FP64 form -- numbers that a larger one does not reach: links that do not
// mix two colours, a neighbour that the projector annihilates, one neighbour
// far above the others --, and so do a NaN, an infinity, all components below
// 2^-895 or one above 2^56, and a handle whose links are not finite or beyond
// 2^+-32 (set_gauge).  A warp with one such lane takes some 25 us longer, a
// fixed tail on small lattices: with the smallest |g| of all six components in
// one sum, one Gaussian lane in 10^5 failed, and 16^4 x 12 took 233 to 245 us
// instead of 217.  Telling them costs 3% of the bare hop (16^4 x 12 209 -> 217
// us).
//
// Measured, bare hop: 16^4 x 12 650 -> 217 us, 24^4 x 16 4.17 -> 1.37 ms (FP64
// form -> this); no pipe is full (FP64 half, integer multiply-add about 60%):
// the chains of dependent integer instructions at 16 warps per SM are what is
// left.
//
// Half of the projections and conversions (spin 0) run on the FP64 pipe (an
// add, an exponent add, a conversion), half (spin 1) as shifts of the
// mantissas: either alone would be the bound.  One body per mu serves both
// signs, to keep the loop within the instruction cache.
struct FxLink {
    int hi, lo;
};
constexpr int kFxCover = 0x140000;   // 1.25 2^52, high word

// |x| of the double v: mantissa aligned to bit 63, moved down by E + 6 - e;
// EB = (E + 6) << 21 | 0x1fffff
__device__ __forceinline__ unsigned long long fx_mag(uint2 v, uint32_t EB) {
    const uint32_t t = (EB - v.y - v.y) >> 21;
    const uint32_t mh = (v.y & 0xfffffu) | 0x100000u;
    const unsigned long long m = (((unsigned long long)mh << 32) | v.x) << 11;
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(t));   // 0 beyond 63
    return r;
}

// a + b in units of 2^(E - 1080); f = -1: a - b
__device__ __forceinline__ long long fx_sum(double a, double b, uint32_t EB, int f) {
    const uint2 va = make_uint2(__double2loint(a), __double2hiint(a)), vb = make_uint2(__double2loint(b), __double2hiint(b));
    const int sa = (int)va.y >> 31, sb = ((int)vb.y >> 31) ^ f;
    const unsigned long long ma = fx_mag(va, EB) ^ (unsigned long long)(long long)sa;
    const unsigned long long mb = fx_mag(vb, EB) ^ (unsigned long long)(long long)sb;
    return (long long)(ma + mb + (unsigned long long)(uint32_t)(-sa - sb));
}

// the same on the FP64 pipe, h = a + b given; sh = (1080 - E) << 20, E <= 1080
// (a zero becomes a number far below one half)
__device__ __forceinline__ long long fx_conv(double h, int sh) {
    return __double2ll_rn(__hiloint2double(__double2hiint(h) + sh, __double2loint(h)));
}

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }

// acc + g, or acc - g where f = -1
__device__ __forceinline__ void fx_add(long long& acc, long long g, int f) {
    acc += (g ^ (long long)f) + (long long)(f & 1);
}

// Spin structure of one direction: the half spinor h_q = u_q - SG A_mu l takes
// lower spin fx_low(MU, q), with a factor i for mu 0, 2, and sign +SG for
// (mu 1, q 0) and (mu 2, q 1), else -SG; -SG A_mu^+ g puts g_q back there.
__host__ __device__ constexpr int fx_low(int mu, int q) { return mu < 2 ? 3 - q : 2 + q; }
__host__ __device__ constexpr bool fx_itype(int mu) { return mu == 0 || mu == 2; }
__host__ __device__ constexpr bool fx_plus(int mu, int q) { return (mu == 1 && q == 0) || (mu == 2 && q == 1); }

// a half spinor split into signed words
struct FxHalf {
    int h1r[2][3], h0r[2][3], h1i[2][3], h0i[2][3];
};

// largest magnitude word of a neighbour's components, 0 if all are zero (or
// denormals below 2^-1042, which set bad): the signed maximum sees the
// positive numbers, the unsigned one the negative
__device__ __forceinline__ uint32_t fx_top(const double2 (&x)[12], bool& bad) {
    int sp = 0;
    uint32_t sn = 0;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const int a = __double2hiint(x[c].x), b = __double2hiint(x[c].y);
        sp = max(sp, max(a, b));
        sn = max(sn, max((uint32_t)a, (uint32_t)b));
    }
    const uint32_t top = max((uint32_t)sp, sn & 0x7fffffffu);
    if (top == 0) {
        uint32_t any = 0;
#pragma unroll
        for (int c = 0; c < 12; ++c) any |= __double2loint(x[c].x) | __double2loint(x[c].y);
        if (any) bad = true;
    }
    return top;
}

// The half spinor of direction MU in the unit of E; P, M = ~P the sign masks
// of +SG and -SG.
template <int MU>
__device__ __forceinline__ void fx_project(const double2 (&x)[12], int P, int E, FxHalf& h) {
    const int M = ~P;
    const uint32_t EB = ((uint32_t)(E + 6) << 21) | 0x1fffffu;
    const int sh = (1080 - E) << 20;
    const double SG = P == 0 ? 1.0 : -1.0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const bool plus = fx_plus(MU, q), im_plus = fx_itype(MU) ? !plus : plus;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 u = x[q * 3 + c], l = x[fx_low(MU, q) * 3 + c];
            const double lr = fx_itype(MU) ? l.y : l.x, li = fx_itype(MU) ? l.x : l.y;
            long long r, i;
            if (q == 0) {
                r = fx_conv(fma(plus ? SG : -SG, lr, u.x), sh);
                i = fx_conv(fma(im_plus ? SG : -SG, li, u.y), sh);
            } else {
                r = fx_sum(u.x, lr, EB, plus ? P : M);
                i = fx_sum(u.y, li, EB, im_plus ? P : M);
            }
            h.h0r[q][c] = (int)r;
            h.h1r[q][c] = (int)(r >> 32) + (int)((uint32_t)h.h0r[q][c] >> 31);
            h.h0i[q][c] = (int)i;
            h.h1i[q][c] = (int)(i >> 32) + (int)((uint32_t)h.h0i[q][c] >> 31);
        }
    }
}

// Row v (re high, re low, im high, im low of three links) times the two half spinors
__device__ __forceinline__ void fx_row(const int4 (&v)[3], const FxHalf& h, long long (&gr)[2], long long (&gi)[2]) {
    long long qr[2], qi[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) qr[q] = qi[q] = 0x80000000ll;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int n1 = -v[b].z, n0 = -v[b].w;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            qr[q] = fx_mad(v[b].x, h.h0r[q][b], qr[q]); qr[q] = fx_mad(v[b].y, h.h1r[q][b], qr[q]);
            qr[q] = fx_mad(n1, h.h0i[q][b], qr[q]); qr[q] = fx_mad(n0, h.h1i[q][b], qr[q]);
            qi[q] = fx_mad(v[b].x, h.h0i[q][b], qi[q]); qi[q] = fx_mad(v[b].y, h.h1i[q][b], qi[q]);
            qi[q] = fx_mad(v[b].z, h.h0r[q][b], qi[q]); qi[q] = fx_mad(v[b].w, h.h1r[q][b], qi[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        gr[q] = (long long)(int)(qr[q] >> 32);
        gi[q] = (long long)(int)(qi[q] >> 32);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int n1 = -v[b].z;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            gr[q] = fx_mad(v[b].x, h.h1r[q][b], gr[q]); gr[q] = fx_mad(n1, h.h1i[q][b], gr[q]);
            gi[q] = fx_mad(v[b].x, h.h1i[q][b], gi[q]); gi[q] = fx_mad(v[b].z, h.h1r[q][b], gi[q]);
        }
    }
}

// high word of the larger part of g
__device__ __forceinline__ int fx_size(long long r, long long i) {
    return max(abs((int)(r >> 32)), abs((int)(i >> 32)));
}

// Direction +mu (k < 4) or -mu in fixed point: acc += W h on the upper spins,
// rebuilt lower spins; E the accumulators' unit, M per colour the sum of the
// smaller |g| (high words), bad set where the FP64 form has to decide (denormals only).
template <int MU, bool DAG>
__device__ __forceinline__ void hop_dir_fx(int k, const double* __restrict__ in, const int* s_nbr,
                                           const FxLink* s_link, int N5, int lane0, long long (&ar)[12],
                                           long long (&ai)[12], int& E, int (&M)[3], bool& bad) {
    const int nb = s_nbr[k];
    if (nb < 0) return;
    const int P = ((k < 4) != DAG) ? 0 : -1, Pm = ~P;   // SG = +1 for (1 - g_mu)
    const double2* src = reinterpret_cast<const double2*>(in) + ((int64_t)nb * 12 * N5 + lane0);
    double2 x[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) x[c] = __ldg(src + (int64_t)c * N5);
    const uint32_t top = fx_top(x, bad);
    if (top == 0) return;
    const int Ed = (int)(top >> 20);
    if (Ed >= E) {
        const int d = min(Ed + 1 - E, 63);
        if (E > 0) {
#pragma unroll
            for (int c = 0; c < 12; ++c) { ar[c] >>= d; ai[c] >>= d; }
#pragma unroll
            for (int c = 0; c < 3; ++c) M[c] >>= min(d, 31);
        }
        E = Ed + 1;
    }
    FxHalf h;
    fx_project<MU>(x, P, E, h);
    const int4* w = reinterpret_cast<const int4*>(s_link) + k * 9;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int4 v[3] = {w[a * 3], w[a * 3 + 1], w[a * 3 + 2]};
        long long gr[2], gi[2];
        fx_row(v, h, gr, gi);
        M[a] += min(fx_size(gr[0], gi[0]), fx_size(gr[1], gi[1]));
        // rebuild: upper += g, lower += -SG A_mu^+ g
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int low = fx_low(MU, q) * 3 + a;
            const bool plus = fx_plus(MU, q);
            ar[q * 3 + a] += gr[q];
            ai[q * 3 + a] += gi[q];
            if (fx_itype(MU)) {
                fx_add(ar[low], gi[q], plus ? Pm : P);
                fx_add(ai[low], gr[q], plus ? P : Pm);
            } else {
                fx_add(ar[low], gr[q], plus ? P : Pm);
                fx_add(ai[low], gi[q], plus ? P : Pm);
            }
        }
    }
}

// The FP64 form of one site and lane (out of line: rarely taken)
template <bool DAG>
__device__ __noinline__ void hop_fx_fallback(const double* in, const int* nb, const double* lk, int N5, int lane0,
                                             double* r, double* i) {
    double ar[12][1], ai[12][1];
#pragma unroll
    for (int c = 0; c < 12; ++c) ar[c][0] = ai[c][0] = 0.0;
    hop_dir<0, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    hop_dir<4, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    hop_dir<1, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    hop_dir<5, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    hop_dir<2, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    hop_dir<6, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    hop_dir<3, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    hop_dir<7, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
#pragma unroll
    for (int c = 0; c < 12; ++c) { r[c] = ar[c][0]; i[c] = ai[c][0]; }
}

// Dh of one site and lane: ar, ai times the returned factor
template <bool DAG>
__device__ __forceinline__ double hop_site_fx(const double* __restrict__ in, const int* nb, const FxLink* lk,
                                              const double* lk64, int2 info, int N5, int lane0,
                                              double (&ar)[12][1], double (&ai)[12][1]) {
    long long r[12], i[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) r[c] = i[c] = 0;
    int E = 0, M[3] = {0, 0, 0};
    bool bad = false;
#pragma unroll 1
    for (int k = 0; k < 8; k += 4) hop_dir_fx<0, DAG>(k, in, nb, lk, N5, lane0, r, i, E, M, bad);
#pragma unroll 1
    for (int k = 1; k < 8; k += 4) hop_dir_fx<1, DAG>(k, in, nb, lk, N5, lane0, r, i, E, M, bad);
#pragma unroll 1
    for (int k = 2; k < 8; k += 4) hop_dir_fx<2, DAG>(k, in, nb, lk, N5, lane0, r, i, E, M, bad);
#pragma unroll 1
    for (int k = 3; k < 8; k += 4) hop_dir_fx<3, DAG>(k, in, nb, lk, N5, lane0, r, i, E, M, bad);
    // E = 0: every neighbour component is zero (or the FP64 form runs)
    if (((E != 0 || bad) && (E < 128 || E > 1080 || min(M[0], min(M[1], M[2])) < kFxCover)) || info.y == 0) {
        double tr[12], ti[12];
        hop_fx_fallback<DAG>(in, nb, lk64, N5, lane0, tr, ti);
#pragma unroll
        for (int c = 0; c < 12; ++c) { ar[c][0] = tr[c]; ai[c][0] = ti[c]; }
        return 1.0;
    }
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        ar[c][0] = __ll2double_rn(r[c]);
        ai[c][0] = __ll2double_rn(i[c]);
    }
    return __hiloint2double(max(E + info.x - 54, 1) << 20, 0);   // 2^(E + exp - 1077)
}

// Output of one site's VL lanes (acc = factor (ar, ai)): PLAIN out = scale * acc; MOO out = M_oo x +
// scale * acc, returning the lanes' |out|^2 (FP32 arithmetic: summed in FP32
// per site, one FP64 add per site, off GB300's slow FP64 pipe).
// Site groups (N5 / VL threads) known at compile time to divide a warp: the
// epilogues take a site's neighbouring fifth-dimension lane by shuffle.
template <int VL, int CN5>
constexpr bool kLaneShfl = CN5 > 0 && CN5 % VL == 0 && CN5 / VL <= 32 && 32 % (CN5 / VL) == 0;

template <class Sout, class R, int VL, bool DAG, int EPI, int CN5>
__device__ __forceinline__ double hop_store(const HopArgs& a, int N5, int64_t site, int lane0,
                                            const R (&ar)[12][VL], const R (&ai)[12][VL], R factor,
                                            const LaneNbrs& nb, int box, const ScanCtx<VL>& sk) {
    const R sc = (R)a.scale * factor;
    if constexpr (EPI == EPI_BMINV) {
        // out = scale B M^-1 acc: non-adjoint upper spins see S_-, lower S_+
        Sout* out = reinterpret_cast<Sout*>(a.out) + (site * 12 * N5 + lane0) * 2;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            float xr[VL], xi[VL];
#pragma unroll
            for (int v = 0; v < VL; ++v) { xr[v] = (float)ar[c][v]; xi[v] = (float)ai[c][v]; }
            if ((c < 6) != DAG) {
                scan_bminv<VL, true>(sk, xr);
                scan_bminv<VL, true>(sk, xi);
            } else {
                scan_bminv<VL, false>(sk, xr);
                scan_bminv<VL, false>(sk, xi);
            }
#pragma unroll
            for (int v = 0; v < VL; ++v) { xr[v] *= (float)sc; xi[v] *= (float)sc; }
            store_lanes<Sout, VL, float, true>(out + (int64_t)c * N5 * 2, xr, xi);
        }
        return 0.0;
    }
    if constexpr (EPI == EPI_POST) {
        static_assert(DAG, "the fused M_pc^+ tail follows the adjoint hop");
        // B^+ acc = b5 acc + c5 S5^+ acc on this site's lanes: S5^+ takes
        // lane s + 1 for the upper spins and s - 1 for the lower ones (walls
        // -mf); the lanes beyond this thread's come from its neighbours in
        // the site group
        const R b5 = (R)a.b5, c5 = (R)a.c5;
        R br[12][VL], bi[12][VL];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            if (c < 6) {
                const R nr = __shfl_sync(nb.mask, ar[c][0], nb.src_up) * (R)nb.f_up;
                const R ni = __shfl_sync(nb.mask, ai[c][0], nb.src_up) * (R)nb.f_up;
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    const R sr = v < VL - 1 ? ar[c][(v + 1) % VL] : nr;
                    const R si = v < VL - 1 ? ai[c][(v + 1) % VL] : ni;
                    br[c][v] = b5 * ar[c][v] + c5 * sr;
                    bi[c][v] = b5 * ai[c][v] + c5 * si;
                }
            } else {
                const R nr = __shfl_sync(nb.mask, ar[c][VL - 1], nb.src_dn) * (R)nb.f_dn;
                const R ni = __shfl_sync(nb.mask, ai[c][VL - 1], nb.src_dn) * (R)nb.f_dn;
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    const R sr = v > 0 ? ar[c][(v + VL - 1) % VL] : nr;
                    const R si = v > 0 ? ai[c][(v + VL - 1) % VL] : ni;
                    br[c][v] = b5 * ar[c][v] + c5 * sr;
                    bi[c][v] = b5 * ai[c][v] + c5 * si;
                }
            }
        }
        // Ap = M_oo^+ t + scale B^+ acc (t = xmoo; M_oo^+ = d + e S5^+ from
        // memory), then x += alpha p, r -= alpha Ap and |r|^2
        const int Ls = a.Ls;
        const int s0 = lane0 % Ls;
        const int rbase = lane0 - s0;
        const int sys = box * a.nrhs + lane0 / Ls;
        const R alpha = (R)a.alpha[sys];
        const bool live = a.run == nullptr || a.run[sys] != 0;
        const bool hi_wrap = (s0 + VL == Ls), lo_wrap = (s0 == 0);
        const int l_above = hi_wrap ? rbase : lane0 + VL;
        const int l_below = lo_wrap ? rbase + Ls - 1 : lane0 - 1;
        const R mf = (R)a.mf, d = (R)a.d, e = (R)a.e;
        // distinct fields: no aliasing, so the loads of later components can
        // be issued ahead of the stores of earlier ones
        const Sout* __restrict__ tb = reinterpret_cast<const Sout*>(a.xmoo) + (site * 12 * N5) * 2;
        float* __restrict__ xb = reinterpret_cast<float*>(a.cg_x) + (site * 12 * N5 + lane0) * 2;
        float* __restrict__ rb = reinterpret_cast<float*>(a.cg_r) + (site * 12 * N5 + lane0) * 2;
        const float* __restrict__ pb = reinterpret_cast<const float*>(a.cg_p) + (site * 12 * N5 + lane0) * 2;
        float nrm = 0.f;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            R tr[VL], ti[VL];
            load_lanes<Sout, VL, R>(tb + (int64_t)(c * N5 + lane0) * 2, tr, ti);
            const bool up = c < 6;   // S5^+: upper spins read s + 1
            R nr, ni, fn;
            if constexpr (kLaneShfl<VL, CN5>) {
                nr = __shfl_sync(nb.mask, up ? tr[0] : tr[VL - 1], up ? nb.src_up : nb.src_dn);
                ni = __shfl_sync(nb.mask, up ? ti[0] : ti[VL - 1], up ? nb.src_up : nb.src_dn);
                fn = (R)(up ? nb.f_up : nb.f_dn);
            } else {
                load_c1<Sout, R>(tb + (int64_t)(c * N5 + (up ? l_above : l_below)) * 2, nr, ni);
                fn = up ? (hi_wrap ? -mf : (R)1) : (lo_wrap ? -mf : (R)1);
            }
            float rr[VL], ri[VL];
            load_lanes<float, VL, float>(rb + (int64_t)c * N5 * 2, rr, ri);
            if (live) {
                float xr[VL], xi[VL], pr[VL], pi[VL];
                load_lanes<float, VL, float>(xb + (int64_t)c * N5 * 2, xr, xi);
                load_lanes<float, VL, float>(pb + (int64_t)c * N5 * 2, pr, pi);
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    R sr, si;
                    if (up) {
                        sr = v == VL - 1 ? fn * nr : tr[(v + 1) % VL];
                        si = v == VL - 1 ? fn * ni : ti[(v + 1) % VL];
                    } else {
                        sr = v == 0 ? fn * nr : tr[(v + VL - 1) % VL];
                        si = v == 0 ? fn * ni : ti[(v + VL - 1) % VL];
                    }
                    const R apr = d * tr[v] + e * sr + sc * br[c][v];
                    const R api = d * ti[v] + e * si + sc * bi[c][v];
                    xr[v] = fmaf((float)alpha, pr[v], xr[v]);
                    xi[v] = fmaf((float)alpha, pi[v], xi[v]);
                    rr[v] = fmaf(-(float)alpha, (float)apr, rr[v]);
                    ri[v] = fmaf(-(float)alpha, (float)api, ri[v]);
                }
                store_lanes<float, VL, float>(xb + (int64_t)c * N5 * 2, xr, xi);
                store_lanes<float, VL, float>(rb + (int64_t)c * N5 * 2, rr, ri);
            }
#pragma unroll
            for (int v = 0; v < VL; ++v) nrm = fmaf(rr[v], rr[v], fmaf(ri[v], ri[v], nrm));
        }
        return (double)nrm;
    }
    Sout* __restrict__ out = reinterpret_cast<Sout*>(a.out) + (site * 12 * N5 + lane0) * 2;
    if (EPI == EPI_PLAIN) {
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            R orr[VL], oi[VL];
#pragma unroll
            for (int v = 0; v < VL; ++v) {
                orr[v] = sc * ar[c][v];
                oi[v] = sc * ai[c][v];
            }
            store_lanes<Sout, VL, R, true>(out + (int64_t)c * N5 * 2, orr, oi);
        }
        return 0.0;
    }
    // M_oo x = d x + e S5 x on this site's lanes; S5 (non-dagger):
    // upper spins x_{s-1}, lower spins x_{s+1}, walls -mf.
    const Sout* __restrict__ xb = reinterpret_cast<const Sout*>(a.xmoo) + (site * 12 * N5) * 2;
    const int Ls = a.Ls;
    const int s0 = lane0 % Ls;
    const int rbase = lane0 - s0;
    const R d = (R)a.d, e = (R)a.e, mf = (R)a.mf;
    // neighbouring lanes below and above this thread's block
    const bool lo_wrap = (s0 == 0);
    const bool hi_wrap = (s0 + VL == Ls);
    const int l_below = lo_wrap ? rbase + Ls - 1 : lane0 - 1;
    const int l_above = hi_wrap ? rbase : lane0 + VL;
    const R f_below = lo_wrap ? -mf : (R)1;
    const R f_above = hi_wrap ? -mf : (R)1;
    double nrm = 0.0;
    float nrm_f = 0.f;
    // FP32: four rows at a time, their loads in flight before the first store
    // (one at a time, each row waited out its own latency: 791 us at 32^4 x 16
    // against 710, the plain epilogue 519; six rows gain nothing more).  FP64 has
    // no registers for more than one row.
    constexpr int NB = sizeof(R) == 8 ? 1 : 4;
#pragma unroll
    for (int c0 = 0; c0 < 12; c0 += NB) {
        R xr[NB][VL], xi[NB][VL], nr[NB], ni[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int c = c0 + b;
            load_lanes<Sout, VL, R>(xb + (int64_t)(c * N5 + lane0) * 2, xr[b], xi[b]);
            // upper spins use S_- (x_{s-1}) unless dagger, lower S_+
            if constexpr (!kLaneShfl<VL, CN5>)
                load_c1<Sout, R>(xb + (int64_t)(c * N5 + ((c < 6) != DAG ? l_below : l_above)) * 2, nr[b], ni[b]);
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int c = c0 + b;
            const bool use_below = (c < 6) != DAG;
            R fn = use_below ? f_below : f_above;
            if constexpr (kLaneShfl<VL, CN5>) {
                // the neighbouring lane is held by the adjacent thread of the site group
                nr[b] = __shfl_sync(nb.mask, use_below ? xr[b][VL - 1] : xr[b][0], use_below ? nb.src_dn : nb.src_up);
                ni[b] = __shfl_sync(nb.mask, use_below ? xi[b][VL - 1] : xi[b][0], use_below ? nb.src_dn : nb.src_up);
                if constexpr (sizeof(R) == 4) fn = (R)(use_below ? nb.f_dn : nb.f_up);   // (nb's factors are FP32)
            }
            R orr[VL], oi[VL];
            float part = 0.f;
#pragma unroll
            for (int v = 0; v < VL; ++v) {
                R sr, si;
                if (use_below) {
                    sr = (v == 0) ? fn * nr[b] : xr[b][v - 1];
                    si = (v == 0) ? fn * ni[b] : xi[b][v - 1];
                } else {
                    sr = (v == VL - 1) ? fn * nr[b] : xr[b][(v + 1) % VL];
                    si = (v == VL - 1) ? fn * ni[b] : xi[b][(v + 1) % VL];
                }
                orr[v] = d * xr[b][v] + e * sr + sc * ar[c][v];
                oi[v] = d * xi[b][v] + e * si + sc * ai[c][v];
                part += (float)(orr[v] * orr[v] + oi[v] * oi[v]);
                if (sizeof(R) == 8 && a.partial != nullptr) nrm += (double)orr[v] * orr[v] + (double)oi[v] * oi[v];
            }
            if (sizeof(R) != 8) nrm_f += part;
            store_lanes<Sout, VL, R, true>(out + (int64_t)c * N5 * 2, orr, oi);
        }
    }
    return sizeof(R) == 8 ? nrm : (double)nrm_f;
}

// Persistent kernel: CTA b takes tiles b, b + gridDim, ...; the links and
// neighbour indices of a tile arrive by bulk copy into one half of a double
// buffer.  There is no CTA-wide barrier in the tile loop: each warp waits for
// its tile's copy on the buffer's mbarrier, and the last warp to finish with
// a buffer (a shared-memory arrival counter) sums the per-warp norm partials
// in warp order and issues the copy of the tile two steps ahead into it, so
// fast warps run on into the next tile.
// CN5 > 0 fixes N5 = Ls * nrhs at compile time (the common single-rhs
// cases), so the row offsets of every spinor load and store are immediates.
// Threads per CTA: 256, two or three CTAs per SM; the fixed-point FP64 hop, one
// CTA of 512 (128 registers and some 30 bytes of spills: 1.34 ms at 24^4 x 16,
// against 1.53 with 384 threads of 168 registers and 1.67 with 2 x 192).
template <class SL>
constexpr int kHopThreads = std::is_same<SL, FxLink>::value ? 512 : 256;

template <class Sin, class Sout, class SL, class R, int VL, bool DAG, int EPI, int CN5>
__global__ void __launch_bounds__(kHopThreads<SL>, std::is_same<SL, FxLink>::value       ? 1
                                                   : (VL == 1 && sizeof(R) == 4) ? 3
                                                                                         : 2)
k_hop(const HopArgs a) {
    constexpr bool FX = std::is_same<SL, FxLink>::value;
    extern __shared__ __align__(128) unsigned char smem[];
    const int N5 = CN5 > 0 ? CN5 : a.N5;
    const int LC = CN5 > 0 ? CN5 : a.lane_chunk;   // lanes of a site this CTA takes, from lc
    const int lc = CN5 > 0 ? 0 : (int)blockIdx.y * LC;
    const int TPS = LC / VL;
    const size_t link_bytes = (size_t)a.T * 144 * sizeof(SL);
    const size_t buf_bytes = link_bytes + (size_t)a.T * 32;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + 2 * buf_bytes);
    int* done = reinterpret_cast<int*>(bar + 2);              // [2] warps finished with a buffer
    double* s_red = reinterpret_cast<double*>(bar + 3);       // [2][nwarps][nrhs]
    const int nt = a.ntiles;
    const int nwarps = (int)(blockDim.x >> 5), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // k-th tile of this CTA: chunks of `chunk` consecutive tiles, strided by the grid
    const int ck = a.chunk;
    auto tile_of = [&](int k) { return ((k / ck) * (int)gridDim.x + (int)blockIdx.x) * ck + k % ck; };

    auto issue = [&](int tile, int b) {
        const int4 t = a.tiles[tile];
        const uint32_t lb = (uint32_t)t.z * 144u * (uint32_t)sizeof(SL);
        const uint32_t nb = (uint32_t)t.z * 32u;
        unsigned char* base = smem + b * buf_bytes;
        // order the generic-proxy reads of this buffer before the async write
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(&bar[b], lb + nb);
        bulk_g2s(base, reinterpret_cast<const SL*>(a.links) + (int64_t)t.y * 144, lb, &bar[b]);
        bulk_g2s(base + link_bytes, a.nbr + (int64_t)t.y * 8, nb, &bar[b]);
    };

    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        done[0] = done[1] = 0;
        fence_mbar_init();
        if (tile_of(0) < nt) issue(tile_of(0), 0);
        if (tile_of(1) < nt) issue(tile_of(1), 1);
    }
    __syncthreads();

    const int G = blockDim.x / TPS;
    const int sg = threadIdx.x / TPS;
    const int lane0 = lc + (threadIdx.x - sg * TPS) * VL;
    const int rhs = lane0 / a.Ls;   // of this thread's lanes (threads without sites add 0)
    const int rhs0 = lc / a.Ls, rhs1 = (lc + LC) / a.Ls;
    const bool part = (EPI == EPI_MOO || EPI == EPI_POST) && a.partial != nullptr;
    ScanCtx<VL> sk{};
    if constexpr (EPI == EPI_BMINV) {
        const int wl = threadIdx.x & 31;
        const int Ls = a.Ls;
        const int tig = lane0 / VL;
        const int gb = wl - tig;
        sk.mask = TPS >= 32 ? 0xffffffffu : (((1u << TPS) - 1u) << gb);
        sk.nthr = Ls / VL;
        sk.j = (lane0 % Ls) / VL;
        sk.seg0 = wl - sk.j;
        sk.a = (float)a.fa;
        sk.inv_d = (float)a.inv_d;
        sk.wc = (float)(a.mf * a.inv_den);
        sk.mf = (float)a.mf;
        sk.b5 = (float)a.b5;
        sk.c5 = (float)a.c5;
        float av = 1.f;
#pragma unroll
        for (int v = 0; v < VL; ++v) av *= sk.a;
#pragma unroll
        for (int l = 0; l < 5; ++l) { sk.astep[l] = av; av *= av; }
        const int s0 = lane0 % Ls;
#pragma unroll
        for (int v = 0; v < VL; ++v) {
            float pd = 1.f, pu = 1.f, cd = 1.f, cu = 1.f;
            for (int q = 0; q < s0 + v + 1; ++q) pd *= sk.a;
            for (int q = 0; q < Ls - s0 - v; ++q) pu *= sk.a;
            for (int q = 0; q < v + 1; ++q) cd *= sk.a;
            for (int q = 0; q < VL - v; ++q) cu *= sk.a;
            sk.pdn[v] = pd; sk.pup[v] = pu; sk.cdn[v] = cd; sk.cup[v] = cu;
        }
    }
    LaneNbrs nbrs{};
    if constexpr (EPI == EPI_POST || (EPI == EPI_MOO && kLaneShfl<VL, CN5>)) {
        // site groups are warp-aligned here (TPS divides 32, checked on the host)
        const int wl = threadIdx.x & 31;
        const int tig = (lane0 - lc) / VL;
        const int gb = wl - tig;
        const int s_first = lane0 % a.Ls, s_last = (lane0 + VL - 1) % a.Ls;
        const int rb = lane0 - s_first;
        const int above = s_last == a.Ls - 1 ? rb : lane0 + VL;
        const int below = s_first == 0 ? rb + a.Ls - 1 : lane0 - 1;
        nbrs.src_up = gb + (above - lc) / VL;
        nbrs.src_dn = gb + (below - lc) / VL;
        nbrs.f_up = s_last == a.Ls - 1 ? -(float)a.mf : 1.f;
        nbrs.f_dn = s_first == 0 ? -(float)a.mf : 1.f;
        nbrs.mask = TPS >= 32 ? 0xffffffffu : (((1u << TPS) - 1u) << gb);
    }

    int k = 0;
    const int2 fx_info = FX ? *reinterpret_cast<const int2*>(a.fx_info) : make_int2(0, 0);
    int turn = 0;   // a.deal: sites done so far mod G, so that the groups that take a tile's
                    // remainder change from tile to tile
    for (int tile = tile_of(0); tile < nt; tile = tile_of(++k)) {
        const int b = k & 1;
        const uint32_t ph = (uint32_t)((k >> 1) & 1);
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&bar[b], ph))) {
            // a lost copy: record it, let it land, stop
            if (lane == 0) {
                atomicOr(a.err, kErrBulkTimeout);
                mbar_wait_bounded(&bar[b], ph);
            }
            return;
        }
        const int4 tl = a.tiles[tile];
        const int begin = tl.y, count = tl.z;
        const SL* s_link_t = reinterpret_cast<const SL*>(smem + b * buf_bytes);
        const int* s_nbr_t = reinterpret_cast<const int*>(smem + b * buf_bytes + link_bytes);
        double* red = s_red + (size_t)b * nwarps * a.nrhs;
        double tile_norm = 0.0;
        int first = sg;
        if (a.deal) {
            first = sg - turn + (sg < turn ? G : 0);
            turn = (turn + count) % G;
        }
        for (int sl = first; sg < G && sl < count; sl += G) {
            // the M_oo input of this site's lanes, into L1 while the last two
            // directions run (earlier, the lines are evicted by the neighbour
            // traffic before the epilogue reads them)
            auto prefetch_moo = [&]() {
                if (EPI == EPI_MOO || EPI == EPI_POST) {
                    const Sout* xb = reinterpret_cast<const Sout*>(a.xmoo) + ((int64_t)(begin + sl) * 12 * N5 + lane0) * 2;
#pragma unroll
                    for (int c = 0; c < 12; ++c)
                        asm volatile("prefetch.global.L1 [%0];" ::"l"(xb + (int64_t)c * N5 * 2));
                }
            };
            R ar[12][VL], ai[12][VL];
            R factor = (R)1;
            const Sin* in = reinterpret_cast<const Sin*>(a.in);
            const int* nb = s_nbr_t + sl * 8;
            const SL* lk = s_link_t + (size_t)sl * 144;
            // +mu and -mu back to back: the row that is the +x neighbour of
            // one site is the -x neighbour of the next, still in L1
            if constexpr (FX) {
                factor = hop_site_fx<DAG>(in, nb, lk, a.links64 + (int64_t)(begin + sl) * 144, fx_info, N5, lane0, ar,
                                          ai);
            } else if constexpr (std::is_same<R, float>::value && VL == 2 && std::is_same<Sin, bf16>::value) {
                float2 pr[12], pi[12];
#pragma unroll
                for (int c = 0; c < 12; ++c) pr[c] = pi[c] = make_float2(0.f, 0.f);
                hop_dir2<0, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
                hop_dir2<4, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
                hop_dir2<1, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
                hop_dir2<5, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
                hop_dir2<2, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
                hop_dir2<6, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
                prefetch_moo();
                hop_dir2<3, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
                hop_dir2<7, DAG, Sin, SL>(in, nb, lk, N5, lane0, pr, pi);
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    ar[c][0] = pr[c].x; ar[c][VL - 1] = pr[c].y;
                    ai[c][0] = pi[c].x; ai[c][VL - 1] = pi[c].y;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 12; ++c)
#pragma unroll
                    for (int v = 0; v < VL; ++v) ar[c][v] = ai[c][v] = (R)0;
                hop_dir<0, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
                hop_dir<4, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
                hop_dir<1, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
                hop_dir<5, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
                hop_dir<2, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
                hop_dir<6, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
                prefetch_moo();
                hop_dir<3, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
                hop_dir<7, DAG, Sin, SL, R, VL>(in, nb, lk, N5, lane0, ar, ai);
            }
            tile_norm += hop_store<Sout, R, VL, DAG, EPI, CN5>(a, N5, begin + sl, lane0, ar, ai, factor, nbrs, tl.x, sk);
        }
        if (part) {
            for (int r = rhs0; r < rhs1; ++r) {
                double v = rhs == r ? tile_norm : 0.0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if (lane == 0) red[warp * a.nrhs + r] = v;
            }
        }
        __syncwarp();   // this warp's reads of buffer b are done
        if (lane == 0) {
            __threadfence_block();
            if (atomicAdd(&done[b], 1) == nwarps - 1) {   // the last warp out
                __threadfence_block();
                if (part)
                    for (int r = rhs0; r < rhs1; ++r) {
                        double sum = 0.0;
                        for (int w = 0; w < nwarps; ++w) sum += red[w * a.nrhs + r];
                        a.partial[(size_t)tile * a.nrhs + r] = sum;
                    }
                done[b] = 0;
                const int next2 = tile_of(k + 2);
                if (next2 < nt) issue(next2, b);
            }
        }
    }
}

// The fixed-point FP64 hop on a domain too small to fill the chip: there a
// lane's chain of eight directions, ~20 us, is the whole time.  Warp k of a CTA
// takes direction k of 32 lanes of its tile, and warps 0..5 add the eight
// directions' half spinors from shared memory, two spin-colour rows each, in
// the largest of the eight units.  4^4 x 8 (1024 lanes): 20.5 us -> 7.9 with
// the call's launch.  Lanes that need the FP64 form take it the same way, a
// direction a warp, its sums in hop_fx_fallback's order.
constexpr int kSplitLanes = 32;

// transported half spinor of direction k in FP64, into g[(q * 3 + colour) * 2 + part][lane]
template <bool DAG>
__device__ __noinline__ void hop_fx_dir64(int k, const double* in, const int* nb, const double* lk, int N5, int lane0,
                                          long long* g) {
    double ar[12][1], ai[12][1];
#pragma unroll
    for (int c = 0; c < 12; ++c) ar[c][0] = ai[c][0] = 0.0;
    switch (k) {
        case 0: hop_dir<0, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai); break;
        case 1: hop_dir<1, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai); break;
        case 2: hop_dir<2, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai); break;
        case 3: hop_dir<3, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai); break;
        case 4: hop_dir<4, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai); break;
        case 5: hop_dir<5, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai); break;
        case 6: hop_dir<6, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai); break;
        default: hop_dir<7, DAG, double, double, double, 1>(in, nb, lk, N5, lane0, ar, ai);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        g[(2 * c) * kSplitLanes] = __double_as_longlong(ar[c][0]);
        g[(2 * c + 1) * kSplitLanes] = __double_as_longlong(ai[c][0]);
    }
}

template <bool DAG, int EPI>
__global__ void __launch_bounds__(256, 2) k_hop_fx_split(const HopArgs a) {
    __shared__ long long s_g[8][12][kSplitLanes];   // [direction][(q * 3 + colour) * 2 + part][lane]
    __shared__ int s_E[8][kSplitLanes];             // unit, 0: nothing, -1: the FP64 form decides
    __shared__ double s_red[256];
    __shared__ double s_sum[kMaxLanes / 2];
    __shared__ unsigned s_fp64;                     // lanes that the FP64 form decides
    const int N5 = a.N5, Ls = a.Ls, nrhs = a.nrhs;
    const int4 tl = a.tiles[blockIdx.x];
    const int items = tl.z * N5;
    const int k = threadIdx.x >> 5, j = threadIdx.x & 31;
    const int2 info = *reinterpret_cast<const int2*>(a.fx_info);
    const double* in = reinterpret_cast<const double*>(a.in);
    const bool part = EPI == EPI_MOO && a.partial != nullptr;
    if (part)
        for (int r = threadIdx.x; r < nrhs; r += blockDim.x) s_sum[r] = 0.0;
    for (int g0 = 0; g0 < items; g0 += kSplitLanes) {
        const bool on = g0 + j < items;
        const int item = on ? g0 + j : 0;
        const int64_t site = tl.y + item / N5;
        const int lane0 = item % N5;
        const int nb = on ? a.nbr[site * 8 + k] : -1;
        int E = 0;
        if (nb >= 0) {
            const double2* src = reinterpret_cast<const double2*>(in) + ((int64_t)nb * 12 * N5 + lane0);
            double2 x[12];
#pragma unroll
            for (int c = 0; c < 12; ++c) x[c] = __ldg(src + (int64_t)c * N5);
            bool bad = false;
            const uint32_t top = fx_top(x, bad);
            if (bad) E = -1;
            if (top != 0) {
                E = (int)(top >> 20) + 1;
                const int P = ((k < 4) != DAG) ? 0 : -1;
                FxHalf h;
                switch (k & 3) {   // the same for the whole warp
                    case 0: fx_project<0>(x, P, E, h); break;
                    case 1: fx_project<1>(x, P, E, h); break;
                    case 2: fx_project<2>(x, P, E, h); break;
                    default: fx_project<3>(x, P, E, h);
                }
                const int4* w = reinterpret_cast<const int4*>(a.links) + (site * 8 + k) * 9;
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const int4 v[3] = {__ldg(w + r * 3), __ldg(w + r * 3 + 1), __ldg(w + r * 3 + 2)};
                    long long gr[2], gi[2];
                    fx_row(v, h, gr, gi);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        s_g[k][(q * 3 + r) * 2][j] = gr[q];
                        s_g[k][(q * 3 + r) * 2 + 1][j] = gi[q];
                    }
                }
            }
        }
        s_E[k][j] = E;
        if (threadIdx.x == 0) s_fp64 = 0;
        __syncthreads();
        double nrm = 0.0, re[2] = {0.0, 0.0}, im[2] = {0.0, 0.0}, factor = 1.0;
        const bool upper = k < 3;   // rows 2 k, 2 k + 1: upper spins for k < 3
        bool fp64 = false;
        if (k < 6 && on) {
            int Em = 0;
            bool bad = false;
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                Em = max(Em, s_E[d][j]);
                bad |= s_E[d][j] < 0;
            }
            fp64 = ((Em != 0 || bad) && (Em < 128 || Em > 1080)) || info.y == 0;
            if (!fp64) {
                long long sr[2] = {0, 0}, si[2] = {0, 0};
                int size[2] = {0, 0};       // each row's own sum of |g| decides here
#pragma unroll
                for (int d = 0; d < 8; ++d) {
                    const int Ek = s_E[d][j];
                    if (Ek <= 0) continue;
                    const int dn = min(Em - Ek, 63);
                    const int P = ((d < 4) != DAG) ? 0 : -1, mu = d & 3;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int c = 2 * k + e, spin = c / 3, col = c - 3 * spin;
                        const int q = upper ? spin : (mu < 2 ? 3 - spin : spin - 2);
                        const long long gr = s_g[d][(q * 3 + col) * 2][j] >> dn, gi = s_g[d][(q * 3 + col) * 2 + 1][j] >> dn;
                        size[e] += fx_size(gr, gi);
                        if (upper) {
                            sr[e] += gr;
                            si[e] += gi;
                        } else {
                            const int f = fx_plus(mu, q) ? P : ~P;   // sign mask of the term (of its im part for i types)
                            if (fx_itype(mu)) { fx_add(sr[e], gi, ~f); fx_add(si[e], gr, f); }
                            else { fx_add(sr[e], gr, f); fx_add(si[e], gi, f); }
                        }
                    }
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) { re[e] = __ll2double_rn(sr[e]); im[e] = __ll2double_rn(si[e]); }
                factor = __hiloint2double(max(Em + info.x - 54, 1) << 20, 0);
                fp64 = Em != 0 && min(size[0], size[1]) < kFxCover;
            }
            if (fp64) atomicOr(&s_fp64, 1u << j);
        }
        if (__syncthreads_or(fp64)) {   // (the sums above are done with s_g)
            const bool redo = (s_fp64 >> j) & 1;
            if (redo)
                hop_fx_dir64<DAG>(k, in, a.nbr + site * 8, a.links64 + site * 144, N5, lane0, &s_g[k][0][j]);
            __syncthreads();
            if (redo && k < 6) {
                factor = 1.0;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int c = 2 * k + e, spin = c / 3, col = c - 3 * spin;
                    re[e] = im[e] = 0.0;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int d = (i >> 1) + 4 * (i & 1), mu = d & 3;
                        const int q = upper ? spin : (mu < 2 ? 3 - spin : spin - 2);
                        const double gr = __longlong_as_double(s_g[d][(q * 3 + col) * 2][j]);
                        const double gi = __longlong_as_double(s_g[d][(q * 3 + col) * 2 + 1][j]);
                        const bool minus = fx_plus(mu, q) == ((d < 4) == DAG);   // sign of the term (of its im part for i types)
                        if (upper) { re[e] += gr; im[e] += gi; }
                        else if (fx_itype(mu)) { re[e] += minus ? gi : -gi; im[e] += minus ? -gr : gr; }
                        else { re[e] += minus ? -gr : gr; im[e] += minus ? -gi : gi; }
                    }
                }
            }
        }
        if (k < 6 && on) {
            const double sc = a.scale * factor;
            const int s = lane0 % Ls;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int c = 2 * k + e;
                const int64_t row = (site * 12 + c) * N5;
                double yr = sc * re[e], yi = sc * im[e];
                if (EPI == EPI_MOO) {
                    const double2* x = reinterpret_cast<const double2*>(a.xmoo) + row;
                    const bool below = (c < 6) != DAG;   // S_- (lane s - 1), else S_+
                    const bool wrap = below ? s == 0 : s == Ls - 1;
                    const int ln = below ? (wrap ? lane0 + Ls - 1 : lane0 - 1) : (wrap ? lane0 - (Ls - 1) : lane0 + 1);
                    const double e5 = wrap ? -a.mf * a.e : a.e;
                    const double2 xo = x[lane0], xn = x[ln];
                    yr = fma(sc, re[e], fma(e5, xn.x, a.d * xo.x));
                    yi = fma(sc, im[e], fma(e5, xn.y, a.d * xo.y));
                    if (part) nrm = fma(yr, yr, fma(yi, yi, nrm));
                }
                reinterpret_cast<double2*>(a.out)[row + lane0] = make_double2(yr, yi);
            }
        }
        if (part) {
            // per right-hand side, added in thread order: lanes change theirs from pass to pass
            s_red[threadIdx.x] = nrm;
            __syncthreads();
            for (int r = k; r < nrhs; r += 8) {
                double v = 0.0;
                for (int t = j; t < 6 * 32; t += 32)
                    if (on && lane0 / Ls == r) v += s_red[t];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if (j == 0) s_sum[r] += v;
            }
        }
        __syncthreads();   // s_g, s_E, s_red are reused
    }
    if (part)
        for (int r = threadIdx.x; r < nrhs; r += blockDim.x) a.partial[(size_t)blockIdx.x * nrhs + r] = s_sum[r];
}

// ------------------------------------------------------------- launcher
static HopArgs hop_args(dwf_handle* h, const HopCall& c, const TileSet& ts, bool FX) {
    const int p = c.out_parity;
    HopArgs a{};
    a.in = c.in;
    a.out = c.out;
    a.xmoo = c.xmoo;
    a.links = FX ? h->d_links_fx[p] : h->d_links[c.prec_link][p];
    a.links64 = static_cast<const double*>(h->d_links[DWF_FP64][p]);
    a.fx_info = h->d_fx_info;
    a.nbr = h->d_nbr[p];
    a.tiles = ts.d_tiles[p];
    a.T = ts.T;
    a.Ls = h->p.Ls;
    a.nrhs = c.nrhs;
    a.N5 = h->p.Ls * c.nrhs;
    a.scale = c.scale;
    a.d = h->f5[0].d;
    a.e = h->f5[0].e;
    a.mf = h->p.mf;
    a.partial = c.partial;
    a.err = h->d_err;
    a.chunk = c.chunk > 0 ? c.chunk : 1;
    a.b5 = h->p.b5;
    a.c5 = h->p.c5;
    a.fa = h->f5[0].a;
    a.inv_d = h->f5[0].inv_d;
    a.inv_den = h->f5[0].inv_den;
    a.cg_x = c.cg_x;
    a.cg_r = c.cg_r;
    a.cg_p = c.cg_p;
    a.alpha = c.alpha;
    a.run = c.run;
    a.ntiles = ts.ntiles[p];
    return a;
}

// Lanes of a site that a CTA takes: all of them, or, with many right-hand
// sides, whole right-hand sides of at most 32 lanes whose threads divide a
// warp (the chunks side by side in the grid), so that a CTA's pass covers a
// row of neighbouring sites that it finds in L1 again; with 256 lanes a pass is
// two sites, 24 KB a row.  Bare hop, whole / chunked, Ls = 16: FP32 12^4 with 16
// right-hand sides 302 / 160 us, 16^4 with 8 305 / 262, 12^4 with 3 49.3 / 45.5;
// 8^4 with 16 (0.5 M lanes) 35.8 / 37.9, so not on small domains; FP64 12^4 with
// 16 1851 / 1406, but with 16-lane chunks 2260; BF16 12^4 with 16 217 / 158, with
// 3 46.2 / 42.8, but 16^4 with 8 232 / 240 (its 128 lanes are 512 bytes).
static int lane_chunk(int Ls, int nrhs, int VL, dwf_prec link, int64_t nsite) {
    const int N5 = Ls * nrhs;
    if (N5 <= 32 || nsite * N5 < (link == DWF_FP64 ? 0 : 1 << 20)) return N5;
    if (link == DWF_BF16 && N5 > 64 && N5 <= 128) return N5;
    for (int k = 32 / Ls; k >= 1; --k)
        if (nrhs % k == 0 && 32 % (k * Ls / VL) == 0 && (link != DWF_FP64 || k * Ls == 32)) return k * Ls;
    return N5;
}

template <class Sin, class Sout, class SL, class R, int VL, int CN5 = 0>
static dwf_status launch_t(dwf_handle* h, const HopCall& c, const TileSet& ts, cudaStream_t s) {
    constexpr bool FX = std::is_same<SL, FxLink>::value;
    HopArgs a = hop_args(h, c, ts, FX);
    a.lane_chunk = CN5 > 0 || c.post || c.bminv ? a.N5 : lane_chunk(h->p.Ls, c.nrhs, VL, c.prec_link, h->nsite[c.out_parity]);
    const int TPS = a.lane_chunk / VL;
    // site groups per CTA: as many as fit in its threads, at most T.  Fixed-point
    // hop, where T groups are fewer than 384 threads and a CTA gets several
    // tiles: as many as the two buffered tiles hold (T / 2 T groups: 16^4 x 10
    // 223 / 198 us, 16^4 x 6 134 / 122; but 16^4 x 12, 384 threads, 211 / 228, and
    // with two tiles per CTA 10^4 x 16 59 / 65, 10^4 x 12 53 / 56).
    // Where they do not divide T, sites are dealt out in turn across tiles: at
    // 16^4 x 12 with 3 right-hand sides 95.7 -> 87.0 us.  (More groups than T in
    // FP32 lost 1 to 6% at 16^4 x 10 and 16^4 x 12.)
    int groups = kHopThreads<SL> / TPS;
    const int most = FX && a.ntiles > 4 * 152 && ts.T * TPS < 384 ? 2 * ts.T : ts.T;
    if (groups > most) groups = most;
    if (groups < 1) {
        set_error("hop: %d threads per site exceed %d", TPS, kHopThreads<SL>);
        return DWF_ERR_ARG;
    }
    a.deal = ts.T % groups != 0;
    int threads = (groups * TPS + 31) / 32 * 32;
    const size_t smem = hop_smem(ts.T, sizeof(SL), threads / 32, c.nrhs);
    const int nt = a.ntiles;
    if (nt == 0) return DWF_OK;
    void (*kern)(const HopArgs);
    const bool moo = c.xmoo != nullptr;
    if (c.post) {
        if constexpr (std::is_same<R, float>::value && std::is_same<Sout, float>::value) {
            if (!c.dagger || !moo || 32 % TPS != 0 || c.cg_x == nullptr || c.cg_r == nullptr ||
                c.cg_p == nullptr || c.alpha == nullptr) {
                set_error("hop: fused M_pc^+ tail needs the adjoint, t, the CG vectors and "
                          "site groups that divide a warp");
                return DWF_ERR_ARG;
            }
            kern = k_hop<Sin, Sout, SL, R, VL, true, EPI_POST, CN5>;
        } else {
            set_error("hop: fused M_pc^+ tail needs FP32 arithmetic and FP32 vectors");
            return DWF_ERR_UNSUPPORTED;
        }
    } else if (c.bminv) {
        if constexpr (std::is_same<R, float>::value) {
            if (moo || 32 % TPS != 0) {
                set_error("hop: fused B M_ee^-1 needs site groups that divide a warp");
                return DWF_ERR_ARG;
            }
            kern = c.dagger ? k_hop<Sin, Sout, SL, R, VL, true, EPI_BMINV, CN5>
                            : k_hop<Sin, Sout, SL, R, VL, false, EPI_BMINV, CN5>;
        } else {
            set_error("hop: fused B M_ee^-1 needs FP32 arithmetic");
            return DWF_ERR_UNSUPPORTED;
        }
    } else if (c.dagger)
        kern = moo ? k_hop<Sin, Sout, SL, R, VL, true, EPI_MOO, CN5>
                   : k_hop<Sin, Sout, SL, R, VL, true, EPI_PLAIN, CN5>;
    else
        kern = moo ? k_hop<Sin, Sout, SL, R, VL, false, EPI_MOO, CN5>
                   : k_hop<Sin, Sout, SL, R, VL, false, EPI_PLAIN, CN5>;
    if (smem > (FX ? kHopMaxSmemFx : kHopMaxSmem)) {
        set_error("hop: tile of %d sites needs %zu bytes of shared memory", ts.T, smem);
        return DWF_ERR_ARG;
    }
    // persistent grid: as many CTAs as are resident at once, at most one per tile
    int grid = 0;
    const int chunks = a.N5 / a.lane_chunk;
    DWF_TRY(persistent_grid((const void*)kern, threads, smem, nt * chunks, &grid));
    kern<<<dim3((grid + chunks - 1) / chunks, chunks), threads, smem, s>>>(a);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

// One CTA of k_hop_fx_split per tile, up to 128 lanes per SM: 8^4 x 8 (16384
// lanes) takes 18.2 us split against 25.9, 8^4 x 16 (32768) 32.7 against 26.9.
static bool fx_split_ok(const dwf_handle* h, const HopCall& c) {
    return h->nsite[c.out_parity] * h->p.Ls * c.nrhs <= 152 * 128;
}

static dwf_status launch_fx_split(dwf_handle* h, const HopCall& c, const TileSet& ts, cudaStream_t s) {
    const HopArgs a = hop_args(h, c, ts, true);
    if (a.ntiles == 0) return DWF_OK;
    void (*kern)(const HopArgs) = c.xmoo != nullptr ? (c.dagger ? k_hop_fx_split<true, EPI_MOO> : k_hop_fx_split<false, EPI_MOO>)
                                                    : (c.dagger ? k_hop_fx_split<true, EPI_PLAIN> : k_hop_fx_split<false, EPI_PLAIN>);
    kern<<<a.ntiles, 256, 0, s>>>(a);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

// FP32-arithmetic hop: two lanes per thread unless the call asks for one
// (FP32 links only).
template <class Sin, class Sout, class SL>
static dwf_status launch_f32(dwf_handle* h, const HopCall& c, const TileSet& ts, cudaStream_t s) {
    const int N5 = h->p.Ls * c.nrhs;
    if constexpr (std::is_same<SL, float>::value) {
        if (c.VL == 1) {
            if (N5 == 12) return launch_t<Sin, Sout, SL, float, 1, 12>(h, c, ts, s);
            if (N5 == 16) return launch_t<Sin, Sout, SL, float, 1, 16>(h, c, ts, s);
            return launch_t<Sin, Sout, SL, float, 1>(h, c, ts, s);
        }
    }
    constexpr bool spec = (std::is_same<SL, float>::value && std::is_same<Sin, float>::value &&
                           std::is_same<Sout, float>::value) ||
                          (std::is_same<Sin, bf16>::value && std::is_same<Sout, bf16>::value);
    if constexpr (spec) {
        if (N5 == 12) return launch_t<Sin, Sout, SL, float, 2, 12>(h, c, ts, s);
        if (N5 == 16) return launch_t<Sin, Sout, SL, float, 2, 16>(h, c, ts, s);
    }
    return launch_t<Sin, Sout, SL, float, 2>(h, c, ts, s);
}

// Raise the dynamic shared-memory limit of every hop instantiation once, so
// that launches recorded into a CUDA graph never need a host-side call.
template <class Sin, class Sout, class SL, class R, int VL, int CN5 = 0>
static cudaError_t hop_attr() {
    cudaError_t e = cudaSuccess;
    void (*k[4])(const HopArgs) = {k_hop<Sin, Sout, SL, R, VL, false, EPI_PLAIN, CN5>,
                                   k_hop<Sin, Sout, SL, R, VL, false, EPI_MOO, CN5>,
                                   k_hop<Sin, Sout, SL, R, VL, true, EPI_PLAIN, CN5>,
                                   k_hop<Sin, Sout, SL, R, VL, true, EPI_MOO, CN5>};
    for (auto f : k) {
        cudaError_t r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             std::is_same<SL, FxLink>::value ? kHopMaxSmemFx : kHopMaxSmem);
        if (r != cudaSuccess) e = r;
    }
    if constexpr (std::is_same<R, float>::value && std::is_same<Sout, float>::value) {
        cudaError_t r = cudaFuncSetAttribute(k_hop<Sin, Sout, SL, R, VL, true, EPI_POST, CN5>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kHopMaxSmem);
        if (r != cudaSuccess) e = r;
    }
    if constexpr (std::is_same<R, float>::value) {
        cudaError_t r = cudaFuncSetAttribute(k_hop<Sin, Sout, SL, R, VL, false, EPI_BMINV, CN5>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kHopMaxSmem);
        if (r != cudaSuccess) e = r;
        r = cudaFuncSetAttribute(k_hop<Sin, Sout, SL, R, VL, true, EPI_BMINV, CN5>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kHopMaxSmem);
        if (r != cudaSuccess) e = r;
    }
    return e;
}

dwf_status init_hop_kernels() {
    DWF_CUDA((hop_attr<double, double, double, double, 1>()));
    DWF_CUDA((hop_attr<double, double, FxLink, double, 1>()));
    DWF_CUDA((hop_attr<double, double, FxLink, double, 1, 12>()));
    DWF_CUDA((hop_attr<double, double, FxLink, double, 1, 16>()));
    DWF_CUDA((hop_attr<float, float, float, float, 2>()));
    DWF_CUDA((hop_attr<float, float, float, float, 1>()));
    DWF_CUDA((hop_attr<bf16, bf16, bf16, float, 2>()));
    DWF_CUDA((hop_attr<bf16, float, bf16, float, 2>()));
    DWF_CUDA((hop_attr<float, bf16, bf16, float, 2>()));
    DWF_CUDA((hop_attr<float, float, bf16, float, 2>()));
    DWF_CUDA((hop_attr<float, float, float, float, 2, 12>()));
    DWF_CUDA((hop_attr<float, float, float, float, 2, 16>()));
    DWF_CUDA((hop_attr<float, float, float, float, 1, 12>()));
    DWF_CUDA((hop_attr<float, float, float, float, 1, 16>()));
    DWF_CUDA((hop_attr<bf16, bf16, bf16, float, 2, 12>()));
    DWF_CUDA((hop_attr<bf16, bf16, bf16, float, 2, 16>()));
    return DWF_OK;
}

bool hop_post_ok(const dwf_handle* h, dwf_prec op, dwf_prec vec, int nrhs, int VL) {
    if (vec != DWF_FP32 || (op != DWF_FP32 && op != DWF_BF16)) return false;
    const int n5 = h->p.Ls * nrhs;
    const int vl = op == DWF_BF16 ? 2 : (VL == 1 ? 1 : 2);
    const int tps = n5 / vl;
    return n5 % vl == 0 && tps <= 32 && 32 % tps == 0;
}

bool hop_bminv_ok(const dwf_handle* h, dwf_prec op, int nrhs, int VL) {
    if (op != DWF_FP32 && op != DWF_BF16) return false;
    if (std::abs(h->f5[0].a) > 1.0) return false;   // the epilogue's scan grows like |a|^Ls
    const int n5 = h->p.Ls * nrhs;
    const int vl = op == DWF_BF16 ? 2 : (VL == 1 ? 1 : 2);
    const int tps = n5 / vl;
    return n5 % vl == 0 && tps <= 32 && 32 % tps == 0;
}

dwf_status launch_hop(dwf_handle* h, const HopCall& c, cudaStream_t s) {
    const TileSet* tsp = nullptr;
    DWF_TRY(get_tiles(h, tile_or_default(c.T), &tsp));
    const TileSet& ts = *tsp;
    if (c.prec_link == DWF_FP64) {
        if (c.prec_in != DWF_FP64 || c.prec_out != DWF_FP64) return DWF_ERR_UNSUPPORTED;
        if (h->fx_links && !c.post && !c.bminv) {
            if (fx_split_ok(h, c)) return launch_fx_split(h, c, ts, s);
            const int N5 = h->p.Ls * c.nrhs;
            if (N5 == 12) return launch_t<double, double, FxLink, double, 1, 12>(h, c, ts, s);
            if (N5 == 16) return launch_t<double, double, FxLink, double, 1, 16>(h, c, ts, s);
            return launch_t<double, double, FxLink, double, 1>(h, c, ts, s);
        }
        return launch_t<double, double, double, double, 1>(h, c, ts, s);
    }
    if (c.prec_link == DWF_FP32) {
        if (c.prec_in != DWF_FP32 || c.prec_out != DWF_FP32) return DWF_ERR_UNSUPPORTED;
        return launch_f32<float, float, float>(h, c, ts, s);
    }
    // BF16 links: FP32 arithmetic, operands FP32 or BF16
    if (c.tc) return launch_hop_tc(h, c, ts, s);
    if (c.prec_in == DWF_BF16 && c.prec_out == DWF_BF16) return launch_f32<bf16, bf16, bf16>(h, c, ts, s);
    if (c.prec_in == DWF_BF16 && c.prec_out == DWF_FP32) return launch_f32<bf16, float, bf16>(h, c, ts, s);
    if (c.prec_in == DWF_FP32 && c.prec_out == DWF_BF16) return launch_f32<float, bf16, bf16>(h, c, ts, s);
    if (c.prec_in == DWF_FP32 && c.prec_out == DWF_FP32) return launch_f32<float, float, bf16>(h, c, ts, s);
    return DWF_ERR_UNSUPPORTED;
}

}  // namespace dwf
