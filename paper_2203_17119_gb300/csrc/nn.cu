// Gauge-covariant parallel-transport convolutional preconditioner K: forward,
// backward and Adam kernels (FP32 arithmetic, BF16 weights for the forward
// pass, FP32 master weights for training).
//
//   T_0 = 1;  T_{1+mu} f(x) = U_mu(x) f(x+mu);  T_{5+mu} f(x) = U_mu(x-mu)^+ f(x-mu);
//   T_9 f(x,s) = f(x,s+1), T_10 f(x,s) = f(x,s-1)  (zero outside [0, Ls));
//   layer 1 (1 -> C):  R_d = T_d r,            phi^a = sum_d W1[a][d] R_d
//   layer 2 (C -> 1):  psi_d = sum_b W2[d][b] phi^b,   z = sum_d T_d psi_d
//
// W[o][i] are complex 4x4 spin matrices (they commute with colour and with
// the transports, so the order of mixing and transport within a layer is
// free).  K acts on the odd checkerboard: the input is embedded with zero on
// even sites and the output is read on odd sites.  Backward: g_psi_d =
// T_d^+ g_z, gW2[d][b] = sum g_psi_d phi_b^+, g_phi_b = sum_d W2[d][b]^+ g_psi_d,
// gW1[a][d] = sum g_phi_a R_d^+ (sums over sites, colour and lanes).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <vector>

#include "dev_common.cuh"
#include "dwf_internal.cuh"

namespace dwf {

constexpr int kNDir = 11;
constexpr int kAdj[kNDir] = {0, 5, 6, 7, 8, 1, 2, 3, 4, 10, 9};

struct TransArgs {
    const float* same;         // parity-p block of the input (field 0)
    const float* opp;          // parity-(1-p) block of the input (field 0)
    float* out;                // parity-p block of the output (field 0)
    const float* links;        // FP32 doubled link table of parity p
    const int* nbr;
    const int4* tiles;
    int dirs[kNDir];           // direction of output (multi) or input (sum) field j
    int ndir, N5, Ls;
    int64_t istride, ostride;  // floats between consecutive input (sum) / output (multi) fields
};

// f = U v (3x3 complex times colour vector) for 4 spins
__device__ __forceinline__ void su3_spinor(const float* __restrict__ w, const float (&vr)[12],
                                           const float (&vi)[12], float (&orr)[12], float (&oi)[12]) {
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float sr = 0.f, si = 0.f;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const float wr = w[2 * (a * 3 + b)], wi = w[2 * (a * 3 + b) + 1];
                sr = fmaf(wr, vr[sp * 3 + b], sr);
                sr = fmaf(-wi, vi[sp * 3 + b], sr);
                si = fmaf(wr, vi[sp * 3 + b], si);
                si = fmaf(wi, vr[sp * 3 + b], si);
            }
            orr[sp * 3 + a] = sr;
            oi[sp * 3 + a] = si;
        }
}

// Value of T_d f at (site, lane) of parity p: 12 complex; same / opp are f's
// blocks of parity p and 1 - p (the link directions read only the latter, the
// others only the former).
__device__ __forceinline__ void transport_at(const TransArgs& a, const float* __restrict__ same,
                                             const float* __restrict__ opp, int d, int64_t site, int lane,
                                             float (&orr)[12], float (&oi)[12]) {
    const int N5 = a.N5;
    if (d == 0 || d == 9 || d == 10) {
        int l = lane;
        if (d != 0) {
            const int s = lane % a.Ls;
            if ((d == 9 && s == a.Ls - 1) || (d == 10 && s == 0)) {
#pragma unroll
                for (int c = 0; c < 12; ++c) orr[c] = oi[c] = 0.f;
                return;
            }
            l = d == 9 ? lane + 1 : lane - 1;
        }
        const float* p = same + (site * 12 * N5 + l) * 2;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const float2 v = *reinterpret_cast<const float2*>(p + (int64_t)c * N5 * 2);
            orr[c] = v.x;
            oi[c] = v.y;
        }
        return;
    }
    const int k = d <= 4 ? d - 1 : d - 5 + 4;     // neighbour / link slot
    const int n = a.nbr[site * 8 + k];
    if (n < 0) {
#pragma unroll
        for (int c = 0; c < 12; ++c) orr[c] = oi[c] = 0.f;
        return;
    }
    float vr[12], vi[12];
    const float* p = opp + ((int64_t)n * 12 * N5 + lane) * 2;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const float2 v = *reinterpret_cast<const float2*>(p + (int64_t)c * N5 * 2);
        vr[c] = v.x;
        vi[c] = v.y;
    }
    su3_spinor(a.links + (site * 8 + k) * 18, vr, vi, orr, oi);
}

// out field j = T_{dirs[j]} in on the sites of parity p (one thread per site x lane)
__global__ void __launch_bounds__(256) k_transport_multi(const TransArgs a) {
    const int4 tl = a.tiles[blockIdx.x];
    const int N5 = a.N5;
    for (int t = threadIdx.x; t < tl.z * N5; t += blockDim.x) {
        const int64_t site = tl.y + t / N5;
        const int lane = t % N5;
        for (int j = 0; j < a.ndir; ++j) {
            float orr[12], oi[12];
            transport_at(a, a.same, a.opp, a.dirs[j], site, lane, orr, oi);
            float* o = a.out + j * a.ostride + (site * 12 * N5 + lane) * 2;
#pragma unroll
            for (int c = 0; c < 12; ++c)
                *reinterpret_cast<float2*>(o + (int64_t)c * N5 * 2) = make_float2(orr[c], oi[c]);
        }
    }
}

// out = sum_j T_{dirs[j]} in_j on the odd sites; in_j is input field j of the
// block that direction reads (odd for 0, 9, 10, even for the links), counted
// from 0 within each block
__global__ void __launch_bounds__(256) k_transport_sum(const TransArgs a) {
    const int4 tl = a.tiles[blockIdx.x];
    const int N5 = a.N5;
    for (int t = threadIdx.x; t < tl.z * N5; t += blockDim.x) {
        const int64_t site = tl.y + t / N5;
        const int lane = t % N5;
        float ar[12], ai[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) ar[c] = ai[c] = 0.f;
        int js = 0, jo = 0;
        for (int j = 0; j < a.ndir; ++j) {
            float orr[12], oi[12];
            const int d = a.dirs[j];
            const bool link = d >= 1 && d <= 8;
            const int64_t f = (link ? jo++ : js++) * a.istride;
            transport_at(a, a.same + f, a.opp + f, d, site, lane, orr, oi);
#pragma unroll
            for (int c = 0; c < 12; ++c) { ar[c] += orr[c]; ai[c] += oi[c]; }
        }
        float* o = a.out + (site * 12 * N5 + lane) * 2;
#pragma unroll
        for (int c = 0; c < 12; ++c)
            *reinterpret_cast<float2*>(o + (int64_t)c * N5 * 2) = make_float2(ar[c], ai[c]);
    }
}

// Pointwise mixing: out[o][so] = sum_{i,si} W[o][so][i][si] in[i][si] at every
// pixel (site, colour, lane) of one parity.  W: [nout][4][nin][4] complex
// (FP32 in shared memory).  One thread per pixel, NOUT * 4 accumulators.
//
// GATHER: the input channels are the link transports R_d = T_d x of the
// inference, d = 1..8 (channel i: neighbour slot i), formed here from the odd
// field x by the thread that needs them (the three colour threads of a site
// and lane share the neighbour's rows through L1): R is never stored.
//
// Bound: the FP32 pipe, reached to 62% (8 x 8 channels at 24^4 x 16: 1.41 ms).
// Two pixels per thread on paired multiply-adds, with the weights doubled in
// shared memory, took 3.25 ms: 250 registers, and the shared loads then bound.
struct MixArgs {
    const float* in;           // input block (GATHER: the odd field)
    float* out;                // output block
    const float* W;
    int nin, N5;
    int64_t npix, fstride;
    const float* links;        // GATHER: FP32 link table and neighbours of this parity
    const int* nbr;
};

template <int NOUT, bool GATHER>
__global__ void __launch_bounds__(128) k_mix(const MixArgs a) {
    extern __shared__ float sW[];
    const int nin = a.nin, N5 = a.N5;
    const int nw = NOUT * 4 * nin * 4 * 2;
    for (int i = threadIdx.x; i < nw; i += blockDim.x) sW[i] = a.W[i];
    __syncthreads();
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.npix; p += (int64_t)gridDim.x * blockDim.x) {
        const int lane = (int)(p % N5);
        const int64_t sc = p / N5;              // site * 3 + colour
        const int colour = (int)(sc % 3);
        const int64_t site = sc / 3;
        const int64_t base = (site * 12 + colour) * N5 + lane;   // complex index of spin 0
        float accr[NOUT][4], acci[NOUT][4];
#pragma unroll
        for (int o = 0; o < NOUT; ++o)
#pragma unroll
            for (int so = 0; so < 4; ++so) accr[o][so] = acci[o][so] = 0.f;
        for (int i = 0; i < nin; ++i) {
            float xr[4], xi[4];
            if (GATHER) {
                const int n = a.nbr[site * 8 + i];
                if (n < 0) continue;            // a cut link carries nothing
                const float2* v = reinterpret_cast<const float2*>(a.in) + (int64_t)n * 12 * N5 + lane;
                const float2* u = reinterpret_cast<const float2*>(a.links) + (site * 8 + i) * 9 + colour * 3;
#pragma unroll
                for (int si = 0; si < 4; ++si) xr[si] = xi[si] = 0.f;
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const float2 w = __ldg(u + b);
#pragma unroll
                    for (int si = 0; si < 4; ++si) {
                        const float2 y = __ldg(v + (int64_t)(si * 3 + b) * N5);
                        xr[si] = fmaf(w.x, y.x, fmaf(-w.y, y.y, xr[si]));
                        xi[si] = fmaf(w.x, y.y, fmaf(w.y, y.x, xi[si]));
                    }
                }
            } else {
#pragma unroll
                for (int si = 0; si < 4; ++si) {
                    const float2 v = *reinterpret_cast<const float2*>(a.in + i * a.fstride +
                                                                      2 * (base + (int64_t)si * 3 * N5));
                    xr[si] = v.x;
                    xi[si] = v.y;
                }
            }
#pragma unroll
            for (int o = 0; o < NOUT; ++o)
#pragma unroll
                for (int so = 0; so < 4; ++so) {
                    const float* w = sW + 2 * (((o * 4 + so) * nin + i) * 4);
#pragma unroll
                    for (int si = 0; si < 4; ++si) {
                        const float wr = w[2 * si], wi = w[2 * si + 1];
                        accr[o][so] = fmaf(wr, xr[si], fmaf(-wi, xi[si], accr[o][so]));
                        acci[o][so] = fmaf(wr, xi[si], fmaf(wi, xr[si], acci[o][so]));
                    }
                }
        }
#pragma unroll
        for (int o = 0; o < NOUT; ++o)
#pragma unroll
            for (int so = 0; so < 4; ++so)
                *reinterpret_cast<float2*>(a.out + o * a.fstride + 2 * (base + (int64_t)so * 3 * N5)) =
                    make_float2(accr[o][so], acci[o][so]);
    }
}

// Inference on odd sites: z = sum_{d=1..8} T_d psi_d (psi on even sites) plus
// the directions 0, 9, 10, which stay on the site and couple five lanes s:
//   z(s) += N0(s) x(s) + N1 x(s+1) + N2 x(s-1) + N3 x(s+2) + N4 x(s-2),
// zero beyond [0, Ls), 4x4 spin matrices summed from W2 W1 (k_mix_weights; N0
// loses a term at each wall: variant (s < Ls - 1) + 2 (s > 0)).  One thread
// per (site, lane).
struct OddArgs {
    const float* x;            // odd field
    const float* psi;          // even block, field j = direction j + 1
    float* z;
    const float* nmat;         // [8][4][4] complex: N0 variants 0..3, N1..N4
    const float* links;
    const int* nbr;
    const int4* tiles;
    int N5, Ls;
    int64_t fstride;
};

__global__ void __launch_bounds__(256) k_odd_sum(const OddArgs a) {
    __shared__ float2 sN[8 * 16];
    for (int e = threadIdx.x; e < 8 * 16; e += blockDim.x) sN[e] = reinterpret_cast<const float2*>(a.nmat)[e];
    __syncthreads();
    const int4 tl = a.tiles[blockIdx.x];
    const int N5 = a.N5, Ls = a.Ls;
    for (int t = threadIdx.x; t < tl.z * N5; t += blockDim.x) {
        const int64_t site = tl.y + t / N5;
        const int lane = t % N5, s = lane % Ls;
        float ar[12], ai[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) ar[c] = ai[c] = 0.f;
        const float2* xs = reinterpret_cast<const float2*>(a.x) + site * 12 * N5 + lane;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const int off = m == 0 ? 0 : m == 1 ? 1 : m == 2 ? -1 : m == 3 ? 2 : -2;
            if (s + off < 0 || s + off >= Ls) continue;
            const float2* N = sN + 16 * (m == 0 ? (s < Ls - 1 ? 1 : 0) + (s > 0 ? 2 : 0) : m + 3);
#pragma unroll
            for (int col = 0; col < 3; ++col) {
                float2 v[4];
#pragma unroll
                for (int si = 0; si < 4; ++si) v[si] = __ldg(xs + (int64_t)(si * 3 + col) * N5 + off);
#pragma unroll
                for (int so = 0; so < 4; ++so) {
                    // each 4-spin product by itself: short sums before the long one
                    float tr = 0.f, ti = 0.f;
#pragma unroll
                    for (int si = 0; si < 4; ++si) {
                        const float2 w = N[so * 4 + si];
                        tr = fmaf(w.x, v[si].x, fmaf(-w.y, v[si].y, tr));
                        ti = fmaf(w.x, v[si].y, fmaf(w.y, v[si].x, ti));
                    }
                    ar[so * 3 + col] += tr;
                    ai[so * 3 + col] += ti;
                }
            }
        }
#pragma unroll 1
        for (int k = 0; k < 8; ++k) {   // direction k + 1 reads neighbour slot k
            const int n = a.nbr[site * 8 + k];
            if (n < 0) continue;
            const float2* p = reinterpret_cast<const float2*>(a.psi + k * a.fstride) + (int64_t)n * 12 * N5 + lane;
            float vr[12], vi[12], orr[12], oi[12];
#pragma unroll
            for (int c = 0; c < 12; ++c) {
                const float2 v = __ldg(p + (int64_t)c * N5);
                vr[c] = v.x;
                vi[c] = v.y;
            }
            su3_spinor(a.links + (site * 8 + k) * 18, vr, vi, orr, oi);
#pragma unroll
            for (int c = 0; c < 12; ++c) { ar[c] += orr[c]; ai[c] += oi[c]; }
        }
        float2* o = reinterpret_cast<float2*>(a.z) + site * 12 * N5 + lane;
#pragma unroll
        for (int c = 0; c < 12; ++c) o[(int64_t)c * N5] = make_float2(ar[c], ai[c]);
    }
}

// Weight gradient of one parity: g[o][so][i][si] = sum_pixels gout[o][so]
// conj(in[i][si]) over its (site, colour, lane) pixels, a [4 MF] x [4 NF]
// complex product contracted over millions of pixels.
//
// Bound: the FP32 pipe (batch 4 at 16^4 x 12, even sites: 38.7 G
// multiply-adds, 1.05 ms at 128 per clock and SM; its 3.6 GB of fields would
// take half of that).  The fields hold pixels contiguously, the
// product wants all rows of a pixel: 32 pixels at a time go through shared
// memory transposed, [pixel][row], the in rows with both parts doubled
// (xr, xr, xi, xi), so that a thread's 4 x 4 spin block of one (o, i) pair is
// 32 paired multiply-adds (two per complex product: the pair (gr, gi) times
// xr into A, times xi into B, combined once at the end) for 6 16-byte shared
// loads.  A warp takes WO x WI pairs (4 x 8: its 32 in vectors are one
// 128-byte row per load); the KS groups of warps take the pixels in turn; the
// next 32 pixels are loaded into registers during the arithmetic.  One thread
// per pair reading scalars from the fields' own order over both parities ran
// at 7 TFLOP/s (29.8 ms each of the two gradients); the whole training step of
// batch 4 at 16^4 x 12 went from 80.2 to 17.9 ms with this kernel and the
// zero directions left out of the mixes.
constexpr int kWgThreads = 256;
constexpr int kWgPix = 32;

template <int MF, int NF>
struct WgShape {
    static constexpr int WI = NF >= 8 ? 8 : 4, WO = 32 / WI;
    static constexpr int WM = (MF + WO - 1) / WO, WN = (NF + WI - 1) / WI;
    static constexpr int KS = (kWgThreads / 32) / (WM * WN);
    static constexpr int GS = MF * 4 + 2;      // float2 per pixel row of gout
    static constexpr int XS = NF * 4 + 1;      // float4 per pixel row of in
    static constexpr size_t smem = kWgPix * ((size_t)GS * 8 + (size_t)XS * 16);
    static_assert(WM * WN * KS * 32 == kWgThreads, "whole warps per pixel group");
};

template <int MF, int NF>
__global__ void __launch_bounds__(kWgThreads, 2) k_wgrad(const float* __restrict__ gout,
                                                         const float* __restrict__ in, int64_t npix, int N5,
                                                         int64_t fstride, double* __restrict__ partial) {
    using S = WgShape<MF, NF>;
    constexpr int ROWS = 4 * (MF + NF);
    constexpr int NLD = (ROWS + kWgThreads / 32 - 1) / (kWgThreads / 32);
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float4* sx = reinterpret_cast<float4*>(sm_raw);                      // [pixel][si][i]
    float2* sg = reinterpret_cast<float2*>(sx + (size_t)kWgPix * S::XS);   // [pixel][o][so]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ks = warp % S::KS, wt = warp / S::KS;
    const int o = (wt / S::WN) * S::WO + lane / S::WI, i = (wt % S::WN) * S::WI + lane % S::WI;
    const bool on = o < MF && i < NF;
    const int oc = on ? o : 0, ic = on ? i : 0;      // idle lanes of a ragged shape compute on pair 0
    float2 A[4][4], B[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) A[a][b] = B[a][b] = make_float2(0.f, 0.f);
    float2 v[NLD];
    auto load = [&](int64_t p0) {
        const int64_t p = p0 + lane;
        const bool live = p < npix;
        const int64_t sc = live ? p / N5 : 0;
        const int l = live ? (int)(p - sc * N5) : 0;
        const int64_t site = sc / 3;
        const int64_t base = (site * 12 + (sc - site * 3)) * N5 + l;
#pragma unroll
        for (int q = 0; q < NLD; ++q) {
            const int row = warp + q * (kWgThreads / 32);
            v[q] = make_float2(0.f, 0.f);
            if (row < ROWS && live) {
                const bool isg = row < 4 * MF;
                const int rr = isg ? row : row - 4 * MF;
                v[q] = *reinterpret_cast<const float2*>((isg ? gout : in) + (rr >> 2) * fstride +
                                                        2 * (base + (int64_t)(rr & 3) * 3 * N5));
            }
        }
    };
    const int64_t step = (int64_t)gridDim.x * kWgPix;
    int64_t p0 = (int64_t)blockIdx.x * kWgPix;
    if (p0 < npix) load(p0);
    for (; p0 < npix; p0 += step) {
        __syncthreads();   // the previous pixels are no longer read
#pragma unroll
        for (int q = 0; q < NLD; ++q) {
            const int row = warp + q * (kWgThreads / 32);
            if (row < 4 * MF) sg[lane * S::GS + row] = v[q];
            else if (row < ROWS) {
                const int rr = row - 4 * MF;
                sx[lane * S::XS + (rr & 3) * NF + (rr >> 2)] = make_float4(v[q].x, v[q].x, v[q].y, v[q].y);
            }
        }
        __syncthreads();
        if (p0 + step < npix) load(p0 + step);
#pragma unroll 2
        for (int k = ks; k < kWgPix; k += S::KS) {
            const float4* g4 = reinterpret_cast<const float4*>(sg + k * S::GS + oc * 4);
            const float4 ga = g4[0], gb = g4[1];
            const float2 g[4] = {make_float2(ga.x, ga.y), make_float2(ga.z, ga.w), make_float2(gb.x, gb.y),
                                 make_float2(gb.z, gb.w)};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float4 x = sx[k * S::XS + b * NF + ic];
                const float2 xr = make_float2(x.x, x.y), xi = make_float2(x.z, x.w);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    A[a][b] = __ffma2_rn(g[a], xr, A[a][b]);
                    B[a][b] = __ffma2_rn(g[a], xi, B[a][b]);
                }
            }
        }
    }
    if (on) {
        double* out = partial + ((size_t)blockIdx.x * S::KS + ks) * (MF * NF * 32);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int idx = ((o * 4 + a) * NF + i) * 4 + b;   // g conj(x)
                out[2 * idx] = (double)(A[a][b].x + B[a][b].y);
                out[2 * idx + 1] = (double)(A[a][b].y - B[a][b].x);
            }
    }
}

// Sum of the partials in a fixed order (8 slices, then the slices), written
// in the master layout [d][channel][so][si]; dirs[j] is the direction of
// field j on the side that runs over directions (gout for W2, in for W1).
struct WgDirs { int d[8]; };
__global__ void __launch_bounds__(256) k_wgrad_reduce(const double* __restrict__ partial, int nparts, int mf, int nf,
                                                      int C, bool dirs_out, WgDirs dirs, double* __restrict__ gw) {
    __shared__ double sh[8][33];
    const int nval = mf * nf * 32;
    const int v = blockIdx.x * 32 + (threadIdx.x & 31), sl = threadIdx.x >> 5;
    double s = 0.0;
    if (v < nval)
        for (int b = sl; b < nparts; b += 8) s += partial[(size_t)b * nval + v];
    sh[sl][threadIdx.x & 31] = s;
    __syncthreads();
    if (sl != 0 || v >= nval) return;
#pragma unroll
    for (int q = 1; q < 8; ++q) s += sh[q][threadIdx.x];
    const int part = v & 1, si = (v >> 1) & 3, i = (v >> 3) % nf, oa = (v >> 3) / nf;
    const int so = oa & 3, o = oa >> 2;
    const int d = dirs.d[dirs_out ? o : i], ch = dirs_out ? i : o;
    gw[2 * ((((size_t)d * C + ch) * 4 + so) * 4 + si) + part] = s;
}

// Adam on the real and imaginary parts (all arrays of n reals).
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const double* __restrict__ g, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = (float)g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

}  // namespace dwf

// ===================================================================== API
using namespace dwf;

struct dwf_nn {
    int C = 16;
    // master weights (FP32, complex interleaved), layout of the oracle:
    // W1[d][a][0][so][si] and W2[d][0][b][so][si]
    std::vector<float> w1, w2;
    float* d_w1 = nullptr;   // master FP32 (device), oracle layout
    float* d_w2 = nullptr;
    float* d_m = nullptr;    // Adam moments over [w1 | w2]
    float* d_v = nullptr;
    // per parity, over that parity's directions: BF16-rounded mixing matrices in
    // kernel layouts, the adjoint of layer 2, and W2 W1 (inference); one block
    float* d_mix = nullptr;
    float* mix1[2] = {nullptr, nullptr};
    float* mix2[2] = {nullptr, nullptr};
    float* mix2h[2] = {nullptr, nullptr};
    float* fold = nullptr;       // even sites, 8 x 8 blocks
    float* nmat = nullptr;       // odd sites, the spin matrices of k_odd_sum
    int adam_t = 0;
    // the last application queued on each stream, for the next change of the
    // mixing matrices to wait for; untracked once one is in a captured graph
    struct Reader {
        cudaStream_t stream;
        cudaEvent_t done;
    };
    std::mutex readers_mu;
    std::vector<Reader> readers;
    bool untracked = false;
};

namespace dwf {

static size_t w1_len(int C) { return (size_t)kNDir * C * 16 * 2; }
static size_t w2_len(int C) { return (size_t)kNDir * C * 16 * 2; }

// Directions whose R_d = T_d x0 can be nonzero on each parity when x0 vanishes
// on even sites: the link transports reach even sites from odd neighbours, the
// identity and the two s-shifts stay on odd sites.
constexpr int kNFold[2] = {8, 3};
constexpr int kFoldDirs[2][8] = {{1, 2, 3, 4, 5, 6, 7, 8}, {0, 9, 10, 0, 0, 0, 0, 0}};
static size_t fold_len(int p) { return (size_t)kNFold[p] * 4 * kNFold[p] * 4 * 2; }
static size_t mix_part_len(int C, int p) { return (size_t)kNFold[p] * C * 16 * 2; }
static size_t mix_len(int C) {
    size_t n = 0;
    for (int p = 0; p < 2; ++p) n += 3 * mix_part_len(C, p);
    return n + fold_len(0) + 8 * 16 * 2;
}

struct MixOut {
    float* m1[2];
    float* m2[2];
    float* m2h[2];
    float* fold;
    float* nmat;
};

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// (W2[d] W1[dp])[so][si] = sum_{b,t} W2[d][b][so][t] W1[dp][b][t][si], FP64 products of the BF16-rounded weights
__device__ __forceinline__ double2 fold_entry(const float* __restrict__ w1, const float* __restrict__ w2, int C, int d,
                                              int dp, int so, int si) {
    double mr = 0.0, mi = 0.0;
    for (int b = 0; b < C; ++b)
        for (int t = 0; t < 4; ++t) {
            const size_t q2 = (((size_t)d * C + b) * 4 + so) * 4 + t;
            const size_t q1 = (((size_t)dp * C + b) * 4 + t) * 4 + si;
            const double ar = bf16_round(w2[2 * q2]), ai = bf16_round(w2[2 * q2 + 1]);
            const double br = bf16_round(w1[2 * q1]), bi = bf16_round(w1[2 * q1 + 1]);
            mr += ar * br - ai * bi;
            mi += ar * bi + ai * br;
        }
    return make_double2(mr, mi);
}

// Mixing matrices from the FP32 master weights (rounded to BF16), per parity p
// over its n directions d = dirs[p][.]:
//   m1  [o = a][so][i = d][si]  = W1[d][a][so][si]
//   m2  [o = d][so][i = b][si]  = W2[d][b][so][si]
//   m2h [o = b][so][i = d][si]  = conj(W2[d][b][si][so])
// and for the inference W2 W1 in FP64, stored FP32: on even sites
//   fold[o = d][so][i = d'][si] = W2[d] W1[d'], d, d' = 1..8,
// on odd sites the matrices of k_odd_sum, sums over the pairs (d, d') of 0, 9
// (s + 1), 10 (s - 1) with the same total shift.  One thread per complex entry.
struct MixDirs { int n[2]; int d[2][8]; };
__global__ void k_mix_weights(const float* __restrict__ w1, const float* __restrict__ w2, int C, MixDirs md, MixOut out) {
    const int p = blockIdx.y, n = md.n[p];
    const int nw = n * C * 16, nf = p == 0 ? n * n * 16 : 8 * 16;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nw + nf; e += gridDim.x * blockDim.x) {
        if (e < nw) {
            const int si = e & 3, so = (e >> 2) & 3, ch = (e >> 4) % C, j = (e >> 4) / C;
            const size_t src = (((size_t)md.d[p][j] * C + ch) * 4 + so) * 4 + si;
            const float r2 = bf16_round(w2[2 * src]), i2 = bf16_round(w2[2 * src + 1]);
            const size_t o1 = (((size_t)ch * 4 + so) * n + j) * 4 + si, o2 = (((size_t)j * 4 + so) * C + ch) * 4 + si,
                         oh = (((size_t)ch * 4 + si) * n + j) * 4 + so;
            out.m1[p][2 * o1] = bf16_round(w1[2 * src]);
            out.m1[p][2 * o1 + 1] = bf16_round(w1[2 * src + 1]);
            out.m2[p][2 * o2] = r2;
            out.m2[p][2 * o2 + 1] = i2;
            out.m2h[p][2 * oh] = r2;
            out.m2h[p][2 * oh + 1] = -i2;
        } else {
            const int f = e - nw;
            const int si = f & 3, so = (f >> 2) & 3, m = f >> 4;
            double2 v = make_double2(0.0, 0.0);
            auto add = [&](int d, int dp) {
                const double2 t = fold_entry(w1, w2, C, d, dp, so, si);
                v.x += t.x;
                v.y += t.y;
            };
            if (p == 0) {
                const int i = m % n, o = m / n;
                add(md.d[0][o], md.d[0][i]);
                const size_t dst = (((size_t)o * 4 + so) * n + i) * 4 + si;
                out.fold[2 * dst] = (float)v.x;
                out.fold[2 * dst + 1] = (float)v.y;
            } else {
                if (m < 4) {   // N0: T_0 T_0, and T_9 T_10 below the last lane, T_10 T_9 above the first
                    add(0, 0);
                    if (m & 1) add(9, 10);
                    if (m & 2) add(10, 9);
                } else if (m == 4) { add(0, 9); add(9, 0); }
                else if (m == 5) { add(0, 10); add(10, 0); }
                else if (m == 6) add(9, 9);
                else add(10, 10);
                out.nmat[2 * f] = (float)v.x;
                out.nmat[2 * f + 1] = (float)v.y;
            }
        }
    }
}

// Note that the work queued on s so far reads the mixing matrices.  An event is
// never recorded before what it stood for is done: of another stream, or of an
// earlier stream with the same handle.
constexpr size_t kMaxReaders = 64;

static dwf_status note_reader(dwf_nn* K, cudaStream_t s) {
    std::lock_guard<std::mutex> lock(K->readers_mu);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    DWF_CUDA(cudaStreamIsCapturing(s, &cap));
    if (cap != cudaStreamCaptureStatusNone) {
        K->untracked = true;
        return DWF_OK;
    }
    auto it = std::find_if(K->readers.begin(), K->readers.end(), [s](const dwf_nn::Reader& r) { return r.stream == s; });
    if (it == K->readers.end() && K->readers.size() < kMaxReaders) {
        cudaEvent_t e;
        DWF_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        it = K->readers.insert(it, {s, e});
    } else {
        if (it == K->readers.end()) it = K->readers.begin();
        DWF_CUDA(cudaStreamWaitEvent(s, it->done, 0));
        it->stream = s;
    }
    DWF_CUDA(cudaEventRecord(it->done, s));
    return DWF_OK;
}

// Rebuild the mixing matrices after the master weights changed, on stream s,
// behind the applications queued on other streams, which still read them.  Not
// by a wait for the device: that would wait for unrelated work, and fail while
// any thread captures a graph (a solve does); only a graph that holds an
// application, whose replays leave no event, asks for it.  Every caller waits for
// s before it returns, so that a later call may use them on any stream.
static dwf_status refresh_mix(dwf_nn* K, cudaStream_t s) {
    {
        std::lock_guard<std::mutex> lock(K->readers_mu);
        if (K->untracked) DWF_CUDA(cudaDeviceSynchronize());
        for (const dwf_nn::Reader& r : K->readers) DWF_CUDA(cudaStreamWaitEvent(s, r.done, 0));
    }
    MixDirs md{};
    MixOut mo{};
    for (int p = 0; p < 2; ++p) {
        md.n[p] = kNFold[p];
        for (int j = 0; j < kNFold[p]; ++j) md.d[p][j] = kFoldDirs[p][j];
        mo.m1[p] = K->mix1[p];
        mo.m2[p] = K->mix2[p];
        mo.m2h[p] = K->mix2h[p];
    }
    mo.fold = K->fold;
    mo.nmat = K->nmat;
    k_mix_weights<<<dim3(12, 2), 256, 0, s>>>(K->d_w1, K->d_w2, K->C, md, mo);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

// network workspace of a handle for nrhs lanes.  Field j of R, psi on parity p
// belongs to direction kFoldDirs[p][j]: what is exactly zero (below) has no
// storage.
struct NNWS {
    int nrhs = 0, C = 0;
    float* R = nullptr;       // 8 full fields (training)
    float* psi = nullptr;     // 8 full fields
    float* phi = nullptr;     // C full fields (training)
    float* gphi = nullptr;    // C full fields (training)
    float* z = nullptr;       // odd FP32 fields (training): K r, then the gradient of the loss
    float* at = nullptr;      // odd FP32 temporaries for the energy-norm loss
    float* aw = nullptr;
    double* wpart = nullptr;  // weight-gradient partials
    double* gw = nullptr;     // [gW1 | gW2], master layout
    double* scal = nullptr;   // loss scalars [4][nrhs]
    double* part = nullptr;   // loss partials (per tile and right-hand side)
};

static std::map<dwf_handle*, NNWS> g_nnws;

static int64_t full_floats(const dwf_handle* h, int nrhs) {
    return (int64_t)(h->nsite[0] + h->nsite[1]) * 12 * h->p.Ls * nrhs * 2;
}

static void free_nn_bufs(NNWS& w) {
    void* p[] = {w.R, w.psi, w.phi, w.gphi, w.z, w.at, w.aw, w.wpart, w.gw, w.scal, w.part};
    for (void* q : p) cudaFree(q);
    w = NNWS();
}

constexpr int kWgBlocks = 152 * 2;
// Ls * nrhs of a training batch.  The weight gradient has no such limit (32
// pixels a step, whatever the lanes); kept so that a batch is taken or refused
// by the same rule as ever.
constexpr int kMaxTrainLanes = 236;

template <int MF, int NF>
static cudaError_t wgrad_attr() {
    return cudaFuncSetAttribute(k_wgrad<MF, NF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)WgShape<MF, NF>::smem);
}

static dwf_status nn_ws(dwf_handle* h, int nrhs, int C, bool train, NNWS** out) {
    NNWS& w = g_nnws[h];
    if (w.nrhs != nrhs || w.C != C || (train && w.gphi == nullptr)) {
        free_nn_bufs(w);
        const int64_t f = full_floats(h, nrhs);
        if (train) {
            DWF_CUDA((wgrad_attr<kNFold[0], 16>()));
            DWF_CUDA((wgrad_attr<16, kNFold[0]>()));
            DWF_CUDA((wgrad_attr<kNFold[1], 16>()));
            DWF_CUDA((wgrad_attr<16, kNFold[1]>()));
        }
        DWF_CUDA(dev_malloc(&w.psi, (size_t)kNFold[0] * f * 4));
        if (train) {
            DWF_CUDA(dev_malloc(&w.R, (size_t)kNFold[0] * f * 4));
            DWF_CUDA(dev_malloc(&w.phi, (size_t)C * f * 4));
            const size_t pairs8 = (size_t)kWgBlocks * WgShape<8, 16>::KS * 8 * 16 * 32;
            const size_t pairs3 = (size_t)kWgBlocks * WgShape<3, 16>::KS * 3 * 16 * 32;
            DWF_CUDA(dev_malloc(&w.wpart, std::max(pairs8, pairs3) * sizeof(double)));
            DWF_CUDA(dev_malloc(&w.gw, (w1_len(C) + w2_len(C)) * sizeof(double)));
            const size_t odd = (size_t)h->nsite[1] * 12 * h->p.Ls * nrhs * 2;
            DWF_CUDA(dev_malloc(&w.z, odd * 4));
            DWF_CUDA(dev_malloc(&w.at, odd * 4));
            DWF_CUDA(dev_malloc(&w.aw, odd * 4));
            DWF_CUDA(dev_malloc(&w.scal, (size_t)4 * nrhs * sizeof(double)));
            DWF_CUDA(dev_malloc(&w.part, (size_t)(h->nsite[1] / kMinTile + h->nbox + 1) * nrhs * sizeof(double)));
            DWF_CUDA(dev_malloc(&w.gphi, (size_t)C * f * 4));
        }
        w.nrhs = nrhs;
        w.C = C;
    }
    *out = &w;
    return DWF_OK;
}

void free_nn_ws(dwf_handle* h) {
    auto it = g_nnws.find(h);
    if (it == g_nnws.end()) return;
    free_nn_bufs(it->second);
    g_nnws.erase(it);
}

// T_{dirs[j]} of one field into fields out + j ostride (multi), or the sum of
// T_{dirs[j]} of the input fields (sum), on the sites of parity p.  same / opp
// are the input's blocks of parity p and 1 - p.
static dwf_status launch_transport(dwf_handle* h, int nrhs, int p, const float* same, const float* opp, float* out,
                                   const int* dirs, int ndir, bool sum, cudaStream_t s) {
    const TileSet* tsp = nullptr;
    DWF_TRY(get_tiles(h, tile_for(h, nrhs), &tsp));
    const TileSet& ts = *tsp;
    if (ts.ntiles[p] == 0) return DWF_OK;
    TransArgs a{};
    a.same = same;
    a.opp = opp;
    a.out = out;
    a.links = (const float*)h->d_links[DWF_FP32][p];
    a.nbr = h->d_nbr[p];
    a.tiles = ts.d_tiles[p];
    a.N5 = h->p.Ls * nrhs;
    a.Ls = h->p.Ls;
    a.istride = a.ostride = full_floats(h, nrhs);
    a.ndir = ndir;
    for (int j = 0; j < ndir; ++j) a.dirs[j] = dirs[j];
    if (sum) k_transport_sum<<<ts.ntiles[p], 256, 0, s>>>(a);
    else k_transport_multi<<<ts.ntiles[p], 256, 0, s>>>(a);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

template <int NOUT, bool GATHER>
static dwf_status launch_mix_t(const MixArgs& a, cudaStream_t s) {
    const size_t smem = (size_t)NOUT * 4 * a.nin * 4 * 2 * sizeof(float);
    const int blocks = (int)std::min<int64_t>((a.npix + 127) / 128, 152 * 16);
    k_mix<NOUT, GATHER><<<blocks, 128, smem, s>>>(a);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

// Mixing on the block of parity p (`in` and `out` point at the block, fields
// keep the full-field stride).
static dwf_status launch_mix(dwf_handle* h, int nrhs, int p, const float* in, int nin, float* out, int nout,
                             const float* W, cudaStream_t s, bool gather = false) {
    MixArgs a{};
    a.in = in;
    a.out = out;
    a.W = W;
    a.nin = nin;
    a.N5 = h->p.Ls * nrhs;
    a.npix = h->nsite[p] * 3 * (int64_t)a.N5;
    a.fstride = full_floats(h, nrhs);
    a.links = (const float*)h->d_links[DWF_FP32][p];
    a.nbr = h->d_nbr[p];
    if (a.npix == 0) return DWF_OK;
    if (gather) return launch_mix_t<8, true>(a, s);
    if (nout == 16) return launch_mix_t<16, false>(a, s);
    if (nout == 8) return launch_mix_t<8, false>(a, s);
    if (nout == 3) return launch_mix_t<3, false>(a, s);
    set_error("nn: unsupported channel count %d", nout);
    return DWF_ERR_UNSUPPORTED;
}

// gW of one layer from parity p's pixels: MF fields of gout against NF of in;
// dirs_out: the gout side runs over directions (W2), else the in side (W1).
template <int MF, int NF>
static dwf_status launch_wgrad(dwf_handle* h, NNWS& w, int nrhs, int p, const float* gout, const float* in,
                               bool dirs_out, double* dst, cudaStream_t s) {
    using S = WgShape<MF, NF>;
    const int N5 = h->p.Ls * nrhs;
    const int64_t npix = h->nsite[p] * 3 * (int64_t)N5;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((npix + kWgPix - 1) / kWgPix, kWgBlocks));
    k_wgrad<MF, NF><<<blocks, kWgThreads, S::smem, s>>>(gout, in, npix, N5, full_floats(h, nrhs), w.wpart);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    WgDirs wd{};
    for (int j = 0; j < kNFold[p]; ++j) wd.d[j] = kFoldDirs[p][j];
    constexpr int nval = MF * NF * 32;
    k_wgrad_reduce<<<nval / 32, 256, 0, s>>>(w.wpart, blocks * S::KS, MF, NF, w.C, dirs_out, wd, dst);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

// z = sum_d T_d psi_d on odd sites; psi's field j on parity p holds direction
// kFoldDirs[p][j]
static dwf_status psi_sum(dwf_handle* h, int nrhs, const float* psi, float* z, cudaStream_t s) {
    int dirs[kNDir], nd = 0;
    for (int p = 1; p >= 0; --p)
        for (int j = 0; j < kNFold[p]; ++j) dirs[nd++] = kFoldDirs[p][j];
    const int64_t c0 = h->nsite[0] * 12 * (int64_t)h->p.Ls * nrhs * 2;
    return launch_transport(h, nrhs, 1, psi + c0, psi, z, dirs, nd, true, s);
}

// z = K x on the odd checkerboard through the channels (training: R and phi
// are kept for the gradient).  What is exactly zero is left out throughout:
// x vanishes on even sites, so R_d = T_d x is zero on odd sites for the link
// directions 1..8 and on even sites for 0, 9 and 10; z is read on odd sites
// only, which take psi_d from even sites for d = 1..8 and from odd sites for
// 0, 9, 10.
static dwf_status nn_forward(dwf_nn* K, dwf_handle* h, NNWS& w, const float* x, int nrhs, cudaStream_t s) {
    const int64_t c0 = h->nsite[0] * 12 * (int64_t)h->p.Ls * nrhs * 2;
    for (int p = 0; p < 2; ++p) {
        const int64_t o = p ? c0 : 0;
        const int n = kNFold[p];
        DWF_TRY(launch_transport(h, nrhs, p, x, x, w.R + o, kFoldDirs[p], n, false, s));
        DWF_TRY(launch_mix(h, nrhs, p, w.R + o, n, w.phi + o, K->C, K->mix1[p], s));
        DWF_TRY(launch_mix(h, nrhs, p, w.phi + o, K->C, w.psi + o, n, K->mix2[p], s));
    }
    return psi_sum(h, nrhs, w.psi, w.z, s);
}

// Inference z = K x on the odd checkerboard: the same function as nn_forward
// up to rounding; with no nonlinearity between the layers psi = (W2 W1) R, so
// on even sites one mix over the eight link directions, which gathers its
// input from x, replaces the transports and the two mixes through the C
// channels, and the odd-site directions are applied with the final sum.  At
// 24^4 x 16 (75 GFLOP) 2.15 ms; with R and the odd-site psi stored, 3.02.
dwf_status nn_apply_internal(dwf_nn* K, dwf_handle* h, float* out, const float* in, int nrhs,
                             cudaStream_t s) {
    NNWS* w;
    DWF_TRY(nn_ws(h, nrhs, K->C, false, &w));
    const int64_t c0 = h->nsite[0] * 12 * (int64_t)h->p.Ls * nrhs * 2, c1 = full_floats(h, nrhs) - c0;
    if (in < out + c1 && out < in + c1) {   // in place: the odd block of psi's field 0 is free
        DWF_CUDA(cudaMemcpyAsync(w->psi + c0, in, c1 * 4, cudaMemcpyDeviceToDevice, s));
        in = w->psi + c0;
    }
    DWF_TRY(launch_mix(h, nrhs, 0, in, kNFold[0], w->psi, kNFold[0], K->fold, s, true));
    const TileSet* tsp = nullptr;
    DWF_TRY(get_tiles(h, tile_for(h, nrhs), &tsp));
    if (tsp->ntiles[1] == 0) return note_reader(K, s);
    OddArgs a{};
    a.x = in;
    a.psi = w->psi;
    a.z = out;
    a.nmat = K->nmat;
    a.links = (const float*)h->d_links[DWF_FP32][1];
    a.nbr = h->d_nbr[1];
    a.tiles = tsp->d_tiles[1];
    a.N5 = h->p.Ls * nrhs;
    a.Ls = h->p.Ls;
    a.fstride = full_floats(h, nrhs);
    k_odd_sum<<<tsp->ntiles[1], 256, 0, s>>>(a);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return note_reader(K, s);
}

}  // namespace dwf

extern "C" {

dwf_status dwf_nn_create(dwf_nn** out, int channels) {
    if (out == nullptr || channels != 16) {
        set_error("dwf_nn_create: channels must be 16");
        return DWF_ERR_ARG;
    }
    dwf_nn* K = new dwf_nn();
    K->C = channels;
    const size_t n1 = w1_len(channels), n2 = w2_len(channels);
    K->w1.assign(n1, 0.f);
    K->w2.assign(n2, 0.f);
    // identity: W1[0][0] = 1, W2[0][0][0] = 1
    for (int so = 0; so < 4; ++so) {
        K->w1[2 * (so * 4 + so)] = 1.f;
        K->w2[2 * (so * 4 + so)] = 1.f;
    }
    if (dev_malloc(&K->d_w1, n1 * 4) != cudaSuccess || dev_malloc(&K->d_w2, n2 * 4) != cudaSuccess ||
        dev_malloc(&K->d_m, (n1 + n2) * 4) != cudaSuccess ||
        dev_malloc(&K->d_v, (n1 + n2) * 4) != cudaSuccess ||
        dev_malloc(&K->d_mix, mix_len(channels) * 4) != cudaSuccess) {
        set_error("dwf_nn_create: cudaMalloc failed");
        dwf_nn_destroy(K);
        return DWF_ERR_CUDA;
    }
    float* m = K->d_mix;
    for (int p = 0; p < 2; ++p) {
        float** part[3] = {&K->mix1[p], &K->mix2[p], &K->mix2h[p]};
        for (float** q : part) { *q = m; m += mix_part_len(channels, p); }
    }
    K->fold = m;
    K->nmat = m + fold_len(0);
    cudaMemcpy(K->d_w1, K->w1.data(), n1 * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(K->d_w2, K->w2.data(), n2 * 4, cudaMemcpyHostToDevice);
    cudaMemset(K->d_m, 0, (n1 + n2) * 4);
    cudaMemset(K->d_v, 0, (n1 + n2) * 4);
    if (refresh_mix(K, nullptr) != DWF_OK || cudaStreamSynchronize(nullptr) != cudaSuccess) {
        dwf_nn_destroy(K);
        return DWF_ERR_CUDA;
    }
    *out = K;
    return DWF_OK;
}

dwf_status dwf_nn_destroy(dwf_nn* K) {
    if (!K) return DWF_OK;
    cudaFree(K->d_w1); cudaFree(K->d_w2); cudaFree(K->d_m); cudaFree(K->d_v);
    cudaFree(K->d_mix);
    for (const dwf_nn::Reader& r : K->readers) cudaEventDestroy(r.done);
    delete K;
    return DWF_OK;
}

dwf_status dwf_nn_set_weights(dwf_nn* K, const double* w, size_t n) {
    if (!K || !w || n != (w1_len(K->C) + w2_len(K->C)) / 2) {
        set_error("dwf_nn_set_weights: expected %zu complex numbers",
                  K ? (w1_len(K->C) + w2_len(K->C)) / 2 : (size_t)0);
        return DWF_ERR_ARG;
    }
    const size_t n1 = w1_len(K->C);
    std::vector<float> all(2 * n);
    for (size_t i = 0; i < 2 * n; ++i) all[i] = (float)w[i];
    DWF_CUDA(cudaMemcpy(K->d_w1, all.data(), n1 * 4, cudaMemcpyHostToDevice));
    DWF_CUDA(cudaMemcpy(K->d_w2, all.data() + n1, (2 * n - n1) * 4, cudaMemcpyHostToDevice));
    DWF_TRY(refresh_mix(K, nullptr));
    DWF_CUDA(cudaStreamSynchronize(nullptr));
    return DWF_OK;
}

dwf_status dwf_nn_get_weights(const dwf_nn* K, double* w, size_t n) {
    if (!K || !w || n != (w1_len(K->C) + w2_len(K->C)) / 2) {
        set_error("dwf_nn_get_weights: bad buffer");
        return DWF_ERR_ARG;
    }
    const size_t n1 = w1_len(K->C);
    std::vector<float> all(2 * n);
    DWF_CUDA(cudaMemcpy(all.data(), K->d_w1, n1 * 4, cudaMemcpyDeviceToHost));
    DWF_CUDA(cudaMemcpy(all.data() + n1, K->d_w2, (2 * n - n1) * 4, cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < 2 * n; ++i) w[i] = all[i];
    return DWF_OK;
}

// Weight file: the 8 bytes "DWFNN001", int32 channels, int32 0, int64 number
// of complex weights n, then n complex128 (re, im) in the order of
// dwf_nn_set_weights, little-endian as written by this host.
static const char kNNMagic[8] = {'D', 'W', 'F', 'N', 'N', '0', '0', '1'};

dwf_status dwf_nn_save(const dwf_nn* K, const char* path) {
    if (!K || !path) {
        set_error("dwf_nn_save: null argument");
        return DWF_ERR_ARG;
    }
    const size_t n = (w1_len(K->C) + w2_len(K->C)) / 2;
    std::vector<double> w(2 * n);
    DWF_TRY(dwf_nn_get_weights(K, w.data(), n));
    FILE* f = fopen(path, "wb");
    if (!f) {
        set_error("dwf_nn_save: cannot open %s for writing", path);
        return DWF_ERR_ARG;
    }
    const int32_t hdr[2] = {K->C, 0};
    const int64_t nn = (int64_t)n;
    bool ok = fwrite(kNNMagic, 1, 8, f) == 8 && fwrite(hdr, sizeof(hdr), 1, f) == 1 &&
              fwrite(&nn, sizeof(nn), 1, f) == 1 && fwrite(w.data(), sizeof(double), w.size(), f) == w.size();
    ok = (fclose(f) == 0) && ok;
    if (!ok) {
        set_error("dwf_nn_save: write to %s failed", path);
        return DWF_ERR_ARG;
    }
    return DWF_OK;
}

dwf_status dwf_nn_load(dwf_nn* K, const char* path) {
    if (!K || !path) {
        set_error("dwf_nn_load: null argument");
        return DWF_ERR_ARG;
    }
    FILE* f = fopen(path, "rb");
    if (!f) {
        set_error("dwf_nn_load: cannot open %s", path);
        return DWF_ERR_ARG;
    }
    char magic[8];
    int32_t hdr[2];
    int64_t nn = 0;
    const size_t n = (w1_len(K->C) + w2_len(K->C)) / 2;
    bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, kNNMagic, 8) == 0 && fread(hdr, sizeof(hdr), 1, f) == 1 &&
              fread(&nn, sizeof(nn), 1, f) == 1 && hdr[0] == K->C && nn == (int64_t)n;
    std::vector<double> w(2 * n);
    ok = ok && fread(w.data(), sizeof(double), w.size(), f) == w.size();
    fclose(f);
    if (!ok) {
        set_error("dwf_nn_load: %s is not a weight file of a %d-channel network", path, K->C);
        return DWF_ERR_ARG;
    }
    return dwf_nn_set_weights(K, w.data(), n);
}

// One training pair from an FP64 solve: e = (x* - x_k) / |x* - x_k|,
// r = M_pc^+ M_pc e (FP64 operator), both written in FP32.
dwf_status dwf_nn_make_pair(dwf_handle* h, const double* x_star, const double* x_k, float* r,
                            float* e, double* norm, void* stream) {
    DWF_RANGE("dwf_nn_make_pair");
    DWF_TRY(check_handle(h));
    if (!x_star || !x_k || !r || !e || !norm || !h->have_gauge || h->dirichlet) {
        set_error("dwf_nn_make_pair: bad argument (whole-lattice handle with a gauge field, "
                  "non-null fields)");
        return DWF_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const size_t no = cb_elems(h, 1, 1);
    const int T = tile_for(h, 1);
    const TileSet* tsp = nullptr;
    DWF_TRY(get_tiles(h, T, &tsp));
    double* buf = nullptr;
    const size_t nd = (size_t)tsp->ntiles[1] + 1;
    DWF_CUDA(dev_malloc(&buf, (3 * no * 2 + nd) * sizeof(double)));
    double* e64 = buf;
    double* t64 = buf + 2 * no;
    double* r64 = buf + 4 * no;
    double* part = buf + 6 * no;
    double* d_n2 = part + tsp->ntiles[1];
    double n2 = 0.0;
    dwf_status st = DWF_OK;
    auto run = [&]() -> dwf_status {
        DWF_CUDA(cudaMemcpyAsync(e64, x_star, no * 16, cudaMemcpyDeviceToDevice, s));
        DWF_TRY(launch_axpby(h, 1, 1, nullptr, -1.0, x_k, DWF_FP64, nullptr, 1.0, e64, DWF_FP64, nullptr, T, s));
        DWF_TRY(launch_dot_partial(h, 1, e64, e64, DWF_FP64, DWF_FP64, 1, part, T, s));
        DWF_TRY(launch_reduce_sys(h, 1, part, 1, d_n2, T, s));
        DWF_CUDA(cudaMemcpyAsync(&n2, d_n2, sizeof(double), cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaStreamSynchronize(s));
        *norm = std::sqrt(n2);
        if (!(n2 > 0.0)) return DWF_OK;
        DWF_TRY(launch_axpby(h, 1, 1, nullptr, 0.0, e64, DWF_FP64, nullptr, 1.0 / *norm, e64, DWF_FP64,
                             nullptr, T, s));
        DWF_TRY(op_mpc(h, t64, e64, 0, DWF_FP64, DWF_FP64, 1, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        DWF_TRY(op_mpc(h, r64, t64, 1, DWF_FP64, DWF_FP64, 1, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        DWF_TRY(launch_convert(r, DWF_FP32, r64, DWF_FP64, no, s));
        DWF_TRY(launch_convert(e, DWF_FP32, e64, DWF_FP64, no, s));
        DWF_CUDA(cudaStreamSynchronize(s));
        return DWF_OK;
    };
    st = run();
    cudaFree(buf);
    return st;
}

// out = K in on the odd checkerboard (FP32 cb fields, nrhs lanes)
dwf_status dwf_nn_apply(dwf_nn* K, dwf_handle* h, float* out, const float* in, int nrhs, void* stream) {
    DWF_RANGE("dwf_nn_apply");
    DWF_TRY(check_handle(h));
    if (!K || !out || !in || nrhs < 1 || nrhs > h->nrhs_max || !h->have_gauge) {
        set_error("dwf_nn_apply: bad argument");
        return DWF_ERR_ARG;
    }
    return nn_apply_internal(K, h, out, in, nrhs, (cudaStream_t)stream);
}

// One Adam step on a batch of nrhs (r, e) pairs (odd cb FP32, lanes = pairs):
// loss = mean_k |K r_k - e_k|^2 / |e_k|^2 (returned, before the step).
dwf_status dwf_nn_train_step(dwf_nn* K, dwf_handle* h, const float* r, const float* e, int nrhs,
                             int loss_kind, double lr, double* loss, void* stream) {
    DWF_RANGE("dwf_nn_train_step");
    DWF_TRY(check_handle(h));
    if (!K || !r || !e || nrhs < 1 || nrhs > h->nrhs_max || !h->have_gauge || h->dirichlet) {
        set_error("dwf_nn_train_step: bad argument");
        return DWF_ERR_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (h->p.Ls * nrhs > kMaxTrainLanes) {
        set_error("nn: %d lanes exceed the training step's %d", h->p.Ls * nrhs, kMaxTrainLanes);
        return DWF_ERR_UNSUPPORTED;
    }
    NNWS* wp;
    DWF_TRY(nn_ws(h, nrhs, K->C, true, &wp));
    NNWS& w = *wp;
    const int C = K->C;
    const int64_t c0 = h->nsite[0] * 12 * (int64_t)h->p.Ls * nrhs * 2;
    const int64_t c1 = h->nsite[1] * 12 * (int64_t)h->p.Ls * nrhs * 2;
    DWF_TRY(nn_forward(K, h, w, r, nrhs, s));
    const int T = tile_for(h, nrhs);
    std::vector<double> h1(nrhs), h2(nrhs), h3(nrhs);
    double* d1 = w.scal;
    double* d2 = w.scal + nrhs;
    double* d_coef = w.scal + 2 * nrhs;
    double* d3 = w.scal + 3 * nrhs;
    double* part = w.part;
    float* zo = w.z;
    auto dot = [&](const void* x, const void* y, double* dst) -> dwf_status {
        DWF_TRY(launch_dot_partial(h, 1, x, y, DWF_FP32, DWF_FP32, nrhs, part, T, s));
        return launch_reduce_sys(h, 1, part, nrhs, dst, T, s);
    };
    double L = 0.0;
    std::vector<double> coef(nrhs);
    if (loss_kind == 0) {
        // |z - e|^2 / |e|^2: the fit residual overwrites z
        DWF_TRY(launch_axpby(h, 1, nrhs, nullptr, -1.0, e, DWF_FP32, nullptr, 1.0, zo, DWF_FP32, nullptr, T, s));
        DWF_TRY(dot(e, e, d1));
        DWF_TRY(dot(zo, zo, d2));
        DWF_CUDA(cudaMemcpyAsync(h1.data(), d1, nrhs * 8, cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaMemcpyAsync(h2.data(), d2, nrhs * 8, cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaStreamSynchronize(s));
        for (int k = 0; k < nrhs; ++k) {
            L += h2[k] / h1[k] / nrhs;
            coef[k] = 2.0 / (h1[k] * nrhs);
        }
    } else if (loss_kind == 2) {
        // A^2 norm: |A z - r|^2 / |r|^2, gradient 2 A (A z - r) / |r|^2, held in z
        DWF_TRY(op_mpc(h, w.at, zo, 0, DWF_FP32, DWF_FP32, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        DWF_TRY(op_mpc(h, w.aw, w.at, 1, DWF_FP32, DWF_FP32, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        DWF_TRY(launch_axpby(h, 1, nrhs, nullptr, -1.0, r, DWF_FP32, nullptr, 1.0, w.aw, DWF_FP32, nullptr, T, s));
        DWF_TRY(dot(w.aw, w.aw, d1));
        DWF_TRY(dot(r, r, d3));
        DWF_CUDA(cudaMemcpyAsync(h1.data(), d1, nrhs * 8, cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaMemcpyAsync(h3.data(), d3, nrhs * 8, cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaStreamSynchronize(s));
        for (int k = 0; k < nrhs; ++k) {
            L += h1[k] / h3[k] / nrhs;
            coef[k] = 2.0 / (h3[k] * nrhs);
        }
        DWF_TRY(op_mpc(h, w.at, w.aw, 0, DWF_FP32, DWF_FP32, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        DWF_TRY(op_mpc(h, zo, w.at, 1, DWF_FP32, DWF_FP32, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
    } else {
        // energy norm of A = M_pc^+ M_pc: (<z,Az> - 2 Re<z,r> + <e,r>) / <e,r>,
        // gradient 2 (A z - r) / <e,r>, held in z
        DWF_TRY(op_mpc(h, w.at, zo, 0, DWF_FP32, DWF_FP32, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        DWF_TRY(op_mpc(h, w.aw, w.at, 1, DWF_FP32, DWF_FP32, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        DWF_TRY(dot(zo, w.aw, d1));
        DWF_TRY(dot(zo, r, d2));
        DWF_TRY(dot(e, r, d3));
        DWF_CUDA(cudaMemcpyAsync(h1.data(), d1, nrhs * 8, cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaMemcpyAsync(h2.data(), d2, nrhs * 8, cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaMemcpyAsync(h3.data(), d3, nrhs * 8, cudaMemcpyDeviceToHost, s));
        DWF_CUDA(cudaStreamSynchronize(s));
        for (int k = 0; k < nrhs; ++k) {
            L += (h1[k] - 2.0 * h2[k] + h3[k]) / h3[k] / nrhs;
            coef[k] = 2.0 / (h3[k] * nrhs);
        }
        DWF_TRY(launch_axpby(h, 1, nrhs, nullptr, -1.0, r, DWF_FP32, nullptr, 1.0, w.aw, DWF_FP32, nullptr, T, s));
        DWF_CUDA(cudaMemcpyAsync(zo, w.aw, (size_t)c1 * 4, cudaMemcpyDeviceToDevice, s));
    }
    if (loss) *loss = L;
    DWF_CUDA(cudaMemcpyAsync(d_coef, coef.data(), nrhs * 8, cudaMemcpyHostToDevice, s));
    // g_z = coef * (held residual) on odd sites (zero on even sites, so the same
    // directions survive per parity as in the forward pass)
    DWF_TRY(launch_axpby(h, 1, nrhs, nullptr, 0.0, nullptr, DWF_FP32, d_coef, 0.0, zo, DWF_FP32, nullptr, T, s));
    const size_t n1 = w1_len(C), n2 = w2_len(C);
    for (int p = 0; p < 2; ++p) {
        const int64_t o = p ? c0 : 0;
        const int n = kNFold[p];
        int adj[kNDir];
        for (int j = 0; j < n; ++j) adj[j] = kAdj[kFoldDirs[p][j]];
        // g_psi_d = T_d^+ g_z, g_phi_b = sum_d W2[d][b]^+ g_psi_d
        DWF_TRY(launch_transport(h, nrhs, p, zo, zo, w.psi + o, adj, n, false, s));
        DWF_TRY(launch_mix(h, nrhs, p, w.psi + o, n, w.gphi + o, C, K->mix2h[p], s));
        // gW2[d][b] = sum g_psi_d phi_b^+, gW1[a][d] = sum g_phi_a R_d^+
        if (p == 0) {
            DWF_TRY((launch_wgrad<kNFold[0], 16>(h, w, nrhs, p, w.psi + o, w.phi + o, true, w.gw + n1, s)));
            DWF_TRY((launch_wgrad<16, kNFold[0]>(h, w, nrhs, p, w.gphi + o, w.R + o, false, w.gw, s)));
        } else {
            DWF_TRY((launch_wgrad<kNFold[1], 16>(h, w, nrhs, p, w.psi + o, w.phi + o, true, w.gw + n1, s)));
            DWF_TRY((launch_wgrad<16, kNFold[1]>(h, w, nrhs, p, w.gphi + o, w.R + o, false, w.gw, s)));
        }
    }
    // Adam (w1 and w2 are separate allocations: two launches over [w1 | w2])
    K->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float bc1 = 1.f - powf(b1, (float)K->adam_t), bc2 = 1.f - powf(b2, (float)K->adam_t);
    k_adam<<<(int)((n1 + 255) / 256), 256, 0, s>>>(K->d_w1, K->d_m, K->d_v, w.gw, (int)n1, (float)lr,
                                                    b1, b2, 1e-8f, bc1, bc2);
    note_launch();
    k_adam<<<(int)((n2 + 255) / 256), 256, 0, s>>>(K->d_w2, K->d_m + n1, K->d_v + n1, w.gw + n1,
                                                    (int)n2, (float)lr, b1, b2, 1e-8f, bc1, bc2);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    DWF_TRY(refresh_mix(K, s));
    DWF_CUDA(cudaStreamSynchronize(s));
    return DWF_OK;
}

// Debug/training access to the raw gradient of the last train step
// (master layout, doubles): used by the gradient parity test.
dwf_status dwf_nn_last_grad(dwf_handle* h, double* g, size_t n) {
    auto it = g_nnws.find(h);
    if (it == g_nnws.end() || it->second.gw == nullptr || !g) {
        set_error("dwf_nn_last_grad: no training step on this handle");
        return DWF_ERR_ARG;
    }
    const int C = it->second.C;
    if (n != (w1_len(C) + w2_len(C)) / 2) {
        set_error("dwf_nn_last_grad: expected %zu complex numbers", (w1_len(C) + w2_len(C)) / 2);
        return DWF_ERR_ARG;
    }
    DWF_CUDA(cudaMemcpy(g, it->second.gw, 2 * n * sizeof(double), cudaMemcpyDeviceToHost));
    return DWF_OK;
}

}  // extern "C"
