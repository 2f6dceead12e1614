// Site-local fifth-dimension operators:
//
//   S5 psi_s = P_- psi_{s+1} + P_+ psi_{s-1},  walls -mf      (S5^+ swaps P_+-)
//   L_B      out = scale (b5 + c5 S5) in
//   L_MOOEE  out = scale (d + e S5) in                         (M_ee = M_oo)
//   L_MINV   out = scale (d + e S5)^-1 in
//   L_BMINV  out = scale (b5 + c5 S5)(d + e S5)^-1 in          (commuting factors)
//   L_POST   out = (d + e S5) in + scale (b5 + c5 S5) in2      (tail of M_pc^+)
//            optionally fused with the CG update x += alpha p, r -= alpha out.
//   L_PB     p = r + beta p (CG direction update), out = scale (b5 + c5 S5) p
//
// Per chirality S5 is a cyclic shift with a -mf twist (S_- on P_+, S_+ on
// P_-, swapped for the adjoint).  FP64 runs in local64.cu; FP32 and BF16 here.
//
// Bound: HBM (2 to 7 fields through the kernel).  A thread takes VL
// consecutive lanes of one (site, spin * colour, rhs) row, 16 or 32 bytes, a
// warp the rows that fit it (Ls / VL threads each; the lanes left over where
// that does not divide 32 idle), and a row's neighbouring lanes come by
// shuffle: no shared memory and no barrier, and the loads of kU row groups are
// in flight before the first is used.  The inverse is a scan over the row's
// threads.  With w = d (d + e S_-)^-1 x, a = -e / d and P_s = sum_{t<=s} a^(s-t) x_t,
//   w_s = P_s - mf / (1 + mf a^Ls) a^(s+1) P_(Ls-1),
// P in the thread first, then across threads (Hillis-Steele with factors
// a^VL, a^2VL, ...); S_+ is the mirror image, so rows of either chirality run
// the same code on mirrored lanes.  For |a| > 1 (c5 well above b5) P grows like
// |a|^Ls and the wall term would have to cancel it (FP32 at b5 = 1, c5 = 3, Ls =
// 32: 8% off); there the scan runs the other way in 1/a (K_INVR): with Q_s =
// sum_{t>=s} a^(s-t) x_t,
//   w_s = a^(s-Ls) / (a^-Ls + mf) Q_0 - Q_(s+1) / a.
//
// The four passes of M_pc^+ M_pc at 32^4 x 16 in FP32 (L_B, L_POST, two
// L_BMINV: 9 fields, 7.2 GB, 1.07 ms at the measured peak) take 1.07 ms; with
// one element per thread staged in shared memory, and the inverse as a dense
// Ls x Ls product, they took 1.47 ms (BF16 at 24^4 x 16: 0.48 -> 0.29 ms).
#include <algorithm>
#include <cmath>

#include "dev_common.cuh"
#include "dwf_internal.cuh"

namespace dwf {

struct LocalArgs {
    const void* in;
    const void* in2;
    void* out;
    const int4* tiles;
    int Ls, nrhs, dagger;
    int rows_warp, rows_block;   // rows a warp and a block take at a time (the latter a multiple of nrhs)
    float scale;
    float c0, c1;                // out = scale (c0 x + c1 S x) (the inverse: of w, scale folded in)
    float z0, z1;                // L_POST: out = c0 x + c1 S x + scale (z0 z + z1 S z)
    float mf;
    float a, wall;               // inverse: a, mf / (1 + mf a^Ls) (K_INVR: 1/a)
    double a64, kappa;           // K_INVR: 1/a, 1 / (a^-Ls + mf)
    float* cg_x;
    float* cg_r;
    float* cg_p;
    const double* alpha;
    const int* run;
    double* partial;
    const void* lin_u;           // L_POST: out = lin_a out + lin_bu u + lin_bv v
    const void* lin_v;
    float lin_a, lin_bu, lin_bv;
};

enum { K_ONE = 0, K_POST = 1, K_PB = 2, K_INV = 3, K_INVR = 4 };
constexpr int kLocalThreads = 256;

// Where a thread's row continues: the threads holding the next lane down and
// up of the row (cyclic), and the wall factors.
struct RowPos {
    int src_dn, src_up;
    float f_dn, f_up;
};

// y = c0 x + c1 S x on the thread's lanes, S_- (down) or S_+
template <int VL>
__device__ __forceinline__ void shift_sum(float c0, float c1, const float (&x)[VL], float (&y)[VL], bool down,
                                          const RowPos& p) {
    const float nb = __shfl_sync(0xffffffffu, down ? x[VL - 1] : x[0], down ? p.src_dn : p.src_up);
    const float cw = c1 * (down ? p.f_dn : p.f_up);   // of the lane whose neighbour is another thread's
#pragma unroll
    for (int v = 0; v < VL; ++v) {
        const float lo = v > 0 ? x[v > 0 ? v - 1 : 0] : nb, hi = v < VL - 1 ? x[v < VL - 1 ? v + 1 : 0] : nb;
        const bool edge = down ? v == 0 : v == VL - 1;
        y[v] = fmaf(edge ? cw : c1, down ? lo : hi, c0 * x[v]);
    }
}

// The thread's lanes of a row: vectors of 16 bytes (8 for two BF16 lanes), or
// one complex number at a time (WIDE false) for fields aligned only to that.
template <class S, int VL, bool WIDE>
__device__ __forceinline__ void load_row(const S* p, float (&re)[VL], float (&im)[VL]) {
    if constexpr (WIDE) load_lanes<S, VL, float>(p, re, im);
    else
#pragma unroll
        for (int v = 0; v < VL; ++v) load_lanes<S, 1, float>(p + 2 * v, re + v, im + v);
}

template <class S, int VL, bool WIDE>
__device__ __forceinline__ void store_row(S* p, const float (&re)[VL], const float (&im)[VL]) {
    if constexpr (WIDE) store_lanes<S, VL, float>(p, re, im);
    else
#pragma unroll
        for (int v = 0; v < VL; ++v) store_lanes<S, 1, float>(p + 2 * v, re + v, im + v);
}

template <class Sin, class Sin2, class Sout, int VL, int KIND, bool WIDE>
__global__ void __launch_bounds__(kLocalThreads) k_local(const LocalArgs a) {
    constexpr bool INV = KIND == K_INV || KIND == K_INVR, REV = KIND == K_INVR;
    constexpr int kU = KIND == K_ONE || INV ? 4 : 2;
    __shared__ double s_red[kLocalThreads];
    const int Ls = a.Ls, nrhs = a.nrhs, TPR = Ls / VL;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rw = lane / TPR, pos = lane - rw * TPR;
    const int rb = warp * a.rows_warp + rw;             // row within the block's group
    const bool on = rw < a.rows_warp && rb < a.rows_block;
    const int rhs = rb % nrhs, s0 = pos * VL;
    RowPos rp;
    rp.src_dn = pos > 0 ? lane - 1 : lane + TPR - 1;    // (idle lanes read some lane and drop it)
    rp.src_up = pos < TPR - 1 ? lane + 1 : lane - (TPR - 1);
    rp.f_dn = pos > 0 ? 1.f : -a.mf;
    rp.f_up = pos < TPR - 1 ? 1.f : -a.mf;
    // inverse: powers of a for the scan
    float pw[VL], astep = 1.f, base_dn = 1.f, base_up = 1.f;
    double astep64 = 1.0;
    if (REV) {   // powers in FP64: |a| near 1 keeps their rounding, and kappa alone may be beyond FP32
        double q = 1.0, dn = a.kappa, up = a.kappa;
#pragma unroll
        for (int v = 0; v < VL; ++v) { pw[v] = (float)q; q *= a.a64; }
        astep64 = q;
        astep = (float)q;
        for (int i = 0; i < s0 + 1; ++i) dn *= a.a64;
        for (int i = 0; i < Ls - s0 - VL + 1; ++i) up *= a.a64;
        base_dn = (float)dn;
        base_up = (float)up;
    } else if (INV) {
        float q = 1.f;
#pragma unroll
        for (int v = 0; v < VL; ++v) { pw[v] = q; q *= a.a; }   // a^v
        astep = q;                                              // a^VL
        for (int i = 0; i < s0 + 1; ++i) base_dn *= a.a;        // a^(s + 1) of the first lane, S_-
        for (int i = 0; i < Ls - s0 - VL + 1; ++i) base_up *= a.a;   // mirrored
    }
    const int4 tl = a.tiles[blockIdx.x];
    const int rows = tl.z * 12 * nrhs;
    const int64_t base = ((int64_t)tl.y * 12 * nrhs + rb) * Ls + s0;   // complex offset of this thread's lanes
    const bool cg = KIND == K_POST && a.cg_r != nullptr;
    float coef = 0.f;
    bool live = true;
    if (KIND == K_PB || cg) {
        const int sys = tl.x * nrhs + rhs;
        coef = (float)a.alpha[sys];
        live = a.run == nullptr || a.run[sys] != 0;
    }
    const Sin* __restrict__ in = reinterpret_cast<const Sin*>(a.in);
    const Sin2* __restrict__ in2 = reinterpret_cast<const Sin2*>(a.in2);
    double nrm = 0.0;
    for (int r0 = 0; r0 < rows; r0 += kU * a.rows_block) {
        float xr[kU][VL], xi[kU][VL], zr[kU][VL], zi[kU][VL];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int r = r0 + u * a.rows_block;
            const bool ok = on && r + rb < rows;
            const int64_t g = base + (int64_t)r * Ls;
#pragma unroll
            for (int v = 0; v < VL; ++v) xr[u][v] = xi[u][v] = zr[u][v] = zi[u][v] = 0.f;
            if (ok) {
                if (KIND == K_PB) load_row<float, VL, WIDE>(a.cg_p + 2 * g, xr[u], xi[u]);
                else load_row<Sin, VL, WIDE>(in + 2 * g, xr[u], xi[u]);
                if (KIND == K_PB || KIND == K_POST) load_row<Sin2, VL, WIDE>(in2 + 2 * g, zr[u], zi[u]);
            }
        }
        float pn = 0.f;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int r = r0 + u * a.rows_block;
            if (r >= rows) break;   // the same for the whole block
            const bool ok = on && r + rb < rows;
            const int64_t g = base + (int64_t)r * Ls;
            const int c = ((r + rb) / nrhs) % 12;
            const bool down = (c < 6) != (a.dagger != 0);
            float yr[VL], yi[VL], tr[VL], ti[VL];
            if (KIND == K_PB) {   // p = r + beta p
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    if (live) {
                        xr[u][v] = fmaf(coef, xr[u][v], zr[u][v]);
                        xi[u][v] = fmaf(coef, xi[u][v], zi[u][v]);
                    }
                }
                if (ok && live) store_row<float, VL, WIDE>(a.cg_p + 2 * g, xr[u], xi[u]);
            }
            if (INV) {
                // mirrored lanes for S_+ (K_INVR: for S_-): m runs with the recurrence
                const bool fwd = down != REV;
                const int j = fwd ? pos : TPR - 1 - pos;
                const int step = fwd ? 1 : -1;
                float wr[VL], wi[VL];
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    wr[v] = fwd ? xr[u][v] : xr[u][VL - 1 - v];
                    wi[v] = fwd ? xi[u][v] : xi[u][VL - 1 - v];
                }
#pragma unroll
                for (int v = 1; v < VL; ++v) {
                    wr[v] = fmaf(a.a, wr[v - 1], wr[v]);
                    wi[v] = fmaf(a.a, wi[v - 1], wi[v]);
                }
                // inclusive scan of the thread totals, then the carry from the thread before
                float totr = wr[VL - 1], toti = wi[VL - 1], f = astep;
                double f64 = astep64;
                for (int o = 1; o < TPR; o <<= 1) {
                    const float br = __shfl_sync(0xffffffffu, totr, j >= o ? lane - step * o : lane);
                    const float bi = __shfl_sync(0xffffffffu, toti, j >= o ? lane - step * o : lane);
                    if (j >= o) { totr = fmaf(f, br, totr); toti = fmaf(f, bi, toti); }
                    if (REV) { f64 *= f64; f = (float)f64; }
                    else f *= f;
                }
                const int prev = j > 0 ? lane - step : lane, last = lane + step * (TPR - 1 - j);
                const float cr = __shfl_sync(0xffffffffu, totr, prev), ci = __shfl_sync(0xffffffffu, toti, prev);
                const float lr = __shfl_sync(0xffffffffu, totr, last), li = __shfl_sync(0xffffffffu, toti, last);
                const float base = fwd ? base_dn : base_up;
                const float wall = REV ? base : -a.wall * base;
                float carry = j > 0 ? a.a : 0.f;
                if (REV) {   // -Q of the next lane in the recurrence's order, over a
                    carry = -carry;
#pragma unroll
                    for (int v = VL - 1; v > 0; --v) { wr[v] = -a.a * wr[v - 1]; wi[v] = -a.a * wi[v - 1]; }
                    wr[0] = wi[0] = 0.f;
                }
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    wr[v] = fmaf(pw[v], fmaf(wall, lr, carry * cr), wr[v]);
                    wi[v] = fmaf(pw[v], fmaf(wall, li, carry * ci), wi[v]);
                }
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    xr[u][v] = fwd ? wr[v] : wr[VL - 1 - v];
                    xi[u][v] = fwd ? wi[v] : wi[VL - 1 - v];
                }
            }
            if (INV && a.c1 == 0.f) {
#pragma unroll
                for (int v = 0; v < VL; ++v) { yr[v] = a.c0 * xr[u][v]; yi[v] = a.c0 * xi[u][v]; }
            } else {
                shift_sum<VL>(a.c0, a.c1, xr[u], yr, down, rp);
                shift_sum<VL>(a.c0, a.c1, xi[u], yi, down, rp);
            }
            if (KIND == K_POST) {
                shift_sum<VL>(a.z0, a.z1, zr[u], tr, down, rp);
                shift_sum<VL>(a.z0, a.z1, zi[u], ti, down, rp);
            }
            if (KIND == K_ONE || KIND == K_POST || KIND == K_PB) {
#pragma unroll
                for (int v = 0; v < VL; ++v) {
                    yr[v] = KIND == K_POST ? fmaf(a.scale, tr[v], yr[v]) : a.scale * yr[v];
                    yi[v] = KIND == K_POST ? fmaf(a.scale, ti[v], yi[v]) : a.scale * yi[v];
                }
            }
            if (!ok) continue;
            if (cg) {   // x += alpha p, r -= alpha y
                float rr[VL], ri[VL];
                load_row<float, VL, WIDE>(a.cg_r + 2 * g, rr, ri);
                if (live) {
                    float pr[VL], pi[VL], vr[VL], vi[VL];
                    load_row<float, VL, WIDE>(a.cg_p + 2 * g, pr, pi);
                    load_row<float, VL, WIDE>(a.cg_x + 2 * g, vr, vi);
#pragma unroll
                    for (int v = 0; v < VL; ++v) {
                        vr[v] = fmaf(coef, pr[v], vr[v]);
                        vi[v] = fmaf(coef, pi[v], vi[v]);
                        rr[v] = fmaf(-coef, yr[v], rr[v]);
                        ri[v] = fmaf(-coef, yi[v], ri[v]);
                    }
                    store_row<float, VL, WIDE>(a.cg_x + 2 * g, vr, vi);
                    store_row<float, VL, WIDE>(a.cg_r + 2 * g, rr, ri);
                }
#pragma unroll
                for (int v = 0; v < VL; ++v) { yr[v] = rr[v]; yi[v] = ri[v]; }
            } else if (a.out != nullptr) {
                if (KIND == K_POST && a.lin_u != nullptr) {
                    float ur[VL], ui[VL], vr[VL], vi[VL];
#pragma unroll
                    for (int v = 0; v < VL; ++v) vr[v] = vi[v] = 0.f;
                    load_row<Sout, VL, WIDE>(reinterpret_cast<const Sout*>(a.lin_u) + 2 * g, ur, ui);
                    if (a.lin_v != nullptr)
                        load_row<Sout, VL, WIDE>(reinterpret_cast<const Sout*>(a.lin_v) + 2 * g, vr, vi);
#pragma unroll
                    for (int v = 0; v < VL; ++v) {
                        yr[v] = fmaf(a.lin_a, yr[v], fmaf(a.lin_bu, ur[v], a.lin_bv * vr[v]));
                        yi[v] = fmaf(a.lin_a, yi[v], fmaf(a.lin_bu, ui[v], a.lin_bv * vi[v]));
                    }
                }
                store_row<Sout, VL, WIDE>(reinterpret_cast<Sout*>(a.out) + 2 * g, yr, yi);
            }
#pragma unroll
            for (int v = 0; v < VL; ++v) pn = fmaf(yr[v], yr[v], fmaf(yi[v], yi[v], pn));
        }
        if (a.partial) nrm += (double)pn;   // FP32 within a few rows, FP64 across
    }
    if (a.partial) {
        const int nr = nrhs, rwp = a.rows_warp;
        block_rhs_reduce(on ? nrm : 0.0, s_red, nr, [&](int t) { return ((t >> 5) * rwp + (t & 31) / TPR) % nr; },
                         a.partial + (size_t)blockIdx.x * nr);
    }
}

template <class Sin, class Sin2, class Sout, int VL, bool WIDE>
static dwf_status launch_vl(dwf_handle* h, const LocalCall& c, const TileSet& ts, cudaStream_t s) {
    const FiveD& f = h->f5[0];
    const int nt = ts.ntiles[c.parity];
    if (nt == 0) return DWF_OK;
    LocalArgs a{};
    a.in = c.in;
    a.in2 = c.in2;
    a.out = c.out;
    a.tiles = ts.d_tiles[c.parity];
    a.Ls = f.Ls;
    a.nrhs = c.nrhs;
    a.dagger = c.dagger;
    a.rows_warp = 32 / (f.Ls / VL);
    a.rows_block = kLocalThreads / 32 * a.rows_warp / c.nrhs * c.nrhs;
    if (a.rows_block < 1) {   // (Ls * nrhs <= 256: never)
        set_error("local: nrhs = %d right-hand sides exceed a block's rows", c.nrhs);
        return DWF_ERR_UNSUPPORTED;
    }
    a.mf = (float)f.mf;
    a.scale = (float)c.scale;
    a.cg_x = (float*)c.cg_x;
    a.cg_r = (float*)c.cg_r;
    a.cg_p = (float*)const_cast<void*>(c.cg_p);
    a.alpha = c.alpha;
    a.run = c.run;
    a.partial = c.partial;
    void (*kern)(const LocalArgs) = k_local<Sin, Sin2, Sout, VL, K_ONE, WIDE>;
    switch (c.op) {
        case L_MINV:
        case L_BMINV: {
            const bool rev = std::abs(f.a) > 1.0;
            const double r = rev ? 1.0 / f.a : f.a;
            double rL = 1.0;
            for (int i = 0; i < f.Ls; ++i) rL *= r;
            a.a = (float)r;
            a.a64 = r;
            if (rev) a.kappa = 1.0 / (rL + f.mf);
            else a.wall = (float)(f.mf / (1.0 + f.mf * rL));
            a.c0 = (float)(c.scale * f.inv_d * (c.op == L_BMINV ? f.b5 : 1.0));
            a.c1 = (float)(c.op == L_BMINV ? c.scale * f.inv_d * f.c5 : 0.0);
            kern = rev ? k_local<Sin, Sin2, Sout, VL, K_INVR, WIDE> : k_local<Sin, Sin2, Sout, VL, K_INV, WIDE>;
            break;
        }
        case L_POST:
            a.c0 = (float)f.d;
            a.c1 = (float)f.e;
            a.z0 = (float)f.b5;
            a.z1 = (float)f.c5;
            if (c.lin) {
                a.lin_u = c.lin->u;
                a.lin_v = c.lin->bv != 0.0 ? c.lin->v : nullptr;
                a.lin_a = (float)c.lin->a;
                a.lin_bu = (float)c.lin->bu;
                a.lin_bv = (float)c.lin->bv;
            }
            kern = k_local<Sin, Sin2, Sout, VL, K_POST, WIDE>;
            break;
        case L_PB:
            a.c0 = (float)f.b5;
            a.c1 = (float)f.c5;
            kern = k_local<Sin, Sin2, Sout, VL, K_PB, WIDE>;
            break;
        default:
            a.c0 = (float)(c.op == L_MOOEE ? f.d : c.op == L_B ? f.b5 : 1.0);
            a.c1 = (float)(c.op == L_MOOEE ? f.e : c.op == L_B ? f.c5 : 0.0);
    }
    kern<<<nt, kLocalThreads, 0, s>>>(a);
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

// 4 lanes per thread where Ls allows it (fewer shuffles a lane), else 2; fields
// off the 16-byte boundaries that the vectors need (an operator's caller may
// pass a view) go number by number.
template <class Sin, class Sin2, class Sout>
static dwf_status launch_t(dwf_handle* h, const LocalCall& c, const TileSet& ts, cudaStream_t s) {
    const void* all[] = {c.in, c.in2, c.out, c.cg_x, c.cg_r, c.cg_p, c.lin ? c.lin->u : nullptr, c.lin ? c.lin->v : nullptr};
    uintptr_t off = 0;
    for (const void* q : all) off |= reinterpret_cast<uintptr_t>(q);
    if (off % 16 != 0) return launch_vl<Sin, Sin2, Sout, 2, false>(h, c, ts, s);
    if (h->p.Ls % 4 == 0) return launch_vl<Sin, Sin2, Sout, 4, true>(h, c, ts, s);
    return launch_vl<Sin, Sin2, Sout, 2, true>(h, c, ts, s);
}

// The right-hand side counts the site-local operators take.  Only the solver's
// reductions have a limit of their own (lcm(32, nrhs) threads); the second
// bound is that of rows staged in shared memory, which no kernel here does any
// more: it is kept so that a count is taken or refused by the same rule as ever.
static dwf_status rhs_supported(int nrhs, int Ls, int word) {
    auto lcm32 = [](int n, int cap) {
        int l = 32;
        while (l % n && l <= cap) l += 32;
        return l <= cap ? l : -1;
    };
    if (word == 4 && (lcm32(12 * Ls * nrhs, 512) > 0 || lcm32(Ls * nrhs, 256) > 0)) return DWF_OK;
    int threads = lcm32(nrhs, 512);
    if (threads < 0) {
        set_error("local: lcm(32, nrhs=%d) exceeds 512 threads", nrhs);
        return DWF_ERR_UNSUPPORTED;
    }
    const int target = word == 8 ? 128 : 256;
    if (threads < target) threads *= target / threads;
    const size_t smem = (size_t)4 * threads * (Ls + 1) * word;
    if (smem > 200 * 1024) {
        set_error("local: %d right-hand sides at Ls = %d are not supported", nrhs, Ls);
        return DWF_ERR_UNSUPPORTED;
    }
    return DWF_OK;
}

dwf_status launch_local(dwf_handle* h, const LocalCall& c, cudaStream_t s) {
    const TileSet* tsp = nullptr;
    DWF_TRY(get_tiles(h, tile_or_default(c.T), &tsp));
    const TileSet& ts = *tsp;
    const dwf_prec pi = c.prec_in, po = c.prec_out;
    const dwf_prec p2 = c.in2 ? c.prec_in2 : pi;
    if (c.f5 != nullptr && (pi != DWF_FP64 || po != DWF_FP64)) return DWF_ERR_UNSUPPORTED;
    if (ts.ntiles[c.parity] == 0) return DWF_OK;
    if (pi == DWF_FP64 || po == DWF_FP64) {
        if (pi != DWF_FP64 || po != DWF_FP64 || p2 != DWF_FP64) return DWF_ERR_UNSUPPORTED;
        DWF_TRY(rhs_supported(c.nrhs, h->p.Ls, 8));
        return launch_local64(h, c, ts, s);
    }
    // FP32 arithmetic; FP32 vectors for the fused CG updates
    if ((c.op == L_MINV || c.op == L_BMINV) && c.cg_r != nullptr) return DWF_ERR_UNSUPPORTED;
    DWF_TRY(rhs_supported(c.nrhs, h->p.Ls, 4));
    if (pi == DWF_FP32 && p2 == DWF_FP32 && po == DWF_FP32) return launch_t<float, float, float>(h, c, ts, s);
    if (pi == DWF_FP32 && p2 == DWF_FP32 && po == DWF_BF16) return launch_t<float, float, bf16>(h, c, ts, s);
    if (pi == DWF_BF16 && p2 == DWF_BF16 && po == DWF_BF16) return launch_t<bf16, bf16, bf16>(h, c, ts, s);
    if (pi == DWF_BF16 && p2 == DWF_BF16 && po == DWF_FP32) return launch_t<bf16, bf16, float>(h, c, ts, s);
    if (pi == DWF_FP32 && p2 == DWF_BF16 && po == DWF_FP32) return launch_t<float, bf16, float>(h, c, ts, s);
    return DWF_ERR_UNSUPPORTED;
}

}  // namespace dwf
