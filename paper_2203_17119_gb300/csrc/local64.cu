// FP64 site-local fifth-dimension operators (the operations of local.cu).
//
// GB300 has 2 FP64 lanes per clock and SM, so these kernels are bound by the
// number of FP64 instructions, not by memory: 24^4 x 16 has 31.8 M complex
// numbers, 0.11 ms per FP64 instruction and real part against 0.075 ms per
// field of HBM traffic.  All constant factors are folded into the
// coefficients on the way in, so that per real number
//   L_B, L_MOOEE  2 (c0 x_s + c1 x_nb)          L_PB    3 (p = r + beta p first)
//   L_POST        4, with the CG update 6, with its norm 7
//   L_MINV        3, L_BMINV 4 (below).
// The kernel before this (one thread per row, recurrences in registers, 3 to 6
// per real) took 0.77 ms for L_B at 24^4 x 16, and 33 us on 4^4 x 8.
//
// Sparse operations (k_local64): one thread per complex number, the site's
// rows staged in shared memory; a thread's s and right-hand side never change
// (the active threads are a multiple of Ls * nrhs; the rest of the last warp
// idles), so its coefficients and neighbours are set up once.
//
// (d + e S)^-1 (k_minv64): with a = -e/d the scaled solution w = d (d + e S)^-1 x
// obeys w_s = x_s + a w_{s-1} (S_-; S_+ the mirror image) and
//   w_0 = [x_0 - mf sum_{t>=1} a^(Ls-t) x_t] / (1 + mf a^Ls),
// one multiply-add per element for the sum, one for the recurrence, and the
// output is c w_s or c0 w_s + c1 w_{s-1} with 1/d and the scale folded in.
// For |a| > 1 (c5 well above b5) that recurrence loses a factor |a|^Ls; it runs
// the other way there (REV), from
//   w_{Ls-1} = sum_t a^-t x_t / (a (a^-Ls + mf)),  w_{s-1} = (w_s - x_s) / a.
// A thread takes the real or the imaginary part of one row; rows lie in shared
// memory Ls + 1 complex numbers apart (Ls is even: no bank conflicts).
#include <algorithm>
#include <cmath>

#include "dev_common.cuh"
#include "dwf_internal.cuh"

namespace dwf {

struct Local64Args {
    const double2* in;
    const double2* in2;
    double2* out;
    const int4* tiles;
    int Ls, nrhs, dagger, active;
    double c0, c1;       // on x: out = c0 x + c1 S x
    double z0, z1;       // L_POST: + z0 z + z1 S z
    double mf;
    double2* cg_x;
    double2* cg_r;
    double2* cg_p;
    const double* alpha;
    const int* run;
    double* partial;
    const double2* lin_u;   // L_POST: out = lin_a out + lin_bu u + lin_bv v
    const double2* lin_v;
    double lin_a, lin_bu, lin_bv;
};

constexpr int kL64Ept = 2;   // elements per thread and chunk

enum { L64_ONE = 0, L64_POST = 1, L64_PB = 2 };

template <int KIND>
__global__ void __launch_bounds__(256) k_local64(const Local64Args a) {
    extern __shared__ __align__(16) double2 sm64[];
    __shared__ double s_red[256];
    const int Ls = a.Ls, nrhs = a.nrhs, N5 = Ls * nrhs, T = a.active, tid = threadIdx.x;
    double2* xs = sm64;
    double2* zs = sm64 + T * kL64Ept;
    const bool on = tid < T;
    const int row0 = tid / Ls, s = tid - row0 * Ls, drow = T / Ls, rhs = row0 % nrhs;
    // S_- reads s - 1 (wall -mf x_{Ls-1}), S_+ reads s + 1
    const int nb_dn = s > 0 ? -1 : Ls - 1, nb_up = s < Ls - 1 ? 1 : 1 - Ls;
    const double tw_dn = s > 0 ? 1.0 : -a.mf, tw_up = s < Ls - 1 ? 1.0 : -a.mf;
    const double c1_dn = a.c1 * tw_dn, c1_up = a.c1 * tw_up, z1_dn = a.z1 * tw_dn, z1_up = a.z1 * tw_up;
    const int4 tl = a.tiles[blockIdx.x];
    const int nel = tl.z * 12 * N5, chunk = T * kL64Ept;
    const int64_t base = (int64_t)tl.y * 12 * N5;
    const bool cg = KIND == L64_POST && a.cg_r != nullptr;
    double coef = 0.0;
    bool live = true;
    if (KIND == L64_PB || cg) {
        const int sys = tl.x * nrhs + rhs;
        coef = a.alpha[sys];
        live = a.run == nullptr || a.run[sys] != 0;
    }
    double nrm = 0.0;
    for (int ch = 0; ch < nel; ch += chunk) {
        const int64_t g0 = base + ch + tid;
        double2 v[kL64Ept], w[kL64Ept];
        if (ch > 0) __syncthreads();   // the previous chunk is no longer read
#pragma unroll
        for (int j = 0; j < kL64Ept; ++j)
            if (on && ch + tid + j * T < nel) {
                const int64_t g = g0 + (int64_t)j * T;
                v[j] = KIND == L64_PB ? a.cg_p[g] : a.in[g];
                if (KIND != L64_ONE) w[j] = a.in2[g];
            }
#pragma unroll
        for (int j = 0; j < kL64Ept; ++j)
            if (on && ch + tid + j * T < nel) {
                if (KIND == L64_PB && live) {   // p = r + beta p
                    v[j] = make_double2(fma(coef, v[j].x, w[j].x), fma(coef, v[j].y, w[j].y));
                    a.cg_p[g0 + (int64_t)j * T] = v[j];
                }
                xs[tid + j * T] = v[j];
                if (KIND == L64_POST) zs[tid + j * T] = w[j];
            }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kL64Ept; ++j) {
            if (!on || ch + tid + j * T >= nel) continue;
            const int64_t g = g0 + (int64_t)j * T;
            const int c = ((ch / Ls + row0 + j * drow) / nrhs) % 12;
            const bool down = (c < 6) != (a.dagger != 0);   // S_- (else S_+)
            const int nb = tid + j * T + (down ? nb_dn : nb_up);
            const double c1 = down ? c1_dn : c1_up;
            const double2 xn = xs[nb];
            double yr = fma(c1, xn.x, a.c0 * v[j].x), yi = fma(c1, xn.y, a.c0 * v[j].y);
            if (KIND == L64_POST) {
                const double z1 = down ? z1_dn : z1_up;
                const double2 zn = zs[nb];
                yr = fma(z1, zn.x, fma(a.z0, w[j].x, yr));
                yi = fma(z1, zn.y, fma(a.z0, w[j].y, yi));
            }
            if (cg) {   // x += alpha p, r -= alpha y
                double2 r = a.cg_r[g];
                if (live) {
                    const double2 p = a.cg_p[g];
                    double2 x = a.cg_x[g];
                    x.x = fma(coef, p.x, x.x);
                    x.y = fma(coef, p.y, x.y);
                    r.x = fma(-coef, yr, r.x);
                    r.y = fma(-coef, yi, r.y);
                    a.cg_x[g] = x;
                    a.cg_r[g] = r;
                }
                yr = r.x;
                yi = r.y;
            } else if (a.out != nullptr) {
                if (KIND == L64_POST && a.lin_u != nullptr) {
                    const double2 u = a.lin_u[g], v = a.lin_v != nullptr ? a.lin_v[g] : make_double2(0.0, 0.0);
                    yr = fma(a.lin_a, yr, fma(a.lin_bu, u.x, a.lin_bv * v.x));
                    yi = fma(a.lin_a, yi, fma(a.lin_bu, u.y, a.lin_bv * v.y));
                }
                a.out[g] = make_double2(yr, yi);
            }
            if (a.partial) nrm = fma(yr, yr, fma(yi, yi, nrm));
        }
    }
    if (a.partial) {
        const int nr = nrhs;
        __syncthreads();
        block_rhs_reduce(on ? nrm : 0.0, s_red, nr, [&](int t) { return (t / Ls) % nr; },
                         a.partial + (size_t)blockIdx.x * nr);
    }
}

struct Minv64Args {
    const double2* in;
    double2* out;
    const int4* tiles;
    int Ls, nrhs, dagger;
    double a, mf, wall;   // wall = 1 / (1 + mf a^Ls); REV: a is 1/a, wall = a / (a^Ls + mf) with that a
    double c0, c1;        // out = c0 w_s + c1 w_{s -+ 1}
};

constexpr int kM64Rows = 64;

template <bool B, bool REV>
__global__ void __launch_bounds__(2 * kM64Rows) k_minv64(const Minv64Args a) {
    extern __shared__ __align__(16) double2 sm64[];
    const int Ls = a.Ls, nrhs = a.nrhs, stride = Ls + 1, tid = threadIdx.x;
    const int4 tl = a.tiles[blockIdx.x];
    const int rows = tl.z * 12 * nrhs;
    const int64_t base = (int64_t)tl.y * 12 * nrhs * Ls;
    const int row = tid >> 1;
    double* part = reinterpret_cast<double*>(sm64) + (size_t)row * stride * 2 + (tid & 1);
    for (int rb = 0; rb < rows; rb += kM64Rows) {
        const int n = min(kM64Rows, rows - rb);
        const double2* in = a.in + base + (int64_t)rb * Ls;
        if (rb > 0) __syncthreads();
        for (int e = tid; e < n * Ls; e += blockDim.x) sm64[e + e / Ls] = in[e];
        __syncthreads();
        if (row < n) {
            const int c = ((rb + row) / nrhs) % 12;
            const bool down = (c < 6) != (a.dagger != 0);
            // S_-: first = 0, upwards; S_+: first = Ls - 1, downwards
            const int first = down ? 0 : 2 * (Ls - 1), st = down ? 2 : -2;
            double acc = 0.0;
            if (REV) {
                const int last = first + (Ls - 1) * st;
                for (int k = 0; k < Ls; ++k) acc = fma(acc, a.a, part[last - k * st]);
                const double top = a.wall * acc;
                double w = top;
                for (int k = 0; k < Ls - 1; ++k) {
                    const int i = last - k * st;
                    const double wn = a.a * (w - part[i]);
                    part[i] = B ? fma(a.c1, wn, a.c0 * w) : a.c0 * w;
                    w = wn;
                }
                part[first] = B ? fma(a.c1 * -a.mf, top, a.c0 * w) : a.c0 * w;
            } else {
                for (int k = 1; k < Ls; ++k) acc = fma(acc, a.a, part[first + k * st]);
                const double w0 = fma(-a.mf * a.a, acc, part[first]) * a.wall;
                double w = w0;
                for (int k = 1; k < Ls; ++k) {
                    const int i = first + k * st;
                    const double wn = fma(a.a, w, part[i]);
                    part[i] = B ? fma(a.c1, w, a.c0 * wn) : a.c0 * wn;
                    w = wn;
                }
                // S w at the first lane: -mf times the last one
                part[first] = B ? fma(a.c1 * -a.mf, w, a.c0 * w0) : a.c0 * w0;
            }
        }
        __syncthreads();
        double2* out = a.out + base + (int64_t)rb * Ls;
        for (int e = tid; e < n * Ls; e += blockDim.x) out[e] = sm64[e + e / Ls];
    }
}

dwf_status launch_local64(dwf_handle* h, const LocalCall& c, const TileSet& ts, cudaStream_t s) {
    const FiveD& f = c.f5 ? *c.f5 : h->f5[0];
    const int nt = ts.ntiles[c.parity];
    if (nt == 0) return DWF_OK;
    const int Ls = h->p.Ls, N5 = Ls * c.nrhs;
    if (c.op == L_MINV || c.op == L_BMINV) {
        Minv64Args a{};
        a.in = (const double2*)c.in;
        a.out = (double2*)c.out;
        a.tiles = ts.d_tiles[c.parity];
        a.Ls = Ls;
        a.nrhs = c.nrhs;
        a.dagger = c.dagger;
        const bool rev = std::abs(f.a) > 1.0;
        a.a = f.a;
        a.mf = f.mf;
        a.wall = f.inv_den * f.d;
        if (rev) {
            a.a = 1.0 / f.a;
            double rL = 1.0;
            for (int i = 0; i < Ls; ++i) rL *= a.a;
            a.wall = a.a / (rL + f.mf);
        }
        a.c0 = c.scale * f.inv_d * (c.op == L_BMINV ? f.b5 : 1.0);
        a.c1 = c.op == L_BMINV ? c.scale * f.inv_d * f.c5 : 0.0;
        if (c.partial != nullptr || c.out == nullptr || c.cg_r != nullptr) {
            set_error("local: the FP64 inverse writes its result, without norms or CG updates");
            return DWF_ERR_UNSUPPORTED;
        }
        const size_t smem = (size_t)kM64Rows * (Ls + 1) * sizeof(double2);
        void (*kern)(const Minv64Args) = c.op == L_BMINV ? (rev ? k_minv64<true, true> : k_minv64<true, false>)
                                                         : (rev ? k_minv64<false, true> : k_minv64<false, false>);
        kern<<<nt, 2 * kM64Rows, smem, s>>>(a);
    } else {
        Local64Args a{};
        a.in = (const double2*)c.in;
        a.in2 = (const double2*)c.in2;
        a.out = (double2*)c.out;
        a.tiles = ts.d_tiles[c.parity];
        a.Ls = Ls;
        a.nrhs = c.nrhs;
        a.dagger = c.dagger;
        a.active = std::max(1, 256 / N5) * N5;
        a.mf = f.mf;
        a.cg_x = (double2*)c.cg_x;
        a.cg_r = (double2*)c.cg_r;
        a.cg_p = (double2*)const_cast<void*>(c.cg_p);
        a.alpha = c.alpha;
        a.run = c.run;
        a.partial = c.partial;
        const int threads = (a.active + 31) / 32 * 32;
        const size_t plane = (size_t)a.active * kL64Ept * sizeof(double2);
        switch (c.op) {
            case L_POST:
                a.c0 = f.d;
                a.c1 = f.e;
                a.z0 = c.scale * f.b5;
                a.z1 = c.scale * f.c5;
                if (c.lin) {
                    a.lin_u = (const double2*)c.lin->u;
                    a.lin_v = c.lin->bv != 0.0 ? (const double2*)c.lin->v : nullptr;
                    a.lin_a = c.lin->a;
                    a.lin_bu = c.lin->bu;
                    a.lin_bv = c.lin->bv;
                }
                k_local64<L64_POST><<<nt, threads, 2 * plane, s>>>(a);
                break;
            case L_PB:
                a.c0 = c.scale * f.b5;
                a.c1 = c.scale * f.c5;
                k_local64<L64_PB><<<nt, threads, plane, s>>>(a);
                break;
            default:
                a.c0 = c.scale * (c.op == L_MOOEE ? f.d : c.op == L_B ? f.b5 : 1.0);
                a.c1 = c.scale * (c.op == L_MOOEE ? f.e : c.op == L_B ? f.c5 : 0.0);
                k_local64<L64_ONE><<<nt, threads, plane, s>>>(a);
        }
    }
    note_launch();
    DWF_CUDA(cudaGetLastError());
    return DWF_OK;
}

}  // namespace dwf
