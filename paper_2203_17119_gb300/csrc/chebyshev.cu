// Chebyshev filter of the normal Schur operator, the recursively built filter
// functions proposed in Sec. 4 for a fast multigrid set-up of the local
// (D_Omega) solves:
//
//   out = T_n(z(A)) in,   A = M_pc^+ M_pc,   z(lam) = (hi + lo - 2 lam) / (hi - lo),
//
// by the three-term recurrence w_{k+1} = 2 z(A) w_k - w_{k-1} (w_0 = in,
// w_1 = z(A) in).  Each step is M_pc and M_pc^+ (the operator kernels, FP64 or
// FP32) with the recurrence's sum in the tail of M_pc^+; on a box handle every
// box is filtered with its own Dirichlet operator at once.
#include "dwf_internal.cuh"

namespace dwf {

dwf_status chebyshev_filter(dwf_handle* h, void* out, const void* in, int order, double lo, double hi,
                            dwf_prec prec, int nrhs, cudaStream_t s) {
    if (!h->have_gauge) {
        set_error("chebyshev: no gauge field loaded");
        return DWF_ERR_ARG;
    }
    if (out == nullptr || in == nullptr || out == in || nrhs < 1 || nrhs > h->nrhs_max || order < 0 ||
        !(hi > lo) || (prec != DWF_FP64 && prec != DWF_FP32)) {
        set_error("chebyshev: bad arguments (distinct odd cb fields, 1 <= nrhs <= nrhs_max, order >= 0, "
                  "hi > lo, FP64 or FP32)");
        return DWF_ERR_ARG;
    }
    const size_t bytes = cb_elems(h, 1, nrhs) * prec_size(prec) * 2;
    if (order == 0) {
        DWF_CUDA(cudaMemcpyAsync(out, in, bytes, cudaMemcpyDeviceToDevice, s));
        return DWF_OK;
    }
    const double c0 = (hi + lo) / (hi - lo), c1 = -2.0 / (hi - lo);
    char* scratch = nullptr;   // two fields: M_pc w_k, and every other w_k
    DWF_CUDA(dev_malloc(&scratch, 2 * bytes));
    void* u = scratch;
    void* other = scratch + bytes;
    // dst = bu src + a A src + bv v: the recurrence's sum in the tail of M_pc^+
    // (as axpby passes it took 14% of the filter)
    auto step = [&](void* dst, const void* src, double a, double bu, const void* v, double bv) -> dwf_status {
        const LinComb lin{a, src, bu, v, bv};
        DWF_TRY(op_mpc(h, u, src, 0, prec, prec, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s));
        return op_mpc(h, dst, u, 1, prec, prec, nrhs, h->d_tmp, h->d_tmp2, nullptr, nullptr, s, &lin);
    };
    auto run = [&]() -> dwf_status {
        // w_1 = c0 in + c1 A in; w_{k+1} = 2 c0 w_k + 2 c1 A w_k - w_{k-1} over
        // w_{k-1}, placed so that w_order ends in out
        void* w[2] = {order % 2 ? other : out, order % 2 ? out : other};   // w_k lives in w[k % 2]
        DWF_TRY(step(w[1], in, c1, c0, nullptr, 0.0));
        for (int k = 1; k < order; ++k)
            DWF_TRY(step(w[(k + 1) % 2], w[k % 2], 2.0 * c1, 2.0 * c0, k == 1 ? in : w[(k + 1) % 2], -1.0));
        return DWF_OK;
    };
    const dwf_status st = run();
    cudaStreamSynchronize(s);
    cudaFree(scratch);
    return st;
}

}  // namespace dwf
