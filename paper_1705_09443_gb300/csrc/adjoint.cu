// Transposed preconditioner P^T = Q^T Sweep^T E^T for the adjoint solve
// A^T mu = rhs (A^T = I + omega^2 M K, the bilinear transpose of Eq. LS_d_c).
//
// Sweep^T.  Algorithm 2 applies S = (I + T N_U)^{-1} (I + T N_L)^{-1} T with
// T = blockdiag(T~_i), N_L[i,i-1] = H_{[i,i-1]}, N_U[i,i+1] = H_{[i,i+1]}, so
// S^T = T^T (I + N_L^T T^T)^{-1} (I + N_U^T T^T)^{-1}: a forward pass
// w_i = v_i - H_{[i-1,i]}^T last(T~_{i-1}^T w_{i-1}) and a backward pass
// x_i = T~_i^T (w_i - H_{[i+1,i]}^T first(x_{i+1})).  It is evaluated
// slab-parallel like the forward sweep: with a'_i = T~_i^T v_i and the maps
//   Lambda'_i = last-layer rows of T~_i^T H_{[i-1,i]}^T,  Gamma'_i = first-layer
//   rows of the same,  Phi'_i = first-layer rows of T~_i^T H_{[i+1,i]}^T,
// the coupling values obey the same three recurrences (lambda', mu', phi') and
// x_i = T~_i^T (v_i - H_{[i-1,i]}^T lambda'_{i-1} - H_{[i+1,i]}^T phi'_{i+1}).
//
// T~_i^T.  Cyclic reduction of S_i^T with the stored factors of S_i: the
// reduced blocks of S_i^T are the transposes of S_i's (lower coupling of row k:
// B_{k-1}^T, upper: C_{k+1}^T, diagonal D_k^T), so
//   level 0 forward:  y_o = D_o^{-T} b_o,  b_e -= B_{e-1}^T y_{e-1} + C_{e+1}^T y_{e+1}
//                     (level 0's stencil bands of the odd rows);
//   level l >= 1:     b_e -= (D^{-1}B)_{e-1}^T b_{e-1} + (D^{-1}C)_{e+1}^T b_{e+1},
//                     then y_o = D_o^{-T} b_o;
//   top:              x_0 = D_top^{-T} b_0;
//   backward:         x_o = y_o - D_o^{-T} (B_{o-1}^T x_{o-1} + C_{o+1}^T x_{o+1})
//                     (B, C of the even rows: level-l blocks, or level 0's bands).
// Both passes run on clusters (cr_cluster.cu).
#include <vector>

#include "cr_cluster.h"
#include "lss_common.cuh"
#include "lss_ctx.h"

namespace {

// One pass over every slab; the runs of equal block width concurrently (the
// 32-wide last slab is the longest chain of a pass).
int pass_t(lss_ctx* c, int mode, const CrcArgs& A, cudaStream_t s) {
    struct Run { int s0, n, ldw; };
    std::vector<Run> runs;
    for (int i = 0; i < c->n_slabs; ++i) {
        if (runs.empty() || c->slabs[i].ldw != runs.back().ldw) runs.push_back({i, 0, c->slabs[i].ldw});
        ++runs.back().n;
    }
    int rc = lss_ensure_aux(c, runs.size());
    if (rc) return rc;
    if (runs.size() > 1) cudaEventRecord(c->fork_event, s);
    for (size_t ri = 0; ri < runs.size() && !rc; ++ri) {
        cudaStream_t su = ri == 0 ? s : c->aux_stream[ri - 1];
        if (ri > 0) cudaStreamWaitEvent(su, c->fork_event, 0);
        rc = lss_cr_cluster(c, mode, true, A, runs[ri].s0, runs[ri].n, runs[ri].ldw, su);
        if (ri > 0) {
            cudaEventRecord(c->aux_event[ri - 1], su);
            cudaStreamWaitEvent(s, c->aux_event[ri - 1], 0);
        }
    }
    return rc;
}

// Maps of the transposed sweep, once per factorization.
template <typename T>
int build_maps_t(lss_ctx* c, cudaStream_t s) {
    using C = cx<T>;
    if (c->iface_t_valid || c->n_slabs == 1) return LSS_OK;
    // 64 bytes of slack for the recurrence's 16-byte aligned copy windows
    const size_t bytes = (size_t)3 * c->n_slabs * c->n_tot * c->n_tot * sizeof(C) + 64;
    if (!c->iface_t) {
        cudaError_t e = cudaMalloc(&c->iface_t, bytes);
        if (e) return lss_check_cuda(c, e, "transposed interface maps");
    }
    const int rc = lss_iface_maps_t(c, s);
    if (!rc) c->iface_t_valid = true;
    return rc;
}

template <typename T>
int sweep_t_impl(lss_ctx* c, const double2* y, double2* r, int R, cudaStream_t s) {
    using C = cx<T>;
    int rc = build_maps_t<T>(c, s);
    if (rc) return rc;
    const long long nt2 = (long long)c->n_tot * c->n_tot;
    const long long vec = (long long)c->n_tot * R;
    rc = lss_grow(c, &c->f_buf, &c->f_cap, (size_t)R * nt2 * sizeof(C));
    if (rc) return rc;
    rc = lss_grow(c, &c->side_buf, &c->side_cap, 4 * (size_t)c->n_slabs * vec * sizeof(C));
    if (rc) return rc;
    // Q^T reads X on the (n+2)^2 region only; slabs write every layer of their D_i
    C* side = (C*)c->side_buf;
    CrcArgs A{};
    A.R = R;
    A.yin = y;
    A.a_first = side;
    A.a_last = side + c->n_slabs * vec;
    C* lam = side + 2 * c->n_slabs * vec;
    C* phi = side + 3 * c->n_slabs * vec;
    A.lam = lam;
    A.phi = phi;
    A.X = c->f_buf;
    if (c->n_slabs > 1) {
        {
            ProfScope ps(c, s, LSS_PROF_SLAB_A, 1);
            rc = pass_t(c, CRC_A, A, s);
        }
        if (rc) return rc;
        rc = lss_recurrences(c, c->iface_t, lam, phi, A.a_first, A.a_last, R, s);
        if (rc) return rc;
    }
    {
        ProfScope ps(c, s, LSS_PROF_SLAB_E, 1);
        rc = pass_t(c, CRC_E, A, s);
    }
    if (rc) return rc;
    return lss_sparsify_t(c, c->f_buf, r, R, s);
}

}  // namespace

int lss_sweep_t(lss_ctx* c, const double2* y, double2* r, int R, cudaStream_t s) {
    return c->prec == LSS_FP64 ? sweep_t_impl<double>(c, y, r, R, s) : sweep_t_impl<float>(c, y, r, R, s);
}

int lss_prepare_sweep_t(lss_ctx* c, cudaStream_t s) {
    return c->prec == LSS_FP64 ? build_maps_t<double>(c, s) : build_maps_t<float>(c, s);
}
