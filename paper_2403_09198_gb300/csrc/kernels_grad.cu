// kernels_grad.cu -- adjoint outer products for x = J^-1 b.
//
// With lambda = J^-T g the derivative of the solve with respect to the stored
// Jacobian is dL/dJ = -lambda x^T, restricted to what is stored:
//   gS[block (i,j)][entry (p,q)] = -lambda_i[p] x_j[q]          (pattern of S_ij)
//   gU[pair of (i,j)]            = -(v . x_j) lambda_i          (column_data)
//   gV[pair of (i,j)]            = -(u . lambda_i) x_j          (row_data)
// The dots v . x_j are pass 1 of the forward matvec on x and u . lambda_i pass 1
// of the transposed matvec on lambda, so both come from the matvec kernels.
#include <cuda_runtime.h>

#include "sts_internal.h"

namespace sts {
namespace {

// lam and x are cell-major here ([cell][b]), so that a warp's entries come out of two
// rows of b values; in the internal layout every entry's factors were sectors of their
// own (S 143 us, pairs 59 us on 128 x 128 cells, N = 60; now 82 and 39).
// One warp per block, lanes over pattern entries; output in the public S layout.
__global__ void __launch_bounds__(128) k_grad_S(double *gS, const double *lam, const double *x, const long long *soff,
                                                const int *blk_row, const int *blk_col, const int *erow,
                                                const int *didx, const int *oidx, int nnzb, int nnz_d, int b) {
    const int lane = threadIdx.x & 31;
    const long long k = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (k >= nnzb) return;
    const int i = blk_row[k], j = blk_col[k];
    const bool diag = i == j;
    const long long s0 = soff[k];
    const int nnz = diag ? nnz_d : (int)(soff[k + 1] - s0);
    const int *__restrict__ rows = erow + (diag ? 0 : nnz_d);
    const int *__restrict__ cols = diag ? didx : oidx;
    const double *__restrict__ li = lam + (size_t)i * b, *__restrict__ xj = x + (size_t)j * b;
    double *__restrict__ g = gS + s0;
#pragma unroll 4
    for (int e = lane; e < nnz; e += 32) g[e] = -__ldg(li + __ldg(rows + e)) * __ldg(xj + __ldg(cols + e));
}

// One warp per pair, lanes over components.
__global__ void __launch_bounds__(128) k_grad_UV(double *gU, double *gV, const double *lam, const double *x,
                                                 const double *cN, const double *cT, const int *pair_cN,
                                                 const int *pair_cT, const int *pair_row, const int *pair_col,
                                                 int n_pairs, int b) {
    const int lane = threadIdx.x & 31;
    const long long pr = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (pr >= n_pairs) return;
    const double cu = -cN[pair_cN[pr]], cv = -cT[pair_cT[pr]];
    const double *__restrict__ li = lam + (size_t)pair_row[pr] * b, *__restrict__ xj = x + (size_t)pair_col[pr] * b;
    double *__restrict__ u = gU + pr * b, *__restrict__ v = gV + pr * b;
#pragma unroll 2
    for (int p = lane; p < b; p += 32) {
        u[p] = cu * __ldg(li + p);
        v[p] = cv * __ldg(xj + p);
    }
}

}  // namespace

sts_status grad(sts_jac_s *h, const double *lam, const double *x, double *gS, double *gU, double *gV) {
    if (!h->g_c) {
        // the transposed pair dots
        STS_TRY(dalloc(h, &h->g_c, (size_t)h->n_tiles * h->mv[1].n_dtasks * kTile + 1));
    }
    // the dots take the vectors as the matvec does; the outer products take them cell-major
    const bool comp = h->layout == STS_LAYOUT_COMPONENT_MAJOR;
    const double *lc = lam, *xc = x;
    if (comp) {
        STS_TRY(comp_to_cell64(h, lam, h->vin));
        STS_TRY(comp_to_cell64(h, x, h->vout));
        lc = h->vin;
        xc = h->vout;
        STS_TRY(mv_dots64(h, 0, Vec<double>{const_cast<double *>(x), 1, h->nc, h->nc, nullptr}, h->c64));
        STS_TRY(mv_dots64(h, 1, Vec<double>{const_cast<double *>(lam), 1, h->nc, h->nc, nullptr}, h->g_c));
    } else {
        STS_TRY(to_internal64(h, lam, h->vin));
        STS_TRY(to_internal64(h, x, h->vout));
        STS_TRY(mv_dots64(h, 0, internal_vec(h, h->vout), h->c64));     // v . x_j   (forward pass 1 on x)
        STS_TRY(mv_dots64(h, 1, internal_vec(h, h->vin), h->g_c));      // u . lambda_i (transposed pass 1 on lambda)
    }
    k_grad_S<<<(unsigned)((h->nnzb + 3) / 4), 128, 0, h->stream>>>(
        gS, lc, xc, h->d_soff, h->g_blk_row, h->g_blk_col, h->g_erow, h->mv[0].pat_idx,
        h->mv[0].pat_idx + h->nnz_d, h->nnzb, h->nnz_d, h->b);
    STS_LAUNCHED();
    if (h->n_pairs > 0) {
        k_grad_UV<<<(unsigned)(((long long)h->n_pairs + 3) / 4), 128, 0, h->stream>>>(
            gU, gV, lc, xc, h->c64, h->g_c, h->g_pair_cN, h->g_pair_cT, h->g_pair_row, h->g_pair_col, h->n_pairs, h->b);
        STS_LAUNCHED();
    }
    return STS_OK;
}

}  // namespace sts
