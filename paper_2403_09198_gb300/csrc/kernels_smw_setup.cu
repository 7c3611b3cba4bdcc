// kernels_smw_setup.cu -- block-Jacobi setup (Section 6; see kernels_smw.cu for
// the method and the apply).  Lane or thread = cell throughout:
//   LU of A_k^0 without pivoting (natural order; for the paper's arrow pattern
//   there is no fill), one lane per cell;
//   W_k = (A_k^0)^-1 U_k   (SMW-1, r sparse solves), one lane per solve;
//   C_k = I + V_k^T W_k    (FP64), one thread per entry; C_k^-1 by Gauss-Jordan
//   with pivoting, one lane per cell; then the apply streams are packed.
// The paper's pattern family has its own LU and solve kernels (arithmetic
// indices, sliding register windows); any other pattern runs the schedule tables.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "sts_internal.h"

namespace sts {
namespace {

struct SetupArgs {
    const double *Sd, *Ud, *Vd;
    double *lu, *dinv, *W, *Wt, *Cinv;
    const int *lu_diag, *src_slot, *d_ptr;
    const int *colL_ptr, *colL_slot, *upd_ptr, *upd_tgt, *upd_src;
    const int *fwd_ptr0, *fwd_col0, *fwd_slot0, *bwd_ptr0, *bwd_col0, *bwd_slot0;
    const int *fwd_ptr1, *fwd_col1, *fwd_slot1, *bwd_ptr1, *bwd_col1, *bwd_slot1;
    int *err_cell;
    int nc, ncp, b, r, nnz_lu, nnz_d, with_T;
};

// Solve A0 w = rhs in place on w[q * ncp + cell] (column of W), N direction.
__device__ void lu_solve_N(const SetupArgs &a, double *w, int cell) {
    const size_t P = a.ncp;
    for (int i = 0; i < a.b; ++i) {
        double acc = w[i * P + cell];
        for (int e = a.fwd_ptr0[i]; e < a.fwd_ptr0[i + 1]; ++e)
            acc = fma(-a.lu[(size_t)a.fwd_slot0[e] * P + cell], w[(size_t)a.fwd_col0[e] * P + cell], acc);
        w[i * P + cell] = acc;
    }
    for (int r = 0; r < a.b; ++r) {
        const int i = a.b - 1 - r;
        double acc = w[i * P + cell];
        for (int e = a.bwd_ptr0[r]; e < a.bwd_ptr0[r + 1]; ++e)
            acc = fma(-a.lu[(size_t)a.bwd_slot0[e] * P + cell], w[(size_t)a.bwd_col0[e] * P + cell], acc);
        w[i * P + cell] = acc * a.dinv[i * P + cell];
    }
}

// Solve A0^T w = rhs in place: U^T (forward, with the pivots), then L^T (unit).
__device__ void lu_solve_T(const SetupArgs &a, double *w, int cell) {
    const size_t P = a.ncp;
    for (int i = 0; i < a.b; ++i) {
        double acc = w[i * P + cell];
        for (int e = a.fwd_ptr1[i]; e < a.fwd_ptr1[i + 1]; ++e)
            acc = fma(-a.lu[(size_t)a.fwd_slot1[e] * P + cell], w[(size_t)a.fwd_col1[e] * P + cell], acc);
        w[i * P + cell] = acc * a.dinv[i * P + cell];
    }
    for (int r = 0; r < a.b; ++r) {
        const int i = a.b - 1 - r;
        double acc = w[i * P + cell];
        for (int e = a.bwd_ptr1[r]; e < a.bwd_ptr1[r + 1]; ++e)
            acc = fma(-a.lu[(size_t)a.bwd_slot1[e] * P + cell], w[(size_t)a.bwd_col1[e] * P + cell], acc);
        w[i * P + cell] = acc;
    }
}

// Setup step 1, one thread per cell: the static-pivot LU of S_kk on the shared
// schedule.  A padding cell gets the identity, so steps 2 and 3 give it W = 0 and
// C^-1 = I without a special case.
__global__ void k_smw_lu(SetupArgs a) {
    const int cell = blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= a.ncp) return;
    const size_t P = a.ncp;
    for (int s = 0; s < a.nnz_lu; ++s) a.lu[s * P + cell] = 0.0;
    if (cell >= a.nc) {
        for (int i = 0; i < a.b; ++i) {
            a.lu[(size_t)a.lu_diag[i] * P + cell] = 1.0;
            a.dinv[i * P + cell] = 1.0;
        }
        return;
    }
    for (int e = 0; e < a.nnz_d; ++e) a.lu[(size_t)a.src_slot[e] * P + cell] = a.Sd[e * P + cell];
    for (int k = 0; k < a.b; ++k) {
        double rowmax = 0.0;
        for (int e = a.d_ptr[k]; e < a.d_ptr[k + 1]; ++e) rowmax = fmax(rowmax, fabs(a.Sd[e * P + cell]));
        const double piv = a.lu[(size_t)a.lu_diag[k] * P + cell];
        if (!(fabs(piv) > 1e-14 * rowmax)) {
            atomicMin(a.err_cell, cell);
            return;
        }
        const double d = 1.0 / piv;
        a.dinv[k * P + cell] = d;
        for (int e = a.colL_ptr[k]; e < a.colL_ptr[k + 1]; ++e) {
            const size_t sl = (size_t)a.colL_slot[e] * P + cell;
            const double l = a.lu[sl] * d;
            a.lu[sl] = l;
            for (int u = a.upd_ptr[e]; u < a.upd_ptr[e + 1]; ++u)
                a.lu[(size_t)a.upd_tgt[u] * P + cell] =
                    fma(-l, a.lu[(size_t)a.upd_src[u] * P + cell], a.lu[(size_t)a.upd_tgt[u] * P + cell]);
        }
    }
}

// Setup step 2, one thread per (cell, pair k, direction): W_k = A0^-1 U_k (SMW-1)
// and, for the adjoint, Wt_k = A0^-T V_k.  Consecutive threads take consecutive
// cells, so every [slot][cell] access of a warp is one coalesced request.
__global__ void k_smw_w(SetupArgs a) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long per_dir = (long long)a.ncp * a.r;
    if (t >= per_dir * (a.with_T ? 2 : 1)) return;
    const int dir = (int)(t / per_dir);
    const long long u = t - dir * per_dir;
    const int k = (int)(u / a.ncp), cell = (int)(u - (long long)k * a.ncp);
    const size_t P = a.ncp;
    double *w = (dir ? a.Wt : a.W) + (size_t)k * a.b * P;
    const double *src = (dir ? a.Vd : a.Ud) + (size_t)k * a.b * P;
    for (int q = 0; q < a.b; ++q) w[q * P + cell] = src[q * P + cell];
    if (dir) lu_solve_T(a, w, cell);
    else lu_solve_N(a, w, cell);
}

// Setup step 3a, one thread per (cell, k, l): C_kl = delta_kl + V_k . W_l (FP64),
// written into the C^-1 array, which step 3b inverts in place.
__global__ void k_smw_cmat(SetupArgs a) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int r = a.r;
    if (t >= (long long)a.ncp * r * r) return;
    const int kl = (int)(t / a.ncp), cell = (int)(t - (long long)kl * a.ncp);
    const int k = kl / r, l = kl - k * r;
    const size_t P = a.ncp;
    const double *v = a.Vd + (size_t)k * a.b * P + cell, *w = a.W + (size_t)l * a.b * P + cell;
    double acc = k == l ? 1.0 : 0.0;
    for (int q = 0; q < a.b; ++q) acc = fma(v[q * P], w[q * P], acc);
    a.Cinv[(size_t)kl * P + cell] = acc;
}

// Setup step 3b, one thread per cell: C^-1 by Gauss-Jordan with partial pivoting,
// in place in the C^-1 array.
__global__ void k_smw_cinv(SetupArgs a) {
    const int cell = blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= a.ncp) return;
    const size_t P = a.ncp;
    const int r = a.r;
    double C[kMaxPairsDiag][kMaxPairsDiag], X[kMaxPairsDiag][kMaxPairsDiag];
    double cmax = 0.0;
    for (int k = 0; k < r; ++k)
        for (int l = 0; l < r; ++l) {
            C[k][l] = a.Cinv[((size_t)k * r + l) * P + cell];
            X[k][l] = k == l ? 1.0 : 0.0;
            cmax = fmax(cmax, fabs(C[k][l]));
        }
    for (int k = 0; k < r; ++k) {
        int pr = k;
        for (int i = k + 1; i < r; ++i)
            if (fabs(C[i][k]) > fabs(C[pr][k])) pr = i;
        if (!(fabs(C[pr][k]) > 1e-14 * cmax)) {
            atomicMin(a.err_cell, cell);
            return;
        }
        if (pr != k)
            for (int j = 0; j < r; ++j) {
                double t = C[k][j]; C[k][j] = C[pr][j]; C[pr][j] = t;
                t = X[k][j]; X[k][j] = X[pr][j]; X[pr][j] = t;
            }
        const double d = 1.0 / C[k][k];
        for (int j = 0; j < r; ++j) { C[k][j] *= d; X[k][j] *= d; }
        for (int i = 0; i < r; ++i) {
            if (i == k) continue;
            const double f = C[i][k];
            for (int j = 0; j < r; ++j) { C[i][j] -= f * C[k][j]; X[i][j] -= f * X[k][j]; }
        }
    }
    for (int k = 0; k < r; ++k)
        for (int l = 0; l < r; ++l) a.Cinv[((size_t)k * r + l) * P + cell] = X[k][l];
}

// ---------------------------------------------------------------------------
// Setup for the paper's pattern family (level band of half-width W plus NF = 3
// dense flow rows and columns).  Its LU has no fill, so LU slot e is pattern
// entry e and every index is arithmetic: the kernels below do the general
// kernels' operations in the same order, with the active window of the
// factorisation (or of a solve) in registers and the next rows' entries loaded
// ahead, where the general ones chase schedule tables through global memory.

// First slot of pattern row p: level rows hold the clipped band and NF columns.
template <int W>
__device__ __forceinline__ int arrow_row(int p, int N, int b) {
    constexpr int NF = kStructNF;
    const int l = min(p, N);
    const int lo = l >= W ? W * (W + 1) / 2 : l * W - l * (l - 1) / 2;       // clipped below column 0
    const int t = max(l - (N - W), 0);                                       // rows clipped above column N - 1
    return l * (2 * W + 1 + NF) - lo - t * (t + 1) / 2 + (p > N ? (p - N) * b : 0);
}
template <int W>
__device__ __forceinline__ size_t arrow_slot(int p, int q, int N, int b) {   // (p, q) with p < N, |p - q| <= W, or p >= N
    return (size_t)(arrow_row<W>(p, N, b) + (p < N ? q - max(p - W, 0) : q));
}
template <int W>
__device__ __forceinline__ size_t arrow_fcol(int p, int f, int N, int b) {   // (p, N + f) with p < N
    return (size_t)(arrow_row<W>(p + 1, N, b) - kStructNF + f);
}

// max(m, |v|) with fmax's treatment of NaN, as integers: an FP64 comparison
// takes an FP64 pipe slot.
__device__ __forceinline__ long long abs_max(long long m, double v) {
    const long long k = __double_as_longlong(v) & 0x7fffffffffffffffll;
    return k <= 0x7ff0000000000000ll && k > m ? k : m;
}
// |piv| > 1e-14 * rowmax, decided on the exponents where they differ by 44 or less
__device__ __forceinline__ bool pivot_ok(double piv, long long rowmax) {
    const int ep = (__double2hiint(piv) >> 20) & 0x7ff, er = (int)(rowmax >> 52);
    if (ep != 0x7ff && er != 0x7ff && ep >= 1 && ep >= er - 44) return true;
    return fabs(piv) > 1e-14 * __longlong_as_double(rowmax);
}

// Static-pivot LU, one lane per cell and one warp per tile of 32 cells.  The
// window holds rows and columns k .. k + W of the band (A), the window rows' flow
// columns (B), the flow rows' window columns (C) and the flow block (D); column k
// costs (W + 3)^2 FMAs, W + 3 products and one reciprocal, about 41 FP64
// instructions at W = 2, which bound the kernel (one warp per sub-partition at
// 128 x 128 cells).  Entry n of the band arrives one column ahead.  Measured on
// 128 x 128 cells, N = 60, W = 2: 939 us for the schedule tables, 164 us here, of which
// 75 us are FP64 pipe time; the rest is one warp's other instructions, which do not
// overlap its FP64 ones.
template <int W>
__global__ void __launch_bounds__(kTile) k_smw_lu_arrow(SetupArgs a) {
    constexpr int NF = kStructNF;
    const int lane = threadIdx.x, cell = blockIdx.x * kTile + lane;
    const size_t P = a.ncp;
    const int b = a.b, N = b - NF;
    const bool pad = cell >= a.nc;                    // padding cells (S = 0) get the identity
    const double *__restrict__ S = a.Sd + cell;
    double *__restrict__ lu = a.lu + cell;
    double A[W + 1][W + 1], B[W + 1][NF], C[NF][W + 1], D[NF][NF];
    long long rm[W + 1], rf[NF];
    // band row n: columns n - W .. n; band column n: rows n - W .. n - 1; flow columns and rows
    double nl[W + 1], nu[W > 0 ? W : 1], nb[NF], nc[NF];
    // rs[i]: first slot of row n - W + i; fr[f]: of flow row N + f.  Running sums of the row lengths
    int rs[W + 2], fr[NF];
    auto row_len = [&](int p) { return p < N ? min(N - 1, p + W) - max(0, p - W) + 1 + NF : 0; };
    auto fetch = [&](int n, const int *r) {           // r[i]: first slot of row n - W + i
        const bool on = n < N;
#pragma unroll
        for (int j = 0; j <= W; ++j) {
            const int q = n - W + j;
            nl[j] = on && q >= 0 ? __ldg(S + (size_t)(r[W] + min(n, W) - W + j) * P) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const int p = n - W + i;
            nu[i] = on && p >= 0 ? __ldg(S + (size_t)(r[i] + n - max(p - W, 0)) * P) : 0.0;
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            nb[f] = on ? __ldg(S + (size_t)(r[W + 1] - NF + f) * P) : 0.0;
            nc[f] = on ? __ldg(S + (size_t)(fr[f] + n) * P) : 0.0;
        }
        if (pad) nl[W] = 1.0;
    };
    // shift the window by one row and column and take entry n in as its last
    auto ingest = [&]() {
#pragma unroll
        for (int i = 0; i < W; ++i) {
#pragma unroll
            for (int j = 0; j < W; ++j) A[i][j] = A[i + 1][j + 1];
#pragma unroll
            for (int f = 0; f < NF; ++f) B[i][f] = B[i + 1][f];
#pragma unroll
            for (int f = 0; f < NF; ++f) C[f][i] = C[f][i + 1];
            rm[i] = abs_max(rm[i + 1], nu[i]);
            A[i][W] = nu[i];
        }
        long long m = 0;
#pragma unroll
        for (int j = 0; j <= W; ++j) {
            A[W][j] = nl[j];
            m = abs_max(m, nl[j]);
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            B[W][f] = nb[f];
            m = abs_max(m, nb[f]);
            C[f][W] = nc[f];
            rf[f] = abs_max(rf[f], nc[f]);
        }
        rm[W] = m;
    };
#pragma unroll
    for (int i = 0; i <= W; ++i) {
        rm[i] = 0;
#pragma unroll
        for (int j = 0; j <= W; ++j) A[i][j] = 0.0;
#pragma unroll
        for (int f = 0; f < NF; ++f) B[i][f] = C[f][i] = 0.0;
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        rf[f] = 0;
#pragma unroll
        for (int g = 0; g < NF; ++g) {
            D[f][g] = pad ? (f == g ? 1.0 : 0.0) : __ldg(S + arrow_slot<W>(N + f, N + g, N, b) * P);
            rf[f] = abs_max(rf[f], D[f][g]);
        }
    }
#pragma unroll
    for (int i = 0; i <= W; ++i) rs[i] = 0;
    rs[W + 1] = row_len(0);
#pragma unroll
    for (int f = 0; f < NF; ++f) fr[f] = arrow_row<W>(N + f, N, b);
    auto advance = [&](int n) {                       // rs for row n
#pragma unroll
        for (int i = 0; i <= W; ++i) rs[i] = rs[i + 1];
        rs[W + 1] += row_len(n);
    };
    fetch(0, rs);
    for (int n = 0; n < W; ++n) {
        ingest();
        advance(n + 1);
        fetch(n + 1, rs);
    }
    bool ok = true;
    for (int k = 0; k < N; ++k) {
        ingest();
        int r0[W + 2];                                // first slots of rows k .. k + W + 1
#pragma unroll
        for (int i = 0; i <= W + 1; ++i) r0[i] = rs[i];
        advance(k + 1 + W);
        if (k + 1 < N) fetch(k + 1 + W, rs);
        const double piv = A[0][0];
        ok = ok && pivot_ok(piv, rm[0]);
        const double d = 1.0 / piv;
        const int nj = min(W, N - 1 - k);
        double *urow = lu + (size_t)(r0[0] + min(k, W)) * P;         // (k, k)
#pragma unroll
        for (int j = 0; j <= W; ++j)
            if (j <= nj) urow[j * P] = A[0][j];
        double *ucol = lu + (size_t)(r0[1] - NF) * P;                // (k, N)
#pragma unroll
        for (int f = 0; f < NF; ++f) ucol[f * P] = B[0][f];
        double l[W + NF];
#pragma unroll
        for (int i = 1; i <= W; ++i) {
            l[i - 1] = A[i][0] * d;
#pragma unroll
            for (int j = 1; j <= W; ++j) A[i][j] = fma(-l[i - 1], A[0][j], A[i][j]);
#pragma unroll
            for (int f = 0; f < NF; ++f) B[i][f] = fma(-l[i - 1], B[0][f], B[i][f]);
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            l[W + f] = C[f][0] * d;
#pragma unroll
            for (int j = 1; j <= W; ++j) C[f][j] = fma(-l[W + f], A[0][j], C[f][j]);
#pragma unroll
            for (int g = 0; g < NF; ++g) D[f][g] = fma(-l[W + f], B[0][g], D[f][g]);
        }
        // the column's results last: a store that waits on a fresh FP64 result holds the warp
        a.dinv[(size_t)k * P + cell] = d;
#pragma unroll
        for (int i = 1; i <= W; ++i)
            if (i <= nj) lu[(size_t)(r0[i] + k - max(k + i - W, 0)) * P] = l[i - 1];
#pragma unroll
        for (int f = 0; f < NF; ++f) lu[(size_t)(fr[f] + k) * P] = l[W + f];
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        ok = ok && pivot_ok(D[k][k], rf[k]);
        const double d = 1.0 / D[k][k];
        a.dinv[(size_t)(N + k) * P + cell] = d;
#pragma unroll
        for (int f = k + 1; f < NF; ++f) {
            D[f][k] *= d;
#pragma unroll
            for (int g = k + 1; g < NF; ++g) D[f][g] = fma(-D[f][k], D[k][g], D[f][g]);
        }
    }
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int g = 0; g < NF; ++g) lu[arrow_slot<W>(N + f, N + g, N, b) * P] = D[f][g];
    if (!ok) atomicMin(a.err_cell, cell);
}

// W_k = A0^-1 U_k (DIR 0) or Wt_k = A0^-T V_k (DIR 1), one warp per (tile, pair,
// direction), lane = cell.  The band recurrences keep their last W values in
// registers and the flow rows accumulate beside them, so a row is W + 3 FMAs in
// each sweep; rows are taken U at a time with the next U rows' coefficients
// loaded ahead.  Bound by the FP64 pipe once a sub-partition holds a few warps.
// Measured on 128 x 128 cells, N = 60, W = 2: nine pairs 300 -> 201 us (FP64 pipe
// busy 77% of it), two pairs in both directions 302 -> 114 us.
template <int W, int DIR>
__device__ __forceinline__ void arrow_solve(const SetupArgs &a, const double *src, double *w, int cell) {
    constexpr int NF = kStructNF, U = W <= 2 ? 4 : 2, R = W + NF;
    const size_t P = a.ncp;
    const int b = a.b, N = b - NF;
    const double *__restrict__ lu = a.lu + cell;
    const double *__restrict__ dinv = a.dinv + cell;
    // coefficient of the lower (i > j) and upper (i < j) factor of this direction
    auto lo_band = [&](int i, int j) { return __ldg(lu + (DIR == 0 ? arrow_slot<W>(i, j, N, b) : arrow_slot<W>(j, i, N, b)) * P); };
    auto lo_flow = [&](int f, int j) { return __ldg(lu + (DIR == 0 ? arrow_slot<W>(N + f, j, N, b) : arrow_fcol<W>(j, f, N, b)) * P); };
    auto up_flow = [&](int i, int f) { return __ldg(lu + (DIR == 0 ? arrow_fcol<W>(i, f, N, b) : arrow_slot<W>(N + f, i, N, b)) * P); };
    auto ff = [&](int f, int g) { return __ldg(lu + arrow_slot<W>(N + (DIR == 0 ? f : g), N + (DIR == 0 ? g : f), N, b) * P); };
    double c[U][R], v[U], s[U], cn[U][R], vn[U], sn[U];
    // ---- forward: rows i = 0 .. N-1
    auto load_f = [&](int i0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u;
            if (i < N) {
#pragma unroll
                for (int k = 0; k < W; ++k) cn[u][k] = i - W + k >= 0 ? lo_band(i, i - W + k) : 0.0;
#pragma unroll
                for (int f = 0; f < NF; ++f) cn[u][W + f] = lo_flow(f, i);
                vn[u] = __ldg(src + (size_t)i * P + cell);
                sn[u] = DIR == 1 ? __ldg(dinv + (size_t)i * P) : 1.0;
            }
        }
    };
    auto take = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int k = 0; k < R; ++k) c[u][k] = cn[u][k];
            v[u] = vn[u];
            s[u] = sn[u];
        }
    };
    double win[W > 0 ? W : 1], acf[NF];
#pragma unroll
    for (int k = 0; k < W; ++k) win[k] = 0.0;
#pragma unroll
    for (int f = 0; f < NF; ++f) acf[f] = __ldg(src + (size_t)(N + f) * P + cell);
    load_f(0);
    for (int i0 = 0; i0 < N; i0 += U) {
        take();
        if (i0 + U < N) load_f(i0 + U);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u >= N) break;
            double acc = v[u];
#pragma unroll
            for (int k = 0; k < W; ++k) acc = fma(-c[u][k], win[k], acc);
            if (DIR == 1) acc *= s[u];
            w[(size_t)(i0 + u) * P + cell] = acc;
#pragma unroll
            for (int f = 0; f < NF; ++f) acf[f] = fma(-c[u][W + f], acc, acf[f]);
#pragma unroll
            for (int k = 0; k + 1 < W; ++k) win[k] = win[k + 1];
            if (W > 0) win[W > 0 ? W - 1 : 0] = acc;
        }
    }
    // ---- flow rows, forward then backward
    double xf[NF], df[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) df[f] = __ldg(dinv + (size_t)(N + f) * P);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        xf[f] = acf[f];
#pragma unroll
        for (int g = 0; g < f; ++g) xf[f] = fma(-ff(f, g), xf[g], xf[f]);
        if (DIR == 1) xf[f] *= df[f];
    }
#pragma unroll
    for (int f = NF - 1; f >= 0; --f) {
#pragma unroll
        for (int g = f + 1; g < NF; ++g) xf[f] = fma(-ff(f, g), xf[g], xf[f]);
        if (DIR == 0) xf[f] *= df[f];
        w[(size_t)(N + f) * P + cell] = xf[f];
    }
    // ---- backward: rows i = N-1-j
    auto load_b = [&](int j0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = N - 1 - j0 - u;
            if (i >= 0) {
#pragma unroll
                for (int k = 0; k < W; ++k)
                    cn[u][k] = i + 1 + k < N ? __ldg(lu + (DIR == 0 ? arrow_slot<W>(i, i + 1 + k, N, b)
                                                                     : arrow_slot<W>(i + 1 + k, i, N, b)) * P)
                                             : 0.0;
#pragma unroll
                for (int f = 0; f < NF; ++f) cn[u][W + f] = up_flow(i, f);
                vn[u] = w[(size_t)i * P + cell];
                sn[u] = DIR == 0 ? __ldg(dinv + (size_t)i * P) : 1.0;
            }
        }
    };
#pragma unroll
    for (int k = 0; k < W; ++k) win[k] = 0.0;          // win[k] = x_{i+1+k}
    load_b(0);
    for (int j0 = 0; j0 < N; j0 += U) {
        take();
        if (j0 + U < N) load_b(j0 + U);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = N - 1 - j0 - u;
            if (i < 0) break;
            double acc = v[u];
#pragma unroll
            for (int k = 0; k < W; ++k) acc = fma(-c[u][k], win[k], acc);
#pragma unroll
            for (int f = 0; f < NF; ++f) acc = fma(-c[u][W + f], xf[f], acc);
            if (DIR == 0) acc *= s[u];
            w[(size_t)i * P + cell] = acc;
#pragma unroll
            for (int k = W - 1; k > 0; --k) win[k] = win[k - 1];
            if (W > 0) win[0] = acc;
        }
    }
}

template <int W>
__global__ void __launch_bounds__(64) k_smw_w_arrow(SetupArgs a) {
    const int n_tiles = a.ncp / kTile;
    const int wid = blockIdx.x * 2 + (threadIdx.x >> 5);
    if (wid >= n_tiles * a.r * (a.with_T ? 2 : 1)) return;
    const int tile = wid % n_tiles, kd = wid / n_tiles, k = kd % a.r;
    const int cell = tile * kTile + (threadIdx.x & 31);
    const size_t off = (size_t)k * a.b * a.ncp;
    if (kd < a.r) arrow_solve<W, 0>(a, a.Ud + off, a.W + off, cell);
    else arrow_solve<W, 1>(a, a.Vd + off, a.Wt + off, cell);
}

// C^-1 by Gauss-Jordan with partial pivoting, in place, one lane per cell and one
// warp per tile, the matrix in shared memory [entry][lane] so that a lane's pivot
// row is one more index (no bank conflict, no divergence).  In place takes r^3 FMAs,
// half of eliminating a [C | I] pair; the pivot search is integer work.  Nine pairs
// on 128 x 128 cells: 152 -> 56 us (the [C | I] pair lived in local memory).  In
// registers the exchanges would be selects over every row: it compiled to spills.
template <int R>
__global__ void __launch_bounds__(kTile) k_smw_cinv_sh(SetupArgs a) {
    __shared__ double sc[R * R][kTile];
    __shared__ int sp[R][kTile];
    const int lane = threadIdx.x, cell = blockIdx.x * kTile + lane;
    const size_t P = a.ncp;
    long long cmax = 0;
#pragma unroll
    for (int i = 0; i < R * R; ++i) {
        const double v = a.Cinv[(size_t)i * P + cell];
        sc[i][lane] = v;
        cmax = abs_max(cmax, v);
    }
    bool ok = true;
#pragma unroll 1
    for (int k = 0; k < R; ++k) {
        // a NaN is never picked over another row, and never given up
        constexpr long long inf = 0x7ff0000000000000ll;
        long long best = __double_as_longlong(sc[k * R + k][lane]) & 0x7fffffffffffffffll;
        int pr = k;
        for (int i = k + 1; i < R; ++i) {
            const long long v = __double_as_longlong(sc[i * R + k][lane]) & 0x7fffffffffffffffll;
            if (v <= inf && v > best) {
                best = v;
                pr = i;
            }
        }
        sp[k][lane] = pr;
        double p[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            p[j] = sc[pr * R + j][lane];
            sc[pr * R + j][lane] = sc[k * R + j][lane];
        }
        const double piv = __longlong_as_double(best);      // |pivot|
        ok = ok && pivot_ok(piv, cmax);
        double d = 0.0;
#pragma unroll
        for (int j = 0; j < R; ++j) d = j == k ? p[j] : d;
        d = 1.0 / d;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            p[j] = (j == k ? 1.0 : p[j]) * d;
            sc[k * R + j][lane] = p[j];
        }
#pragma unroll 1
        for (int i = 0; i < R; ++i) {
            if (i == k) continue;
            const double f = sc[i * R + k][lane];
            double c[R];
#pragma unroll
            for (int j = 0; j < R; ++j) c[j] = j == k ? 0.0 : sc[i * R + j][lane];
#pragma unroll
            for (int j = 0; j < R; ++j) c[j] = fma(-f, p[j], c[j]);
#pragma unroll
            for (int j = 0; j < R; ++j) sc[i * R + j][lane] = c[j];
        }
    }
    // row exchanges of the matrix are column exchanges of its inverse, undone in reverse
#pragma unroll 1
    for (int k = R - 1; k >= 0; --k) {
        const int pr = sp[k][lane];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const double x = sc[j * R + k][lane], y = sc[j * R + pr][lane];
            sc[j * R + k][lane] = y;
            sc[j * R + pr][lane] = x;
        }
    }
#pragma unroll
    for (int i = 0; i < R * R; ++i) a.Cinv[(size_t)i * P + cell] = sc[i][lane];
    if (!ok) atomicMin(a.err_cell, cell);
}

// Write the general apply's streams from the packing tables (SmwPlan); the zeros of the
// padding were written when they were allocated.
template <typename T>
__global__ void k_smw_pack(T *out, const double *lu, const double *dinv, const int *pk_slot,
                           const int *pk_scale, int len, int ncp) {
    const long long total = (long long)len * ncp;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int cell = (int)(i % ncp), pos = (int)(i / ncp);
        const int sl = pk_slot[pos], sc = pk_scale[pos];
        double v;
        if (sl < -1) continue;
        if (sl >= 0) {
            v = lu[(size_t)sl * ncp + cell];
            if (sc >= 0) v *= dinv[(size_t)sc * ncp + cell];
        } else {
            v = dinv[(size_t)sc * ncp + cell];
        }
        out[i] = (T)v;
    }
}

template <typename T>
__global__ void k_round(T *out, const double *in, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        out[i] = (T)in[i];
}

// Structured stream packing: per position a source code and argument
//   src >= 0: LU slot (times the pivot inverse of row arg if arg >= 0)
//   src = -1: pivot inverse of row arg      src = -2: dot vector entry arg
//   src = -3: W entry arg                   src = -4: zero
//   src = -5: folded tail entry, written by k_smw_fold
// One warp per tile and run of 16-byte vectors: a position's code is the same for
// the whole warp, so no lane computes indices of its own and every access is one
// coalesced request.  `list` names the vectors that hold a value, the n_scaled that
// need a product with a pivot inverse first: a product that a predicate switches
// off still takes its FP64 pipe slot, so the others run a loop without one.  The
// zeros of the other vectors were written when the stream was allocated.
// Measured on 128 x 128 cells, N = 60: two pairs 68 -> 51 us per direction.
constexpr int kPackWarps = 4;
template <typename T> struct PackVec;
template <> struct PackVec<double> { using type = double2; };
template <> struct PackVec<float> { using type = float4; };

template <typename T>
struct PackArgs {
    T *out;
    const double *lu, *dinv, *DV, *WW;
    const int *src, *arg, *list;
    int n_scaled, n_list, Lt, ncp;
};

// Part `part` of `parts` of the tile blockIdx.x.
template <typename T>
__device__ __forceinline__ void pack_part(const PackArgs<T> &A, int part, int parts) {
    constexpr int VEC = 16 / (int)sizeof(T);
    using V = typename PackVec<T>::type;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t cell = (size_t)blockIdx.x * kTile + lane;
    const size_t ncp = A.ncp;
    T *o = A.out + ((size_t)blockIdx.x * A.Lt) * kTile + (size_t)lane * VEC;
    const int step = parts * kPackWarps;
    auto run = [&](auto scaled, int i0, int i1) {
#pragma unroll 4
        for (int i = i0; i < i1; i += step) {
            const int pv = __ldg(A.list + i);
            alignas(16) T v[VEC];
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                // loads without branches, so that the unrolled vectors' loads are in flight together
                const int sv = __ldg(A.src + pv * VEC + j), ag = __ldg(A.arg + pv * VEC + j);
                const double *s = sv >= 0 ? A.lu : sv == -2 ? A.DV : sv == -3 ? A.WW : A.dinv;
                double e = __ldg(s + (size_t)(sv >= 0 ? sv : sv > -4 ? ag : 0) * ncp + cell);
                if constexpr (decltype(scaled)::value) {
                    const bool on = sv >= 0 && ag >= 0;
                    const double d = __ldg(A.dinv + (size_t)(on ? ag : 0) * ncp + cell);
                    e *= on ? d : 1.0;
                }
                v[j] = sv > -4 ? (T)e : T(0);
            }
            *reinterpret_cast<V *>(o + (size_t)pv * kTile * VEC) = *reinterpret_cast<V *>(v);
        }
    };
    const int w = part * kPackWarps + warp;
    run(std::true_type{}, w, A.n_scaled);
    run(std::false_type{}, A.n_scaled + w, A.n_list);
}

template <typename T>
__global__ void __launch_bounds__(kPackWarps * kTile) k_smw_spack(PackArgs<T> A) {
    pack_part(A, blockIdx.y, gridDim.y);
}

// Folded tail entries (W C^-1)[q][a] = sum_l W[l][q] C^-1[l][a] (transposed: W'
// and C^-T), in FP64, into their stream positions tp[a * b + q] of the FP64
// stream and, where there is one, the FP32 stream.  One warp per tile and rows
// q; the r entries of W are read once for the r sums, C^-1 sits in shared
// memory.  r^2 FMAs a row: bound by the FP64 pipe.  The rest of the FP64 stream, bound
// by memory, is packed beside it by `parts` of the blocks of every tile, which alternate
// with the folding ones as far as they go.  Nine pairs on 128 x 128 cells, N = 60:
// 280 us in one kernel that formed a fold entry per position, 68 + 173 us as two kernels
// (133 us of FP64 pipe time), 217 us here.
constexpr int kFoldWarps = 4;

template <int R>
__global__ void __launch_bounds__(kFoldWarps * kTile) k_smw_fold(PackArgs<double> A, int parts, float *out32,
                                                                 const int *tp64, const int *tp32, int Lt32,
                                                                 const double *Cinv, int b, int trans) {
    __shared__ double sc[R * R][kTile];
    const int y = blockIdx.y, folds = gridDim.y - parts, both = min(parts, folds);
    const int part = y < 2 * both ? y >> 1 : y - both;
    if (y < 2 * both ? !(y & 1) : parts > folds) {
        pack_part(A, part, parts);
        return;
    }
    double *out64 = A.out;
    const double *WW = A.WW;
    const int Lt64 = A.Lt, ncp = A.ncp;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t tile = blockIdx.x, cell = tile * kTile + lane;
    for (int i = warp; i < R * R; i += kFoldWarps)           // sc[l * R + a]
        sc[i][lane] = __ldg(Cinv + (size_t)(trans ? (i % R) * R + i / R : i) * ncp + cell);
    __syncthreads();
    for (int q = part * kFoldWarps + warp; q < b; q += folds * kFoldWarps) {
        double w[R];
#pragma unroll
        for (int l = 0; l < R; ++l) w[l] = __ldg(WW + ((size_t)l * b + q) * ncp + cell);
#pragma unroll
        for (int aa = 0; aa < R; ++aa) {
            double v = 0.0;
#pragma unroll
            for (int l = 0; l < R; ++l) v = fma(w[l], sc[l * R + aa][lane], v);
            const int p64 = __ldg(tp64 + aa * b + q);
            out64[((tile * Lt64 + (p64 & ~1)) * kTile + 2 * lane) + (p64 & 1)] = v;
            if (out32) {
                const int p32 = __ldg(tp32 + aa * b + q);
                out32[((tile * Lt32 + (p32 & ~3)) * kTile + 4 * lane) + (p32 & 3)] = (float)v;
            }
        }
    }
}

inline int grid_for(long long n, int block) {
    long long g = (n + block - 1) / block;
    if (g > 152LL * 64) g = 152LL * 64;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

sts_status smw_setup(sts_jac_s *h) {
    SmwPlan &M = h->smw;
    const bool was_ready = M.ready;
    M.ready = false;
    SetupArgs a;
    a.Sd = M.Sd; a.Ud = M.Ud; a.Vd = M.Vd;
    a.lu = M.lu; a.dinv = M.dinv; a.W = M.W; a.Wt = M.Wt; a.Cinv = M.Cinv;
    a.lu_diag = M.lu_diag; a.src_slot = M.src_slot; a.d_ptr = M.d_ptr;
    a.colL_ptr = M.f_colL_ptr; a.colL_slot = M.f_colL_slot;
    a.upd_ptr = M.f_upd_ptr; a.upd_tgt = M.f_upd_tgt; a.upd_src = M.f_upd_src;
    a.fwd_ptr0 = M.ap_fwd_ptr[0]; a.fwd_col0 = M.ap_fwd_col[0]; a.fwd_slot0 = M.ap_fwd_slot[0];
    a.bwd_ptr0 = M.ap_bwd_ptr[0]; a.bwd_col0 = M.ap_bwd_col[0]; a.bwd_slot0 = M.ap_bwd_slot[0];
    a.fwd_ptr1 = M.ap_fwd_ptr[1]; a.fwd_col1 = M.ap_fwd_col[1]; a.fwd_slot1 = M.ap_fwd_slot[1];
    a.bwd_ptr1 = M.ap_bwd_ptr[1]; a.bwd_col1 = M.ap_bwd_col[1]; a.bwd_slot1 = M.ap_bwd_slot[1];
    a.err_cell = M.err_cell;
    a.nc = h->nc; a.ncp = h->ncp; a.b = h->b; a.r = h->r_diag; a.nnz_lu = M.nnz_lu;
    a.nnz_d = h->nnz_d; a.with_T = h->has_T ? 1 : 0;
    constexpr int kNone = 0x7f7f7f7f;       // above any cell
    STS_CK(cudaMemsetAsync(M.err_cell, 0x7f, sizeof(int), h->stream));
    if (M.structured) {
        auto lu = M.s_w == 0 ? k_smw_lu_arrow<0> : M.s_w == 1 ? k_smw_lu_arrow<1> : M.s_w == 2 ? k_smw_lu_arrow<2>
                  : M.s_w == 3 ? k_smw_lu_arrow<3> : k_smw_lu_arrow<4>;
        lu<<<h->n_tiles, kTile, 0, h->stream>>>(a);
    } else {
        k_smw_lu<<<(h->ncp + 63) / 64, 64, 0, h->stream>>>(a);
    }
    STS_LAUNCHED();
    const long long nw = (long long)h->ncp * a.r * (a.with_T ? 2 : 1);
    if (nw > 0) {
        if (M.structured) {
            auto ws = M.s_w == 0 ? k_smw_w_arrow<0> : M.s_w == 1 ? k_smw_w_arrow<1> : M.s_w == 2 ? k_smw_w_arrow<2>
                      : M.s_w == 3 ? k_smw_w_arrow<3> : k_smw_w_arrow<4>;
            ws<<<(unsigned)((nw + 63) / 64), 64, 0, h->stream>>>(a);
        } else {
            k_smw_w<<<(unsigned)((nw + 63) / 64), 64, 0, h->stream>>>(a);
        }
        STS_LAUNCHED();
        const long long nc2 = (long long)h->ncp * a.r * a.r;
        k_smw_cmat<<<(unsigned)((nc2 + 255) / 256), 256, 0, h->stream>>>(a);
        STS_LAUNCHED();
        using Cinv = void (*)(SetupArgs);
        static const Cinv cinv[11] = {nullptr, k_smw_cinv_sh<1>, k_smw_cinv_sh<2>, k_smw_cinv_sh<3>, k_smw_cinv_sh<4>,
                                      k_smw_cinv_sh<5>, k_smw_cinv_sh<6>, k_smw_cinv_sh<7>, k_smw_cinv_sh<8>,
                                      k_smw_cinv_sh<9>, k_smw_cinv_sh<10>};
        if (a.r <= 10) cinv[a.r]<<<h->n_tiles, kTile, 0, h->stream>>>(a);
        else k_smw_cinv<<<(h->ncp + 63) / 64, 64, 0, h->stream>>>(a);      // more than any structured instance holds
        STS_LAUNCHED();
    }
    const size_t P = h->ncp;
    const int b = h->b, r = h->r_diag;
    for (int dir = 0; dir < 2; ++dir) {
        if (dir == 1 && !h->has_T) continue;
        const double *DV = dir == 0 ? M.Vd : M.Ud;
        const double *WW = dir == 0 ? M.W : M.Wt;
        if (M.structured) {
            const int nt = h->n_tiles;
            auto ysplit = [&](int work) {       // blocks per tile: a few thousand warps in all, at least 4 units each
                return (unsigned)std::max(1, std::min((work + 4 * kPackWarps - 1) / (4 * kPackWarps),
                                                      (h->nsm * 64 + nt * kPackWarps - 1) / (nt * kPackWarps)));
            };
            const PackArgs<double> p64{M.ap64[dir], M.lu, M.dinv, DV, WW, M.spk_src[0][dir], M.spk_arg[0][dir],
                                       M.spk_list[0][dir], M.spk_scaled[0][dir], M.spk_n[0][dir], M.s_lt[0], h->ncp};
            const unsigned parts = ysplit(M.spk_n[0][dir]);
            if (M.ap32[dir]) {
                const PackArgs<float> p32{M.ap32[dir], M.lu, M.dinv, DV, WW, M.spk_src[1][dir], M.spk_arg[1][dir],
                                          M.spk_list[1][dir], M.spk_scaled[1][dir], M.spk_n[1][dir], M.s_lt[1], h->ncp};
                k_smw_spack<float><<<dim3(nt, ysplit(M.spk_n[1][dir])), kPackWarps * kTile, 0, h->stream>>>(p32);
                STS_LAUNCHED();
            }
            if (M.tail_pos[0] && r > 0) {
                static_assert(kPackWarps == kFoldWarps, "one split rule");
                using Fold = void (*)(PackArgs<double>, int, float *, const int *, const int *, int, const double *, int, int);
                static const Fold fold[11] = {nullptr, k_smw_fold<1>, k_smw_fold<2>, k_smw_fold<3>, k_smw_fold<4>,
                                              k_smw_fold<5>, k_smw_fold<6>, k_smw_fold<7>, k_smw_fold<8>,
                                              k_smw_fold<9>, k_smw_fold<10>};
                fold[r]<<<dim3(nt, parts + ysplit(b)), kFoldWarps * kTile, 0, h->stream>>>(
                    p64, (int)parts, M.ap32[dir], M.tail_pos[0], M.tail_pos[1], M.s_lt[1], M.Cinv, b, dir);
            } else {
                k_smw_spack<double><<<dim3(nt, parts), kPackWarps * kTile, 0, h->stream>>>(p64);
            }
            STS_LAUNCHED();
            continue;
        }
        const int len = kGenWarps * M.g_wlen[dir];
        const long long n = (long long)len * P;
        k_smw_pack<double><<<grid_for(n, 256), 256, 0, h->stream>>>(M.ap64[dir], M.lu, M.dinv, M.pk_slot[dir],
                                                                     M.pk_scale[dir], len, h->ncp);
        STS_LAUNCHED();
        if (M.ap32[dir]) {
            k_smw_pack<float><<<grid_for(n, 256), 256, 0, h->stream>>>(M.ap32[dir], M.lu, M.dinv, M.pk_slot[dir],
                                                                       M.pk_scale[dir], len, h->ncp);
            STS_LAUNCHED();
            const long long nw = (long long)r * b * P;
            if (nw > 0) {
                k_round<float><<<grid_for(nw, 256), 256, 0, h->stream>>>(M.W32[dir], WW, nw);
                STS_LAUNCHED();
                k_round<float><<<grid_for(nw, 256), 256, 0, h->stream>>>(M.DV32[dir], DV, nw);
                STS_LAUNCHED();
            }
        }
    }
    // one look at the device for the whole setup, after the packing (which a failed cell
    // makes useless, not wrong): the wait flag and, beside it, the first failing cell
    h->streams_dirty = true;
    int flags[2] = {0, kNone};
    STS_CK(cudaMemcpyAsync(flags, h->d_err, sizeof(flags), cudaMemcpyDeviceToHost, h->stream));
    STS_CK(cudaStreamSynchronize(h->stream));
    if (flags[1] != kNone) {
        STS_TRY(report_wait(h, flags[0]));
        return set_error(STS_ERR_SINGULAR,
                         "block-Jacobi setup: cell %d has a pivot below 1e-14 x its row maximum "
                         "(static pivot order) or a singular capacitance matrix C_k", flags[1]);
    }
    // a wait that gave up earlier is this call's error: what was not set up stays so
    M.ready = was_ready || !flags[0];
    return report_wait(h, flags[0]);
}

}  // namespace sts
