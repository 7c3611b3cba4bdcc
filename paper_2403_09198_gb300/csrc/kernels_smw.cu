// kernels_smw.cu -- block-Jacobi through the Sherman-Morrison-Woodbury formula
// (Section 6).  Each diagonal block is A_k = A_k^0 + U_k V_k^T with A_k^0 = S_kk
// sparse (Eq. R1_Block_Jacobian).
//
// Setup: kernels_smw_setup.cu.
// Apply (SMW-1..3): x0 = (A_k^0)^-1 b_k, t = V_k^T x0, z = C_k^-1 t (FP64),
//   x_k = x0 - W_k z.  The paper prints "+ W_k z"; with C_k = I + V^T A0^-1 U the
//   Woodbury identity needs the minus sign, which is what is computed here.
// Transposed apply: (A0 + U V^T)^-T = (A0^T + V U^T)^-1, i.e. the same steps with
//   A0^T (solved from the same LU factors), U and V swapped and C_k^T.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <type_traits>
#include <vector>

#include "ring.cuh"
#include "smw_sapply.cuh"
#include "sts_internal.h"

namespace sts {
namespace {

template <typename T>
struct ApplyArgs {
    const T *st;            // [kGenWarps][wlen][ncp] coefficients of every warp, in its order
    const short *row;       // [kGenWarps][wlen] row that a coefficient updates, -1: none
    const int *n_fwd, *n_bwd;   // [b] coefficients of every warp for column j, forward and backward
    const T *dv;            // [r][b][ncp] dot vectors (V for N, U for T)
    const T *W;             // [r][b][ncp] (W for N, Wt for T)
    const double *Cinv;     // [r][r][ncp]
    Vec<T> x, y;
    int wlen, b, r, ncp, trans;
};


// Any pattern: one block of four warps per 32 cells, one lane per cell.  The working
// vector lives in shared memory [q][lane]; the sweeps go column by column, and the rows
// that a column updates are dealt to the warps, so that four FP64 pipes share a tile's
// work with one barrier per column.  Forward updates reach a row in ascending column
// order, the order of a serial sweep over the rows.  Each warp's coefficients are one
// sequence, loaded a batch of four ahead of its use and brought into L2 well before.
//
// As one warp's serial program over the rows a tile took 85 us for 33 x 33 blocks (41 x 37
// cells, 15% filled before the factorisation), mostly one dependent step after
// another; now 32 us.  Rings of bulk or cp.async stages in front of the batches took 39 us:
// with one block on most SMs a warp's instructions per coefficient set the time.
constexpr int kGenAhead = 4;        // coefficients of a batch; padding behind every warp's sequence
constexpr int kGenPrefetch = 64;    // coefficients between one used and one brought into L2
constexpr int kGenSum = 8;          // pairs whose partial sums are added at once

template <typename T, int RMAX>
__global__ void __launch_bounds__(kGenWarps * kTile) k_smw_apply(ApplyArgs<T> a) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int U = kGenAhead, KC = RMAX < kGenSum ? RMAX : kGenSum;
    T *part = reinterpret_cast<T *>(smem_raw);                     // [kGenWarps][KC][32]
    T *w = part + kGenWarps * KC * kTile;                           // [b][32]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cell = blockIdx.x * kTile + lane, b = a.b;
    const size_t P = a.ncp;
    const T *__restrict__ x = a.x.at(cell);
    const T *__restrict__ st = a.st + (size_t)warp * a.wlen * P + cell;
    const short *__restrict__ row = a.row + (size_t)warp * a.wlen;
    // the next batch; the sequences end in U padding positions, there to be read
    T vn[U];
    int rn[U], left = a.wlen;
    auto advance = [&](int n) {
        st += (size_t)n * P;
        row += n;
        left -= n;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            vn[u] = __ldg(st + (size_t)u * P);
            rn[u] = __ldg(row + u);
            if (u < n && kGenPrefetch + u < left) prefetch_l2(st + (size_t)(kGenPrefetch + u) * P);
        }
    };
    for (int k = 0; k < min(kGenPrefetch + U, a.wlen); ++k) prefetch_l2(st + (size_t)k * P);
    advance(0);
    for (int i = warp; i < b; i += kGenWarps) w[i * kTile + lane] = __ldg(x + i * a.x.sq);
    __syncthreads();
    // n updates w[row] -= coefficient * xj: the rows of one column are distinct
    auto column = [&](T xj, int n) {
        for (int s = 0; s < n; s += U) {
            T v[U], c[U];
            int r[U];
            const int m = min(U, n - s);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                v[u] = vn[u];
                r[u] = u < m ? rn[u] : -1;
            }
            advance(m);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (r[u] >= 0) c[u] = w[r[u] * kTile + lane];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (r[u] >= 0) w[r[u] * kTile + lane] = fma(-v[u], xj, c[u]);
        }
    };
    for (int j = 0; j < b; ++j) {
        const int n = __ldg(a.n_fwd + j);
        if (n == 0) continue;
        column(w[j * kTile + lane], n);
        __syncthreads();
    }
    // pivot inverses: ceil(b / kGenWarps) positions of every warp, the last one padding where
    // the warps are too many
    for (int i = warp; i < b; i += kGenWarps) {
        const T v = vn[0];
        advance(1);
        w[i * kTile + lane] *= v;
    }
    if (b % kGenWarps && warp >= b % kGenWarps) advance(1);
    __syncthreads();
    for (int j = b - 1; j >= 0; --j) {
        const int n = __ldg(a.n_bwd + j);
        if (n == 0) continue;
        column(w[j * kTile + lane], n);
        __syncthreads();
    }
    // t = dv^T x0 over the warps' rows, z = C^-1 t (FP64), x = x0 - W z
    T t[RMAX];
#pragma unroll
    for (int k = 0; k < RMAX; ++k) t[k] = T(0);
    const T *__restrict__ dv = a.dv + cell;
#pragma unroll 4
    for (int q = warp; q < b; q += kGenWarps) {
        const T xq = w[q * kTile + lane];
#pragma unroll
        for (int k = 0; k < RMAX; ++k)
            if (k < a.r) t[k] = fma(__ldg(dv + ((size_t)k * b + q) * P), xq, t[k]);
    }
#pragma unroll
    for (int k0 = 0; k0 < RMAX; k0 += KC) {
        if (k0 >= a.r) break;
#pragma unroll
        for (int k = 0; k < KC; ++k)
            if (k0 + k < a.r) part[(warp * KC + k) * kTile + lane] = t[k0 + k];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KC; ++k)
            if (k0 + k < a.r) {
                T s = part[k * kTile + lane];
#pragma unroll
                for (int v = 1; v < kGenWarps; ++v) s += part[(v * KC + k) * kTile + lane];
                t[k0 + k] = s;
            }
        __syncthreads();
    }
    T z[RMAX];
#pragma unroll
    for (int k = 0; k < RMAX; ++k) {
        double s = 0.0;
        if (k < a.r) {
#pragma unroll
            for (int l = 0; l < RMAX; ++l)
                if (l < a.r) {
                    const double cij = a.trans ? __ldg(a.Cinv + ((size_t)l * a.r + k) * P + cell)
                                               : __ldg(a.Cinv + ((size_t)k * a.r + l) * P + cell);
                    s = fma(cij, (double)t[l], s);
                }
        }
        z[k] = (T)s;
    }
    const T *__restrict__ Wp = a.W + cell;
    long long ystep;
    T *__restrict__ y = a.y.out(cell, ystep);
#pragma unroll 4
    for (int q = warp; q < b; q += kGenWarps) {
        T v = w[q * kTile + lane];
#pragma unroll
        for (int k = 0; k < RMAX; ++k)
            if (k < a.r) v = fma(-__ldg(Wp + ((size_t)k * b + q) * P), z[k], v);
        y[q * ystep] = v;
    }
}

}  // namespace

// Host: symbolic factorisation of the shared diagonal pattern and the programs
// of the two apply directions.
sts_status smw_build(sts_jac_s *h) {
    SmwPlan &M = h->smw;
    const int b = h->b;
    if (b > 4095) return set_error(STS_ERR_INVALID_ARG, "block_size above 4095 is not supported by the SMW apply");
    if (h->r_diag > kMaxPairsDiag)
        return set_error(STS_ERR_INVALID_ARG, "r_diag = %d exceeds the supported %d pairs per diagonal block",
                         h->r_diag, kMaxPairsDiag);
    std::vector<char> nz((size_t)b * b, 0);
    for (int p = 0; p < b; ++p)
        for (int e = h->dptr[p]; e < h->dptr[p + 1]; ++e) nz[(size_t)p * b + h->didx[e]] = 1;
    for (int k = 0; k < b; ++k)               // symbolic elimination, natural order
        for (int i = k + 1; i < b; ++i)
            if (nz[(size_t)i * b + k])
                for (int j = k + 1; j < b; ++j)
                    if (nz[(size_t)k * b + j]) nz[(size_t)i * b + j] = 1;
    std::vector<int> slot((size_t)b * b, -1);
    M.h_lu_ptr.assign(b + 1, 0);
    M.h_lu_idx.clear();
    M.h_lu_diag.assign(b, -1);
    for (int i = 0; i < b; ++i) {
        for (int j = 0; j < b; ++j)
            if (nz[(size_t)i * b + j]) {
                slot[(size_t)i * b + j] = (int)M.h_lu_idx.size();
                if (i == j) M.h_lu_diag[i] = (int)M.h_lu_idx.size();
                M.h_lu_idx.push_back(j);
            }
        M.h_lu_ptr[i + 1] = (int)M.h_lu_idx.size();
    }
    M.nnz_lu = (int)M.h_lu_idx.size();
    const int sw = struct_band(b, h->dptr, h->didx);
    M.structured = sw >= 0 && sap_rmax(h->r_diag, sw) > 0 && M.nnz_lu == h->nnz_d;
    M.h_src_slot.assign(h->nnz_d, 0);
    for (int p = 0; p < b; ++p)
        for (int e = h->dptr[p]; e < h->dptr[p + 1]; ++e) M.h_src_slot[e] = slot[(size_t)p * b + h->didx[e]];
    // factorisation schedule (the structured family's setup has arithmetic indices instead)
    std::vector<int> colL_ptr(b + 1, 0), colL_slot, upd_ptr(1, 0), upd_tgt, upd_src;
    for (int k = 0; k < b && !M.structured; ++k) {
        for (int i = k + 1; i < b; ++i) {
            if (slot[(size_t)i * b + k] < 0) continue;
            colL_slot.push_back(slot[(size_t)i * b + k]);
            for (int j = k + 1; j < b; ++j)
                if (slot[(size_t)k * b + j] >= 0) {
                    upd_tgt.push_back(slot[(size_t)i * b + j]);
                    upd_src.push_back(slot[(size_t)k * b + j]);
                }
            upd_ptr.push_back((int)upd_tgt.size());
        }
        colL_ptr[k + 1] = (int)colL_slot.size();
    }
    // apply programs.  dir 0 (A0):  forward  L rows   (i, j<i), coefficient L_ij
    //                               backward U rows   (i, j>i), coefficient U_ij * dinv_i
    //                  dir 1 (A0^T): forward  U cols   (j<i, i), coefficient U_ji * dinv_j
    //                               backward L cols   (j>i, i), coefficient L_ji
    // Setup solves use the unscaled LU slots with the same row lists.
    for (int dir = 0; dir < 2 && !M.structured; ++dir) {
        std::vector<int> fptr(b + 1, 0), fcol, fslot, fscale, bptr(b + 1, 0), bcol, bslot, bscale;
        // the setup's unscaled solves use (fcol, fslot) and (bcol, bslot); the
        // apply streams carry the scaled coefficients described by (fscale, bscale)
        for (int i = 0; i < b; ++i) {
            for (int j = 0; j < i; ++j) {
                const int sl = dir == 0 ? slot[(size_t)i * b + j] : slot[(size_t)j * b + i];
                if (sl < 0) continue;
                fcol.push_back(j);
                fslot.push_back(sl);
                fscale.push_back(dir == 0 ? -1 : j);
            }
            fptr[i + 1] = (int)fcol.size();
        }
        for (int r = 0; r < b; ++r) {
            const int i = b - 1 - r;
            for (int j = i + 1; j < b; ++j) {
                const int sl = dir == 0 ? slot[(size_t)i * b + j] : slot[(size_t)j * b + i];
                if (sl < 0) continue;
                bcol.push_back(j);
                bslot.push_back(sl);
                bscale.push_back(dir == 0 ? i : -1);
            }
            bptr[r + 1] = (int)bcol.size();
        }
        STS_TRY(upload(h, &M.ap_fwd_ptr[dir], fptr));
        STS_TRY(upload(h, &M.ap_fwd_col[dir], fcol));
        STS_TRY(upload(h, &M.ap_fwd_slot[dir], fslot));
        STS_TRY(upload(h, &M.ap_bwd_ptr[dir], bptr));
        STS_TRY(upload(h, &M.ap_bwd_col[dir], bcol));
        STS_TRY(upload(h, &M.ap_bwd_slot[dir], bslot));
        // apply program of any other pattern (k_smw_apply): columns forward, the pivot
        // inverses, columns backward, every column's rows dealt to the warps
        struct Entry {
            int row, slot, scale;
        };
        std::vector<std::vector<Entry>> fc(b), bc(b);
        for (int i = 0; i < b; ++i)
            for (int e = fptr[i]; e < fptr[i + 1]; ++e) fc[fcol[e]].push_back({i, fslot[e], fscale[e]});
        for (int r = 0; r < b; ++r)
            for (int e = bptr[r]; e < bptr[r + 1]; ++e) bc[bcol[e]].push_back({b - 1 - r, bslot[e], bscale[e]});
        std::vector<int> nf(b), nb(b), pk_slot[kGenWarps], pk_scale[kGenWarps];
        std::vector<short> row[kGenWarps];
        auto deal = [&](const std::vector<Entry> &col) {
            const int n = ((int)col.size() + kGenWarps - 1) / kGenWarps;
            for (int k = 0; k < n * kGenWarps; ++k) {
                const bool on = k < (int)col.size();
                row[k % kGenWarps].push_back(on ? (short)col[k].row : (short)-1);
                pk_slot[k % kGenWarps].push_back(on ? col[k].slot : -2);
                pk_scale[k % kGenWarps].push_back(on ? col[k].scale : -1);
            }
            return n;
        };
        for (int j = 0; j < b; ++j) nf[j] = deal(fc[j]);
        std::vector<Entry> piv(b);
        for (int i = 0; i < b; ++i) piv[i] = {i, -1, i};
        deal(piv);
        for (int j = b - 1; j >= 0; --j) nb[j] = deal(bc[j]);
        for (int v = 0; v < kGenWarps; ++v) {
            row[v].insert(row[v].end(), kGenAhead, (short)-1);
            pk_slot[v].insert(pk_slot[v].end(), kGenAhead, -2);
            pk_scale[v].insert(pk_scale[v].end(), kGenAhead, -1);
        }
        M.g_wlen[dir] = (int)row[0].size();
        std::vector<int> all_slot, all_scale;
        std::vector<short> all_row;
        for (int v = 0; v < kGenWarps; ++v) {
            all_slot.insert(all_slot.end(), pk_slot[v].begin(), pk_slot[v].end());
            all_scale.insert(all_scale.end(), pk_scale[v].begin(), pk_scale[v].end());
            all_row.insert(all_row.end(), row[v].begin(), row[v].end());
        }
        STS_TRY(upload(h, &M.pk_slot[dir], all_slot));
        STS_TRY(upload(h, &M.pk_scale[dir], all_scale));
        STS_TRY(upload(h, &M.g_row[dir], all_row));
        STS_TRY(upload(h, &M.g_nf[dir], nf));
        STS_TRY(upload(h, &M.g_nb[dir], nb));
    }
    // structured apply tables (both directions; FP64 and, for mixed handles, FP32)
    if (M.structured) {
        const int NF = kStructNF, N = b - NF, r = h->r_diag;
        M.s_w = sw;
        auto sl = [&](int i, int j) { return slot[(size_t)i * b + j]; };
        const int RMAX = sap_rmax(r, sw);      // the kernel instance chosen at apply time
        for (int prec = 0; prec < 2; ++prec) {
            if (prec == 1 && h->dtype != STS_MIXED) continue;
            const int elem = prec == 0 ? 8 : 4, vec = 16 / elem, K = kSApChunkBytes / (kTile * elem);
            for (int dir = 0; dir < 2; ++dir) {
                std::vector<int> src, arg, gsrc, garg;
                auto put = [&](int s_, int a_) { gsrc.push_back(s_); garg.push_back(a_); };
                auto zero = [&](int n) { for (int k = 0; k < n; ++k) put(-4, 0); };
                // close one group: whole vectors, never straddling a chunk (zero padding)
                bool fits = true;
                auto group = [&]() {
                    while (gsrc.size() % vec) put(-4, 0);
                    const int G = (int)gsrc.size(), off = (int)(src.size() % K);
                    if (G > K) fits = false;
                    if (off + G > K)
                        for (int k = off; k < K; ++k) { src.push_back(-4); arg.push_back(0); }
                    src.insert(src.end(), gsrc.begin(), gsrc.end());
                    arg.insert(arg.end(), garg.begin(), garg.end());
                    gsrc.clear();
                    garg.clear();
                };
                auto vd = [&](int q) {              // dot-vector entries of unknown q, padded to RMAX
                    for (int k = 0; k < RMAX; ++k) put(k < r ? -2 : -4, k < r ? k * b + q : 0);
                };
                // lower factor of this direction: dir 0 L, dir 1 U'^T (U scaled by the row pivot inverse)
                auto lo = [&](int i, int j) {       // coefficient (i, j), i > j
                    if (dir == 0) put(sl(i, j), -1);
                    else put(sl(j, i), j);
                };
                // upper factor after the pivot scaling: dir 0 U' = D^-1 U, dir 1 L^T
                auto up = [&](int i, int j) {       // coefficient (i, j), i < j
                    if (dir == 0) put(sl(i, j), i);
                    else put(sl(j, i), -1);
                };
                const int FW = sw + NF, UF = sap_fwd_rows(FW, vec, NF);
                for (int i0 = 0; i0 < N; i0 += UF) {
                    for (int i = i0; i < i0 + UF; ++i) {
                        if (i >= N) {
                            zero(FW);
                            continue;
                        }
                        for (int k = 0; k < sw; ++k) {
                            const int j = i - sw + k;
                            if (j >= 0) lo(i, j);
                            else put(-4, 0);
                        }
                        for (int f = 0; f < NF; ++f) lo(N + f, i);
                    }
                    group();
                }
                lo(N + 1, N);
                lo(N + 2, N);
                lo(N + 2, N + 1);
                group();
                const bool fsplit = sap_round(6 + 3 * RMAX, vec) > K;   // as FSPLIT in the kernel
                put(-1, N + 2);
                vd(N + 2);
                if (fsplit) group();
                put(-1, N + 1);
                up(N + 1, N + 2);
                vd(N + 1);
                if (fsplit) group();
                put(-1, N);
                up(N, N + 1);
                up(N, N + 2);
                vd(N);
                group();
                const int BW = 1 + NF + sw + RMAX, UB = sap_group_rows(BW, vec);
                for (int j0 = 0; j0 < N; j0 += UB) {
                    for (int j = j0; j < j0 + UB; ++j) {
                        const int i = N - 1 - j;
                        if (i < 0) {
                            zero(BW);
                            continue;
                        }
                        put(-1, i);
                        for (int f = 0; f < NF; ++f) up(i, N + f);
                        for (int k = sw - 1; k >= 0; --k) {
                            const int jj = i + 1 + k;
                            if (jj < N) up(i, jj);
                            else put(-4, 0);
                        }
                        vd(i);
                    }
                    group();
                }
                const int UT = sap_group_rows(RMAX, vec);
                const int tail_src = sap_fold(RMAX, sw) ? -5 : -3;
                for (int q0 = 0; q0 < b; q0 += UT) {
                    for (int q = q0; q < q0 + UT; ++q) {
                        if (q >= b) {
                            zero(RMAX);
                            continue;
                        }
                        for (int k = 0; k < RMAX; ++k) put(k < r ? tail_src : -4, k < r ? k * b + q : 0);
                    }
                    group();
                }
                while (src.size() % K) {
                    src.push_back(-4);
                    arg.push_back(0);
                }
                if (!fits) return set_error(STS_ERR_INVALID_ARG, "internal: structured apply group wider than a chunk");
                for (size_t e = 0; e < src.size(); ++e)
                    if (src[e] < -5 || (src[e] >= 0 && src[e] >= M.nnz_lu))
                        return set_error(STS_ERR_INVALID_ARG, "internal: structured apply table");
                M.s_lt[prec] = (int)src.size();
                if (sap_fold(RMAX, sw) && dir == 0) {       // positions of the folded tail, alike in both directions
                    std::vector<int> tp((size_t)std::max(r, 1) * b, 0);
                    for (size_t e = 0; e < src.size(); ++e)
                        if (src[e] == -5) tp[arg[e]] = (int)e;
                    STS_TRY(upload(h, &M.tail_pos[prec], tp));
                }
                // vectors to pack: those that scale an entry first; none for all zeros or folded tails
                std::vector<int> list, plain;
                for (int v = 0; v < (int)src.size() / vec; ++v) {
                    bool any = false, scaled = false, folded = false;
                    for (int e = v * vec; e < (v + 1) * vec; ++e) {
                        any = any || src[e] > -4;
                        scaled = scaled || (src[e] >= 0 && arg[e] >= 0);
                        folded = folded || src[e] == -5;
                    }
                    // a packed vector is written whole, beside the kernel's folding blocks
                    if (any && folded) return set_error(STS_ERR_INVALID_ARG, "internal: structured apply vector");
                    if (any) (scaled ? list : plain).push_back(v);
                }
                M.spk_scaled[prec][dir] = (int)list.size();
                list.insert(list.end(), plain.begin(), plain.end());
                M.spk_n[prec][dir] = (int)list.size();
                STS_TRY(upload(h, &M.spk_list[prec][dir], list));
                STS_TRY(upload(h, &M.spk_src[prec][dir], src));
                STS_TRY(upload(h, &M.spk_arg[prec][dir], arg));
            }
        }
    }
    if (!M.structured) {
        STS_TRY(upload(h, &M.lu_diag, M.h_lu_diag));
        STS_TRY(upload(h, &M.src_slot, M.h_src_slot));
        STS_TRY(upload(h, &M.d_ptr, h->dptr));
        STS_TRY(upload(h, &M.f_colL_ptr, colL_ptr));
        STS_TRY(upload(h, &M.f_colL_slot, colL_slot));
        STS_TRY(upload(h, &M.f_upd_ptr, upd_ptr));
        STS_TRY(upload(h, &M.f_upd_tgt, upd_tgt));
        STS_TRY(upload(h, &M.f_upd_src, upd_src));
    }
    const size_t P = h->ncp;
    const int r = h->r_diag;
    // zero in the padding cells and in the pairs that a block does not have (u = v = 0
    // leaves A_k unchanged and adds an identity row and column to C_k)
    STS_TRY(dalloc_zero(h, &M.Sd, (size_t)h->nnz_d * P));
    STS_TRY(dalloc_zero(h, &M.Ud, (size_t)std::max(r, 1) * b * P));
    STS_TRY(dalloc_zero(h, &M.Vd, (size_t)std::max(r, 1) * b * P));
    STS_TRY(dalloc(h, &M.lu, (size_t)M.nnz_lu * P));
    STS_TRY(dalloc(h, &M.dinv, (size_t)b * P));
    STS_TRY(dalloc(h, &M.W, (size_t)std::max(r, 1) * b * P));
    if (h->has_T) STS_TRY(dalloc(h, &M.Wt, (size_t)std::max(r, 1) * b * P));
    STS_TRY(dalloc(h, &M.Cinv, (size_t)std::max(r * r, 1) * P));
    for (int dir = 0; dir < 2; ++dir) {
        if (dir == 1 && !h->has_T) continue;
        const size_t len = M.structured ? (size_t)M.s_lt[0] : (size_t)kGenWarps * M.g_wlen[dir];
        const size_t len32 = M.structured ? (size_t)M.s_lt[1] : len;
        // the structured streams' zero padding is written here and never again
        STS_TRY(dalloc_zero(h, &M.ap64[dir], len * P));
        if (h->dtype == STS_MIXED) {
            STS_TRY(dalloc_zero(h, &M.ap32[dir], len32 * P));
            STS_TRY(dalloc(h, &M.W32[dir], (size_t)std::max(r, 1) * b * P));
            STS_TRY(dalloc(h, &M.DV32[dir], (size_t)std::max(r, 1) * b * P));
        }
    }
    M.err_cell = h->d_err + 1;
    return STS_OK;
}

template <typename T>
static sts_status smw_apply_t(sts_jac_s *h, int dir, const T *st, const T *dv, const T *W, const Vec<T> &x,
                              const Vec<T> &z) {
    const SmwPlan &M = h->smw;
    ApplyArgs<T> a;
    a.st = st; a.row = M.g_row[dir]; a.n_fwd = M.g_nf[dir]; a.n_bwd = M.g_nb[dir];
    a.dv = dv; a.W = W; a.Cinv = M.Cinv; a.x = x; a.y = z;
    a.wlen = M.g_wlen[dir]; a.b = h->b; a.r = h->r_diag; a.ncp = h->ncp; a.trans = dir;
    const int rmax = a.r <= 2 ? 2 : a.r <= 4 ? 4 : kMaxPairsDiag;
    const size_t smem = ((size_t)kGenWarps * std::min(rmax, kGenSum) + h->b) * kTile * sizeof(T);
    auto kern = rmax == 2 ? k_smw_apply<T, 2> : rmax == 4 ? k_smw_apply<T, 4> : k_smw_apply<T, kMaxPairsDiag>;
    if (smem > 48 * 1024) STS_CK(allow_all_smem(kern));
    kern<<<h->n_tiles, kGenWarps * kTile, smem, h->stream>>>(a);
    STS_LAUNCHED();
    return STS_OK;
}

bool smw_apply_any_layout(const sts_jac_s *h, int elem) { return !h->smw.structured || !sap_in_y(h->b, elem); }

sts_status smw_apply64(sts_jac_s *h, int dir, const Vec<double> &x, const Vec<double> &z) {
    const SmwPlan &M = h->smw;
    if (M.structured) return smw_sapply_t<double>(h, dir, M.ap64[dir], x, z);
    return smw_apply_t<double>(h, dir, M.ap64[dir], dir == 0 ? M.Vd : M.Ud, dir == 0 ? M.W : M.Wt, x, z);
}

sts_status smw_apply32(sts_jac_s *h, int dir, const Vec<float> &x, const Vec<float> &z) {
    const SmwPlan &M = h->smw;
    if (M.structured) return smw_sapply32(h, dir, x, z);
    return smw_apply_t<float>(h, dir, M.ap32[dir], M.DV32[dir], M.W32[dir], x, z);
}

}  // namespace sts
