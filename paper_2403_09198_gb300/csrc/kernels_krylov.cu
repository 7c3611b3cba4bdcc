// kernels_krylov.cu -- restarted right-preconditioned GMRES(m) on the device.
//
// Section 6 (Eq. right_precond_system): solve (A M) y = b, x = M y.  Each
// cycle starts from the true FP64 residual r = b - A x, builds the Krylov basis
// by classical Gram-Schmidt with a second pass (CGS2: dots, update and dots
// in one sweep, update and norm; same result as modified Gram-Schmidt in exact
// arithmetic), reduces the Hessenberg matrix with Givens rotations in FP64 (on the
// device in cycles that run as a graph, on the host in the others) and updates
// x += Z y with Z = [M v_0, ..., M v_{k-1}] (for a fixed M this equals x += M (V y)).  Convergence is declared on the recomputed true
// residual only.  Mixed mode (flexible GMRES): z_j = M32(v_j) and w = A32 z_j in
// FP32; the basis, the orthogonalisation, x and the residual refresh stay FP64.
// Left preconditioning (Eq. left_precond_system, (M A) x = M b): the cycle's
// first vector is M r / ||M r||, each step forms w = M (A v_j), x += V y, and a
// cycle stops when the preconditioned residual has fallen by the factor the
// true residual still needs.
//
// All reductions are deterministic: a fixed grid writes per-block partial sums
// and the block that finishes last adds them in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "ring.cuh"
#include "sts_internal.h"

namespace sts {
namespace {

constexpr int kRedThreads = 256;
constexpr int kRedMax = 304;        // blocks of a reduction with several totals at most: two per SM
constexpr int kOrthChunk = 31;      // vectors per sweep: their dots and w . w fill a warp's 32 lanes

// Blocks of the sweeps over n elements and cnt vectors, one element per thread at
// least.  The sums depend on this number: it is a function of n and cnt alone, so that
// every caller gets the same bits.  Above kTwoBlocks vectors the accumulators leave
// room for one block per SM; the last sweep has none, and four blocks per SM hide its
// serial FMA chains (128 x 128 cells, N = 60, 28 / 30 vectors: 86 / 94 -> 71 / 75 us;
// 24 and fewer are faster in two blocks: 61 against 63 us, 2 vectors 15.5 against 16.9).
constexpr int kTwoBlocks = 24;
inline int orth_blocks(long long n, int cnt, bool norm_only = false) {
    const long long most = cnt <= kTwoBlocks ? kRedMax : norm_only ? 2 * kRedMax : kRedMax / 2;
    return (int)std::max(1LL, std::min(most, (n + kRedThreads - 1) / kRedThreads));
}

// Whether a sweep is launched early (programmatic dependent launch): on small grids,
// where its blocks wait beside the previous kernel's.  On full ones they take the
// place of blocks that have work (measured on 125 x 121 cells, N = 60: GMRES 1.55 -> 1.59 ms).
inline bool early_start(int blocks) { return blocks < kRedMax / 2; }

// Sum each of the NV values of v over the warp: lane l returns the sum of value
// l >> (5 - log2 of NV rounded up to a power of two).  Every exchange halves the values
// that a lane still carries, so NV values take NV - 1 + (5 - log2 NV) FP64 additions
// instead of 5 NV (an FP64 addition holds the pipe for 64 cycles whatever the lanes).
template <int NV>
__device__ __forceinline__ double warp_sums(double (&v)[NV], int lane) {
    static_assert(NV >= 1 && NV <= 32 && (NV & (NV - 1)) == 0, "a power of two");
    int mask = 16;
#pragma unroll
    for (int half = NV / 2; half >= 1; half /= 2, mask /= 2) {
        const bool up = lane & mask;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const double send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
        }
    }
    double s = v[0];
    for (; mask >= 1; mask /= 2) s += __shfl_xor_sync(0xffffffffu, s, mask);
    return s;
}

// Totals of NV values over the whole grid, into out[0..NV), by the block that finishes
// last; true in that block (after its stores).  Every block's sums go to
// partial[block][0..NV); the last block adds them in a fixed order (warp w takes
// blocks w, w + 8, ..., lane = value, then the warps in order), so the result never
// depends on which block is last.  The ticket counts finished blocks and is reset.
template <int NV>
__device__ __forceinline__ bool grid_totals(double (&v)[NV], int used, double *partial, double *out,
                                            unsigned int *ticket) {
    constexpr int NW = kRedThreads / 32, SH = NV == 32 ? 0 : NV == 16 ? 1 : NV == 8 ? 2 : NV == 4 ? 3 : NV == 2 ? 4 : 5;
    __shared__ double sh[NW][NV];
    __shared__ bool last;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double s = warp_sums<NV>(v, lane);
    if ((lane & ((1 << SH) - 1)) == 0) sh[w][lane >> SH] = s;
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = sh[0][threadIdx.x];
#pragma unroll
        for (int k = 1; k < NW; ++k) t += sh[k][threadIdx.x];
        partial[(size_t)blockIdx.x * NV + threadIdx.x] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
    // 32 / NV blocks side by side in a warp, so that every lane adds
    const int per = 1 << SH, o = lane & (NV - 1), b0 = w * per + lane / NV;
    double t = 0.0;
    for (int b = b0; b < (int)gridDim.x; b += NW * per) t += __ldcg(partial + (size_t)b * NV + o);
#pragma unroll
    for (int m = 16; m >= NV; m /= 2) t += __shfl_xor_sync(0xffffffffu, t, m);
    if (lane < NV) sh[w][lane] = t;
    __syncthreads();
    if (threadIdx.x < used) {
        t = sh[0][threadIdx.x];
#pragma unroll
        for (int k = 1; k < NW; ++k) t += sh[k][threadIdx.x];
        out[threadIdx.x] = t;
    }
    if (threadIdx.x == 0) *ticket = 0u;
    __syncthreads();
    return true;
}

// State of the device-side rotations (see givens_step); H = NULL: none.
struct Givens {
    int j, m;
    const double *h1, *h2;
    double *H, *cs, *sn, *g, *hist, *par;
    int *state;
    cudaGraphConditionalHandle next;
    int has_next;
};

// Step j's rotations, by one block: h1, h2 the two passes' coefficients of column j, hn2
// the squared norm of w after them (before them it is hn2 plus the squares of the
// first ones, the basis being orthonormal); par: stop threshold, history
// scale, 1 / h(j+1,j) (output), steps allowed; state: steps taken, stop reason (0 none,
// 1 criterion met, 2 NaN or Inf).  An FP64 operation takes a whole warp 64 cycles or
// more, so what can run beside the recurrence does, in other lanes (the products with
// the column's entries) and other warps (the square root of w2, 1 / hn), and a step of
// the recurrence is one FMA.  As one thread's loop over global memory it took 5.6 us
// (j = 0) to 14 us (j = 29).
constexpr int kGivensMax = 64;
__device__ __noinline__ void givens_step(const Givens &G, double hn2) {
    // t[i]: column entry i after rotations 0 .. i - 1; u[i], v[i]: c_i, s_i times entry i + 1
    __shared__ double c[kGivensMax], sn[kGivensMax], t[kGivensMax], u[kGivensMax], v[kGivensMax], hn, w2;
    const int j = G.j, m = G.m, x = threadIdx.x;
    int bad = 0;
    if (x <= j) {
        const double h = G.h1[x] + G.h2[x];
        bad = !isfinite(h);
        if (x == 0) t[0] = h;
        else {
            c[x - 1] = G.cs[x - 1];
            sn[x - 1] = G.sn[x - 1];
            u[x - 1] = c[x - 1] * h;
            v[x - 1] = sn[x - 1] * h;
        }
    }
    if (x >= 64 && x < 96) {
        double q = 0.0;
        for (int i = x - 64; i <= j; i += 32) q = fma(G.h1[i], G.h1[i], q);
#pragma unroll
        for (int k = 16; k >= 1; k /= 2) q += __shfl_xor_sync(0xffffffffu, q, k);
        if (x == 64) {
            w2 = q + hn2;
            bad = !isfinite(w2);        // it tells a breakdown from an overflow
        }
    } else if (x == 96) {
        hn = sqrt(hn2);
        G.par[2] = 1.0 / hn;
        bad = !isfinite(hn);
    }
    bad = __syncthreads_or(bad);
    if (x == 0) {
        int stop = 2;
        if (!bad) {
            double a = t[0];
            for (int i = 0; i < j; ++i) {
                a = fma(-sn[i], a, u[i]);
                t[i + 1] = a;
            }
            // hypot(a, hn) where neither square leaves the range
            const int ea = (__double2hiint(a) >> 20) & 0x7ff, eh = (__double2hiint(hn) >> 20) & 0x7ff, e = max(ea, eh);
            const double den = e > 1023 - 450 && e < 1023 + 450 ? sqrt(fma(a, a, hn * hn)) : hypot(a, hn);
            const double inv = 1.0 / den, cj = a * inv, sj = hn * inv, gj = G.g[j], gn = -sj * gj;
            G.cs[j] = cj;
            G.sn[j] = sj;
            G.g[j + 1] = gn;
            G.g[j] = cj * gj;
            G.hist[j] = fabs(gn) * G.par[1];
            G.H[(size_t)j * m + j] = den;
            const bool happy = hn2 <= 1e-28 * w2;
            stop = happy || fabs(gn) <= G.par[0] || (double)(j + 1) >= G.par[3] ? 1 : 0;
        }
        G.state[0] = j + 1;
        G.state[1] = stop;
        if (G.has_next) cudaGraphSetConditional(G.next, stop ? 0u : 1u);
    }
    __syncthreads();
    if (x < j) G.H[(size_t)x * m + j] = fma(c[x], t[x], v[x]);
    if (x == j + 1) G.H[(size_t)x * m + j] = 0.0;
}

// One sweep over w and CNT basis vectors V (contiguous, n apart):
//   kDots        out[i] = V_i . w, out[CNT] = w . w
//   kDotsOnly    out[i] = V_i . w
//   kUpdateDots  w -= sum_i h_i V_i, then out[i] = V_i . w with the same loaded V
//   kUpdateNorm  w -= sum_i h_i V_i, out[0] = w . w, and the rotations that need it
// The count is a template parameter: a predicated-off FP64 FMA still takes its pipe
// slot, so the loop issues exactly the FMAs it needs.  U elements per thread and
// iteration keep several loads in flight where CNT is small.  Bound by the FP64 pipe
// from about eight vectors on (one FMA per loaded value, two in kUpdateDots), by
// memory below.  Measured on 128 x 128 cells, N = 60 (1.03 M elements): with dots,
// update, dots and update as four sweeps and 5 additions per value and warp in the
// reductions, the 163 steps of a Newton step (16 vectors on average) took 31.3 ms, now
// 22.4 ms, the rotations included; 18.2 ms are FP64 pipe time.
enum { kDots, kDotsOnly, kUpdateDots, kUpdateNorm };

constexpr int pow2_at_least(int n) { return n <= 1 ? 1 : n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : n <= 16 ? 16 : 32; }

template <int CNT, int MODE>
__global__ void __launch_bounds__(kRedThreads, CNT <= kTwoBlocks ? 2 : MODE == kUpdateNorm ? 4 : 1)
    k_orth(double *w, const double *V, long long n, const double *hcoef, double *partial, double *out,
           int n_out, unsigned int *ticket, Givens G) {
    constexpr int U = CNT <= 1 ? 8 : CNT <= 3 ? 4 : CNT <= (MODE == kUpdateNorm ? kTwoBlocks - 1 : 6) ? 2 : 1;
    constexpr int C1 = CNT > 0 ? CNT : 1;
    constexpr bool UPD = MODE == kUpdateDots || MODE == kUpdateNorm;
    // the same tree in all modes that return dots, so that they return the same bits
    constexpr int NO = MODE == kUpdateNorm ? 1 : CNT + 1, NV = pow2_at_least(NO);
    __shared__ double h[C1];
    pdl_wait();
    pdl_trigger();
    if (UPD) {
        if (threadIdx.x < CNT) h[threadIdx.x] = __ldcg(hcoef + threadIdx.x);
        __syncthreads();
    }
    double acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    auto step = [&](double we, const double (&v)[C1], long long e) {
        if (UPD) {
#pragma unroll
            for (int i = 0; i < CNT; ++i) we = fma(-h[i], v[i], we);
            w[e] = we;
        }
        if (MODE != kUpdateNorm) {
#pragma unroll
            for (int i = 0; i < CNT; ++i) acc[i] = fma(v[i], we, acc[i]);
        }
        if (MODE == kDots || MODE == kUpdateNorm) acc[NO - 1] = fma(we, we, acc[NO - 1]);
    };
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; e + (U - 1) * stride < n; e += U * stride) {
        double we[U], v[U][C1];
#pragma unroll
        for (int u = 0; u < U; ++u) we[u] = w[e + u * stride];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < CNT; ++i) v[u][i] = __ldg(V + (size_t)i * n + e + u * stride);
#pragma unroll
        for (int u = 0; u < U; ++u) step(we[u], v[u], e + u * stride);
    }
    for (; e < n; e += stride) {
        double v[C1];
#pragma unroll
        for (int i = 0; i < CNT; ++i) v[i] = __ldg(V + (size_t)i * n + e);
        step(w[e], v, e);
    }
    const bool last = grid_totals<NV>(acc, n_out, partial, out, ticket);
    if (MODE == kUpdateNorm && last && G.H) givens_step(G, out[0]);
}

using OrthKernel = void (*)(double *, const double *, long long, const double *, double *, double *, int,
                            unsigned int *, Givens);
template <int MODE, int... I>
OrthKernel orth_kernel(int cnt, std::integer_sequence<int, I...>) {
    // kDots without vectors is the norm; the other modes have at least one
    constexpr int least = MODE == kDots ? 0 : 1;
    static const OrthKernel k[] = {k_orth<I + least, MODE>...};
    return k[cnt - least];
}

sts_status orth_launch(int mode, int cnt, double *w, const double *V, long long n, const double *hcoef,
                       double *partial, double *out, int n_out, unsigned int *ticket, cudaStream_t st,
                       const Givens &G = {}) {
    using All = std::make_integer_sequence<int, kOrthChunk>;
    const OrthKernel k = mode == kDots ? orth_kernel<kDots>(cnt, std::make_integer_sequence<int, kOrthChunk + 1>{})
                         : mode == kDotsOnly ? orth_kernel<kDotsOnly>(cnt, All{})
                         : mode == kUpdateDots ? orth_kernel<kUpdateDots>(cnt, All{}) : orth_kernel<kUpdateNorm>(cnt, All{});
    const int blocks = orth_blocks(n, cnt, mode == kUpdateNorm);
    if (early_start(blocks))
        STS_CK(launch_pdl(k, dim3(blocks), dim3(kRedThreads), 0, st, w, V, n, hcoef, partial, out, n_out, ticket, G));
    else
        k<<<blocks, kRedThreads, 0, st>>>(w, V, n, hcoef, partial, out, n_out, ticket, G);
    STS_LAUNCHED();
    return STS_OK;
}

__global__ void k_sub(double *r, const double *b, const double *y, long long n) {
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        r[e] = b[e] - y[e];
}

// What k_residual leaves beside the norm after a graph cycle (err = NULL: nothing): a copy
// of the handle's error flag, and whether the solve ends here with a result, as the host
// will decide it from the same numbers (its square root and quotient round alike): steps
// that did not break down, a finite norm, and rtol reached or none of the `left` steps left.
struct CycleEnd {
    const int *err, *state;
    double bnorm, rtol;
    int left;
    int *err_out, *done;
};

// r = b - y and out[0] = r . r, in the order of a difference followed by a norm.
__global__ void __launch_bounds__(kRedThreads, 2) k_residual(double *r, const double *b, const double *y, long long n,
                                                             double *partial, double *out, unsigned int *ticket,
                                                             CycleEnd E) {
    constexpr int U = 4;
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; e + (U - 1) * stride < n; e += U * stride) {
        double v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = b[e + u * stride] - y[e + u * stride];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            r[e + u * stride] = v[u];
            acc[0] = fma(v[u], v[u], acc[0]);
        }
    }
    for (; e < n; e += stride) {
        const double v = b[e] - y[e];
        r[e] = v;
        acc[0] = fma(v, v, acc[0]);
    }
    if (grid_totals<1>(acc, 1, partial, out, ticket) && E.err && threadIdx.x == 0) {
        const double norm = sqrt(out[0]);
        *E.err_out = *E.err;
        *E.done = E.state[1] != 2 && isfinite(norm) && (norm / E.bnorm <= E.rtol || E.state[0] >= E.left);
    }
}

// out[y] = ||v_y||^2 of the two vectors, blockIdx.y = y, each in the order of its own sweep.
__global__ void __launch_bounds__(kRedThreads, 2) k_two_norms(const double *v0, const double *v1, long long n,
                                                              double *partial, double *out, unsigned int *ticket) {
    constexpr int U = 8;
    const double *v = blockIdx.y ? v1 : v0;
    double acc[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; e + (U - 1) * stride < n; e += U * stride) {
        double x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = v[e + u * stride];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[0] = fma(x[u], x[u], acc[0]);
    }
    for (; e < n; e += stride) acc[0] = fma(v[e], v[e], acc[0]);
    grid_totals<1>(acc, 1, partial + blockIdx.y * kRedMax, out + blockIdx.y, ticket + blockIdx.y);
}

// Least-squares coefficients of a finished graph cycle, y = R^-1 g for the k steps taken
// (k = 0 after a NaN): one warp, lane = rows l and l + 32, pivots inverted beforehand so
// that a step of the back substitution is a product and an FMA.
__global__ void __launch_bounds__(kTile) k_cycle_y(const double *H, const double *g, int m, int *state, double *y) {
    const int l = threadIdx.x, k = state[1] == 2 ? 0 : state[0];
    double s[2], inv[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = l + 32 * h;
        s[h] = i < k ? g[i] : 0.0;
        inv[h] = i < k ? 1.0 / H[(size_t)i * m + i] : 0.0;
    }
    for (int i = k - 1; i >= 0; --i) {
        const double yi = __shfl_sync(0xffffffffu, i < 32 ? s[0] * inv[0] : s[1] * inv[1], i & 31);
        if (l == 0) y[i] = yi;
        if (l < i) s[0] = fma(-H[(size_t)l * m + i], yi, s[0]);
        if (l + 32 < i) s[1] = fma(-H[(size_t)(l + 32) * m + i], yi, s[1]);
    }
}

__global__ void k_scale(double *out, const double *in, double s, long long n) {
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        out[e] = in[e] * s;
}

// state: with it, the number of vectors is the steps of a graph cycle (see k_cycle_y)
template <typename T>
__global__ void k_axpy_multi(double *x, const T *Z, long long n, const double *y, int k, const int *state) {
    __shared__ double ys[64];
    if (state) k = state[1] == 2 ? 0 : state[0];
    for (int i0 = 0; i0 < k; i0 += 64) {
        const int cnt = min(64, k - i0);
        __syncthreads();
        if (threadIdx.x < cnt) ys[threadIdx.x] = y[i0 + threadIdx.x];
        __syncthreads();
        for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
             e += (long long)gridDim.x * blockDim.x) {
            double v = x[e];
            for (int i = 0; i < cnt; ++i) v = fma(ys[i], (double)Z[(size_t)(i0 + i) * n + e], v);
            x[e] = v;
        }
    }
}

template <typename To, typename Ti>
__global__ void k_convert(To *out, const Ti *in, long long n) {
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        out[e] = (To)in[e];
}

inline int grid_for(long long n, int block) {
    long long g = (n + block - 1) / block;
    if (g > 152LL * 32) g = 152LL * 32;
    if (g < 1) g = 1;
    return (int)g;
}

// Operators shared with the public entry points.
sts_status opA64(sts_jac_s *h, int dir, const double *x, double *y) {
    if (h->rep == STS_REP_DENSE_BSR) return dense_matvec(h, x, y);
    return mv_apply64(h, dir, internal_vec(h, x), internal_vec(h, y), h->c64);
}
sts_status opM64(sts_jac_s *h, int dir, const double *x, double *z) {
    if (h->rep == STS_REP_DENSE_BSR) return dense_apply(h, x, z);
    return smw_apply64(h, dir, internal_vec(h, x), internal_vec(h, z));
}

struct Red {
    sts_jac_s *h;
    long long n;
    // device: per-block partials in h->kry.partial, totals written by each
    // kernel's last block (h->kry.ticket)
    sts_status dots(const double *V, int k, const double *w, int self, double *out) {
        Krylov &K = h->kry;
        for (int i0 = 0; i0 < k; i0 += kOrthChunk) {
            const int cnt = std::min(kOrthChunk, k - i0);
            const int sf = self && i0 + cnt == k;
            STS_TRY(orth_launch(sf ? kDots : kDotsOnly, cnt, const_cast<double *>(w), V + (size_t)i0 * n, n, nullptr,
                                K.partial, out + i0, cnt + (sf ? 1 : 0), K.ticket, h->stream));
        }
        return STS_OK;
    }
    // the squared norm goes to out[0] (norm = 1) and, with G.H, on to the rotations
    sts_status update(double *w, const double *V, int k, const double *hcoef, int norm, double *out,
                      const Givens &G = {}) {
        Krylov &K = h->kry;
        for (int i0 = 0; i0 < k; i0 += kOrthChunk) {
            const int cnt = std::min(kOrthChunk, k - i0), fin = norm && i0 + cnt == k;
            STS_TRY(orth_launch(kUpdateNorm, cnt, w, V + (size_t)i0 * n, n, hcoef + i0, K.partial, out, fin, K.ticket,
                                h->stream, fin ? G : Givens{}));
        }
        return STS_OK;
    }
    // update with hcoef, then the dots of the result
    sts_status update_dots(double *w, const double *V, int k, const double *hcoef, double *out) {
        Krylov &K = h->kry;
        if (k <= kOrthChunk)
            return orth_launch(kUpdateDots, k, w, V, n, hcoef, K.partial, out, k, K.ticket, h->stream);
        STS_TRY(update(w, V, k, hcoef, 0, nullptr));
        return dots(V, k, w, 0, out);
    }
    sts_status norm2(const double *v, double *out) {
        Krylov &K = h->kry;
        return orth_launch(kDots, 0, const_cast<double *>(v), v, n, nullptr, K.partial, out, 1, K.ticket, h->stream);
    }
};

sts_status ensure_workspace(sts_jac_s *h, int m, bool mixed) {
    Krylov &K = h->kry;
    const size_t n = (size_t)h->b * h->ncp;
    if (K.m < m) {
        // a larger restart replaces the basis buffers (the stream is idle here:
        // every solve ends with a synchronisation)
        STS_CK(cudaStreamSynchronize(h->stream));
        dev_free(h, K.V);
        dev_free(h, K.Z);
        dev_free(h, K.Z32);
        dev_free(h, K.partial);
        dev_free(h, K.red);
        K.V = K.Z = K.partial = K.red = nullptr;
        // the cycle graphs hold the old buffers and sizes
        for (auto &row : K.gexec)
            for (auto &ge : row) {
                if (ge) cudaGraphExecDestroy(ge);
                ge = nullptr;
            }
        dev_free(h, K.gbuf);
        K.gbuf = nullptr;
        if (K.g_pinned) cudaFreeHost(K.g_pinned);
        K.g_pinned = nullptr;
        K.Z32 = nullptr;
        K.m = 0;
        STS_TRY(dalloc(h, &K.V, (size_t)(m + 1) * n));
        STS_TRY(dalloc(h, &K.Z, (size_t)m * n));
        STS_TRY(dalloc(h, &K.partial, (size_t)kRedMax * 32));      // at least two rows of kRedMax
        STS_TRY(dalloc(h, &K.red, (size_t)3 * (m + 2)));
        if (!K.ticket) {
            STS_TRY(dalloc_zero(h, &K.ticket, 2));
        }
        if (!K.w) {
            STS_TRY(dalloc(h, &K.w, n));
            STS_TRY(dalloc(h, &K.r, n));
            STS_TRY(dalloc(h, &K.xb, n));
            STS_TRY(dalloc(h, &K.bb, n));
            STS_TRY(dalloc(h, &K.tmp, n));
        }
        if (K.h_pinned) cudaFreeHost(K.h_pinned);
        K.h_pinned = nullptr;
        STS_CK(cudaMallocHost(&K.h_pinned, sizeof(double) * 3 * (m + 2)));
        K.m = m;
    }
    if (mixed && !K.Z32) {
        STS_TRY(dalloc(h, &K.Z32, (size_t)K.m * n));
        if (!K.t32a) {
            STS_TRY(dalloc(h, &K.t32a, n));
            STS_TRY(dalloc(h, &K.t32b, n));
        }
    }
    return STS_OK;
}

// ---------------------------------------------------------------------------
// One Arnoldi cycle as a CUDA graph.  Step j of the cycle is the body of a
// conditional (IF) node, nested in step j - 1's body: z_j = M v_j, w = A z_j,
// the two Gram-Schmidt passes,
// of which the last folds the new Hessenberg column into the rotations on
// the device (the host loop's rotations, rounded otherwise: FMAs of products formed
// beforehand, reciprocals for quotients, a square root for hypot, and a breakdown
// judged against ||w||^2 from the first pass's coefficients, the basis being
// orthonormal, instead of w . w; the two need not agree in the last bits), records the
// rotated residual, and switches step j + 1 on or off, and finally v_{j+1} =
// w / h(j+1, j).  The host launches the graph once per cycle and reads the
// rotated system back once, instead of synchronising after every step.

__global__ void k_scale_dev(double *out, const double *in, const double *s, long long n) {
    pdl_wait();
    pdl_trigger();
    const double f = *s;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        out[e] = in[e] * f;
}

// Build (once per restart length, direction, preconditioning and stream) the
// graph of a whole cycle of m steps.  The kernels of a step are recorded by
// capturing the ordinary host code on a private stream into the step's body.
sts_status cycle_graph(sts_jac_s *h, int m, int dir, bool pre) {
    Krylov &K = h->kry;
    cudaGraphExec_t &exec = K.gexec[dir][pre ? 1 : 0];
    if (exec && K.g_m[dir][pre ? 1 : 0] == m && K.g_stream[dir][pre ? 1 : 0] == h->stream) return STS_OK;
    if (exec) cudaGraphExecDestroy(exec);
    exec = nullptr;
    if (!K.gbuf) {
        // what the host writes before a cycle and reads after it first, in one piece
        const size_t M = (size_t)K.m, io = 8 + (M + 1) + M;
        STS_TRY(dalloc(h, &K.gbuf, io + (M + 1) * M + 3 * M));
        K.gpar = K.gbuf;
        K.gstate = reinterpret_cast<int *>(K.gbuf + 4);
        K.grn = K.gbuf + 5;
        K.gerr = reinterpret_cast<int *>(K.gbuf + 6);
        K.gdone = reinterpret_cast<int *>(K.gbuf + 7);
        K.gg = K.gbuf + 8;
        K.ghist = K.gg + (M + 1);
        K.gH = K.gbuf + io;
        K.gcs = K.gH + (M + 1) * M;
        K.gsn = K.gcs + M;
        K.gy = K.gsn + M;
        STS_CK(cudaMallocHost(&K.g_pinned, sizeof(double) * io));
    }
    const long long n = (long long)h->b * h->ncp;
    const int ld = m + 2, nb = grid_for(n, 256);
    cudaGraph_t graph = nullptr;
    STS_CK(cudaGraphCreate(&graph, 0));
    cudaStream_t cs = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        cudaGraphDestroy(graph);
        return set_error(STS_ERR_CUDA, "gmres graph: cudaStreamCreate failed: %s", cudaGetErrorString(e));
    }
    std::vector<cudaGraphConditionalHandle> hd(m);
    sts_status st = STS_OK;
    for (int j = 0; j < m && e == cudaSuccess; ++j)
        e = cudaGraphConditionalHandleCreate(&hd[j], graph, j == 0 ? 1u : 0u, cudaGraphCondAssignDefault);
    cudaStream_t saved = h->stream;
    // step j + 1's conditional node sits at the end of step j's body, so once a
    // step switches the next one off nothing further of the cycle is evaluated
    cudaGraph_t parent = graph;
    std::vector<cudaGraphNode_t> deps;
    Red R{h, n};
    for (int j = 0; j < m && e == cudaSuccess && st == STS_OK; ++j) {
        cudaGraphNodeParams p = {};
        p.type = cudaGraphNodeTypeConditional;
        p.conditional.handle = hd[j];
        p.conditional.type = cudaGraphCondTypeIf;
        p.conditional.size = 1;
        cudaGraphNode_t node = nullptr;
        e = cudaGraphAddNode(&node, parent, deps.empty() ? nullptr : deps.data(), nullptr, deps.size(), &p);
        if (e != cudaSuccess) break;
        cudaGraph_t body = p.conditional.phGraph_out[0];
        e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
        if (e != cudaSuccess) break;
        h->stream = cs;
        auto step = [&]() -> sts_status {
            double *vj = K.V + (size_t)j * n, *zj = K.Z + (size_t)j * n;
            if (pre) STS_TRY(opM64(h, dir, vj, zj));
            else STS_CK(cudaMemcpyAsync(zj, vj, n * sizeof(double), cudaMemcpyDeviceToDevice, cs));
            STS_TRY(opA64(h, dir, zj, K.w));
            double *h1 = K.red, *h2 = K.red + ld, *nr = K.red + 2 * ld;
            const int has_next = j + 1 < m ? 1 : 0;
            const Givens G{j, m, h1, h2, K.gH, K.gcs, K.gsn, K.gg, K.ghist, K.gpar, K.gstate,
                           has_next ? hd[j + 1] : hd[j], has_next};
            STS_TRY(R.dots(K.V, j + 1, K.w, 0, h1));
            STS_TRY(R.update_dots(K.w, K.V, j + 1, h1, h2));
            STS_TRY(R.update(K.w, K.V, j + 1, h2, 1, nr, G));
            if (has_next) {
                double *vn = K.V + (size_t)(j + 1) * n;
                if (early_start(nb)) STS_CK(launch_pdl(k_scale_dev, dim3(nb), dim3(256), 0, cs, vn, K.w, K.gpar + 2, n));
                else k_scale_dev<<<nb, 256, 0, cs>>>(vn, K.w, K.gpar + 2, n);
                STS_LAUNCHED();
            }
            return STS_OK;
        };
        st = step();
        h->stream = saved;
        if (st == STS_OK) {
            cudaStreamCaptureStatus cst;
            const cudaGraphNode_t *last = nullptr;
            size_t nlast = 0;
            e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, nullptr, &last, nullptr, &nlast);
            if (e == cudaSuccess) deps.assign(last, last + nlast);
        }
        cudaGraph_t captured = nullptr;
        const cudaError_t e2 = cudaStreamEndCapture(cs, &captured);
        if (e == cudaSuccess) e = e2;
        parent = body;
    }
    h->stream = saved;
    if (st == STS_OK && e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    cudaStreamDestroy(cs);
    if (st != STS_OK) return st;
    if (e != cudaSuccess) {
        exec = nullptr;
        return set_error(STS_ERR_CUDA, "gmres graph: building the cycle graph failed: %s", cudaGetErrorString(e));
    }
    K.g_m[dir][pre ? 1 : 0] = m;
    K.g_stream[dir][pre ? 1 : 0] = h->stream;
    return STS_OK;
}

}  // namespace

// Krylov building blocks on one handle's internal vectors of n = b * ncp
// entries, for the domain-decomposed driver (kernels_dd.cu).  Reductions leave
// their totals in device memory (out_dev); the caller copies them out.
sts_status kry_reserve(sts_jac_s *h, int m) { return ensure_workspace(h, m, false); }
sts_status kry_dots(sts_jac_s *h, const double *V, int k, const double *w, int self, double *out_dev) {
    Red R{h, (long long)h->b * h->ncp};
    return R.dots(V, k, w, self, out_dev);
}
sts_status kry_update(sts_jac_s *h, double *w, const double *V, int k, const double *hcoef_dev, int norm,
                      double *out_dev) {
    Red R{h, (long long)h->b * h->ncp};
    return R.update(w, V, k, hcoef_dev, norm, out_dev);
}
sts_status kry_norm2(sts_jac_s *h, const double *v, double *out_dev) {
    Red R{h, (long long)h->b * h->ncp};
    return R.norm2(v, out_dev);
}
sts_status kry_sub(sts_jac_s *h, double *r, const double *b, const double *y) {
    const long long n = (long long)h->b * h->ncp;
    k_sub<<<grid_for(n, 256), 256, 0, h->stream>>>(r, b, y, n);
    STS_LAUNCHED();
    return STS_OK;
}
sts_status kry_scale(sts_jac_s *h, double *out, const double *in, double s) {
    const long long n = (long long)h->b * h->ncp;
    k_scale<<<grid_for(n, 256), 256, 0, h->stream>>>(out, in, s, n);
    STS_LAUNCHED();
    return STS_OK;
}
sts_status kry_axpy(sts_jac_s *h, double *x, const double *Z, int k, const double *y_dev) {
    const long long n = (long long)h->b * h->ncp;
    k_axpy_multi<double><<<grid_for(n, 256), 256, 0, h->stream>>>(x, Z, n, y_dev, k, nullptr);
    STS_LAUNCHED();
    return STS_OK;
}

sts_status op_matvec64(sts_jac_s *h, int dir, const double *x, double *y) { return opA64(h, dir, x, y); }
sts_status op_apply64(sts_jac_s *h, int dir, const double *x, double *z) { return opM64(h, dir, x, z); }

// *checked: the solve has read the handle's error flag after its last kernel that may set it,
// and found it clear.
sts_status gmres(sts_jac_s *h, const double *b_pub, double *x_pub, const sts_gmres_opts *o,
                 sts_gmres_info *info, bool *checked) {
    *checked = false;
    sts_gmres_opts d{};
    if (o) d = *o;
    const int m = d.restart > 0 ? d.restart : 30;
    const int max_iters = d.max_iters > 0 ? d.max_iters : 1000;
    const double rtol = d.rtol > 0 ? d.rtol : 1e-10;
    const double inner = d.inner_rtol > 0 ? d.inner_rtol : 1e-6;
    const bool pre = d.precond != STS_PRECOND_NONE;
    const int dir = d.trans ? 1 : 0;
    const bool mixed = d.mixed != 0;
    const bool left = d.left != 0;
    // graph cycles for right preconditioning in FP64, unless the caller asks for
    // host-driven steps; restart lengths above 64 keep the host loop (a step's
    // conditional node is nested in the previous step's body)
    const bool use_graph = d.arnoldi != STS_ARNOLDI_HOST && !left && !mixed && m <= 64;
    if (left && (!pre || mixed))
        return set_error(STS_ERR_INVALID_ARG, "gmres: left preconditioning needs precond BJ and mixed = 0");
    if (d.precond != STS_PRECOND_BJ && d.precond != STS_PRECOND_NONE)
        return set_error(STS_ERR_INVALID_ARG, "gmres: unknown precond %d", d.precond);
    if (m > 512) return set_error(STS_ERR_INVALID_ARG, "gmres: restart %d exceeds 512", m);
    if (dir == 1 && (!h->has_T || h->rep != STS_REP_FACTORED))
        return set_error(STS_ERR_INVALID_ARG, "gmres: trans = 1 needs a factored handle created with enable_transpose");
    if (mixed && (h->dtype != STS_MIXED || h->rep != STS_REP_FACTORED))
        return set_error(STS_ERR_INVALID_ARG, "gmres: mixed = 1 needs a factored handle created with dtype STS_MIXED");
    if (pre) {
        const bool ready = h->rep == STS_REP_FACTORED ? h->smw.ready : h->dense.ready;
        if (!ready) return set_error(STS_ERR_NOT_SETUP, "gmres: block-Jacobi preconditioner used before sts_jac_bjacobi_setup");
    }
    STS_TRY(ensure_workspace(h, m, mixed));
    Krylov &K = h->kry;
    const long long n = (long long)h->b * h->ncp;
    Red R{h, n};
    const int nb = grid_for(n, 256);
    const size_t vbytes = (size_t)h->nc * h->b * sizeof(double);
    // inputs into the internal layout
    const double *b_src = b_pub;
    const double *x_src = x_pub;
    if (d.vectors_on_host) {
        STS_CK(cudaMemcpyAsync(h->vin, b_pub, vbytes, cudaMemcpyHostToDevice, h->stream));
        STS_TRY(to_internal64(h, h->vin, K.bb));
        STS_CK(cudaMemcpyAsync(h->vin, x_pub, vbytes, cudaMemcpyHostToDevice, h->stream));
        STS_TRY(to_internal64(h, h->vin, K.xb));
    } else {
        STS_TRY(to_internal64(h, b_src, K.bb));
        STS_TRY(to_internal64(h, x_src, K.xb));
    }
    double *hp = K.h_pinned;
    // ||b||^2 and ||x0||^2: a zero guess starts from r = b without a product
    k_two_norms<<<dim3(orth_blocks(n, 0), 2), kRedThreads, 0, h->stream>>>(K.bb, K.xb, n, K.partial, K.red, K.ticket);
    STS_LAUNCHED();
    STS_CK(cudaMemcpyAsync(hp, K.red, 2 * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    STS_CK(cudaStreamSynchronize(h->stream));
    const double bnorm = std::sqrt(hp[0]);
    bool zero_guess = hp[1] == 0.0;
    if (!std::isfinite(bnorm)) return set_error(STS_ERR_NUMERIC, "gmres: right-hand side has NaN or Inf");
    sts_gmres_info inf{0, 0, 1, 0.0, 0, 0};
    sts_status status = STS_OK;
    bool written = false;       // x_pub holds the result, and the error flag has been read
    if (bnorm == 0.0) {
        STS_CK(cudaMemsetAsync(K.xb, 0, n * sizeof(double), h->stream));
    } else {
        std::vector<double> H((size_t)(m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
        int its = 0;
        // r = b - A x and its squared norm
        auto residual = [&](double *norm, const CycleEnd &end) -> sts_status {
            STS_TRY(opA64(h, dir, K.xb, K.w));
            k_residual<<<orth_blocks(n, 0), kRedThreads, 0, h->stream>>>(K.r, K.bb, K.w, n, K.partial, norm, K.ticket,
                                                                         end);
            STS_LAUNCHED();
            return STS_OK;
        };
        double beta_known = -1.0;       // the residual's norm where the last cycle has brought it along
        for (;;) {
            NvtxRange nvtx_cycle("gmres cycle");
            // true residual r = b - A x (r = b exactly for the zero guess)
            double beta = bnorm;
            const double *r = K.r;
            if (zero_guess) {
                r = K.bb;
                zero_guess = false;
            } else if (beta_known >= 0.0 || std::isnan(beta_known)) {
                beta = beta_known;
                beta_known = -1.0;
            } else {
                STS_TRY(residual(K.red, CycleEnd{}));
                ++inf.matvecs;
                STS_CK(cudaMemcpyAsync(hp, K.red, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
                STS_CK(cudaStreamSynchronize(h->stream));
                beta = std::sqrt(hp[0]);
            }
            if (!std::isfinite(beta)) {
                status = set_error(STS_ERR_NUMERIC, "gmres: residual norm is NaN or Inf");
                break;
            }
            inf.true_rel_residual = beta / bnorm;
            if (beta / bnorm <= rtol) { inf.converged = 1; break; }
            if (its >= max_iters) { inf.converged = 0; break; }
            double stop_abs = mixed ? std::max(rtol * bnorm, inner * beta) : rtol * bnorm;
            double g0 = beta, hscale = 1.0 / bnorm;
            if (left) {
                // z = M r; the cycle works on the preconditioned residual
                STS_TRY(opM64(h, dir, r, K.tmp));
                ++inf.applies;
                STS_TRY(R.norm2(K.tmp, K.red));
                STS_CK(cudaMemcpyAsync(hp, K.red, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
                STS_CK(cudaStreamSynchronize(h->stream));
                g0 = std::sqrt(hp[0]);
                if (!std::isfinite(g0) || g0 == 0.0) {
                    status = set_error(STS_ERR_NUMERIC, "gmres: preconditioned residual norm is %g", g0);
                    break;
                }
                stop_abs = g0 * (rtol * bnorm / beta);
                hscale = beta / (g0 * bnorm);
            }
            k_scale<<<nb, 256, 0, h->stream>>>(K.V, left ? K.tmp : r, 1.0 / g0, n);
            STS_LAUNCHED();
            std::fill(g.begin(), g.end(), 0.0);
            g[0] = g0;
            int k = 0;
            if (use_graph) {
                // the whole cycle on the device, then x, its residual and (for device vectors, if
                // the solve ends here with a result: the caller's x stays as it was after a
                // failure) the result, so that one synchronisation ends a cycle whether it is the
                // last or not (it took four; one-cycle solves on 16 x 16 cells, N = 10
                // 338 -> 290 us, with the shorter rotations)
                NvtxRange nvtx_graph("gmres cycle graph");
                STS_TRY(cycle_graph(h, m, dir, pre));
                double *pp = K.g_pinned, *pg = pp + 8, *ph = pg + (K.m + 1);
                const int *ps = reinterpret_cast<const int *>(pp + 4), *pe = reinterpret_cast<const int *>(pp + 6);
                const int *pd = reinterpret_cast<const int *>(pp + 7);
                pp[0] = stop_abs;
                pp[1] = hscale;
                pp[2] = 0.0;
                pp[3] = (double)std::min(m, max_iters - its);
                for (int i = 0; i <= m; ++i) pg[i] = g[i];
                STS_CK(cudaMemcpyAsync(K.gbuf, pp, sizeof(double) * (8 + m + 1), cudaMemcpyHostToDevice, h->stream));
                STS_CK(cudaGraphLaunch(K.gexec[dir][pre ? 1 : 0], h->stream));
                k_cycle_y<<<1, kTile, 0, h->stream>>>(K.gH, K.gg, m, K.gstate, K.gy);
                STS_LAUNCHED();
                k_axpy_multi<double><<<nb, 256, 0, h->stream>>>(K.xb, K.Z, n, K.gy, 0, K.gstate);
                STS_LAUNCHED();
                STS_TRY(residual(K.grn, CycleEnd{h->d_err, K.gstate, bnorm, rtol, max_iters - its, K.gerr, K.gdone}));
                if (!d.vectors_on_host) STS_TRY(from_internal64(h, K.xb, x_pub, K.gdone));
                STS_CK(cudaMemcpyAsync(pp, K.gbuf, sizeof(double) * (8 + (K.m + 1) + K.m), cudaMemcpyDeviceToHost,
                                       h->stream));
                STS_CK(cudaStreamSynchronize(h->stream));
                k = ps[0];
                if (ps[1] == 2) {
                    status = set_error(STS_ERR_NUMERIC, "gmres: NaN or Inf in the Arnoldi process");
                    break;
                }
                for (int i = 0; i < k; ++i)
                    if (d.history && its + i < max_iters) d.history[its + i] = ph[i];
                its += k;
                inf.matvecs += k + 1;       // the steps' and the residual's
                if (pre) inf.applies += k;
                ++inf.restarts;
                written = !d.vectors_on_host && *pd && *pe == 0;
                beta_known = std::sqrt(pp[5]);
                continue;
            }
            for (int j = 0; j < m; ++j) {
                NvtxRange nvtx_step("gmres arnoldi step");
                double *vj = K.V + (size_t)j * n;
                // z_j = M v_j, w = A z_j (left: w = M (A v_j))
                if (left) {
                    STS_TRY(opA64(h, dir, vj, K.tmp));
                    STS_TRY(opM64(h, dir, K.tmp, K.w));
                    ++inf.matvecs;
                    ++inf.applies;
                } else if (!mixed) {
                    double *zj = K.Z + (size_t)j * n;
                    if (pre) STS_TRY(opM64(h, dir, vj, zj));
                    else STS_CK(cudaMemcpyAsync(zj, vj, n * sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
                    STS_TRY(opA64(h, dir, zj, K.w));
                    ++inf.matvecs;
                    if (pre) ++inf.applies;
                } else {
                    float *zj = K.Z32 + (size_t)j * n;
                    k_convert<float, double><<<nb, 256, 0, h->stream>>>(pre ? K.t32a : zj, vj, n);
                    STS_LAUNCHED();
                    if (pre) STS_TRY(smw_apply32(h, dir, internal_vec(h, K.t32a), internal_vec(h, zj)));
                    STS_TRY(mv_apply32(h, dir, internal_vec(h, zj), internal_vec(h, K.t32b), h->c32));
                    k_convert<double, float><<<nb, 256, 0, h->stream>>>(K.w, K.t32b, n);
                    STS_LAUNCHED();
                }
                // CGS2: h1 = V^T w (+ w.w), w -= V h1; h2 = V^T w, w -= V h2, ||w||^2
                double *h1 = K.red, *h2 = K.red + (m + 2), *nr = K.red + 2 * (m + 2);
                STS_TRY(R.dots(K.V, j + 1, K.w, 1, h1));
                STS_TRY(R.update_dots(K.w, K.V, j + 1, h1, h2));
                STS_TRY(R.update(K.w, K.V, j + 1, h2, 1, nr));
                STS_CK(cudaMemcpyAsync(hp, K.red, sizeof(double) * 3 * (m + 2), cudaMemcpyDeviceToHost, h->stream));
                STS_CK(cudaStreamSynchronize(h->stream));
                const double *H1 = hp, *H2 = hp + (m + 2);
                const double w0 = std::sqrt(H1[j + 1]);
                double hn = std::sqrt(hp[2 * (m + 2)]);
                bool bad = !std::isfinite(w0) || !std::isfinite(hn);
                for (int i = 0; i <= j; ++i) {
                    H[(size_t)i * m + j] = H1[i] + H2[i];
                    bad = bad || !std::isfinite(H[(size_t)i * m + j]);
                }
                if (bad) { status = set_error(STS_ERR_NUMERIC, "gmres: NaN or Inf in the Arnoldi process"); break; }
                H[(size_t)(j + 1) * m + j] = hn;
                for (int i = 0; i < j; ++i) {
                    const double a = H[(size_t)i * m + j], c = H[(size_t)(i + 1) * m + j];
                    H[(size_t)i * m + j] = cs[i] * a + sn[i] * c;
                    H[(size_t)(i + 1) * m + j] = -sn[i] * a + cs[i] * c;
                }
                const double hjj = H[(size_t)j * m + j];
                const double den = std::hypot(hjj, hn);
                cs[j] = hjj / den;
                sn[j] = hn / den;
                H[(size_t)j * m + j] = den;
                H[(size_t)(j + 1) * m + j] = 0.0;
                g[j + 1] = -sn[j] * g[j];
                g[j] = cs[j] * g[j];
                ++its;
                k = j + 1;
                if (d.history && its <= max_iters) d.history[its - 1] = std::fabs(g[j + 1]) * hscale;
                const bool happy = hn <= 1e-14 * w0;
                if (happy || std::fabs(g[j + 1]) <= stop_abs || its >= max_iters) break;
                k_scale<<<nb, 256, 0, h->stream>>>(K.V + (size_t)(j + 1) * n, K.w, 1.0 / hn, n);
                STS_LAUNCHED();
            }
            if (status != STS_OK) break;
            for (int i = k - 1; i >= 0; --i) {
                double s = g[i];
                for (int l = i + 1; l < k; ++l) s -= H[(size_t)i * m + l] * y[l];
                y[i] = s / H[(size_t)i * m + i];
            }
            std::copy(y.begin(), y.begin() + k, hp);
            STS_CK(cudaMemcpyAsync(K.red, hp, sizeof(double) * k, cudaMemcpyHostToDevice, h->stream));
            if (!mixed) k_axpy_multi<double><<<nb, 256, 0, h->stream>>>(K.xb, left ? K.V : K.Z, n, K.red, k, nullptr);
            else k_axpy_multi<float><<<nb, 256, 0, h->stream>>>(K.xb, K.Z32, n, K.red, k, nullptr);
            STS_LAUNCHED();
            ++inf.restarts;
        }
        inf.iterations = its;
    }
    *checked = written && status == STS_OK;
    if (!written && (status == STS_OK || status == STS_ERR_NOT_CONVERGED)) {
        if (d.vectors_on_host) {
            STS_TRY(from_internal64(h, K.xb, h->vout));
            STS_CK(cudaMemcpyAsync(x_pub, h->vout, vbytes, cudaMemcpyDeviceToHost, h->stream));
        } else {
            STS_TRY(from_internal64(h, K.xb, x_pub));
        }
        STS_CK(cudaStreamSynchronize(h->stream));
    }
    if (info) *info = inf;
    if (status != STS_OK) return status;
    if (!inf.converged)
        return set_error(STS_ERR_NOT_CONVERGED, "gmres: %d iterations, true relative residual %.3e > rtol %.3e",
                         inf.iterations, inf.true_rel_residual, rtol);
    return STS_OK;
}

}  // namespace sts
