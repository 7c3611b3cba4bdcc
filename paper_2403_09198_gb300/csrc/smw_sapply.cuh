// smw_sapply.cuh -- the structured block-Jacobi apply (see kernels_smw.cu) and its launch,
// instantiated for FP64 in kernels_smw.cu and for FP32 in kernels_smw32.cu.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "ring.cuh"
#include "smw_stream.cuh"
#include "sts_internal.h"

namespace sts {
namespace {

// ---------------------------------------------------------------------------
// Structured apply for the paper's pattern family (level band of half-width W
// plus NF = 3 dense flow rows / columns).  Its LU has no fill:
//   L: level row i holds the band (i, i-W..i-1); flow rows are dense.
//   U: level row i holds (i, i..i+W) and the flow columns; the flow block is
//      upper triangular.
// Both directions are "forward unit-lower arrow-band sweep, then backward
// scaled unit-upper arrow-band sweep" over a per-direction coefficient stream:
//   forward level row i:  W band coefficients (oldest first), then the NF
//                          coefficients of the flow rows in column i, which
//                          feed NF independent accumulators;
//   forward flow rows:    the 3 coefficients among the flow unknowns;
//   backward flow rows:   per row its pivot inverse and coefficients, then the
//                          RMAX dot-vector entries of t = V^T x0 for that unknown
//                          (one group, or one group per row where the three
//                          rows are wider than a chunk);
//   backward level row i: pivot inverse, NF flow coefficients, W band
//                          coefficients (farthest first), RMAX dot-vector entries;
//   tail:                 W[a][q] for the correction x = x0 - W C^-1 t, with
//                          C^-1 read per cell (FP64, r x r registers); in the
//                          instances that fold (sap_fold) the capacitance solve
//                          is folded into the tail instead: (W C^-1)[q][a],
//                          formed in FP64 when the stream is packed, and
//                          x = x0 - (W C^-1) t needs neither C^-1 nor its registers.
// A cell with fewer than RMAX pairs has zero dot and tail entries.
// The band recurrences keep their last W values in registers, so the only
// dependency chain is one FMA per row.
//
// Stream layout.  Rows are packed in groups of whole 16-byte vectors (VEC =
// 16 / sizeof(T) positions): a group is a run of consecutive rows of one
// section whose width is a multiple of VEC and at least 16 positions (rows
// past the end of the section are zero; see sap_group_rows), or one single row
// padded with zeros.  Groups never
// straddle a chunk of K positions (8 KB), and each tile's stream is padded to
// whole chunks, so one tile's stream is Lt contiguous positions stored as
// [tile][position / VEC][lane][VEC]: a chunk is one bulk copy and a lane reads
// VEC positions with one 16-byte shared-memory load.
template <typename T, bool BARE>
struct SApplyArgs {
    const T *st;            // [n_tiles][Lt / VEC][32][VEC]
    const double *Cinv;     // [r][r][ncp] (instances that do not fold only)
    std::conditional_t<BARE, Bare<T>, Vec<T>> x, y;     // internal layout where the working vector lives in y
    int *err;               // set when a bounded wait gave up
    int Lt, b, N, r, ncp, trans, n_tiles;
    int pre;                // the stream and C^-1 may be read before the grid-dependency wait
    int evict_first;        // the stream of one call is larger than L2
    int bulk;               // x starts on a 16-byte boundary
};

constexpr int kApWarps = 4;              // consumer warps per block of the structured apply (one per sub-partition)
constexpr int kSApStages = 5;            // ring stages of the structured apply (three chunks in flight)
constexpr int kSApChunkBytes = 8192;     // bytes per stage (one bulk copy)

// Pair slots RMAX of the structured apply instance for r pairs per diagonal
// block and band half-width w: 2, 4, or nine (one source pair plus two per face
// of a 2D cell, Section 4.3).  Ten for w = 4, whose backward rows are then 18
// positions wide instead of 17 (two 17-wide rows would not fit one chunk), and
// for w = 2, whose 16-wide rows then form one-row groups: the extra zero slot
// costs two FMAs per row but frees the registers a second row would hold.
// 0: more pairs than any structured instance holds.
__host__ __device__ constexpr int sap_rmax_big(int w) { return w == 2 || w == 4 ? 10 : 9; }
__host__ __device__ constexpr int sap_rmax(int r, int w) {
    return r <= 2 ? 2 : r <= 4 ? 4 : r <= sap_rmax_big(w) ? sap_rmax_big(w) : 0;
}
// Whether the instance folds C^-1 into its tail vectors: always above four
// pairs, and wherever the r x r FP64 registers of the unfolded form would spill
// (more than two pairs, or band half-width 1 or 4, by the ptxas register
// reports).  Where both fit, the unfolded form measured faster (band 2, two pairs).
__host__ __device__ constexpr bool sap_fold(int rmax, int w) { return rmax > 2 || w == 1 || w == 4; }

// Rows per group: the fewest rows of whole vectors, repeated up to at least 16
// positions (the per-group bookkeeping is then spread over 16 or more FMAs);
// forward groups hold at most NF + 1 rows, so that their working-vector reads
// past the last level row stay inside the block.
__host__ __device__ constexpr int sap_group_rows(int width, int vec) {
    return sap_rows(width, vec) * ((16 + sap_rows(width, vec) * width - 1) / (sap_rows(width, vec) * width));
}
__host__ __device__ constexpr int sap_fwd_rows(int width, int vec, int nf) {
    return sap_group_rows(width, vec) <= nf + 1 ? sap_group_rows(width, vec)
                                                : (sap_rows(width, vec) > nf + 1 ? sap_rows(width, vec) : nf + 1 -
                                                   (nf + 1) % sap_rows(width, vec));
}
// shared memory of one consumer warp: stages, 128 bytes of mbarriers (full,
// empty, the first tile's x), working vector [b][32]
constexpr int kSApBarBytes = 128;
static_assert((2 * kSApStages + 1) * 8 <= kSApBarBytes, "full, empty and x barriers fit");
__host__ __device__ inline size_t sap_warp_bytes(int b, int elem) {
    const size_t raw = (size_t)kSApStages * kSApChunkBytes + kSApBarBytes + (size_t)b * kTile * elem;
    return (raw + 127) / 128 * 128;
}


// Consumer warp w of block k takes tiles w * gridDim.x + k, + nc * gridDim.x,
// ... so that tiles are dealt to SMs round-robin and no sub-partition runs two
// tiles while another idles; the block's last warp is the producer, whose
// lane 0 issues every bulk copy of the block's rings.  A consumer's tiles form
// one continuous stream for its ring, so the next tile's first chunks arrive
// during the current tail; the next tile's x is copied into the working vector
// one group of rows at a time as the tail frees it.  Within a section the next group
// (coefficients and working-vector entries) is loaded into registers before
// the current one is used, so the shared-memory latency overlaps the FMAs.
//
// GW: the working vector lives in y instead of shared memory (the forward
// sweep reads x from global memory and writes its rows into y; the backward
// sweep and the tail read and rewrite them in place, loaded a group ahead so
// the L2 latency overlaps the FMAs).  Chosen where b rows per warp would leave
// fewer than four consumers per SM (b > 65 in FP64, b > 131 in FP32): the ring
// alone then fits four.  Plain (coherent) loads throughout, since the kernel
// rewrites the rows it reads and x may be y.  wl is then not used.
//
// INT: the vectors are in the internal layout (GW always is), whose addresses the FP32
// kernel, bound by its instructions, cannot spare (11.2 against 12.8 us through strides on
// 128 x 128 cells, N = 60).  FP32 and GW instances on it do without the strides as arguments,
// too: unused, they still cost 2-6% (96 x 96 cells: N = 30 FP32 7.07 -> 7.33 us, N = 100
// FP64 in y 90.8 -> 96.2); FP64 in shared memory is as fast or faster beside them (W = 2,
// two pairs 44.5 against 45.1 us, 248 registers against 255).
__host__ __device__ constexpr bool sap_bare(int elem, bool gw, bool in) { return gw || (in && elem == 4); }
template <typename T, int W, int RMAX, bool GW, bool INT>
__global__ void __launch_bounds__((kApWarps + 1) * 32) k_smw_sapply(SApplyArgs<T, sap_bare((int)sizeof(T), GW, INT)> a) {
    static_assert(INT || !GW, "the working vector in y needs the internal layout");
    constexpr int NF = kStructNF, VEC = 16 / (int)sizeof(T);
    constexpr int K = kSApChunkBytes / (kTile * (int)sizeof(T));
    constexpr int FW = W + NF, UF = sap_fwd_rows(FW, VEC, NF), GF = UF * FW;
    constexpr int GFF = sap_round(3, VEC), GBF = sap_round(6 + 3 * RMAX, VEC);
    // the three backward flow rows form one group, or one group each where that is wider than a chunk
    constexpr bool FSPLIT = GBF > K;
    constexpr int G2 = sap_round(1 + RMAX, VEC), G1 = sap_round(2 + RMAX, VEC), G0 = sap_round(3 + RMAX, VEC);
    constexpr int BW = 1 + NF + W + RMAX, UB = sap_group_rows(BW, VEC), GB = UB * BW;
    constexpr int UT = sap_group_rows(RMAX, VEC), GT = UT * RMAX;
    static_assert(GF % VEC == 0 && GB % VEC == 0 && GT % VEC == 0, "groups are whole vectors");
    static_assert(GF <= K && G0 <= K && GB <= K && GT <= K, "groups fit a chunk");
    constexpr bool FOLD = sap_fold(RMAX, W);
    static_assert(UF <= NF + 1, "forward rows read past N stay inside the block");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nc = (int)(blockDim.x >> 5) - 1;                  // consumer warps
    const size_t wbytes = sap_warp_bytes(GW ? 0 : a.b, (int)sizeof(T));
    const int nw = nc * gridDim.x;
    const int nch = a.Lt / K;
    if (threadIdx.x == 0) {
        for (int w = 0; w < nc; ++w) {
            const uint32_t full = smem_addr(smem_raw + (size_t)w * wbytes + (size_t)kSApStages * kSApChunkBytes);
#pragma unroll
            for (int st = 0; st < kSApStages; ++st) {
                mbar_init(full + 8u * st, 1);
                mbar_init(full + 8u * (kSApStages + st), 32);
            }
            mbar_init(full + 8u * (2 * kSApStages), 1);     // the first tile's x
        }
        mbar_init_fence();
    }
    __syncthreads();
    if (warp == nc) {
        // ---- producer
        if (lane == 0) {
            // the L2 policy of the copies is a template argument: a test in the
            // issue loop slowed the FP32 apply (about 1 us at 128 x 128 cells)
            auto produce = [&](auto evict_first) {
                RingProducer<T, K, kSApStages, kApWarps, decltype(evict_first)::value> pr;
                pr.src = a.st;
                pr.seg_elems = (size_t)a.Lt * kTile;
                pr.nc = nc;
                pr.seg_step = nw;
                pr.nch = nch;
                pr.maxc = 0;
#pragma unroll
                for (int w = 0; w < kApWarps; ++w) {
                    unsigned char *reg = smem_raw + (size_t)min(w, nc - 1) * wbytes;
                    pr.stg[w] = reinterpret_cast<T *>(reg);
                    pr.full[w] = smem_addr(reg + (size_t)kSApStages * kSApChunkBytes);
                    pr.empty[w] = pr.full[w] + 8u * kSApStages;
                    pr.seg0[w] = w * gridDim.x + blockIdx.x;
                    pr.nseg[w] = (w < nc && pr.seg0[w] < a.n_tiles) ? (a.n_tiles - 1 - pr.seg0[w]) / nw + 1 : 0;
                    pr.issued[w] = 0;
                    pr.pk[w] = 0;
                    pr.pl[w] = 0;
                    pr.maxc = max(pr.maxc, pr.nseg[w] * nch);
                }
                bool ok = a.pre ? pr.issue_upto(kSApStages) : true;
                pdl_wait();
                pdl_trigger();
                if (ok) ok = pr.run();
                if (!ok) atomicExch(a.err, 1);
                pr.drain();
            };
            if (a.evict_first) produce(std::true_type{});
            else produce(std::false_type{});
        } else {
            pdl_wait();
            pdl_trigger();
        }
        return;
    }
    // ---- consumers
    const int gw = warp * gridDim.x + blockIdx.x;
    if (gw >= a.n_tiles) return;
    const int my = (a.n_tiles - 1 - gw) / nw + 1;
    const size_t P = a.ncp;
    const int N = a.N, b = a.b, r = a.r;
    unsigned char *mine = smem_raw + (size_t)warp * wbytes;
    const uint32_t full = smem_addr(mine + (size_t)kSApStages * kSApChunkBytes);
    T *wl = reinterpret_cast<T *>(mine + (size_t)kSApStages * kSApChunkBytes + kSApBarBytes) + lane;  // row i at wl[i * 32]
    RingConsumer<T, K, kSApStages> R;
    R.start(reinterpret_cast<T *>(mine), full, full + 8u * kSApStages, lane);
    pdl_wait();
    pdl_trigger();
    // The first tile's x.  FP64: one bulk copy per row (rows lane, lane + 32,
    // ...), completed on the warp's x barrier; per-lane cp.async of the b rows
    // measured slower (their issue stalls once the SM's outstanding loads
    // fill).  FP32 (128-byte rows): per-lane cp.async measured faster (11.5
    // against 12.9 us on 128 x 128 cells, N = 60).
    constexpr bool XBULK = !GW && sizeof(T) == 8;
    const uint32_t xbar = full + 8u * (2 * kSApStages);
    const bool bulk = XBULK && INT && a.bulk;
    if (bulk) {
        if (lane == 0) mbar_expect_tx(xbar, (uint32_t)((size_t)b * kTile * sizeof(T)));
        __syncwarp();
        for (int i = lane; i < b; i += kTile)
            bulk_copy_g2s(smem_addr(wl - lane + (size_t)i * kTile), a.x.p + (size_t)i * P + (size_t)gw * kTile,
                          (uint32_t)(kTile * sizeof(T)), xbar);
    } else if constexpr (!GW) {
        const T *x0 = a.x.template cell<INT>(gw * kTile + lane);
        size_t xq = P;
        if constexpr (!INT) xq = (size_t)a.x.sq;
        for (int i = 0; i < b; ++i) cp_async_elem(wl + i * kTile, x0 + (size_t)i * xq);
        cp_async_commit();
    }
    for (int k = 0; k < my; ++k) {
        const int cell = (gw + k * nw) * kTile + lane;
        // row j of the working vector, and row j of this tile's x
        auto wv = [&](int j) -> T & {
            if constexpr (GW) return a.y.p[(size_t)j * P + cell];
            else return wl[j * kTile];
        };
        auto xin = [&](int j) -> T {
            if constexpr (GW) return a.x.p[(size_t)j * P + cell];
            else return wl[j * kTile];
        };
        double cz[FOLD ? 1 : RMAX * RMAX];      // C^-1 (transposed for A^T), zero outside r x r
        if constexpr (!FOLD) {
#pragma unroll
            for (int i = 0; i < RMAX; ++i)
#pragma unroll
                for (int l = 0; l < RMAX; ++l)
                    cz[i * RMAX + l] =
                        (i < r && l < r) ? __ldg(a.Cinv + (a.trans ? (size_t)l * r + i : (size_t)i * r + l) * P + cell)
                                         : 0.0;
        }
        if constexpr (!GW) {
            if (bulk && k == 0) {
                if (!mbar_wait_bounded(xbar, 0)) goto fail;
            } else {
                cp_async_wait<0>();             // copied in by the previous tile's tail (or, FP32, before it)
            }
            __syncwarp();
        }
        // ---- forward sweep over the level rows: row i = [W band, oldest first | NF flow]
        T win[W > 0 ? W : 1];
#pragma unroll
        for (int q = 0; q < W; ++q) win[q] = T(0);
        T accf[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) accf[f] = T(0);
        sap_section<T, GF, UF>(
            R, N, [&](int j) { return xin(min(j, b - 1)); },
            [&](const Group<T, GF> &g, T acc, int u, int) {
#pragma unroll
                for (int q = 0; q < W; ++q) acc = fma(-g[u * FW + q], win[q], acc);
#pragma unroll
                for (int f = 0; f < NF; ++f) accf[f] = fma(g[u * FW + W + f], acc, accf[f]);
#pragma unroll
                for (int q = 0; q + 1 < W; ++q) win[q] = win[q + 1];
                if (W > 0) win[W > 0 ? W - 1 : 0] = acc;
                return acc;
            },
            [&](int j, T v) { wv(j) = v; });
        // ---- forward flow rows: (N+1,N), (N+2,N), (N+2,N+1)
        T wf[NF];
        {
            Group<T, GFF> g;
            g.load(R.take(GFF));
            wf[0] = xin(N) - accf[0];
            wf[1] = fma(-g[0], wf[0], xin(N + 1) - accf[1]);
            wf[2] = fma(-g[2], wf[1], fma(-g[1], wf[0], xin(N + 2) - accf[2]));
        }
        // ---- backward flow rows, with t = V^T x0 accumulated on the way
        T t[RMAX];
#pragma unroll
        for (int q = 0; q < RMAX; ++q) t[q] = T(0);
        T xf[NF];
        {
            // rows [d2, V(N+2) | d1, u(N+1,N+2), V(N+1) | d0, u(N,N+1), u(N,N+2), V(N)], V padded to RMAX
            auto flow = [&](auto e2, auto e1, auto e0) {
                xf[2] = e2(0) * wf[2];
#pragma unroll
                for (int q = 0; q < RMAX; ++q) t[q] = fma(e2(1 + q), xf[2], t[q]);
                xf[1] = fma(-e1(1), xf[2], e1(0) * wf[1]);
#pragma unroll
                for (int q = 0; q < RMAX; ++q) t[q] = fma(e1(2 + q), xf[1], t[q]);
                xf[0] = fma(-e0(2), xf[2], fma(-e0(1), xf[1], e0(0) * wf[0]));
#pragma unroll
                for (int q = 0; q < RMAX; ++q) t[q] = fma(e0(3 + q), xf[0], t[q]);
            };
            if constexpr (FSPLIT) {
                Group<T, G2> g2;
                Group<T, G1> g1;
                Group<T, G0> g0;
                g2.load(R.take(G2));
                g1.load(R.take(G1));
                g0.load(R.take(G0));
                flow([&](int e) { return g2[e]; }, [&](int e) { return g1[e]; }, [&](int e) { return g0[e]; });
            } else {
                constexpr int o1 = 1 + RMAX, o0 = o1 + 2 + RMAX;
                Group<T, GBF> g;
                g.load(R.take(GBF));
                flow([&](int e) { return g[e]; }, [&](int e) { return g[o1 + e]; }, [&](int e) { return g[o0 + e]; });
            }
        }
        if (R.failed) goto fail;
        // ---- backward level rows i = N-1-j: [pivot inverse | NF flow | W band, farthest first | V (RMAX)]
        {
            T xw[W > 0 ? W : 1];
#pragma unroll
            for (int q = 0; q < W; ++q) xw[q] = T(0);
            sap_section<T, GB, UB>(
                R, N, [&](int j) { return wv(max(N - 1 - j, 0)); },
                [&](const Group<T, GB> &g, T wi, int u, int) {
                    T acc = g[u * BW] * wi;
#pragma unroll
                    for (int f = 0; f < NF; ++f) acc = fma(-g[u * BW + 1 + f], xf[f], acc);
#pragma unroll
                    for (int q = 0; q < W; ++q) acc = fma(-g[u * BW + 1 + NF + q], xw[W - 1 - q], acc);
#pragma unroll
                    for (int q = 0; q < RMAX; ++q) t[q] = fma(g[u * BW + 1 + NF + W + q], acc, t[q]);
#pragma unroll
                    for (int q = W - 1; q > 0; --q) xw[q] = xw[q - 1];
                    if (W > 0) xw[0] = acc;
                    return acc;
                },
                [&](int j, T v) { wv(N - 1 - j) = v; });
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) wv(N + f) = xf[f];
        // ---- z = C^-1 t in FP64, then x = x0 - W z (tail row q = W[0..RMAX)[q]);
        //      folded: z = t and tail row q = (W C^-1)[q][0..RMAX)
        {
            T z[RMAX];
#pragma unroll
            for (int i = 0; i < RMAX; ++i) {
                if constexpr (FOLD) {
                    z[i] = t[i];
                } else {
                    double sacc = 0.0;
#pragma unroll
                    for (int l = 0; l < RMAX; ++l) sacc = fma(cz[i * RMAX + l], (double)t[l], sacc);
                    z[i] = (T)sacc;
                }
            }
            const T *xn = a.x.p + (size_t)cell + (size_t)nw * kTile;
            T *y = a.y.p + cell;
            size_t sq = P;                  // of x and of y
            bool on = true;                 // padding lanes of a vector in place write nothing
            if constexpr (!INT) {
                xn = a.x.at(cell + nw * kTile);
                y = a.y.p + (size_t)cell * (size_t)a.y.sc;
                sq = (size_t)a.x.sq;
                on = cell < a.y.cells;
            }
            // the next tile's x is copied in one group of rows at a time, at
            // the group's last row (all its rows have been read by then): a
            // test of the runtime flag on every row measured about 25 cycles
            // a row even when never taken
            const bool more = k + 1 < my;
            sap_section<T, GT, UT>(
                R, b, [&](int j) { return wv(min(j, b - 1)); },
                [&](const Group<T, GT> &g, T val, int u, int j) {
#pragma unroll
                    for (int l = 0; l < RMAX; ++l) val = fma(-g[u * RMAX + l], z[l], val);
                    if constexpr (!GW) {
                        if (u == UT - 1 && more) {
#pragma unroll
                            for (int q = 0; q < UT; ++q)
                                cp_async_elem(wl + (j - q) * kTile, xn + (size_t)(j - q) * sq);
                        }
                    }
                    return val;
                },
                [&](int j, T v) { if (on) y[(size_t)j * sq] = v; });
            if constexpr (!GW) {
                if (more) {
                    for (int j = b / UT * UT; j < b; ++j) cp_async_elem(wl + j * kTile, xn + (size_t)j * sq);  // ragged last group
                    cp_async_commit();
                }
            }
        }
        if (R.failed) goto fail;
        R.end_segment();
    }
    return;
fail:
    // the producer waits (bounded) for every copy it issued before it exits;
    // this warp waits (bounded) for its own copies of the first tile's x
    if (lane == 0) atomicExch(a.err, 1);
    if (bulk) mbar_wait_bounded(xbar, 0);
    cp_async_wait<0>();
}

// The working vector moves to y where b rows per warp would leave fewer than kApWarps
// consumers per SM.
inline bool sap_in_y(int b, int elem) { return (size_t)(227 * 1024) / sap_warp_bytes(b, elem) < (size_t)kApWarps; }

template <typename T, int W, bool GW, bool INT>
void (*sap_kernel_of(int rmax))(SApplyArgs<T, sap_bare((int)sizeof(T), GW, INT)>) {
    return rmax == 2 ? k_smw_sapply<T, W, 2, GW, INT> : rmax == 4 ? k_smw_sapply<T, W, 4, GW, INT>
                                                                   : k_smw_sapply<T, W, sap_rmax_big(W), GW, INT>;
}
template <typename T, bool GW, bool INT>
auto sap_kernel(int w, int rmax) {
    return w == 0 ? sap_kernel_of<T, 0, GW, INT>(rmax) : w == 1 ? sap_kernel_of<T, 1, GW, INT>(rmax)
           : w == 2 ? sap_kernel_of<T, 2, GW, INT>(rmax) : w == 3 ? sap_kernel_of<T, 3, GW, INT>(rmax)
                                                                 : sap_kernel_of<T, 4, GW, INT>(rmax);
}

template <typename T>
sts_status smw_sapply_t(sts_jac_s *h, int dir, const T *st, const Vec<T> &x, const Vec<T> &z) {
    const SmwPlan &M = h->smw;
    SApplyArgs<T, false> a;
    a.st = st; a.Cinv = M.Cinv; a.x = x; a.y = z; a.err = h->d_err;
    a.Lt = M.s_lt[sizeof(T) == 8 ? 0 : 1]; a.b = h->b; a.N = h->b - kStructNF; a.r = h->r_diag; a.ncp = h->ncp;
    a.trans = dir; a.n_tiles = h->n_tiles;
    a.pre = h->streams_dirty ? 0 : 1;
    a.evict_first = (double)a.n_tiles * a.Lt * kTile * sizeof(T) > (double)h->l2_bytes ? 1 : 0;
    const bool gw = sap_in_y(h->b, (int)sizeof(T));
    const bool in = x.internal(h->ncp);
    a.bulk = reinterpret_cast<uintptr_t>(x.p) % 16 == 0 ? 1 : 0;
    const size_t per_warp = sap_warp_bytes(gw ? 0 : h->b, (int)sizeof(T));
    const int wpb = (int)std::min<size_t>(kApWarps, (size_t)(227 * 1024) / per_warp);
    if (wpb < 1)
        return set_error(STS_ERR_INVALID_ARG, "block size %d needs %zu bytes of shared memory per warp", h->b, per_warp);
    const size_t smem = (size_t)wpb * per_warp;
    const int rm = sap_rmax(h->r_diag, M.s_w);
    bool &attr = h->sap_attr[sizeof(T) == 8 ? 0 : 1][in ? 1 : 0];
    const int blocks = std::max(1, std::min(h->nsm, (h->n_tiles + wpb - 1) / wpb));
    auto launch = [&](auto kern, const auto &args) -> sts_status {
        if (!attr && smem > 48 * 1024) STS_CK(allow_all_smem(kern));
        attr = true;
        STS_CK(launch_pdl(kern, dim3(blocks), dim3((wpb + 1) * kTile), smem, h->stream, args));
        STS_LAUNCHED();
        return STS_OK;
    };
    const SApplyArgs<T, true> bare{a.st, a.Cinv, {a.x.p}, {a.y.p}, a.err, a.Lt, a.b, a.N, a.r, a.ncp, a.trans,
                                   a.n_tiles, a.pre, a.evict_first, a.bulk};
    if (gw) STS_TRY(launch(sap_kernel<T, true, true>(M.s_w, rm), bare));
    else if (!in) STS_TRY(launch(sap_kernel<T, false, false>(M.s_w, rm), a));
    else if constexpr (sap_bare((int)sizeof(T), false, true)) STS_TRY(launch(sap_kernel<T, false, true>(M.s_w, rm), bare));
    else STS_TRY(launch(sap_kernel<T, false, true>(M.s_w, rm), a));
    h->streams_dirty = false;
    return STS_OK;
}

}  // namespace
}  // namespace sts
