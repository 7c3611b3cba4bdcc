// kernels_values.cu -- public Jacobian values into the kernels' streams
// (sts_jac_create, sts_jac_update_values).
//
// The public arrays hold one block (or one pair vector) after another; the streams
// hold [tile][position][lane = cell].  A warp takes one unit, 32 consecutive
// entries of one block slot (or components of one pair slot) of the 32 cells of a
// tile: it reads each cell's run of 32 with one coalesced request, turns the 32 x 32
// piece round in shared memory and writes every entry's 32 cells with one coalesced
// request to each place that holds it: the pass-2 stream or the pass-1 stream, their
// FP32 copies, and the diagonal block's copy for the block-Jacobi setup.  Every
// value is thus read once per direction whatever the number of its destinations.
// Positions that no value reaches (padding, absent blocks and pairs) are zeroed when
// the streams are allocated and never written again.
//
// Bound by HBM.  Measured on 128 x 128 cells, N = 60: 9 / 2 pairs (1.46 GB read and
// written) 654 -> 287 us, 5.1 TB/s; 2 / 1 pairs, both directions, 790 -> 396 us.
// Before, one thread per stream position gathered its value from the public array,
// once for every destination.  The runs' loads have to be issued before the first
// value is used (490 us otherwise, the warps waiting on one load after another).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "sts_internal.h"

namespace sts {
namespace {

constexpr int kLoadWarps = 4;

struct LoadArgs {
    const double *S, *AX, *DV;      // values; axpy vectors (pass-2 stream) and dot vectors (pass-1 stream)
    const int *blk;                 // [n_tiles][n_slots][32]
    const long long *soff;
    const int *pbase;
    const int4 *unit;               // [n_units]: slot, pair within its block or -1, first entry, entries
    const int2 *dst;                // [n_units][32]: pass-2 position or -1, pass-1 position or -1
    double *main64, *dot64;
    float *main32, *dot32;
    double *Sd, *AXd, *DVd;         // diagonal-block copies [entry][ncp], or NULL
    long long tile_len, dlen;
    int n_units, n_slots, b, ncp;
};

// Position pos of this lane in the FP32 pass-1 stream [pos / 4][lane][4].
__device__ __forceinline__ size_t vec4_at(size_t pos, int lane) { return (pos & ~(size_t)3) * kTile + 4 * lane + (pos & 3); }

__global__ void __launch_bounds__(kLoadWarps * kTile) k_load_values(LoadArgs a) {
    __shared__ double sh[kLoadWarps][kTile][kTile + 1];
    const int lane = threadIdx.x & 31;
    double(*piece)[kTile + 1] = sh[threadIdx.x >> 5];
    const int per_tile = (a.n_units + kLoadWarps - 1) / kLoadWarps;
    const size_t tile = blockIdx.x / per_tile;
    const int u = (int)(blockIdx.x - tile * per_tile) * kLoadWarps + (threadIdx.x >> 5);
    if (u >= a.n_units) return;
    const int4 un = __ldg(a.unit + u);
    const int slot = un.x, local = un.y, e0 = un.z, cnt = un.w;
    const bool pair = local >= 0;
    const int k = __ldg(a.blk + (tile * a.n_slots + slot) * kTile + lane);
    long long base = -1;
    if (k >= 0) {
        if (!pair) base = __ldg(a.soff + k) + e0;
        else if (local < __ldg(a.pbase + k + 1) - __ldg(a.pbase + k)) base = (long long)(__ldg(a.pbase + k) + local) * a.b + e0;
    }
    const int2 to = __ldg(a.dst + (size_t)u * kTile + lane);
    const size_t cell = tile * kTile + lane;
    // bring 32 runs in and turn them round: piece[entry][cell]
    auto bring = [&](const double *__restrict__ src) {
        // half the runs at a time, every load issued before the first value is used
#pragma unroll
        for (int c0 = 0; c0 < kTile; c0 += kTile / 2) {
            double v[kTile / 2];
#pragma unroll
            for (int c = 0; c < kTile / 2; ++c) {
                const long long at = __shfl_sync(0xffffffffu, base, c0 + c);
                v[c] = 0.0;
                if (at >= 0 && lane < cnt) v[c] = __ldg(src + at + lane);     // runs share sectors: cached loads (294 against 301 us)
            }
#pragma unroll
            for (int c = 0; c < kTile / 2; ++c) piece[lane][c0 + c] = v[c];
        }
        __syncwarp();
    };
    const size_t m0 = tile * a.tile_len, d0 = tile * a.dlen;
    auto put_main = [&](int pos, double v) {
        a.main64[(m0 + pos) * kTile + lane] = v;
        if (a.main32) a.main32[(m0 + pos) * kTile + lane] = (float)v;
    };
    auto put_dot = [&](int pos, double v) {
        a.dot64[(d0 + pos) * kTile + lane] = v;
        if (a.dot32) a.dot32[d0 * kTile + vec4_at(pos, lane)] = (float)v;
    };
    const bool on = base >= 0;
    if (!pair) {
        bring(a.S);
        double *sd = slot == 0 ? a.Sd : nullptr;
        for (int e = 0; e < cnt; ++e) {
            const int mp = __shfl_sync(0xffffffffu, to.x, e), dp = __shfl_sync(0xffffffffu, to.y, e);
            if (!on) continue;
            const double v = piece[e][lane];
            if (mp >= 0) put_main(mp, v);
            if (dp >= 0) put_dot(dp, v);
            if (sd) sd[(size_t)(e0 + e) * a.ncp + cell] = v;
        }
        return;
    }
    const size_t pd = (size_t)local * a.b + e0;         // first component in the diagonal copies
    bring(a.AX);
    for (int e = 0; e < cnt; ++e) {
        const int mp = __shfl_sync(0xffffffffu, to.x, e);
        if (!on) continue;
        const double v = piece[e][lane];
        put_main(mp, v);
        if (slot == 0 && a.AXd) a.AXd[(pd + e) * a.ncp + cell] = v;
    }
    __syncwarp();
    bring(a.DV);
    for (int e = 0; e < cnt; ++e) {
        const int dp = __shfl_sync(0xffffffffu, to.y, e);
        if (!on) continue;
        const double v = piece[e][lane];
        put_dot(dp, v);
        if (slot == 0 && a.DVd) a.DVd[(pd + e) * a.ncp + cell] = v;
    }
}

}  // namespace

// Units and destinations of one direction from its stream positions: kind and
// argument of every pass-2 position (pk, pa) and pass-1 position (dk, da), src[k] the
// public entry of every entry of pattern k, nnz_d the entries of pattern 0.
sts_status values_plan(sts_jac_s *h, MvPlan &P, const std::vector<int> &pk, const std::vector<int> &pa,
                       const std::vector<int> &dk, const std::vector<int> &da, const std::vector<int> (&src)[2],
                       const std::vector<int> &pslot_slot, const std::vector<int> &pslot_local) {
    const int nnz[2] = {h->nnz_d, h->nnz_o}, b = h->b;
    // first unit of every slot's S entries, then of every pair slot's components
    std::vector<int4> unit;
    std::vector<int> s0(P.n_slots), p0(P.n_pslots);
    auto add = [&](int slot, int local, int n) {
        const int first = (int)unit.size();
        for (int e = 0; e < n; e += kTile) unit.push_back(make_int4(slot, local, e, std::min(kTile, n - e)));
        return first;
    };
    for (int s = 0; s < P.n_slots; ++s) s0[s] = add(s, -1, nnz[s ? 1 : 0]);
    for (int k = 0; k < P.n_pslots; ++k) p0[k] = add(pslot_slot[k], pslot_local[k], b);
    std::vector<int2> dst(unit.size() * kTile, make_int2(-1, -1));
    auto place = [&](int kind, int arg) -> int2 & {
        if (kind < 0) return dst[(size_t)p0[-1 - kind] * kTile + arg];
        const int kd = kind ? 1 : 0;
        return dst[(size_t)s0[kind] * kTile + src[kd][arg - (kd ? h->nnz_d : 0)]];
    };
    for (size_t p = 0; p < pk.size(); ++p)
        if (pk[p] != kPosZero) place(pk[p], pa[p]).x = (int)p;
    for (size_t p = 0; p < dk.size(); ++p)
        if (dk[p] != kPosZero) place(dk[p], da[p]).y = (int)p;
    P.n_units = (int)unit.size();
    STS_TRY(upload(h, &P.unit, unit));
    return upload(h, &P.unit_dst, dst);
}

sts_status values_load(sts_jac_s *h, int dir, const double *S, const double *U, const double *V) {
    const MvPlan &P = h->mv[dir];
    LoadArgs a;
    a.S = S;
    a.AX = dir == 0 ? U : V;
    a.DV = dir == 0 ? V : U;
    a.blk = P.blk;
    a.soff = h->d_soff;
    a.pbase = h->d_pbase;
    a.unit = P.unit;
    a.dst = P.unit_dst;
    a.main64 = P.main64;
    a.main32 = P.main32;
    a.dot64 = P.dotv64;
    a.dot32 = P.dotv32;
    // the block-Jacobi setup's copies come with the forward direction
    a.Sd = dir == 0 ? h->smw.Sd : nullptr;
    a.AXd = dir == 0 ? h->smw.Ud : nullptr;
    a.DVd = dir == 0 ? h->smw.Vd : nullptr;
    a.tile_len = P.tile_len;
    a.dlen = (long long)P.n_dtasks * P.Lp;
    a.n_units = P.n_units;
    a.n_slots = P.n_slots;
    a.b = h->b;
    a.ncp = h->ncp;
    const long long blocks = (long long)h->n_tiles * ((P.n_units + kLoadWarps - 1) / kLoadWarps);
    k_load_values<<<(unsigned)blocks, kLoadWarps * kTile, 0, h->stream>>>(a);
    STS_LAUNCHED();
    return STS_OK;
}

}  // namespace sts
