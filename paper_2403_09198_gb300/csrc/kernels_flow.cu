// kernels_flow.cu -- residual and r1-sparse Jacobian of a toy HLL-flux flow
// model (Section 2.1 model, Section 3.2 Eq. HLL_flux, Section 3.3 Eq.
// system_residual, Section 4.1 Eqs. r1_flux_left / r1_flux_right).
//
// k_flow_mix forms every cell's mixture scalars (lane = cell), k_flow_face_* the
// scalars of 8 cells and their 32 directed faces (lane = (cell, face)); k_flow_jac and
// k_flow_res then run one warp per cell, lanes over the species.
// Every face is evaluated from both of its cells (once per block row), which keeps
// the writes of a block row in one warp: no atomics, deterministic.
//
// A warp-wide FP64 instruction holds a sub-partition's pipe for 64 cycles whatever the
// number of lanes that need it, so nothing scalar is computed by a whole warp, and
// every entry that varies over the species is written as an affine form of q_c, r_c,
// cv_c and e0_c with coefficients formed once per face: about 72 FP64 operations per
// cell and species (10 per face for the four pair vectors, 5 per block for S).  A_n is
// linear in the normal, so the diagonal block's face sum sum_f (1/2 + a_f) A_{n_f}(q_i)
// is A_n(q_i) at the summed normal.
//
// Measured on 128 x 128 cells, N = 60 (band 2): Jacobian (571 MB written) 1326 us with the
// scalars formed by every warp and every entry on its own, now 24 + 29 + 238 us (scalars
// of cells, of faces, entries); residual 540 us, now 26 + 12 + 47.  The entries keep the
// FP64 pipe 63% busy (134 of the 238 us are pipe time); more warps per SM or four faces
// at once without branches between them left the time as it was.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>
#include <vector>

#include "ring.cuh"
#include "sts_internal.h"

namespace sts {
namespace {

constexpr int kMixCells = 32;     // cells per block of k_flow_mix
constexpr int kFlowCells = 8;     // cells per warp of k_flow_face (8 x 4 faces) and per block of the kernels after it

// Per-cell scalars, component-major: M[field * nc + cell].
enum { mRho, mR, mC, mU, mV, mT, mKe, mP, mE, mA, mG0, mG1, mG2, mGT, mKap, mSb, kMixFields };

struct FlowDev {
    int Lx, nc, N, b, w, nnz_d, nnz_o;
    const double *r, *cv, *e0, *beta, *ws, *K;
    const double *dtK;      // dt K, plus 1 on the diagonal
    double A, theta, dt;
    const int *bptr, *bidx, *pip;
    const long long *soff;
    const int *d_ptr;       // row starts of the diagonal pattern (the neighbour pattern's are 4p, then 4N + b (p-N))
    const short2 *d_pq;     // (row, column) of the diagonal pattern's level-row entries
    double *mix;            // [2][kMixFields][nc]: scalars of Q, then of Qn
    double *face;           // [blocks of 8 cells][kFaceFields][32 faces]: coefficients of the faces
    double *cell;           // [blocks of 8 cells][kCellFields][8 cells]: of the diagonal blocks
};

struct Mix {
    double rho, R, C, u, v, T, ke, p, e, a;      // e: rho e_tot
};

__device__ __forceinline__ Mix mix_of(const double *M, int nc, int i) {
    Mix m;
    m.rho = M[mRho * (size_t)nc + i];
    m.R = M[mR * (size_t)nc + i];
    m.C = M[mC * (size_t)nc + i];
    m.u = M[mU * (size_t)nc + i];
    m.v = M[mV * (size_t)nc + i];
    m.T = M[mT * (size_t)nc + i];
    m.ke = M[mKe * (size_t)nc + i];
    m.p = M[mP * (size_t)nc + i];
    m.e = M[mE * (size_t)nc + i];
    m.a = M[mA * (size_t)nc + i];
    return m;
}

// Species sums and scalars of the states Q (blockIdx.y = 0) and Qn (1), one lane per
// cell: the 32 rows are staged in shared memory with an odd stride, each of four
// warps adds every fourth species in four interleaved sums.  A warp-wide sum over
// species, one cell at a time, costs 28 FP64 instructions a state against 5 N / 32,
// and the Jacobian needed it at the cell and at each of its neighbours.
// da/dq_c = G0 + G1 cv_c + G2 r_c for a species (from a^2 = T g, g = (C + R) R / (rho C),
// with R - g rho = -R^2 / C), GT for T, 0 for the velocities.
template <bool EARLY>
__global__ void __launch_bounds__(128) k_flow_mix(FlowDev F, const double *Q, const double *Qn) {
    extern __shared__ double rows[];             // [32][b | 1], species constants [N][4], partial sums [4][5][32]
    const int b = F.b, N = F.N, st = b | 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c0 = blockIdx.x * kMixCells, n = min(kMixCells, F.nc - c0);
    if (EARLY) {
        pdl_wait();
        pdl_trigger();
    }
    const double *src = (blockIdx.y ? Qn : Q) + (size_t)c0 * b;
    double *cst = rows + 32 * st;
    double(*part)[5][32] = reinterpret_cast<double(*)[5][32]>(cst + 4 * N);
    for (int k = threadIdx.x; k < N; k += 128) {
        cst[4 * k] = __ldg(F.r + k);
        cst[4 * k + 1] = __ldg(F.cv + k);
        cst[4 * k + 2] = __ldg(F.e0 + k);
        cst[4 * k + 3] = __ldg(F.beta + k);
    }
#pragma unroll 4
    for (int e = threadIdx.x; e < n * b; e += 128) {
        const int c = e / b;
        rows[c * st + e - c * b] = __ldg(src + e);
    }
    __syncthreads();
    const double *q = rows + min(lane, n - 1) * st;
    double s[4][5] = {};
    // Qn gives the conserved variables only: its sums of r and beta are left out
    auto sums = [&](auto all) {
        for (int k = warp; k < N; k += 16) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int kk = k + 4 * h;
                if (kk >= N) break;
                const double x = q[kk];
                s[h][0] += x;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (decltype(all)::value || j == 1 || j == 2) s[h][j + 1] = fma(x, cst[4 * kk + j], s[h][j + 1]);
            }
        }
    };
    if (blockIdx.y) sums(std::false_type{});
    else sums(std::true_type{});
#pragma unroll
    for (int j = 0; j < 5; ++j) part[warp][j][lane] = (s[0][j] + s[1][j]) + (s[2][j] + s[3][j]);
    __syncthreads();
    if (lane >= n) return;
    auto total = [&](int j) { return (part[0][j][lane] + part[1][j][lane]) + (part[2][j][lane] + part[3][j][lane]); };
    const double T = q[N + 2];
    double *M = F.mix + (size_t)blockIdx.y * kMixFields * F.nc + c0 + lane;
    const size_t P = F.nc;
    // the scalars' dependent chains on a warp each
    if (warp == 0 && blockIdx.y == 0) {
        const double rho = total(0), R = total(1), C = total(2);
        const double g = (C + R) * R / (rho * C), a = sqrt(g * T);
        M[mA * P] = a;
        const double cga = T / (2.0 * a * rho * C);
        M[mG0 * P] = -cga * ((C + R) * R / rho);
        M[mG1 * P] = -cga * (R * R / C);
        M[mG2 * P] = cga * (2.0 * R + C);
        M[mGT * P] = a / (2.0 * T);
    } else if (warp == 1) {
        const double rho = total(0), R = total(1), C = total(2), u = q[N], v = q[N + 1];
        const double ke = 0.5 * (u * u + v * v);
        M[mRho * P] = rho;
        M[mR * P] = R;
        M[mC * P] = C;
        M[mU * P] = u;
        M[mV * P] = v;
        M[mT * P] = T;
        M[mKe * P] = ke;
        M[mP * P] = R * T;
        M[mE * P] = total(3) + C * T + rho * ke;
    } else if (warp == 2 && blockIdx.y == 0) {
        M[mKap * P] = F.A * exp(-F.theta / T);
        M[mSb * P] = total(4);
    }
}

struct Face {
    double nx, ny, sL, sR, inv_den;
    int iL, iR;
};

// HLL bounds of the face from cell L to cell R: the extreme of 0, L's and R's
// wave speed, ties to the first; iL, iR name the one taken
__device__ __forceinline__ Face face_of(const Mix &mL, const Mix &mR, double nx, double ny) {
    Face f;
    f.nx = nx;
    f.ny = ny;
    const double unL = nx * mL.u + ny * mL.v, unR = nx * mR.u + ny * mR.v;
    f.sL = 0.0;
    f.iL = 0;
    if (unL - mL.a < f.sL) { f.sL = unL - mL.a; f.iL = 1; }
    if (unR - mR.a < f.sL) { f.sL = unR - mR.a; f.iL = 2; }
    f.sR = 0.0;
    f.iR = 0;
    if (unL + mL.a > f.sR) { f.sR = unL + mL.a; f.iR = 1; }
    if (unR + mR.a > f.sR) { f.sR = unR + mR.a; f.iR = 2; }
    f.inv_den = 1.0 / (f.sR - f.sL);
    return f;
}

__device__ __forceinline__ void normal_of(int Lx, int i, int j, double &nx, double &ny) {
    const int d = j - i;
    nx = d == 1 ? 1.0 : d == -1 ? -1.0 : 0.0;
    ny = d == Lx ? 1.0 : d == -Lx ? -1.0 : 0.0;
    if (Lx == 1) {      // a one-column grid: every neighbour is vertical
        nx = 0.0;
        ny = d > 0 ? 1.0 : -1.0;
    }
}

// Lane = (cell, face) of a block's cells: the face's neighbour block, its cell and
// the number of faces; false for a lane without a face.
struct FaceLane {
    int i, f, nf, kd, k, j;
    bool on;
};
__device__ __forceinline__ FaceLane face_lane(const FlowDev &F, int blk, int lane) {
    FaceLane L;
    L.i = blk * kFlowCells + (lane >> 2);
    L.f = lane & 3;
    L.on = L.i < F.nc;
    if (!L.on) L.i = F.nc - 1;
    const int k0 = F.bptr[L.i], k1 = F.bptr[L.i + 1];
    L.nf = k1 - k0 - 1;
    L.kd = k0;
    for (int k = k0; k < k1; ++k)
        if (F.bidx[k] == L.i) L.kd = k;
    L.on = L.on && L.f < L.nf;
    L.k = L.on ? k0 + L.f + (k0 + L.f >= L.kd ? 1 : 0) : L.kd;
    L.j = F.bidx[L.k];
    return L;
}

// Sum of x over a cell's faces, in face order, on the lane of its first face.
__device__ __forceinline__ double face_sum(double x, int lane, int nf) {
    double s = x;
#pragma unroll
    for (int f = 1; f < 4; ++f) {
        const double y = __shfl_sync(0xffffffffu, x, (lane & ~3) + f);
        if (f < nf) s += y;
    }
    return s;
}

// Coefficients of one block's entries: with q the block's state, level row p
// holds diag on (p, p) and cx q_p, cy q_p in the first two flow columns; flow row N + e
// holds mx + mxr r_c, my + myr r_c and h0 + he e0_c + hc cv_c + hr r_c in the level
// columns and corner[e][.] in the flow columns.
struct BlockCoef {
    double diag, cx, cy, mx, mxr, my, myr, h0, he, hc, hr, corner[3][3];
};

// Block ax A_x + ay A_y + h H of the state m (H = du/dq, A_n the flux Jacobian, linear
// in the normal), where (ax, ay) is the weighted normal.
__device__ __forceinline__ BlockCoef block_coef(const Mix &m, double ax, double ay, double h) {
    const double un = ax * m.u + ay * m.v, w = un + h, H = m.e + m.p;
    BlockCoef B;
    B.diag = w;
    B.cx = ax;
    B.cy = ay;
    B.mx = m.u * w;
    B.mxr = m.T * ax;
    B.my = m.v * w;
    B.myr = m.T * ay;
    B.he = w;
    B.h0 = w * m.ke;
    B.hc = w * m.T;
    B.hr = un * m.T;
    const double ru = m.rho * m.u, rv = m.rho * m.v;
    B.corner[0][0] = fma(m.rho, w, ru * ax);
    B.corner[0][1] = ru * ay;
    B.corner[0][2] = m.R * ax;
    B.corner[1][0] = rv * ax;
    B.corner[1][1] = fma(m.rho, w, rv * ay);
    B.corner[1][2] = m.R * ay;
    B.corner[2][0] = fma(ru, w, H * ax);
    B.corner[2][1] = fma(rv, w, H * ay);
    B.corner[2][2] = fma(m.C, w, m.R * un);
    return B;
}

// Fields of the coefficient arrays.  Block coefficients take kBlockFields from their first.
constexpr int kBlockFields = 20;
enum { fUi, fUj,            // U of the first pair: ui q_i - uj q_j (both with dt)
       fG,                  // V of a species: g da/dq, pairs 1 and 2 of q_i, pairs 1 and 2 of q_j
       fU = fG + 4,         // flow components of the pairs: U [2][3], V [4][3]
       fV = fU + 6,
       fB = fV + 12,        // the neighbour block
       fH = fB + kBlockFields,      // da/dq of q_j: G0, G1, G2 (0 where q_j gives no wave speed)
       kFaceFields = fH + 3 };
enum { cKap, cVT,           // source pair: kap beta_c, and its T component
       cB,                  // the diagonal block (without the band K and H's identity)
       kCellFields = cB + kBlockFields };
enum { rB, rD };            // residual: fields of a face (of the same array) ...
enum { rA, rOm };           // ... and of a cell
enum { bDiag, bCx, bCy, bMx, bMxr, bMy, bMyr, bH0, bHe, bHc, bHr, bCorner };      // BlockCoef in order
static_assert(bCorner + 9 == kBlockFields, "block coefficients");

// Scalars of 8 cells and their 32 directed faces, one warp, lane = (cell, face), each
// face from both of its cells.  In a kernel of its own: as the first step of the
// kernels that use the coefficients it left seven of eight warps waiting at a barrier
// (k_flow_jac 280 us on 128 x 128 cells, N = 60).
template <bool EARLY>
__global__ void __launch_bounds__(64) k_flow_face_jac(FlowDev F) {
    const int lane = threadIdx.x & 31, blk = blockIdx.x * 2 + (threadIdx.x >> 5), nc = F.nc;
    if (blk * kFlowCells >= nc) return;
    const double dt = F.dt;
    const double *M = F.mix;
    const FaceLane L = face_lane(F, blk, lane);
    if (EARLY) {
        pdl_wait();
        pdl_trigger();
    }
    const Mix mi = mix_of(M, nc, L.i), mj = mix_of(M, nc, L.j);
    double nx, ny;
    normal_of(F.Lx, L.i, L.j, nx, ny);
    const Face f = face_of(mi, mj, nx, ny);
    // a_f and c_f by division: on a supersonic face a_f is exactly +-1/2 and the
    // upwind side's weight 1/2 -+ a_f exactly zero
    const double den = f.sR - f.sL, sum = f.sL + f.sR;
    const double af = L.on ? 0.5 * sum / den : -0.5, cf = L.on ? f.sL * f.sR / den : 0.0;
    const double wL = 0.5 + af, wR = 0.5 - af;
    const double uni = nx * mi.u + ny * mi.v, unj = nx * mj.u + ny * mj.v;
    double *o = F.face + (size_t)blk * kFaceFields * 32 + lane;
    auto put = [&](int field, double v) { o[field * 32] = v; };
    put(fUi, dt * uni);
    put(fUj, dt * unj);
    const double fi[3] = {mi.rho * mi.u * uni + mi.p * nx, mi.rho * mi.v * uni + mi.p * ny, (mi.e + mi.p) * uni};
    const double fj[3] = {mj.rho * mj.u * unj + mj.p * nx, mj.rho * mj.v * unj + mj.p * ny, (mj.e + mj.p) * unj};
    const double ci[3] = {mi.rho * mi.u, mi.rho * mi.v, mi.e}, cj[3] = {mj.rho * mj.u, mj.rho * mj.v, mj.e};
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        put(fU + e, dt * (fi[e] - fj[e]));
        put(fU + 3 + e, dt * (cj[e] - ci[e]));
    }
    // V = (sR^k dsL - sL^k dsR) / den^2 (k = 1, 2) with dsL = n - da where this side
    // gives s_L, dsR = n + da where it gives s_R: A n - G da, n along the velocities.  A
    // side that gives neither has V = 0 even where its da is no number (T <= 0)
    const double i2 = f.inv_den * f.inv_den;
    auto pair = [&](bool l, bool r, int s, double gT) {
        double A1 = 0.0, G1 = 0.0, A2 = 0.0, G2 = 0.0;
        if (l && r) {
            A1 = f.inv_den;
            G1 = sum * i2;
            A2 = sum * f.inv_den;
            G2 = (f.sR * f.sR + f.sL * f.sL) * i2;
        } else if (l) {
            A1 = G1 = f.sR * i2;
            A2 = G2 = f.sR * f.sR * i2;
        } else if (r) {
            G1 = f.sL * i2;
            G2 = f.sL * f.sL * i2;
            A1 = -G1;
            A2 = -G2;
        }
        put(fG + s, -G1);
        put(fG + s + 1, -G2);
        put(fV + 3 * s, A1 * nx);
        put(fV + 3 * s + 1, A1 * ny);
        put(fV + 3 * s + 2, l || r ? -G1 * gT : 0.0);
        put(fV + 3 * s + 3, A2 * nx);
        put(fV + 3 * s + 4, A2 * ny);
        put(fV + 3 * s + 5, l || r ? -G2 * gT : 0.0);
    };
    pair(f.iL == 1, f.iR == 1, 0, M[mGT * (size_t)nc + L.i]);
    pair(f.iL == 2, f.iR == 2, 2, M[mGT * (size_t)nc + L.j]);
    auto put_block = [&](double *to, int stride, const BlockCoef &B) {
        const double v[bCorner] = {B.diag, B.cx, B.cy, B.mx, B.mxr, B.my, B.myr, B.h0, B.he, B.hc, B.hr};
#pragma unroll
        for (int e = 0; e < bCorner; ++e) to[e * stride] = v[e];
#pragma unroll
        for (int e = 0; e < 9; ++e) to[(bCorner + e) * stride] = B.corner[e / 3][e % 3];
    };
#pragma unroll
    for (int e = 0; e < 3; ++e) put(fH + e, f.iL == 2 || f.iR == 2 ? M[(mG0 + e) * (size_t)nc + L.j] : 0.0);
    put_block(o + fB * 32, 32, block_coef(mj, dt * (wR * nx), dt * (wR * ny), dt * cf));
    // the diagonal block's face sum is A_n at the summed weighted normal
    const double sx = face_sum(L.on ? wL * nx : 0.0, lane, L.nf), sy = face_sum(L.on ? wL * ny : 0.0, lane, L.nf);
    const double sc = face_sum(cf, lane, L.nf);
    if (L.f) return;
    BlockCoef X = block_coef(mi, dt * sx, dt * sy, -(dt * sc));
    // H itself on the flow rows (the level rows' identity is added to the band)
    const double he = 1.0 + X.he;
    X.mx += mi.u;
    X.my += mi.v;
    X.he = he;
    X.h0 = he * mi.ke;
    X.hc = he * mi.T;
    X.corner[0][0] += mi.rho;
    X.corner[1][1] += mi.rho;
    X.corner[2][0] += mi.rho * mi.u;
    X.corner[2][1] += mi.rho * mi.v;
    X.corner[2][2] += mi.C;
    double *c = F.cell + (size_t)blk * kCellFields * kFlowCells + (lane >> 2);
    const double kap = M[mKap * (size_t)nc + L.i];
    c[cKap * kFlowCells] = kap;
    c[cVT * kFlowCells] = kap * F.theta / (mi.T * mi.T) * M[mSb * (size_t)nc + L.i];
    put_block(c + cB * kFlowCells, kFlowCells, X);
}

// Jacobian entries, one warp per cell, lanes over the species.
template <bool EARLY>
__global__ void __launch_bounds__(kFlowCells * 32) k_flow_jac(FlowDev F, const double *Q, double *S, double *U,
                                                              double *V) {
    __shared__ double sh[kFlowCells][kFaceFields * 4 + kCellFields];
    __shared__ long long sk[kFlowCells][4];          // neighbour blocks: first S value,
    __shared__ int sj[kFlowCells][4], spo[kFlowCells][4];      // cell and first pair
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = F.b, N = F.N, w = F.w, nc = F.nc;
    const double dt = F.dt;
    const double *M = F.mix;
    const int i = blockIdx.x * kFlowCells + warp;
    if (i >= nc) return;
    const int k0 = F.bptr[i], nf = F.bptr[i + 1] - k0 - 1;
    if (EARLY) pdl_wait();
    // this cell's coefficients: fc[field * 4 + face], cc[field]
    double *fc = sh[warp], *cc = fc + kFaceFields * 4;
    const double *gf = F.face + (size_t)blockIdx.x * kFaceFields * 32 + warp * 4;
    for (int e = lane; e < kFaceFields * 4; e += 32) fc[e] = gf[(e >> 2) * 32 + (e & 3)];
    if (lane < kCellFields) cc[lane] = F.cell[((size_t)blockIdx.x * kCellFields + lane) * kFlowCells + warp];
    // lane k of the row's at most five blocks
    const int col = lane <= nf ? F.bidx[k0 + lane] : -1;
    const int at = __ffs(__ballot_sync(0xffffffffu, col == i)) - 1, kd = k0 + at;
    if (lane <= nf && lane != at) {
        const int f = lane - (lane > at ? 1 : 0);
        sj[warp][f] = col;
        spo[warp][f] = F.pip[k0 + lane];
        sk[warp][f] = F.soff[k0 + lane];
    }
    __syncwarp();
    const double *qi = Q + (size_t)i * b;
    const double g0 = M[mG0 * (size_t)nc + i], g1 = M[mG1 * (size_t)nc + i], g2 = M[mG2 * (size_t)nc + i];
    const size_t ps = (size_t)F.pip[kd];
    double *Sd = S + F.soff[kd];
    // ---- level columns of the flow rows and level components of the pairs, lanes over species
    for (int c0 = 0; c0 < N; c0 += 32) {
        const int c = c0 + lane;
        const bool on = c < N;
        const double x = on ? qi[c] : 0.0, rc = on ? __ldg(F.r + c) : 0.0, cvc = on ? __ldg(F.cv + c) : 0.0,
                     e0c = on ? __ldg(F.e0 + c) : 0.0;
        double ys[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) ys[f] = on && f < nf ? __ldg(Q + (size_t)sj[warp][f] * b + c) : 0.0;
        const double ga = fma(g2, rc, fma(g1, cvc, g0));
        if (on) {
            const double *B = cc + cB;
            double *Sf = Sd + F.d_ptr[N] + c;
            Sf[0] = fma(B[bMxr], rc, B[bMx]);
            Sf[b] = fma(B[bMyr], rc, B[bMy]);
            Sf[2 * b] = fma(B[bHr], rc, fma(B[bHc], cvc, fma(B[bHe], e0c, B[bH0])));
            U[ps * b + c] = -dt * __ldg(F.ws + c);
            V[ps * b + c] = cc[cKap] * __ldg(F.beta + c);
        }
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            if (f >= nf) break;
            const int j = sj[warp][f];
            const bool horizontal = F.Lx > 1 && (j == i + 1 || j == i - 1);
            const double *o = fc + f, *B = o + fB * 4;              // field e at o[4 e]
            const double y = ys[f];
            const double gj = fma(o[4 * (fH + 2)], rc, fma(o[4 * (fH + 1)], cvc, o[4 * fH]));
            const size_t pd = ps + 1 + 2 * f, po = (size_t)spo[warp][f];
            double *Sk = S + sk[warp][f];
            if (on) {
                const double u1 = fma(o[4 * fUi], x, -(o[4 * fUj] * y)), u2 = dt * (y - x);
                U[pd * b + c] = u1;
                U[(pd + 1) * b + c] = u2;
                U[po * b + c] = u1;
                U[(po + 1) * b + c] = u2;
                V[pd * b + c] = o[4 * fG] * ga;
                V[(pd + 1) * b + c] = o[4 * fG + 4] * ga;
                V[po * b + c] = o[4 * fG + 8] * gj;
                V[(po + 1) * b + c] = o[4 * fG + 12] * gj;
                // the normal is along one axis: one momentum row is constant over the species
                const int m = horizontal ? bMx : bMy;
                const double t = fma(B[4 * (m + 1)], rc, B[4 * m]), u = B[4 * (bMx + bMy - m)];
                double *Sf = Sk + 4 * N + c;
                Sf[0] = horizontal ? t : u;
                Sf[b] = horizontal ? u : t;
                Sf[2 * b] = fma(B[4 * bHr], rc, fma(B[4 * bHc], cvc, fma(B[4 * bHe], e0c, B[4 * bH0])));
            }
            // neighbour block's level rows [diag, cx q, cy q, 0]: 32 rows are 128 consecutive
            // entries; one of cx, cy is zero
            const double z = B[4 * (horizontal ? bCx : bCy)] * y, d = B[4 * bDiag];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const double zr = __shfl_sync(0xffffffffu, z, r * 8 + (lane >> 2));
                const int col = lane & 3;
                if (c0 + r * 8 + (lane >> 2) < N)
                    Sk[4 * c0 + r * 32 + lane] = col == 0 ? d : col == (horizontal ? 1 : 2) ? zr : 0.0;
            }
        }
    }
    // where da/dq_i is no number, 0 times it was none: the pairs of the faces that take no bound
    // from q_i (both G are 0), after the loop, which has no instruction to spare for them; by the
    // exponents, since two sums and a comparison are FP64 instructions of the whole warp
    auto no_number = [](double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; };
    if (no_number(g0) || no_number(g1) || no_number(g2))
        for (int f = 0; f < nf; ++f) {
            const double *o = fc + f;
            if (o[4 * fG] != 0.0 || o[4 * fG + 4] != 0.0) continue;
            double *v = V + (ps + 1 + 2 * f) * b;
            for (int c = lane; c < N; c += 32) v[c] = v[b + c] = 0.0;       // the lane that wrote them
        }
    // ---- flow components: computed by k_flow_face_jac, only written here
    for (int f = 0; f < nf; ++f) {
        const double *o = fc + f;
        const size_t pd = ps + 1 + 2 * f, po = (size_t)spo[warp][f];
        if (lane < 24) {
            const int row = lane / 3, e = lane - 3 * row;         // U pd, pd+1, po, po+1, then V of the same
            const size_t at = ((row & 2 ? po : pd) + (row & 1)) * b + N + e;
            if (row < 4) U[at] = o[4 * (fU + 3 * (row & 1) + e)];
            else V[at] = o[4 * (fV + 3 * (row & 3) + e)];
        }
        if (lane < 9) S[sk[warp][f] + 4 * N + (size_t)(lane / 3) * b + N + lane % 3] = o[4 * (fB + bCorner + lane)];
    }
    if (lane < 9) Sd[F.d_ptr[N] + (lane / 3) * b + N + lane % 3] = cc[cB + bCorner + lane];
    if (lane < 3) {
        U[ps * b + N + lane] = 0.0;
        V[ps * b + N + lane] = lane == 2 ? cc[cVT] : 0.0;
    }
    // ---- the diagonal block's level rows: band K (plus H = 1 and the face terms on the
    // diagonal) and the flow columns, lanes over the pattern's consecutive entries
    const int nl = F.d_ptr[N];
#pragma unroll 4
    for (int e = lane; e < nl; e += 32) {
        const short2 pq = F.d_pq[e];
        const int p = pq.x, c = pq.y;
        double base = 0.0, coef = 0.0, x = 1.0;
        if (c < N) {
            base = __ldg(F.dtK + (size_t)p * (2 * w + 1) + (c - p + w));
            coef = c == p ? cc[cB + bDiag] : 0.0;
        } else {
            coef = c == N ? cc[cB + bCx] : c == N + 1 ? cc[cB + bCy] : 0.0;
            x = qi[p];
        }
        Sd[e] = fma(coef, x, base);
    }
}

// Residual scalars, as k_flow_face_jac; the flow components are complete here.  With
// the flux (s_R f_i - s_L f_j + s_L s_R (u_j - u_i)) / (s_R - s_L) the species flux of a
// face is ca q_i - cb q_j + cd (q_j - q_i).
template <bool EARLY>
__global__ void __launch_bounds__(64) k_flow_face_res(FlowDev F, double *R) {
    const int lane = threadIdx.x & 31, blk = blockIdx.x * 2 + (threadIdx.x >> 5), nc = F.nc;
    if (blk * kFlowCells >= nc) return;
    const double *M = F.mix, *Mn = F.mix + (size_t)kMixFields * nc;
    const FaceLane L = face_lane(F, blk, lane);
    if (EARLY) {
        pdl_wait();
        pdl_trigger();
    }
    const Mix mi = mix_of(M, nc, L.i), mj = mix_of(M, nc, L.j);
    double nx, ny;
    normal_of(F.Lx, L.i, L.j, nx, ny);
    const Face f = face_of(mi, mj, nx, ny);
    const double uni = nx * mi.u + ny * mi.v, unj = nx * mj.u + ny * mj.v;
    const double ca = f.sR * f.inv_den, cb = f.sL * f.inv_den, cd = f.sL * f.sR * f.inv_den;
    const double fi[3] = {mi.rho * mi.u * uni + mi.p * nx, mi.rho * mi.v * uni + mi.p * ny, (mi.e + mi.p) * uni};
    const double fj[3] = {mj.rho * mj.u * unj + mj.p * nx, mj.rho * mj.v * unj + mj.p * ny, (mj.e + mj.p) * unj};
    const double ci[3] = {mi.rho * mi.u, mi.rho * mi.v, mi.e}, cj[3] = {mj.rho * mj.u, mj.rho * mj.v, mj.e};
    double *o = F.face + (size_t)blk * kFaceFields * 32 + lane;
    o[rB * 32] = cb * unj;
    o[rD * 32] = cd;
    const double sum = face_sum(L.on ? ca * uni : 0.0, lane, L.nf);
    double fl[3];
#pragma unroll
    for (int e = 0; e < 3; ++e)
        fl[e] = face_sum(L.on ? (ca * fi[e] - cb * fj[e]) + cd * (cj[e] - ci[e]) : 0.0, lane, L.nf);
    if (L.f || blk * kFlowCells + (lane >> 2) >= nc) return;
    double *c = F.cell + (size_t)blk * kCellFields * kFlowCells + (lane >> 2);
    c[rA * kFlowCells] = sum;
    c[rOm * kFlowCells] = M[mKap * (size_t)nc + L.i] * M[mSb * (size_t)nc + L.i];
    const Mix mn = mix_of(Mn, nc, L.i);
    const double cn[3] = {mn.rho * mn.u, mn.rho * mn.v, mn.e};
#pragma unroll
    for (int e = 0; e < 3; ++e) R[(size_t)L.i * F.b + F.N + e] = (ci[e] - cn[e]) + F.dt * fl[e];
}

// Residual of the species, one warp per cell, lanes over the species.
template <bool EARLY>
__global__ void __launch_bounds__(kFlowCells * 32) k_flow_res(FlowDev F, const double *Q, const double *Qn,
                                                              double *R) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = F.b, N = F.N, w = F.w, bw = 2 * w + 1;
    const int i = blockIdx.x * kFlowCells + warp;
    if (i >= F.nc) return;
    const int k0 = F.bptr[i], nf = F.bptr[i + 1] - k0 - 1;
    int j[4];                                   // neighbours in block order
#pragma unroll
    for (int f = 0, k = k0; f < 4; ++f, ++k) {
        if (f < nf && F.bidx[k] == i) ++k;
        j[f] = f < nf ? F.bidx[k] : i;
    }
    if (EARLY) pdl_wait();
    const double *gf = F.face + (size_t)blockIdx.x * kFaceFields * 32 + warp * 4;
    const double *gc = F.cell + (size_t)blockIdx.x * kCellFields * kFlowCells + warp;
    double fb[4], fd[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        fb[f] = gf[rB * 32 + f];
        fd[f] = gf[rD * 32 + f];
    }
    const double ca = gc[rA * kFlowCells], omega = gc[rOm * kFlowCells];
    const double *qi = Q + (size_t)i * b, *qn = Qn + (size_t)i * b;
    for (int c = lane; c < N; c += 32) {
        const double x = qi[c], xn = qn[c];
        double y[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) y[f] = __ldg(Q + (size_t)j[f] * b + c);
        double acc = ca * x;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            if (f >= nf) break;
            acc = fma(-fb[f], y[f], acc);
            acc = fma(fd[f], y[f] - x, acc);
        }
        double src = 0.0;
        for (int l = max(0, c - w); l < min(N, c + w + 1); ++l)
            src = fma(-__ldg(F.K + (size_t)c * bw + (l - c + w)), qi[l], src);
        src = fma(__ldg(F.ws + c), omega, src);
        R[(size_t)i * b + c] = (x - xn) + F.dt * (acc - src);
    }
}

constexpr int kNormBlocks = 304;     // 2 x 152 SMs
constexpr int kNormThreads = 256;

// Per-block sums of squares (block tree in shared memory); the host adds the
// kNormBlocks partials in block order, so the norm is deterministic.
__global__ void __launch_bounds__(kNormThreads) k_flow_sumsq(const double *x, long long n, double *partial) {
    __shared__ double sh[kNormThreads];
    double s = 0.0;
    for (long long i = (long long)blockIdx.x * kNormThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kNormThreads)
        s = fma(x[i], x[i], s);
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = kNormThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

// y = a + alpha * d   (alpha = 0 and a = 0: y = -d when neg is set)
__global__ void k_flow_axpy(double *y, const double *a, double alpha, const double *d, long long n, int neg) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = neg ? -d[i] : fma(alpha, d[i], a[i]);
}

}  // namespace
}  // namespace sts

using namespace sts;

struct sts_flow_s {
    FlowDev dev{};
    cudaStream_t stream = nullptr;
    int Lx = 0, Ly = 0;
    std::vector<int> bptr, bidx, dptr, didx, optr, oidx, pip;
    long long nnz_S = 0;
    std::vector<void *> bufs;
    // Newton workspace, allocated on the first sts_flow_newton
    double *S = nullptr, *U = nullptr, *V = nullptr, *R = nullptr, *Rt = nullptr, *rhs = nullptr,
           *dQ = nullptr, *Qt = nullptr, *partial = nullptr, *h_partial = nullptr;
};

namespace {

void flow_free(sts_flow_s *f) {
    for (void *p : f->bufs) cudaFree(p);
    f->bufs.clear();
    if (f->h_partial) cudaFreeHost(f->h_partial);
    f->h_partial = nullptr;
}

sts_status flow_alloc(sts_flow_s *f, double **p, size_t n) {
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, (n ? n : 1) * sizeof(double));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(STS_ERR_ALLOC, "flow generator: cudaMalloc of %zu doubles failed: %s", n,
                         cudaGetErrorString(e));
    }
    f->bufs.push_back(q);
    *p = static_cast<double *>(q);
    return STS_OK;
}

// Small grids: the launches set the time, so each kernel after the first is launched early
// (EARLY instances: programmatic dependent launch).  As three dependent kernels the calls
// had become slower there than the single kernel they came from (a column of 200 cells, N =
// 20: residual 22.3, then 25.4, now 20.6 us).  Early blocks take room from the kernel they
// wait for: a Jacobian of 24 x 24 cells (72 blocks) takes 39.1 and 34.7 us, of 32 x 32 (128)
// 38.6 and 39.0, of 48 x 48 47.8 and 54.8; so below one block of the last kernel per two SMs.
constexpr int kEarlyCells = 152 / 2 * kFlowCells;

template <bool EARLY, typename... KArgs, typename... Args>
sts_status flow_launch(sts_flow_s *f, void (*kern)(KArgs...), int cells, int threads, Args... args) {
    const unsigned blocks = (f->dev.nc + cells - 1) / cells;
    if (EARLY) STS_CK(launch_pdl(kern, dim3(blocks), dim3(threads), 0, f->stream, args...));
    else kern<<<blocks, threads, 0, f->stream>>>(args...);
    STS_LAUNCHED();
    return STS_OK;
}

template <bool EARLY>
sts_status flow_mix(sts_flow_s *f, const double *Q, const double *Qn) {
    const int b = f->dev.b;
    const size_t smem = (32 * (size_t)(b | 1) + 4 * (size_t)f->dev.N + 4 * 5 * 32) * sizeof(double);
    if (smem > 48 * 1024) STS_CK(allow_all_smem(k_flow_mix<EARLY>));
    k_flow_mix<EARLY><<<dim3((f->dev.nc + kMixCells - 1) / kMixCells, Qn ? 2 : 1), 128, smem, f->stream>>>(f->dev, Q, Qn);
    STS_LAUNCHED();
    return STS_OK;
}

template <bool EARLY>
sts_status flow_res_as(sts_flow_s *f, const double *Q, const double *Qn, double *R) {
    STS_TRY(flow_mix<EARLY>(f, Q, Qn));
    STS_TRY(flow_launch<EARLY>(f, k_flow_face_res<EARLY>, 2 * kFlowCells, 64, f->dev, R));
    return flow_launch<EARLY>(f, k_flow_res<EARLY>, kFlowCells, kFlowCells * 32, f->dev, Q, Qn, R);
}
sts_status flow_res(sts_flow_s *f, const double *Q, const double *Qn, double *R) {
    return f->dev.nc < kEarlyCells ? flow_res_as<true>(f, Q, Qn, R) : flow_res_as<false>(f, Q, Qn, R);
}

template <bool EARLY>
sts_status flow_jac_as(sts_flow_s *f, const double *Q, double *S, double *U, double *V) {
    STS_TRY(flow_mix<EARLY>(f, Q, nullptr));
    STS_TRY(flow_launch<EARLY>(f, k_flow_face_jac<EARLY>, 2 * kFlowCells, 64, f->dev));
    return flow_launch<EARLY>(f, k_flow_jac<EARLY>, kFlowCells, kFlowCells * 32, f->dev, Q, S, U, V);
}
sts_status flow_jac(sts_flow_s *f, const double *Q, double *S, double *U, double *V) {
    return f->dev.nc < kEarlyCells ? flow_jac_as<true>(f, Q, S, U, V) : flow_jac_as<false>(f, Q, S, U, V);
}

// ||x||_2 of a device vector of the generator's stream (synchronous)
sts_status flow_norm(sts_flow_s *f, const double *x, long long n, double *out) {
    k_flow_sumsq<<<kNormBlocks, kNormThreads, 0, f->stream>>>(x, n, f->partial);
    STS_LAUNCHED();
    STS_CK(cudaMemcpyAsync(f->h_partial, f->partial, kNormBlocks * sizeof(double), cudaMemcpyDeviceToHost, f->stream));
    STS_CK(cudaStreamSynchronize(f->stream));
    double s = 0.0;
    for (int i = 0; i < kNormBlocks; ++i) s += f->h_partial[i];
    *out = std::sqrt(s);
    return STS_OK;
}

unsigned flow_grid(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 152LL * 16); }

sts_status flow_newton(sts_flow_s *f, sts_jac_t jac, double *Q, const double *Qn, const sts_newton_opts *o,
                       sts_newton_info *info) {
    if (!f || !jac || !Q || !Qn) return set_error(STS_ERR_INVALID_ARG, "sts_flow_newton: NULL argument");
    sts_newton_opts d{};
    if (o) d = *o;
    const int max_newton = d.max_newton > 0 ? d.max_newton : 20;
    const double rtol = d.rtol > 0 ? d.rtol : 1e-10;
    const double atol = d.atol > 0 ? d.atol : 0.0;
    const int max_halvings = d.max_halvings > 0 ? d.max_halvings : 8;
    if (d.gmres.vectors_on_host) return set_error(STS_ERR_INVALID_ARG, "sts_flow_newton: gmres.vectors_on_host must be 0");
    if (d.gmres.trans) return set_error(STS_ERR_INVALID_ARG, "sts_flow_newton: gmres.trans must be 0");
    // the handle must hold this generator's layout
    if (jac->layout != STS_LAYOUT_CELL_MAJOR || jac->nc != f->dev.nc ||
        jac->b != f->dev.b || jac->bidx != f->bidx || jac->bptr != f->bptr || jac->pbase != f->pip ||
        jac->dptr != f->dptr || jac->didx != f->didx || jac->optr != f->optr || jac->oidx != f->oidx)
        return set_error(STS_ERR_INVALID_ARG, "sts_flow_newton: jac is not a cell-major handle of this "
                                              "generator's layout");
    const long long n = (long long)f->dev.nc * f->dev.b;
    if (!f->R) {
        STS_TRY(flow_alloc(f, &f->S, (size_t)f->nnz_S));
        STS_TRY(flow_alloc(f, &f->U, (size_t)f->pip.back() * f->dev.b));
        STS_TRY(flow_alloc(f, &f->V, (size_t)f->pip.back() * f->dev.b));
        STS_TRY(flow_alloc(f, &f->R, n));
        STS_TRY(flow_alloc(f, &f->Rt, n));
        STS_TRY(flow_alloc(f, &f->rhs, n));
        STS_TRY(flow_alloc(f, &f->dQ, n));
        STS_TRY(flow_alloc(f, &f->Qt, n));
        STS_TRY(flow_alloc(f, &f->partial, kNormBlocks));
        STS_CK(cudaMallocHost(&f->h_partial, kNormBlocks * sizeof(double)));
    }
    const unsigned eg = flow_grid(n);
    sts_newton_info inf{0, 0, 0, 0, 0.0, 0.0};
    STS_TRY(flow_res(f, Q, Qn, f->R));
    double r = 0.0;
    STS_TRY(flow_norm(f, f->R, n, &r));
    inf.res0 = inf.res = r;
    if (d.history) d.history[0] = r;
    if (!std::isfinite(r)) {
        if (info) *info = inf;
        return set_error(STS_ERR_NUMERIC, "sts_flow_newton: the initial residual is NaN or Inf");
    }
    const double tol = std::max(rtol * r, atol);
    sts_status status = STS_OK;
    // inexact Newton forcing (Eisenstat & Walker, choice 2; Kelley's safeguards)
    constexpr double kEtaMax = 0.9, kGamma = 0.9;
    double eta = kEtaMax, r_prev = r;
    while (true) {
        if (r <= tol) {
            inf.converged = 1;
            break;
        }
        if (inf.iterations >= max_newton) break;
        NvtxRange nvtx_it("newton iteration");
        // Jacobian at Q into the handle, block-Jacobi, then J dQ = -R
        STS_TRY(flow_jac(f, Q, f->S, f->U, f->V));
        k_flow_axpy<<<eg, 256, 0, f->stream>>>(f->rhs, nullptr, 0.0, f->R, n, 1);
        STS_LAUNCHED();
        STS_CK(cudaMemsetAsync(f->dQ, 0, n * sizeof(double), f->stream));
        STS_CK(cudaStreamSynchronize(f->stream));
        STS_TRY(sts_jac_update_values(jac, f->S, f->U, f->V, 0));
        if (d.gmres.precond != STS_PRECOND_NONE) STS_TRY(sts_jac_bjacobi_setup(jac));
        sts_gmres_info gi{};
        sts_gmres_opts go = d.gmres;
        if (d.forcing) {
            if (inf.iterations > 0) {
                const double ea = kGamma * (r / r_prev) * (r / r_prev);
                const double eb = kGamma * eta * eta > 0.1 ? std::max(ea, kGamma * eta * eta) : ea;
                eta = std::min(kEtaMax, std::max(eb, 0.5 * tol / r));
            }
            go.rtol = eta;
        }
        const sts_status gs = sts_gmres_solve(jac, f->rhs, f->dQ, &go, &gi);
        if (gs != STS_OK && gs != STS_ERR_NOT_CONVERGED) return gs;
        inf.linear_iterations += gi.iterations;
        // line search: alpha = 1, 1/2, ... until ||R|| decreases
        double alpha = 1.0, rt = 0.0;
        bool accepted = false;
        for (int hv = 0; hv <= max_halvings; ++hv) {
            k_flow_axpy<<<eg, 256, 0, f->stream>>>(f->Qt, Q, alpha, f->dQ, n, 0);
            STS_LAUNCHED();
            STS_TRY(flow_res(f, f->Qt, Qn, f->Rt));
            STS_TRY(flow_norm(f, f->Rt, n, &rt));
            if (std::isfinite(rt) && rt < r) {
                accepted = true;
                break;
            }
            alpha *= 0.5;
            ++inf.halvings;
        }
        ++inf.iterations;
        if (!accepted) {
            status = set_error(STS_ERR_NOT_CONVERGED, "sts_flow_newton: no decrease of ||R|| = %.3e after %d halvings "
                                                      "(iteration %d)", r, max_halvings, inf.iterations);
            break;
        }
        STS_CK(cudaMemcpyAsync(Q, f->Qt, n * sizeof(double), cudaMemcpyDeviceToDevice, f->stream));
        std::swap(f->R, f->Rt);
        r_prev = r;
        r = rt;
        inf.res = r;
        if (d.history) d.history[inf.iterations] = r;
    }
    STS_CK(cudaStreamSynchronize(f->stream));
    if (info) *info = inf;
    if (status != STS_OK) return status;
    if (!inf.converged)
        return set_error(STS_ERR_NOT_CONVERGED, "sts_flow_newton: %d iterations, ||R|| = %.3e > %.3e", inf.iterations,
                         r, tol);
    return STS_OK;
}

template <typename T>
sts_status flow_upload(sts_flow_s *f, const T **dst, const T *src, size_t n) {
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, (n ? n : 1) * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(STS_ERR_ALLOC, "sts_flow_create: cudaMalloc failed: %s", cudaGetErrorString(e));
    }
    f->bufs.push_back(p);
    if (n) STS_CK(cudaMemcpyAsync(p, src, n * sizeof(T), cudaMemcpyHostToDevice, f->stream));
    *dst = static_cast<const T *>(p);
    return STS_OK;
}

sts_status flow_create(const sts_flow_desc *d, sts_flow_t *out) {
    if (!out) return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: out is NULL");
    *out = nullptr;
    if (!d) return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: desc is NULL");
    const int N = d->n_species, w = d->band;
    if (d->Lx < 1 || d->Ly < 1 || N < 1 || w < 0)
        return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: need Lx, Ly, n_species >= 1 and band >= 0");
    if (N + 3 > 256) return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: block size N + 3 must be <= 256");
    if ((long long)d->Lx * d->Ly * (N + 3) > (1LL << 31) - 1)
        return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: n_cells * block_size must fit in int32");
    if (!d->r || !d->cv || !d->e0 || !d->beta || !d->ws || !d->K)
        return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: a constant array is NULL");
    for (int k = 0; k < N; ++k) {
        if (!(d->r[k] > 0.0) || !(d->cv[k] > 0.0) || !std::isfinite(d->r[k]) || !std::isfinite(d->cv[k]))
            return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: r[%d] and cv[%d] must be finite and > 0", k, k);
        if (!std::isfinite(d->e0[k]) || !std::isfinite(d->beta[k]) || !std::isfinite(d->ws[k]))
            return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: non-finite constant of species %d", k);
    }
    for (long long e = 0; e < (long long)N * (2 * w + 1); ++e)
        if (!std::isfinite(d->K[e])) return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: non-finite K");
    if (!std::isfinite(d->A) || !std::isfinite(d->theta) || !std::isfinite(d->dt))
        return set_error(STS_ERR_INVALID_ARG, "sts_flow_create: non-finite A, theta or dt");

    sts_flow_s *f = new sts_flow_s();
    f->stream = static_cast<cudaStream_t>(d->stream);
    f->Lx = d->Lx;
    f->Ly = d->Ly;
    const int Lx = d->Lx, Ly = d->Ly, nc = Lx * Ly, b = N + 3;
    // mesh adjacency: i-Lx, i-1, i, i+1, i+Lx where present
    f->bptr.assign(1, 0);
    for (int i = 0; i < nc; ++i) {
        const int ix = i % Lx, iy = i / Lx;
        if (iy > 0) f->bidx.push_back(i - Lx);
        if (ix > 0) f->bidx.push_back(i - 1);
        f->bidx.push_back(i);
        if (ix < Lx - 1) f->bidx.push_back(i + 1);
        if (iy < Ly - 1) f->bidx.push_back(i + Lx);
        f->bptr.push_back((int)f->bidx.size());
    }
    // patterns (the kernels write them in this order)
    f->dptr.assign(1, 0);
    f->optr.assign(1, 0);
    for (int p = 0; p < b; ++p) {
        if (p < N) {
            for (int c = std::max(0, p - w); c <= std::min(N - 1, p + w); ++c) f->didx.push_back(c);
            for (int c = N; c < b; ++c) f->didx.push_back(c);
            f->oidx.push_back(p);
            for (int c = N; c < b; ++c) f->oidx.push_back(c);
        } else {
            for (int c = 0; c < b; ++c) {
                f->didx.push_back(c);
                f->oidx.push_back(c);
            }
        }
        f->dptr.push_back((int)f->didx.size());
        f->optr.push_back((int)f->oidx.size());
    }
    // S offsets and pairs: 1 + 2 per face on the diagonal block, 2 on a neighbour block
    const int nnzb = (int)f->bidx.size();
    std::vector<long long> soff(nnzb + 1, 0);
    f->pip.assign(nnzb + 1, 0);
    for (int i = 0; i < nc; ++i) {
        const int deg = f->bptr[i + 1] - f->bptr[i] - 1;
        for (int k = f->bptr[i]; k < f->bptr[i + 1]; ++k) {
            const bool diag = f->bidx[k] == i;
            soff[k + 1] = soff[k] + (diag ? (long long)f->didx.size() : (long long)f->oidx.size());
            f->pip[k + 1] = f->pip[k] + (diag ? 1 + 2 * deg : 2);
        }
    }
    f->nnz_S = soff[nnzb];
    FlowDev &D = f->dev;
    D.Lx = Lx;
    D.nc = nc;
    D.N = N;
    D.b = b;
    D.w = w;
    D.nnz_d = (int)f->didx.size();
    D.nnz_o = (int)f->oidx.size();
    D.A = d->A;
    D.theta = d->theta;
    D.dt = d->dt;
    std::vector<double> dtK((size_t)N * (2 * w + 1));
    for (size_t e = 0; e < dtK.size(); ++e) dtK[e] = d->dt * d->K[e] + ((int)(e % (2 * w + 1)) == w ? 1.0 : 0.0);
    std::vector<short2> pq;
    for (int p = 0; p < N; ++p)
        for (int e = f->dptr[p]; e < f->dptr[p + 1]; ++e) pq.push_back(make_short2((short)p, (short)f->didx[e]));
    sts_status st = STS_OK;
    do {
        if ((st = flow_alloc(f, &D.mix, 2 * (size_t)kMixFields * nc)) != STS_OK) break;
        const size_t blocks = (nc + kFlowCells - 1) / kFlowCells;
        if ((st = flow_alloc(f, &D.face, blocks * kFaceFields * 32)) != STS_OK) break;
        if ((st = flow_alloc(f, &D.cell, blocks * kCellFields * kFlowCells)) != STS_OK) break;
        if ((st = flow_upload(f, &D.dtK, dtK.data(), dtK.size())) != STS_OK) break;
        if ((st = flow_upload(f, &D.d_pq, pq.data(), pq.size())) != STS_OK) break;
        if ((st = flow_upload(f, &D.r, d->r, N)) != STS_OK) break;
        if ((st = flow_upload(f, &D.cv, d->cv, N)) != STS_OK) break;
        if ((st = flow_upload(f, &D.e0, d->e0, N)) != STS_OK) break;
        if ((st = flow_upload(f, &D.beta, d->beta, N)) != STS_OK) break;
        if ((st = flow_upload(f, &D.ws, d->ws, N)) != STS_OK) break;
        if ((st = flow_upload(f, &D.K, d->K, (size_t)N * (2 * w + 1))) != STS_OK) break;
        if ((st = flow_upload(f, &D.bptr, f->bptr.data(), f->bptr.size())) != STS_OK) break;
        if ((st = flow_upload(f, &D.bidx, f->bidx.data(), f->bidx.size())) != STS_OK) break;
        if ((st = flow_upload(f, &D.pip, f->pip.data(), f->pip.size())) != STS_OK) break;
        if ((st = flow_upload(f, &D.soff, soff.data(), soff.size())) != STS_OK) break;
        if ((st = flow_upload(f, &D.d_ptr, f->dptr.data(), f->dptr.size())) != STS_OK) break;
        cudaError_t e = cudaStreamSynchronize(f->stream);   // the host vectors above are temporaries
        if (e != cudaSuccess) st = set_error(STS_ERR_CUDA, "sts_flow_create: %s", cudaGetErrorString(e));
    } while (false);
    if (st != STS_OK) {
        cudaStreamSynchronize(f->stream);
        flow_free(f);
        delete f;
        return st;
    }
    *out = f;
    return STS_OK;
}

}  // namespace

#define STS_FLOW_GUARD(body)                                                      \
    try {                                                                         \
        body                                                                      \
    } catch (const std::bad_alloc &) {                                            \
        return set_error(STS_ERR_ALLOC, "host allocation failed");                \
    } catch (...) {                                                               \
        return set_error(STS_ERR_INVALID_ARG, "unexpected exception");            \
    }

extern "C" {

sts_status sts_flow_create(const sts_flow_desc *d, sts_flow_t *out) {
    NvtxRange nvtx_range("sts_flow_create");
    STS_FLOW_GUARD(return flow_create(d, out);)
}

sts_status sts_flow_get_sizes(sts_flow_t f, sts_flow_sizes *s) {
    if (!f || !s) return set_error(STS_ERR_INVALID_ARG, "sts_flow_get_sizes: NULL argument");
    s->n_cells = f->dev.nc;
    s->block_size = f->dev.b;
    s->nnzb = (int)f->bidx.size();
    s->nnz_d = f->dev.nnz_d;
    s->nnz_o = f->dev.nnz_o;
    s->n_pairs = f->pip.back();
    s->nnz_S = f->nnz_S;
    return STS_OK;
}

sts_status sts_flow_get_layout(sts_flow_t f, int *block_indptr, int *block_indices, int *d_indptr, int *d_indices,
                               int *o_indptr, int *o_indices, int *pair_indptr) {
    if (!f || !block_indptr || !block_indices || !d_indptr || !d_indices || !o_indptr || !o_indices || !pair_indptr)
        return set_error(STS_ERR_INVALID_ARG, "sts_flow_get_layout: NULL argument");
    std::copy(f->bptr.begin(), f->bptr.end(), block_indptr);
    std::copy(f->bidx.begin(), f->bidx.end(), block_indices);
    std::copy(f->dptr.begin(), f->dptr.end(), d_indptr);
    std::copy(f->didx.begin(), f->didx.end(), d_indices);
    std::copy(f->optr.begin(), f->optr.end(), o_indptr);
    std::copy(f->oidx.begin(), f->oidx.end(), o_indices);
    std::copy(f->pip.begin(), f->pip.end(), pair_indptr);
    return STS_OK;
}

sts_status sts_flow_residual(sts_flow_t f, const double *Q, const double *Qn, double *R) {
    NvtxRange nvtx_range("sts_flow_residual");
    if (!f || !Q || !Qn || !R) return set_error(STS_ERR_INVALID_ARG, "sts_flow_residual: NULL argument");
    return flow_res(f, Q, Qn, R);
}

sts_status sts_flow_jacobian(sts_flow_t f, const double *Q, double *S, double *U, double *V) {
    NvtxRange nvtx_range("sts_flow_jacobian");
    if (!f || !Q || !S || !U || !V) return set_error(STS_ERR_INVALID_ARG, "sts_flow_jacobian: NULL argument");
    return flow_jac(f, Q, S, U, V);
}

sts_status sts_flow_newton(sts_flow_t f, sts_jac_t jac, double *Q, const double *Qn, const sts_newton_opts *opts,
                           sts_newton_info *info) {
    NvtxRange nvtx_range("sts_flow_newton");
    STS_FLOW_GUARD(return flow_newton(f, jac, Q, Qn, opts, info);)
}

sts_status sts_flow_destroy(sts_flow_t f) {
    if (!f) return STS_OK;
    cudaStreamSynchronize(f->stream);
    flow_free(f);
    delete f;
    return STS_OK;
}

}  // extern "C"
