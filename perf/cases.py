"""Performance cases of the block r1-sparse Jacobian library: what its users have it do.

An implicit flow solver generates its Jacobian (flow), loads it into a handle and sets
the preconditioner up (refresh), applies J, J^T, M and M^T (matvec, apply, general) and
solves with GMRES (gmres, mixed), once per Newton iteration (newton); an adjoint code
differentiates the solve (adjoint).  Every case goes through the package's public Python
entry points.  Inputs are seeded synthetic Jacobians with the structure of the paper's
quad-grid state-to-state problems, drawn on the GPU.

Fields of a case: kind (above), Lx, Ly (grid), N (levels; the block size is N + 3), w (level
band), rd, ro (rank-one pairs per diagonal / neighbour block), ppf (pairs that a diagonal
block gains per face neighbour), dt (pseudo time step: 1/dt sits on the diagonal), layout
("cell": the default block vectors, "component": the kernels' own), pattern ("paper": band,
dense flow rows and columns; "shared": the diagonal-block pattern on the neighbours too;
"random": arbitrary sparsity).
"""
import math

import numpy as np
import torch

from paper_2403_09198_gb300.autograd import ImplicitSolve
from paper_2403_09198_gb300.binding import StsFlow, StsJacobian

F64 = torch.float64


def _case(name, kind, Lx, Ly, N, w=2, rd=2, ro=1, ppf=0, dt=1e-3, layout="cell", pattern="paper"):
    c = dict(kind=kind, Lx=Lx, Ly=Ly, N=N, w=w, rd=rd, ro=ro, ppf=ppf, dt=dt, layout=layout, pattern=pattern)
    return dict(c, name=name) if name else c


def listed():
    return [
        # J x and J^T x on a small problem (a coarse-grid or unit-test call): latency and launches
        _case("matvec_16x16_N10", "matvec", 16, 16, 10),
        # the same at the ordinary size, vectors kept in the kernels' layout as a Krylov user keeps them
        _case("matvec_128x128_N60", "matvec", 128, 128, 60, layout="component"),
        # the same at the largest size: 200 levels, wider band, three pairs
        _case("matvec_256x256_N200", "matvec", 256, 256, 200, w=4, rd=3),
        # J, J^T, M and M^T of a Jacobian whose sparsity is not the paper's (another mechanism), ragged grid
        _case("general_41x37_N30", "general", 41, 37, 30, pattern="random"),
        # block-Jacobi M x and M^T x, the preconditioner of a user's own Krylov loop
        _case("apply_128x128_N60", "apply", 128, 128, 60, layout="component"),
        # new values into a handle, preconditioner set up, one product and one apply: a Jacobian refresh
        # with the paper's pair counts (one source pair and two per face)
        _case("refresh_128x128_N60", "refresh", 128, 128, 60, rd=1, ro=2, ppf=2),
        # preconditioned GMRES to 1e-10 on a small problem
        _case("gmres_16x16_N10", "gmres", 16, 16, 10),
        # the same at the ordinary size with a larger time step (more iterations), ragged grid
        _case("gmres_125x121_N60", "gmres", 125, 121, 60, dt=2e-2),
        # FP32 operators inside FP64 flexible GMRES
        _case("mixed_256x256_N60", "mixed", 256, 256, 60, layout="component"),
        # implicit solve and its gradients with respect to the right-hand side and all Jacobian values
        _case("adjoint_128x128_N60", "adjoint", 128, 128, 60),
        # residual and r1-sparse Jacobian of the HLL-flux flow model
        _case("flow_128x128_N60", "flow", 128, 128, 60, dt=0.5),
        # one whole implicit pseudo-time step (Newton, each linear solve by GMRES)
        _case("newton_128x128_N60", "newton", 128, 128, 60, dt=0.5),
    ]


# work limit (cells x block size) of the drawn cases of each kind: the listed one's, or less
_CAP = {"matvec": 256 * 256 * 203, "general": 128 * 64 * 33, "apply": 256 * 128 * 63, "refresh": 128 * 128 * 63,
        "gmres": 128 * 128 * 63, "mixed": 256 * 256 * 63, "adjoint": 128 * 128 * 63, "flow": 128 * 128 * 63,
        "newton": 96 * 96 * 63}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(sorted(_CAP))
    N = _log(rng, 4, 40) if kind == "general" else _log(rng, 8, 100) if kind in ("flow", "newton") else _log(rng, 6, 200)
    cells = _log(rng, 60, max(64, _CAP[kind] // (N + 3)))
    Lx = max(1, min(cells, int(round(math.sqrt(cells) * math.exp(rng.uniform(-0.7, 0.7))))))
    Ly = max(1, cells // Lx)
    w = rng.randint(1, 4)
    rd, ro, ppf = rng.choice([(2, 1, 0), (3, 1, 0), (1, 2, 2)])
    dt = math.exp(rng.uniform(math.log(1e-3), math.log(2e-2)))
    pattern = "paper"
    if kind == "general":
        pattern, rd, ro, ppf = rng.choice(["random", "shared"]), 2, 1, 0
    if kind in ("flow", "newton"):
        rd, ro, ppf, dt = 1, 2, 2, rng.uniform(0.1, 0.5)
    layout = "cell" if kind in ("adjoint", "flow", "newton") else rng.choice(["cell", "component"])
    return _case(None, kind, Lx, Ly, N, w, rd, ro, ppf, dt, layout, pattern)


# ------------------------------------------------------------------ structure


class _Layout:
    """Index arrays of one case (numpy, host), as StsJacobian takes them."""


def _mesh(Lx, Ly):
    i = np.arange(Lx * Ly)
    ix, iy = i % Lx, i // Lx
    cand = np.stack([i - Lx, i - 1, i, i + 1, i + Lx], 1)
    ok = np.stack([iy > 0, ix > 0, ix >= 0, ix < Lx - 1, iy < Ly - 1], 1)
    ptr = np.concatenate([[0], np.cumsum(ok.sum(1))])
    return ptr.astype(np.int32), cand[ok].astype(np.int32)


def _csr(mask):
    ptr = np.concatenate([[0], np.cumsum(mask.sum(1))])
    return ptr.astype(np.int32), np.nonzero(mask)[1].astype(np.int32)


def _layout(c):
    L, N = _Layout(), c["N"]
    L.N, L.b, L.nc = N, N + 3, c["Lx"] * c["Ly"]
    b = L.b
    L.block_indptr, L.block_indices = _mesh(c["Lx"], c["Ly"])
    if c["pattern"] == "random":
        r = np.random.default_rng(1000 + N)
        d, o = r.random((b, b)) < 0.15, r.random((b, b)) < 0.15
        d |= np.eye(b, dtype=bool)
        o[np.arange(b), r.integers(0, b, b)] = True
    else:
        p, q = np.mgrid[0:b, 0:b]
        flow = (p >= N) | (q >= N)
        d = flow | (abs(p - q) <= c["w"])
        o = d if c["pattern"] == "shared" else flow | (p == q)
    L.d_indptr, L.d_indices = _csr(d)
    L.o_indptr, L.o_indices = _csr(o)
    L.rows = np.repeat(np.arange(L.nc), np.diff(L.block_indptr))
    L.diag = L.rows == L.block_indices
    deg = np.diff(L.block_indptr) - 1
    counts = np.where(L.diag, c["rd"] + c["ppf"] * deg[L.rows], c["ro"])
    L.pairs = np.concatenate([[0], np.cumsum(counts)])
    L.r_diag, L.r_off = int(counts[L.diag].max()), c["ro"]
    L.pair_indptr = L.pairs.astype(np.int32) if c["ppf"] else None
    L.soff = np.concatenate([[0], np.cumsum(np.where(L.diag, len(L.d_indices), len(L.o_indices)))])
    L.nnz_S, L.n_pairs, L.n = int(L.soff[-1]), int(L.pairs[-1]), L.nc * b
    return L


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _values(c, L, seed):
    """S, U, V, a right-hand side and loss weights on the GPU: diagonal entries 1/dt + |z|,
    other S entries 0.1 z, pairs z / sqrt(b)."""
    g = _gen(seed)
    randn = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=F64)  # noqa: E731
    S = randn(L.nnz_S).mul_(0.1)
    on = np.flatnonzero(np.repeat(np.arange(L.b), np.diff(L.d_indptr)) == L.d_indices)
    at = torch.from_numpy(L.soff[:-1][L.diag]).cuda()[:, None] + torch.from_numpy(on).cuda()[None, :]
    S[at] = randn(L.nc, L.b).abs_() + 1.0 / c["dt"]
    U = randn(L.n_pairs, L.b).div_(math.sqrt(L.b))
    V = randn(L.n_pairs, L.b).div_(math.sqrt(L.b))
    return S, U, V, randn(L.n), torch.rand(L.n, generator=g, device="cuda", dtype=F64) + 0.5


class _Flow:
    """Constants and states of one flow case, with the fields StsFlow takes."""


def _flow(c, seed):
    f, N, Lx, Ly = _Flow(), c["N"], c["Lx"], c["Ly"]
    r = np.random.default_rng(seed)
    f.Lx, f.Ly, f.N, f.w, f.dt, f.A, f.theta = Lx, Ly, N, c["w"], c["dt"], 1.0, 2.0
    f.r, f.cv = r.uniform(0.25, 0.45, N), r.uniform(0.6, 1.2, N)
    f.e0 = 0.05 * np.arange(N) + r.uniform(0.0, 0.02, N)
    f.beta, f.ws, f.K = r.uniform(0.0, 1.0, N), 0.1 * r.standard_normal(N), r.uniform(0.0, 0.5, (N, 2 * f.w + 1))
    g, nc = _gen(seed), Lx * Ly
    noise = lambda *s: 1.0 + 0.05 * torch.randn(*s, generator=g, device="cuda", dtype=F64)  # noqa: E731
    i = torch.arange(nc, device="cuda")
    x, y = ((i % Lx) + 0.5) / Lx, ((i // Lx) + 0.5) / Ly
    x, y = x.to(F64), y.to(F64)
    pop = torch.exp(-torch.outer(1.0 / (0.5 + 0.3 * x), torch.from_numpy(2.0 * f.e0).cuda()))
    rho = 1.0 + 0.3 * torch.sin(math.pi * x) * torch.cos(math.pi * y)
    Q = torch.empty(nc, N + 3, device="cuda", dtype=F64)
    Q[:, :N] = rho[:, None] * pop / pop.sum(1, keepdim=True) * noise(nc, N)
    Q[:, N] = 0.28 * (1.0 + 0.3 * torch.sin(2 * math.pi * y)) * noise(nc)
    Q[:, N + 1] = 0.112 * torch.cos(math.pi * x) * noise(nc)
    Q[:, N + 2] = (1.0 + 0.2 * torch.cos(2 * math.pi * x) * torch.sin(math.pi * y)) * noise(nc)
    f.Qn = Q * (1.0 + 0.01 * torch.randn(nc, N + 3, generator=g, device="cuda", dtype=F64))
    f.Q = Q
    return f


# ------------------------------------------------------------------ the passes


def _vec(c, L, x):
    """A cell-major vector in the case's layout."""
    return x if c["layout"] == "cell" else x.view(L.nc, L.b).t().contiguous().view(-1)


def prepare(case, seed):
    c, s = case, {"case": case}
    if c["kind"] in ("flow", "newton"):
        f = _flow(c, seed)
        s["flow"], s["Q"], s["Qn"] = StsFlow(f), f.Q, f.Qn
        if c["kind"] == "newton":
            s["jac"] = s["flow"].jacobian_handle()
        return s
    L = _layout(c)
    S, U, V, x, W = _values(c, L, seed)
    keep = c["kind"] in ("refresh", "adjoint")
    first = [0.5 * a for a in (S, U, V)] if keep else (S, U, V)     # those calls bring the values in themselves
    s["jac"] = StsJacobian(L, *first, layout=c["layout"], mixed=c["kind"] == "mixed",
                           transpose=c["kind"] in ("matvec", "general", "apply", "adjoint"), n_levels=c["N"])
    del first
    s["x"] = _vec(c, L, x)
    if keep:
        s["S"], s["U"], s["V"] = S, U, V
    if c["kind"] == "adjoint":
        s["W"] = W
    if c["kind"] in ("general", "apply", "gmres", "mixed"):
        s["jac"].bjacobi_setup()
    return s


def run(state):
    kind, x, jac = state["case"]["kind"], state.get("x"), state.get("jac")
    if kind == "matvec":
        return {"y": jac.matvec(x), "yt": jac.matvec(x, trans=True)}
    if kind == "apply":
        return {"z": jac.bjacobi_apply(x), "zt": jac.bjacobi_apply(x, trans=True)}
    if kind == "general":
        return {"y": jac.matvec(x), "yt": jac.matvec(x, trans=True),
                "z": jac.bjacobi_apply(x), "zt": jac.bjacobi_apply(x, trans=True)}
    if kind == "refresh":
        jac.update_values(state["S"], state["U"], state["V"])
        jac.bjacobi_setup()
        return {"y": jac.matvec(x), "z": jac.bjacobi_apply(x)}
    if kind in ("gmres", "mixed"):
        return {"x": jac.gmres(x, rtol=1e-10, mixed=kind == "mixed")[0]}
    if kind == "adjoint":
        leaves = [a.detach().requires_grad_() for a in (x, state["S"], state["U"], state["V"])]
        sol = ImplicitSolve.apply(*leaves, jac)
        grads = torch.autograd.grad(0.5 * (state["W"] * sol).square().sum(), leaves)
        return {"x": sol.detach(), "gb": grads[0], "gS": grads[1], "gU": grads[2], "gV": grads[3]}
    if kind == "flow":
        S, U, V = state["flow"].jacobian(state["Q"])
        return {"S": S, "U": U, "V": V, "R": state["flow"].residual(state["Q"], state["Qn"])}
    Q = state["Q"].clone()
    state["flow"].newton(jac, Q, state["Qn"])
    return {"Q": Q}


# ------------------------------------------------------------------ what a pass cannot do without


def work(case):
    c = case
    L = _layout(dict(c, rd=1, ro=2, ppf=2) if c["kind"] in ("flow", "newton") else c)
    n, b = L.n, L.b
    pd, po = int((L.pairs[1:] - L.pairs[:-1])[L.diag].sum()), int((L.pairs[1:] - L.pairs[:-1])[~L.diag].sum())
    vals = L.nnz_S + 2 * L.n_pairs * b                       # values of the Jacobian
    dvals = L.nc * len(L.d_indices) + 2 * pd * b             # values of its diagonal blocks
    r2 = int(((L.pairs[1:] - L.pairs[:-1])[L.diag] ** 2).sum())
    mv_b, mv_f = 8 * (vals + 2 * n), 2 * vals                # one product: values and x read, y written
    ap_b, ap_f = 8 * (dvals + r2 + 2 * n), 2 * (dvals + r2)  # one apply: factors (no larger than the pattern), W, V, C^-1
    # factorisation: every L entry of column k updates the rest of row k's pattern (band and flow columns)
    w = min(c["w"], c["N"])
    st_f = 2 * L.nc * c["N"] * (w + 3) * (w + 4) + 2 * 2 * dvals + 2 * r2 * b
    st_b = 8 * (2 * dvals + r2)
    k = c["kind"]
    if k == "matvec":
        return {"bytes": 2 * mv_b, "flops": 2 * mv_f}
    if k == "apply":
        return {"bytes": 2 * ap_b, "flops": 2 * ap_f}
    if k == "general":
        return {"bytes": 2 * (mv_b + ap_b), "flops": 2 * (mv_f + ap_f)}
    if k == "refresh":
        return {"bytes": 8 * 2 * vals + st_b + mv_b + ap_b, "flops": st_f + mv_f + ap_f}
    its = 4 if c["dt"] < 2e-3 else 8                          # Arnoldi steps, about
    orth_b, orth_f = 8 * n * its * (its + 1) * 1.5, 8 * n * its * (its + 1) / 2
    solve_b, solve_f = (its + 1) * (mv_b + ap_b) + orth_b, (its + 1) * (mv_f + ap_f) + orth_f
    if k == "gmres":
        return {"bytes": solve_b, "flops": solve_f}
    if k == "mixed":
        return {"bytes": its * (mv_b + ap_b) / 2 + 2 * mv_b + orth_b, "flops": solve_f}
    if k == "adjoint":
        return {"bytes": 8 * 2 * vals + st_b + 2 * solve_b + 8 * (vals + 2 * n), "flops": st_f + 2 * solve_f + 2 * vals}
    if k == "flow":
        return {"bytes": 8 * (vals + 4 * n), "flops": 4 * vals}
    steps, its = 6, 30
    orth_b, orth_f = 8 * n * its * (its + 1) * 1.5, 8 * n * its * (its + 1) / 2
    return {"bytes": steps * (8 * 3 * vals + st_b + its * (mv_b + ap_b) + orth_b),
            "flops": steps * (st_f + its * (mv_f + ap_f) + orth_f)}


# ------------------------------------------------------------------ the same in plain torch, 64 bits


class _Plain:
    """J as its arrays, with products and block-Jacobi by torch alone (cell-major vectors [nc, b])."""

    def __init__(self, L, S, U, V):
        cu = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int64)).cuda()  # noqa: E731
        self.L, self.S, self.U, self.V = L, S, U, V
        self.kinds = []
        for on, ptr, idx in ((L.diag, L.d_indptr, L.d_indices), (~L.diag, L.o_indptr, L.o_indices)):
            p = np.repeat(np.arange(L.b), np.diff(ptr))
            self.kinds.append([cu(a) for a in (L.soff[:-1][on], L.rows[on], L.block_indices[on], p, idx)])
        blk = np.repeat(np.arange(len(L.rows)), np.diff(L.pairs))
        self.prow, self.pcol, self.pdiag = cu(L.rows[blk]), cu(L.block_indices[blk]), cu(np.flatnonzero(L.diag[blk]))
        self.lu = None

    def mv(self, x, trans=False):
        y = torch.zeros_like(x)
        for off, r, col, p, q in self.kinds:
            i, j, pi, pj = (col, r, q, p) if trans else (r, col, p, q)
            step = max(1, (1 << 27) // max(1, len(p)))
            for a in range(0, len(off), step):
                sl = slice(a, a + step)
                v = self.S[off[sl, None] + torch.arange(len(p), device=x.device)] * x[j[sl]][:, pj]
                y.index_add_(0, i[sl], torch.zeros(len(v), x.shape[1], device=x.device, dtype=F64).index_add_(1, pi, v))
        (i, j, u, v) = (self.pcol, self.prow, self.V, self.U) if trans else (self.prow, self.pcol, self.U, self.V)
        return y.index_add_(0, i, u * (v * x[j]).sum(1, keepdim=True))

    def blocks(self):
        nc, b = self.L.nc, self.L.b
        off, _, _, p, q = self.kinds[0]
        A = torch.zeros(nc, b, b, device="cuda", dtype=F64)
        A[:, p, q] = self.S[off[:, None] + torch.arange(len(p), device="cuda")]
        k = self.pdiag
        for a in range(0, len(k), 1 << 14):
            s = k[a:a + (1 << 14)]
            A.index_add_(0, self.prow[s], self.U[s][:, :, None] * self.V[s][:, None, :])
        return A

    def bj(self, x, trans=False):
        if self.lu is None:
            self.lu = torch.linalg.lu_factor(self.blocks())
        return torch.linalg.lu_solve(*self.lu, x[:, :, None], adjoint=trans)[:, :, 0]

    def solve(self, b, trans=False, rtol=1e-15, m=40, most=400):
        """GMRES(m) preconditioned from the right, refined until the residual no longer falls."""
        x, best, its = torch.zeros_like(b), math.inf, 0
        while its < most:
            r = b - self.mv(x, trans)
            beta = float(r.norm())
            if beta <= rtol * float(b.norm()) or beta > 0.5 * best:
                break
            best = beta
            vs, zs, H = [r / beta], [], np.zeros((m + 1, m))
            for j in range(m):
                zs.append(self.bj(vs[j], trans))
                u = self.mv(zs[j], trans)
                for _ in range(2):
                    for i in range(j + 1):
                        h = float((vs[i] * u).sum())
                        H[i, j] += h
                        u = u - h * vs[i]
                H[j + 1, j] = float(u.norm())
                e = np.zeros(j + 2)
                e[0] = beta
                y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
                its += 1
                res = np.linalg.norm(H[:j + 2, :j + 1] @ y - e)
                if res <= 1e-9 * beta or res <= rtol * float(b.norm()):
                    break
                vs.append(u / H[j + 1, j])
            for a, z in zip(y, zs):
                x = x + float(a) * z
        return x


def _plain_flow(c, f, Q):
    """Residual terms and the r1-sparse Jacobian of the flow model by torch alone.
    Returns (layout, S, U, V, residual function)."""
    L = _layout(dict(c, rd=1, ro=2, ppf=2))
    N, b, nc, Lx, dt = L.N, L.b, L.nc, c["Lx"], f.dt
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    rk, cv, e0, beta, ws, K = (cu(a) for a in (f.r, f.cv, f.e0, f.beta, f.ws, f.K))
    off = ~L.diag
    fi, fj = cu(L.rows[off].astype(np.int64)), cu(L.block_indices[off].astype(np.int64))
    d = (fj - fi)
    vert = torch.ones_like(d, dtype=torch.bool) if Lx == 1 else d.abs() != 1
    if Lx > 1:
        vert = d.abs() == Lx
    sgn = torch.sign(d).to(F64)
    nx, ny = torch.where(vert, torch.zeros_like(sgn), sgn), torch.where(vert, sgn, torch.zeros_like(sgn))

    def mix(q):
        s = q[:, :N]
        m = dict(q=q, rho=s.sum(1), R=s @ rk, C=s @ cv, E=s @ e0, u=q[:, N], v=q[:, N + 1], T=q[:, N + 2])
        m["ke"] = 0.5 * (m["u"] ** 2 + m["v"] ** 2)
        m["p"] = m["R"] * m["T"]
        m["e"] = m["E"] + m["C"] * m["T"] + m["rho"] * m["ke"]
        m["g"] = (m["C"] + m["R"]) * m["R"] / (m["rho"] * m["C"])
        m["a"] = torch.sqrt(m["g"] * m["T"])
        return m

    def cons(m):
        return torch.cat([m["q"][:, :N], torch.stack([m["rho"] * m["u"], m["rho"] * m["v"], m["e"]], 1)], 1)

    def flux(m, nx, ny):
        un = nx * m["u"] + ny * m["v"]
        return torch.cat([m["q"][:, :N] * un[:, None],
                          torch.stack([m["rho"] * m["u"] * un + m["p"] * nx, m["rho"] * m["v"] * un + m["p"] * ny,
                                       (m["e"] + m["p"]) * un], 1)], 1)

    def at(m, i):
        return {k: v[i] for k, v in m.items()}

    def speeds(l, r):
        ul, ur = nx * l["u"] + ny * l["v"], nx * r["u"] + ny * r["v"]
        z = torch.zeros_like(ul)
        sL, iL = torch.stack([z, ul - l["a"], ur - r["a"]]).min(0)
        sR, iR = torch.stack([z, ul + l["a"], ur + r["a"]]).max(0)
        return sL, sR, iL, iR

    def source(q, T):
        om = -(sum(torch.nn.functional.pad(q[:, :N], (f.w, f.w))[:, k:k + N] * K[:, k] for k in range(2 * f.w + 1)))
        return om + ws * (f.A * torch.exp(-f.theta / T) * (q[:, :N] @ beta))[:, None]

    def residual(Q, Qn):
        m = mix(Q)
        l, r = at(m, fi), at(m, fj)
        sL, sR, _, _ = (a[:, None] for a in speeds(l, r))
        F = (sR * flux(l, nx, ny) - sL * flux(r, nx, ny) + sL * sR * (cons(r) - cons(l))) / (sR - sL)
        R = torch.zeros_like(Q).index_add_(0, fi, F)
        R[:, :N] -= source(Q, m["T"])
        return cons(m) - cons(mix(Qn)) + dt * R

    def H(m):
        n = len(m["u"])
        A = torch.zeros(n, b, b, device="cuda", dtype=F64)
        A[:, range(N), range(N)] = 1.0
        A[:, N, :N], A[:, N + 1, :N] = m["u"][:, None], m["v"][:, None]
        A[:, N, N] = A[:, N + 1, N + 1] = m["rho"]
        A[:, N + 2, :N] = e0 + cv * m["T"][:, None] + m["ke"][:, None]
        A[:, N + 2, N], A[:, N + 2, N + 1], A[:, N + 2, N + 2] = m["rho"] * m["u"], m["rho"] * m["v"], m["C"]
        return A

    def An(m, nx, ny):
        n, un = len(m["u"]), nx * m["u"] + ny * m["v"]
        A = torch.zeros(n, b, b, device="cuda", dtype=F64)
        A[:, range(N), range(N)] = un[:, None]
        A[:, :N, N], A[:, :N, N + 1] = m["q"][:, :N] * nx[:, None], m["q"][:, :N] * ny[:, None]
        rT = rk * m["T"][:, None]
        A[:, N, :N] = (m["u"] * un)[:, None] + rT * nx[:, None]
        A[:, N + 1, :N] = (m["v"] * un)[:, None] + rT * ny[:, None]
        A[:, N + 2, :N] = (e0 + cv * m["T"][:, None] + m["ke"][:, None] + rT) * un[:, None]
        A[:, N, N], A[:, N, N + 1], A[:, N, N + 2] = m["rho"] * (un + m["u"] * nx), m["rho"] * m["u"] * ny, m["R"] * nx
        A[:, N + 1, N], A[:, N + 1, N + 1], A[:, N + 1, N + 2] = (m["rho"] * m["v"] * nx, m["rho"] * (un + m["v"] * ny),
                                                                  m["R"] * ny)
        h = m["e"] + m["p"]
        A[:, N + 2, N], A[:, N + 2, N + 1] = m["rho"] * m["u"] * un + h * nx, m["rho"] * m["v"] * un + h * ny
        A[:, N + 2, N + 2] = (m["C"] + m["R"]) * un
        return A

    def grad_a(m):
        dn = (cv + rk) * m["R"][:, None] + (m["C"] + m["R"])[:, None] * rk
        dd = m["C"][:, None] + m["rho"][:, None] * cv
        G = torch.zeros(len(m["u"]), b, device="cuda", dtype=F64)
        G[:, :N] = (m["T"] / (2 * m["a"] * m["rho"] * m["C"]))[:, None] * (dn - m["g"][:, None] * dd)
        G[:, N + 2] = m["a"] / (2 * m["T"])
        return G

    m = mix(Q)
    S = torch.zeros(L.nnz_S, device="cuda", dtype=F64)
    U, V = (torch.zeros(L.n_pairs, b, device="cuda", dtype=F64) for _ in range(2))
    l, r = at(m, fi), at(m, fj)
    sL, sR, iL, iR = speeds(l, r)
    den = sR - sL
    af, cf = 0.5 * (sL + sR) / den, sL * sR / den
    p_o, q_o = cu(np.repeat(np.arange(b), np.diff(L.o_indptr)).astype(np.int64)), cu(L.o_indices.astype(np.int64))
    p_d, q_d = cu(np.repeat(np.arange(b), np.diff(L.d_indptr)).astype(np.int64)), cu(L.d_indices.astype(np.int64))
    so, sd = cu(L.soff[:-1][off]), cu(L.soff[:-1][L.diag])
    for a in range(0, len(fi), 1 << 13):
        k = slice(a, a + (1 << 13))
        rr = {x: v[k] for x, v in r.items()}
        B = dt * ((0.5 - af[k])[:, None, None] * An(rr, nx[k], ny[k]) + cf[k][:, None, None] * H(rr))
        S[so[k, None] + torch.arange(len(p_o), device="cuda")] = B[:, p_o, q_o]
    w = 0.5 + af
    acc = torch.zeros(nc, 3, device="cuda", dtype=F64).index_add_(0, fi, torch.stack([cf, w * nx, w * ny], 1))
    for a in range(0, nc, 1 << 13):
        k = slice(a, a + (1 << 13))
        mm = {x: v[k] for x, v in m.items()}
        h = H(mm)
        B = h + dt * (An(mm, acc[k, 1], acc[k, 2]) - acc[k, 0][:, None, None] * h)
        for j in range(2 * f.w + 1):
            lo, hi = max(0, f.w - j), min(N, N + f.w - j)
            if lo < hi:
                i = torch.arange(lo, hi, device="cuda")
                B[:, i, i + j - f.w] += dt * K[lo:hi, j]
        S[sd[k, None] + torch.arange(len(p_d), device="cuda")] = B[:, p_d, q_d]
    # pairs: the face's place among its row's neighbours picks its pair of the diagonal block
    ptr = L.block_indptr.astype(np.int64)
    order = np.arange(len(L.rows)) - ptr[L.rows]
    dpos = order[L.diag]
    kd = np.flatnonzero(L.diag)
    place = (order - (order > dpos[L.rows]))[off]
    pd, po = cu(L.pairs[kd[L.rows[off]]] + 1 + 2 * place), cu(L.pairs[:-1][off])
    u1, u2 = dt * (flux(l, nx, ny) - flux(r, nx, ny)), dt * (cons(r) - cons(l))
    gn = torch.zeros(len(fi), b, device="cuda", dtype=F64)
    gn[:, N], gn[:, N + 1] = nx, ny
    gl, gr = grad_a(l), grad_a(r)
    on = lambda i, k: (i == k).to(F64)[:, None]  # noqa: E731
    LL, LR, RL, RR = on(iL, 1) * (gn - gl), on(iL, 2) * (gn - gr), on(iR, 1) * (gn + gl), on(iR, 2) * (gn + gr)
    sL, sR, i2 = sL[:, None], sR[:, None], (1.0 / den ** 2)[:, None]
    U[pd] = U[po] = u1
    U[pd + 1] = U[po + 1] = u2
    V[pd], V[po] = (sR * LL - sL * RL) * i2, (sR * LR - sL * RR) * i2
    V[pd + 1], V[po + 1] = (sR ** 2 * LL - sL ** 2 * RL) * i2, (sR ** 2 * LR - sL ** 2 * RR) * i2
    ps = cu(L.pairs[kd])
    U[ps, :N] = -dt * ws
    kap = f.A * torch.exp(-f.theta / m["T"])
    V[ps, :N] = kap[:, None] * beta
    V[ps, N + 2] = kap * f.theta / m["T"] ** 2 * (Q[:, :N] @ beta)
    return L, S, U, V, residual


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("flow", "newton"):
        f = _flow(c, seed)
        L, S, U, V, residual = _plain_flow(c, f, f.Q)
        if k == "flow":
            return {"S": S, "U": U, "V": V, "R": residual(f.Q, f.Qn)}
        Q, R = f.Q.clone(), residual(f.Q, f.Qn)
        for _ in range(30):
            L, S, U, V, residual = _plain_flow(c, f, Q)
            d = _Plain(L, S, U, V).solve(-R, rtol=1e-11, m=60)
            a = 1.0
            while a > 1e-3 and not float(residual(Q + a * d, f.Qn).norm()) < float(R.norm()):
                a *= 0.5
            if a <= 1e-3:
                break
            Q = Q + a * d
            R = residual(Q, f.Qn)
        return {"Q": Q}
    L = _layout(c)
    S, U, V, x, W = _values(c, L, seed)
    J = _Plain(L, S, U, V)
    x = x.view(L.nc, L.b)
    out = lambda y: _vec(c, L, y.reshape(-1))  # noqa: E731
    got = {}
    if k in ("matvec", "general", "refresh"):
        got["y"] = out(J.mv(x))
    if k in ("matvec", "general"):
        got["yt"] = out(J.mv(x, True))
    if k in ("apply", "general", "refresh"):
        got["z"] = out(J.bj(x))
    if k in ("apply", "general"):
        got["zt"] = out(J.bj(x, True))
    if k in ("gmres", "mixed", "adjoint"):
        sol = J.solve(x)
        got["x"] = out(sol)
    if k == "adjoint":
        W = W.view(L.nc, L.b)
        lam = J.solve(W * W * sol, True)
        got["gb"] = out(lam)
        gS = torch.empty_like(S)
        for off, r, col, p, q in J.kinds:
            for a in range(0, len(off), 1 << 14):
                t = slice(a, a + (1 << 14))
                gS[off[t, None] + torch.arange(len(p), device="cuda")] = -lam[r[t]][:, p] * sol[col[t]][:, q]
        got["gS"] = gS
        got["gU"] = -(V * sol[J.pcol]).sum(1, keepdim=True) * lam[J.prow]
        got["gV"] = -(U * lam[J.prow]).sum(1, keepdim=True) * sol[J.pcol]
    return got
