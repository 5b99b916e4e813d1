"""Performance cases of the blocked AMG reuse phase.

Every case is work that a program using this package has it do through its
public binding: assembling an operator from a blocked COO stream, products
with one and with several vectors, the Galerkin recompute on a cached plan,
whole reuse steps (re-assembly, hierarchy update, CG solve), several
right-hand sides at once and a batch of problems.  The inputs are 3D linear
elasticity on the unit cube, Q1 or Q2 hexahedra, clamped at x = 0, with a
per-element stiffness perturbation drawn from the seed.
"""
import math

import numpy as np
import torch

from paper_2606_24748_gb300 import bamg as B

RTOL, MAXIT = 1e-8, 200
NU = 0.3


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------- problem

def _shape_1d(p, t):
    if p == 1:
        return np.array([1.0 - t, t]), np.array([-1.0, 1.0])
    return (np.array([(1.0 - t) * (1.0 - 2.0 * t), 4.0 * t * (1.0 - t), t * (2.0 * t - 1.0)]),
            np.array([4.0 * t - 3.0, 4.0 - 8.0 * t, 4.0 * t - 1.0]))


def _reference_blocks(nu, p):
    """Stiffness of the unit cube (E = 1) as node-pair blocks (nn * nn, 3, 3)."""
    lam, mu = nu / ((1.0 + nu) * (1.0 - 2.0 * nu)), 1.0 / (2.0 * (1.0 + nu))
    D = np.zeros((6, 6))
    D[:3, :3] = lam
    D[range(3), range(3)] += 2.0 * mu
    D[range(3, 6), range(3, 6)] = mu
    pts, wts = np.polynomial.legendre.leggauss(p + 1)
    pts, wts = 0.5 * (pts + 1.0), 0.5 * wts
    q, nn = p + 1, (p + 1) ** 3
    ax, ay, az = np.arange(nn) % q, (np.arange(nn) // q) % q, np.arange(nn) // (q * q)
    K = np.zeros((3 * nn, 3 * nn))
    for x, wx in zip(pts, wts):
        for y, wy in zip(pts, wts):
            for z, wz in zip(pts, wts):
                (fx, dx), (fy, dy), (fz, dz) = _shape_1d(p, x), _shape_1d(p, y), _shape_1d(p, z)
                g = np.stack([dx[ax] * fy[ay] * fz[az], fx[ax] * dy[ay] * fz[az], fx[ax] * fy[ay] * dz[az]], 1)
                S = np.zeros((6, nn, 3))
                S[0, :, 0], S[1, :, 1], S[2, :, 2] = g[:, 0], g[:, 1], g[:, 2]
                S[3, :, 0], S[3, :, 1] = g[:, 1], g[:, 0]
                S[4, :, 1], S[4, :, 2] = g[:, 2], g[:, 1]
                S[5, :, 0], S[5, :, 2] = g[:, 2], g[:, 0]
                S = S.reshape(6, 3 * nn)
                K += (wx * wy * wz) * (S.T @ D @ S)
    return K.reshape(nn, 3, nn, 3).transpose(0, 2, 1, 3).reshape(nn * nn, 3, 3).copy()


class _Problem:
    """Mesh, COO coordinates and the seeded COO values on the device."""

    def __init__(self, ne, p, nu):
        self.ne, self.p, self.nu, self.m = ne, p, nu, p * ne + 1
        self.n, self.n_el, self.nn = self.m ** 3, ne ** 3, (p + 1) ** 3
        dev, m = _device(), self.m
        e = torch.arange(self.n_el, device=dev)
        base = p * (e % ne + m * ((e // ne) % ne) + m * m * (e // (ne * ne)))
        a = torch.arange(self.nn, device=dev)
        q = p + 1
        self.conn = base[:, None] + (a % q + m * ((a // q) % q) + m * m * (a // (q * q)))[None, :]
        node = torch.arange(self.n, device=dev)
        self.clamped = node % m == 0
        fixed = node[self.clamped]
        shape = (self.n_el, self.nn, self.nn)
        self.bi = torch.cat([self.conn[:, :, None].expand(shape).reshape(-1), fixed]).to(torch.int32)
        self.bj = torch.cat([self.conn[:, None, :].expand(shape).reshape(-1), fixed]).to(torch.int32)
        self.kref = torch.as_tensor(_reference_blocks(nu, p), device=dev)

    def values(self, seed=None):
        """COO values: scale_e * K_ref per element, zero where a clamped node
        is touched, identity blocks on the clamped nodes.  A seed perturbs the
        element stiffness by up to 1%."""
        dev = self.conn.device
        scale = torch.full((self.n_el,), 1.0 / self.ne, dtype=torch.float64, device=dev)
        if seed is not None:
            g = torch.Generator(device="cpu").manual_seed(int(seed))
            d = torch.rand(self.n_el, generator=g, dtype=torch.float64) * 0.02 - 0.01
            scale = scale * (1.0 + d.to(dev))
        nb = self.nn * self.nn
        v = torch.empty((self.bi.numel(), 3, 3), dtype=torch.float64, device=dev)
        el = v[: nb * self.n_el].view(self.n_el, nb, 3, 3)
        torch.mul(scale[:, None, None, None], self.kref[None], out=el)
        c = self.clamped[self.conn]
        el.masked_fill_((c[:, :, None] | c[:, None, :]).reshape(self.n_el, nb)[:, :, None, None], 0.0)
        v[nb * self.n_el:] = torch.eye(3, dtype=torch.float64, device=dev)
        return v

    def coords(self):
        k = np.arange(self.n, dtype=np.int64)
        return np.stack([k % self.m, (k // self.m) % self.m, k // (self.m * self.m)], 1).astype(np.float64) / (self.m - 1)

    def dirichlet(self):
        return (np.arange(self.n, dtype=np.int64) % self.m == 0).astype(np.uint8)

    def load(self):
        """Consistent load of a unit body force in -z."""
        w = torch.ones(1, dtype=torch.float64)
        w1 = torch.tensor([0.5, 0.5] if self.p == 1 else [1 / 6, 2 / 3, 1 / 6], dtype=torch.float64)
        for _ in range(3):
            w = (w[:, None] * w1[None, :]).reshape(-1)
        f = torch.zeros(self.n, dtype=torch.float64, device=self.conn.device)
        f.index_add_(0, self.conn.reshape(-1), (-(1.0 / self.ne) ** 3 * w).to(f.device).repeat(self.n_el))
        b = torch.zeros((self.n, 3), dtype=torch.float64, device=f.device)
        b[:, 2] = f
        b[self.clamped] = 0.0
        return b.reshape(-1)

    def gaussian(self, seed, k=1, dtype=torch.float64):
        """k standard normal vectors, vector-minor (n_dofs, k), zero on clamped dofs."""
        g = torch.Generator(device="cpu").manual_seed(int(seed) + 1)
        x = torch.randn((self.n, 3, k), generator=g, dtype=torch.float64).to(self.conn.device)
        x[self.clamped] = 0.0
        return x.reshape(3 * self.n, k).to(dtype)

    def blocks(self, v):
        """(row, column, value) of the assembled blocks, sorted by row then column."""
        key, inv = torch.unique(self.bi.long() * self.n + self.bj.long(), return_inverse=True)
        out = torch.zeros((key.numel(), 9), dtype=torch.float64, device=v.device)
        out.index_add_(0, inv, v.reshape(-1, 9))
        return key // self.n, key % self.n, out.view(-1, 3, 3)

    def prolongator(self, v):
        """A smoothed rigid-body prolongator over 3 x 3 x 3 node aggregates as
        unique blocks (row, aggregate, value 3 x 6) of the operator with COO values v."""
        dev, m = v.device, self.m
        na = max(1, m // 3)
        k = torch.arange(self.n, device=dev)
        ijk = torch.stack([k % m, (k // m) % m, k // (m * m)], 1)
        a3 = torch.clamp(ijk // 3, max=na - 1)
        agg = a3[:, 0] + na * (a3[:, 1] + na * a3[:, 2])
        nc = na ** 3
        x = ijk.double()
        cen = torch.zeros((nc, 3), dtype=torch.float64, device=dev).index_add_(0, agg, x)
        cnt = torch.bincount(agg, minlength=nc).double()
        x = (x - cen[agg] / cnt[agg][:, None]) * 0.7
        T = torch.zeros((self.n, 3, 6), dtype=torch.float64, device=dev)
        T[:, range(3), range(3)] = 1.0
        T[:, 0, 3], T[:, 1, 3] = -x[:, 1], x[:, 0]
        T[:, 1, 4], T[:, 2, 4] = -x[:, 2], x[:, 1]
        T[:, 2, 5], T[:, 0, 5] = -x[:, 0], x[:, 2]
        T /= cnt[agg].sqrt()[:, None, None]
        T[self.clamped] = 0.0
        D = torch.zeros((self.n, 3), dtype=torch.float64, device=dev)
        i, j = self.bi.long(), self.bj.long()
        on = i == j
        D.index_add_(0, i[on], torch.diagonal(v[on], dim1=1, dim2=2))
        key, inv = torch.unique(i * nc + agg[j], return_inverse=True)
        P = torch.zeros((key.numel(), 3, 6), dtype=torch.float64, device=dev)
        for s in range(0, i.numel(), 1 << 21):
            e = slice(s, s + (1 << 21))
            P.index_add_(0, inv[e], (-0.5 / D[i[e]])[:, :, None] * torch.bmm(v[e], T[j[e]]))
        own = torch.searchsorted(key, k * nc + agg)
        P[own] += T
        return key // nc, key % nc, P, nc


# --------------------------------------------------------------------- cases

def listed():
    return [
        # operator assembly of one nonlinear or time step, 64^3 Q1 elements
        {"name": "coo_q1_64", "kind": "coo", "ne": 64, "order": 1},
        # one operator application inside a caller's own Krylov method
        {"name": "spmv_fp64_q1_64", "kind": "spmv", "ne": 64, "order": 1, "prec": 64},
        # the same in single precision on quadratic elements (rows of 75 to 125 blocks), odd node count
        {"name": "spmv_fp32_q2_21", "kind": "spmv", "ne": 21, "order": 2, "prec": 32},
        # one operator applied to 16 vectors (block methods, modal analysis), single precision
        {"name": "spmm16_fp32_q1_48", "kind": "spmm", "ne": 48, "order": 1, "prec": 32, "k": 16},
        # new operator values and the Galerkin recompute on the cached plan
        {"name": "ptap_fp64_q1_64", "kind": "ptap", "ne": 64, "order": 1, "prec": 64},
        # the mixed form's single-precision recompute, ragged aggregates
        {"name": "ptap_fp32_q1_47", "kind": "ptap", "ne": 47, "order": 1, "prec": 32},
        # the smallest whole step: latency and launches
        {"name": "step_fp64_q1_12", "kind": "step", "ne": 12, "order": 1, "prec": 64, "mis": False},
        # the ordinary whole step: re-assembly, hierarchy update, CG to 1e-8
        {"name": "step_fp64_q1_64", "kind": "step", "ne": 64, "order": 1, "prec": 64, "mis": False},
        # the mixed-precision whole step, odd size
        {"name": "step_mixed_q1_51", "kind": "step", "ne": 51, "order": 1, "prec": 32, "mis": False},
        # the whole step on a hierarchy built from the strength graph (irregular, denser coarse operators)
        {"name": "step_fp64_mis_q1_24", "kind": "step", "ne": 24, "order": 1, "prec": 64, "mis": True},
        # 16 load cases solved together on one hierarchy
        {"name": "multi16_fp64_q1_32", "kind": "multi", "ne": 32, "order": 1, "prec": 64, "k": 16},
        # uneven independent problems solved by one launch
        {"name": "batch8_fp64_q1", "kind": "batch", "count": 8, "lo": 16, "hi": 28, "prec": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["coo", "spmv", "spmm", "ptap", "step", "step", "multi", "batch"])
    order = 2 if kind != "batch" and rng.random() < 0.25 else 1
    case = {"kind": kind, "prec": rng.choice([64, 32])}
    if kind == "batch":
        lo = rng.randint(8, 24)
        return {**case, "count": rng.randint(2, 8), "lo": lo, "hi": lo + rng.randint(1, 8)}
    hi = {"coo": 64, "spmv": 64, "spmm": 48, "ptap": 64, "step": 60, "multi": 32}[kind]
    # a quadratic mesh of ne elements has 8 times the nodes and 2.4 times the blocks per row
    case.update(ne=_log_int(rng, 8, hi) if order == 1 else _log_int(rng, 4, {"step": 16, "multi": 10}.get(kind, 24)), order=order)
    if kind == "spmm":
        case["k"] = rng.choice([2, 3, 4, 5, 8, 12, 16])
    if kind == "multi":
        case["k"] = rng.choice([2, 3, 5, 8, 16])
    if kind == "step":
        case["mis"] = order == 1 and 12 <= case["ne"] <= 24 and rng.random() < 0.5
    return case


class _State:
    """Handles and tensors of one case; destroyed with the object."""

    def __init__(self):
        self.undo = []

    def keep(self, handle, destroy):
        self.undo.append((handle, destroy))
        return handle

    def __del__(self):
        while self.undo:
            handle, destroy = self.undo.pop()
            destroy(handle)


def _operator(s, pr, v):
    s.ctx = s.keep(B.bamg_ctx_create(torch.cuda.current_stream()), B.bamg_ctx_destroy)
    s.A = s.keep(B.bamg_bsr_create(s.ctx, 3, 3, pr.n, pr.n), B.bamg_bsr_destroy)
    B.bamg_bsr_coo_preallocate(s.ctx, s.A, pr.bi, pr.bj)
    B.bamg_bsr_coo_set_values(s.ctx, s.A, v, 0)


def _hierarchy(s, pr, prec, mis=False):
    o = B.bamg_mg_opts_default()
    o.grid[0] = o.grid[1] = o.grid[2] = pr.m
    o.precision = B.BAMG_FP32 if prec == 32 else B.BAMG_FP64
    o.aggregation = B.BAMG_AGG_MIS if mis else B.BAMG_AGG_GEOMETRIC
    s.mg = s.keep(B.bamg_mg_setup(s.ctx, s.A, pr.coords(), pr.dirichlet(), o), B.bamg_mg_destroy)


def _batch_problems(case, seed):
    g = np.random.default_rng(int(seed) + 5)
    sizes = [case["lo"] + (7 * i) % (case["hi"] - case["lo"] + 1) for i in range(case["count"])]
    return [(ne, float(nu)) for ne, nu in zip(sizes, g.uniform(0.2, 0.45, len(sizes)))]


def prepare(case, seed):
    s = _State()
    s.kind, s.prec = case["kind"], B.BAMG_FP32 if case.get("prec") == 32 else B.BAMG_FP64
    if s.kind == "batch":
        s.ctx = s.keep(B.bamg_ctx_create(torch.cuda.current_stream()), B.bamg_ctx_destroy)
        s.parts = []
        for ne, nu in _batch_problems(case, seed):
            q, pr = _State(), _Problem(ne, 1, nu)
            _operator(q, pr, pr.values(seed))
            _hierarchy(q, pr, case["prec"])
            q.b = pr.load()
            q.x = torch.zeros_like(q.b)
            s.parts.append(q)
        s.bs, s.xs = [q.b for q in s.parts], [q.x for q in s.parts]
        s.bt = s.keep(B.bamg_batch_create(s.ctx, [q.mg for q in s.parts]), B.bamg_batch_destroy)
        B.bamg_batch_autotune(s.ctx, s.bt, s.bs, s.xs, RTOL, MAXIT)
        return s
    pr = _Problem(case["ne"], case["order"], NU)
    dt = torch.float32 if case.get("prec") == 32 else torch.float64
    if s.kind in ("step", "multi"):
        # the hierarchy is set up once; each step brings new values
        _operator(s, pr, pr.values())
        _hierarchy(s, pr, case["prec"], case.get("mis", False))
        s.v = pr.values(seed)
        if s.kind == "step":
            s.b = pr.load()
        else:
            s.k = case["k"]
            s.b = pr.gaussian(seed, s.k)
            B.bamg_bsr_coo_set_values(s.ctx, s.A, s.v, 0)
            B.bamg_mg_update(s.ctx, s.mg)
            del s.v
        s.x = torch.zeros_like(s.b)
        return s
    s.v = pr.values(seed)
    _operator(s, pr, s.v)
    if s.kind == "coo":
        s.out = torch.empty(B.bamg_bsr_info(s.A)["nnzb"] * 9, dtype=torch.float64, device="cuda")
    elif s.kind in ("spmv", "spmm"):
        s.k = case.get("k", 1)
        s.x = pr.gaussian(seed, s.k, dt).contiguous()
        s.y = torch.empty_like(s.x)
        if s.kind == "spmv":
            B.bamg_bsr_spmv(s.ctx, s.A, s.x, s.y, s.prec)
            B.bamg_bsr_autotune(s.ctx, s.A)
        del s.v
    elif s.kind == "ptap":
        B.bamg_bsr_set_symmetric(s.ctx, s.A, 1)
        pi, pj, pv, nc = pr.prolongator(s.v)
        s.P = s.keep(B.bamg_bsr_create(s.ctx, 3, 6, pr.n, nc), B.bamg_bsr_destroy)
        B.bamg_bsr_coo_preallocate(s.ctx, s.P, pi.to(torch.int32), pj.to(torch.int32))
        B.bamg_bsr_coo_set_values(s.ctx, s.P, pv, 0)
        plan, Ac = B.bamg_ptap_symbolic(s.ctx, s.A, s.P)
        s.Ac = s.keep(Ac, B.bamg_bsr_destroy)
        s.plan = s.keep(plan, B.bamg_ptap_destroy)
        if s.prec == B.BAMG_FP32:  # the recomputed operator holds FP32 values only: its product is what a program can read
            s.xc = _coarse_vector(nc, seed).float()
            s.out = torch.empty_like(s.xc)
        else:
            s.out = torch.empty(B.bamg_bsr_info(s.Ac)["nnzb"] * 36, dtype=torch.float64, device="cuda")
    return s


def _coarse_vector(nc, seed):
    g = torch.Generator(device="cpu").manual_seed(int(seed) + 3)
    return torch.randn(6 * nc, generator=g, dtype=torch.float64).to(_device())


def run(s):
    if s.kind == "coo":
        B.bamg_bsr_coo_set_values(s.ctx, s.A, s.v, 0)
        B.bamg_bsr_get_values(s.ctx, s.A, s.out)
        return s.out
    if s.kind == "spmv":
        B.bamg_bsr_spmv(s.ctx, s.A, s.x, s.y, s.prec)
        return s.y
    if s.kind == "spmm":
        B.bamg_bsr_spmm(s.ctx, s.A, s.x, s.y, s.k, s.prec)
        return s.y
    if s.kind == "ptap":
        B.bamg_bsr_coo_set_values(s.ctx, s.A, s.v, 0)
        B.bamg_ptap_numeric_prec(s.ctx, s.plan, s.A, s.P, s.Ac, s.prec)
        if s.prec == B.BAMG_FP32:
            B.bamg_bsr_spmv(s.ctx, s.Ac, s.xc, s.out, s.prec)
        else:
            B.bamg_bsr_get_values(s.ctx, s.Ac, s.out)
        return s.out
    if s.kind == "step":
        B.bamg_bsr_coo_set_values(s.ctx, s.A, s.v, 0)
        B.bamg_mg_update(s.ctx, s.mg)
        B.bamg_cg_solve(s.ctx, s.mg, s.b, s.x, RTOL, MAXIT)
        return s.x
    if s.kind == "multi":
        B.bamg_cg_solve_multi(s.ctx, s.mg, s.b, s.x, s.k, RTOL, MAXIT)
        return s.x
    B.bamg_batch_cg_solve(s.ctx, s.bt, s.bs, s.xs, RTOL, MAXIT)
    return s.xs


# ---------------------------------------------------------------------- work

def _sizes(ne, p):
    """(nodes, stored blocks, COO entries, prolongator blocks, coarse blocks)."""
    m = p * ne + 1
    if p == 1:
        nz1 = 3 * m - 2
    else:  # vertex nodes couple with 5 (3 at the ends), middle nodes with 3
        nz1 = 5 * (ne + 1) - 4 + 3 * ne
    na = max(1, m // 3)
    r = 1 if p == 1 else 2
    p1 = sum(min((min(i + r, m - 1)) // 3, na - 1) - min(max(i - r, 0) // 3, na - 1) + 1 for i in range(m))
    c1 = 3 * na - 2 if na > 1 else 1
    return m ** 3, nz1 ** 3, ne ** 3 * (p + 1) ** 6 + m * m, p1 ** 3, c1 ** 3


def _solve_work(ne, p, prec, k):
    """One PCG solve: what 20 iterations with a V(2,2) cycle cannot do without
    on the finest level (five operator and two transfer passes each)."""
    n, nz, _, npb, _ = _sizes(ne, p)
    w, its = prec // 8, 20
    ops = 4 * (nz * (9 * w + 4)) + nz * 76 + 2 * npb * (18 * w + 4)
    vec = k * 3 * n * (16 * w + 64)
    return its * (ops + vec), its * k * (5 * 18 * nz + 2 * 36 * npb)


def work(case):
    if case["kind"] == "batch":
        got = [_solve_work(ne, 1, case["prec"], 1) for ne, _ in _batch_problems(case, 0)]
        return {"bytes": sum(b for b, _ in got), "flops": sum(f for _, f in got)}
    n, nz, nco, npb, ncb = _sizes(case["ne"], case["order"])
    w, kind = case.get("prec", 64) // 8, case["kind"]
    coo = nco * 76 + nz * 72
    if kind == "coo":
        return {"bytes": coo + nz * 72, "flops": 9 * nco}
    if kind in ("spmv", "spmm"):
        k = case.get("k", 1)
        return {"bytes": nz * (9 * w + 4) + 6 * n * w * k, "flops": 18 * nz * k}
    # A P pairs every operator block with the prolongator blocks of its column
    # row; P^T (A P) pairs prolongator blocks with the upper half of its row
    ptap_flops = 108 * nz * npb / n + 216 * npb * 13 / 2
    ptap = nz * (9 * w + 4) + npb * (18 * w + 4) + ncb * (36 * w + 4)
    if kind == "ptap":
        return {"bytes": coo + ptap + ncb * 36 * 8, "flops": 9 * nco + ptap_flops}
    b, f = _solve_work(case["ne"], case["order"], case["prec"], case.get("k", 1))
    if kind == "multi":
        return {"bytes": b, "flops": f}
    # a step adds the assembly, the recompute and 16 eigen-estimate products
    return {"bytes": coo + ptap + 16 * nz * 76 + b, "flops": 9 * nco + ptap_flops + 16 * 18 * nz + f}


# --------------------------------------------------------------------- exact

def _csr(pr, v):
    i, j, a = pr.blocks(v)
    r = torch.arange(3, device=v.device)
    rows = (3 * i[:, None, None] + r[None, :, None]).expand(-1, 3, 3).reshape(-1)
    cols = (3 * j[:, None, None] + r[None, None, :]).expand(-1, 3, 3).reshape(-1)
    order = torch.argsort(rows * (3 * pr.n) + cols)
    ptr = torch.zeros(3 * pr.n + 1, dtype=torch.int64, device=v.device)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=3 * pr.n), 0)
    d = torch.zeros(3 * pr.n, dtype=torch.float64, device=v.device)
    on = rows == cols
    d[rows[on]] = a.reshape(-1)[on]
    return torch.sparse_csr_tensor(ptr, cols[order], a.reshape(-1)[order], (3 * pr.n, 3 * pr.n)), d


def _solve(pr, v, b):
    """Diagonally preconditioned CG to 1e-13 in plain torch; b (n_dofs, k)."""
    A, d = _csr(pr, v)
    x, r = torch.zeros_like(b), b.clone()
    z = r / d[:, None]
    p, rz, stop = z.clone(), (r * z).sum(0), 1e-13 * b.norm(dim=0)
    for it in range(20000):
        q = A @ p
        alpha = rz / torch.clamp((p * q).sum(0), min=1e-300)
        x += alpha * p
        r -= alpha * q
        if it % 20 == 0 and bool((r.norm(dim=0) <= stop).all()):
            break
        z = r / d[:, None]
        new = (r * z).sum(0)
        p = z + (new / torch.clamp(rz, min=1e-300)) * p
        rz = new
    return x


def _sum_pairs(key, fn, width):
    """Sum the blocks fn(pairs) over equal keys, sorted by key."""
    uniq, inv = torch.unique(key, return_inverse=True)
    out = torch.zeros((uniq.numel(), width), dtype=torch.float64, device=key.device)
    for s in range(0, key.numel(), 1 << 21):
        out.index_add_(0, inv[s:s + (1 << 21)], fn(slice(s, s + (1 << 21))).reshape(-1, width))
    return uniq, out


def _row_pairs(rows, of, n):
    """For each entry e, the entries of row of[e] of a row-sorted list `rows`: (e, entry)."""
    cnt = torch.bincount(rows, minlength=n)
    start = torch.cumsum(cnt, 0) - cnt
    num = cnt[of]
    e = torch.repeat_interleave(torch.arange(of.numel(), device=of.device), num)
    first = torch.cumsum(num, 0) - num
    return e, start[of[e]] + torch.arange(e.numel(), device=of.device) - first[e]


def exact(case, seed):
    if case["kind"] == "batch":
        got = []
        for ne, nu in _batch_problems(case, seed):
            pr = _Problem(ne, 1, nu)
            got.append(_solve(pr, pr.values(seed), pr.load()[:, None]).reshape(-1))
        return got
    pr = _Problem(case["ne"], case["order"], NU)
    v = pr.values(seed)
    kind = case["kind"]
    if kind == "coo":
        return pr.blocks(v)[2].reshape(-1)
    if kind in ("spmv", "spmm"):
        x = pr.gaussian(seed, case.get("k", 1), torch.float32 if case["prec"] == 32 else torch.float64).double()
        i, j, a = pr.blocks(v)
        y = torch.zeros((pr.n, 3, x.shape[1]), dtype=torch.float64, device=v.device)
        xb = x.view(pr.n, 3, -1)
        for s in range(0, i.numel(), 1 << 20):
            e = slice(s, s + (1 << 20))
            y.index_add_(0, i[e], torch.bmm(a[e], xb[j[e]]))
        return y.reshape(x.shape)
    if kind == "step":
        return _solve(pr, v, pr.load()[:, None]).reshape(-1)
    if kind == "multi":
        return _solve(pr, v, pr.gaussian(seed, case["k"]))
    i, j, a = pr.blocks(v)
    pi, pj, pv, nc = pr.prolongator(v)
    e, t = _row_pairs(pi, j, pr.n)
    zk, z = _sum_pairs(i[e] * nc + pj[t], lambda q: torch.bmm(a[e[q]], pv[t[q]]), 18)
    zi, zj, z = zk // nc, zk % nc, z.view(-1, 3, 6)
    f, u = _row_pairs(zi, pi, pr.n)
    ck, c = _sum_pairs(pj[f] * nc + zj[u], lambda q: torch.bmm(pv[f[q]].transpose(1, 2), z[u[q]]), 36)
    if case["prec"] == 64:
        return c.reshape(-1)
    x = _coarse_vector(nc, seed).float().double().view(nc, 6, 1)
    y = torch.zeros((nc, 6, 1), dtype=torch.float64, device=v.device)
    return y.index_add_(0, ck // nc, torch.bmm(c.view(-1, 6, 6), x[ck % nc])).reshape(-1)
