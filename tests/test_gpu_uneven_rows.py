"""Multi-vector kernels on matrices whose rows are placed by length and whose
last, partly filled slice is as wide as others or wider."""
import numpy as np
import pytest
import torch

from paper_2606_24748_gb300 import bamg as B
from workloads.elasticity import gaussian_rhs

from gpu_helpers import TOL64, GpuProblem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("last", [1, 31, 33])
@pytest.mark.parametrize("bs", [(3, 3), (3, 6), (6, 3), (6, 6)])
@pytest.mark.parametrize("prec", [64, 32])
def test_spmm_with_a_wide_last_slice(last, bs, prec):
    """1,024 rows of 40 and 3 blocks in turn, then rows of 27 blocks; a sum of
    at most 240 products against extended precision, its operands exact in
    either precision, and untouched values in front of and behind Y."""
    br, bc = bs
    nbr, nbc = 1024 + last, 64
    rng = np.random.default_rng(nbr + br)
    rows = [np.sort(rng.choice(nbc, 27 if i >= 1024 else [40, 3][i % 2], replace=False)) for i in range(nbr)]
    bi = np.repeat(np.arange(nbr), [r.size for r in rows]).astype(np.int32)
    bj = np.concatenate(rows).astype(np.int32)
    dt = torch.float64 if prec == 64 else torch.float32
    eps = 2.0 ** -53 if prec == 64 else 2.0 ** -24
    v = rng.standard_normal((bi.size, br, bc)).astype(np.float32).astype(np.float64)
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A = B.bamg_bsr_create(ctx, br, bc, nbr, nbc)
    try:
        B.bamg_bsr_coo_preallocate(ctx, A, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda())
        B.bamg_bsr_coo_set_values(ctx, A, torch.from_numpy(v).cuda(), 0)
        assert B.bamg_bsr_storage(A)["rows_sorted"]
        for k in (3, 4, 16):
            x = rng.standard_normal((nbc, bc, k)).astype(np.float32).astype(np.float64)
            ref, mag = np.zeros((nbr, br, k), dtype=np.longdouble), np.zeros((nbr, br, k))
            np.add.at(ref, bi, np.einsum("nrc,nck->nrk", v.astype(np.longdouble), x[bj].astype(np.longdouble)))
            np.add.at(mag, bi, np.einsum("nrc,nck->nrk", abs(v), abs(x[bj])))
            guard, n = 512, nbr * br * k
            whole = torch.full((n + 2 * guard,), -5.0, dtype=dt, device="cuda")
            Y = whole[guard:guard + n]
            B.bamg_bsr_spmm(ctx, A, torch.from_numpy(x).to(dt).cuda().reshape(-1), Y, k,
                            B.BAMG_FP64 if prec == 64 else B.BAMG_FP32)
            assert (whole[:guard] == -5.0).all() and (whole[guard + n:] == -5.0).all()
            got = Y.cpu().numpy().astype(np.longdouble).reshape(nbr, br, k)
            assert np.all(np.abs(got - ref) <= 2 * 40 * bc * eps * mag)
    finally:
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)


@pytest.mark.parametrize("ne,order,aggregation", [(6, 2, B.BAMG_AGG_GEOMETRIC), (10, 2, B.BAMG_AGG_GEOMETRIC),
                                                  (12, 1, B.BAMG_AGG_MIS), (24, 1, B.BAMG_AGG_MIS)])
@pytest.mark.parametrize("precision,tol", [(B.BAMG_FP64, TOL64), (B.BAMG_FP32, 1e-5)])
def test_multi_cycle_against_single_cycles(ne, order, aggregation, precision, tol):
    """Prolongators and coarse operators with such slices: every column is the
    single-vector cycle in another summation order (TOL64 in FP64; in FP32 a
    few hundred roundings of 6e-8)."""
    gp = GpuProblem(ne, order=order, aggregation=aggregation, precision=precision, max_coarse_dofs=300)
    try:
        Bh = np.stack([gaussian_rhs(gp.mesh, s) for s in range(5)], axis=1)
        for lanes in (1, 4):
            B.bamg_mg_set_lanes(gp.ctx, gp.mg, lanes)
            for k in (1, 5):
                Bd = torch.from_numpy(np.ascontiguousarray(Bh[:, :k])).cuda()
                X = torch.zeros_like(Bd)
                B.bamg_mg_vcycle_multi(gp.ctx, gp.mg, Bd, X, k)
                for j in range(k):
                    x = torch.zeros(Bh.shape[0], dtype=torch.float64, device="cuda")
                    B.bamg_vcycle(gp.ctx, gp.mg, torch.from_numpy(np.ascontiguousarray(Bh[:, j])).cuda(), x)
                    assert rel(X[:, j].cpu().numpy(), x.cpu().numpy()) <= tol, (lanes, k, j)
    finally:
        gp.close()


@pytest.mark.parametrize("ne,order,aggregation", [(10, 2, B.BAMG_AGG_GEOMETRIC), (24, 1, B.BAMG_AGG_MIS)])
def test_multi_solve_reaches_its_tolerance(ne, order, aggregation):
    gp = GpuProblem(ne, order=order, aggregation=aggregation)
    try:
        Bh = np.stack([gaussian_rhs(gp.mesh, s) for s in range(4)], axis=1)
        X = torch.zeros(Bh.shape, dtype=torch.float64, device="cuda")
        infos = B.bamg_cg_solve_multi(gp.ctx, gp.mg, torch.from_numpy(Bh).cuda(), X, 4, 1e-8, 200)
        for j, info in enumerate(infos):
            bn = np.linalg.norm(Bh[:, j])
            assert info["converged"] and info["true_rnorm"] <= 1.05e-8 * bn
            y = torch.zeros(Bh.shape[0], dtype=torch.float64, device="cuda")
            B.bamg_bsr_spmv(gp.ctx, gp.A, X[:, j].contiguous(), y)
            assert np.linalg.norm(y.cpu().numpy() - Bh[:, j]) <= 1.05e-8 * bn
            x = torch.zeros_like(y)
            out = B.bamg_cg_solve(gp.ctx, gp.mg, torch.from_numpy(np.ascontiguousarray(Bh[:, j])).cuda(), x, 1e-8, 200)
            assert abs(out["iterations"] - info["iterations"]) <= 1
            assert rel(X[:, j].cpu().numpy(), x.cpu().numpy()) <= 1e-7
    finally:
        gp.close()
