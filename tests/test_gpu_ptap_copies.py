"""Operand copies of a Galerkin plan: built by the products that read them, and
renewed when P changes whichever precision ran first on the new values."""
import numpy as np
import pytest
import torch

from paper_2606_24748_gb300 import bamg as B

pytestmark = pytest.mark.gpu


def fill(ctx, M, rng, i, j, shape):
    v = torch.from_numpy(rng.standard_normal((i.size, *shape)))
    B.bamg_bsr_coo_set_values(ctx, M, v.cuda(), 0)


def values(ctx, Ac, n):
    v = torch.empty((B.bamg_bsr_info(Ac)["nnzb"], n, n), dtype=torch.float64, device="cuda")
    B.bamg_bsr_get_values(ctx, Ac, v)
    return v


@pytest.mark.parametrize("bs,bsp", [(3, 6), (6, 6), (3, 3)])
def test_fp32_products_leave_the_fp64_copies_to_fp64_products(bs, bsp):
    rng = np.random.default_rng(bs * bsp)
    n, nc, per = 3000, 40, 8
    i = np.arange(n, dtype=np.int32)
    pi = np.repeat(i, per)
    pj = np.concatenate([np.sort(rng.choice(nc, per, replace=False)) for _ in range(n)]).astype(np.int32)
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A, P = B.bamg_bsr_create(ctx, bs, bs, n, n), B.bamg_bsr_create(ctx, bs, bsp, n, nc)
    plans = []
    try:
        for M, r, c in ((A, i, i), (P, pi, pj)):
            B.bamg_bsr_coo_preallocate(ctx, M, torch.from_numpy(r).cuda(), torch.from_numpy(c).cuda())
        fill(ctx, A, rng, i, i, (bs, bs))
        fill(ctx, P, rng, pi, pj, (bs, bsp))
        plan, Ac = B.bamg_ptap_symbolic(ctx, A, P)
        plans.append((plan, Ac))
        B.bamg_ptap_numeric_prec(ctx, plan, A, P, Ac, B.BAMG_FP32)
        used32 = B.bamg_device_memory(ctx)[0]
        B.bamg_ptap_numeric_prec(ctx, plan, A, P, Ac, B.BAMG_FP64)
        # the first FP64 product brings copies of both operands, no smaller than these
        assert B.bamg_device_memory(ctx)[0] - used32 >= 8 * (n * bs * bs + pi.size * bs * bsp)
        for order in ((B.BAMG_FP32, B.BAMG_FP64), (B.BAMG_FP64, B.BAMG_FP32, B.BAMG_FP64)):
            fill(ctx, P, rng, pi, pj, (bs, bsp))
            for prec in order:
                B.bamg_ptap_numeric_prec(ctx, plan, A, P, Ac, prec)
            got = values(ctx, Ac, bsp)
            fresh = B.bamg_ptap_symbolic(ctx, A, P)
            plans.append(fresh)
            B.bamg_ptap_numeric_prec(ctx, fresh[0], A, P, fresh[1], B.BAMG_FP64)
            assert torch.equal(got, values(ctx, fresh[1], bsp))
    finally:
        for plan, Ac in plans:
            B.bamg_ptap_destroy(plan)
            B.bamg_bsr_destroy(Ac)
        B.bamg_bsr_destroy(P)
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)
