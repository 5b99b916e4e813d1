"""Component-split products of 6-row blocks, whose slices are shared by clusters
of CTAs where the matrix has few of them: against extended precision."""
import numpy as np
import pytest
import torch

from paper_2606_24748_gb300 import bamg as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [3, 6])
@pytest.mark.parametrize("nbr,longest", [(1, 3), (33, 17), (70, 130), (1200, 40), (10000, 9)])
def test_split_products_over_slice_counts(bc, nbr, longest):
    """From one slice to more slices than are shared, rows of 0 blocks to more
    than a cluster's warps; a sum of n products is off by at most n 2^-53
    (2^-24 in FP32) of the sum of |a| |x|, doubled for its own rounding."""
    rng = np.random.default_rng(nbr + bc)
    nbc = 150
    lengths = rng.integers(0, longest + 1, nbr)
    lengths[0] = longest
    bi = np.repeat(np.arange(nbr), lengths).astype(np.int32)
    bj = np.concatenate([np.sort(rng.choice(nbc, k, replace=False)) for k in lengths]).astype(np.int32)
    v = rng.standard_normal((bi.size, 6, bc))
    x = rng.standard_normal(nbc * bc)
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A = B.bamg_bsr_create(ctx, 6, bc, nbr, nbc)
    try:
        B.bamg_bsr_coo_preallocate(ctx, A, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda())
        B.bamg_bsr_coo_set_values(ctx, A, torch.from_numpy(v).cuda(), 0)
        xb = x.reshape(-1, bc)[bj]
        want, mag = np.zeros((nbr, 6), dtype=np.longdouble), np.zeros((nbr, 6))
        np.add.at(want, bi, np.einsum("krc,kc->kr", v.astype(np.longdouble), xb.astype(np.longdouble)))
        np.add.at(mag, bi, np.einsum("krc,kc->kr", np.abs(v), np.abs(xb)))
        n = bc * lengths[:, None]
        for prec, dt, eps in ((B.BAMG_FP64, torch.float64, 2.0 ** -52), (B.BAMG_FP32, torch.float32, 2.0 ** -23)):
            xd = torch.from_numpy(x).cuda().to(dt)
            for lanes in (-1, -2, -4):
                B.bamg_bsr_set_lanes_prec(ctx, A, prec, lanes)
                y = torch.full((nbr * 6,), 3.0, dtype=dt, device="cuda")
                B.bamg_bsr_spmv(ctx, A, xd, y, prec)
                got = y.cpu().numpy().reshape(nbr, 6).astype(np.longdouble)
                # the FP32 product also rounds each operand once
                assert np.all(np.abs(got - want) <= (n + 2 * (prec == B.BAMG_FP32)) * eps * mag), (prec, lanes)
                again = torch.empty_like(y)
                B.bamg_bsr_spmv(ctx, A, xd, again, prec)
                assert torch.equal(y, again)
    finally:
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)
