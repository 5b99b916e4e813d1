"""Values into and out of the sliced storage: blocked COO sums and the
block-CSR read-back, exactly, over block shapes and ragged rows; products of
matrices whose rows are placed by length."""
import numpy as np
import pytest
import torch

from paper_2606_24748_gb300 import bamg as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bs", [(3, 3), (1, 1), (2, 5), (3, 6), (6, 6), (7, 7), (8, 8)])
@pytest.mark.parametrize("nbr", [1, 33, 70])
def test_coo_sums_and_read_back_exactly(bs, nbr):
    """Rows of 0 to 40 blocks (several passes of the read-back), blocks of 1
    to 9 contributions side by side in a warp, ignored entries, ADD mode: the
    sums are those of the contributions in input order."""
    rng = np.random.default_rng(nbr + 10 * bs[0])
    nbc = 48
    blocks = [(i, j) for i in range(nbr) for j in rng.choice(nbc, [40, 0, 1, 17, 27][i % 5], replace=False)]
    if not blocks:
        blocks = [(0, 3)]
    reps = rng.integers(1, 10, len(blocks))
    idx = np.repeat(np.arange(len(blocks)), reps)
    rng.shuffle(idx)
    bi = np.array([blocks[k][0] for k in idx], dtype=np.int32)
    bj = np.array([blocks[k][1] for k in idx], dtype=np.int32)
    drop = rng.random(idx.size) < 0.05
    drop[[np.nonzero(idx == k)[0][0] for k in range(len(blocks))]] = False  # every block keeps a contribution
    bi[drop] = -1
    v = rng.standard_normal((idx.size, *bs))
    want = {}
    for k in range(idx.size):
        if not drop[k]:
            key = (int(bi[k]), int(bj[k]))
            want[key] = v[k] if key not in want else want[key] + v[k]
    ref = np.stack([want[k] for k in sorted(want)])
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A = B.bamg_bsr_create(ctx, bs[0], bs[1], nbr, nbc)
    try:
        B.bamg_bsr_coo_preallocate(ctx, A, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda())
        assert B.bamg_bsr_info(A)["nnzb"] == len(ref)
        vd = torch.from_numpy(v).cuda()
        got = torch.empty(ref.shape, dtype=torch.float64, device="cuda")
        B.bamg_bsr_coo_set_values(ctx, A, vd, 0)
        B.bamg_bsr_get_values(ctx, A, got)
        assert np.array_equal(got.cpu().numpy(), ref)
        B.bamg_bsr_coo_set_values(ctx, A, vd, 1)
        B.bamg_bsr_get_values(ctx, A, got)
        assert np.array_equal(got.cpu().numpy(), ref + ref)
    finally:
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)


@pytest.mark.parametrize("nbr", [31, 33, 1024, 1057, 2500])
@pytest.mark.parametrize("prec", [64, 32])
def test_rows_placed_by_length(nbr, prec):
    """Rows of 0 to 40 blocks in turn (sorted within windows of 1,024 rows, the
    slices then by width; one part of a slice, of a window, several windows):
    values read back in pattern order, and the product with a vector."""
    rng = np.random.default_rng(nbr)
    nbc = 64
    rows = [np.sort(rng.choice(nbc, [40, 3, 17, 0, 27][i % 5], replace=False)) for i in range(nbr)]
    bi = np.repeat(np.arange(nbr), [r.size for r in rows]).astype(np.int32)
    bj = np.concatenate(rows).astype(np.int32)
    dt = torch.float64 if prec == 64 else torch.float32
    v = rng.standard_normal((bi.size, 3, 3))
    x = rng.standard_normal((nbc, 3))
    if prec == 32:
        v, x = v.astype(np.float32).astype(np.float64), x.astype(np.float32).astype(np.float64)
    ref, mag = np.zeros((nbr, 3)), np.zeros((nbr, 3))
    np.add.at(ref, bi, np.einsum("krc,kc->kr", v, x[bj]))
    np.add.at(mag, bi, np.einsum("krc,kc->kr", abs(v), abs(x[bj])))
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A = B.bamg_bsr_create(ctx, 3, 3, nbr, nbc)
    try:
        B.bamg_bsr_coo_preallocate(ctx, A, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda())
        B.bamg_bsr_coo_set_values(ctx, A, torch.from_numpy(v).cuda(), 0)
        got = torch.empty(v.shape, dtype=torch.float64, device="cuda")
        B.bamg_bsr_get_values(ctx, A, got)
        assert np.array_equal(got.cpu().numpy(), v)
        xd = torch.from_numpy(x).to(dt).cuda().reshape(-1)
        y = torch.full((nbr * 3,), float("nan"), dtype=dt, device="cuda")
        B.bamg_bsr_spmv(ctx, A, xd, y, B.BAMG_FP64 if prec == 64 else B.BAMG_FP32)
        # sums of at most 120 products: 122 roundings of the terms' magnitudes
        eps = 2.0 ** -53 if prec == 64 else 2.0 ** -24
        assert (np.abs(y.cpu().numpy().astype(np.float64).reshape(nbr, 3) - ref) <= 122 * eps * mag + 1e-300).all()
    finally:
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)
