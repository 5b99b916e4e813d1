"""FP64 products that are partly formed in fixed point: every scalar row of a
product against sums in extended precision, with the bound n 2^-52 of its own
sum of |a| |x| that FP64 multiply-adds keep too (n 2^-53 for the products, as
much again for the few roundings of the parts' sums), at row lengths around the
carry and flush steps and for values of unlike size in a block."""
import numpy as np
import pytest
import torch

from paper_2606_24748_gb300 import bamg as B

pytestmark = pytest.mark.gpu


def operator(rng, lengths, nbc, bs, decades):
    """Block COO arrays of a matrix whose row i has lengths[i] blocks."""
    br, bc = bs
    bi = np.repeat(np.arange(len(lengths)), lengths).astype(np.int32)
    bj = np.concatenate([np.sort(rng.choice(nbc, k, replace=False)) for k in lengths]).astype(np.int32)
    v = rng.standard_normal((bi.size, br, bc)) * 10.0 ** rng.uniform(-decades, decades, (bi.size, 1, 1))
    v[rng.random(bi.size) < 0.05] = 0.0
    return bi, bj, v


def reference(bi, bj, v, x, nbr):
    """Products, sums of |a| |x| and the number of terms of each scalar row."""
    br, bc = v.shape[1:]
    xb = x.reshape(-1, bc)
    y = np.zeros((nbr, br), dtype=np.longdouble)
    mag, n = np.zeros((nbr, br), dtype=np.longdouble), np.zeros(nbr)
    for i, j, a in zip(bi, bj, v):
        y[i] += (a.astype(np.longdouble) * xb[j].astype(np.longdouble)).sum(1)
        mag[i] += (np.abs(a).astype(np.longdouble) * np.abs(xb[j]).astype(np.longdouble)).sum(1)
        n[i] += bc
    return y, mag, n[:, None]


def within(got, ref, scale=1.0):
    y, mag, n = ref
    return np.all(np.abs(got.reshape(y.shape).astype(np.longdouble) / scale - y) <= n * 2.0 ** -52 * mag)


@pytest.mark.parametrize("bs", [(3, 3), (3, 6), (6, 3)])
def test_products_at_carry_and_flush_lengths(bs):
    rng = np.random.default_rng(5)
    lengths = [1, 19, 20, 21, 39, 40, 41, 60, 80, 81, 120, 0, 2, 7] + [27] * 40
    nbc, nbr = 130, len(lengths)
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A = B.bamg_bsr_create(ctx, bs[0], bs[1], nbr, nbc)
    try:
        bi, bj, v = operator(rng, lengths, nbc, bs, 2.0)
        B.bamg_bsr_coo_preallocate(ctx, A, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda())
        B.bamg_bsr_coo_set_values(ctx, A, torch.from_numpy(v).cuda(), 0)
        x = rng.standard_normal(nbc * bs[1]) * 10.0 ** rng.uniform(-3, 3, nbc * bs[1])
        ref = reference(bi, bj, v, x, nbr)
        xd = torch.from_numpy(x).cuda()
        single = torch.full((nbr * bs[0],), 7.0, dtype=torch.float64, device="cuda")
        for lanes in ((-264, -272, -288) if bs == (6, 3) else ()) + (4, 32, 1):
            B.bamg_bsr_set_lanes(ctx, A, lanes)
            B.bamg_bsr_spmv(ctx, A, xd, single)
            assert within(single.cpu().numpy(), ref), lanes
        # several vectors: the single one-lane product bit for bit, whatever its sign and scale
        for f in (1.0, -1.0, 2.0 ** 40, -(2.0 ** -70)):
            X = torch.stack([f * xd, xd, torch.zeros_like(xd), -xd], 1).contiguous()
            Y = torch.empty((nbr * bs[0], 4), dtype=torch.float64, device="cuda")
            B.bamg_bsr_spmm(ctx, A, X, Y, 4)
            assert torch.equal(Y[:, 0], f * single) and torch.equal(Y[:, 1], single)
            assert torch.equal(Y[:, 3], -single) and not Y[:, 2].any()
        # columns that are no multiple of four take the one-column kernel
        X = torch.stack([xd, 2 * xd, -xd], 1).contiguous()
        Y = torch.empty((nbr * bs[0], 3), dtype=torch.float64, device="cuda")
        B.bamg_bsr_spmm(ctx, A, X, Y, 3)
        assert all(within(Y[:, j].cpu().numpy(), ref, f) for j, f in enumerate((1.0, 2.0, -1.0)))
    finally:
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)


def unlike_sizes(rng, mode, v, bi, bj, nbr, nbc):
    """Scales the blocks in place, and returns the scales of x's entries."""
    _, br, bc = v.shape
    xs = np.ones((nbc, bc))
    if mode in ("rows", "both"):  # unknowns in other units, weakly coupled components
        v *= (10.0 ** rng.uniform(-12, 12, (nbr, br)))[bi][:, :, None]
    if mode in ("columns", "both"):
        xs = 10.0 ** rng.uniform(-12, 12, (nbc, bc))
        if mode == "both":
            v /= xs[bj][:, None, :]
    if mode == "entries":
        v *= 10.0 ** rng.uniform(-15, 15, v.shape)
        xs = 10.0 ** rng.uniform(-15, 15, xs.shape)
    if mode == "identity":  # each row sees one of x's entries
        v[:] = np.resize(np.eye(max(br, bc)), (max(br, bc), max(br, bc)))[:br, :bc]
        xs = 10.0 ** rng.uniform(-20, 20, xs.shape)
    if mode == "penalty":  # one large entry on a dof of some rows
        v[rng.random(len(bi)) < 0.3, br - 2, bc - 1] *= 1e18
    return xs


@pytest.mark.parametrize("mode", ["rows", "columns", "both", "entries", "identity", "penalty"])
@pytest.mark.parametrize("bs", [(3, 3), (3, 6), (6, 3)])
def test_values_of_unlike_size_in_a_block(bs, mode):
    """Small scalar rows beside large ones, and small entries of x beside large ones."""
    rng = np.random.default_rng(len(mode) + bs[1])
    lengths = [1, 2, 5, 27, 60, 81] + [27] * 90
    nbc, nbr = 130, len(lengths)
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A = B.bamg_bsr_create(ctx, bs[0], bs[1], nbr, nbc)
    try:
        bi, bj, v = operator(rng, lengths, nbc, bs, 0.0)
        x = rng.standard_normal((nbc, bs[1])) * unlike_sizes(rng, mode, v, bi, bj, nbr, nbc)
        ref = reference(bi, bj, v, x, nbr)
        B.bamg_bsr_coo_preallocate(ctx, A, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda())
        B.bamg_bsr_coo_set_values(ctx, A, torch.from_numpy(v).cuda(), 0)
        xd = torch.from_numpy(x.reshape(-1)).cuda()
        y = torch.empty(nbr * bs[0], dtype=torch.float64, device="cuda")
        for lanes in ((-1, -4, -258, -264, -288) if bs == (6, 3) else ()) + (1, 2, 8):
            B.bamg_bsr_set_lanes(ctx, A, lanes)
            B.bamg_bsr_spmv(ctx, A, xd, y)
            assert within(y.cpu().numpy(), ref), lanes
        for k in (3, 8):
            X = torch.stack([xd] * k, 1).contiguous()
            Y = torch.empty((nbr * bs[0], k), dtype=torch.float64, device="cuda")
            B.bamg_bsr_spmm(ctx, A, X, Y, k)
            assert all(within(Y[:, j].cpu().numpy(), ref) for j in range(k)), k
    finally:
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)


@pytest.mark.parametrize("bs,lanes", [((3, 3), 1), ((3, 3), 4), ((3, 6), 1), ((6, 3), -264)])
def test_values_outside_the_scales(bs, lanes):
    """Infinities, NaN, subnormals, the largest and smallest magnitudes and
    zero blocks beside huge x give what FP64 multiply-adds give."""
    rng = np.random.default_rng(9)
    nbr = nbc = 64
    lengths = [9] * nbr
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    A = B.bamg_bsr_create(ctx, bs[0], bs[1], nbr, nbc)
    try:
        bi, bj, v = operator(rng, lengths, nbc, bs, 1.0)
        x = rng.standard_normal(nbc * bs[1])
        v[9 * 3 + 2, -2, 1] = np.inf
        v[9 * 5 + 1, -1, 0] = np.nan
        v[9 * 7:9 * 8] *= 1e-300
        v[9 * 9:9 * 10] *= 2.0 ** 900
        v[9 * 11:9 * 12] *= 2.0 ** -1060
        v[9 * 13:9 * 14] = 0.0
        v[9 * 15 + 4] = 0.0
        x[bj[9 * 15 + 4] * bs[1]] = 2.0 ** 800
        B.bamg_bsr_coo_preallocate(ctx, A, torch.from_numpy(bi).cuda(), torch.from_numpy(bj).cuda())
        B.bamg_bsr_coo_set_values(ctx, A, torch.from_numpy(v).cuda(), 0)
        B.bamg_bsr_set_lanes(ctx, A, lanes)
        y = torch.empty(nbr * bs[0], dtype=torch.float64, device="cuda")
        B.bamg_bsr_spmv(ctx, A, torch.from_numpy(x).cuda(), y)
        got = y.cpu().numpy().reshape(nbr, bs[0])
        with np.errstate(all="ignore"):
            want = np.zeros((nbr, bs[0]))
            np.add.at(want, bi, np.einsum("krc,kc->kr", v, x.reshape(-1, bs[1])[bj]))
            tol = np.zeros((nbr, bs[0]))
            np.add.at(tol, bi, np.einsum("krc,kc->kr", np.abs(v), np.abs(x.reshape(-1, bs[1])[bj])))
        fine = np.isfinite(want)
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(got[~fine & ~np.isnan(want)], want[~fine & ~np.isnan(want)])
        # both sides sum 27 or 54 products in FP64 or better; subnormal sums are
        # off by at most one unit per term
        n = 9 * bs[1]
        bound = n * 2.0 ** -51 * tol + n * 2.0 ** -1074
        off = np.abs(got - want, where=fine, out=np.zeros_like(want))
        assert (off <= bound)[fine].all()
        assert not got[13].any()
    finally:
        B.bamg_bsr_destroy(A)
        B.bamg_ctx_destroy(ctx)


@pytest.mark.parametrize("bs,bsp", [(3, 6), (6, 6), (3, 3)])
@pytest.mark.parametrize("symmetric", [0, 1])
def test_galerkin_product_at_carry_and_flush_lengths(bs, bsp, symmetric):
    """P^T A P against extended precision, with gather lists of 1 to some 100
    pairs: 2^-52 per product, twice, on at most 300 products of entries within
    a factor of about 8 of their root mean square stays below 1e-12 normwise."""
    galerkin(bs, bsp, symmetric, False)


@pytest.mark.parametrize("bs,bsp", [(3, 6), (6, 6), (3, 3)])
@pytest.mark.parametrize("symmetric", [0, 1])
def test_galerkin_product_of_unlike_units(bs, bsp, symmetric):
    """The same with the fine unknowns in units over 24 decades and the coarse
    ones over 16 more: entry by entry, Z = A P is off by at most n 2^-52 of
    |A| |P| and P^T Z by as much of |P|^T |Z|, with n at most 720 in either."""
    galerkin(bs, bsp, symmetric, True)


def galerkin(bs, bsp, symmetric, unlike):
    rng = np.random.default_rng(bs + bsp)
    n, nc = 120, 4
    hit = rng.random((n, n)) < np.linspace(0.02, 0.9, n)[:, None]
    hit = hit | hit.T | np.eye(n, dtype=bool)
    hp = rng.random((n, nc)) < np.array([0.9, 0.5, 0.2, 0.03])
    hp[:, 0] |= ~hp.any(1)
    bi, bj = (t.astype(np.int32) for t in np.nonzero(hit))
    pi, pj = (t.astype(np.int32) for t in np.nonzero(hp))
    A = np.zeros((n, bs, n, bs))
    A[bi, :, bj, :] = rng.standard_normal((bi.size, bs, bs))
    A = (A.reshape(n * bs, n * bs) + A.reshape(n * bs, n * bs).T).reshape(n, bs, n, bs)
    pv = rng.standard_normal((pi.size, bs, bsp))
    if unlike:
        d, dc = 10.0 ** rng.uniform(-12, 12, (n, bs)), 10.0 ** rng.uniform(-8, 8, (nc, bsp))
        A *= d[:, :, None, None] * d
        pv *= dc[pj][:, None, :] / d[pi][:, :, None]
    v = A[bi, :, bj, :]
    P = np.zeros((n, bs, nc, bsp))
    P[pi, :, pj, :] = pv
    Pl, Al = P.reshape(n * bs, -1).astype(np.longdouble), A.reshape(n * bs, -1).astype(np.longdouble)
    want = (Pl.T @ (Al @ Pl)).astype(np.float64)
    mag = (np.abs(Pl).T @ (np.abs(Al) @ np.abs(Pl))).astype(np.float64)
    ctx = B.bamg_ctx_create(torch.cuda.current_stream())
    Ah, Ph = B.bamg_bsr_create(ctx, bs, bs, n, n), B.bamg_bsr_create(ctx, bs, bsp, n, nc)
    plan = Ac = None
    try:
        for M, i, j, w in ((Ah, bi, bj, v), (Ph, pi, pj, pv)):
            B.bamg_bsr_coo_preallocate(ctx, M, torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda())
            B.bamg_bsr_coo_set_values(ctx, M, torch.from_numpy(np.ascontiguousarray(w)).cuda(), 0)
        B.bamg_bsr_set_symmetric(ctx, Ah, symmetric)
        plan, Ac = B.bamg_ptap_symbolic(ctx, Ah, Ph)
        B.bamg_ptap_numeric(ctx, plan, Ah, Ph, Ac)
        info = B.bamg_bsr_info(Ac)
        rp = torch.empty(info["nbr"] + 1, dtype=torch.int32, device="cuda")
        ci = torch.empty(info["nnzb"], dtype=torch.int32, device="cuda")
        vals = torch.empty((info["nnzb"], bsp, bsp), dtype=torch.float64, device="cuda")
        B.bamg_bsr_get_pattern(ctx, Ac, rp, ci)
        B.bamg_bsr_get_values(ctx, Ac, vals)
        rows = np.repeat(np.arange(nc), np.diff(rp.cpu().numpy()))
        got = np.zeros((nc, bsp, nc, bsp))
        got[rows, :, ci.cpu().numpy(), :] = vals.cpu().numpy()
        off = np.abs(got.reshape(want.shape) - want)
        assert np.all(off <= 2 * n * bs * 2.0 ** -52 * mag)
        if not unlike:
            assert np.linalg.norm(off) <= 1e-12 * np.linalg.norm(want)
        # a value outside the scales goes through FP64 multiply-adds
        v[0, -1, -1] = np.nan
        B.bamg_bsr_coo_set_values(ctx, Ah, torch.from_numpy(np.ascontiguousarray(v)).cuda(), 0)
        B.bamg_ptap_numeric(ctx, plan, Ah, Ph, Ac)
        B.bamg_bsr_get_values(ctx, Ac, vals)
        assert torch.isnan(vals).any()
        with pytest.raises(B.BamgError):
            B.bamg_ctx_sync(ctx)  # the assembly reports the NaN it wrote
    finally:
        if plan is not None:
            B.bamg_ptap_destroy(plan)
            B.bamg_bsr_destroy(Ac)
        B.bamg_bsr_destroy(Ph)
        B.bamg_bsr_destroy(Ah)
        B.bamg_ctx_destroy(ctx)
