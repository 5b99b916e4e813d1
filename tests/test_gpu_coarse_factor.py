"""The dense coarsest factorisation at the edges of its 32-wide tiles."""
import numpy as np
import pytest
import torch

from paper_2606_24748_gb300 import bamg as B
from gpu_helpers import GpuProblem
from oracle_cases import problem

pytestmark = pytest.mark.gpu


# 81 = 2 tiles and 17 rows, 192 = 6 whole tiles, 375 = 11 tiles and 23 rows,
# 648 = 20 tiles and 8 rows (one panel of the diagonal tile)
@pytest.mark.parametrize("ne", [2, 3, 4, 5])
def test_single_level_dense_solve(ne):
    """The cycle of a single-level hierarchy applies the inverse of the
    operator: the residual of b - A x is rounding, n eps |A| |x| at most."""
    _, _, A = problem(ne)
    gp = GpuProblem(ne, max_coarse_dofs=10 ** 6, coarse_solver=1)
    try:
        assert B.bamg_mg_num_levels(gp.mg) == 1
        S = A.scalar().tocsr()
        b = np.random.default_rng(ne).standard_normal(S.shape[0])
        x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
        B.bamg_vcycle(gp.ctx, gp.mg, torch.from_numpy(b).cuda(), x)
        got = x.cpu().numpy()
        norm = abs(S).sum(axis=1).max()
        # x = L^-T L^-1 b with the inverse formed: its error, and so the
        # residual, carries the condition of L, below 1e3 for these sizes
        bound = S.shape[0] * 2.0 ** -52 * norm * 1e3 * np.abs(got).max()
        assert np.abs(b - S @ got).max() <= bound
    finally:
        gp.close()
