"""The multifrontal solve over shapes of the subdomain grid: thin and odd grids, single leaves, fronts
cut into parts and fronts of one part, both interface degrees; against the band LU's solution."""

import numpy as np
import pytest
import torch

from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mx,my,degree", [(2, 1, 0), (1, 40, 0), (5, 3, 0), (17, 16, 0), (33, 20, 0), (64, 3, 1),
                                          (18, 17, 1)])
def test_coupling_solve_matches_the_band_lu(mx, my, degree):
    from paper_2606_08883_gb300 import mrcm
    n = (4 * mx, 4 * my)
    prob = W.random_problem((n[0], n[1], 1), seed=mx + my, contrast=1e2)
    r = torch.randn(n[0] * n[1], dtype=torch.float64, generator=torch.Generator().manual_seed(3)).cuda()
    c = []
    for solver in (0, 1):
        s = mrcm.Solver(prob, W.Params(sub=(4, 4, 1), oversample=1, smooth_steps=0, iface_degree=degree,
                                       coarse_solver=solver))
        s.factor()
        assert (s.coarse_method() == "multifrontal") == (solver == 0)
        s.apply_precond(r)
        c.append([s.debug(mrcm.MRCM_DBG_COARSE)])
        s.apply_precond(2.0 * r)          # a second solve takes no value of the first
        c[-1].append(s.debug(mrcm.MRCM_DBG_COARSE))
    for k in (0, 1):
        # both FP64: eps times the condition number of G (1e4 to 1e5 on these fields)
        assert np.linalg.norm(c[0][k] - c[1][k]) <= 1e-9 * np.linalg.norm(c[1][k])
    assert np.array_equal(2.0 * c[0][0], c[0][1])
