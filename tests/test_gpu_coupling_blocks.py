"""Coupling systems whose larger pivot blocks one CTA inverts (their size is no multiple of the cluster): the
widest register layouts of the elimination, against the band LU."""

import numpy as np
import pytest
import torch

from paper_2606_08883_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("mx,my,degree,block", [(45, 45, 0, 90), (47, 49, 0, 94), (49, 49, 0, 98), (63, 63, 0, 126), (31, 31, 1, 124)])
def test_large_pivot_blocks_match_the_band_lu(mx, my, degree, block):
    from paper_2606_08883_gb300 import mrcm
    n = (4 * mx, 4 * my)
    prob = W.random_problem((n[0], n[1], 1), seed=mx + my, contrast=1e2)
    q = dict(sub=(4, 4, 1), oversample=1, smooth_steps=0, iface_degree=degree)
    one_cta = [f["np"] for f in mrcm.plan_mf_export(prob, W.Params(**q))["fronts"] if f["np"] < 64 or f["np"] % 8]
    assert max(one_cta) == block
    r = torch.randn(n[0] * n[1], dtype=torch.float64, generator=torch.Generator().manual_seed(3)).cuda()
    c = []
    for solver in (0, 1):
        s = mrcm.Solver(prob, W.Params(coarse_solver=solver, **q))
        s.factor()
        assert (s.coarse_method() == "multifrontal") == (solver == 0)
        s.apply_precond(r)
        c.append(s.debug(mrcm.MRCM_DBG_COARSE))
    # both FP64: eps times the condition number of G (1e4 to 1e5 on these fields)
    assert np.linalg.norm(c[0] - c[1]) <= 1e-9 * np.linalg.norm(c[1])
