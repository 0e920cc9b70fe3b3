"""The operator by the marching kernel (grids above half a million cells) and by one thread per cell: odd
widths around a warp's 31 columns, a last group of one row, grids of few rows or columns."""

import numpy as np
import pytest
import torch

from oracle.grid import matvec, transmissibilities
from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sub", [((724, 725), 32), ((31 * 33, 517), 20), ((4098, 129), 32), ((129, 4097), 32),
                                   ((1999, 1101), 32), ((723, 723), 32), ((33, 35), 16)])
def test_operator_matches_the_oracle(n, sub):
    from paper_2606_08883_gb300 import mrcm
    prob = W.random_problem((n[0], n[1], 1), seed=n[0], contrast=1e3, bc_kind=[0, 1, 1, 0, 1, 1])
    q = W.Params(sub=(sub, sub, 1), oversample=0, smooth_steps=0, restart=1, local_prec=W.PREC_FP32)
    s = mrcm.Solver(prob, q)
    s.factor()
    v = np.random.default_rng(2).standard_normal((1, n[1], n[0]))
    w = s.apply_operator(torch.as_tensor(v.ravel(), device="cuda")).cpu().numpy()
    ref = matvec(transmissibilities(prob.K, prob.h, 2, prob.bc_kind), v, 2).ravel()
    # a handful of rounded operations per cell on terms of the size of the largest face product
    assert np.linalg.norm(w - ref) <= 1e-14 * np.linalg.norm(ref)
