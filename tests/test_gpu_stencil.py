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


def test_apply_precond_on_a_large_odd_grid():
    """T where the reconstruction takes four rows per thread and the FP32 sweep's residual is marched, on a
    grid whose sides divide by neither."""
    from oracle.solve import build
    from paper_2606_08883_gb300 import mrcm
    n = (725, 727)
    prob = W.random_problem((n[0], n[1], 1), seed=5, contrast=10.0)
    r = np.random.default_rng(6).standard_normal((1, n[1], n[0]))
    ref = build(prob.K, prob.h, 2, prob.bc_kind, (32, 32, 1), 2, 1, 10.0).apply(r).ravel()
    # FP64: rounding times the boxes' condition (1e4); FP32 local solves: 6e-8 times the same
    for prec, tol in ((W.PREC_FP64, 1e-10), (W.PREC_FP32, 1e-3)):
        s = mrcm.Solver(prob, W.Params(sub=(32, 32, 1), oversample=2, smooth_steps=1, alpha=10.0, local_prec=prec))
        s.factor()
        z = s.apply_precond(torch.as_tensor(r.ravel(), device="cuda")).cpu().numpy()
        assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref)
        s.close()
