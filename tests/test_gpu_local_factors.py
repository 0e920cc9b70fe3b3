"""FP64 line-block factorisation over box widths: the edges of its register layouts, odd widths, boxes
of one and two lines, the widest box."""

import numpy as np
import pytest
import torch

from oracle.solve import build
from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sub,l", [((9, 6), (3, 2), 0), ((5, 4), (5, 1), 0), ((40, 33), (15, 16), 0), ((40, 36), (17, 17), 1),
                                     ((44, 54), (20, 24), 2), ((62, 59), (29, 28), 2), ((70, 64), (32, 32), 0),
                                     ((70, 68), (33, 32), 2), ((80, 72), (36, 32), 2), ((86, 92), (41, 44), 2),
                                     ((100, 96), (48, 48), 0), ((110, 104), (49, 52), 0), ((124, 120), (60, 60), 2)])
def test_apply_precond_over_box_widths(n, sub, l):
    from paper_2606_08883_gb300 import mrcm
    prob = W.random_problem((n[0], n[1], 1), seed=n[0], contrast=1e3)
    q = W.Params(sub=sub + (1,), oversample=l, smooth_steps=1, tol=1e-9, restart=30)
    s = mrcm.Solver(prob, q)
    s.factor()
    r = np.random.default_rng(7).standard_normal((1, n[1], n[0]))
    z = s.apply_precond(torch.as_tensor(r.ravel(), device="cuda")).cpu().numpy()
    ref = build(prob.K, prob.h, 2, prob.bc_kind, q.sub, l, 1, q.alpha).apply(r).ravel()
    # both sides in FP64: the boxes' condition numbers (contrast 1e3, up to 64 cells across) times 1e-16
    assert np.linalg.norm(z - ref) <= 1e-10 * np.linalg.norm(ref)
