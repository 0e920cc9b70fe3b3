"""GMRES over vector lengths: one cluster of one to eight CTAs, few CTAs that each form every total, the
three-barrier form, a last CTA with few elements, and cycles longer than a block has warps."""

import numpy as np
import pytest

from oracle.solve import solve
from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,restart,sweeps", [((12, 11), 30, 1), ((36, 16), 30, 1), ((64, 64), 30, 1), ((64, 64), 40, 0),
                                              ((68, 64), 30, 1), ((128, 64), 30, 1), ((129, 65), 40, 0), ((160, 111), 30, 1)])
def test_gmres_matches_the_oracle_over_vector_lengths(n, restart, sweeps):
    from paper_2606_08883_gb300 import mrcm
    prob = W.random_problem((n[0], n[1], 1), seed=n[1], contrast=1e2)
    l = 2 if sweeps else 0       # without overlap and sweeps the cycles run past 32 steps
    s = mrcm.Solver(prob, W.Params(sub=(8, 8, 1), oversample=l, smooth_steps=sweeps, tol=1e-9, restart=restart, max_iter=400))
    s.factor()
    p, info = s.solve()
    ref, oinfo, _ = solve(prob.K, prob.h, 2, prob.bc_kind, prob.bc_val, prob.f, sub=(8, 8, 1), l=l, smooth_steps=sweeps,
                          tol=1e-9, restart=restart, max_iter=400)
    assert info["iterations"] == oinfo["iterations"]
    # the same iterate up to FP64 rounding carried through the cycles
    assert np.linalg.norm(p.cpu().numpy() - ref.ravel()) <= 1e-8 * np.linalg.norm(ref)
