"""Entries handed from front to front inside a coupling solve: each value whole and of the present solve."""

import numpy as np
import pytest
import torch

from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_repeated_solves_take_no_half_of_another():
    """Two right-hand sides whose entries differ in both 32-bit halves, in turn on one handle: a half of the
    other solve's entry, or a late one, changes the bits."""
    from paper_2606_08883_gb300 import mrcm
    n = 256                                       # 64 x 64 subdomains: nine levels of fronts
    prob = W.random_problem((n, n, 1), seed=8, contrast=1e2)
    s = mrcm.Solver(prob, W.Params(sub=(4, 4, 1), oversample=1, smooth_steps=0))
    s.factor()
    assert s.coarse_method() == "multifrontal"
    gen = torch.Generator().manual_seed(9)
    rs = [torch.randn(n * n, dtype=torch.float64, generator=gen).cuda() for _ in range(2)]
    rs[1] *= -1e-3
    want = []
    for r in rs:
        s.apply_precond(r)
        want.append(s.debug(mrcm.MRCM_DBG_COARSE))
    assert np.isfinite(want).all()
    halves = [w.view(np.uint32).reshape(-1, 2) for w in want]
    assert (halves[0] != halves[1]).mean() > 0.99
    z = [s.empty() for _ in rs]
    first = [s.apply_precond(r, out).clone() for r, out in zip(rs, z)]
    for _ in range(100):
        for k in (0, 1):
            s.apply_precond(rs[k], z[k])
        assert torch.equal(z[0], first[0]) and torch.equal(z[1], first[1])
