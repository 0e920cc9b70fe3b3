"""Device waits that give up: a short limit makes them run out, the call reports it, the next one without a
set-up refuses, and a set-up makes the handle good again."""

import ctypes as C

import numpy as np
import pytest

from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coarse_solver", [0,      # the coupling solve's messages run out first
                                           1])     # band coupling solve, without waits: the Arnoldi barrier
def test_a_wait_that_gives_up_is_reported_and_cured_by_a_set_up(coarse_solver):
    from paper_2606_08883_gb300 import mrcm
    prob = W.random_problem((160, 128, 1), seed=2, contrast=1e2)      # 20 CTAs in the Arnoldi step
    s = mrcm.Solver(prob, W.Params(sub=(8, 8, 1), oversample=2, smooth_steps=1, tol=1e-9, restart=30,
                                   coarse_solver=coarse_solver))
    s.factor()
    assert (s.coarse_method() == "multifrontal") == (coarse_solver == 0)
    want, info = s.solve()
    want = want.cpu().numpy()

    def limit(polls):
        assert mrcm.mrcm_debug_wait_limit(s.handle, C.c_int64(polls)) == mrcm.MRCM_OK

    def refused():
        with pytest.raises(mrcm.MRCMError) as e:
            s.solve()
        assert e.value.status == mrcm.MRCM_ERR_TIMEOUT and "coupling solve" in str(e.value)

    limit(1)
    refused()
    limit(0)
    refused()               # the status stands until a set-up clears it
    s.factor()
    p, again = s.solve()
    assert np.array_equal(p.cpu().numpy(), want) and again["iterations"] == info["iterations"]


def test_a_negative_limit_is_refused():
    from paper_2606_08883_gb300 import mrcm
    s = mrcm.Solver(W.random_problem((16, 16, 1)), W.Params(sub=(8, 8, 1), oversample=0, smooth_steps=0))
    assert mrcm.mrcm_debug_wait_limit(s.handle, C.c_int64(-1)) == mrcm.MRCM_ERR_INVALID_ARG
