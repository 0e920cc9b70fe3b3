"""The library stays inside the workspace that mrcm_footprint() asks for."""

import ctypes as C

import pytest
import torch

from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GUARD = 1 << 16


@pytest.mark.parametrize("n,sub,l,sweeps,degree,prec", [((128, 128), 4, 2, 1, 0, W.PREC_FP64),    # 1,024 subdomains
                                                        ((264, 264), 6, 2, 2, 0, W.PREC_FP64),    # 1,936
                                                        ((131, 75), 8, 2, 1, 1, W.PREC_FP64),     # uneven
                                                        ((160, 96), 16, 2, 1, 0, W.PREC_FP32),
                                                        ((64, 64), 64, 0, 0, 0, W.PREC_FP64)])    # one subdomain
def test_nothing_is_written_past_the_footprint(n, sub, l, sweeps, degree, prec):
    from paper_2606_08883_gb300 import mrcm
    prob = W.random_problem((n[0], n[1], 1), seed=4, contrast=1e2)
    q = W.Params(sub=(sub, sub, 1), oversample=l, smooth_steps=sweeps, iface_degree=degree, local_prec=prec,
                 refine_setup=1 if prec else 0, tol=1e-8, restart=20, max_iter=200)
    need = mrcm.footprint(prob, q)
    ws = torch.full((need + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    K = torch.as_tensor(prob.K.ravel(), device="cuda")
    f = torch.as_tensor(prob.f.ravel(), device="cuda")
    p = torch.zeros(n[0] * n[1], dtype=torch.float64, device="cuda")
    mp, mq = mrcm.make_problem(prob, K.data_ptr(), f_ptr=f.data_ptr()), mrcm.make_params(q)
    h, res = C.c_void_p(), mrcm.mrcm_result()
    stream = torch.cuda.current_stream().cuda_stream
    assert mrcm.mrcm_setup(C.byref(mp), C.byref(mq), ws.data_ptr(), need, stream, C.byref(h)) == mrcm.MRCM_OK
    try:
        assert mrcm.mrcm_factor_local(h, stream) == mrcm.MRCM_OK
        assert mrcm.mrcm_gmres_solve(h, None, p.data_ptr(), None, None, None, C.byref(res), stream) == mrcm.MRCM_OK
        torch.cuda.synchronize()
        assert bool((ws[need:] == 0xA5).all()), "bytes past the footprint were written"
    finally:
        mrcm.mrcm_destroy(h)
