"""The order of the FP64 arithmetic, bit for bit.  On channels of contrast 1e6 with a tensor K or linear
interface spaces T r is rounding times a condition number of 1e6 and more, so a factorisation that sums
the same terms in another order moves it by 1e-9 to 1e-3.  The recorded values come from the plain
order: Cholesky, inverse of L and L^-T L^-1 column by column in increasing k; fronts assembled as
original + first child + second child, eliminated as a_ij -= a_ik (a_kj / a_kk), products summed in
increasing k; each inner product of the Krylov basis summed over slices of 1,024 elements.

The fields are made of integers, so every machine forms the same inputs."""

import hashlib
import json
import os

import numpy as np
import pytest

from paper_2606_08883_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RECORDED = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp64_rounding_order.json")

#        grid, subdomain, overlap, sweeps, degree, multiplicative, tensor
CASES = {"tensor": ((100, 84), 16, 3, 2, 0, 0, 1),
         "linear": ((100, 84), 16, 3, 1, 1, 1, 0),
         "tensor-linear": ((117, 83), 32, 4, 2, 1, 0, 1),
         "scalar": ((117, 83), 32, 4, 2, 0, 0, 0),
         "wide-boxes": ((129, 118), 56, 4, 1, 0, 0, 0),
         "many-subdomains": ((128, 132), 4, 1, 1, 0, 0, 0),      # pivot blocks on a cluster
         "large-blocks": ((180, 180), 4, 1, 1, 0, 0, 0)}         # and of 90 unknowns on one CTA


def integers(n, seed):
    """n well mixed integers of 20 bits"""
    x = np.arange(n, dtype=np.uint64) * np.uint64(2654435761) + np.uint64(seed * 40503 + 1)
    x = (x ^ (x >> np.uint64(15))) * np.uint64(2246822519) % np.uint64(1 << 32)
    x = (x ^ (x >> np.uint64(13))) * np.uint64(3266489917) % np.uint64(1 << 32)
    return (x >> np.uint64(12)).astype(np.int64) % (1 << 20)


def channels(nx, ny, seed):
    """Zigzag channels of permeability 1e6 along x, at most 9 cells wide, over a background of 1."""
    K = np.ones((1, ny, nx))
    i, j = np.arange(nx)[None, :], np.arange(ny)[:, None]
    for a, b, c, d in integers(4 * 6, seed).reshape(6, 4):
        period, amplitude = 20 + int(b) % 60, 4 + int(c) % 16
        phase = (i + int(d)) % (2 * period)
        zigzag = np.minimum(phase, 2 * period - phase) * amplitude // period
        K[0, np.abs(j - int(a) % ny - zigzag) <= 1 + int(a) % 4] = 1e6
    return K


def problem(case):
    (nx, ny), sub, l, sweeps, degree, mult, tensor = CASES[case]
    K = channels(nx, ny, 1)
    if tensor:
        K = np.stack([K, channels(nx, ny, 2)])
    ends = [W.DIRICHLET, W.DIRICHLET] + 4 * [W.NEUMANN]
    prob = W.Problem(2, (nx, ny, 1), (1.0, 1.0, 1.0), K, ends, [np.ones((1, ny)), np.zeros((1, ny))] + 4 * [None])
    return prob, W.Params(sub=(sub, sub, 1), oversample=l, smooth_steps=sweeps, alpha=10.0, tol=1e-8, restart=100, max_iter=100,
                          smooth_kind=mult, iface_degree=degree)


def record(a):
    a = np.asarray(a, dtype=np.float64).ravel() + 0.0      # one kind of zero
    return {"sha256": hashlib.sha256(a.astype("<f8").tobytes()).hexdigest(),
            "samples": [float(v).hex() for v in a[:: max(1, a.size // 16)]]}


def check(case, what, a):
    with open(RECORDED) as f:
        want = json.load(f)[case][what]
    got = record(a)
    w, g = (np.array([float.fromhex(v) for v in r["samples"]]) for r in (want, got))
    assert np.array_equal(w, g), f"largest difference {np.abs(w - g).max() / np.abs(w).max():.1e} of the samples' largest"
    assert want["sha256"] == got["sha256"]


def solver(case):
    from paper_2606_08883_gb300 import mrcm
    prob, q = problem(case)
    s = mrcm.Solver(prob, q)
    s.factor()
    return s


@pytest.mark.parametrize("case", list(CASES))
def test_local_factors(case):
    """Side moments of the basis functions: boundary problems on both kinds of boxes."""
    from paper_2606_08883_gb300 import mrcm
    check(case, "moments", solver(case).debug(mrcm.MRCM_DBG_MOMENTS))


@pytest.mark.parametrize("case", list(CASES))
def test_coupling_system(case):
    """Interface coefficients and T r: assembly, elimination and products of the fronts, their solves."""
    import torch
    from paper_2606_08883_gb300 import mrcm
    s = solver(case)
    z = s.apply_precond(torch.as_tensor((integers(s.n, 3) - (1 << 19)) / float(1 << 19), device="cuda"))
    check(case, "coupling", s.debug(mrcm.MRCM_DBG_COARSE))
    check(case, "precond", z.cpu().numpy())


@pytest.mark.parametrize("case", list(CASES))
def test_solution(case):
    """p of a whole solve, which the inner products of the Krylov basis enter too."""
    p, info = solver(case).solve()
    check(case, "solve", p.cpu().numpy())
