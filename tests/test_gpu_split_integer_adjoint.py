"""The adjoint's split-integer form at the edges of its loops, tiles and ranges, against the
CPU adjoint.

Tolerance, derived before the first run: the integer sums carry about 2^-51 of a gradient entry's
natural scale (the root sum of squares of its terms), the largest entry of a gradient is at
least that scale, and the FP64 sums add a few 2^-53: 2^-47 of the largest entry.
"""

import numpy as np
import pytest

import oracle
from paper_2008_11326_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -47


@pytest.fixture(scope="module")
def gpp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11326_gb300 import gpp as g
    return g


def check(gpp, prob, ga, gs, occ="all", tol=TOL):
    import torch
    dp = gpp.DeviceProblem.from_host(prob, device="cuda")
    got = gpp.sigma_backward(dp, torch.from_numpy(ga).cuda(), torch.from_numpy(gs).cuda(),
                             occ_mode=occ)
    torch.cuda.synchronize()
    ref = oracle.sigma_adjoint(prob, ga, gs, occ_mode=0 if occ == "all" else 1)
    for k, r in ref.items():
        scale = np.abs(r).max()
        err = np.abs(got[k].cpu().numpy() - r).max()
        assert err <= tol * scale, (k, err / max(scale, 1e-300), prob.shape)


def cotangents(W, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return (rng.standard_normal(W) + 1j * rng.standard_normal(W),
            rng.standard_normal(W) + 1j * rng.standard_normal(W))


# bands around a reduction (4), the staged weights (64) and the modular sums (1024); columns
# around a tile (8); G-vectors around a warp; every number of frequencies
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (3, 31, 7, 2), (4, 32, 8, 3), (5, 33, 9, 4),
                                   (63, 40, 5, 5), (64, 65, 3, 6), (65, 33, 17, 7), (7, 70, 9, 8),
                                   (1027, 9, 2, 3), (2051, 5, 1, 1)])
def test_loop_edges(gpp, shape):
    B, G, P, W = shape
    prob = inputs.make_problem(B, 2, G, P, W, seed=B + G)
    check(gpp, prob, *cotangents(W, 1))
    check(gpp, prob.replace(nvband=(2 * B) // 3), *cotangents(W, 2), occ="occupied")
    check(gpp, prob.replace(nvband=0), *cotangents(W, 3), occ="occupied")


@pytest.mark.parametrize("kind", ["zero", "ach", "asx", "spread", "huge"])
def test_cotangents(gpp, kind):
    prob = inputs.make_problem(12, 2, 70, 9, 3, seed=5)
    ga, gs = cotangents(3, 4)
    if kind in ("zero", "asx"):
        ga = np.zeros_like(ga)
    if kind in ("zero", "ach"):
        gs = np.zeros_like(gs)
    if kind == "spread":
        ga, gs = ga * np.array([1.0, 1e-6, 1e-12]), gs * np.array([1e-9, 1.0, 1e-3])
    if kind == "huge":     # beyond the integer scaling's range: the FP64 form
        ga, gs = ga * 1e100, gs * 1e100
    check(gpp, prob, ga, gs)


def test_warps_of_both_forms_in_a_tile(gpp):
    """Columns whose poles lie outside the split-integer range (below 2^(E-7), Re w < 0, more
    than twice the largest frequency), a sentinel and repeated columns, beside ordinary ones
    of the same tile; limbs that end on half units. The FP64 form's tolerance, 1e-12: next to
    x = -w (Re w < 0) it and the oracle are each off by 2^-47 of the largest entry."""
    prob = inputs.make_problem(9, 2, 75, 16, 3, seed=8)
    wt = prob.wtilde_array.copy()
    wt[1] *= 0.03
    wt[3, 40:] *= -1.0
    wt[6] = (np.floor(wt[6].real * 2 ** 26) + 0.5) / 2 ** 26 + \
        1j * (np.floor(wt[6].imag * 2 ** 26) + 0.5) / 2 ** 26
    inv = prob.inv_igp_index.copy()
    inv[4] = prob.ncouls
    inv[9] = inv[2]
    inv[13] = inv[2]
    prob = prob.replace(wtilde_array=wt, inv_igp_index=inv)
    check(gpp, prob, *cotangents(3, 6), tol=1e-12)
    check(gpp, prob.replace(wx_array=prob.wx_array * 0.1), *cotangents(3, 7), tol=1e-12)
    check(gpp, prob.replace(wx_array=prob.wx_array - 6.0), *cotangents(3, 8), tol=1e-12)
