"""Accuracy of every output relative to its own terms, where other bands hold far larger
weights: the occupied bands against the rest.

Tolerance, derived before the first run: at a scale of its own an output carries about 2^-52 of the
root of the sum of its terms' squares; partial fractions, FP64 sums and the oracle add a few
2^-52 each: 2^-48 of that root.
"""

import numpy as np
import pytest

import oracle
from paper_2008_11326_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -48


@pytest.fixture(scope="module")
def gpp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11326_gb300 import gpp as g
    return g


def natural(prob, nocc, sexcut=0.0):
    """Root of the sum of the squares of what each output adds up: M I w u on branch 1 for
    achtemp; in the bands of asxtemp half of M I w u and of M I w v (the forms it is summed in)."""
    g = prob.indinv[prob.inv_igp_index]
    am = np.abs(prob.aqsmtemp[:, g]) * prob.vcoul[g]
    M2 = (am[:, :, None] * np.abs(prob.aqsntemp)[:, None, :]) ** 2
    w, Iw2 = prob.wtilde_array, np.abs(prob.I_eps_array * prob.wtilde_array) ** 2
    ach, asx = [], []
    for k in range(prob.nw):
        x = prob.wx_array[:, k][:, None, None]
        a, s = np.abs(x - w) ** 2, np.abs(x + w) ** 2
        u = M2 * Iw2 * (a > 0.25) / a
        v = M2 * Iw2 / s
        if sexcut:   # the terms themselves
            t = np.where(a > 0.25, np.abs(w) ** 2 / a / s, 0.25 / s)
            t = M2 * Iw2 * t * ~((x < 0) & (t * np.abs(w) ** 2 > sexcut ** 2))
        else:
            t = 0.25 * (u + v)
        ach.append(u.sum())
        asx.append(t[:nocc].sum())
    return np.sqrt(ach), np.sqrt(asx)


def check(gpp, prob, occ="all", tol=TOL, sexcut=0.0):
    import torch
    dp = gpp.DeviceProblem.from_host(prob, device="cuda")
    got = gpp.sigma(dp, occ_mode=occ, sexcut=sexcut)
    torch.cuda.synchronize()
    ref = oracle.sigma(prob, occ_mode=0 if occ == "all" else 1, sexcut=sexcut)
    size = natural(prob, prob.number_bands if occ == "all" else prob.nvband, sexcut)
    for g, r, s in zip(got, ref, size):
        err = np.abs(g.cpu().numpy() - r)
        assert np.all(err <= tol * s), (err / s, prob.shape)


@pytest.mark.parametrize("nw", [1, 3, 5])
@pytest.mark.parametrize("scale", [1e-2, 1e-4, 1e-6, 1e-8, 1e-12, 1e6])
def test_occupied_weights_of_another_size(gpp, scale, nw):
    prob = inputs.make_problem(64, 8, 100, 5, nw, seed=41)
    for side in ("aqsmtemp", "aqsntemp"):
        a = getattr(prob, side).copy()
        a[:8] *= scale
        check(gpp, prob.replace(**{side: a}), occ="occupied")
