"""Accuracy of every output relative to its own terms, where other bands hold far larger
weights: the occupied bands against the rest, a heavy band that branch 2 or the cutoff
removes, a light band that alone sets the scale of the reciprocals.

Tolerance, derived before the first run: an output whose terms are 2^-6 of its scale carries at
most 2^-50 of the root of the sum of its terms' squares, weaker ones are FP64's, and partial
fractions, FP64 sums and the oracle add a few 2^-52 each: 2^-48 of that root. Entries of the gradients, single and of fewer terms: 2^-47, the
adjoint's bound elsewhere.
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


@pytest.mark.parametrize("heavy", [1e1, 1e2, 1e4, 1e6, 1e12])
def test_heavy_band_in_branch_2(gpp, heavy):
    """Band 5 lies within 1/2 of every pole at the first of four frequencies only."""
    rng = np.random.Generator(np.random.PCG64(43))
    prob = inputs.make_problem(24, 24, 96, 4, 4, seed=43)
    w = rng.uniform(1.5, 1.7, (4, 96)) + 1j * rng.uniform(-0.05, 0.05, (4, 96))
    wx = prob.wx_array.copy()
    wx[:, 0] = np.where(np.abs(wx[:, 0] - 1.6) < 0.7, 2.5, wx[:, 0])
    wx[5] = [1.6, 4.0, 5.0, 6.0]
    am = prob.aqsmtemp.copy()
    am[5] *= heavy
    check(gpp, prob.replace(wtilde_array=w, wx_array=wx, aqsmtemp=am))
    # some lanes of each warp only
    w[:, ::3] += 3.0
    check(gpp, prob.replace(wtilde_array=w, wx_array=wx, aqsmtemp=am))


@pytest.mark.parametrize("light", [1.0, 1e-2, 1e-6])
def test_light_band_at_the_pole(gpp, light):
    """All bands far from the poles, where |u| is about 1/40, but one light one at |x - w| = 0.55."""
    rng = np.random.Generator(np.random.PCG64(44))
    prob = inputs.make_problem(32, 32, 96, 4, 2, seed=44)
    wx = rng.uniform(40.0, 46.0, (32, 2))
    wx[7] = 3.0
    am = prob.aqsmtemp.copy()
    am[7] *= light
    check(gpp, prob.replace(wtilde_array=2.45 + 0.01j * rng.standard_normal((4, 96)), wx_array=wx,
                            aqsmtemp=am), tol=2.0 ** -47)   # the partial fractions' x / |w|: 2^4.2


@pytest.mark.parametrize("part", ["all", "heavy"])
def test_terms_dropped_by_the_cutoff(gpp, part):
    """Every term beyond the cutoff: asxtemp is exactly zero; or only one heavy band's."""
    rng = np.random.Generator(np.random.PCG64(45))
    prob = inputs.make_problem(12, 12, 96, 3, 2, seed=45)
    wx = -rng.uniform(1.0, 2.0, (12, 2)) if part == "all" else rng.uniform(-8.0, -5.0, (12, 2))
    wx[4] = -1.5
    am = prob.aqsmtemp.copy()
    am[4] *= 1.0 if part == "all" else 1e5
    w = rng.uniform(1.2, 1.8, (3, 96)) + 0j
    prob = prob.replace(wx_array=wx, aqsmtemp=am, wtilde_array=w)
    if part == "all":
        import torch
        got = gpp.sigma(gpp.DeviceProblem.from_host(prob, device="cuda"), sexcut=0.05)
        torch.cuda.synchronize()
        assert np.all(got[1].cpu().numpy() == 0) and np.all(
            np.asarray(oracle.sigma(prob, sexcut=0.05)[1]) == 0)
    check(gpp, prob, sexcut=0.05 if part == "all" else 0.4)


@pytest.mark.parametrize("nw", [2, 3, 7])
@pytest.mark.parametrize("occ", ["all", "occupied"])
def test_sums_that_cancel(gpp, nw, occ):
    """Bands in pairs of opposite weights and almost equal frequencies: every sum is far below its
    terms, which are strong all the same."""
    prob = inputs.make_problem(20, 12, 100, 5, nw, seed=46)
    am, an, wx = prob.aqsmtemp.copy(), prob.aqsntemp.copy(), prob.wx_array.copy()
    am[1::2], an[1::2], wx[1::2] = -am[::2], an[::2], wx[::2] + 1e-7
    prob = prob.replace(aqsmtemp=am, aqsntemp=an, wx_array=wx)
    check(gpp, prob, occ=occ)
    check(gpp, prob.replace(wx_array=wx - 5.0), occ=occ, sexcut=3.0)


def test_small_cotangents(gpp):
    """The gradients are linear in the cotangents, also where those squared are below FP64's range."""
    import torch
    prob = inputs.make_problem(12, 7, 70, 9, 3, seed=47)
    ga, gs = inputs.cotangents(48, 3)
    dp = gpp.DeviceProblem.from_host(prob, device="cuda")
    ref = oracle.sigma_adjoint(prob, ga, gs, occ_mode=1)
    for k in (-300, -500, -536, -544, -600, -900):
        s = 2.0 ** k
        got = gpp.sigma_backward(dp, torch.from_numpy(ga * s).cuda(), torch.from_numpy(gs * s).cuda(),
                                 occ_mode="occupied")
        for name, r in ref.items():
            err = np.abs(got[name].cpu().numpy() / s - r).max()
            assert err <= 2.0 ** -47 * np.abs(r).max(), (name, k, err)


def natural_gradients(prob, ga, gs, nocc):
    """The root of the sum of the squares of what every gradient entry adds up (partial fractions)."""
    B, (P, G) = prob.number_bands, prob.wtilde_array.shape
    g = prob.indinv[prob.inv_igp_index]
    am2 = (np.abs(prob.aqsmtemp[:, g]) * prob.vcoul[g]) ** 2        # [B][P]
    an2 = np.abs(prob.aqsntemp) ** 2
    w, I = prob.wtilde_array, prob.I_eps_array
    occ = (np.arange(B) < nocc)[:, None, None]
    q, h = np.zeros((B, P, G)), np.zeros((B, P, G))                # of GI and of GW, squared
    for k in range(prob.nw):
        x = prob.wx_array[:, k][:, None, None]
        a2, s2 = np.abs(x - w) ** 2, np.abs(x + w) ** 2
        c = np.where(occ, abs(ga[k].conj() + gs[k].conj() / 2), abs(ga[k])) ** 2 * (a2 > 0.25)
        s = occ * abs(gs[k] / 2) ** 2
        q += c / a2 + s / s2
        h += x * x * (c / a2 ** 2 + s / s2 ** 2)
    M2, Iw2 = am2[:, :, None] * an2[:, None, :], np.abs(I * w) ** 2
    aqsm = np.zeros((B, G))
    aqsm[:, g] = prob.vcoul[g] * np.sqrt(np.einsum("bg,pg,bpg->bp", an2, Iw2, q))
    return dict(I_eps=np.abs(w) * np.sqrt((M2 * q).sum(0)), wtilde=np.abs(I) * np.sqrt((M2 * h).sum(0)),
                aqsn=np.sqrt(np.einsum("bp,pg,bpg->bg", am2, Iw2, q)), aqsm=aqsm)


def check_gradients(gpp, prob, ga, gs, occ="occupied"):
    import torch
    dp = gpp.DeviceProblem.from_host(prob, device="cuda")
    got = gpp.sigma_backward(dp, torch.from_numpy(ga).cuda(), torch.from_numpy(gs).cuda(),
                             occ_mode=occ)
    torch.cuda.synchronize()
    ref = oracle.sigma_adjoint(prob, ga, gs, occ_mode=0 if occ == "all" else 1)
    size = natural_gradients(prob, ga, gs, prob.number_bands if occ == "all" else prob.nvband)
    for k, r in ref.items():
        err = np.abs(got[k].cpu().numpy() - r)
        bad = err > 2.0 ** -47 * size[k]
        assert not bad.any(), (k, bad.sum(), np.nanmax(err[bad] / size[k][bad]), prob.shape)


def random_cotangents(nw, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    z = rng.standard_normal((4, nw))
    return z[0] + 1j * z[1], z[2] + 1j * z[3]


@pytest.mark.parametrize("scale", [1e-2, 1e-4, 1e-8, 1e-12, 1e6])
def test_gradients_occupied_weights_of_another_size(gpp, scale):
    prob = inputs.make_problem(40, 7, 70, 9, 3, seed=49)
    am = prob.aqsmtemp.copy()
    am[:7] *= scale
    prob = prob.replace(aqsmtemp=am)
    ga, gs = random_cotangents(3, 50)
    check_gradients(gpp, prob, ga, gs)
    check_gradients(gpp, prob, 0 * ga, gs)


@pytest.mark.parametrize("scale", [1e-2, 1e-4, 1e-8, 1e-20, 0.0])
@pytest.mark.parametrize("nw", [1, 3])
def test_gradients_cotangents_of_two_sizes(gpp, scale, nw):
    prob = inputs.make_problem(40, 17, 70, 9, nw, seed=51)
    ga, gs = random_cotangents(nw, 52)
    check_gradients(gpp, prob, scale * ga, gs)
    check_gradients(gpp, prob, ga, scale * gs)


def check_weak_gradients(gpp, prob, ga, gs, occ="all"):
    """Where entries of a warp lie on both sides of the lines below which they are taken from FP64
    (2^-8 of the scale for a band's rows; for the pairs' sums 2^-11 and 2^-13, and for half of a warp 2^-7
    and 2^-9), errors of 2^-56 of the scale: a tensor's root mean square error within 2^-47 of
    its terms', a single entry's within 2^-43 of its own, four times that at the most."""
    import torch
    dp = gpp.DeviceProblem.from_host(prob, device="cuda")
    got = gpp.sigma_backward(dp, torch.from_numpy(ga).cuda(), torch.from_numpy(gs).cuda(),
                             occ_mode=occ)
    torch.cuda.synchronize()
    ref = oracle.sigma_adjoint(prob, ga, gs, occ_mode=0 if occ == "all" else 1)
    size = natural_gradients(prob, ga, gs, prob.number_bands if occ == "all" else prob.nvband)
    for k, r in ref.items():
        err = np.abs(got[k].cpu().numpy() - r)
        assert np.all(err <= 2.0 ** -41 * size[k]), (k, np.max(err / np.maximum(size[k], 1e-300)))
        some = size[k] > 0      # (rows of columns that no local column reaches are zero)
        if some.any():
            rel = np.sqrt(np.mean((err[some] / size[k][some]) ** 2))
            assert rel <= 2.0 ** -47, (k, rel)


@pytest.mark.parametrize("heavy", [1e1, 1e2, 1e4, 1e8, 1e12])
@pytest.mark.parametrize("nw", [1, 2])
def test_gradients_heavy_band_in_branch_2(gpp, heavy, nw):
    rng = np.random.Generator(np.random.PCG64(53))
    prob = inputs.make_problem(24, 24, 70, 9, nw, seed=53)
    w = rng.uniform(1.5, 1.7, (9, 70)) + 1j * rng.uniform(-0.05, 0.05, (9, 70))
    wx = prob.wx_array.copy()
    wx[:, 0] = np.where(np.abs(wx[:, 0] - 1.6) < 0.7, 2.5, wx[:, 0])
    wx[5] = 1.6
    am = prob.aqsmtemp.copy()
    am[5] *= heavy
    prob = prob.replace(wtilde_array=w, wx_array=wx, aqsmtemp=am)
    ga, gs = random_cotangents(nw, 54)
    check_weak_gradients(gpp, prob, ga, 0 * gs)
    check_weak_gradients(gpp, prob, ga, gs)


@pytest.mark.parametrize("small", [1.0, 1e-1, 1e-2, 1e-4, 1e-8, 0.0])
def test_gradients_of_small_frequencies(gpp, small):
    """x << |w| in what counts: all bands but a light one; or the one frequency with a cotangent."""
    rng = np.random.Generator(np.random.PCG64(55))
    prob = inputs.make_problem(40, 40, 70, 9, 3, seed=55)
    wx = small * rng.uniform(0.0, 1.0, (40, 3))
    wx[5] = 8.0
    am = prob.aqsmtemp.copy()
    am[5] *= 1e-6 if small else 0.0
    ga, gs = random_cotangents(3, 56)
    check_weak_gradients(gpp, prob.replace(wx_array=wx, aqsmtemp=am), ga, gs)
    wx = prob.wx_array.copy()
    wx[:, 0] = small * rng.uniform(0.0, 1.0, 40)
    one = np.array([1.0, 0.0, 0.0])
    check_weak_gradients(gpp, prob.replace(wx_array=wx), ga * one, gs * one)


@pytest.mark.parametrize("small", [0.3, 1e-2, 1e-4, 1e-8, 1e-22, 1e-60])
@pytest.mark.parametrize("occ", ["all", "occupied"])
def test_gradients_cotangents_of_different_frequencies(gpp, small, occ):
    """Rows of bands whose large cotangent meets branch 2: only the small ones reach them."""
    rng = np.random.Generator(np.random.PCG64(57))
    prob = inputs.make_problem(30, 12, 70, 9, 3, seed=57)
    w = rng.uniform(1.5, 1.7, (9, 70)) + 1j * rng.uniform(-0.05, 0.05, (9, 70))
    wx = prob.wx_array.copy()
    wx[::5, 0] = 1.6
    ga, gs = random_cotangents(3, 58)
    ga = ga * np.array([1.0, small, small])
    check_weak_gradients(gpp, prob.replace(wtilde_array=w, wx_array=wx), ga, small * gs, occ)
    check_weak_gradients(gpp, prob.replace(wtilde_array=w, wx_array=wx), ga, 0 * gs, occ)
    check_weak_gradients(gpp, prob.replace(wx_array=wx), ga, gs, occ)


# bands around the FP32 low sums' eight (forward) and the reductions' four (adjoint)
@pytest.mark.parametrize("B", [3, 4, 5, 7, 8, 9])
@pytest.mark.parametrize("nw", [1, 3, 4])
def test_few_bands(gpp, B, nw):
    prob = inputs.make_problem(B, (B + 1) // 2, 65, 9, nw, seed=59)
    ga, gs = random_cotangents(nw, 60)
    for occ in ("all", "occupied"):
        check(gpp, prob, occ=occ)
        check_weak_gradients(gpp, prob, ga, gs, occ)


@pytest.mark.parametrize("nw", [2, 5])
@pytest.mark.parametrize("zero", ["occupied", "rest", "columns"])
def test_bands_without_weights(gpp, zero, nw):
    """A class of bands whose weights are all zero (padding), and G-vectors without any."""
    prob = inputs.make_problem(40, 9, 100, 5, nw, seed=61)
    am, an = prob.aqsmtemp.copy(), prob.aqsntemp.copy()
    if zero == "columns":
        an[:, 40:70] = 0.0
    else:
        am[slice(0, 9) if zero == "occupied" else slice(9, 40)] = 0.0
    prob = prob.replace(aqsmtemp=am, aqsntemp=an)
    ga, gs = random_cotangents(nw, 62)
    check(gpp, prob, occ="occupied")
    check(gpp, prob.replace(wx_array=prob.wx_array - 5.0), occ="occupied", sexcut=3.0)
    check_weak_gradients(gpp, prob, ga, gs, "occupied")


@pytest.mark.parametrize("small", [0.3, 1e-2, 1e-4, 1e-8, 1e-22])
@pytest.mark.parametrize("nw", [1, 3])
def test_gradients_of_bands_all_in_branch_2(gpp, small, nw):
    """Bands whose every frequency is in branch 2 for every pole: asxtemp's cotangent alone, a small
    one, reaches their rows."""
    rng = np.random.Generator(np.random.PCG64(63))
    prob = inputs.make_problem(30, 12, 70, 1, nw, seed=63)
    w = rng.uniform(1.5, 1.7, (1, 70)) + 1j * rng.uniform(-0.05, 0.05, (1, 70))
    wx = prob.wx_array.copy()
    wx[::5] = 1.6
    ga, gs = random_cotangents(nw, 64)
    for occ in ("all", "occupied"):
        check_weak_gradients(gpp, prob.replace(wtilde_array=w, wx_array=wx), ga, small * gs, occ)
