"""GPU parity of the FP64 sum's split-integer form (gpp_terms_fix.cuh) at the edges of its
range and of its loops, against the CPU oracle.

Tolerance, derived before the first run: a pair's sum carries at most about 2^-51 of its root
mean square, pairs are independent, and the final FP64 additions add a few 2^-53; so every
output lies within 2^-48 (3.6e-15) of the root mean square of its kind, whatever cancels.
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


def check(gpp, prob, occ="all", **opts):
    import torch
    dp = gpp.DeviceProblem.from_host(prob, device="cuda")
    got = gpp.sigma(dp, occ_mode=occ, **opts)
    torch.cuda.synchronize()
    ref = oracle.sigma(prob, occ_mode=0 if occ == "all" else 1)
    for g, r in zip(got, ref):
        rms = np.sqrt(np.mean(np.abs(r) ** 2))
        err = np.max(np.abs(g.cpu().numpy() - r))
        assert err <= TOL * rms, (err / rms, prob.shape)


# bands: one, around the FP32 low sums (16), the staged weights (64), the modular sums (1024);
# G-vectors around a warp and a tile; every frequency group (1, 2, 3, 2+2, 3+2, 3+3, 3+2+2, 3+3+2)
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 33, 3, 2), (15, 127, 5, 3), (16, 128, 4, 4),
                                   (17, 129, 4, 5), (63, 511, 3, 6), (64, 513, 3, 7),
                                   (65, 130, 3, 8), (1023, 40, 2, 3), (1025, 40, 2, 3),
                                   (2049, 33, 1, 1)])
def test_loop_edges(gpp, shape):
    B, G, P, W = shape
    prob = inputs.make_problem(B, 2, G, P, W, seed=B + G)
    check(gpp, prob)
    check(gpp, prob.replace(nvband=B // 2), occ="occupied")


# largest frequency at the edge of each binary scale (0.75 2^E) and past the last one; |w| from
# below 2^(E-7) to above 1.375 2^E - max x
@pytest.mark.parametrize("xmax", [0.4, 3.0, 3.0001, 6.0, 12.0, 23.9, 47.999, 48.0, 48.001, 90.0])
def test_frequency_and_pole_range(gpp, xmax):
    rng = np.random.Generator(np.random.PCG64(int(xmax * 1000)))
    prob = inputs.make_problem(20, 2, 320, 4, 3, seed=7)
    wx = rng.uniform(0.0, xmax, size=prob.wx_array.shape)
    wx[3, 1] = xmax
    wx[4, 0] = 0.0
    E = 2
    while E < 6 and xmax > 0.75 * 2 ** E:
        E += 1
    wt = prob.wtilde_array.copy()
    lo, hi = 2.0 ** (E - 7), 1.375 * 2 ** E - xmax
    for p in range(4):   # segments of one warp each, just inside and just outside the bounds
        for k, mod in enumerate((lo * 1.0001, lo * 0.9999, 3 * lo, hi * 0.9999, hi * 1.0001)):
            if mod > 0:
                ph = rng.uniform(-1.5, 1.5, size=32)
                wt[p, 64 * k:64 * k + 32] = mod * np.exp(1j * ph)
    check(gpp, prob.replace(wx_array=wx, wtilde_array=wt))


@pytest.mark.parametrize("spread", [0.5, 2.0, 6.0])
def test_weight_range(gpp, spread):
    """Weights spread over e^(+-2 spread) per band and column (the widest leaves most pairs to
    the FP64 form), zero rows, zero columns, very large and very small scales."""
    rng = np.random.Generator(np.random.PCG64(int(10 * spread)))
    prob = inputs.make_problem(24, 2, 256, 6, 3, seed=3)
    am = prob.aqsmtemp * np.exp(spread * rng.standard_normal((24, 256)))
    an = prob.aqsntemp * np.exp(spread * rng.standard_normal((24, 256)))
    an[:, 5] = 0.0
    an[:, 64:96] *= 1e-90
    an[:, 100] *= 1e-250           # below the integer scaling's range: FP64
    am[7] = 0.0
    check(gpp, prob.replace(aqsmtemp=am, aqsntemp=an))
    check(gpp, prob.replace(aqsmtemp=am * 1e30, aqsntemp=an * 1e-20))


def test_one_column_of_each_extreme(gpp):
    """A column whose largest weight and largest aqsntemp fall in different bands (their
    product is far below the product of the maxima), beside ordinary ones."""
    prob = inputs.make_problem(8, 2, 96, 3, 2, seed=21)
    g = prob.indinv[prob.inv_igp_index]
    am, an = prob.aqsmtemp.copy(), prob.aqsntemp.copy()
    am[:, g[1]] *= 1e-4
    am[2, g[1]] = 1.0
    an[2, 40:60] *= 1e-5
    check(gpp, prob.replace(aqsmtemp=am, aqsntemp=an))


def test_limb_edges(gpp):
    """Poles, frequencies and weights whose low 32-bit limbs are exactly the most negative
    integer, or whose values are exact in few bits (halves and multiples of the high limb's
    unit, 2^-26 for frequencies up to 12; powers of two; equal magnitudes)."""
    rng = np.random.Generator(np.random.PCG64(11))
    prob = inputs.make_problem(19, 2, 256, 8, 3, seed=13)
    u = 2.0 ** -26
    wt = prob.wtilde_array.copy()
    half = lambda a: (np.floor(a / u) + 0.5) * u  # noqa: E731
    wt[0:2] = half(wt[0:2].real) + 1j * half(wt[0:2].imag)
    wt[2:4] = half(wt[2:4].real) + 1j * np.round(wt[2:4].imag / u) * u
    wt[4:6] = wt[4:6].real + 1j * half(wt[4:6].imag)
    wt[6] = wt[6].real                              # real poles
    wt[7] = rng.choice([0.25, 0.5, 1.0, 2.0], size=256) + 0.5j * rng.choice([-1, 0, 1], size=256)
    wx = prob.wx_array.copy()
    wx[:6] = half(wx[:6])
    wx[6] = [0.0, 4.0, 12.0]
    am, an = prob.aqsmtemp.copy(), prob.aqsntemp.copy()
    an[3:6] = rng.choice([-1.0, 1.0], size=(3, 256)) + 1j * rng.choice([-1.0, 1.0], size=(3, 256))
    an[7:9] = half(an[7:9].real) + 1j * half(an[7:9].imag)
    am[4] = 1.0 - 2.0 ** -53
    am[5] = -1.0 + 2.0 ** -53
    check(gpp, prob.replace(wtilde_array=wt, wx_array=wx, aqsmtemp=am, aqsntemp=an))


@pytest.mark.parametrize("sexcut", [1e-3, 0.3, 1.2, 4.0, 8.0, 15.0, 40.0])
@pytest.mark.parametrize("occ", ["all", "occupied"])
def test_negative_frequencies_with_cutoff(gpp, sexcut, occ):
    """The screened-exchange cutoff on the split-integer form: frequencies of both signs, many
    next to -Re w, poles from 0.15 up (the lowest need the reduced scale, the highest cutoffs
    send warps to the FP64 form).

    Tolerance: a kept term next to x = -w is taken at a scale up to 2^-6 below the others', so
    with a relative error up to 2^-47, and such terms are few: 2^-45 of the outputs' root mean
    square."""
    import torch
    rng = np.random.Generator(np.random.PCG64(int(1000 * sexcut) + len(occ)))
    prob = inputs.make_problem(40, 17, 300, 12, 3, seed=29)
    wx = rng.uniform(-9.0, 9.0, size=prob.wx_array.shape)
    wx[::3] = -rng.uniform(0.1, 3.1, size=wx[::3].shape)
    wx[1] = [0.0, -0.0, -1e-12]
    wt = prob.wtilde_array.copy()
    wt[3] = rng.uniform(0.15, 0.3, size=300) + 1j * rng.uniform(-0.01, 0.01, size=300)
    prob = prob.replace(wx_array=wx, wtilde_array=wt)
    dp = gpp.DeviceProblem.from_host(prob, device="cuda")
    got = gpp.sigma(dp, sexcut=sexcut, ch_half=True, occ_mode=occ)
    torch.cuda.synchronize()
    ref = oracle.sigma(prob, sexcut=sexcut, ch_half=True, occ_mode=0 if occ == "all" else 1)
    for g, r in zip(got, ref):
        rms = np.sqrt(np.mean(np.abs(r) ** 2))
        err = np.max(np.abs(g.cpu().numpy() - r))
        assert err <= 2.0 ** -45 * rms, err / rms


@pytest.mark.parametrize("sexcut", [0.7, 4.0, 10.0])
def test_cutoff_decisions_near_the_edge(gpp, sexcut):
    """Terms on both sides of the cutoff, down to a relative distance of 2^-45, on both
    branches and for poles from 0.15 to 9: every one is decided as the oracle decides it. Each
    term is a problem of its own in the comparison (one column's G-vectors carry the distances;
    a wrong decision changes the sum by a term, 1e-3 of it)."""
    import torch
    rng = np.random.Generator(np.random.PCG64(int(10 * sexcut)))
    B = 12
    prob = inputs.make_problem(B, 2, 256, B, 1, seed=31)
    delta = 2.0 ** -rng.uniform(3, 45, 256) * rng.choice([-1.0, 1.0], 256)
    w0 = np.geomspace(0.16, 6.0, B)
    wx = np.empty((B, 1))
    wt = prob.wtilde_array.copy()
    for b in range(B):
        if b % 2 == 0:   # branch 1, |x| > w: w^2 / (x^2 - w^2) = sexcut (1 + delta)
            x = -w0[b] * np.sqrt(1 + 1 / sexcut)
            t = sexcut * (1 + delta)
            wt[b] = abs(x) * np.sqrt(t / (1 + t))
        else:            # |x| < w: w^2 / (w^2 - x^2) where that can reach the cutoff
            x = -w0[b] * np.sqrt(max(1 - 1 / sexcut, 0.1))
            t = np.maximum(sexcut * (1 + delta), 1.05)
            wt[b] = abs(x) * np.sqrt(t / (t - 1))
        wx[b, 0] = x
    prob = prob.replace(wx_array=wx, wtilde_array=wt)
    for b in range(B):
        sub = prob.columns(slice(b, b + 1))
        dp = gpp.DeviceProblem.from_host(sub, device="cuda")
        got = gpp.sigma(dp, sexcut=sexcut)[1]
        torch.cuda.synchronize()
        ref = oracle.sigma(sub, sexcut=sexcut)[1]
        assert abs(got.cpu().numpy()[0] - ref[0]) <= 1e-9 * np.abs(sub.vcoul).max() * 256, b


# weights of nearly one phase, so that the sums of 300 bands pass 2^64 many times over, upwards
# and downwards, with the scale of u above ("far": |x - w| >= 1/2, |x + w| > 2) and below that
# of v ("low": |x + w| < 1/2); (x + |w|) / 2 |w| is at most 4, so the difference of the two sums
# that asxtemp takes costs two of the tolerance's bits
@pytest.mark.parametrize("where", ["far", "low"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_sums_beyond_64_bits(gpp, where, sign):
    rng = np.random.Generator(np.random.PCG64(77))
    prob = inputs.make_problem(300, 120, 70, 3, 2, seed=78)
    B, G = prob.aqsmtemp.shape
    P = prob.wtilde_array.shape[0]

    def near_one(shape):
        return 1.0 + 0.01 * (rng.standard_normal(shape) + 1j * rng.standard_normal(shape))
    far = where == "far"
    w = rng.uniform(1.0, 3.0, (P, G)) if far else rng.uniform(0.2, 0.4, (P, G))
    x = rng.uniform(0.0, 7.0, (B, 2)) if far else rng.uniform(0.0, 1.2, (B, 2))
    prob = prob.replace(aqsmtemp=sign * (0.9 - 0.3j) * near_one((B, G)),
                        aqsntemp=(0.6 + 0.5j) * near_one((B, G)), wx_array=x,
                        wtilde_array=w + 1j * rng.uniform(-0.05, 0.05, (P, G)))
    check(gpp, prob)
    check(gpp, prob, occ="occupied")
