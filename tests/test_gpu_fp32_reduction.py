"""GPU parity of the FP32-bulk tile reduction for every number of frequencies and tile shape.

Tolerance, derived before the first run: a term's FP32 form is right to about eight units of
2^-24, independent from term to term, so an output lies within 2^-21 of the root sum of squares
of its terms; the outputs' own root mean square is of that size to a factor of four.
"""

import numpy as np
import pytest

import oracle
from paper_2008_11326_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -19


@pytest.fixture(scope="module")
def gpp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_11326_gb300 import gpp as g
    return g


@pytest.mark.parametrize("threads", [64, 96, 256])
@pytest.mark.parametrize("nw", [1, 2, 3, 4, 5, 6, 7, 8])
def test_every_value_lands_in_its_place(gpp, nw, threads):
    import torch
    prob = inputs.make_problem(9, 2, 301, 5, nw, seed=nw)
    dp = gpp.DeviceProblem.from_host(prob, device="cuda", c64=True)
    got = gpp.sigma(dp, precision="fp32_bulk", block_threads=threads)
    torch.cuda.synchronize()
    for g, r in zip(got, oracle.sigma(prob)):
        assert np.max(np.abs(g.cpu().numpy() - r)) <= TOL * np.sqrt(np.mean(np.abs(r) ** 2))


# at and past the lines of the default tile depth for few bands, on any count of SMs up to 160:
# the default gives the bits of the depth it stands for
@pytest.mark.parametrize("B,P,G,depth", [(3, 330, 8192, 4), (40, 330, 8065, 4), (41, 330, 8065, 2),
                                         (3, 1300, 8192, 8), (5, 100, 1000, 2)])
def test_default_depth(gpp, B, P, G, depth):
    import torch
    prob = inputs.make_problem(B, 2, G, P, 3, seed=B)
    dp = gpp.DeviceProblem.from_host(prob, device="cuda", c64=True)
    got = gpp.sigma(dp, precision="fp32_bulk")
    want = gpp.sigma(dp, precision="fp32_bulk", ig_per_thread=depth)
    torch.cuda.synchronize()
    for g, w, r in zip(got, want, oracle.sigma(prob)):
        assert torch.equal(g, w)
        assert np.max(np.abs(g.cpu().numpy() - r)) <= TOL * np.sqrt(np.mean(np.abs(r) ** 2))
