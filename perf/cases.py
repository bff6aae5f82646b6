"""The work that a user of this framework has it do, as a list of measurable cases.

A case is one call (or one training step) through the package's public entry points on one
GPP instance or batch: ``gpp.sigma`` (FP64 and FP32-bulk), ``gpp.GppSigma`` / ``gpp.sigma_backward``
(the adjoint), ``gpp.BatchedPlan`` (many instances, a replayed graph) and ``gpp.sigma_host``
(host arrays). Sizes are those of ``inputs.CONFIGS``, ``inputs.batched_shapes`` and the tests.

Inputs follow the distributions of ``inputs.make_problem`` and are drawn on the device.
``exact`` evaluates the written branch formulas with plain torch in 64 bits.
"""

from __future__ import annotations

import math

import torch

from paper_2008_11326_gb300 import gpp

DEVICE = "cuda"


def listed():
    return [
        # the smallest everyday call: the package's "tiny" workload, latency and launches
        dict(name="fp64 tiny", kind="fp64", B=32, P=64, G=512, W=3),
        # an odd, ragged instance with the paper's two frequencies and few occupied bands
        dict(name="fp64 ragged", kind="fp64", B=37, P=95, G=1901, W=2, nvband=11),
        # one ordinary instance: a forward pass at the gradient workload's size
        dict(name="fp64 ordinary", kind="fp64", B=128, P=410, G=8192, W=3),
        # the paper-shaped sum with all of the benchmark's bands (the largest case)
        dict(name="fp64 large", kind="fp64", B=512, P=819, G=16384, W=3),
        # the Sigma code around the kernel: bands on both sides of the level (x of both signs),
        # the screened-exchange cutoff, the half Coulomb hole, occupied bands only in asxtemp
        dict(name="fp64 sigma code", kind="fp64", B=96, P=205, G=4096, W=3, nvband=40,
             signs=True, sexcut=4.0, ch_half=True),
        # the mixed-precision sum at the benchmark's full size, complex64 copy kept by the user
        dict(name="fp32 large", kind="fp32", B=512, P=1638, G=32768, W=3, c64=True),
        # mixed precision at an odd size, the library converting in the call
        dict(name="fp32 ragged", kind="fp32", B=100, P=301, G=6001, W=3),
        # a training step on a small instance: forward and backward through autograd
        dict(name="step tiny", kind="step", B=32, P=64, G=512, W=3),
        # the gradient workload: every gradient of one instance
        dict(name="adjoint", kind="adjoint", B=128, P=410, G=8192, W=3),
        # many uneven instances in one replayed graph, FP64 and mixed precision
        dict(name="batched fp64", kind="batched64", n=12, Bmin=24, Bmax=96, Gmin=1024, Gmax=8192, W=3),
        dict(name="batched fp32", kind="batched32", n=24, Bmin=64, Bmax=256, Gmin=2048, Gmax=16384, W=3),
        # a host code's call: page-locked arrays in, copies overlapped with the sum
        dict(name="host fp64", kind="host", B=64, P=410, G=8192, W=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Most (band, column, G-vector) triples times frequencies of a drawn case, by kind: each stays
# below the time of the largest listed case.
_MOST = {"fp64": 1.0e10, "fp32": 6.0e10, "step": 4.0e8, "adjoint": 1.3e9, "batched64": 3.0e9,
         "batched32": 2.0e10, "host": 1.5e9}


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "fp64", "fp32", "fp32", "step", "adjoint", "batched64",
                       "batched32", "host"])
    W = rng.choice([1, 2, 3, 3, 3, 4])
    if kind.startswith("batched"):
        small = kind == "batched64"
        n = rng.randint(3, 14 if small else 28)
        bmin = _log_int(rng, 6, 64)
        gmin = _log_int(rng, 300, 2048)
        return dict(kind=kind, n=n, Bmin=bmin, Bmax=bmin + rng.randint(1, 64 if small else 192),
                    Gmin=gmin, Gmax=_log_int(rng, gmin + 1, 8192 if small else 16384), W=W)
    while True:
        B = _log_int(rng, 5, 512)
        G = _log_int(rng, 300, 32768)
        P = min(G, max(1, _log_int(rng, G / 60.0 + 1, G / 8.0 + 1)))
        if 1.0e5 <= float(B) * P * G * W <= _MOST[kind]:
            break
    case = dict(kind=kind, B=B, P=P, G=G, W=W)
    if rng.random() < 0.4:
        case["nvband"] = rng.randint(1, B)
    if kind == "fp64" and rng.random() < 0.35:
        case.update(signs=True, sexcut=rng.choice([2.0, 4.0, 8.0]), ch_half=rng.random() < 0.5)
    if kind == "fp32" and rng.random() < 0.5:
        case["c64"] = True
    return case


def _shapes(case):
    """(B, P, G) of every instance of a case; a batch's are spread over its ranges (G over its
    logarithm) in a fixed irregular order, P = G // 20 as in inputs.batched_shapes."""
    if not case["kind"].startswith("batched"):
        return [(case["B"], case["P"], case["G"])]
    n, out = case["n"], []
    for i in range(n):
        f, h = (i * 0.6180339887) % 1.0, (i * 0.7548776662) % 1.0
        G = int(round(case["Gmin"] * (case["Gmax"] / case["Gmin"]) ** f))
        B = case["Bmin"] + int(h * (case["Bmax"] - case["Bmin"] + 1))
        out.append((B, max(1, G // 20), G))
    return out


def _arrays(B, P, G, W, seed, signs=False, nvband=2):
    """The instance's arrays on the device, with the distributions of inputs.make_problem.
    With ``signs`` the band energies span both sides of the level, e_n1 ~ U(0, 20)."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))

    def u(shape, lo, hi):
        return torch.rand(shape, generator=g, dtype=torch.float64, device=DEVICE) * (hi - lo) + lo

    def c(shape, rl, rh, il, ih):
        return torch.complex(u(shape, rl, rh), u(shape, il, ih))

    a = dict(number_bands=B, nvband=nvband, ncouls=G, ngpown=P, nw=W)
    a["aqsmtemp"] = c((B, G), -1.0, 1.0, -1.0, 1.0)
    a["aqsntemp"] = c((B, G), -1.0, 1.0, -1.0, 1.0)
    a["I_eps_array"] = c((P, G), 0.5, 1.5, -0.1, 0.1)
    a["wtilde_array"] = c((P, G), 0.2, 3.0, -0.05, 0.05)
    a["vcoul"] = u((G,), 0.1, 10.0)
    a["inv_igp_index"] = torch.randperm(G, generator=g, device=DEVICE)[:P].to(torch.int32)
    ind = torch.empty(G + 1, dtype=torch.int32, device=DEVICE)
    ind[:G] = torch.randperm(G, generator=g, device=DEVICE).to(torch.int32)
    ind[G] = G
    a["indinv"] = ind
    e_n1 = u((B,), 0.0, 20.0 if signs else 10.0)
    iw = torch.arange(W, dtype=torch.float64, device=DEVICE)
    a["wx_array"] = ((10.0 - e_n1)[:, None] + iw[None, :]).contiguous()
    a["g_ach"] = torch.complex(torch.randn(W, generator=g, dtype=torch.float64, device=DEVICE),
                               torch.zeros(W, dtype=torch.float64, device=DEVICE))
    a["g_asx"] = torch.complex(torch.zeros(W, dtype=torch.float64, device=DEVICE),
                               torch.randn(W, generator=g, dtype=torch.float64, device=DEVICE))
    return a


def _draws(case, seed):
    shapes = _shapes(case)
    return [_arrays(B, P, G, case["W"], seed * len(shapes) + i, bool(case.get("signs")),
                    int(case.get("nvband", 2))) for i, (B, P, G) in enumerate(shapes)]


def _problem(a):
    return gpp.DeviceProblem(**{k: v for k, v in a.items() if k not in ("g_ach", "g_asx")})


def _options(case):
    o = {}
    if case["kind"] in ("fp32", "batched32"):
        o["precision"] = "fp32_bulk"
    if "nvband" in case:
        o["occ_mode"] = "occupied"
    if case.get("sexcut"):
        o["sexcut"] = case["sexcut"]
    if case.get("ch_half"):
        o["ch_half"] = True
    return o


def prepare(case, seed):
    kind, opts = case["kind"], _options(case)
    drawn = _draws(case, seed)
    s = dict(kind=kind, opts=opts)
    if kind.startswith("batched"):
        dps = [_problem(a) for a in drawn]
        if kind == "batched32":
            for d in dps:
                d.make_c64()
        s["plan"] = gpp.BatchedPlan(dps, use_graph=True, **opts)
        return s
    a = drawn[0]
    if kind == "host":
        h = {k: (v.cpu().pin_memory() if torch.is_tensor(v) else v) for k, v in a.items()}
        s["dp"] = _problem(h)
        s["workspace"] = torch.empty(gpp.host_workspace_size(s["dp"], **opts), dtype=torch.uint8,
                                     device=DEVICE)
        s["out"] = tuple(torch.empty(case["W"], dtype=torch.complex128).pin_memory()
                         for _ in range(2))
        return s
    if kind == "step":
        s["leaves"] = [a[k].requires_grad_() for k in ("aqsmtemp", "aqsntemp", "I_eps_array",
                                                       "wtilde_array")]
        s["rest"] = [a[k] for k in ("vcoul", "inv_igp_index", "indinv", "wx_array")]
        s["nvband"] = a["nvband"]
    else:
        s["dp"] = _problem(a)
        if case.get("c64"):
            s["dp"].make_c64()
    s["g"] = (a["g_ach"], a["g_asx"])
    return s


def run(state):
    kind, opts = state["kind"], state["opts"]
    if kind.startswith("batched"):
        return [list(o) for o in state["plan"].run()]
    if kind == "host":
        return list(gpp.sigma_host(state["dp"], workspace=state["workspace"], out=state["out"],
                                   **opts))
    if kind == "adjoint":
        return gpp.sigma_backward(state["dp"], *state["g"], **opts)
    if kind == "step":
        outs = gpp.GppSigma.apply(*state["leaves"], *state["rest"], state["nvband"],
                                  opts.get("occ_mode", "all"))
        grads = torch.autograd.grad(outs, state["leaves"], grad_outputs=state["g"])
        return dict(ach=outs[0].detach(), asx=outs[1].detach(),
                    **{k: v for k, v in zip(("aqsm", "aqsn", "I_eps", "wtilde"), grads)})
    return list(gpp.sigma(state["dp"], **opts))


def work(case):
    """Each input read once, each output written once (of aqsmtemp only the gathered columns);
    operations of the written formulas per (band, column, G-vector) and frequency."""
    W, nbytes, flops = case["W"], 0.0, 0.0
    adj = case["kind"] in ("adjoint", "step")
    esize = 8 if case.get("c64") or case["kind"] == "batched32" else 16
    for B, P, G in _shapes(case):
        n = float(B) * P * G
        nbytes += 16.0 * B * P + esize * float(B) * G + 32.0 * P * G + 12.0 * G + 4.0 * P + 8.0 * B * W + 32.0 * W
        if case["kind"] != "adjoint":
            flops += n * (51.0 * W + 6.0)
        if adj:  # u, v, their squares and four complex products per frequency; M, Q, four sums
            flops += n * (56.0 * W + 44.0)
            nbytes += 32.0 * B * G + 32.0 * P * G
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------
# The written formulas in 64 bits with plain torch.


def _columns(a):
    """(global columns, live mask) of the local columns."""
    G = a["ncouls"]
    g = a["indinv"].long()[a["inv_igp_index"].long()]
    live = (g >= 0) & (g < G)
    return torch.where(live, g, torch.zeros_like(g)), live


def _terms(x, wr, wi, w2abs, sexcut):
    """Per (column, G-vector), for one real frequency x: u = 1/(x - w) and v = 1/(x + w) as
    (re, im), and the masks of branch 1, of branch 2 and of the terms that asxtemp keeps."""
    ar, sr = x - wr, x + wr
    wi2 = wi * wi
    a2, s2 = ar * ar + wi2, sr * sr + wi2
    b1 = (a2 > 0.25) & (w2abs < 250000.0 * a2)
    b2 = ~b1 & (w2abs > 1.0e-12 * a2)
    u = (ar / a2, wi / a2)
    v = (sr / s2, -wi / s2)
    keep = b1 | b2
    if sexcut and x < 0.0:
        big = torch.where(b1, w2abs * w2abs > sexcut * sexcut * a2 * s2,
                          w2abs > 4.0 * sexcut * sexcut * s2)
        keep = keep & ~big
    return u, v, b1, keep


def _cmul(p, q):
    return p[0] * q[0] - p[1] * q[1], p[0] * q[1] + p[1] * q[0]


def _exact_forward(a, opts):
    B, W = a["number_bands"], a["nw"]
    sexcut, occupied = opts.get("sexcut", 0.0), opts.get("occ_mode") == "occupied"
    g, live = _columns(a)
    am = (a["aqsmtemp"][:, g].conj() * a["vcoul"][g]) * live
    wx = a["wx_array"].tolist()
    ach = torch.zeros(W, dtype=torch.complex128, device=DEVICE)
    asx = torch.zeros(W, dtype=torch.complex128, device=DEVICE)
    step = max(1, (1 << 25) // a["ncouls"])  # columns at a time
    for p0 in range(0, a["ngpown"], step):
        wt, eps = a["wtilde_array"][p0:p0 + step], a["I_eps_array"][p0:p0 + step]
        w = (wt.real.contiguous(), wt.imag.contiguous())
        w2abs = w[0] * w[0] + w[1] * w[1]
        iw_ = wt * eps
        Iw = (iw_.real.contiguous(), iw_.imag.contiguous())

        def bilinear(b, t):  # sum over columns and G-vectors of am an (t I w)
            k = torch.complex(*_cmul(t, Iw))
            return (am[b, p0:p0 + step, None] * (k @ a["aqsntemp"][b])[:, None]).sum()

        for b in range(B):
            occ = not occupied or b < a["nvband"]
            for k in range(W):
                u, v, b1, keep = _terms(wx[b][k], *w, w2abs, sexcut)
                ach[k] += bilinear(b, (u[0] * b1, u[1] * b1))
                if occ:  # branch 1: w u v; branch 2: -v / 2 (both times I w)
                    h = _cmul(w, _cmul(u, v))
                    asx[k] += bilinear(b, tuple(
                        torch.where(b1, p, -0.5 * q) * keep for p, q in zip(h, v)))
    if opts.get("ch_half"):
        ach = 0.5 * ach
    return ach, asx


def _exact_adjoint(a, opts):
    B, W = a["number_bands"], a["nw"]
    occupied = opts.get("occ_mode") == "occupied"
    g, live = _columns(a)
    am = (a["aqsmtemp"][:, g].conj() * a["vcoul"][g]) * live
    wx = a["wx_array"].tolist()
    wt, eps, an = a["wtilde_array"], a["I_eps_array"], a["aqsntemp"]
    w = (wt.real.contiguous(), wt.imag.contiguous())
    w2abs = w[0] * w[0] + w[1] * w[1]
    ca, cs = a["g_ach"].conj(), a["g_asx"].conj()
    gw, gI = torch.zeros_like(wt), torch.zeros_like(wt)
    gn, gm = torch.zeros_like(an), torch.zeros_like(a["aqsmtemp"])
    Iw = eps * wt
    for b in range(B):
        GI, GW = torch.zeros_like(wt), torch.zeros_like(wt)
        occ = not occupied or b < a["nvband"]
        for k in range(W):
            x = wx[b][k]
            u, v, b1, keep = _terms(x, *w, w2abs, 0.0)
            u, v = torch.complex(*u), torch.complex(*v)
            u = torch.where(b1, u, torch.zeros_like(u))
            GI += ca[k] * u
            GW += ca[k] * x * u * u
            if occ:
                uv = u * v
                zero = torch.zeros_like(v)
                GI += cs[k] * torch.where(b1, wt * uv, torch.where(keep, -0.5 * v, zero))
                GW += cs[k] * torch.where(b1, 2.0 * x * x * wt * uv * uv,
                                          torch.where(keep, -0.5 * x * v * v, zero))
        M = am[b][:, None] * an[b][None, :]
        gI += M * wt * GI
        gw += M * eps * GW
        Q = Iw * GI
        gn[b] = (am[b][:, None] * Q).sum(0).conj()
        r = (an[b][None, :] * Q).sum(1) * live
        gm[b].index_add_(0, g, a["vcoul"][g] * r)
    return dict(wtilde=gw.conj() * live[:, None], I_eps=gI.conj() * live[:, None], aqsm=gm, aqsn=gn)


def exact(case, seed):
    kind, opts = case["kind"], _options(case)
    if sum(float(B) * P * G for B, P, G in _shapes(case)) * case["W"] > 2.5e10:
        return None  # takes over 20 seconds
    drawn = _draws(case, seed)
    if kind.startswith("batched"):
        return [list(_exact_forward(a, opts)) for a in drawn]
    a = drawn[0]
    if kind == "adjoint":
        return _exact_adjoint(a, opts)
    ach, asx = _exact_forward(a, opts)
    if kind == "step":
        return dict(ach=ach, asx=asx, **_exact_adjoint(a, opts))
    return [ach.cpu(), asx.cpu()] if kind == "host" else [ach, asx]
