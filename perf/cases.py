"""Performance cases: what a user of the library has it do, through its public entry points.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges, ``prepare(case,
seed)`` the inputs and handles that a program holds before the call, ``run(state)`` one pass,
``work(case)`` the bytes and operations a pass cannot do without, and ``exact(case, seed)`` what
``run`` returns for the same inputs, from plain torch in 64 bits.

Kinds of case:
  fit     loss and gradient of one field (a call of an optimiser that lives outside the library)
  steps   a fit from its starting point: n AdaBelief updates inside the library
  batch   loss and gradient of many uneven fields in one call
  renew   a batch whose data, noise and PSFs are replaced before its evaluation (the first
          evaluation of every new set of fields: folding and spectra of the PSFs included)
  psf     loss and gradient of a PSF reconstruction from star cutouts
  noise   the Monte Carlo prior weights of one field

The loss is evaluated in FP32 arithmetic (its sums are accumulated beyond that), so it is taken
in single precision, like the gradient.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2402_08725_gb300.binding import Batch, Problem, noise_weights, optim_cfg

# noise level per detail plane of the B3 starlet for unit white noise (published table)
_STARLET_NOISE = (0.8908, 0.2007, 0.0856, 0.0413, 0.0205, 0.0103, 0.0052, 0.0026)
_SIZES = (32, 48, 64, 96, 128)  # stamp sizes of survey batches


def listed():
    return [
        # the smallest fit: four epochs of a supernova stamp; latency and launches are its cost
        {"name": "fit_4x32", "kind": "fit", "E": 4, "N": 32, "f": 2, "K": 64, "M": 2, "J": 4, "lam": 3.0},
        # the ordinary fit: a lensed quasar, four images, 300 epochs of LSST-like seeing
        {"name": "fit_300x64", "kind": "fit", "E": 300, "N": 64, "f": 2, "K": 64, "M": 4, "J": 4, "lam": 2.0},
        # a ragged one with the prior on the point sources (Eq. 11's third term): odd stamp, odd
        # PSF, supersampling 3, a source count that is no power of two
        {"name": "fit_pts_37x45", "kind": "fit", "E": 37, "N": 45, "f": 3, "K": 51, "M": 3, "J": 5, "lam": 2.0,
         "pts": 1.0},
        # stamps beyond the sizes whose transforms fit in shared memory
        {"name": "fit_12x210", "kind": "fit", "E": 12, "N": 210, "f": 2, "K": 65, "M": 6, "J": 5, "lam": 2.0},
        # the wide field: six frames of 512x512, large PSFs, forty compact sources on an arc
        {"name": "fit_6x512", "kind": "fit", "E": 6, "N": 512, "f": 3, "K": 255, "M": 40, "J": 6, "lam": 2.0},
        # dithered and rotated frames (each with its own shift and angle of the extended channel)
        {"name": "fit_rot_24x64", "kind": "fit", "E": 24, "N": 64, "f": 2, "K": 64, "M": 2, "J": 4, "lam": 2.0,
         "rot": True},
        # a whole light-curve fit: 1000 epochs of 32x32, twenty updates from the starting point
        {"name": "steps_1000x32", "kind": "steps", "E": 1000, "N": 32, "f": 2, "K": 64, "M": 1, "J": 4, "lam": 2.0,
         "n_steps": 20},
        # a night's uneven batch: 256 supernova + host fields of 10 to 500 epochs
        {"name": "batch_256", "kind": "batch", "n": 256, "shapes": 4, "N_max": 128, "E_min": 10, "E_max": 500},
        # a small batch of small stamps, as one filter of one night gives
        {"name": "batch_24", "kind": "batch", "n": 24, "shapes": 9, "N_max": 64, "E_min": 10, "E_max": 60},
        # new inputs for a batch, then its evaluation
        {"name": "renew_32", "kind": "renew", "n": 32, "shapes": 5, "N_max": 128, "E_min": 10, "E_max": 120},
        # PSF reconstruction from 16 stars on a 128x128 fine grid
        {"name": "psf_16x64", "kind": "psf", "S": 16, "N": 64, "f": 2, "J": 5, "lam": 2.0},
        # prior weights of the 300-epoch field, the 5000 realisations of App. B
        {"name": "noise_5000x64", "kind": "noise", "E": 300, "N": 64, "f": 2, "K": 64, "J": 4, "n_real": 5000},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("fit", "fit", "fit", "wide", "rot", "steps", "batch", "renew", "psf", "noise"))
    if kind == "fit":
        case = {"kind": "fit", "E": _logint(rng, 2, 500), "N": rng.randint(20, 128), "f": rng.choice((1, 2, 2, 3)),
                "K": rng.randint(21, 64), "M": rng.randint(0, 4), "J": rng.randint(3, 5), "lam": 2.0}
        if case["f"] == 3:  # fine grids up to 256 pixels
            case["N"] = min(case["N"], 85)
        if case["M"] and rng.random() < 0.3:
            case["pts"] = 1.0
        return case
    if kind == "wide":
        return {"kind": "fit", "E": rng.randint(2, 8), "N": rng.randint(140, 512), "f": rng.choice((2, 3)),
                "K": rng.randint(49, 255), "M": _logint(rng, 1, 40), "J": rng.randint(4, 6), "lam": 2.0}
    if kind == "rot":
        return {"kind": "fit", "E": _logint(rng, 2, 40), "N": rng.randint(24, 96), "f": 2, "K": rng.randint(21, 64),
                "M": rng.randint(1, 4), "J": rng.randint(3, 5), "lam": 2.0, "rot": True}
    if kind == "steps":
        return {"kind": "steps", "E": _logint(rng, 20, 1000), "N": rng.randint(24, 64), "f": 2,
                "K": rng.randint(31, 64), "M": rng.randint(1, 4), "J": 4, "lam": 2.0, "n_steps": rng.randint(5, 20)}
    if kind in ("batch", "renew"):
        return {"kind": kind, "n": _logint(rng, 4, 128), "shapes": rng.randint(100, 10 ** 6),
                "N_max": rng.choice(_SIZES[1:]), "E_min": 10, "E_max": _logint(rng, 20, 200)}
    if kind == "psf":
        return {"kind": "psf", "S": _logint(rng, 3, 64), "N": rng.randint(20, 96), "f": rng.choice((2, 2, 3)),
                "J": rng.randint(3, 5), "lam": 2.0}
    return {"kind": "noise", "E": _logint(rng, 4, 300), "N": rng.randint(24, 72), "f": rng.choice((1, 2, 2)),
            "K": rng.randint(21, 64), "J": rng.randint(3, 4), "n_real": _logint(rng, 300, 5000)}


# --- inputs -----------------------------------------------------------------------------------
def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)


def _uniform(g, lo, hi, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32) * (hi - lo) + lo


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def _offsets(n, c):
    return torch.arange(n, device="cuda", dtype=torch.float32) - c


def _psfs(g, E, K):
    """[E][K][K] narrow PSFs of unit sum, each epoch its own width and wing; the wide ones carry an
    aberration (a smooth 5 % field), as space-telescope PSFs do."""
    fwhm, beta = _uniform(g, 3.0, 9.0 if K < 100 else 5.0, E, 1, 1), _uniform(g, 2.0, 4.0, E, 1, 1)
    alpha = fwhm / (2.0 * torch.sqrt(2.0 ** (1.0 / beta) - 1.0))
    r2 = _offsets(K, K // 2)[:, None] ** 2 + _offsets(K, K // 2)[None, :] ** 2
    s = (1.0 + r2[None] / alpha ** 2) ** (-beta)
    if K >= 100:
        rough = _normal(g, E, 1, K // 4 + 2, K // 4 + 2)
        rough = torch.nn.functional.interpolate(rough, size=(K, K), mode="bilinear", align_corners=False)[:, 0]
        s = s * (1.0 + 0.05 * rough)
    return (s / s.sum(dim=(1, 2), keepdim=True)).contiguous(), fwhm.reshape(E)


def _field(seed, salt, c):
    """One field: data, noise, PSFs, prior weights and the packed parameters of an evaluation near
    its solution (the point a fit spends its time at)."""
    g = _gen(seed, salt)
    E, N, f, K, M, J = c["E"], c["N"], c["f"], c["K"], c["M"], c["J"]
    F = f * N
    s, fwhm = _psfs(g, E, K)
    fwhm_d = torch.sqrt(fwhm ** 2 + 4.0) / f  # seeing on the data grid
    # host: a disc and a bulge with a texture, on a faint noise floor as a reconstructed image has
    u = _offsets(F, (F - 1) / 2.0)
    rr = torch.sqrt(u[:, None] ** 2 / 0.6 + u[None, :] ** 2)
    h = 40.0 * torch.exp(-rr / (0.10 * F)) + 60.0 * torch.exp(-rr / (0.03 * F + 1.0))
    h = h * (1.0 + 0.1 * _normal(g, F, F)) + 0.3 * _normal(g, F, F)
    # the host on the data grid at the mean seeing (separable)
    sig = float(0.5 / f + 3.0 / (f * 2.355))
    y = _offsets(N, (N - 1) / 2.0)
    G = torch.exp(-0.5 * ((y[:, None] - u[None, :] / f) / sig) ** 2) / (sig * math.sqrt(2.0 * math.pi))
    hd = G @ h @ G.T
    base = torch.exp(_uniform(g, math.log(1e3), math.log(1e4), 1, M))
    a = base * torch.exp(0.2 * _normal(g, E, M))
    pos = _uniform(g, -N / 6.0, N / 6.0, M, 2)
    delta = (1.0 if c.get("rot") else 0.1) * _normal(g, E, 2)
    model = hd[None].expand(E, N, N).clone()
    s2 = ((fwhm_d / 2.355) ** 2)[:, None, None]
    for k in range(M):
        dx = y[None, None, :] - (pos[k, 0] + delta[:, 0])[:, None, None]
        dy = y[None, :, None] - (pos[k, 1] + delta[:, 1])[:, None, None]
        model += a[:, k, None, None] / (2.0 * math.pi * s2) * torch.exp(-0.5 * (dx * dx + dy * dy) / s2)
    sky = _uniform(g, 3.0, 10.0, E, 1, 1)
    sigma = torch.sqrt(sky ** 2 + model.clamp(min=0.0))
    d = model + sigma * _normal(g, E, N, N)
    level = 6.0 / (f * math.sqrt(E))
    sigma = torch.where(torch.rand((E, N, N), generator=g, device="cuda") < 0.002,
                        torch.full_like(sigma, math.inf), sigma)  # bad pixels are masked
    W = [w * level for w in _STARLET_NOISE[:J - 1]]
    gamma = 0.1 * _normal(g, E)
    params = torch.cat([x.reshape(-1) for x in (h, a, pos, delta, gamma)]).contiguous()
    theta = (2.0 * math.pi) * np.random.default_rng([int(seed) & 0x7FFFFFFF, salt]).random(E) if c.get("rot") else None
    return {"d": d, "sigma": sigma, "s": s, "W": W, "params": params, "theta": theta}


def _problem(c, fd, inputs=True):
    p = Problem("deconv", c["E"], c["N"], c["f"], c["K"], c["M"], c["J"], c["lam"])
    if inputs:
        p.set_data(fd["d"])
        p.set_noise(fd["sigma"])
        p.set_psfs(fd["s"])
    p.set_weights(fd["W"])
    if c.get("pts"):
        p.set_lambda_pts(c["pts"])
    if c.get("rot"):
        p.set_translate_h(True)
        p.set_rotations(fd["theta"])
    return p


def _shapes(c):
    """The fields of a batch: uneven stamps, epochs and starlet depths."""
    r = np.random.default_rng(c["shapes"])
    sizes = [n for n in _SIZES if n <= c["N_max"]]
    return [{"E": int(r.integers(c["E_min"], c["E_max"] + 1)), "N": int(r.choice(sizes)), "f": 2, "K": 64, "M": 1,
             "J": int(r.integers(4, 7)), "lam": 2.0} for _ in range(c["n"])]


def _lrs(c):
    return (0.02, 20.0, 5e-3, 2e-3, 1e-2)


def _stars(seed, c):
    g = _gen(seed)
    S, N, f, J = c["S"], c["N"], c["f"], c["J"]
    F = f * N
    beta, fwhm = 2.5, 3.0
    alpha = fwhm / (2.0 * math.sqrt(2.0 ** (1.0 / beta) - 1.0))
    a = torch.exp(_uniform(g, math.log(1e4), math.log(1e5), S))
    pos = _uniform(g, -1.0, 1.0, S, 2)
    u = _offsets(F, F // 2)
    moff = (1.0 + (u[:, None] ** 2 + u[None, :] ** 2) / alpha ** 2) ** (-beta)
    b = 0.05 * moff / moff.sum() * _normal(g, F, F) + 1e-6 * _normal(g, F, F)
    fw = math.sqrt(fwhm ** 2 + 4.0) / f
    ad = fw / (2.0 * math.sqrt(2.0 ** (1.0 / beta) - 1.0))
    y = _offsets(N, (N - 1) / 2.0)
    dx = y[None, None, :] - pos[:, 0, None, None]
    dy = y[None, :, None] - pos[:, 1, None, None]
    model = a[:, None, None] * (beta - 1.0) / (math.pi * ad * ad) * (1.0 + (dx * dx + dy * dy) / ad ** 2) ** (-beta)
    model = model * (1.0 + 0.05 * _normal(g, 1, N, N))
    sigma = torch.sqrt(100.0 + model)
    t = model + sigma * _normal(g, S, N, N)
    W = [w * 10.0 / (f * math.sqrt(S)) for w in _STARLET_NOISE[:J - 1]]
    shape = torch.tensor([alpha, beta], device="cuda")
    params = torch.cat([x.reshape(-1) for x in (b, shape, a, pos)]).contiguous()
    return {"d": t, "sigma": sigma, "W": W, "params": params}


def _noise_inputs(seed, c):
    g = _gen(seed)
    E, N = c["E"], c["N"]
    sigma = _uniform(g, 3.0, 10.0, E, 1, 1) * (1.0 + 0.3 * torch.rand((1, N, N), generator=g, device="cuda"))
    sigma = torch.where(torch.rand((E, N, N), generator=g, device="cuda") < 0.002, torch.full_like(sigma, math.inf),
                        sigma).contiguous()
    s1 = _psfs(g, 1, c["K"])[0][0].contiguous()
    return sigma, s1


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fit":
        fd = _field(seed, 0, case)
        p = _problem(case, fd)
        return {"kind": kind, "problem": p, "params": fd["params"], "grad": torch.empty_like(fd["params"])}
    if kind == "steps":
        fd = _field(seed, 0, case)
        return {"kind": kind, "problem": _problem(case, fd), "start": fd["params"], "params": fd["params"].clone(),
                "cfg": optim_cfg("adabelief", lr=_lrs(case)), "n_steps": case["n_steps"],
                "losses": torch.empty(case["n_steps"], dtype=torch.float64, device="cuda")}
    if kind in ("batch", "renew"):
        shapes = _shapes(case)
        fields = [_field(seed, i + 1, c) for i, c in enumerate(shapes)]
        probs = [_problem(c, fd) for c, fd in zip(shapes, fields)]
        b = Batch(probs)
        st = {"kind": kind, "batch": b, "params": b.pack([fd["params"] for fd in fields]),
              "losses": torch.empty(len(probs), dtype=torch.float64, device="cuda")}
        st["grad"] = torch.empty_like(st["params"])
        if kind == "renew":
            for key in ("d", "sigma", "s"):
                st[key] = torch.cat([fd[key].reshape(-1) for fd in fields])
        return st
    if kind == "psf":
        sd = _stars(seed, case)
        p = Problem("psf", case["S"], case["N"], case["f"], J=case["J"], lam=case["lam"])
        p.set_data(sd["d"])
        p.set_noise(sd["sigma"])
        p.set_weights(sd["W"])
        return {"kind": kind, "problem": p, "params": sd["params"], "grad": torch.empty_like(sd["params"])}
    sigma, s1 = _noise_inputs(seed, case)
    return {"kind": kind, "case": case, "sigma": sigma, "s1": s1, "seed": int(seed)}


def run(state):
    kind = state["kind"]
    if kind in ("fit", "psf"):
        loss, grad = state["problem"].loss_and_grad(state["params"], state["grad"], sync=False)
        return [loss.float(), grad]
    if kind == "steps":
        p = state["problem"]
        state["params"].copy_(state["start"])
        p.reset_optimizer()
        p.step(state["params"], state["n_steps"], state["cfg"], state["losses"], sync=False)
        return [state["losses"].float(), state["params"]]
    if kind in ("batch", "renew"):
        b = state["batch"]
        if kind == "renew":
            b.set_psfs(state["s"])
            b.set_noise(state["sigma"])
            b.set_data(state["d"])
        total, grad = b.loss_and_grad(state["params"], state["grad"], state["losses"], sync=False)
        return [total.float(), state["losses"].float(), grad]
    c = state["case"]
    W, W_map, _ = noise_weights(c["N"], c["f"], c["K"], c["J"], state["sigma"], state["s1"], c["n_real"],
                                state["seed"])
    return [W, W_map]


# --- bytes and operations of a pass --------------------------------------------------------------
def _fold_size(N, f, K):
    return N + (K + 2 * f) // (2 * f)  # circular size that keeps the stamp free of wrap-around


def _field_work(c, raw=True):
    """Each input read once (data, noise or weights, PSFs, parameters), each output written once;
    the model and its adjoint as transforms of the folded problem, the starlet and its adjoint."""
    E, N, f, K, M, J = c["E"], c["N"], c["f"], c["K"], c["M"], c["J"]
    F, L = f * N, _fold_size(N, f, K)
    n = F * F + E * M + 2 * M + 3 * E
    transforms = 2 * 2.5 * L * L * math.log2(L * L)           # model and adjoint of an epoch
    products = f * f * (L * L / 2) * 2 * 8.0                  # by the phases' kernel spectra
    flops = E * (transforms + products + 12.0 * N * N) + (J - 1) * 40.0 * F * F
    return 4.0 * (2 * E * N * N + E * K * K + 2 * n), flops


def work(case):
    kind = case["kind"]
    if kind in ("fit", "steps"):
        b, fl = _field_work(case)
        k = case.get("n_steps", 1)
        return {"bytes": b * k, "flops": fl * k}
    if kind in ("batch", "renew"):
        w = [_field_work(c) for c in _shapes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "psf":
        S, N, f, J = case["S"], case["N"], case["f"], case["J"]
        F = f * N
        n = F * F + 2 + 3 * S
        return {"bytes": 4.0 * (2 * S * N * N + 2 * n),
                "flops": S * 2 * (2 * 34.0 * F * F) + (J - 1) * 40.0 * F * F}
    E, N, f, K, J, R = case["E"], case["N"], case["f"], case["K"], case["J"], case["n_real"]
    F = f * N
    L = F + K // 2
    return {"bytes": 4.0 * (E * N * N + K * K + (J - 1) * F * F),
            "flops": R * (5.0 * L * L * math.log2(L * L) + 4.0 * L * L + 40.0 * F * F + (J - 1) * 24.0 * F * F)}


# --- the same in 64 bits ---------------------------------------------------------------------------
def _mirror(n, off):
    i = (torch.arange(n, device="cuda") + off).abs()
    return torch.where(i > n - 1, 2 * (n - 1) - i, i)


def _starlet(c0, J):
    """Detail planes of the B3 starlet with whole-sample mirror borders (last two axes)."""
    taps, F, out = (1.0, 4.0, 6.0, 4.0, 1.0), c0.shape[-1], []
    for j in range(J - 1):
        idx = [_mirror(F, (k - 2) * 2 ** j) for k in range(5)]
        x = sum(t / 16.0 * c0.index_select(-1, i) for t, i in zip(taps, idx))
        x = sum(t / 16.0 * x.index_select(-2, i) for t, i in zip(taps, idx))
        out.append(c0 - x)
        c0 = x
    return out


def _prior(img, J, W):
    return sum(w * p.abs().sum() for w, p in zip(W, _starlet(img, J)))


def _f64(x):
    """A 32-bit value as the library takes it, in 64 bits."""
    return float(np.float32(x))


def _gauss(F, centre):
    """1-D factor of the unit Gaussian of FWHM 2 at each centre: [..., F]."""
    u = torch.arange(F, device="cuda", dtype=torch.float64)
    return math.sqrt(math.log(2.0) / math.pi) * torch.exp2(-(u - centre[..., None]) ** 2)


def _warp(h, theta, shift):
    """h seen by frames turned by theta and moved by shift (fine pixels): bilinear, zero outside."""
    F = h.shape[-1]
    u0 = 0.5 * (F - 1)
    u = torch.arange(F, device="cuda", dtype=torch.float64)
    dx = u[None, None, :] - u0 - shift[:, 0, None, None]
    dy = u[None, :, None] - u0 - shift[:, 1, None, None]
    c, s = torch.cos(theta)[:, None, None], torch.sin(theta)[:, None, None]
    qx, qy = u0 + c * dx + s * dy, u0 - s * dx + c * dy
    x0, y0 = torch.floor(qx.detach()), torch.floor(qy.detach())
    tx, ty = qx - x0, qy - y0
    out = 0.0
    for ky, wy in ((0, 1.0 - ty), (1, ty)):
        for kx, wx in ((0, 1.0 - tx), (1, tx)):
            xi, yi = (x0 + kx).long(), (y0 + ky).long()
            ok = (xi >= 0) & (xi < F) & (yi >= 0) & (yi < F)
            v = h[yi.clamp(0, F - 1), xi.clamp(0, F - 1)]
            out = out + torch.where(ok, v, torch.zeros_like(v)) * wy * wx
    return out


def _exact_field(c, fd, params):
    """(loss, gradient) of one field at the packed 64-bit parameters."""
    E, N, f, K, M, J = c["E"], c["N"], c["f"], c["K"], c["M"], c["J"]
    F, o = f * N, K // 2
    n_h = F * F
    x = params.detach().clone().requires_grad_(True)
    P = F + K - 1
    chunk = max(1, int(2 ** 25 // (P * P)))
    W = [_f64(w) for w in fd["W"]]
    total = 0.0

    def parts():
        h = x[:n_h].reshape(F, F)
        a = x[n_h:n_h + E * M].reshape(E, M)
        r = x[n_h + E * M:]
        return h, a, r[:2 * M].reshape(M, 2), r[2 * M:2 * M + 2 * E].reshape(E, 2), r[2 * M + 2 * E:]

    for i in range(0, E, chunk):
        h, a, pos, delta, gamma = parts()
        sl = slice(i, min(E, i + chunk))
        dl = delta[sl]
        if c.get("rot"):
            th = torch.tensor(fd["theta"][sl], device="cuda", dtype=torch.float64)
            th = torch.atan2(torch.sin(th).float().double(), torch.cos(th).float().double())
            img = _warp(h, th, f * dl)
            cs, sn = torch.cos(th), torch.sin(th)
            px = cs[:, None] * pos[None, :, 0] - sn[:, None] * pos[None, :, 1]
            py = sn[:, None] * pos[None, :, 0] + cs[:, None] * pos[None, :, 1]
        else:
            img = h[None]
            px, py = pos[None, :, 0].expand(dl.shape[0], M), pos[None, :, 1].expand(dl.shape[0], M)
        if M:
            gx = _gauss(F, 0.5 * (F - 1) + f * (px + dl[:, 0, None]))
            gy = _gauss(F, 0.5 * (F - 1) + f * (py + dl[:, 1, None]))
            img = img + torch.einsum("ek,eky,ekx->eyx", a[sl], gy, gx)
        S = torch.fft.rfft2(fd["s"][sl].double(), s=(P, P))
        conv = torch.fft.irfft2(torch.fft.rfft2(img, s=(P, P)) * S, s=(P, P))[:, o:o + F, o:o + F]
        m = conv.reshape(-1, N, f, N, f).sum(dim=(2, 4)) + f * f * gamma[sl, None, None]
        w = 1.0 / fd["sigma"][sl].double() ** 2
        part = 0.5 * (w * (fd["d"][sl].double() - m) ** 2).sum()
        part.backward()
        total += float(part.detach())
    h, a, pos, _, _ = parts()
    prior = _f64(c["lam"]) * _prior(h, J, W)
    if c.get("pts") and M:
        gx, gy = _gauss(F, 0.5 * (F - 1) + f * pos[:, 0]), _gauss(F, 0.5 * (F - 1) + f * pos[:, 1])
        prior = prior + c["pts"] * _prior(torch.einsum("k,ky,kx->yx", a.mean(dim=0), gy, gx), J, W)
    prior.backward()
    return total + float(prior.detach()), x.grad


def _exact_psf(c, sd):
    S, N, f, J = c["S"], c["N"], c["f"], c["J"]
    F = f * N
    x = sd["params"].double().requires_grad_(True)
    b = x[:F * F].reshape(F, F)
    alpha, beta = x[F * F], x[F * F + 1]
    a = x[F * F + 2:F * F + 2 + S]
    pos = x[F * F + 2 + S:].reshape(S, 2)
    u = torch.arange(F, device="cuda", dtype=torch.float64) - F // 2
    r2 = u[:, None] ** 2 + u[None, :] ** 2
    s = (beta - 1.0) / (math.pi * alpha ** 2) * (1.0 + r2 / alpha ** 2) ** (-beta) + b
    d = torch.arange(F, device="cuda", dtype=torch.float64)
    lag = d[:, None] - d[None, :]
    c0 = 0.5 * (F - 1) - F // 2
    k0 = math.sqrt(math.log(2.0) / math.pi)
    gx = k0 * torch.exp2(-(lag[None] - (c0 + f * pos[:, 0])[:, None, None]) ** 2)
    gy = k0 * torch.exp2(-(lag[None] - (c0 + f * pos[:, 1])[:, None, None]) ** 2)
    t = a[:, None, None] * (gy @ s[None] @ gx.transpose(1, 2))
    m = t.reshape(S, N, f, N, f).sum(dim=(2, 4))
    w = 1.0 / sd["sigma"].double() ** 2
    loss = 0.5 * (w * (sd["d"].double() - m) ** 2).sum()
    loss = loss + _f64(c["lam"]) * _prior(b, J, [_f64(v) for v in sd["W"]])
    loss.backward()
    return loss.detach(), x.grad


def _exact_steps(c, fd):
    """AdaBelief from zero moments, with the projection a >= 0."""
    E, M, n = c["E"], c["M"], c["n_steps"]
    F = c["f"] * c["N"]
    sizes = (F * F, E * M, 2 * M, 2 * E, E)
    lr = torch.cat([torch.full((k,), _f64(v), device="cuda", dtype=torch.float64) for k, v in zip(sizes, _lrs(c))])
    b1, b2, eps = _f64(0.9), _f64(0.999), _f64(1e-16)
    x = fd["params"].double()
    m, v = torch.zeros_like(x), torch.zeros_like(x)
    losses = []
    for t in range(1, n + 1):
        loss, grad = _exact_field(c, fd, x)
        losses.append(loss)
        m = b1 * m + (1.0 - b1) * grad
        v = b2 * v + (1.0 - b2) * (grad - m) ** 2 + eps
        x = x - lr * (m / (1.0 - b1 ** t)) / (torch.sqrt(v / (1.0 - b2 ** t)) + eps)
        x[F * F:F * F + E * M].clamp_(min=0.0)
    return torch.tensor(losses, dtype=torch.float64), x


def _normals(seed, first, n):
    """Numbers first .. first + n of the library's stream: Philox4x64-10, two Box-Muller pairs of
    24-bit uniforms per block (first and n multiples of 4)."""
    bits = np.random.Philox(counter=(first // 4 - 1) % 2 ** 256, key=int(seed) & (2 ** 64 - 1)).random_raw(n)
    u = torch.from_numpy((bits >> np.uint64(40)).astype(np.int64)).cuda().double().add_(1.0).mul_(2.0 ** -24)
    u = u.reshape(-1, 2, 2)
    rad = torch.sqrt(-2.0 * torch.log(u[..., 0]))
    return torch.stack((rad * torch.cos(2.0 * math.pi * u[..., 1]), rad * torch.sin(2.0 * math.pi * u[..., 1])),
                       dim=-1).reshape(-1)


def _exact_noise(c, seed):
    N, f, K, J, R = c["N"], c["f"], c["K"], c["J"], c["n_real"]
    sigma, s1 = _noise_inputs(seed, c)
    F = f * N
    inv = torch.sqrt((1.0 / sigma.double() ** 2).sum(dim=0))
    inv = inv.repeat_interleave(f, 0).repeat_interleave(f, 1)
    P, o = F + K, K // 2
    S = torch.fft.rfft2(s1.double(), s=(P, P)).conj()
    sums = torch.zeros((J - 1, 2, F, F), device="cuda", dtype=torch.float64)
    step = max(4, int(2 ** 23 // (F * F)) // 4 * 4)  # a multiple of 4 realisations: whole blocks
    for r in range(0, R, step):
        k = min(step, R - r)
        pad = (-k * F * F) % 4
        z = _normals(seed, r * F * F, k * F * F + pad)[:k * F * F].reshape(k, F, F) * inv
        y = torch.fft.irfft2(torch.fft.rfft2(z, s=(P, P)) * S, s=(P, P))
        y = torch.roll(y, (o, o), dims=(1, 2))[:, :F, :F]
        for j, w in enumerate(_starlet(y, J)):
            sums[j, 0] += w.sum(dim=0)
            sums[j, 1] += (w * w).sum(dim=0)
    var = (sums[:, 1] - sums[:, 0] ** 2 / R) / (R - 1)
    t0, t1, n = sums[:, 0].sum(dim=(1, 2)), sums[:, 1].sum(dim=(1, 2)), R * F * F
    return torch.sqrt((t1 - t0 * t0 / n) / (n - 1)), torch.sqrt(var.clamp(min=0.0))


def exact(case, seed):
    kind = case["kind"]
    if kind == "fit":
        fd = _field(seed, 0, case)
        loss, grad = _exact_field(case, fd, fd["params"].double())
        return [torch.tensor(loss, dtype=torch.float64), grad]
    if kind == "steps":
        return list(_exact_steps(case, _field(seed, 0, case)))
    if kind in ("batch", "renew"):
        losses, grads = [], []
        for i, c in enumerate(_shapes(case)):
            fd = _field(seed, i + 1, c)
            loss, grad = _exact_field(c, fd, fd["params"].double())
            losses.append(loss)
            grads.append(grad)
        losses = torch.tensor(losses, dtype=torch.float64)
        return [losses.sum(), losses, torch.cat(grads)]
    if kind == "psf":
        return list(_exact_psf(case, _stars(seed, case)))
    return list(_exact_noise(case, seed))
