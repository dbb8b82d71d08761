"""The workloads whose speed counts: what users of the library have it do, through its Python entry points.

A case is one kind of call on one grid. Kinds:
  filter   G applied to a batch of fields (the filter itself, as a flow code or a data generator calls it)
  solve    the deconvolution of a batch of equal fields by one method, in physical or spectral space
  batched  the deconvolution of a list of fields of uneven size in one call
  closure  the sub-filter stress of a deconvolved velocity
  infer    the learned initial guess of a batch of 3D fields
  grad     loss and weight gradient of the learned guess, one training minibatch

Solves run a fixed number of passes (tol = 0), as structural closures use them: the pass count is then an input, and
few enough passes for the Krylov iterates to be determined by their inputs rather than by rounding.
"""

import math

import torch

import paper_1707_09177_gb300 as gad

TAPS, CH = 27, 32


def listed():
    return [
        # one small double-precision field filtered: the smallest call, the cost of a call itself
        {"name": "filter_2d_128_f64", "kind": "filter", "shape": "128x128", "batch": 1, "dtype": "f64", "gamma": 0.1},
        # the paper's Van Cittert closure on a small vorticity field, double precision, 20 passes
        {"name": "vc_2d_128_f64", "kind": "solve", "shape": "128x128", "batch": 1, "dtype": "f64", "gamma": 0.1,
         "method": "vancittert", "space": "physical", "passes": 20},
        # one coarse 2D snapshot (the paper's 256^2 LES grid): a latency-bound Krylov solve
        {"name": "cg_2d_256_f32", "kind": "solve", "shape": "256x256", "batch": 1, "dtype": "f32", "gamma": 0.1,
         "method": "cg", "space": "physical", "passes": 5},
        # a velocity on an anisotropic box whose sides have factors 3
        {"name": "filter_3d_ragged_f32", "kind": "filter", "shape": "96x72x144", "batch": 3, "dtype": "f32",
         "gamma": 0.1},
        # the benchmark's ensemble: 16 snapshots of the paper's fine 2D grid
        {"name": "bicgstab_2d_2048x16_f32", "kind": "solve", "shape": "2048x2048", "batch": 16, "dtype": "f32",
         "gamma": 0.01, "method": "bicgstab", "space": "physical", "passes": 3},
        # the three velocity components of the paper's fine 3D grid: the largest call
        {"name": "bicgstab_3d_512x3_f32", "kind": "solve", "shape": "512x512x512", "batch": 3, "dtype": "f32",
         "gamma": 0.01, "method": "bicgstab", "space": "physical", "passes": 3},
        # preconditioned CG of a velocity, the passes it takes to 1e-5
        {"name": "pcg_3d_256x3_f32", "kind": "solve", "shape": "256x256x256", "batch": 3, "dtype": "f32",
         "gamma": 0.1, "method": "pcg", "space": "physical", "passes": 5},
        # 12 fields of uneven size, 2D and 3D, in one call
        {"name": "bicgstab_uneven_f32", "kind": "batched", "sizes": "256,768,1024,1536,2304,4096;64,64,96,128,192,288",
         "gamma": 0.1, "method": "bicgstab", "space": "physical", "passes": 3},
        # the ensemble of fine 2D snapshots iterated on its half spectra
        {"name": "bicgstab_spectral_2048x16_f32", "kind": "solve", "shape": "2048x2048", "batch": 16, "dtype": "f32",
         "gamma": 0.01, "method": "bicgstab", "space": "spectral", "passes": 3},
        # the closure stress of a 3D velocity: six pairs
        {"name": "closure_3d_256_f32", "kind": "closure", "shape": "256x256x256", "batch": 1, "dtype": "f32",
         "gamma": 0.1},
        # the learned guess for a 3D velocity (bf16 tensor-core layers)
        {"name": "infer_3d_256x3", "kind": "infer", "shape": "256x256x256", "batch": 3, "gamma": 0.1},
        # one training minibatch of the learned guess: eight 64^3 pairs
        {"name": "grad_3d_64x8", "kind": "grad", "shape": "64x64x64", "batch": 8, "gamma": 0.01},
    ]


# --- drawn cases ------------------------------------------------------------

def _sides(lo, hi):
    return sorted(2 ** a * 3 ** b for b in range(3) for a in range(2, 13) if lo <= 2 ** a * 3 ** b <= hi)


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(rng, lo, hi):
    x = _log_uniform(rng, lo, hi)
    return min(_sides(lo, hi), key=lambda n: abs(math.log(n / x)))


def _grid(rng, most):
    """A 2D or 3D shape and a batch of at most `most` points in all, the points spread over their logarithm."""
    while True:
        if rng.random() < 0.5:
            shape = [_side(rng, 64, 4096) for _ in range(2)]
        else:
            shape = [_side(rng, 24, 512) for _ in range(3)]
        points = math.prod(shape)
        batch = int(_log_uniform(rng, 1, 32))
        if points * batch <= most and max(shape) <= 4 * min(shape):
            return shape, batch


def draw(rng):
    kind = rng.choice(["filter", "filter", "solve", "solve", "solve", "solve", "batched", "closure", "infer", "grad"])
    case = {"kind": kind}
    if kind in ("infer", "grad"):
        sides = [_side(rng, 24, 192) for _ in range(2)]
        x = rng.choice([32, 64, 96, 128, 256] if kind == "infer" else [32, 64, 96, 128])
        batch = max(1, min(rng.randint(1, 8), (48 << 20 if kind == "infer" else 8 << 20) // (math.prod(sides) * x)))
        case.update(shape="%dx%dx%d" % (sides[0], sides[1], x), batch=batch, gamma=rng.choice([0.01, 0.1]))
        return case
    if kind == "batched":
        two = [_side(rng, 64, 2304) for _ in range(rng.randint(1, 6))]
        three = [_side(rng, 24, 256) for _ in range(rng.randint(1, 6))]
        case.update(sizes=",".join(map(str, two)) + ";" + ",".join(map(str, three)), gamma=0.1,
                    method=rng.choice(["vancittert", "cg", "bicgstab"]), space=rng.choice(["physical", "spectral"]),
                    passes=rng.randint(1, 3))
        return case
    shape, batch = _grid(rng, {"filter": 256 << 20, "solve": 96 << 20, "closure": 24 << 20}[kind])
    dtype = rng.choice(["f32", "f32", "f32", "f64"])
    if dtype == "f64":
        batch = max(1, batch // 4)
    case.update(shape="x".join(map(str, shape)), batch=batch, dtype=dtype, gamma=0.01 if max(shape) >= 512 else 0.1)
    if kind == "solve":
        methods = ["vancittert", "cg", "bicgstab", "sd"] + (["pcg"] if case["gamma"] == 0.1 else [])
        method = rng.choice(methods)
        case.update(method=method, space=rng.choice(["physical", "physical", "spectral"]),
                    passes=rng.randint(1, 12 if method == "vancittert" else 4 if method == "cg" else 3))
    return case


# --- inputs -----------------------------------------------------------------

def _shape(text):
    return tuple(int(n) for n in text.split("x"))


def _shapes(case):
    two, three = case["sizes"].split(";")
    return [(int(n),) * 2 for n in two.split(",")] + [(int(n),) * 3 for n in three.split(",")]


def _k2(shape):
    """|k|^2 of the integer wavenumbers on the rfft half grid, float64."""
    k2 = None
    for d, n in enumerate(shape):
        f = torch.fft.rfftfreq(n, 1.0 / n) if d == len(shape) - 1 else torch.fft.fftfreq(n, 1.0 / n)
        view = [1] * len(shape)
        view[d] = -1
        f = f.to("cuda", torch.float64).reshape(view) ** 2
        k2 = f if k2 is None else k2 + f
    return k2


def _ghat(shape, gamma):
    kc2 = (gamma * min(shape) / 2.0) ** 2
    return 1.0 / (1.0 + _k2(shape) / kc2)


def _field(shape, gen, gamma=None):
    """One random field of unit RMS and zero mean with the turbulence spectrum of the repository's workloads (2D: k^-3 beyond
    k = 10, cut at 600; 3D: k^-5/3 beyond k = 4, cut at 100), filtered by G when gamma is given; and the same unfiltered."""
    k2 = _k2(shape)
    k = torch.sqrt(k2)
    if len(shape) == 2:
        x2, shell = k2 / 100.0, 2.0 * math.pi * k
        e = x2 ** 2 / (1.0 + x2) ** 3.5 * torch.exp(-k2 / 600.0 ** 2)
    else:
        x2, shell = k2 / 16.0, 4.0 * math.pi * k2
        e = x2 ** 2 / (1.0 + x2) ** (17.0 / 6.0) * torch.exp(-k2 / 100.0 ** 2)
    amp = torch.where(k2 > 0, torch.sqrt(e / torch.where(k2 > 0, shell, torch.ones_like(k2))), torch.zeros_like(k2))
    h = torch.fft.rfftn(torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)) * amp
    u = torch.fft.irfftn(h, s=shape)
    scale = 1.0 / torch.sqrt(torch.mean(u * u))
    if gamma is None:
        return u * scale, None
    return torch.fft.irfftn(h * _ghat(shape, gamma), s=shape) * scale, u * scale


def _batch(shape, n, gen, dtype, gamma=None):
    out = torch.empty((n,) + shape, device="cuda", dtype=dtype)
    raw = torch.empty_like(out) if gamma is not None else None
    for i in range(n):
        a, b = _field(shape, gen, gamma)
        out[i] = a
        if raw is not None:
            raw[i] = b
    return out, raw


def _weights(gen):
    """Network weights where training starts: the 7-point inverse stencil carried by two channels, and He noise."""
    sizes, fans = [TAPS * CH, TAPS * CH * CH, TAPS * CH * CH, TAPS * CH], [27, 27 * CH, 27 * CH, 27 * CH]
    w = [torch.randn(n, generator=gen, device="cuda") * (0.1 * math.sqrt(2.0 / f)) for n, f in zip(sizes, fans)]
    w1, w2, w3, w4 = w[0].view(TAPS, CH), w[1].view(TAPS, CH, CH), w[2].view(TAPS, CH, CH), w[3].view(TAPS, CH)
    w1[:, :2] = 0.0
    w4[:, :2] = 0.0
    for tap, c in [(13, -6.0)] + [(t, 1.0) for t in (4, 22, 10, 16, 12, 14)]:
        w1[tap, 0], w1[tap, 1] = c, -c
    for m in (w2, w3):
        m[:, :, :2] = 0.0
        m[13, 0, 0] = m[13, 1, 1] = 1.0
    w4[13, 0], w4[13, 1] = -1.0, 1.0
    return torch.cat(w)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    state = {"case": case}
    kind, dtype = case["kind"], torch.float64 if case.get("dtype") == "f64" else torch.float32
    if kind == "batched":
        state["fields"] = [_batch(s, 1, gen, torch.float32, case["gamma"])[0][0] for s in _shapes(case)]
        return state
    shape, n = _shape(case["shape"]), case["batch"]
    if kind == "filter":
        state["u"] = _batch(shape, n, gen, dtype)[0]
    elif kind == "closure":
        ubar, u = _batch(shape, n * len(shape), gen, dtype, case["gamma"])
        lead = (n, len(shape)) + shape
        state["ubar"], state["ustar"] = ubar.view(lead), u.view(lead)
    elif kind == "solve":
        state["ubar"] = _batch(shape, n, gen, dtype, case["gamma"])[0]
    else:
        state["ubar"], state["utrue"] = _batch(shape, n, gen, torch.float32, case["gamma"])
        state["weights"] = _weights(gen)
    return state


# --- one pass ---------------------------------------------------------------

def run(state):
    case = state["case"]
    kind, gamma = case["kind"], case["gamma"]
    if kind == "batched":
        u, its, status, _ = gad.deconvolve_batched(state["fields"], [gamma] * len(state["fields"]),
                                                   method=case["method"], tol=0.0, maxit=case["passes"],
                                                   history=False, space=case["space"])
        return {"u": u, "iterations": its, "status": status}
    ndim = len(_shape(case["shape"]))
    if kind == "filter":
        return gad.filter(state["u"], gamma, ndim=ndim)
    if kind == "closure":
        return gad.closure(state["ubar"], state["ustar"], gamma, ncomp=ndim, ndim=ndim)
    if kind == "infer":
        return gad.guess_infer(state["weights"], state["ubar"], gamma)
    if kind == "grad":
        loss, grad = gad.guess_grad(state["weights"], state["ubar"], state["utrue"], gamma)
        return {"loss": loss, "grad": grad}
    double = case["dtype"] == "f64"
    res = gad.deconvolve(state["ubar"], gamma, method=case["method"], tol=0.0, maxit=case["passes"], ndim=ndim,
                         history=double, space=case["space"])
    out = {"u": res.u, "iterations": res.iterations, "status": res.status}
    if double:
        out["history"] = res.history
    return out


# --- what a pass cannot do without ------------------------------------------

def _fft_flops(points):
    return 5.0 * points * math.log2(points)          # a real transform and its inverse: 2.5 P log2 P each


def work(case):
    kind, real = case["kind"], 8 if case.get("dtype") == "f64" else 4
    per_pass = {"vancittert": (1, 4), "sd": (1, 8), "cg": (1, 10), "pcg": (1, 24), "bicgstab": (2, 22)}
    if kind == "batched":
        ng, nv = per_pass[case["method"]]
        points = [math.prod(s) for s in _shapes(case)]
        return {"bytes": 8.0 * sum(points),
                "flops": sum(case["passes"] * (ng * _fft_flops(p) + nv * p) + _fft_flops(p) for p in points)}
    shape, n = _shape(case["shape"]), case["batch"]
    p = math.prod(shape)
    if kind == "filter":
        return {"bytes": 2.0 * real * n * p, "flops": n * _fft_flops(p)}
    if kind == "closure":
        c = len(shape)
        pairs = c * (c + 1) // 2
        return {"bytes": real * n * p * (2.0 * c + pairs), "flops": n * pairs * (_fft_flops(p) + 3.0 * p)}
    if kind in ("infer", "grad"):
        flops = 2.0 * TAPS * (2 * CH + 2 * CH * CH) * n * p
        return {"bytes": 8.0 * n * p, "flops": flops * (3.0 if kind == "grad" else 1.0)}
    ng, nv = per_pass[case["method"]]
    if case["space"] == "spectral":
        flops = _fft_flops(p) + case["passes"] * nv * p
    else:
        flops = _fft_flops(p) + case["passes"] * (ng * _fft_flops(p) + nv * p)
    return {"bytes": 2.0 * real * n * p, "flops": n * flops}


# --- the same in 64 bits, in plain torch ------------------------------------

def _apply(x, g):
    return torch.fft.irfftn(torch.fft.rfftn(x) * g, s=x.shape)


def _dot(a, b):
    return float(torch.sum(a * b))


def _precondition(r, kc):
    z = r.clone()
    for d, n in enumerate(r.shape):
        z += (n / (2.0 * math.pi * kc)) ** 2 * (2.0 * r - torch.roll(r, 1, d) - torch.roll(r, -1, d))
    return z


def _solve(ubar, gamma, method, passes):
    """u after `passes` passes of the paper's Algorithms 1-4 (or of CG preconditioned by the finite-difference inverse of G) from
    u = u_bar, and the residual norms by ||u_bar - G u_bar||."""
    g, kc = _ghat(ubar.shape, gamma), gamma * min(ubar.shape) / 2.0
    u = ubar.clone()
    r = ubar - _apply(ubar, g)
    norm = [math.sqrt(_dot(r, r))]
    p = q = None
    f0, rho, alpha, omega = r.clone(), _dot(r, r), 1.0, 1.0
    for n in range(passes):
        if method == "vancittert":
            u += r
            r = r - _apply(r, g)
        elif method == "sd":
            d = _apply(r, g)
            alpha = _dot(r, r) / _dot(r, d)
            u += alpha * r
            r = r - alpha * d
        elif method in ("cg", "pcg"):
            z = _precondition(r, kc) if method == "pcg" else r
            new = _dot(r, z)
            p = z.clone() if n == 0 else z + (new / rho) * p
            rho = new
            d = _apply(p, g)
            alpha = rho / _dot(p, d)
            u += alpha * p
            r = r - alpha * d
        else:
            if n:
                new = _dot(f0, r)
                p = r + (new / rho) * (alpha / omega) * (p - omega * q)
                rho = new
            else:
                p = r.clone()
            q = _apply(p, g)
            alpha = rho / _dot(f0, q)
            s = r - alpha * q
            t = _apply(s, g)
            omega = _dot(s, t) / _dot(t, t)
            u += alpha * p + omega * s
            r = s - omega * t
        norm.append(math.sqrt(_dot(r, r)))
    return u, [x / norm[0] for x in norm]


def _conv(h, w):
    """Periodic 3x3x3 convolution of channels-last h [Z, Y, X, in] with w [27, in, out]."""
    out = None
    for tap in range(TAPS):
        a, b, c = tap // 9, tap // 3 % 3, tap % 3
        t = torch.roll(h, (1 - a, 1 - b, 1 - c), (0, 1, 2)) @ w[tap]
        out = t if out is None else out + t
    return out


def _network(weights, ubar, gamma):
    cut = [0, TAPS * CH, TAPS * CH * (1 + CH), TAPS * CH * (1 + 2 * CH), TAPS * CH * (2 + 2 * CH)]
    w1, w2, w3, w4 = (weights[a:b] for a, b in zip(cut, cut[1:]))
    sigma = torch.sqrt(torch.mean(ubar * ubar))
    h = (ubar / sigma).unsqueeze(-1)
    for w in (w1.view(TAPS, 1, CH), w2.view(TAPS, CH, CH), w3.view(TAPS, CH, CH)):
        h = torch.relu(_conv(h, w))
    return ubar + sigma / (math.pi * gamma) ** 2 * _conv(h, w4.view(TAPS, CH, 1)).squeeze(-1)


def exact(case, seed):
    state = prepare(case, seed)
    kind, gamma = case["kind"], case["gamma"]
    if kind == "batched":
        u = [_solve(x.double(), gamma, case["method"], case["passes"])[0] for x in state["fields"]]
        return {"u": u, "iterations": None, "status": None}
    shape, n = _shape(case["shape"]), case["batch"]
    if kind == "filter":
        g = _ghat(shape, gamma)
        return torch.stack([_apply(x.double(), g) for x in state["u"]])
    if kind == "closure":
        g, c = _ghat(shape, gamma), len(shape)
        out = torch.empty((n, c * (c + 1) // 2) + shape, device="cuda", dtype=torch.float64)
        for v in range(n):
            ub, us, k = state["ubar"][v].double(), state["ustar"][v].double(), 0
            for i in range(c):
                for j in range(i, c):
                    out[v, k] = ub[i] * ub[j] - _apply(us[i] * us[j], g)
                    k += 1
        return out
    if kind == "infer":
        w = state["weights"].double()
        return torch.stack([_network(w, x.double(), gamma) for x in state["ubar"]])
    if kind == "grad":
        w = state["weights"].double().requires_grad_()
        total = 0.0
        for x, t in zip(state["ubar"], state["utrue"]):
            x, t = x.double(), t.double()
            loss = torch.sum((_network(w, x, gamma) - t) ** 2) / torch.sum(t * t) / n
            loss.backward()
            total += float(loss.detach())
        return {"loss": total, "grad": w.grad}
    u = torch.empty_like(state["ubar"], dtype=torch.float64)
    hist = []
    for i, x in enumerate(state["ubar"]):
        u[i], h = _solve(x.double(), gamma, case["method"], case["passes"])
        hist.append(h)
    out = {"u": u, "iterations": None, "status": None}
    if case["dtype"] == "f64":
        out["history"] = torch.tensor(hist, device="cuda", dtype=torch.float64)
    return out
