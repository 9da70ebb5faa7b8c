"""Performance cases: the transforms, loops and gradients of aberration-space holography through the package's entry points.

A case names an operation, the SLM grid (nx columns, ny rows), the spot count N, the mode count D (Noll 2 .. D + 1) and, where
the operation loops, its iterations. The spots lie on a square lattice over +-0.45 Nyquist; D = 5 and 10 take the piecewise
constant aberrations of 50 isoplanatic patches (sigma 0.5 rad) under a Gaussian illumination, D = 11 five defocus planes in
+-20 rad, smooth aberrations with 0.3 rad noise and a flat-top illumination. Loops and gradients start from the superposition
hologram arg sum_n T_n exp(i theta_n) conj(K_n) with random spot phases, as a program does that starts from a first guess.
"""
import math

import torch

from paper_2505_08777_gb300 import Batch, Hologram
from paper_2505_08777_gb300.autograd import spot_field, spot_intensity_loss

DEVICE = "cuda"
SPAN = 0.45                    # spots lie within this fraction of the Nyquist tilt
MOST_TERMS = 22.2e9            # spot x pixel terms of the largest listed case
OFFSETS = [-1.5, -1.0, -0.5, 0.0, 0.5, 1.0, 1.5]   # calibration sweep, radians


def listed():
    return [
        # one small correction while a user tunes a trap by hand: launches and latency
        {"name": "forward-256", "op": "forward", "nx": 256, "ny": 256, "N": 16, "D": 10},
        # a whole small hologram from a first guess, 4 x 4 tweezers
        {"name": "wgs-256", "op": "wgs", "nx": 256, "ny": 256, "N": 16, "D": 10, "iters": 20},
        # the 20 x 20 tweezer array on a 1024^2 modulator: evaluating a hologram, making one, and the loop that refines it
        {"name": "forward-array", "op": "forward", "nx": 1024, "ny": 1024, "N": 400, "D": 10},
        {"name": "adjoint-array", "op": "adjoint", "nx": 1024, "ny": 1024, "N": 400, "D": 10},
        {"name": "wgs-array", "op": "wgs", "nx": 1024, "ny": 1024, "N": 400, "D": 10, "iters": 10},
        # the 3D lattice of 2000 spots on a full 1920 x 1152 modulator, one superposition and the loop
        {"name": "adjoint-volume", "op": "adjoint", "nx": 1920, "ny": 1152, "N": 2000, "D": 11},
        {"name": "wgs-volume", "op": "wgs", "nx": 1920, "ny": 1152, "N": 2000, "D": 11, "iters": 2},
        # one step of gradient descent on the phase and the aberration coefficients of 32 x 32 spots
        {"name": "autograd-1024", "op": "autograd", "nx": 1024, "ny": 1024, "N": 1024, "D": 10},
        # the same on a region of interest with odd sizes, 3D spots
        {"name": "autograd-ragged", "op": "autograd", "nx": 901, "ny": 611, "N": 230, "D": 11},
        # a measured complex nearfield of odd size (no phase-only nearfield), few modes
        {"name": "field-ragged", "op": "field", "nx": 517, "ny": 389, "N": 131, "D": 5},
        # one order of a calibration: seven offsets of one mode through the system
        {"name": "sweep-array", "op": "sweep", "nx": 1024, "ny": 1024, "N": 400, "D": 10},
        # sixteen uneven small holograms (256^2 to 512^2, 10 to 300 spots) solved together
        {"name": "batch-small", "op": "batch", "count": 16, "shapes": 3, "iters": 5},
    ]


def draw(rng):
    op = rng.choice(["forward", "adjoint", "wgs", "wgs", "autograd", "field", "sweep", "batch"])
    if op == "batch":
        return {"op": op, "count": rng.randint(4, 24), "shapes": rng.randint(10, 1 << 20), "iters": rng.randint(2, 6)}
    while True:
        ny = int(round(math.exp(rng.uniform(math.log(200), math.log(1152)))))
        nx = min(1920, int(round(ny * rng.uniform(0.8, 1.67))))
        N = int(round(math.exp(rng.uniform(math.log(10), math.log(2500)))))
        c = {"op": op, "nx": nx, "ny": ny, "N": N, "D": rng.choice([5, 10, 11])}
        if op == "wgs":
            c["iters"] = rng.randint(2, 12)
        # a hologram has many more pixels than spots
        if N * 60 < nx * ny and terms(c) <= MOST_TERMS:
            return c


# --- the shapes of a case -------------------------------------------------------

def members(case):
    """The (nx, ny, N, D) of a batch's holograms."""
    g = torch.Generator().manual_seed(int(case["shapes"]))
    out = []
    for _ in range(case["count"]):
        n = (256, 384, 512)[int(torch.randint(3, (1,), generator=g))]
        N = int(round(math.exp(float(torch.rand(1, generator=g)) * math.log(30.0) + math.log(10.0))))
        out.append((n, n, N, (5, 10, 11)[int(torch.randint(3, (1,), generator=g))]))
    return out


def passes(case):
    """Transforms (of N x nx ny terms each) in one pass."""
    return {"forward": 1, "adjoint": 1, "field": 1, "autograd": 3, "sweep": len(OFFSETS)}.get(case["op"]) or 2 * case["iters"] + 1


def terms(case):
    if case["op"] == "batch":
        return passes(case) * sum(nx * ny * N for nx, ny, N, _ in members(case))
    return passes(case) * case["nx"] * case["ny"] * case["N"]


def work(case):
    """Bytes: illumination, coefficients and the arrays a pass is given and gives back. Flops: a term is the D-long phase
    product, a sine, a cosine and a complex multiply-accumulate, 2 D + 8 operations with a sine or cosine as one."""
    if case["op"] == "batch":
        b = sum(4 * (3 * nx * ny + N * (D + 3)) for nx, ny, N, D in members(case))
        f = sum((2 * D + 8) * nx * ny * N for nx, ny, N, D in members(case))
        return {"bytes": b, "flops": passes(case) * f}
    M, N, D = case["nx"] * case["ny"], case["N"], case["D"]
    pixel = {"forward": 8, "adjoint": 8, "field": 8, "wgs": 12, "autograd": 12, "sweep": 8}[case["op"]]
    spot = {"forward": 2, "adjoint": 2, "field": 2, "wgs": 5, "autograd": D + 1, "sweep": len(OFFSETS)}[case["op"]]
    return {"bytes": pixel * M + 4 * N * (D + spot), "flops": passes(case) * (2 * D + 8) * M * N}


# --- inputs -----------------------------------------------------------------------

def lattice(g, span):
    t = torch.linspace(-span, span, g, dtype=torch.float64) if g > 1 else torch.zeros(1, dtype=torch.float64)
    v, u = torch.meshgrid(t, t, indexing="ij")
    return torch.stack([u.ravel(), v.ravel()], 1)


def quadratic(p, modes, gen):
    """A smooth random field per mode: a quadratic polynomial of the position with N(0, 0.5 rad) coefficients."""
    cols = [torch.ones(len(p), dtype=torch.float64)] + [p[:, i] for i in range(p.shape[1])]
    cols += [p[:, i] * p[:, j] for i in range(p.shape[1]) for j in range(i, p.shape[1])]
    return lambda: torch.stack(cols, 1) @ (0.5 * torch.randn(len(cols), modes, generator=gen, dtype=torch.float64))


def coefficients(nx, ny, N, D, gen):
    R = min(nx, ny) / 2
    C = torch.zeros(N, D, dtype=torch.float64)
    if D == 11:
        uv = lattice(math.ceil(math.sqrt(N / 5)), SPAN)
        z = torch.linspace(-20, 20, 5, dtype=torch.float64)
        p = torch.cat([torch.cat([uv, torch.full((len(uv), 1), float(d), dtype=torch.float64)], 1) for d in z])[:N]
        C[:, 2] = p[:, 2]
        field = quadratic(p / torch.tensor([SPAN, SPAN, 20.0], dtype=torch.float64), D - 3, gen)()
        C[:, 3:] = field + 0.3 * torch.randn(N, D - 3, generator=gen, dtype=torch.float64)
    else:
        p = lattice(math.ceil(math.sqrt(N)), SPAN)[:N]
        centres = 2 * torch.rand(50, 2, generator=gen, dtype=torch.float64) - 1
        near = torch.cdist(p / SPAN, centres).argmin(1)
        C[:, 2:] = quadratic(centres, D - 2, gen)()[near]
    C[:, :2] = p[:, :2] * math.pi * R
    return C.float().to(DEVICE)


def amplitude(nx, ny, D):
    """Gaussian of waist 0.4 apertures, or flat for the 3D lattice; unit power."""
    i = torch.arange(nx, dtype=torch.float64, device=DEVICE) - (nx - 1) / 2
    j = torch.arange(ny, dtype=torch.float64, device=DEVICE) - (ny - 1) / 2
    r2 = i[None, :] ** 2 + j[:, None] ** 2
    a = torch.ones_like(r2) if D == 11 else torch.exp(-r2 / (0.4 * min(nx, ny)) ** 2)
    return (a / a.square().sum().sqrt()).float()


def hologram(nx, ny, N, D, gen):
    """What every operation starts from: illumination, coefficients, targets, spot values, first guess."""
    p = {"nx": nx, "ny": ny, "D": D, "amp": amplitude(nx, ny, D), "coeff": coefficients(nx, ny, N, D, gen)}
    t = 0.5 + 0.5 * torch.rand(N, generator=gen) if D == 11 else torch.ones(N)
    theta = 2 * math.pi * torch.rand(N, generator=gen)
    p["target"] = t.to(DEVICE)
    p["y"] = torch.polar(t * (0.5 + torch.rand(N, generator=gen)), theta).to(DEVICE)
    p["loss_target"] = (0.5 + torch.rand(N, generator=gen)).to(DEVICE)
    return p


def guess(p):
    """The superposition hologram of the spots y, in 64 bits, as a phase."""
    return adjoint(p, p["coeff"], p["y"]).angle().float()


def prepare(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    if case["op"] == "batch":
        ps = [hologram(*m, gen) for m in members(case)]
        for p in ps:
            p["phase"] = guess(p)
        b = Batch([(p["amp"], p["coeff"], list(range(2, 2 + p["D"]))) for p in ps])
        return {"op": "batch", "iters": case["iters"], "ps": ps, "holo": b,
                "phases": [p["phase"].clone() for p in ps], "weights": [p["target"].clone() for p in ps]}
    p = hologram(case["nx"], case["ny"], case["N"], case["D"], gen)
    if case["op"] == "field":
        g = torch.Generator(device=DEVICE).manual_seed(int(seed))
        p["field"] = p["amp"] * torch.randn(case["ny"], case["nx"], dtype=torch.complex64, device=DEVICE, generator=g)
    elif case["op"] != "adjoint":
        p["phase"] = guess(p)
    s = {"op": case["op"], "p": p, "iters": case.get("iters"),
         "holo": Hologram(p["amp"], p["coeff"], noll=list(range(2, 2 + case["D"])))}
    if case["op"] == "wgs":
        s["phase"], s["weights"] = p["phase"].clone(), p["target"].clone()
    if case["op"] == "autograd":
        s["phase"], s["coeff"] = p["phase"].clone().requires_grad_(), p["coeff"].clone().requires_grad_()
    return s


# --- one pass -----------------------------------------------------------------------

def run(s):
    op, h = s["op"], s["holo"]
    if op == "batch":
        for p, ph, w in zip(s["ps"], s["phases"], s["weights"]):
            ph.copy_(p["phase"])
            w.copy_(p["target"])
        met = h.wgs(s["phases"], s["weights"], [p["target"] for p in s["ps"]], s["iters"])
        return {"metrics": met, "weights": list(s["weights"])}
    p = s["p"]
    if op == "forward":
        return h.forward(p["phase"])
    if op == "field":
        return h.forward_field(p["field"])
    if op == "adjoint":
        return h.adjoint(p["y"])[0]
    if op == "sweep":
        return h.zsub_sweep(p["phase"], 2, OFFSETS)
    if op == "autograd":
        E = spot_field(h, s["phase"], s["coeff"])
        loss = spot_intensity_loss(E, p["loss_target"])
        dphase, dcoeff = torch.autograd.grad(loss, [s["phase"], s["coeff"]])
        return {"loss": loss.detach(), "dphase": dphase, "dcoeff": dcoeff}
    # The loop's phase is the argument of a speckle field: where that is nearly 0, and at the seam of +-pi, it is not
    # determined to any number of digits. E is the transform of the whole phase, so the phase is judged through it.
    s["phase"].copy_(p["phase"])
    s["weights"].copy_(p["target"])
    E, met = h.wgs(s["phase"], s["weights"], p["target"], s["iters"])
    return {"E": E, "metrics": met, "weights": s["weights"]}


# --- the same in 64 bits ---------------------------------------------------------------

def zernike(j, x, y):
    """Noll mode j, peak 1 at the unit circle, from its radial polynomial."""
    n = 0
    while (n + 1) * (n + 2) // 2 < j:
        n += 1
    k = j - n * (n + 1) // 2 - 1
    m = 2 * ((k + 1) // 2) if n % 2 == 0 else 2 * (k // 2) + 1
    rho, th = torch.hypot(x, y), torch.atan2(y, x)
    r = torch.zeros_like(rho)
    f = math.factorial
    for s in range((n - m) // 2 + 1):
        r += (-1) ** s * f(n - s) / (f(s) * f((n + m) // 2 - s) * f((n - m) // 2 - s)) * rho ** (n - 2 * s)
    return r * (torch.cos(m * th) if j % 2 == 0 or m == 0 else torch.sin(m * th))


def kernel_rows(p, C):
    """(first pixel, last pixel, Z (D, pixels), exp(-i C Z)) by chunks of pixels."""
    nx, ny, C = p["nx"], p["ny"], C.double()
    R = min(nx, ny) / 2
    step = max(1, (1 << 24) // len(C))
    for a in range(0, nx * ny, step):
        m = torch.arange(a, min(nx * ny, a + step), device=DEVICE)
        x = ((m % nx).double() - (nx - 1) / 2) / R
        y = (torch.div(m, nx, rounding_mode="floor").double() - (ny - 1) / 2) / R
        Z = torch.stack([zernike(j, x, y) for j in range(2, 2 + p["D"])])
        ph = C @ Z
        yield a, a + len(m), Z, torch.complex(torch.cos(ph), -torch.sin(ph))


def forward(p, C, f):
    return sum(K @ f[a:b] for a, b, _, K in kernel_rows(p, C))


def adjoint(p, C, y):
    return torch.cat([y.to(torch.complex128) @ K.conj() for _, _, _, K in kernel_rows(p, C)]).reshape(p["ny"], p["nx"])


def wgs(p, iters):
    A, C, T = p["amp"].double().ravel(), p["coeff"], p["target"].double()
    E, w = forward(p, C, torch.polar(A, p["phase"].double().ravel())), T.clone()
    for _ in range(iters):
        w = w * (T / T.norm()) / (E.abs() / E.norm())
        w = w / w.norm()
        g = adjoint(p, C, w * torch.exp(1j * E.angle())).ravel()
        E = forward(p, C, torch.polar(A, g.angle()))
    I, q = E.abs() ** 2, E.abs() ** 2 / T ** 2
    met = torch.stack([1 - (q.max() - q.min()) / (q.max() + q.min()), I.sum() / (A.numel() * (A * A).sum()), I.sum(), q.min()])
    return E, met, w


def exact(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    if case["op"] == "batch":
        ps = [hologram(*m, gen) for m in members(case)]
        for p in ps:
            p["phase"] = guess(p)
        r = [wgs(p, case["iters"]) for p in ps]
        return {"metrics": torch.stack([x[1] for x in r]), "weights": [x[2] for x in r]}
    p = hologram(case["nx"], case["ny"], case["N"], case["D"], gen)
    op, C = case["op"], p["coeff"].double()
    A = p["amp"].double().ravel()
    if op == "field":
        g = torch.Generator(device=DEVICE).manual_seed(int(seed))
        f = p["amp"] * torch.randn(case["ny"], case["nx"], dtype=torch.complex64, device=DEVICE, generator=g)
        return forward(p, C, f.to(torch.complex128).ravel())
    if op == "adjoint":
        return adjoint(p, C, p["y"])
    p["phase"] = guess(p)
    f = torch.polar(A, p["phase"].double().ravel())
    if op == "forward":
        return forward(p, C, f)
    if op == "wgs":
        E, met, w = wgs(p, case["iters"])
        return {"E": E, "metrics": met, "weights": w}
    if op == "sweep":
        out = []
        for d in OFFSETS:
            S = C.clone()
            S[:, 2] -= float(torch.tensor(d, dtype=torch.float32))
            out.append(forward(p, S, f).abs() ** 2)
        return torch.stack(out)
    E = forward(p, C, f)
    I, t = E.abs() ** 2, p["loss_target"].double()
    mu = I.mean()
    d = I / mu - t
    dI = 2 * d / mu - 2 * (d * I).sum() / (mu * mu * len(I))
    gE = 2 * dI * E
    dphase, dC = torch.empty_like(A), torch.zeros_like(C)
    for a, b, Z, K in kernel_rows(p, C):
        # dE_n / dphase_m = i K_nm f_m, dE_n / dC_nd = -i sum_m Z_dm K_nm f_m
        q = (gE.conj()[:, None] * K) * f[a:b]
        dphase[a:b] = -q.imag.sum(0)
        dC += q.imag @ Z.T
    return {"loss": d.square().sum(), "dphase": dphase.reshape(p["ny"], p["nx"]), "dcoeff": dC}
