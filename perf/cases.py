"""Performance cases: the calls that a program using the solver makes, over their real range.

A case is one of
  * "product": y = A x, A(chi') A(chi) x, or the same for several vectors at once, on a grid
    of any shape, FP64 or complex64, TE, TM or the three-plane magnetic system;
  * "solve": restarted GMRES from a plane wave to a tolerance, plain or regularised and
    deflated, FP64 or with complex64 products inside a cycle, one right-hand side or one per
    incidence angle;
  * "forward" / "gradients": the learned preconditioner's network on a batch.

Solves ask for 1e-12 or less, so that their solutions are those of the system and not of
where the iteration happened to stop.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1104_4263_gb300 import die, workloads as W

POL = {"te": die.DIE_TE, "tm": die.DIE_TM, "mag": die.DIE_TE_MAG}


def listed():
    return [
        # One regularised FP64 product on the 61^2 grid of the paper's Section 4 squares: the
        # smallest systems solved in earnest, where latency and launches count.
        {"name": "product_f64_square_61", "what": "product", "map": "square", "n1": 61, "n2": 61, "pol": "te",
         "bits": 64, "reg": True, "batch": 1},
        # The product inside the FP32-inner solves, on the benchmark's 512^2 core-shell.
        {"name": "product_c64_coreshell_512", "what": "product", "map": "core_shell", "n1": 512, "n2": 512,
         "pol": "te", "bits": 32, "reg": True, "batch": 1},
        # The same product in FP64: every restart residual, and every step of the FP64 solves.
        {"name": "product_f64_coreshell_512", "what": "product", "map": "core_shell", "n1": 512, "n2": 512,
         "pol": "te", "bits": 64, "reg": True, "batch": 1},
        # Eight incidence angles at once on the 233^2 grid of Section 5's sinusoidal object (a
        # size that no transform length fits exactly).
        {"name": "batch_c64_sinusoidal_233", "what": "product", "map": "sinusoidal", "n1": 233, "n2": 233,
         "pol": "te", "bits": 32, "reg": True, "batch": 8},
        # The largest grid: the 2048^2 composite of random cylinders, 8.4 million unknowns.
        {"name": "product_c64_cylinders_2048", "what": "product", "map": "cylinders", "n1": 2048, "n2": 2048,
         "pol": "te", "bits": 32, "reg": True, "batch": 1},
        # The three-plane system with magnetic contrast in FP64 (transform length 3 * 2^8).
        {"name": "product_f64_magnetic_384", "what": "product", "map": "core_shell", "n1": 384, "n2": 384,
         "pol": "mag", "bits": 64, "reg": False, "batch": 1},
        # Section 4's plasma-like square, plain FP64 GMRES(40) to convergence: many short steps.
        {"name": "solve_f64_square_61", "what": "solve", "map": "plasma", "n": 61, "pol": "te", "inner": 64,
         "reg": False, "restart": 40, "tol": 1e-13, "steps": 20000, "r": 0, "rhs": 1, "graph": False},
        # The method of the paper on a 512^2 grid: regularised, deflated, FP32-inner GMRES(30)
        # with FP64 refinement to convergence, cycles as graphs.
        {"name": "solve_mixed_cylinder_512", "what": "solve", "map": "cylinder", "n": 512, "pol": "te", "inner": 32,
         "reg": True, "restart": 30, "tol": 1e-12, "steps": 3000, "r": 8, "rhs": 1, "graph": True},
        # A long Krylov space in FP64, as in the paper's large-memory runs (Section 5): restart
        # 400 on the 133^2 grid of its sweep, a lossy random field.
        {"name": "solve_f64_long_133", "what": "solve", "map": "lossy", "n": 133, "pol": "te", "inner": 64,
         "reg": True, "restart": 400, "tol": 1e-12, "steps": 2000, "r": 0, "rhs": 1, "graph": False},
        # One scatterer under eight incidence angles, solved concurrently.
        {"name": "solve_batch_lossy_64", "what": "solve", "map": "lossy", "n": 64, "pol": "te", "inner": 32,
         "reg": True, "restart": 60, "tol": 1e-12, "steps": 4000, "r": 8, "rhs": 8, "graph": False},
        # The learned preconditioner inside flexible GMRES: one field at a time.
        {"name": "network_forward_128", "what": "forward", "width": 32, "modes": 16, "layers": 4, "hidden": 128,
         "H": 128, "W": 128, "batch": 1},
        # One training batch: forward, backward and the gradients.
        {"name": "network_gradients_128x16", "what": "gradients", "width": 32, "modes": 16, "layers": 4,
         "hidden": 128, "H": 128, "W": 128, "batch": 16},
    ]


def _spread(rng, lo, hi):
    """An integer between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["product", "product", "product", "batch", "magnetic", "solve", "solve", "network"])
    if kind == "product":
        bits = rng.choice([64, 32])
        top = 2048 if bits == 32 else 1024
        n1 = _spread(rng, 24, top)
        n2 = rng.choice([n1, _spread(rng, 24, top)])
        if rng.random() < 0.4:          # a power of two, as most users choose
            n1 = n2 = 1 << rng.randint(5, 11 if bits == 32 else 10)
        return {"what": "product", "map": "random", "n1": n1, "n2": n2, "pol": rng.choice(["te", "te", "tm"]),
                "bits": bits, "reg": rng.random() < 0.6, "batch": 1}
    if kind == "batch":
        return {"what": "product", "map": "random", "n1": _spread(rng, 24, 512), "n2": _spread(rng, 24, 512),
                "pol": "te", "bits": rng.choice([64, 32]), "reg": rng.random() < 0.6, "batch": rng.randint(2, 8)}
    if kind == "magnetic":
        return {"what": "product", "map": "random", "n1": _spread(rng, 24, 512), "n2": _spread(rng, 24, 512),
                "pol": "mag", "bits": rng.choice([64, 32]), "reg": rng.random() < 0.5, "batch": 1}
    if kind == "solve":
        inner = rng.choice([64, 32])
        reg = inner == 32 or rng.random() < 0.5
        kind = rng.choice(["lossy", "cylinder"])
        return {"what": "solve", "map": kind, "n": _spread(rng, 100, 320) if kind == "cylinder" else _spread(rng, 24, 64),
                "pol": rng.choice(["te", "te", "tm"]), "inner": inner, "reg": reg, "restart": rng.randint(40, 80),
                "tol": 1e-12, "steps": 3000,
                "r": rng.choice([0, 0, rng.randint(2, 10)]) if reg else 0, "rhs": rng.choice([1, 1, rng.randint(2, 6)]),
                "graph": rng.random() < 0.5}
    width, modes = rng.choice([16, 24, 32, 48]), rng.randint(4, 16)
    return {"what": rng.choice(["forward", "gradients"]), "width": width, "modes": modes, "layers": rng.randint(2, 4),
            "hidden": rng.choice([64, 128]), "H": rng.choice([48, 64, 96, 100, 128]), "W": rng.choice([48, 64, 96, 100, 128]),
            "batch": rng.randint(1, 16)}


# ------------------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _map(case, seed):
    """(eps_r, h, mu_r): the scatterer of a case (sizes and values of the paper and the benchmark)."""
    if case["what"] == "solve":
        n1 = n2 = case["n"]
    else:
        n1, n2 = case["n1"], case["n2"]
    kind, h = case["map"], 1.0 / 60.0
    if kind == "square":
        p = W.square(n1, h, 16.0 + 0j)
        eps, h = p.eps_r, p.h
    elif kind == "plasma":
        p = W.square(n1, h, -16.0 + 1.5j)
        eps, h = p.eps_r, p.h
    elif kind == "core_shell":
        p = W.config2(n1)
        eps, h = p.eps_r, p.h
    elif kind == "sinusoidal":
        p = W.sinusoidal(n1)
        eps, h = p.eps_r, p.h
    elif kind == "cylinders":
        p = W.random_cylinders(n1, seed_index=int(seed) % 1000)
        eps, h = p.eps_r, p.h
    elif kind == "cylinder":
        p = W.config1(n1)
        eps, h = p.eps_r, p.h
    elif kind == "lossy":          # a random lossy dielectric field, smooth over 0.3 wavelengths
        p = W.config4_field(int(seed) % 100000, n1, re_lo=1.0)
        eps, h = p.eps_r, p.h
    else:                          # cell-wise random values
        eps = W.random_field(np.random.default_rng(int(seed)), n1, n2)
    mu = None
    if case["pol"] == "mag":
        mu = np.where(np.asarray(eps).real != 1.0, 2.0 + 0.1j, 1.0 + 0j)
    return eps, h, mu


def _waves(n1, n2, h, k, psi, device):
    """exp(i k (x1 cos psi + x2 sin psi)) at the cell centres, (len(psi), n2, n1)."""
    x1 = (torch.arange(n1, dtype=torch.float64, device=device) + 0.5) * h - 0.5 * n1 * h
    x2 = (torch.arange(n2, dtype=torch.float64, device=device) + 0.5) * h - 0.5 * n2 * h
    return torch.stack([torch.exp(1j * k * (x1[None, :] * math.cos(a) + x2[:, None] * math.sin(a))) for a in psi])


def _field(case, seed, h):
    """Vectors for the products: plane waves with as much complex noise, one per vector."""
    g = _generator(seed)
    planes = 3 if case["pol"] == "mag" else 2
    shape = (case["batch"], planes, case["n2"], case["n1"])
    noise = torch.randn(shape, dtype=torch.complex128, device="cuda", generator=g)
    psi = [2.0 * math.pi * (seed % 997 / 997 + k / case["batch"]) for k in range(case["batch"])]
    x = noise + _waves(case["n1"], case["n2"], h, 2.0 * math.pi, psi, "cuda")[:, None]
    if case["pol"] == "tm":
        x[:, 1] = 0
    return x.to(torch.complex128 if case["bits"] == 64 else torch.complex64)


def _angles(case, seed):
    return [2.0 * math.pi * (seed % 997 / 997 + k / case["rhs"]) for k in range(case["rhs"])]


def _shapes(case):
    """The network's parameters in the order of the parameter vector: (name, shape, scale)."""
    c, m, hid = case["width"], case["modes"], case["hidden"]
    out = [("P", (c, 6), 6 ** -0.5), ("p", (c,), 0.1)]
    for l in range(case["layers"]):
        out += [(f"W{l}", (c, c), c ** -0.5), (f"w{l}", (c,), 0.1),
                (f"R{l}", (2, c, c, m, m, 2), 1.0 / c)]
    return out + [("Q1", (hid, c), c ** -0.5), ("q1", (hid,), 0.1), ("Q2", (4, hid), hid ** -0.5), ("q2", (4,), 0.1)]


def _network_inputs(case, seed):
    """Parameters (float32), input channels and the gradient of the output."""
    rng = np.random.default_rng(int(seed))
    params = np.concatenate([(s * rng.standard_normal(shape, dtype=np.float32)).ravel() for _, shape, s in _shapes(case)])
    g = _generator(seed)
    x = torch.randn((case["batch"], 6, case["H"], case["W"]), device="cuda", generator=g)
    gy = torch.randn((case["batch"], 4, case["H"], case["W"]), device="cuda", generator=g) / (case["H"] * case["W"])
    return params.astype(np.float32), x, gy


def prepare(case, seed):
    if case["what"] in ("forward", "gradients"):
        params, x, gy = _network_inputs(case, seed)
        net = die.FNO(6, 4, case["width"], case["modes"], case["layers"], case["hidden"], case["H"], case["W"],
                      case["batch"])
        net.set_params(params)
        return {"case": case, "net": net, "x": x, "gy": gy}
    eps, h, mu = _map(case, seed)
    prec = die.DIE_FP64 if case.get("bits", 64) == 64 else die.DIE_FP32_INNER
    op = die.Operator(eps, h, prec=prec, pol=POL[case["pol"]], mu_r=mu)
    if case["what"] == "product":
        x = _field(case, seed, h)
        x = x if case["batch"] > 1 else x[0].contiguous()
        return {"case": case, "op": op, "x": x, "y": torch.empty_like(x)}
    b = torch.stack([op.plane_wave(a) for a in _angles(case, seed)])
    inner = die.DIE_FP64 if case["inner"] == 64 else die.DIE_FP32_INNER
    D = die.Deflation(op, case["r"], regularized=case["reg"], inner=inner) if case["r"] else None
    return {"case": case, "op": op, "b": b, "inner": inner, "D": D}


# --------------------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    if case["what"] == "product":
        op, x, y = state["op"], state["x"], state["y"]
        if case["batch"] > 1:
            return op.apply_batch(x, y, regularized=case["reg"])
        return op.apply_regularized(x, y) if case["reg"] else op.apply(x, y)
    if case["what"] == "solve":
        kw = dict(restart=case["restart"], tol=case["tol"], max_iters=case["steps"], regularized=case["reg"],
                  inner=state["inner"], deflation=state["D"], graph=case["graph"])
        if case["rhs"] > 1:
            return state["op"].solve_batch(state["b"], **kw)[0]
        return state["op"].solve(state["b"][0], **kw)[0]
    net = state["net"]
    y = net.forward(state["x"])
    if case["what"] == "forward":
        return y
    net.zero_grads()
    gx = net.backward(state["gy"], want_gx=True)
    return {"y": y, "gx": gx, "grads": net.get_grads()}


# ------------------------------------------------------------- what a pass cannot do without
def _conv_flops(n1, n2, planes):
    """Real operations of one zero-padded 2-D FFT convolution (5 L log2 L per transform of
    length L, transforms of zero lines left out) with its planes x planes multiply."""
    M1, M2 = 2 * n1, 2 * n2
    rows = planes * n2 * 2 * 5 * M1 * math.log2(M1)
    cols = planes * M1 * 2 * 5 * M2 * math.log2(M2)
    return rows + cols + 8 * planes * planes * M1 * M2 + 8 * planes * n1 * n2


def work(case):
    if case["what"] == "product":
        n, planes, e = case["n1"] * case["n2"], 3 if case["pol"] == "mag" else 2, case["bits"] // 4
        spectra = 6 if planes == 3 else 3
        return {"bytes": e * (2 * planes * n * case["batch"] + (1 + case["reg"]) * n + spectra * n),
                "flops": case["batch"] * (2 if case["reg"] else 1) * _conv_flops(case["n1"], case["n2"], planes)}
    if case["what"] == "solve":
        # one cycle's worth of Arnoldi steps per right-hand side: the basis read twice a step
        # (projections and update), the product's operands, two sweeps of 8 operations per entry
        n, m = 2 * case["n"] ** 2, min(case["restart"], case["steps"])
        e = case["inner"] // 4
        steps = m * case["rhs"]
        return {"bytes": steps * (16 * n * m + 4 * e * n), "flops": steps * ((2 if case["reg"] else 1) * _conv_flops(case["n"], case["n"], 2)
                                                                          + 8 * n * m)}
    c, m, hid, b = case["width"], case["modes"], case["hidden"], case["batch"]
    hw = case["H"] * case["W"]
    layer = 2 * c * c * hw + 2 * c * 2 * m * hw + 2 * c * m * 2 * case["H"] * 4 * m
    fwd = 2 * hw * (6 * c + c * hid + hid * 4) + case["layers"] * (2 * layer - 2 * c * c * hw + 2 * 2 * m * m * 4 * c * c)
    params = sum(math.prod(s) for _, s, _ in _shapes(case))
    if case["what"] == "forward":
        return {"bytes": 4 * (b * 10 * hw + params), "flops": b * fwd}
    return {"bytes": 4 * (b * 20 * hw + 2 * params), "flops": 3 * b * fwd}


# ---------------------------------------------------------------- the same in plain FP64
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _hankel(x):
    """H0 and H1 of the first kind for x > 0: Hankel's expansion from 25 on, below it Miller's
    downward recurrence for J and Neumann's series for Y."""
    z = torch.where(x < 25, x, torch.full_like(x, 25.0))
    hi, lo = torch.zeros_like(z), torch.full_like(z, 1e-280)
    total, y0, y1 = torch.zeros_like(z), torch.zeros_like(z), torch.zeros_like(z)
    for n in range(81, 0, -1):           # (J_{n+1}, J_n) = (hi, lo), up to a common factor
        if n % 2 == 0:
            k = n // 2
            total, y0 = total + 2 * lo, y0 + (-1) ** k * lo / k
        elif n > 1:
            k = (n - 1) // 2
            y1 = y1 + (-1) ** k * (2 * k + 1) / (k * (k + 1)) * lo
        hi, lo = lo, 2 * n / z * lo - hi
        s = torch.where(lo.abs() > 1e200, torch.full_like(z, 1e-200), torch.ones_like(z))
        hi, lo, total, y0, y1 = hi * s, lo * s, total * s, y0 * s, y1 * s
    total = total + lo
    J0, J1, y0, y1 = lo / total, hi / total, y0 / total, y1 / total
    lg = torch.log(z / 2) + 0.57721566490153286061
    Y0 = 2 / math.pi * lg * J0 - 4 / math.pi * y0
    Y1 = -2 / (math.pi * z) * J0 + 2 / math.pi * (lg - 1) * J1 - 2 / math.pi * y1
    z = torch.where(x < 25, torch.full_like(x, 25.0), x)
    out = []
    for nu, J, Y in ((0, J0, Y0), (1, J1, Y1)):
        term = acc = torch.ones_like(z, dtype=torch.complex128)
        for k in range(1, 31):
            term = term * (1j * (4 * nu * nu - (2 * k - 1) ** 2) / (8.0 * k)) / z
            acc = acc + term
        ph = z - (nu / 2 + 0.25) * math.pi
        far = torch.sqrt(2 / (math.pi * z)) * torch.polar(torch.ones_like(z), ph) * acc
        out.append(torch.where(x < 25, torch.complex(J, Y), far))
    return out


def _spectra(n1, n2, h, k, pol, dev):
    """Spectra of the kernel planes on the (2 n2) x (2 n1) circle, {(l, q): plane}."""
    p = torch.arange(2 * n1, dtype=torch.float64, device=dev)
    q = torch.arange(2 * n2, dtype=torch.float64, device=dev)
    p, q = torch.where(p < n1, p, p - 2 * n1), torch.where(q < n2, q, q - 2 * n2)
    d1, d2 = p[None, :] * h, q[:, None] * h
    keep = (p.abs() < n1)[None, :] & (q.abs() < n2)[:, None]
    a1 = torch.arange(n1 + 1, dtype=torch.float64, device=dev) * h
    a2 = torch.arange(n2 + 1, dtype=torch.float64, device=dev) * h
    r = torch.hypot(a1[None, :].expand(n2 + 1, n1 + 1), a2[:, None].expand(n2 + 1, n1 + 1))
    r[0, 0] = 1.0
    H0, H1 = (v[q.abs().long()][:, p.abs().long()] for v in _hankel(k * r))
    own = (p == 0)[None, :] & (q == 0)[:, None]
    r = r[q.abs().long()][:, p.abs().long()]
    t1, t2, c = d1 / r, d2 / r, (k * h) ** 2
    a = k * h / math.sqrt(math.pi)
    disc = 0.5j * math.pi * a * complex(_hankel(torch.tensor([a], dtype=torch.float64))[1][0])

    def plane(v, at_zero):
        v = torch.where(own, torch.full_like(v, at_zero), v)
        return torch.fft.fft2(torch.where(keep, v, torch.zeros_like(v)))

    if pol == "tm":
        g = plane(0.25j * c * H0, disc - 1.0)
        return {(0, 0): g, (1, 1): g}
    P, Q = 0.5j / (k * r) * H1 - 0.25j * H0, 0.25j * H0 - 0.25j / (k * r) * H1
    s = -(1.0 - 0.5 * disc)
    G = {(0, 0): plane(c * (P * t1 * t1 + Q), s), (1, 1): plane(c * (P * t2 * t2 + Q), s)}
    G[0, 1] = G[1, 0] = plane(c * P * t1 * t2, 0.0)
    if pol == "mag":
        G[0, 2] = G[2, 0] = plane(0.25 * c * H1 * t2, 0.0)
        G[1, 2] = G[2, 1] = plane(-0.25 * c * H1 * t1, 0.0)
        G[2, 2] = plane(0.25j * c * H0, disc - 1.0)
    return G


class _Plain:
    """A and A(chi') by torch.fft in FP64, for one vector (planes, n2, n1)."""

    def __init__(self, case, seed):
        eps, h, mu = _map(case, seed)
        self.n2, self.n1 = eps.shape
        self.h, self.k, dev = h, 2.0 * math.pi, _device()
        self.planes = 3 if case["pol"] == "mag" else 2
        self.G = _spectra(self.n1, self.n2, h, self.k, case["pol"], dev)
        eps = torch.from_numpy(np.ascontiguousarray(eps)).to(dev)
        chi_m = [torch.from_numpy(mu).to(dev) - 1.0] if mu is not None else []
        self.chi = torch.stack([eps - 1.0, eps - 1.0] + chi_m)
        self.chi_reg = torch.stack([1.0 / eps - 1.0, 1.0 / eps - 1.0] + chi_m)

    def _times(self, chi, u):
        w = torch.fft.fft2(chi * u, s=(2 * self.n2, 2 * self.n1))
        z = torch.stack([sum(self.G[l, q] * w[q] for q in range(self.planes) if (l, q) in self.G) for l in range(self.planes)])
        return u - torch.fft.ifft2(z)[:, :self.n2, :self.n1]

    def apply(self, u, reg):
        v = self._times(self.chi, u)
        return self._times(self.chi_reg, v) if reg else v

    def wave(self, psi, pol):
        e = _waves(self.n1, self.n2, self.h, self.k, [psi], self.chi.device)[0]
        if pol == "tm":
            return torch.stack([e, torch.zeros_like(e)])
        return torch.stack([-math.sin(psi) * e, math.cos(psi) * e])

    def solve(self, b, restart=100, steps=4000, tol=2e-14):
        """The system's solution by GMRES with repeated Gram-Schmidt."""
        b = b.reshape(-1)
        mul = lambda v: self._times(self.chi, v.reshape(self.planes, self.n2, self.n1)).reshape(-1)  # noqa: E731
        x, done, scale = torch.zeros_like(b), 0, float(torch.linalg.norm(b))
        while done < steps:
            r = b - mul(x)
            beta = float(torch.linalg.norm(r))
            if beta <= tol * scale:
                break
            m = min(restart, steps - done)
            V = torch.empty((m + 1, b.numel()), dtype=b.dtype, device=b.device)
            H = torch.zeros((m + 1, m), dtype=b.dtype, device=b.device)
            V[0] = r / beta
            for j in range(m):
                w = mul(V[j])
                for _ in range(2):
                    c = V[:j + 1].conj() @ w
                    w = w - c @ V[:j + 1]
                    H[:j + 1, j] += c
                H[j + 1, j] = torch.linalg.norm(w)
                V[j + 1] = w / H[j + 1, j]
            e = np.zeros(m + 1, dtype=np.complex128)
            e[0] = beta
            y = np.linalg.lstsq(H.cpu().numpy(), e, rcond=None)[0]
            x = x + torch.from_numpy(y).to(b.device) @ V[:m]
            done += m
        return x.reshape(self.planes, self.n2, self.n1)


def _network(case, params, x):
    """The network in FP64 on torch.fft; params: {name: tensor}."""
    m, H, Wd = case["modes"], case["H"], case["W"]
    mix = lambda A, a, h: torch.einsum("oi,bihw->bohw", A, h) + a[None, :, None, None]  # noqa: E731
    gelu = lambda v: v * torch.special.ndtr(v)  # noqa: E731
    h = mix(params["P"], params["p"], x)
    for l in range(case["layers"]):
        R = torch.view_as_complex(params[f"R{l}"])
        X = torch.fft.rfft2(h)
        low = torch.einsum("bixy,ioxy->boxy", X[:, :, :m, :m], R[0])
        high = torch.einsum("bixy,ioxy->boxy", X[:, :, H - m:, :m], R[1])
        mid = torch.zeros(low.shape[:2] + (H - 2 * m, m), dtype=low.dtype, device=low.device)
        Y = torch.nn.functional.pad(torch.cat([low, mid, high], dim=2), (0, Wd // 2 + 1 - m))
        h = mix(params[f"W{l}"], params[f"w{l}"], h) + torch.fft.irfft2(Y, s=(H, Wd))
        h = gelu(h) if l < case["layers"] - 1 else h
    return mix(params["Q2"], params["q2"], gelu(mix(params["Q1"], params["q1"], h)))


def exact(case, seed):
    if case["what"] in ("forward", "gradients"):
        flat, x, gy = _network_inputs(case, seed)
        dev, params, at = x.device, {}, 0
        for name, shape, _ in _shapes(case):
            n = math.prod(shape)
            params[name] = torch.from_numpy(flat[at:at + n].astype(np.float64)).reshape(shape).to(dev).requires_grad_()
            at += n
        x = x.double().requires_grad_()
        y = _network(case, params, x)
        if case["what"] == "forward":
            return y.detach()
        (y * gy.double()).sum().backward()
        grads = torch.cat([params[name].grad.reshape(-1) for name, _, _ in _shapes(case)])
        return {"y": y.detach(), "gx": x.grad, "grads": grads.cpu().numpy()}
    plain = _Plain(case, seed)
    if case["what"] == "product":
        x = _field(case, seed, plain.h).to(torch.complex128)
        y = torch.stack([plain.apply(v, case["reg"]) for v in x])
        return y if case["batch"] > 1 else y[0]
    x = torch.stack([plain.solve(plain.wave(a, case["pol"])) for a in _angles(case, seed)])
    return x if case["rhs"] > 1 else x[0]
