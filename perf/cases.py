"""The work that users of this library have it do, as measured cases.

Each case is one call pattern of ``paper_1504_02897_gb300.ddi`` with its sizes:

``ddi``        ``Plan.apply``: one dipolar potential on a 3D or 2D grid (any precision)
``split``      ``Plan.apply`` of a plan built for the improved split algorithm (3D)
``batch``      ``Batch.apply``: many 2D densities in one call (recorded graph, autotuned)
``step``       ``Plan.gpe_step`` / ``gpe_step_ex``: a few time-splitting steps in place, with a
               fixed axis, a rotating axis (``set_axes`` before every step) or three-body loss
``ground``     ``Plan.ground_state``: a stretch of the normalised gradient flow
``gradient``   ``Plan.trap_gradient``: J and dJ/dV through the steps' adjoint

``exact`` evaluates the same sums in FP64 with plain torch: the quadrature sum of a ring of
nodes (one k_z) factors into a transform along z and one in the plane, so the direct sum
needs no NUFFT.
"""
import math

import numpy as np
import torch

from paper_1504_02897_gb300 import ddi

SIZES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024)


# ---- the cases --------------------------------------------------------------------------------
def _ddi3(n, length, prec, rule=(0, 0, 0), axes="tilted", split=False):
    return {"kind": "split" if split else "ddi", "dim": 3, "nx": n[0], "ny": n[1], "nz": n[2], "lx": length[0],
            "ly": length[1], "lz": length[2], "prec": prec, "nr": rule[0], "ntheta": rule[1], "nphi": rule[2],
            "axes": axes}


def listed():
    return [
        # the smallest call: a 24^3 density with a 16 x 16 x 32 rule (launches and latency)
        dict(_ddi3((24, 24, 24), (12.0, 12.0, 12.0), "fp32", (16, 16, 32), "z"), name="ddi3d_24_fp32"),
        # a box of unequal sides and spacings with two dipole axes, default rule
        dict(_ddi3((96, 64, 48), (18.0, 14.0, 12.0), "fp32", axes="two"), name="ddi3d_96x64x48_fp32"),
        # the headline workload: 128^3, tilted axis, 128 x 64 x 128 nodes
        dict(_ddi3((128, 128, 128), (24.0, 24.0, 24.0), "fp32"), name="ddi3d_128_fp32"),
        # a large grid with its own default rule (3.5 M nodes)
        dict(_ddi3((192, 192, 192), (36.0, 36.0, 36.0), "fp32"), name="ddi3d_192_fp32"),
        # the FP64 path of the headline workload
        dict(_ddi3((128, 128, 128), (24.0, 24.0, 24.0), "fp64"), name="ddi3d_128_fp64"),
        # the split algorithm on a large grid (its ball rule does not grow with the grid)
        dict(_ddi3((256, 256, 256), (48.0, 48.0, 48.0), "fp32", split=True), name="split_256_fp32"),
        # one 2D density, default 2N x 2N rule
        {"name": "ddi2d_512_fp32", "kind": "ddi", "dim": 2, "nx": 512, "ny": 512, "lx": 24.0, "ly": 24.0,
         "prec": "fp32", "nr": 0, "nphi": 0, "axes": "tilted"},
        # a batch of 2D densities of mixed sizes, boxes and tilts
        {"name": "batch2d_24_fp32", "kind": "batch", "count": 24, "least": 128, "most": 1024, "shape_seed": 0},
        # real-time dynamics: four steps at 128^3, fixed axis, FP32
        {"name": "step_128_fp32", "kind": "step", "n": 128, "half": 10.0, "prec": "fp32", "steps": 4,
         "beta": 207.16, "lam": 33.1456, "dt": 1e-3, "mode": "fixed"},
        # real-time dynamics with a rotating dipole axis in FP64: new node weights every step
        {"name": "step_rotating_64_fp64", "kind": "step", "n": 64, "half": 8.0, "prec": "fp64", "steps": 2,
         "beta": 207.16, "lam": 103.58, "dt": 2e-3, "mode": "rotating"},
        # a stretch of the gradient flow to the ground state at 96^3
        {"name": "ground_96_fp32", "kind": "ground", "n": 96, "half": 12.0, "prec": "fp32", "steps": 5,
         "beta": 207.16, "lam": 103.58, "dt": 1e-2},
        # the gradient of a final-time observable with respect to the trap at 64^3
        {"name": "gradient_64_fp32", "kind": "gradient", "n": 64, "half": 8.0, "prec": "fp32", "steps": 8, "every": 4,
         "beta": 207.16, "lam": 33.1456, "dt": 1e-3},
    ]


def _size(rng, least, most):
    """A built grid size in [least, most], spread over the logarithm."""
    return rng.choice([n for n in SIZES if least <= n <= most])


def draw(rng):
    kind = rng.choice(["ddi3", "ddi3", "ddi2", "split", "batch", "step", "ground", "gradient"])
    if kind in ("ddi3", "split"):
        prec = "fp32" if kind == "split" else rng.choice(["fp32", "fp32", "fp64"])
        top = _size(rng, 64 if kind == "split" else 16, 256 if kind == "split" else (192 if prec == "fp32" else 96))
        # up to a factor of two between the axes
        n = [rng.choice([m for m in SIZES if top / 2 <= m <= top]) for _ in range(3)]
        n[rng.randrange(3)] = top
        h = rng.uniform(0.12, 0.25)
        if kind == "split":  # the window's ball (6 k0, k0 = 9.6 / the shortest side) has to fit the band
            n = [max(m, top // 2) for m in n]
            length = [m * h for m in n]
            return _ddi3(n, length, prec, axes=rng.choice(["z", "tilted", "two"]), split=True)
        length = [m * h * rng.uniform(0.8, 1.25) for m in n]
        rule = (0, 0, 0)
        if rng.random() < 0.5:  # a rule of the user's own, odd counts among them
            rule = (rng.randint(max(4, top // 2), top), rng.randint(max(3, top // 4), top // 2),
                    2 * rng.randint(max(4, top // 4), top // 2))
        return _ddi3(n, length, prec, rule, rng.choice(["z", "tilted", "two"]))
    if kind == "ddi2":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        top = _size(rng, 32, 1024 if prec == "fp32" else 256)
        n = [rng.choice([m for m in SIZES if top / 2 <= m <= top]), top]
        h = rng.uniform(0.04, 0.25)
        rule = (0, 0) if rng.random() < 0.5 else (rng.randint(top, 2 * top), 2 * rng.randint(top // 2, top))
        return {"kind": "ddi", "dim": 2, "nx": n[0], "ny": n[1], "lx": n[0] * h, "ly": n[1] * h * rng.uniform(0.8, 1.25),
                "prec": prec, "nr": rule[0], "nphi": rule[1], "axes": rng.choice(["tilted", "two"])}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 24), "least": 64, "most": _size(rng, 128, 768),
                "shape_seed": rng.randrange(1 << 20)}
    case = {"kind": kind, "n": _size(rng, 16, 96), "half": round(rng.uniform(6.0, 10.0), 3),
            "prec": rng.choice(["fp32", "fp64"]), "steps": rng.randint(1, 5), "beta": round(rng.uniform(50.0, 250.0), 3),
            "lam": round(rng.uniform(10.0, 100.0), 3), "dt": round(rng.uniform(5e-4, 4e-3), 6)}
    if case["prec"] == "fp64":
        case["n"] = min(case["n"], 48)
    if kind == "step":
        case["mode"] = rng.choice(["fixed", "rotating", "loss"])
    if kind == "gradient":
        case["every"] = rng.randint(1, case["steps"])
    return case


# ---- inputs -----------------------------------------------------------------------------------
def _dtypes(prec):
    return (torch.float64, torch.complex128, ddi.FP64) if prec == "fp64" else (torch.float32, torch.complex64, ddi.FP32)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _axes_of(name):
    s, c = math.sin(math.radians(30.0)), math.cos(math.radians(30.0))
    if name == "z":
        return (0.0, 0.0, 1.0), None
    if name == "tilted":
        return (s, 0.0, c), None
    return (s, 0.0, c), (0.0, 0.6, 0.8)


def _coords(n, lo, length):
    return [lo[a] + torch.arange(n[a], dtype=torch.float64, device=_device()) * (length[a] / n[a])
            for a in range(len(n))]


def _outer(parts):
    """Product of per-axis factors (x, y[, z]) on the grid [z][y][x] / [y][x]."""
    if len(parts) == 3:
        return parts[2][:, None, None] * parts[1][None, :, None] * parts[0][None, None, :]
    return parts[1][:, None] * parts[0][None, :]


def _mixture(n, lo, length, seed, count):
    """A sum of axis-aligned Gaussians of discrete mass 1 (FP64)."""
    rng = np.random.default_rng(seed)
    x = _coords(n, lo, length)
    rho = 0.0
    for _ in range(count):
        parts = []
        for a in range(len(n)):
            c = rng.uniform(-length[a] / 6.0, length[a] / 6.0)
            w = rng.uniform(0.5, 2.0) * length[a] / 24.0
            parts.append(torch.exp(-(x[a] - c) ** 2 / (2.0 * w * w)))
        rho = rho + rng.uniform(0.5, 1.5) * _outer(parts)
    dv = math.prod(length[a] / n[a] for a in range(len(n)))
    return rho / (dv * rho.sum())


def _geometry(case):
    """(n, lo, length, rule, axis_n, axis_m) of a ddi / split case."""
    names = ("x", "y", "z")[: case["dim"]]
    n = tuple(case["n" + a] for a in names)
    length = tuple(case["l" + a] for a in names)
    rule = {k: case[k] for k in ("nr", "ntheta", "nphi") if k in case}
    axis_n, axis_m = _axes_of(case["axes"])
    return n, tuple(-0.5 * v for v in length), length, rule, axis_n, axis_m


def _batch_items(case):
    """Sizes, boxes and tilts of a batch (fixed by the case; the densities come from the seed)."""
    rng = np.random.default_rng(case["shape_seed"])
    sizes = [m for m in (64, 128, 256, 512, 1024) if case["least"] <= m <= case["most"]]
    items = []
    for _ in range(case["count"]):
        n = int(sizes[rng.integers(0, len(sizes))])
        half, tilt = float(rng.uniform(8.0, 16.0)), math.radians(float(rng.uniform(0.0, 90.0)))
        items.append(((n, n), (-half, -half), (2 * half, 2 * half), (math.sin(tilt), 0.0, math.cos(tilt))))
    return items


def _gpe_inputs(case, seed):
    """(n, lo, length, trap, state): a harmonic trap and its Gaussian with a smooth perturbation."""
    n, half = (case["n"],) * 3, case["half"]
    lo, length = (-half,) * 3, (2.0 * half,) * 3
    x = _coords(n, lo, length)
    gam = (1.0, 1.0, 2.0)
    V = 0.5 * (x[2][:, None, None] ** 2 * gam[2] ** 2 + x[1][None, :, None] ** 2 * gam[1] ** 2
               + x[0][None, None, :] ** 2 * gam[0] ** 2)
    psi = _outer([torch.exp(-0.5 * gam[a] * x[a] ** 2) for a in range(3)])
    rng = np.random.default_rng(seed)
    eta = torch.zeros_like(psi)
    for _ in range(8):
        p, ab = rng.integers(-3, 4, 3), rng.standard_normal(2)
        e = _outer([torch.exp(2j * math.pi * float(p[a]) * (x[a] - lo[a]) / length[a]) for a in range(3)])
        eta += float(ab[0]) * e.real + float(ab[1]) * e.imag
    psi = psi * (1.0 + 0.05 * eta / eta.abs().max())
    dv = math.prod(length[a] / n[a] for a in range(3))
    return n, lo, length, V, (psi / torch.sqrt(dv * (psi * psi).sum())).to(torch.complex128)


def _rotating(case, k):
    """The rotating axis at the midpoint of step k."""
    t = (k + 0.5) * case["dt"] * 50.0
    return math.sin(t / 5.0), 0.0, math.cos(t / 5.0)


def prepare(case, seed):
    dev = _device()
    if case["kind"] in ("ddi", "split"):
        n, lo, length, rule, axis_n, axis_m = _geometry(case)
        real, _, prec = _dtypes(case["prec"])
        kw = dict(rule, split_k0=-1.0) if case["kind"] == "split" else rule
        plan = ddi.Plan(case["dim"], n, lo, length, axis_n, axis_m, precision=prec, **kw)
        rho = _mixture(n, lo, length, seed, 8 if case["dim"] == 3 else 4).to(real)
        return {"case": case, "plan": plan, "rho": rho, "phi": torch.empty_like(rho)}
    if case["kind"] == "batch":
        items = _batch_items(case)
        batch = ddi.Batch([ddi.make_desc(2, n, lo, ln, axis, precision=ddi.FP32) for n, lo, ln, axis in items])
        rhos = [_mixture(n, lo, ln, seed * 1000 + i, 4).float() for i, (n, lo, ln, _) in enumerate(items)]
        return {"case": case, "batch": batch, "rhos": rhos, "phis": [torch.empty_like(r) for r in rhos]}
    real, cplx, prec = _dtypes(case["prec"])
    n, lo, length, V, psi = _gpe_inputs(case, seed)
    plan = ddi.Plan(3, n, lo, length, (0.0, 0.0, 1.0), precision=prec)
    return {"case": case, "plan": plan, "V": V.to(real), "psi": psi.to(cplx).to(dev)}


# ---- one pass ---------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("ddi", "split"):
        return state["plan"].apply(state["rho"], state["phi"])
    if kind == "batch":
        return state["batch"].apply(state["rhos"], state["phis"])
    plan, V, beta, lam, dt = state["plan"], state["V"], case["beta"], case["lam"], case["dt"]
    if kind == "step":
        psi = state["psi"]  # evolves in place
        if case["mode"] == "fixed":
            return plan.gpe_step(psi, V, beta, lam, dt, case["steps"])
        if case["mode"] == "loss":
            return plan.gpe_step_ex(psi, V, beta, lam, dt, case["steps"], damping=ddi.DAMP_POWER, delta=3.512, q=2.0)
        for k in range(case["steps"]):
            plan.set_axes(_rotating(case, k))
            plan.gpe_step(psi, V, beta, lam, dt, 1)
        return psi
    if kind == "ground":
        phi = state["psi"].clone()  # every search starts from the initial guess
        st = plan.ground_state(phi, V, beta, lam, dt, 1e-14, max_steps=case["steps"], check_every=10)
        return phi, [st[k] for k in ("E", "mu", "Ekin", "Epot", "Eint", "Edip", "mass")]
    J, grad = plan.trap_gradient(state["psi"], V, beta, lam, dt, case["steps"], case["every"])
    return J, grad


# ---- the work a pass cannot do without -----------------------------------------------------------
def _rule3(n, rule):
    m = max(n)
    return rule.get("nr") or m, rule.get("ntheta") or m // 2, rule.get("nphi") or m


def _split_rule(length):
    k = 6.0 * 9.6 / min(length) * math.sqrt(sum(v * v for v in length))

    def up(v, least):
        return max(least, int(math.ceil(v / 8.0) * 8))
    return up(0.48 * k, 16), up(0.32 * k, 8), up(0.64 * k, 16)


def _ddi_work(n, nodes, real, taps, fft_sweeps=1):
    """One DDI: the density and the potential once each and a position and a weight per node
    of one half of the set; w^d complex taps per node and transform, and the fine grid's FFTs
    (a quarter of whole transforms: real data, zero padding)."""
    cells = math.prod(n)
    fine = cells * 2 ** len(n)
    fft = 2 * fft_sweeps * 0.25 * 5.0 * fine * math.log2(fine)
    return {"bytes": real * (2.0 * cells + 0.5 * nodes * (len(n) + 1)), "flops": 2 * 0.5 * nodes * 4.0 * taps + fft}


def work(case):
    if case["kind"] in ("ddi", "split"):
        n, _, length, rule, _, _ = _geometry(case)
        real, w = (8, 14) if case["prec"] == "fp64" else (4, 8)
        if case["dim"] == 2:
            nodes = (rule["nr"] or 2 * max(n)) * (rule["nphi"] or 2 * max(n))
        elif case["kind"] == "split":
            nodes = math.prod(_split_rule(length))
        else:
            nodes = math.prod(_rule3(n, rule))
        return _ddi_work(n, nodes, real, w ** case["dim"], 2 if case["kind"] == "split" else 1)
    if case["kind"] == "batch":
        parts = [_ddi_work(n, 4 * n[0] * n[0], 4, 64) for n, _, _, _ in _batch_items(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n = (case["n"],) * 3
    real, w = (8, 14) if case["prec"] == "fp64" else (4, 8)
    cells = math.prod(n)
    one = _ddi_work(n, math.prod(_rule3(n, {})), real, w ** 3)
    fft = 2 * 5.0 * cells * math.log2(cells)
    # DDIs and kinetic transform pairs of a pass; the state and the trap are read and written once a step
    ddis, ffts = {"step": (1, 1), "ground": (1.4, 10), "gradient": (4, 5)}[case["kind"]]
    return {"bytes": case["steps"] * (ddis * one["bytes"] + 5.0 * real * cells),
            "flops": case["steps"] * (ddis * one["flops"] + ffts * fft)}


# ---- the same results in FP64 by plain torch --------------------------------------------------------
def _legendre(count):
    x, w = np.polynomial.legendre.leggauss(count)
    return x, w


class _Direct3:
    """Phi = Re sum_q W_q e^{i k_q.x} h^3 sum_j rho_j e^{-i k_q.x_j} over the spherical rule,
    ring by ring: e^{-i k.x} = e^{-i k_z z} e^{-i k_y y} e^{-i k_x x} with one k_z per ring."""

    def __init__(self, n, lo, length, rule, axis_n, axis_m=None, kmax=0.0, window=0.0):
        self.n, self.dev = n, _device()
        self.x = _coords(n, lo, length)
        h = [length[a] / n[a] for a in range(3)]
        self.dv = math.prod(h)
        nr, nt, nphi = rule
        R = kmax or math.pi / min(h)
        xr, wr = _legendre(nr)
        u, wu = _legendre(nt)
        r, wr = 0.5 * R * (1.0 + xr), 0.5 * R * wr
        ang = 2.0 * math.pi * np.arange(nphi // 2) / nphi  # one node of each +-k pair, twice
        kr, kz = np.outer(r, np.sqrt(1.0 - u * u)).ravel(), np.outer(r, u).ravel()
        wgt = (np.outer(wr * r * r, wu) * (2.0 * math.pi / nphi)).ravel()
        if window:
            wgt = wgt * np.exp(-(kr * kr + kz * kz) / window ** 2)
        self.ring = [torch.from_numpy(v).to(self.dev) for v in (kr, kz, wgt)]
        self.cs = torch.from_numpy(np.stack([np.cos(ang), np.sin(ang)])).to(self.dev)
        self.dirs = torch.from_numpy(np.stack([np.broadcast_to(np.sqrt(1.0 - u * u), (nr, nt)).ravel(),
                                               np.broadcast_to(u, (nr, nt)).ravel()])).to(self.dev)
        self.set_axes(axis_n, axis_m)

    def set_axes(self, axis_n, axis_m=None):
        self.a, self.b = axis_n, axis_m or axis_n

    def __call__(self, rho):
        nx, ny, nz = self.n
        kr, kz, wgt = self.ring
        out = torch.zeros(nz, ny * nx, dtype=torch.float64, device=self.dev)
        flat = rho.reshape(nz, ny * nx).to(torch.float64)
        m = self.cs.shape[1]
        step = max(1, min(kr.numel(), int(6e7 // max(ny * nx, m * max(nx, ny)))))
        nm = sum(p * q for p, q in zip(self.a, self.b))
        for i in range(0, kr.numel(), step):
            j = slice(i, i + step)
            az = kz[j, None] * self.x[2][None, :]
            cz, sz = torch.cos(az), torch.sin(az)
            G = torch.complex(cz @ flat, -(sz @ flat)).reshape(-1, ny, nx)
            ax = (kr[j, None] * self.cs[0])[:, :, None] * self.x[0]
            ay = (kr[j, None] * self.cs[1])[:, :, None] * self.x[1]
            Ex, Ey = torch.complex(torch.cos(ax), -torch.sin(ax)), torch.complex(torch.cos(ay), -torch.sin(ay))
            f = (torch.bmm(Ey, G) * Ex).sum(-1)
            st, u = self.dirs[0][j, None], self.dirs[1][j, None]
            nk = st * (self.a[0] * self.cs[0] + self.a[1] * self.cs[1]) + u * self.a[2]
            mk = st * (self.b[0] * self.cs[0] + self.b[1] * self.cs[1]) + u * self.b[2]
            c = f * (2.0 * self.dv * wgt[j, None] * (3.0 * nk * mk - nm) / (2.0 * math.pi) ** 3)
            T = torch.bmm(Ey.conj().transpose(1, 2), c[:, :, None] * Ex.conj()).reshape(-1, ny * nx)
            out += cz.T @ T.real - sz.T @ T.imag  # Re(e^{+i kz z} T)
        return out.reshape(nz, ny, nx)


def _direct2(rho, n, lo, length, nr, nphi, axis_n, axis_m=None):
    """The 2D quadrature sum by its definition, in blocks of nodes."""
    x, y = _coords(n, lo, length)
    h = [length[a] / n[a] for a in range(2)]
    xr, wr = _legendre(nr)
    R = math.pi / min(h)
    r, wr = 0.5 * R * (1.0 + xr), 0.5 * R * wr
    ang = 2.0 * math.pi * np.arange(nphi // 2) / nphi
    c, s = np.cos(ang), np.sin(ang)
    b = axis_m or axis_n
    sym = 1.5 * ((axis_n[0] * c + axis_n[1] * s) * (b[0] * c + b[1] * s) - axis_n[2] * b[2])
    dev = _device()
    kx, ky, W = (torch.from_numpy(v.ravel()).to(dev) for v in
                 (np.outer(r, c), np.outer(r, s),
                  2.0 * h[0] * h[1] * np.outer(wr * r * r, sym) * (2.0 * math.pi / nphi) / (2.0 * math.pi) ** 2))
    src = rho.to(torch.float64)
    out = torch.zeros_like(src)
    step = 1 << 15
    for i in range(0, kx.numel(), step):
        ax, ay = kx[i:i + step, None] * x, ky[i:i + step, None] * y
        cx, sx, cy, sy = torch.cos(ax), torch.sin(ax), torch.cos(ay), torch.sin(ay)
        P, Q = cx @ src.T, sx @ src.T  # sum over x: P - i Q
        fr, fi = (cy * P - sy * Q).sum(1), -(cy * Q + sy * P).sum(1)
        fr, fi = (fr * W[i:i + step])[:, None], (fi * W[i:i + step])[:, None]
        # Re[(fr + i fi) e^{i ky y} e^{i kx x}]
        out += (fr * cy - fi * sy).T @ cx - (fr * sy + fi * cy).T @ sx
    return out


def _smooth_part(rho, n, length, axis_n, axis_m, k0):
    """The split algorithm's smooth part: the zero-padded FFT convolution with (1 - q) Uhat."""
    dev, b = rho.device, axis_m or axis_n
    k = [2.0 * math.pi * torch.fft.fftfreq(2 * n[a], d=length[a] / n[a], dtype=torch.float64, device=dev)
         for a in range(3)]
    kz, ky, kx = k[2][:, None, None], k[1][None, :, None], k[0][None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    f = torch.where(k2 > 0, -torch.expm1(-k2 / k0 ** 2) / torch.where(k2 > 0, k2, torch.ones_like(k2)),
                    torch.full_like(k2, 1.0 / k0 ** 2))
    nk = axis_n[0] * kx + axis_n[1] * ky + axis_n[2] * kz
    mk = b[0] * kx + b[1] * ky + b[2] * kz
    P = f * (3.0 * nk * mk - sum(p * q for p, q in zip(axis_n, b)) * k2)
    del f, nk, mk, k2
    F = torch.fft.fftn(rho.to(torch.float64), s=[2 * v for v in reversed(n)])
    return torch.fft.ifftn(F * P)[: n[2], : n[1], : n[0]].real.contiguous()


class _SelfAdjoint(torch.autograd.Function):
    @staticmethod
    def forward(ctx, rho, op):
        ctx.op = op
        return op(rho)

    @staticmethod
    def backward(ctx, g):
        return ctx.op(g), None


def _kinetic(psi, length, f):
    mu = [2.0 * math.pi * torch.fft.fftfreq(psi.shape[2 - a], d=1.0 / psi.shape[2 - a], dtype=torch.float64,
                                            device=psi.device) / length[a] for a in range(3)]
    m2 = mu[2][:, None, None] ** 2 + mu[1][None, :, None] ** 2 + mu[0][None, None, :] ** 2
    return torch.fft.ifftn(torch.fft.fftn(psi) * torch.exp(1j * f * m2)), m2


def _step(psi, V, beta, lam, dt, length, op, loss=False):
    psi, _ = _kinetic(psi, length, -0.25 * dt)
    rho = psi.real ** 2 + psi.imag ** 2
    if not loss:
        psi = psi * torch.exp(-1j * dt * (V + beta * rho + lam * op(rho)))
    else:  # three-body loss f = delta rho^2, sigma = 1
        q, delta = 2.0, 3.512
        L = torch.log1p(2.0 * q * delta * dt * rho ** q)
        safe = torch.where(rho > 0, rho, torch.ones_like(rho))
        g = torch.where(rho > 0, torch.expm1((1.0 - 1.0 / q) * L) / (2.0 * delta * (q - 1.0) * safe ** (q - 1.0)),
                        torch.zeros_like(rho))
        psi = psi * torch.exp(-1j * (dt * V + beta * g + lam * op(g)) - L / (2.0 * q))
    return _kinetic(psi, length, -0.25 * dt)[0]


def _flow(case, psi, V, length, op):
    """Backward-Euler gradient flow with converged solves, and the energies at its end."""
    beta, lam, dt = case["beta"], case["lam"], case["dt"]
    dv = math.prod(length[a] / case["n"] for a in range(3))
    _, m2 = _kinetic(psi, length, 0.0)

    def unit(a):
        return a / torch.sqrt(dv * (a.real ** 2 + a.imag ** 2).sum())
    phi = unit(psi)
    for _ in range(case["steps"]):
        rho = phi.real ** 2 + phi.imag ** 2
        W = V + beta * rho + lam * op(rho)
        alpha = 0.5 * (W.max() + W.min())
        cur = phi
        for _ in range(200):
            new = torch.fft.ifftn(torch.fft.fftn(phi / dt + (alpha - W) * cur) / (1.0 / dt + alpha + 0.5 * m2))
            done = (new - cur).abs().max() <= 1e-14
            cur = new
            if done:
                break
        phi = unit(cur)
    rho = phi.real ** 2 + phi.imag ** 2
    hat = torch.fft.fftn(phi)
    kin = float(0.5 * dv / rho.numel() * (m2 * (hat.real ** 2 + hat.imag ** 2)).sum())
    pot, inter = float(dv * (V * rho).sum()), float(0.5 * beta * dv * (rho * rho).sum())
    dip, mass = float(0.5 * lam * dv * (op(rho) * rho).sum()), float(dv * rho.sum())
    E = kin + pot + inter + dip
    return phi, [E, E + inter + dip, kin, pot, inter, dip, mass]


def _reachable3(n, nodes):
    """Whether the direct sum stays within seconds (about 4 (rings nz + nodes) nx ny FP64 operations)."""
    return math.prod(n[:2]) * (nodes * 1.5) < 2e11


def exact(case, seed):
    with torch.no_grad():
        return _exact(case, seed)


def _exact(case, seed):
    if case["kind"] in ("ddi", "split"):
        n, lo, length, rule, axis_n, axis_m = _geometry(case)
        rho = _mixture(n, lo, length, seed, 8 if case["dim"] == 3 else 4).to(_dtypes(case["prec"])[0]).double()
        if case["dim"] == 2:
            if max(n) > 512:
                return None
            return _direct2(rho, n, lo, length, rule["nr"] or 2 * max(n), rule["nphi"] or 2 * max(n), axis_n, axis_m)
        if case["kind"] == "ddi":
            sizes = _rule3(n, rule)
            if not _reachable3(n, math.prod(sizes)):
                return None
            return _Direct3(n, lo, length, sizes, axis_n, axis_m)(rho)
        k0 = 9.6 / min(length)
        ball = _Direct3(n, lo, length, _split_rule(length), axis_n, axis_m, kmax=6.0 * k0, window=k0)
        return ball(rho) + _smooth_part(rho, n, length, axis_n, axis_m, k0)
    if case["kind"] == "batch":
        out = []
        for i, (n, lo, ln, axis) in enumerate(_batch_items(case)):
            rho = _mixture(n, lo, ln, seed * 1000 + i, 4).float().double()
            out.append(_direct2(rho, n, lo, ln, 2 * n[0], 2 * n[0], axis) if n[0] <= 256 else None)
        return out
    real, cplx, _ = _dtypes(case["prec"])
    n, lo, length, V, psi = _gpe_inputs(case, seed)
    V, psi = V.to(real).double(), psi.to(cplx).to(torch.complex128)
    op = _Direct3(n, lo, length, _rule3(n, {}), (0.0, 0.0, 1.0))
    beta, lam, dt = case["beta"], case["lam"], case["dt"]
    if case["kind"] == "step":
        for k in range(case["steps"]):
            if case["mode"] == "rotating":
                op.set_axes(_rotating(case, k))
            psi = _step(psi, V, beta, lam, dt, length, op, case["mode"] == "loss")
        return psi
    if case["kind"] == "ground":
        return _flow(case, psi, V, length, op)
    with torch.enable_grad():
        Vg = V.clone().requires_grad_(True)
        cur = psi
        for _ in range(case["steps"]):
            cur = _step(cur, Vg, beta, lam, dt, length, lambda r: _SelfAdjoint.apply(r, op))
        x2 = _coords(n, lo, length)[2] ** 2
        J = math.prod(length[a] / n[a] for a in range(3)) * (x2[:, None, None] * (cur.real ** 2 + cur.imag ** 2)).sum()
        (g,) = torch.autograd.grad(J, Vg)
    return float(J), g
