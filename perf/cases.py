"""The work this library is used for, as cases of measurable size.

Every case runs one of the library's public entry points the way a program calls it: the
reaction table of one element on one substrate (FP64 and FP32-mixed, one or four rotation
classes), a batched sweep of substrates and frequencies, the reduced matrix of an array
(a few elements up to the 10,000-element array), an objective with its gradient, the
reduced system's solution, and the 2-D Cartesian form.  Sizes are those of the library's
own workloads (``workloads/``, ``bench.py``) and generic ones between them.

``exact`` evaluates the same definitions in plain torch in float64: the contour sum with
exact exponentials, the angular quadrature, the array sums.
"""
import math

import numpy as np
import torch

import workloads
from paper_1404_7357_gb300 import autograd, cfft

DEVICE = 0
DEV = "cuda:%d" % DEVICE
K0 = 2.0 * math.pi
Z0 = 376.730313668
TAPS = 20           # Lagrange taps of exact()'s grids ...
OVERSAMPLE = 16     # ... whose spacing is 2 pi / (OVERSAMPLE * beta_max)
PORT = 37           # basis function that carries the delta-gap port


# ----------------------------------------------------------------------------- the cases

def _table(name, **kw):
    c = {"name": name, "kind": "table", "element": "patch", "m": 4, "precision": "fp32", "classes": 1,
         "n": 16384, "n_rho": 8192, "rho_max": 50.0, "q_max": 16, "eps_r": 4.4, "h": 0.03}
    c.update(kw)
    return c


def _array(name, kind, **kw):
    return _table(name, kind=kind, **kw)


def listed():
    return [
        # one strip dipole in FP64: the smallest table, launches and host work count
        _table("strip table fp64", element="strip", m=1, precision="fp64", n=1024, n_rho=1024, rho_max=10.0,
               q_max=4, eps_r=2.2, h=0.05),
        # the patch of 200 rooftops, 16 MBF pairs, 50 wavelengths: the ordinary table
        _table("patch table fp32"),
        # the same element in FP64 over a quarter of the range
        _table("patch table fp64", precision="fp64", n=4096, n_rho=2047, rho_max=12.5),
        # two MBFs, rotated elements, a contour length that is no power of two, a ragged rho grid
        _table("rotated table fp32", m=2, classes=4, n=6144, n_rho=3001, rho_max=24.0, q_max=11),
        # sweep over frequencies and substrates with uneven contours, one graph per sweep
        {"name": "sweep fp32", "kind": "sweep", "m": 4, "freqs": 4, "subs": 4, "n_rho": 2048, "rho_max": 50.0,
         "q_max": 16},
        # a few elements: the fill's latency
        _array("fill 24 fp32", "fill", layout="irregular", elements=24, radius=2.6, n_rho=1024, rho_max=6.0,
               n=2048, q_max=8),
        # the paper's 25 x 25 regular array, FP64
        _array("fill regular 625 fp64", "fill", layout="regular", elements=625, radius=0.0, precision="fp64",
               n=4096, n_rho=2048, rho_max=18.0, q_max=8),
        # the large irregular array: 10,000 rotated elements, a 40,000 x 40,000 matrix
        _array("fill irregular 10000 fp32", "fill", layout="irregular", elements=10000, radius=60.0, classes=4,
               n_rho=16384, rho_max=121.0),
        # objective and gradient with respect to positions and substrate (forward and backward)
        _array("gradient 2000 fp32", "grad", layout="irregular", elements=2000, radius=25.0, classes=4),
        # the reduced system of 2,000 elements, complex64
        {"name": "solve 8000 c64", "kind": "solve", "n": 8000, "m": 4, "dtype": "c64", "refine": False},
        # a reduced system to float64 accuracy: complex64 factors refined in float64
        {"name": "solve 2500 c128 refined", "kind": "solve", "n": 2500, "m": 4, "dtype": "c128", "refine": True},
        # the 2-D Cartesian form: its table and a fill of unrotated elements
        {"name": "cartesian 128 fp32", "kind": "cartesian", "m": 4, "precision": "fp32", "n_grid": 128,
         "elements": 200, "rho_max": 2.5, "eps_r": 4.4, "h": 0.03, "height": 0.1},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_table(rng, n_rho_max, rho_hi, fp64_share):
    fp64 = rng.random() < fp64_share
    strip = rng.random() < 0.2
    n = 16 * 2 ** rng.randrange(3, 7) * rng.choice([1, 2, 3, 5, 7, 8])
    eps_r = round(rng.uniform(2.0, 6.0), 2)
    n = min(n, 4096 if fp64 else 16384)
    rho_max = round(min(_log(rng, 4.0, rho_hi), 0.4 * math.pi * n / (5.0 * K0 * math.sqrt(eps_r))), 2)
    if fp64:
        rho_max = min(rho_max, 16.0)
    # at least 80 points a wavelength in the largest tables, more in the small ones
    n_rho = int(min(2048 if fp64 else n_rho_max, _log(rng, 90.0 * rho_max, 200.0 * rho_max) + 64))
    return {"element": "strip" if strip else "patch", "m": 1 if strip else rng.choice([1, 2, 3, 4, 4, 4]),
            "precision": "fp64" if fp64 else "fp32", "classes": rng.choice([1, 1, 4]), "n": n, "n_rho": n_rho,
            "rho_max": rho_max, "q_max": rng.randrange(4, 17), "eps_r": eps_r, "h": round(rng.uniform(0.02, 0.08), 3)}


def draw(rng):
    kind = rng.choice(["table", "table", "sweep", "fill", "fill", "grad", "solve", "cartesian"])
    if kind == "table":
        return dict(_draw_table(rng, 8192, 50.0, 0.3), kind="table")
    if kind == "sweep":
        return {"kind": "sweep", "m": rng.choice([1, 2, 4]), "freqs": rng.randrange(1, 5), "subs": rng.randrange(1, 5),
                "n_rho": int(_log(rng, 300, 2049)), "rho_max": round(_log(rng, 8.0, 50.0), 1),
                "q_max": rng.randrange(4, 17)}
    if kind == "solve":
        m = rng.choice([1, 2, 4])
        dtype = rng.choice(["c64", "c64", "c128"])
        n = m * max(1, int(_log(rng, 24, 6000 if dtype == "c64" else 2000)) // m)
        return {"kind": "solve", "n": n, "m": m, "dtype": dtype, "refine": dtype == "c128" and rng.random() < 0.5}
    if kind == "cartesian":
        n, eps_r = rng.choice([64, 128, 128, 256]), round(rng.uniform(2.0, 5.0), 2)
        reach = n * math.pi / (2.0 * 5.0 * K0 * math.sqrt(eps_r))       # half the table's width
        return {"kind": "cartesian", "m": rng.choice([1, 2, 4]), "precision": rng.choice(["fp32", "fp32", "fp64"]),
                "n_grid": n, "elements": int(_log(rng, 4, 300)), "rho_max": round(rng.uniform(0.4, 0.9) * reach, 2),
                "eps_r": eps_r, "h": round(rng.uniform(0.02, 0.08), 3), "height": round(rng.uniform(0.05, 0.15), 3)}
    c = _draw_table(rng, 8192, 44.0, 0.3 if kind == "fill" else 0.0)
    most = (800 if c["precision"] == "fp64" else 6000) if kind == "fill" else 2000
    a = int(_log(rng, 8, most))
    # the array's disc follows its element count (about the density of the large array) within the table
    radius = min(0.49 * c["rho_max"], 0.5 * math.sqrt(2.2 * a) + 0.6)
    a = min(a, int((radius / 0.5) ** 2 * 1.2))
    c.update(kind=kind, elements=max(2, a), radius=round(radius, 3), layout="irregular")
    if kind == "fill" and c["classes"] == 1 and rng.random() < 0.4:
        side = max(2, min(int(math.sqrt(a)), int(0.98 * c["rho_max"] / (0.6 * math.sqrt(2.0)))))
        c.update(layout="regular", elements=side * side, radius=0.0)
    return c


# ---------------------------------------------------------------- inputs made from the seed

def _rng(seed):
    return np.random.default_rng([7919, int(seed)])


def _substrate(case, seed):
    u = _rng(seed).uniform(-1.0, 1.0, 2)
    return case["eps_r"] * (1.0 + 0.02 * u[0]), case["h"] * (1.0 + 0.02 * u[1])


def _element(case, seed):
    """Mesh and MBF coefficients: a 0.5 x 0.5 patch of 200 rooftops with complex-normal
    coefficients drawn with the seed, or one strip dipole (its length follows the seed)."""
    if case.get("element") == "strip":
        return workloads.strip_element(length=0.45 + 0.01 * float(_rng(seed).uniform(-1.0, 1.0)))
    return workloads.patch_rooftops(n_mbf=case["m"], seed=1000 + int(seed))


def _contour(case, eps_r, n, rho_max):
    """5 k_d long, parabola to 1.3 k_d, six node spacings high with height * rho_max <= 3."""
    sub = workloads.Substrate(eps_r, case["h"])
    c = workloads.default_contour(sub, n)
    c.height = min(c.height, 3.0 / rho_max)
    return c


def _positions(case, seed):
    if case["layout"] == "regular":
        side = int(round(math.sqrt(case["elements"])))
        pitch = 0.5 + 0.02 * float(_rng(seed).uniform(0.0, 1.0))
        g = np.arange(side) * pitch
        return np.stack(np.meshgrid(g, g, indexing="ij"), -1).reshape(-1, 2).copy()
    return workloads.poisson_disc(case["elements"], case["radius"], 0.5, seed=2000 + int(seed))


def _rotations(case, seed):
    if case["classes"] == 1:
        return None
    return workloads.rotations(case["elements"], seed=3000 + int(seed))


def _sweep_items(case, seed):
    """Substrates over eps_r 2..10 and h 0.02..0.1, frequencies 0.8..1.2, contours of 4k..64k
    nodes in a fixed uneven order, lengthened until their s period covers the table three times."""
    rng = _rng(seed)
    items = []
    for fi in range(case["freqs"]):
        f = 0.8 + 0.4 * (fi + 0.5) / case["freqs"]
        for si in range(case["subs"]):
            eps = (2.0 + 8.0 * (si + 0.5) / case["subs"]) * (1.0 + 0.02 * rng.uniform(-1.0, 1.0))
            h = (0.02 + 0.08 * ((3 * si + 1) % case["subs"] + 0.5) / case["subs"]) * (1.0 + 0.02 * rng.uniform(-1.0, 1.0))
            kd = K0 * f * math.sqrt(eps)
            n = 4096 * 2 ** ((3 * fi + 2 * si) % 4)
            while K0 / (5.0 * kd / n) < 6.0 * case["rho_max"]:
                n *= 2
            step = 5.0 * kd / n
            items.append({"eps_r": eps, "h": h, "k0": K0 * f, "n": n, "beta_max": 5.0 * kd,
                          "beta_p": round(1.3 * kd / step) * step,
                          "height": min(6.0 * step, 3.0 / case["rho_max"]), "taylor_order": -1})
    return items


def _reduced_system(case, seed):
    """A matrix with the structure of a reduced array matrix: M x M blocks, self blocks on the
    diagonal, couplings by a space wave exp(-j k0 r) / (k0 r) and a weaker surface wave
    / sqrt(k0 r) with a pattern in the azimuth, as well conditioned as an array's; excitation."""
    n, m = case["n"], case["m"]
    a = n // m
    rng = _rng(seed)
    side = int(math.ceil(math.sqrt(a)))
    g = np.stack(np.meshgrid(np.arange(side), np.arange(side), indexing="ij"), -1).reshape(-1, 2)[:a]
    pos = torch.tensor(0.62 * g + rng.uniform(-0.06, 0.06, (a, 2)), device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(4000 + int(seed))
    d = pos[:, None] - pos[None]
    r = torch.hypot(d[..., 0], d[..., 1]) + torch.eye(a, device=DEV, dtype=torch.float64)
    w = torch.polar(1.0 / (K0 * r) + 0.02 / torch.sqrt(K0 * r), -K0 * r) * (1.0 + 0.3 * d[..., 0] * d[..., 1] / r ** 2)
    w.fill_diagonal_(0.0)
    c0 = torch.randn((m, m), generator=gen, device=DEV, dtype=torch.complex128)
    self_block = (3.0 - 1.5j) * torch.linalg.qr(c0)[0]
    cpl = 0.35 * torch.randn((m, m), generator=gen, device=DEV, dtype=torch.complex128)
    z = torch.einsum("mn,ab->manb", w, cpl)
    k = torch.arange(a, device=DEV)
    z[k, :, k, :] += self_block
    v = torch.randn(n, generator=gen, device=DEV, dtype=torch.complex128)
    dt = torch.complex64 if case["dtype"] == "c64" else torch.complex128
    return z.reshape(n, n).to(dt).contiguous(), v.to(dt).contiguous()


def _vectors(n, seed):
    return (torch.tensor(workloads.complex_normal(n, 5000 + 2 * int(seed) + i), device=DEV).to(torch.complex64)
            for i in range(2))


def _beta_max_cartesian(case, eps_r):
    return 5.0 * K0 * math.sqrt(eps_r)


# ----------------------------------------------------------------------------- prepare, run

def _precision(case):
    return cfft.CFFT_FP64 if case["precision"] == "fp64" else cfft.CFFT_FP32_MIXED


def _set_element(ctx, el):
    if el.kind == "strip":
        ctx.set_mbf_spectra_strip(el.length, el.strip_width)
    else:
        ctx.set_mbf_spectra(np.stack([el.cx, el.cy], 1), el.direction, el.half_len, el.width, el.q)


def _tabulate(ctx, case, sub, c):
    ctx.set_substrate(sub[0], sub[1], K0)
    ctx.build_contour(c.n, c.beta_max, c.beta_p, c.height)
    ctx.tabulate_reactions(case["q_max"], case["rho_max"], case["n_rho"], _precision(case), case["classes"])


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "solve":
        s["ctx"] = cfft.Context(DEVICE)
        s["z"], s["v"] = _reduced_system(case, seed)
        return s
    el = _element(case, seed)
    if kind == "sweep":
        s["ctx"] = cfft.Context(DEVICE)
        _set_element(s["ctx"], el)
        s["items"] = _sweep_items(case, seed)
        s["out"] = torch.empty((len(s["items"]), case["m"] ** 2, 2 * case["q_max"] + 1, case["n_rho"]),
                               dtype=torch.complex64, device=DEV)
        return s
    sub = s["sub"] = _substrate(case, seed)
    if kind == "cartesian":
        ctx = s["ctx"] = cfft.Context(DEVICE)
        _set_element(ctx, el)
        s["pos"] = torch.tensor(_cartesian_positions(case, seed), device=DEV)
        n = case["elements"] * case["m"]
        s["z"] = torch.empty((n, n), device=DEV,
                             dtype=torch.complex128 if case["precision"] == "fp64" else torch.complex64)
        return s
    c = s["contour"] = _contour(case, sub[0], case["n"], case["rho_max"])
    if kind == "table":
        s["ctx"] = cfft.Context(DEVICE)
        _set_element(s["ctx"], el)
        s["out"] = torch.empty((case["classes"], case["m"] ** 2, 2 * case["q_max"] + 1, case["n_rho"]), device=DEV,
                               dtype=torch.complex128 if case["precision"] == "fp64" else torch.complex64)
        return s
    pos = _positions(case, seed)
    rot = _rotations(case, seed)
    s["pos"] = torch.tensor(pos, device=DEV)
    s["rot"] = None if rot is None else torch.tensor(rot, device=DEV)
    if kind == "fill":
        s["ctx"] = cfft.Context(DEVICE)
        _set_element(s["ctx"], el)
        _tabulate(s["ctx"], case, sub, c)
        n = case["elements"] * case["m"]
        s["z"] = torch.empty((n, n), device=DEV,
                             dtype=torch.complex128 if case["precision"] == "fp64" else torch.complex64)
        return s
    s["problem"] = autograd.FillProblem(el, K0, c, case["q_max"], case["rho_max"], case["n_rho"],
                                        case["precision"], rot=s["rot"], device=DEVICE)
    s["eps_h"] = torch.tensor(sub, dtype=torch.float64, device=DEV)
    s["v"], s["t"] = _vectors(case["elements"] * case["m"], seed)
    return s


def _cartesian_positions(case, seed):
    """Distinct points of a jittered lattice whose largest distance stays below rho_max."""
    side = int(math.ceil(math.sqrt(case["elements"])))
    g = np.stack(np.meshgrid(np.arange(side), np.arange(side), indexing="ij"), -1).reshape(-1, 2)[:case["elements"]]
    p = (g + _rng(seed).uniform(-0.2, 0.2, g.shape)) / (side + 0.4)
    return 0.98 * case["rho_max"] / math.sqrt(2.0) * p


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "table":
        _tabulate(s["ctx"], case, s["sub"], s["contour"])
        return s["ctx"].copy_table(out=s["out"])
    if kind == "sweep":
        s["ctx"].tabulate_batch(s["items"], case["q_max"], case["rho_max"], case["n_rho"], cfft.CFFT_FP32_MIXED,
                                out=s["out"], graph=True)
        return list(s["out"].unbind(0))
    if kind == "fill":
        return s["ctx"].fill_reduced_matrix(s["pos"], s["rot"], s["z"])
    if kind == "grad":
        pos = s["pos"].detach().requires_grad_(True)
        eps_h = s["eps_h"].detach().requires_grad_(True)
        z = autograd.ReducedMatrix.apply(pos, eps_h, s["problem"])
        loss = ((z @ s["v"] - s["t"]).abs() ** 2).sum()
        loss.backward()
        return {"loss": loss.detach(), "z": z.detach(), "grad_pos": pos.grad, "grad_eps_h": eps_h.grad}
    if kind == "solve":
        return s["ctx"].solve_reduced(s["z"], s["v"], refine=case["refine"])
    ctx = s["ctx"]
    ctx.set_substrate(s["sub"][0], s["sub"][1], K0)
    bm = _beta_max_cartesian(case, s["sub"][0])
    ctx.build_contour(case["n_grid"], bm, 0.26 * bm, case["height"])
    ctx.tabulate_cartesian(case["n_grid"], case["rho_max"], _precision(case))
    ctx.fill_cartesian(s["pos"], s["z"])
    return {"table": ctx.cartesian_table(), "z": s["z"]}


# ------------------------------------------------------------------------------------ work

def _table_work(n, beta_max, radius, basis, m, q_max, rho_max, n_rho, classes, sigma):
    """Operations of one tabulation: spectra and kernel at every (node, angle), the harmonics, one
    zero-padded FFT per (pair, harmonic), and the quadrature over the table's own samples."""
    na = 2.0 * beta_max * radius + 2.0 * q_max + 32.0
    nh, pairs, cc = 2 * q_max + 1, m * m, 1 if classes == 1 else 3
    series = cc * pairs * nh
    length = sigma * n
    flops = n * na * (8.0 * basis * 2.0 * m + cc * pairs * (16.0 + 5.0 * math.log2(na)))
    flops += series * 5.0 * length * math.log2(length)
    flops += series * n_rho * 8.0 * beta_max * rho_max / 4.0
    return flops


def work(case):
    kind = case["kind"]
    wide = case.get("precision") == "fp64" or case.get("dtype") == "c128"
    e = 16 if wide else 8
    if kind == "solve":
        n = case["n"]
        return {"bytes": n * n * e + 2 * n * e, "flops": 8.0 * n ** 3 / 3.0 + 8.0 * n * n}
    m = case["m"]
    if kind == "sweep":
        flops, out = 0.0, 0
        for it in _sweep_items(case, 0):
            flops += _table_work(it["n"], it["beta_max"], 0.32, 200, m, case["q_max"], case["rho_max"], case["n_rho"], 1, 4)
            out += m * m * (2 * case["q_max"] + 1) * case["n_rho"] * 8
        return {"bytes": out + 200 * (36 + 16 * m), "flops": flops}
    if kind == "cartesian":
        order = 8                                       # the series order of height * rho_max ~ 0.4
        p = 2 * case["n_grid"]
        mono = (order + 1) * (order + 2) // 2
        flops = mono * m * m * (10.0 * p * p * math.log2(p) + 8.0 * p * p) + case["n_grid"] ** 2 * 8.0 * 200 * 2 * m
        flops += case["elements"] ** 2 * m * m * 36.0
        return {"bytes": (m * p) ** 2 * e + (case["elements"] * m) ** 2 * e, "flops": flops}
    basis = 1 if case["element"] == "strip" else 200
    beta_max = 5.0 * K0 * math.sqrt(case["eps_r"])
    nh = 2 * case["q_max"] + 1
    table = case["classes"] * m * m * nh * case["n_rho"] * e
    tab_flops = _table_work(case["n"], beta_max, 0.32, basis, m, case["q_max"], case["rho_max"], case["n_rho"],
                            case["classes"], 8 if wide else 4)
    if kind == "table":
        return {"bytes": table + basis * (36 + 16 * m), "flops": tab_flops}
    a = case["elements"]
    # per entry: the harmonic sum, and the interpolation of its stencil's taps
    fill = a * a * m * m * (8.0 * nh + 4.0 * (16 if wide else 8))
    z = (a * m) ** 2 * e
    if kind == "fill":
        return {"bytes": table + a * 20 + z, "flops": fill}
    # forward, objective, and the backward pass: the table with its two substrate derivatives, the adjoint
    return {"bytes": 2 * z + table + a * 36, "flops": 4.0 * tab_flops + 5.0 * fill + 16.0 * (a * m) ** 2}


# ----------------------------------------------------------------------------------- exact

def _nodes(n, beta_max, beta_p, height):
    step = beta_max / n
    br = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * step
    inside = br < beta_p
    bi = torch.where(inside, 4.0 * height * br * (beta_p - br) / beta_p ** 2, 0.0)
    slope = torch.where(inside, 4.0 * height * (beta_p - 2.0 * br) / beta_p ** 2, 0.0)
    return torch.complex(br, bi), step * torch.complex(torch.ones_like(br), slope)


def _green(beta_sq, eps_r, h, k0):
    """(P, R) of the grounded slab's dyadic P I - R k k^T at beta^2 (exp(+j w t), Im k2 <= 0)."""
    k1 = torch.sqrt(eps_r * k0 ** 2 - beta_sq)
    k2 = -1j * torch.sqrt(beta_sq - k0 ** 2)
    c, s = torch.cos(k1 * h), torch.sin(k1 * h)
    common = (-1j * Z0 / k0) * s / ((k1 * c + 1j * k2 * s) * (eps_r * k2 * c + 1j * k1 * s))
    return k0 ** 2 * (eps_r * k2 * c + 1j * k1 * s) * common, (k2 * c + 1j * k1 * s) * common


def _sinc(z):
    small = z.abs() < 1e-3
    safe = torch.where(small, torch.ones_like(z), z)
    return torch.where(small, 1.0 - z * z / 6.0 + z ** 4 / 120.0, torch.sin(safe) / safe)


def _spectra(el, kx, ky):
    """MBF spectra M_a(k) and their conjugate-side continuation: two (x, y) pairs of (M, points)."""
    f64 = {"dtype": torch.float64, "device": DEV}
    if el.kind == "strip":
        u = kx * el.length / 2.0
        u = torch.where(u.real < 0.0, -u, u)
        fx = (math.pi * el.length / 2.0) * _sinc(math.pi / 2.0 - u) / (math.pi / 2.0 + u) * _sinc(ky * el.strip_width / 2.0)
        zero = torch.zeros_like(fx)[None]
        return (fx[None], zero), (fx[None], zero)
    q = torch.tensor(el.q, device=DEV)
    side = {1: [], -1: []}
    for direction, ku, kv in ((0, kx, ky), (1, ky, kx)):
        i = np.flatnonzero(el.direction == direction)
        a, w = float(el.half_len[i[0]]), float(el.width[i[0]])       # one rooftop shape per direction
        shape = a * _sinc(ku * a / 2.0) ** 2 * _sinc(kv * w / 2.0)
        ph = -1j * (torch.outer(torch.tensor(el.cx[i], **f64).to(kx.dtype), kx) +
                    torch.outer(torch.tensor(el.cy[i], **f64).to(kx.dtype), ky))
        qi = q[torch.tensor(i, device=DEV)]
        side[1].append((qi.conj().T @ torch.exp(ph)) * shape)
        side[-1].append((qi.T @ torch.exp(-ph)) * shape)
    return tuple(side[1]), tuple(side[-1])


def _harmonics(el, beta_c, weight, q_max, classes, greens, radius=0.36):
    """[channel][class][pair][harmonic][node]: the kernel's azimuthal harmonics times beta w, for
    each (P, R) of ``greens``; class order (0,0), (0,90), (90,0), (90,90)."""
    need = 2.0 * float(beta_c.abs().max()) * radius * 1.5 + 2.0 * q_max + 48.0
    na = 4 * int(math.ceil(need / 4.0))
    alpha = torch.arange(na, dtype=torch.float64, device=DEV) * (2.0 * math.pi / na)
    ca, sa = torch.cos(alpha), torch.sin(alpha)
    qs = torch.arange(-q_max, q_max + 1, device=DEV) % na
    m, n = el.n_mbf, beta_c.numel()
    rots = [(0, 0)] if classes == 1 else [(0, 0), (0, 1), (1, 0), (1, 1)]
    out = torch.empty((len(greens), len(rots), m * m, 2 * q_max + 1, n), dtype=torch.complex128, device=DEV)
    chunk = max(1, 600_000 // na)
    for j in range(0, n, chunk):
        b = beta_c[j:j + chunk]
        shape = (b.numel(), na)
        kx, ky = b[:, None] * ca, b[:, None] * sa
        sides = [[x.reshape((m,) + shape) for x in xy] for xy in _spectra(el, kx.reshape(-1), ky.reshape(-1))]

        def rotated(side, r):
            x, y = sides[side]
            if not r:
                return x, y
            return -torch.roll(y, na // 4, -1), torch.roll(x, na // 4, -1)

        for ic, (rt, rb) in enumerate(rots):
            (tx, ty), (bx, by) = rotated(0, rt), rotated(1, rb)
            dot = tx[:, None] * bx[None] + ty[:, None] * by[None]
            kk = (kx * tx + ky * ty)[:, None] * (kx * bx + ky * by)[None]
            for ch, (p, r) in enumerate(greens):
                hk = p[j:j + chunk, None] * dot - r[j:j + chunk, None] * kk
                hq = torch.fft.fft(hk, dim=-1)[..., qs] / na
                hq = hq * (b * weight[j:j + chunk])[:, None]
                out[ch, ic, :, :, j:j + chunk] = hq.permute(0, 1, 3, 2).reshape(m * m, 2 * q_max + 1, -1)
    return out


def _lagrange(x, derivative=False):
    """Weights (.., TAPS) of the Lagrange stencil at nodes 0..TAPS-1, or those of its slope."""
    t = torch.arange(TAPS, dtype=torch.float64, device=x.device)
    den = torch.tensor([math.factorial(i) * math.factorial(TAPS - 1 - i) * (-1.0) ** (TAPS - 1 - i) for i in range(TAPS)],
                       dtype=torch.float64, device=x.device)
    d = x[..., None] - t
    left, right = torch.ones_like(d), torch.ones_like(d)
    left[..., 1:] = torch.cumprod(d[..., :-1], -1)
    right[..., :-1] = torch.flip(torch.cumprod(torch.flip(d[..., 1:], [-1]), -1), [-1])
    if not derivative:
        return left * right / den
    dl, dr = torch.zeros_like(d), torch.zeros_like(d)
    for i in range(1, TAPS):
        dl[..., i] = dl[..., i - 1] * d[..., i - 1] + left[..., i - 1]
        k = TAPS - 1 - i
        dr[..., k] = dr[..., k + 1] * d[..., k + 1] + right[..., k + 1]
    return (dl * right + left * dr) / den


def _rho_table(y, beta_c, beta_max, q_max, rho):
    """Z_q(rho) = 1/(2 pi^2) int_0^pi cos(q a) g_q(rho cos a) da for y[..., harmonic, node] at the
    points ``rho`` (ascending): g by its exact exponential sum on a fine grid, the midpoint rule in a."""
    lead = y.shape[:-2]
    nh = 2 * q_max + 1
    ds = 2.0 * math.pi / (OVERSAMPLE * beta_max)
    top = int(math.ceil(float(rho[-1]) / ds)) + TAPS
    s = torch.arange(-top, top + 1, dtype=torch.float64, device=DEV) * ds
    yt = y.reshape(-1, y.shape[-1]).T.contiguous()                    # (node, series)
    g = torch.empty((s.numel(), yt.shape[1]), dtype=torch.complex128, device=DEV)
    # nodes off the real axis (a prefix): exponential by exponential; the others, equally spaced on
    # the axis, by one zero-padded FFT on the same grid
    n = beta_c.numel()
    off = int((beta_c.imag != 0).sum())
    rows = max(1, 60_000_000 // max(1, off))
    for k in range(0, s.numel(), rows):
        g[k:k + rows] = torch.exp(-1j * torch.outer(s[k:k + rows].to(torch.complex128), beta_c[:off])) @ yt[:off]
    k = torch.arange(-top, top + 1, device=DEV)
    turn = torch.polar(torch.ones_like(s), -math.pi / (OVERSAMPLE * n) * k.to(torch.float64))
    for c in range(0, yt.shape[1], 256):
        x = torch.zeros((OVERSAMPLE * n, yt[:, c:c + 256].shape[1]), dtype=torch.complex128, device=DEV)
        x[off:n] = yt[off:, c:c + 256]
        g[:, c:c + 256] += torch.fft.fft(x, dim=0)[k % (OVERSAMPLE * n)] * turn[:, None]
    g = torch.view_as_real(g.reshape(s.numel(), -1, nh)).permute(2, 0, 1, 3).contiguous()   # (nh, s, lead, 2)
    out = torch.empty((nh, rho.numel(), g.shape[2], 2), dtype=torch.float64, device=DEV)
    bmax = float(beta_c.abs().max())
    qv = torch.arange(0, q_max + 1, dtype=torch.float64, device=DEV)
    step = 32
    for r0 in range(0, rho.numel(), step):
        r = rho[r0:r0 + step]
        z = bmax * float(r[-1])
        npr = int(math.ceil((z + q_max + 44.0 + 8.0 * z ** (1.0 / 3.0)) / 2.0)) + 1
        half = int(math.ceil(float(r[-1]) / ds)) + TAPS
        a = (torch.arange(npr, dtype=torch.float64, device=DEV) + 0.5) * (math.pi / npr)
        u = (r[:, None] * torch.cos(a)) / ds + half
        i0 = torch.floor(u).long() - (TAPS // 2 - 1)
        w = _lagrange(u - i0)                                         # (rows, npr, TAPS)
        width = 2 * half + 1
        at = (torch.arange(r.numel(), device=DEV)[:, None, None] * width + i0[..., None] +
              torch.arange(TAPS, device=DEV)).reshape(-1)
        for q in range(q_max + 1):
            mat = torch.zeros(r.numel() * width, dtype=torch.float64, device=DEV)
            mat.index_add_(0, at, (w * torch.cos(qv[q] * a)[None, :, None]).reshape(-1))
            mat = mat.reshape(r.numel(), width) * (1.0 / (2.0 * math.pi * npr))
            for sgn in {q, -q}:
                seg = g[sgn + q_max, top - half:top + half + 1].reshape(width, -1)
                out[sgn + q_max, r0:r0 + r.numel()] = (mat @ seg).reshape(r.numel(), -1, 2)
    return torch.view_as_complex(out).permute(2, 0, 1).reshape(lead + (nh, rho.numel()))


def _fine_table(y, beta_c, beta_max, q_max, rho_max):
    """(row spacing, rows from -TAPS..) of Z_q on a grid fine enough for _lagrange at any rho:
    [.., row][harmonic], rows at negative rho from Z_q(-rho) = (-1)^q Z_q(rho)."""
    d = 2.0 * math.pi / (OVERSAMPLE * beta_max)
    n = int(math.ceil(rho_max / d)) + TAPS + 1
    z = _rho_table(y, beta_c, beta_max, q_max, torch.arange(n, dtype=torch.float64, device=DEV) * d)
    sign = (-1.0) ** torch.arange(-q_max, q_max + 1, device=DEV, dtype=torch.float64)
    z = torch.cat([torch.flip(z[..., 1:TAPS + 1], [-1]) * sign[:, None], z], -1)
    return d, z


def _case_harmonics(case, seed, derivatives=False):
    el, (eps_r, h) = _element(case, seed), _substrate(case, seed)
    c = _contour(case, eps_r, case["n"], case["rho_max"])
    beta_c, w = _nodes(c.n, c.beta_max, c.beta_p, c.height)
    b2 = beta_c * beta_c
    greens = [_green(b2, eps_r, h, K0)]
    if derivatives:
        for de, dh in ((1e-4 * eps_r, 0.0), (0.0, 1e-4 * h)):
            lo2, lo, hi, hi2 = [_green(b2, eps_r + f * de, h + f * dh, K0) for f in (-2, -1, 1, 2)]
            greens.append(tuple((8.0 * (y - x) - (y2 - x2)) / (12.0 * (de + dh))
                                for x2, x, y, y2 in zip(lo2, lo, hi, hi2)))
    return _harmonics(el, beta_c, w, case["q_max"], case["classes"], greens), beta_c, c


def _pairs(pos, rot):
    """Displacement, distance, azimuth and rotation class of every ordered element pair."""
    d = pos[:, None] - pos[None]
    rho = torch.hypot(d[..., 0], d[..., 1])
    phi = torch.atan2(d[..., 1], d[..., 0])
    cls = torch.zeros_like(rho, dtype=torch.long) if rot is None else 2 * rot[:, None].long() + rot[None].long()
    return rho, phi, cls


def _exact_fill(case, seed, grads=None):
    """The reduced matrix; with grads = (v, t) also the objective and its gradients."""
    y, beta_c, c = _case_harmonics(case, seed, derivatives=grads is not None)
    d, tab = _fine_table(y, beta_c, c.beta_max, case["q_max"], case["rho_max"])
    ch, cl, pp, nh, nr = tab.shape
    tab = tab.permute(1, 4, 0, 2, 3).reshape(cl * nr, ch, pp, nh).contiguous()
    pos = torch.tensor(_positions(case, seed), device=DEV)
    rot = _rotations(case, seed)
    rho, phi, cls = _pairs(pos, None if rot is None else torch.tensor(rot, device=DEV))
    a, m = pos.shape[0], case["m"]
    qs = torch.arange(-case["q_max"], case["q_max"] + 1, dtype=torch.float64, device=DEV)
    rows = max(1, int(2e8 // (a * ch * pp * nh)))

    def blocks(i):
        """Stencil sums of the pairs of test elements i..i+rows: values and rho slopes [pair][channel][ab][q]."""
        r, ph, cc = (x[i:i + rows].reshape(-1) for x in (rho, phi, cls))
        u = r / d + TAPS
        i0 = torch.floor(u).long() - (TAPS // 2 - 1)
        w = _lagrange(u - i0)
        dw = _lagrange(u - i0, True) / d if grads is not None else None
        val = torch.zeros((r.numel(), ch, pp, nh), dtype=torch.complex128, device=DEV)
        slope = torch.zeros((r.numel(), pp, nh), dtype=torch.complex128, device=DEV) if grads is not None else None
        for t in range(TAPS):
            x = tab[cc * nr + i0 + t]
            val.addcmul_(x, w[:, t, None, None, None].to(x.dtype))
            if slope is not None:
                slope.addcmul_(x[:, 0], dw[:, t, None, None].to(x.dtype))
        e = torch.exp(1j * ph[:, None] * qs)
        return r, ph, val, slope, e

    z = torch.empty((a, m, a, m), dtype=torch.complex128, device=DEV)
    for i in range(0, a, rows):
        r, ph, val, _, e = blocks(i)
        blk = torch.einsum("pkq,pq->pk", val[:, 0], e).reshape(-1, a, m, m)
        z[i:i + rows] = blk.permute(0, 2, 1, 3)
    z = z.reshape(a * m, a * m)
    if grads is None:
        return z
    v, t = (x.to(torch.complex128) for x in grads)
    res = z @ v - t
    gp = torch.zeros((a, 2), dtype=torch.float64, device=DEV)
    gt = torch.zeros(2, dtype=torch.float64, device=DEV)
    for i in range(0, a, rows):
        r, ph, val, slope, e = blocks(i)
        g = 2.0 * torch.einsum("ia,jb->ijab", res.reshape(a, m)[i:i + rows], v.reshape(a, m).conj()).reshape(-1, m * m)
        cg = g.conj()
        g_rho = (cg * torch.einsum("pkq,pq->pk", slope, e)).sum(-1).real
        g_phi = (cg * torch.einsum("pkq,pq->pk", val[:, 0], e * (1j * qs))).sum(-1).real
        inv = torch.where(r > 0, 1.0 / torch.where(r > 0, r, 1.0), 0.0)
        g_rho = torch.where(r > 0, g_rho, 0.0)
        gx = torch.cos(ph) * g_rho - torch.sin(ph) * inv * g_phi
        gy = torch.sin(ph) * g_rho + torch.cos(ph) * inv * g_phi
        gd = torch.stack([gx, gy], -1).reshape(-1, a, 2)
        gp[i:i + rows] += gd.sum(1)
        gp -= gd.sum(0)
        for k in range(2):
            gt[k] += (cg * torch.einsum("pkq,pq->pk", val[:, 1 + k], e)).sum().real
    return {"loss": (res.abs() ** 2).sum(), "z": z, "grad_pos": gp, "grad_eps_h": gt}


def _exact_cartesian(case, seed):
    el, (eps_r, h) = _element(case, seed), _substrate(case, seed)
    n, m = case["n_grid"], case["m"]
    bm = _beta_max_cartesian(case, eps_r)
    bp, height = 0.26 * bm, case["height"]
    dk = 2.0 * bm / n
    k = -bm + dk * torch.arange(n, dtype=torch.float64, device=DEV)
    kx, ky = torch.meshgrid(k, k, indexing="ij")
    br = torch.hypot(kx, ky)
    inside = br < bp
    slope = torch.where(inside, 4.0 * height * (bp - 2.0 * br) / bp ** 2, 0.0)
    gamma = torch.where(inside, 4.0 * height * (bp - br) / bp ** 2, 0.0)
    one = torch.complex(torch.ones_like(gamma), gamma)
    kcx, kcy = (kx * one).reshape(-1), (ky * one).reshape(-1)
    p, r = _green(kcx * kcx + kcy * kcy, eps_r, h, K0)
    (tx, ty), (bx, by) = _spectra(el, kcx, kcy)
    hk = p * (tx[:, None] * bx[None] + ty[:, None] * by[None]) - \
        r * (kcx * tx + kcy * ty)[:, None] * (kcx * bx + kcy * by)[None]
    jac = (torch.complex(torch.ones_like(slope), slope) * one).reshape(-1)
    hk = torch.where((br <= bm).reshape(-1), hk * jac, 0.0).reshape(m * m, n, n)
    # the rectangle rule with the exact contour factor, separable per column of ky: a plain
    # Fourier sum of every Taylor monomial to far beyond double precision
    size = 2 * n
    x = -n * math.pi / (2.0 * bm) + math.pi / (2.0 * bm) * torch.arange(size, dtype=torch.float64, device=DEV)
    e = torch.exp(-1j * torch.outer(x, k))
    out = torch.zeros((m * m, size, size), dtype=torch.complex128, device=DEV)
    order = 0
    reach = height * case["rho_max"]
    while reach ** (order + 1) / math.factorial(order + 1) > 1e-17:
        order += 1
    for a in range(order + 1):
        for b in range(order + 1 - a):
            f = e @ (hk * (gamma * kx) ** a * (gamma * ky) ** b) @ e.T
            out += f * (x[:, None] ** a * x[None] ** b) / (math.factorial(a) * math.factorial(b))
    out *= dk * dk / (4.0 * math.pi ** 2)
    # the table itself reaches beyond rho_max, where its own series is cut: no value for it
    pos = torch.tensor(_cartesian_positions(case, seed), device=DEV)
    d = (pos[:, None] - pos[None]).reshape(-1, 2)
    u = (d - x[0]) / (x[1] - x[0])
    i0 = torch.round(u).long()
    f = u - i0
    w = torch.stack([0.5 * f * (f - 1.0), 1.0 - f * f, 0.5 * f * (f + 1.0)], -1).to(torch.complex128)
    z = 0.0
    for s in range(3):
        for t in range(3):
            z = z + w[:, 0, s] * w[:, 1, t] * out[:, i0[:, 0] - 1 + s, i0[:, 1] - 1 + t]
    a = pos.shape[0]
    z = z.reshape(m, m, a, a).permute(2, 0, 3, 1).reshape(a * m, a * m)
    return {"table": None, "z": z}


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        z, v = _reduced_system(case, seed)
        return torch.linalg.solve(z.to(torch.complex128), v.to(torch.complex128))
    if kind == "cartesian":
        return _exact_cartesian(case, seed)
    if kind == "table":
        y, beta_c, c = _case_harmonics(case, seed)
        rho = torch.linspace(0.0, case["rho_max"], case["n_rho"], dtype=torch.float64, device=DEV)
        return _rho_table(y[0], beta_c, c.beta_max, case["q_max"], rho)
    if kind == "sweep":
        el = _element(case, seed)
        items = _sweep_items(case, seed)
        one = min(range(len(items)), key=lambda i: items[i]["n"] * items[i]["beta_max"])
        it = items[one]
        beta_c, w = _nodes(it["n"], it["beta_max"], it["beta_p"], it["height"])
        y = _harmonics(el, beta_c, w, case["q_max"], 1, [_green(beta_c * beta_c, it["eps_r"], it["h"], it["k0"])])
        rho = torch.linspace(0.0, case["rho_max"], case["n_rho"], dtype=torch.float64, device=DEV)
        z = _rho_table(y[0, 0], beta_c, it["beta_max"], case["q_max"], rho)
        return [z if i == one else None for i in range(len(items))]
    if kind == "grad":
        return _exact_fill(case, seed, grads=tuple(_vectors(case["elements"] * case["m"], seed)))
    if case["elements"] > 2500:
        return None
    return _exact_fill(case, seed)
