"""Performance cases: the work that a user of this library has it do.

Every case goes through the public entry points (the C ABI through its ctypes
binding).  The kinds, and what each stands for:

  product   y = (I - A) x, the operator of eq. 9, as a user's own Krylov solver
            or eigenvalue search calls it on device vectors: the FP64 and the
            FP32 (mixed) product, on the square tree, and the FP64 product on
            the regular-triangle tree
  block     one fundamental block from its geometry to its Bragg coefficients
            (create, mixed solve to 1e-6, coefficients, destroy): the benchmark's
            step, and what a design loop over geometries repeats
  crystal   one frequency of a band-gap curve of Sec. 4 (create, mixed solve,
            ETC on the right edge, destroy), with host vectors, as bandgap.py
  sweep     a chunk of band-gap-sweep instances of uneven sizes solved in one
            batched call on handles already made
  field     a field map: u^s and its x1-derivative at points between the fibers
  train     one Adam step of the warm-start network on a batch
  forward   the network on a batch of blocks' features

Sizes come from workloads.py, the tests and bench.py.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_1910_10863_gb300 import pfmbem as pf
from paper_1910_10863_gb300 import workloads as W


def listed():
    return [
        # the smallest block of the tests: latency of one launch and of the call itself
        {"name": "product_small", "kind": "product", "lattice": "square", "cols": 2, "rows": 2, "n": 64, "kH": 2.0,
         "mixed": False, "tree": 0},
        # the benchmark's block, in both precisions: what a solve on it repeats
        {"name": "product_hexagon", "kind": "product", "lattice": "hexagon", "cols": 8, "rows": 8, "n": 256,
         "kH": 5.0, "mixed": False, "tree": 0},
        {"name": "product_hexagon_mixed", "kind": "product", "lattice": "hexagon", "cols": 8, "rows": 8, "n": 256,
         "kH": 5.0, "mixed": True, "tree": 0},
        # the largest block of the benchmark (131072 elements): operators larger than the L2
        {"name": "product_large", "kind": "product", "lattice": "square", "cols": 32, "rows": 32, "n": 128,
         "kH": 20.0, "mixed": False, "tree": 0},
        {"name": "product_large_mixed", "kind": "product", "lattice": "square", "cols": 32, "rows": 32, "n": 128,
         "kH": 20.0, "mixed": True, "tree": 0},
        # the paper's own tree on the benchmark's block
        {"name": "product_triangle", "kind": "product", "lattice": "hexagon", "cols": 8, "rows": 8, "n": 256,
         "kH": 5.0, "mixed": False, "tree": 1},
        # the benchmark's step: a new geometry to its Bragg coefficients
        {"name": "block_hexagon", "kind": "block", "lattice": "hexagon", "cols": 8, "rows": 8, "n": 256, "kH": 5.0},
        # a point of Table 3's curves, on the scatterers without a rotation symmetry (full same-fiber blocks)
        {"name": "crystal_round_square", "kind": "crystal", "lattice": "square", "scatterer": "roundsquare",
         "f": 0.35, "n": 256, "ka": 0.62},
        # a chunk of the band-gap sweep: 64..256 elements per fiber, odd counts, both lattices
        {"name": "sweep_32", "kind": "sweep", "count": 32, "layout": 1912},
        # a field map on the benchmark's block
        {"name": "field_map", "kind": "field", "cols": 8, "rows": 8, "n": 256, "kH": 5.0, "points": 1024},
        # the warm start's training step and its inference over a test set, at the defaults of warmstart.py
        {"name": "mlp_train", "kind": "train", "inputs": 50, "outputs": 1088, "batch": 256},
        {"name": "mlp_forward", "kind": "forward", "inputs": 50, "outputs": 1088, "batch": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: odd element counts, ragged blocks, blocks wider than their period."""
    kind = rng.choice(["product", "product", "product", "block", "crystal", "sweep", "field", "train", "forward"])
    if kind == "product":
        if rng.random() < 0.5:
            rows = _log_int(rng, 2, 32)
            cols = max(1, min(int(round(rows * rng.uniform(0.5, 1.6))), 1024 // rows))
            n = _log_int(rng, 17, max(18, min(256, 131072 // (rows * cols))))
            return {"kind": kind, "lattice": "square", "cols": cols, "rows": rows, "n": n,
                    "kH": round(rng.uniform(0.5, 4.0 + 0.5 * rows), 3), "mixed": rng.random() < 0.5, "tree": 0}
        rows = rng.randint(3, 9)
        tree = 1 if rng.random() < 0.3 else 0
        cols = rng.randint(2, rows)
        return {"kind": kind, "lattice": "hexagon", "cols": cols, "rows": rows, "n": _log_int(rng, 33, 256),
                "kH": round(rng.uniform(1.0, 8.0), 3), "mixed": tree == 0 and rng.random() < 0.5, "tree": tree}
    if kind == "block":
        rows = rng.randint(3, 8)
        return {"kind": kind, "lattice": rng.choice(["square", "hexagon"]), "cols": rng.randint(2, rows),
                "rows": rows, "n": _log_int(rng, 48, 256), "kH": round(rng.uniform(1.0, 6.0), 3)}
    if kind == "crystal":
        return {"kind": kind, "lattice": rng.choice(["square", "hexagon"]),
                "scatterer": rng.choice(["circular", "roundsquare"]), "f": rng.choice([0.35, 0.5]),
                "n": _log_int(rng, 96, 256), "ka": round(rng.uniform(0.1, 1.1), 3)}
    if kind == "sweep":
        return {"kind": kind, "count": _log_int(rng, 3, 32), "layout": rng.randint(1, 9999)}
    if kind == "field":
        rows = rng.randint(2, 8)
        return {"kind": kind, "cols": rng.randint(2, rows), "rows": rows, "n": _log_int(rng, 33, 256),
                "kH": round(rng.uniform(1.0, 6.0), 3), "points": _log_int(rng, 9, 1024)}
    wide = rng.random() < 0.7                        # one row per block, or one row per fiber
    return {"kind": kind, "inputs": 50, "outputs": 1088 if wide else 68,
            "batch": _log_int(rng, 17, 1024 if wide else 4096)}


# ---------------------------------------------------------------- inputs
def _angle(rng, kH):
    while True:
        theta = float(rng.uniform(0.0, 0.45 * math.pi))
        if W.wood_distance(kH, theta) > 0.02:
            return theta


def _geometry(case, seed):
    """The block (workloads.Workload) of a case: its nodes, wavenumbers and incidence, from the seed alone."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "crystal":
        ka = case["ka"] + float(rng.uniform(-0.02, 0.02))
        while W.wood_distance(6 * 2 * math.pi * ka, 0.0) < 0.02:
            ka += 0.004
        return W.table3_block(ka, f=case["f"], lattice=case["lattice"], scatterer=case["scatterer"], n=case["n"])
    theta = _angle(rng, case["kH"])
    if case.get("lattice", "hexagon") == "hexagon":
        return W.hexagon_block(case["cols"], case["rows"], 1.0, case["n"], case["kH"], theta, int(seed) % (1 << 31))
    return W.square_block(case["cols"], case["rows"], 1.0, float(rng.uniform(0.15, 0.3)), case["n"], case["kH"],
                          theta)


def _instances(case, seed):
    """The sweep's blocks (sizes from the case's layout) at frequencies and angles from the seed."""
    rng = np.random.default_rng(seed)
    out = []
    for w in W.batch_instances(case["count"], seed=case["layout"]):
        kH = float(rng.uniform(0.5, 8.0))
        theta = _angle(rng, kH)
        f = kH / w.H / w.k
        out.append(dataclasses.replace(w, k=w.k * f, k1=w.k1 * f, theta=theta))
    return out


def _options(case):
    if case.get("tree"):
        return dict(tree=1, leaf_max=16, **W.hexagon_block_lattice(1.0, case["rows"]))
    return {}


def _vector(E, seed):
    """Half a smooth density, half noise: what the products of a Krylov solver meet."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    z = torch.randn(2 * E, dtype=torch.complex128, device="cuda", generator=g)
    e = torch.arange(2 * E, dtype=torch.float64, device="cuda")
    ph = torch.rand(2, dtype=torch.float64, device="cuda", generator=g)
    return 0.5 * z + torch.polar(torch.ones_like(e), 0.003 * e + 6.28 * ph[0]) * (1.0 + ph[1])


def _smooth(w):
    """The incident field and its normal derivative at the elements: a density of the size of a solution."""
    a, b = _ends(w)
    c, d = 0.5 * (a + b), b - a
    h = np.hypot(d[:, 0], d[:, 1])
    dr = np.array([math.cos(w.theta), math.sin(w.theta)])
    u = np.exp(1j * w.k * (c @ dr))
    nu = np.stack([d[:, 1], -d[:, 0]], axis=1) / h[:, None]
    psi = np.empty(2 * len(h), dtype=np.complex128)
    psi[0::2] = u
    psi[1::2] = u * (nu @ dr)
    return psi


def _ends(w):
    a = w.nodes
    off = np.concatenate([[0], np.cumsum(w.nodes_per_fiber)])
    nxt = np.arange(len(a)) + 1
    nxt[off[1:] - 1] = off[:-1]
    return a, a[nxt]


def _points(w, count, seed):
    """Points of the block outside the fibers."""
    rng = np.random.default_rng(seed)
    x1 = float(np.max(w.centres[:, 0] + w.radii))
    got = np.empty((0, 2))
    while len(got) < count:
        p = rng.uniform([0.0, 0.0], [x1, w.H], size=(2 * count, 2))
        keep = np.ones(len(p), dtype=bool)
        for (cx, cy), r in zip(w.centres, w.radii):
            for m in (-1, 0, 1):
                keep &= np.hypot(p[:, 0] - cx, p[:, 1] - cy - m * w.H) > 1.02 * r
        got = np.concatenate([got, p[keep]])
    return np.ascontiguousarray(got[:count])


def _network(case, seed):
    """Layer widths and seeded weights (flat: per layer W [out][in], b [out])."""
    dims = [case["inputs"], 256, 256, 256, case["outputs"]]
    rng = np.random.default_rng(seed)
    flat = []
    for i, o in zip(dims[:-1], dims[1:]):
        flat += [rng.uniform(-1, 1, size=i * o) * math.sqrt(3.0 / i), 0.1 * rng.standard_normal(o)]
    return dims, np.concatenate(flat).astype(np.float32)


def _rows(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    X = torch.rand(case["batch"], case["inputs"], device="cuda", generator=g)
    T = 0.5 * torch.randn(case["batch"], case["outputs"], device="cuda", generator=g)
    return X, T


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "product":
        w = _geometry(case, seed)
        s = pf.Solver(w, precision=pf.MIXED if case["mixed"] else pf.FP64, **_options(case))
        x = _vector(s.E, seed)
        return {"kind": kind, "solver": s, "x": x, "y": torch.zeros_like(x),
                "precision": pf.MIXED if case["mixed"] else pf.FP64}
    if kind == "block":
        w = _geometry(case, seed)
        return {"kind": kind, "w": w, "psi": torch.zeros(2 * w.E, dtype=torch.complex128, device="cuda")}
    if kind == "crystal":
        w = _geometry(case, seed)
        return {"kind": kind, "w": w, "x1": _right_edge(case)}
    if kind == "sweep":
        ws = _instances(case, seed)
        ss = [pf.Solver(w, precision=pf.MIXED) for w in ws]
        return {"kind": kind, "solvers": ss, "handles": [s.h for s in ss],
                "psis": [torch.zeros(2 * s.E, dtype=torch.complex128, device="cuda") for s in ss]}
    if kind == "field":
        w = _geometry(case, seed)
        n = case["points"]
        return {"kind": kind, "solver": pf.Solver(w), "psi": torch.from_numpy(_smooth(w)).cuda(),
                "points": _points(w, n, seed), "u": np.zeros(n, np.complex128), "du": np.zeros(n, np.complex128)}
    dims, flat = _network(case, seed)
    net = pf.MLP(dims[0], 256, 3, dims[-1])
    net.set_params(flat)
    X, T = _rows(case, seed)
    if kind == "train":
        return {"kind": kind, "net": net, "X": X, "T": T, "grad": torch.zeros(len(flat), device="cuda")}
    return {"kind": kind, "net": net, "X": X, "Y": torch.zeros_like(T)}


def _right_edge(case):
    return 4 * 0.5 * (1.0 if case["lattice"] == "square" else math.sqrt(3.0) / 2.0)


def run(state):
    kind = state["kind"]
    if kind == "product":
        state["solver"].matvec(state["x"], state["y"], state["precision"])
        return state["y"]
    if kind == "block":
        s = pf.Solver(state["w"], precision=pf.MIXED)
        s.solve(state["psi"], tol=1e-6, check=False)
        orders, R, T, energy = pf.pfmbem_coefficients(s.h, state["psi"])
        s.close()
        return {"psi": state["psi"], "orders": orders, "R": R, "T": T, "energy": energy}
    if kind == "crystal":
        s = pf.Solver(state["w"], precision=pf.MIXED)
        psi = np.zeros(2 * s.E, dtype=np.complex128)
        s.solve(psi, tol=1e-6, check=False)
        etc = pf.pfmbem_etc(s.h, psi, state["x1"], 256)
        s.close()
        return {"psi": psi, "etc": etc}
    if kind == "sweep":
        pf.pfmbem_solve_batch(state["handles"], state["psis"], tol=1e-6)
        return state["psis"]
    if kind == "field":
        u, du = pf.pfmbem_field_dx1(state["solver"].h, state["psi"], state["points"], state["u"], state["du"])
        return {"u": u, "du": du}
    net, X = state["net"], state["X"]
    if kind == "forward":
        return net.forward(X, state["Y"])
    # the C call itself: the binding's own train() brings the gradient to the host
    loss = pf.ctypes.c_float(0)
    st = pf.lib().pfmbem_mlp_train(net.h, X.shape[0], pf.addr(X), pf.addr(state["T"]), 1e-3, pf.ctypes.byref(loss),
                                   pf.addr(state["grad"]))
    if st != 0:
        raise pf.PfmbemError(st, "pfmbem_mlp_train")
    return {"loss": loss.value, "grad": state["grad"]}


# ---------------------------------------------------------------- work
def work(case):
    """Bytes and flops of one pass that no form of the method does without.

    A product reads x, the geometry (node, midpoint, normal: 48 bytes an element) and
    writes y; its arithmetic is the near field (about 100 sources an element, four
    complex multiply-adds each), P2M and L2P (2 x 49 each way) and the same-fiber
    blocks (FFT).  A solve is 10 products and reads its geometry once; a field point
    meets every element and its two nearest images (about 100 flops a pair)."""
    kind = case["kind"]

    def product(E):
        return {"bytes": E * (64.0 + 48.0), "flops": E * (100 * 4 * 8 + 4 * 49 * 8 + 600.0)}

    if kind == "product":
        return product(case["cols"] * case["rows"] * case["n"])
    if kind in ("block", "crystal", "sweep"):
        E = case["cols"] * case["rows"] * case["n"] if kind == "block" else \
            24 * case["n"] if kind == "crystal" else case["count"] * 16 * 155
        p = product(E)
        return {"bytes": 48.0 * E + 32.0 * E, "flops": 10 * p["flops"]}
    if kind == "field":
        E = case["cols"] * case["rows"] * case["n"]
        return {"bytes": E * 80.0 + case["points"] * 48.0, "flops": case["points"] * 3.0 * E * 100}
    dims = [case["inputs"], 256, 256, 256, case["outputs"]]
    params = sum(i * o + o for i, o in zip(dims[:-1], dims[1:]))
    mac = case["batch"] * sum(i * o for i, o in zip(dims[:-1], dims[1:]))
    io = 4.0 * case["batch"] * (case["inputs"] + case["outputs"])
    if kind == "forward":
        return {"bytes": 4.0 * params + io, "flops": 2.0 * mac}
    return {"bytes": 4.0 * params * 8 + io, "flops": 6.0 * mac - 2.0 * case["batch"] * case["inputs"] * 256}


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """The outputs in FP64 by dense collocation with torch (no tree, no expansions): every
    element integral by Gauss quadrature of the kernel (16 nodes within 12 element
    lengths, 4 beyond), self integrals by their series, the images |m| <= q summed
    directly and the rest through their plane-wave integrals; solves by GMRES on the
    dense matrix.  None for the largest blocks (a matrix of 131072 elements)."""
    kind = case["kind"]
    if kind in ("train", "forward"):
        return _exact_network(case, seed)
    if kind == "sweep":
        return [_solve_dense(_Dense(w)) for w in _instances(case, seed)]
    w = _geometry(case, seed)
    if w.E > 17000:
        return None
    d = _Dense(w)
    if kind == "product":
        return d.operator()[1](_vector(w.E, seed))
    if kind == "block":
        psi = _solve_dense(d)
        orders, R, T, energy = d.bragg(psi)
        return {"psi": psi, "orders": orders, "R": R, "T": T, "energy": energy}
    if kind == "crystal":
        psi = _solve_dense(d)
        y0, x1 = 0.0, _right_edge(case)
        p = torch.tensor([[x1, y0 + w.H * (i + 0.5) / 256] for i in range(256)], dtype=torch.float64, device="cuda")
        u, du = d.field(psi, p)
        c, s = math.cos(w.theta), math.sin(w.theta)
        inc = 1j * w.k * c * torch.exp(1j * w.k * (c * p[:, 0] + s * p[:, 1]))
        return {"psi": psi.cpu().numpy(), "etc": float((du + inc).abs().mean() / w.k)}
    psi = torch.from_numpy(_smooth(w)).cuda()
    u, du = d.field(psi, torch.from_numpy(_points(w, case["points"], seed)).cuda())
    return {"u": u.cpu().numpy(), "du": du.cpu().numpy()}


def _exact_network(case, seed):
    dims, flat = _network(case, seed)
    X, T = (v.double() for v in _rows(case, seed))
    p = torch.from_numpy(flat).cuda().double().requires_grad_(True)
    a, o = X, 0
    for l, (i, n) in enumerate(zip(dims[:-1], dims[1:])):
        a = a @ p[o:o + i * n].view(n, i).T + p[o + i * n:o + i * n + n]
        o += i * n + n
        if l < len(dims) - 2:
            a = torch.nn.functional.gelu(a)
    if case["kind"] == "forward":
        return a.detach()
    loss = ((a - T) ** 2).mean()
    loss.backward()
    return {"loss": float(loss), "grad": p.grad}


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()


def _hankel_fits():
    """Chebyshev coefficients in y = 10/x - 1 (x >= 5) of H_n(x) sqrt(pi x/2) e^{-i(x - n pi/2 - pi/4)}, n = 0, 1,
    sampled through its Laplace integral by Gauss-Hermite quadrature (torch's own Bessel functions carry 1e-6)."""
    s, g = np.polynomial.hermite.hermgauss(160)
    y = np.cos((np.arange(18) + 0.5) * np.pi / 18)
    f = 1 + 1j * s[None, :] ** 2 * (y[:, None] + 1) / 20.0
    v = (g * f ** -0.5).sum(1) / np.sqrt(np.pi), (g * s ** 2 * f ** 0.5).sum(1) * 2 / np.sqrt(np.pi)
    return [np.polynomial.chebyshev.cheb2poly(np.polynomial.chebyshev.chebfit(y, p, 17))
            for h in v for p in (h.real, h.imag)]


_FITS = _hankel_fits()


def _hankel(x):
    """H_0 and H_1 (first kind) of x > 0: ascending series below 5, the fits above."""
    lo = torch.clamp(x, max=5.0)
    q, t = -0.25 * lo * lo, torch.ones_like(lo)
    lg = (2 / math.pi) * (torch.log(0.5 * lo) + 0.57721566490153286)
    j0, j1, y0, y1, har = t.clone(), t.clone(), 0 * t, t.clone(), 0.0
    for k in range(1, 24):
        t = t * q / (k * k)
        har += 1.0 / k
        j0 = j0 + t
        y0 = y0 - har * t
        j1 = j1 + t / (k + 1)
        y1 = y1 + (2 * har + 1.0 / (k + 1)) * t / (k + 1)
    y0 = lg * j0 + (2 / math.pi) * y0
    j1 = 0.5 * lo * j1
    y1 = lg * j1 - (2 / math.pi) / lo - (0.5 / math.pi) * lo * y1
    hi = torch.clamp(x, min=5.0)
    y = 10.0 / hi - 1.0
    v = []
    for c in _FITS:
        a = torch.full_like(y, float(c[-1]))
        for b in c[-2::-1].tolist():
            a = a * y + b
        v.append(a)
    e = torch.polar(torch.sqrt(2 / (math.pi * hi)), hi - 0.25 * math.pi)
    big = x >= 5.0
    return (torch.where(big, e * torch.complex(v[0], v[1]), torch.complex(j0, y0)),
            torch.where(big, -1j * e * torch.complex(v[2], v[3]), torch.complex(j1, y1)))


def _integrals(kap, x, nx, c, t, nu, h, nodes):
    """Element integrals of S, D, K, T of (i/4) H0(kap r); all arguments broadcast, vectors as pairs."""
    S = D = K = T = 0
    xs, ws = _gauss(nodes)
    for a, b in zip(xs.tolist(), ws.tolist()):
        z1 = x[0] - c[0] - 0.5 * a * h * t[0]
        z2 = x[1] - c[1] - 0.5 * a * h * t[1]
        r = torch.sqrt(z1 * z1 + z2 * z2)
        H0, H1 = _hankel(kap * r)
        zx, zy = (z1 * nx[0] + z2 * nx[1]) / r, (z1 * nu[0] + z2 * nu[1]) / r
        f = 0.125j * b * h
        kH1 = kap * H1
        S = S + f * H0
        D = D + f * kH1 * zy
        K = K - f * kH1 * zx
        T = T + f * (kH1 / r * (nx[0] * nu[0] + nx[1] * nu[1]) + zx * zy * (kap * kap * H0 - 2 * kH1 / r))
    return S, D, K, T


def _self(kap, h):
    """S and the finite-part T of a flat element at its midpoint, from int_0^{kap h/2} H0 by series."""
    x = 0.5 * kap * h
    q = -0.25 * x * x
    term, har, ij, iy = x.clone(), 0.0, x.clone(), torch.zeros_like(x)
    lg = torch.log(0.5 * x) + 0.57721566490153286
    iy = (2 / math.pi) * (lg - 1.0) * x
    for k in range(1, 25):
        term = term * q / (k * k)
        har += 1.0 / k
        ij = ij + term / (2 * k + 1)
        iy = iy + (2 / math.pi) * term / (2 * k + 1) * (lg - har - 1.0 / (2 * k + 1))
    ih = torch.complex(ij, iy)
    return 0.5j / kap * ih, 0.5j * kap * (ih - _hankel(x)[1])


class _Dense:
    """The dense operator of eq. 9 of one block and its outputs, FP64."""

    def __init__(self, w):
        self.w = w
        a, b = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in _ends(w))
        d = b - a
        self.h = torch.hypot(d[:, 0], d[:, 1])
        t = d / self.h[:, None]
        m = 0.5 * (a + b)
        self.c, self.t, self.nu = m.T.contiguous(), t.T.contiguous(), torch.stack([t[:, 1], -t[:, 0]])
        self.E = len(self.h)
        self.eta = w.k
        self.c2 = 2.0 / (1j * self.eta * (1.0 + w.rho_ratio))
        self.alpha = complex(math.cos(w.k * w.H * math.sin(w.theta)), math.sin(w.k * w.H * math.sin(w.theta)))
        width = float(self.c[0].max() - self.c[0].min()) + 0.5 * w.H
        self.q = max(1, math.ceil(w.k * width * width / (12.0 * w.H)))
        self.x0 = 0.5 * float(self.c[0].max() + self.c[0].min())
        self.y0 = 0.5 * float(self.c[1].max() + self.c[1].min())

    def waves(self):
        """Plane waves of the images |m| > q: exponents (a, b) of e^{a z1 + b z2} and their weights."""
        w = self.w
        V = 7.0 / math.sqrt(0.5 * self.q * w.H)
        edges = [0.0] + [V * 2.0 ** (-i) for i in range(11, 2, -1)] + [V * i / 8 for i in range(2, 9)]
        x, g = np.polynomial.legendre.leggauss(24)
        v = np.concatenate([0.5 * (r - l) * (x + 1) + l for l, r in zip(edges[:-1], edges[1:])])
        gw = np.concatenate([0.5 * (r - l) * g for l, r in zip(edges[:-1], edges[1:])])
        root = np.sqrt(v * v - 2j * w.k)
        mu, t = v * v - 1j * w.k, v * root
        A, B, C = [], [], []
        for sg, al in ((1, self.alpha), (-1, 1 / self.alpha)):       # images m > q, m < -q
            e = al * np.exp(-mu * w.H)
            f = gw / (2 * math.pi * root) * e ** (self.q + 1) / (1 - e)
            for st in (1, -1):
                A.append(1j * st * t)
                B.append(sg * mu)
                C.append(f)
        return (torch.from_numpy(np.concatenate(z)).cuda() for z in (A, B, C))

    def sources(self, A, B):
        """[waves][2E]: element integrals of e^{-(a y1 + b y2)} for phi (d/dnu_y) and varphi (-i eta)."""
        e = torch.exp(-(A[:, None] * (self.c[0] - self.x0) + B[:, None] * (self.c[1] - self.y0)))
        s = 0
        for a, b in zip(*(z.tolist() for z in _gauss(6))):
            u = 0.5 * a * self.h
            s = s + 0.5 * b * self.h * torch.exp(-(A[:, None] * (u * self.t[0]) + B[:, None] * (u * self.t[1])))
        e = e * s
        return torch.stack([-e * (A[:, None] * self.nu[0] + B[:, None] * self.nu[1]), -1j * self.eta * e],
                           dim=2).reshape(len(A), 2 * self.E)

    def operator(self):
        """The dense matrix without the far images, and the whole operator as a function of a vector."""
        w, E, eta = self.w, self.E, self.eta
        M = torch.empty(E, 2, E, 2, dtype=torch.complex128, device="cuda")
        fib = torch.repeat_interleave(torch.arange(w.M, device="cuda"),
                                      torch.from_numpy(w.nodes_per_fiber.astype(np.int64)).cuda())
        st = max(1, 4_000_000 // E)
        for r0 in range(0, E, st):
            r1 = min(E, r0 + st)
            x, nx = self.c[:, r0:r1, None], self.nu[:, r0:r1, None]
            blk = [0, 0, 0, 0]
            for m in range(-self.q, self.q + 1):
                c = torch.stack([self.c[0], self.c[1] + m * w.H])[:, None, :]
                got = self.pairs(w.k, x, nx, c, r0, r1, m == 0)
                blk = [p + self.alpha ** m * g for p, g in zip(blk, got)]
            S, D, K, T = blk
            M[r0:r1, 0, :, 0], M[r0:r1, 0, :, 1] = D, -1j * eta * S
            M[r0:r1, 1, :, 0], M[r0:r1, 1, :, 1] = self.c2 * T, -1j * eta * self.c2 * K
        # the fiber operators (k1), within each fiber
        off = 0
        for n in w.nodes_per_fiber.tolist():
            sl = slice(off, off + n)
            sub = _Sub(self, sl)
            S, D, K, T = sub.pairs(w.k1, sub.c[:, :, None], sub.nu[:, :, None], sub.c[:, None, :], 0, n, True)
            M[sl, 0, sl, 0] -= D
            M[sl, 0, sl, 1] += 1j * eta * S
            M[sl, 1, sl, 0] -= self.c2 * w.rho_ratio * T
            M[sl, 1, sl, 1] += 1j * eta * self.c2 * w.rho_ratio * K
            off += n
        M = M.reshape(2 * E, 2 * E)
        A, B, C = self.waves()
        V = self.sources(A, B)
        U = C * torch.exp(A * (self.c[0] - self.x0)[:, None] + B * (self.c[1] - self.y0)[:, None])
        Un = self.c2 * U * (A * self.nu[0][:, None] + B * self.nu[1][:, None])
        M.diagonal().add_(1.0)
        far = torch.stack([U, Un], dim=1).reshape(2 * E, len(A))
        return M, lambda v: M @ v + far @ (V @ v)

    def pairs(self, kap, x, nx, c, r0, r1, own):
        """Integrals of targets r0..r1 against all elements at c: 4 nodes, 16 for the near pairs, closed forms for own."""
        t, nu, h = self.t[:, None, :], self.nu[:, None, :], self.h[None, :]
        if own:          # the self pair's kernel is singular: moved away here, replaced below
            eye = torch.zeros(r1 - r0, self.E, dtype=torch.float64, device="cuda")
            i = torch.arange(r0, r1, device="cuda")
            eye[i - r0, i] = 1.0
            x = torch.stack([x[0] + eye, x[1] + 0 * eye])
        S, D, K, T = _integrals(kap, x, nx, c, t, nu, h, 4)
        near = torch.hypot(x[0] - c[0], x[1] - c[1]) < 12 * h
        i, j = near.nonzero(as_tuple=True)
        if len(i):
            xi = [torch.broadcast_to(v, near.shape)[i, j] for v in x]
            ni = [torch.broadcast_to(v, near.shape)[i, j] for v in nx]
            cj = [torch.broadcast_to(v, near.shape)[i, j] for v in c]
            got = _integrals(kap, xi, ni, cj, self.t[:, j], self.nu[:, j], self.h[j], 16)
            for dst, g in zip((S, D, K, T), got):
                dst[i, j] = g
        if own:
            i = torch.arange(r0, r1, device="cuda")
            s, tt = _self(kap, self.h[r0:r1])
            S[i - r0, i], T[i - r0, i] = s, tt
            D[i - r0, i] = K[i - r0, i] = 0
        return S, D, K, T

    def rhs(self):
        w = self.w
        d1, d2 = math.cos(w.theta), math.sin(w.theta)
        u = torch.exp(1j * w.k * (d1 * self.c[0] + d2 * self.c[1]))
        return torch.stack([-u, -self.c2 * 1j * w.k * (d1 * self.nu[0] + d2 * self.nu[1]) * u], dim=1).reshape(-1)

    def field(self, psi, p):
        """u^s and du^s/dx1 at the points p."""
        w = self.w
        u, du = [], []
        A, B, C = self.waves()
        vec = self.sources(A, B) @ psi
        st = max(1, 4_000_000 // self.E)
        phi, var = psi[0::2], -1j * self.eta * psi[1::2]
        nx = (torch.ones((), dtype=torch.float64, device="cuda"), torch.zeros((), dtype=torch.float64, device="cuda"))
        for r0 in range(0, len(p), st):
            q = p[r0:r0 + st]
            x = q.T.contiguous()[:, :, None]
            n0 = torch.stack([torch.broadcast_to(v, (len(q), 1)) for v in nx])
            # the copy of the point in the period that the elements fill
            mp = torch.floor((x[1] - (self.y0 - 0.5 * w.H)) / w.H)
            x = torch.stack([x[0], x[1] - mp * w.H])
            a = b = 0
            for m in range(-self.q, self.q + 1):
                c = torch.stack([self.c[0], self.c[1] + m * w.H])[:, None, :]
                S, D, K, T = self.pairs(w.k, x, n0, c, 0, 0, False)
                a = a + self.alpha ** m * (D @ phi + S @ var)
                b = b + self.alpha ** m * (T @ phi + K @ var)
            e = C * torch.exp(A * (x[0] - self.x0) + B * (x[1] - self.y0))
            ph = self.alpha ** mp[:, 0]
            u.append(ph * (a + e @ vec))
            du.append(ph * (b + (e * A) @ vec))
        return torch.cat(u), torch.cat(du)

    def bragg(self, psi):
        w = self.w
        ks = w.k * math.sin(w.theta)
        lim = int(w.k * w.H / math.pi) + 2
        orders = [n for n in range(-lim, lim + 1) if abs(ks + 2 * math.pi * n / w.H) < w.k]
        R, T, en = [], [], 0.0
        for n in orders:
            kap = ks + 2 * math.pi * n / w.H
            kn = math.sqrt(w.k ** 2 - kap ** 2)
            v = []
            for w1 in (kn, -kn):
                ph = torch.exp(-1j * (w1 * self.c[0] + kap * self.c[1]))
                a = 0.5 * self.h * (w1 * self.t[0] + kap * self.t[1])
                bra = -1j * (w1 * self.nu[0] + kap * self.nu[1]) * psi[0::2] - 1j * self.eta * psi[1::2]
                v.append(complex((1j / (2 * w.H * kn)) * (self.h * torch.sinc(a / math.pi) * ph * bra).sum()))
            T.append(v[0] + (1.0 if n == 0 else 0.0))
            R.append(v[1])
            en += kn / (w.k * math.cos(w.theta)) * (abs(R[-1]) ** 2 + abs(T[-1]) ** 2)
        return np.array(orders, dtype=np.int32), np.array(R), np.array(T), en


class _Sub(_Dense):
    """One fiber of a block (for its k1 operators)."""

    def __init__(self, d, sl):
        self.c, self.t, self.nu, self.h = d.c[:, sl], d.t[:, sl], d.nu[:, sl], d.h[sl]
        self.E = len(self.h)


def _solve_dense(d):
    """GMRES on the dense matrix, preconditioned by the fibers' diagonal blocks, to FP64 rounding."""
    (M, apply), b = d.operator(), d.rhs()
    lu, off = [], 0
    for n in d.w.nodes_per_fiber.tolist():
        sl = slice(2 * off, 2 * (off + n))
        lu.append((sl, torch.linalg.inv(M[sl, sl])))
        off += n

    def solve(v):
        z = torch.empty_like(v)
        for sl, f in lu:
            z[sl] = f @ v[sl]
        return z

    x = torch.zeros_like(b)
    for _ in range(4):
        r = b - apply(x)
        beta = torch.linalg.vector_norm(r)
        if float(beta / torch.linalg.vector_norm(b)) < 1e-14:
            break
        Q, Z, H = [r / beta], [], np.zeros((61, 60), dtype=np.complex128)
        for j in range(60):
            Z.append(solve(Q[j]))
            v = apply(Z[j])
            B = torch.stack(Q)
            for _ in range(2):
                g = B.conj() @ v
                v = v - g @ B
                H[:j + 1, j] += g.cpu().numpy()
            H[j + 1, j] = float(torch.linalg.vector_norm(v))
            Q.append(v / float(H[j + 1, j].real))
            e = np.zeros(j + 2, dtype=np.complex128)
            e[0] = float(beta)
            y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
            if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) < 1e-12 * float(beta):
                break
        x = x + torch.from_numpy(y).cuda() @ torch.stack(Z)
    return x
