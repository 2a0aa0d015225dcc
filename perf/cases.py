"""The work that is timed: the calls that linear-stability runs of the lid-driven cube are made of.

A case is a dict of plain values.  `kind` names the call; sizes are cells per
axis; `prec` is the arithmetic form a run chooses (fp64, mixed, ff).  The base
flow is the smooth vortex sample field that throughput runs use, scaled a
little by the seed; right-hand sides are Gaussian velocity fields (walls zero),
as Krylov start vectors are.  `exact` restates every call that has a closed
answer in float64 torch, from the definitions of the method: the staggered
finite-volume operators, and pressure solves by the eigenbases of the 1-D
Neumann operators.
"""
import math

import numpy as np
import torch

import paper_1704_08521_gb300 as fv

PI4 = math.pi / 4
MAPS = ("cosine", "sine0975", "uniform")


# ------------------------------------------------------------------ cases --

def _krylov(name, n, prec, map="cosine", alpha=0.0, re=1000.0, sigma=0.0, eps=1e-8, wait=True, p=True):
    nx, ny, nz = (n, n, n) if isinstance(n, int) else n
    return {"name": name, "kind": "krylov", "nx": nx, "ny": ny, "nz": nz, "prec": prec, "map": map,
            "alpha": alpha, "re": re, "sigma": sigma, "eps": eps, "wait": wait, "p": p}


def listed():
    return [
        # one Krylov vector on the 16^3 cosine grid (the plain-method configuration): all latency
        _krylov("krylov_mixed_16", 16, "mixed"),
        # the headline workload: 100^3 cosine grid, Re 1900, queued without waiting as a Krylov method does
        _krylov("krylov_mixed_100", 100, "mixed", re=1900.0, wait=False),
        # a vector of the shifted operator as GMRES and Arnoldi ask for it, on uneven odd sizes
        _krylov("krylov_ff_83x61x47", (83, 61, 47), "ff", "sine0975", 0.3, 1500.0, 10.0, 1e-10, False, False),
        # the diagonal-lid configuration, 150^3 cosine, in the form its eigenvalues are computed in
        _krylov("krylov_ff_150", 150, "ff", "cosine", PI4, 2300.0, 10.0, 1e-10, False, False),
        # the paper's largest grid, 256^3 with its own stretching
        _krylov("krylov_ff_256", 256, "ff", "sine0975", 0.0, 1926.0, 0.0, 1e-8, False, False),
        # the plain float64 form on the 100^3 configuration
        _krylov("krylov_fp64_100", 100, "fp64", re=1900.0),
        # twelve instances per launch, {48, 64, 80, 96}^3 x Re {1700, 1900, 2100}, both lid directions
        {"name": "batch_12", "kind": "batch", "sizes": "48,64,80,96", "res": "1700,1900,2100", "map": "cosine",
         "eps": 1e-8, "sigma": 0.0},
        # leading eigenvalues by restarted Arnoldi from a Gaussian start vector
        {"name": "arnoldi_48", "kind": "arnoldi", "nx": 48, "ny": 48, "nz": 48, "prec": "ff", "map": "sine0975",
         "alpha": 0.0, "re": 1000.0, "m": 40, "nev": 2, "tol": 1e-8},
        # a steady state by Newton from rest: the first stage of a continuation in Re
        {"name": "newton_16", "kind": "newton", "nx": 16, "ny": 16, "nz": 16, "prec": "ff", "map": "cosine",
         "alpha": 0.0, "re": 200.0},
        # the iterative pressure solve, as far as float64 conjugate gradients take it
        {"name": "multigrid_100", "kind": "mg", "nx": 100, "ny": 100, "nz": 100, "map": "cosine", "rtol": 1e-12},
        # forward and backward pass of the learned guess on its smallest training grid
        {"name": "unet_64", "kind": "unet", "nx": 64, "ny": 64, "nz": 64},
        # a flow projected onto the (x, z) planes with its vector potential, for pictures
        {"name": "planes_100", "kind": "planes", "nx": 100, "ny": 100, "nz": 100, "map": "cosine", "plane": "xz"},
    ]


def _size(rng, lo, hi):
    """Cells of one axis, even over the logarithm, odd ones among them."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """Three axes: a cube half of the time, else uneven."""
    n = _size(rng, lo, hi)
    if rng.random() < 0.5:
        return n, n, n
    return tuple(max(lo, min(hi, int(round(n * rng.uniform(0.6, 1.4))))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["mixed", "ff", "ff", "fp64", "batch", "mg", "planes", "unet", "newton"])
    flow = {"map": rng.choice(MAPS), "alpha": rng.choice([0.0, 0.3, PI4]), "re": round(rng.uniform(200.0, 2500.0), 1)}
    if kind in ("mixed", "ff", "fp64"):
        nx, ny, nz = _box(rng, 8, {"mixed": 112, "ff": 256, "fp64": 128}[kind])
        return {"kind": "krylov", "nx": nx, "ny": ny, "nz": nz, "prec": kind, **flow,
                "sigma": rng.choice([0.0, 10.0]), "eps": 1e-8, "wait": rng.random() < 0.5,
                "p": kind != "ff" and rng.random() < 0.5}   # the pressure of a Krylov vector is context, seldom asked for
    if kind == "batch":
        n = sorted({_size(rng, 12, 100) for _ in range(rng.randint(2, 4))})
        return {"kind": "batch", "sizes": ",".join(map(str, n)), "res": "1700,%d" % rng.randint(1800, 2100),
                "map": flow["map"], "eps": 1e-8, "sigma": rng.choice([0.0, 10.0])}
    if kind == "mg":
        nx, ny, nz = _box(rng, 24, 128)
        return {"kind": "mg", "nx": nx, "ny": ny, "nz": nz, "map": rng.choice(["cosine", "sine0975"]), "rtol": 1e-12}
    if kind == "planes":
        nx, ny, nz = _box(rng, 12, 128)
        return {"kind": "planes", "nx": nx, "ny": ny, "nz": nz, "map": flow["map"],
                "plane": rng.choice(["xz", "yz", "xy"])}
    if kind == "unet":
        nx, ny, nz = (8 * rng.randint(2, 12) for _ in range(3))
        return {"kind": "unet", "nx": nx, "ny": ny, "nz": nz}
    n = rng.randint(9, 16)
    return {"kind": "newton", "nx": n, "ny": n + rng.randint(-2, 2), "nz": n, "prec": "ff", "map": "cosine",
            "alpha": flow["alpha"], "re": float(rng.randint(50, 200))}


# ----------------------------------------------------------------- inputs --

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _faces(n, map):
    xi = np.arange(n + 1) / n
    if map == "cosine":
        x = 0.5 * (1.0 - np.cos(np.pi * xi))
    elif map == "sine0975":
        x = xi - 0.0975 * np.sin(2.0 * np.pi * xi)
    else:
        x = xi
    x[0], x[-1] = 0.0, 1.0
    return x


def _walls(q):
    q[0, :, :, 0] = 0.0
    q[1, :, 0, :] = 0.0
    q[2, 0, :, :] = 0.0
    return q.reshape(-1)


def _gaussian(shape, gen):
    return _walls(torch.randn((3, *shape), dtype=torch.float64, device="cuda", generator=gen))


def _vortex(shape, map, alpha, gen):
    """One recirculating vortex turned by the lid angle plus a weak secondary flow, sampled at the faces."""
    nz, ny, nx = shape
    amp = float(1.0 + 0.05 * torch.randn((), dtype=torch.float64, device="cuda", generator=gen))
    X, Y, Z = (torch.tensor(_faces(n, map), device="cuda") for n in (nx, ny, nz))
    xc, yc, zc = ((a[1:] + a[:-1]) / 2 for a in (X, Y, Z))

    def s(t):
        return torch.sin(np.pi * t)

    def ds(t):
        return np.pi * torch.sin(2 * np.pi * t)

    ca, sa = math.cos(alpha), math.sin(alpha)
    at = lambda x, y, z: (x[None, None, :], y[None, :, None], z[:, None, None])  # noqa: E731
    x, y, z = at(X[:-1], yc, zc)
    u = 4 * ca * ds(z) * s(x) ** 2 * s(y) ** 2 + 0.3 * s(x) ** 2 * ds(y) * s(z) ** 2
    x, y, z = at(xc, Y[:-1], zc)
    v = 4 * sa * ds(z) * s(x) ** 2 * s(y) ** 2 - 0.3 * ds(x) * s(y) ** 2 * s(z) ** 2
    x, y, z = at(xc, yc, Z[:-1])
    w = -4 * s(z) ** 2 * (ca * ds(x) * s(y) ** 2 + sa * s(x) ** 2 * ds(y))
    return _walls(amp * torch.stack([u, v, w]))


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _empty(n):
    return torch.empty(n, dtype=torch.float64, device="cuda")


def _instances(case):
    out = []
    for n in case["sizes"].split(","):
        for re in case["res"].split(","):
            out.append((int(n), float(re), 0.0 if len(out) % 2 == 0 else PI4))
    return out


def _inputs(case, seed):
    """The arrays of a case, made from the seed alone."""
    gen = _gen(seed)
    kind = case["kind"]
    if kind in ("krylov", "arnoldi"):
        return {"U": _vortex(_shape(case), case["map"], case["alpha"], gen), "v": _gaussian(_shape(case), gen)}
    if kind == "batch":
        return {"U": [_vortex((n, n, n), case["map"], a, gen) for n, _, a in _instances(case)],
                "v": [_gaussian((n, n, n), gen) for n, _, _ in _instances(case)]}
    if kind == "newton":   # from rest, or nearly: a continuation never starts twice from the same field
        return {"U": 1e-3 * _vortex(_shape(case), case["map"], case["alpha"], gen)}
    if kind == "mg":
        ops = _Ops(_shape(case), case["map"])
        return {"r": ops.div(ops.full(_gaussian(_shape(case), gen))).reshape(-1).contiguous()}
    if kind == "planes":   # a flow with a component the projection removes
        s = _shape(case)
        return {"v": _vortex(s, case["map"], 0.0, gen) + 0.1 * _gaussian(s, gen)}
    n = case["nx"] * case["ny"] * case["nz"]
    planes = torch.randn(4, n, device="cuda", generator=gen)
    return {"planes": planes, "target": torch.randn(n, device="cuda", generator=gen), "params": _unet_params(gen)}


def prepare(case, seed):
    st = {"case": case, **_inputs(case, seed)}
    kind = case["kind"]
    if kind == "unet":
        st["net"] = net = fv.UNet(seed=0)
        net.set_params(st["params"])
        st["out"] = torch.empty(st["target"].numel(), device="cuda")
        st["grads"] = torch.empty(net.n_param, device="cuda")
        return st
    if kind == "batch":
        inst = _instances(case)
        st["grids"] = [fv.Grid(n, n, n, case["map"], alpha=a, re=re) for n, re, a in inst]
        st["batch"] = fv.Batch(st["grids"])
        st["out"] = [torch.empty_like(x) for x in st["v"]]
        return st
    st["g"] = g = fv.Grid(case["nx"], case["ny"], case["nz"], case["map"], alpha=case.get("alpha", 0.0),
                          re=case.get("re", 1000.0))
    if kind == "krylov":
        g.set_base(st["U"])   # a Krylov method registers its base flow once
        st["out"] = _empty(g.n_vel)
        st["p"] = _empty(g.n_cell) if case["p"] else None
    elif kind == "newton":
        st["Uo"], st["P"] = _empty(g.n_vel), _empty(g.n_cell)
    elif kind == "mg":
        st["phi"] = _empty(g.n_cell)
    elif kind == "planes":
        nz, ny, nx = g.shape
        a, c = {"xz": (0, 2), "yz": (1, 2), "xy": (0, 1)}[case["plane"]]
        dims = [nx, ny, nz]
        dims[a] += 1
        dims[c] += 1
        st["vp"], st["psi"] = _empty(g.n_vel), _empty(dims[0] * dims[1] * dims[2])
    return st


# -------------------------------------------------------------------- run --

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "krylov":
        fv.simple_krylov_solve(st["g"], None, st["v"], st["out"], st["p"], eps=case["eps"], prec=case["prec"],
                               sigma=case["sigma"], async_=not case["wait"])
        return {"v": st["out"], "p": st["p"]} if case["p"] else {"v": st["out"]}
    if kind == "batch":
        st["batch"].krylov(st["U"], st["v"], st["out"], eps=case["eps"], sigma=case["sigma"], sync=False)
        return st["out"]
    if kind == "arnoldi":
        lam, _ = fv.arnoldi_leading(st["g"], st["U"], st["v"], m=case["m"], nev=case["nev"], tol=case["tol"],
                                    prec=case["prec"])
        return [x for z in lam for x in (z.real, z.imag)]
    if kind == "newton":
        st["Uo"].copy_(st["U"])
        fv.newton_steady(st["g"], st["Uo"], st["P"], prec=case["prec"])
        return {"U": st["Uo"], "P": st["P"]}
    if kind == "mg":
        fv.fv_pressure_solve_mg(st["g"], st["r"], st["phi"], rtol=case["rtol"])
        return st["phi"]
    if kind == "planes":
        fv.fv_plane_projection(st["g"], st["v"], case["plane"], st["vp"], st["psi"])
        return {"v": st["vp"], "psi": st["psi"]}
    net = st["net"]
    net.forward((case["nx"], case["ny"], case["nz"]), st["planes"], st["out"])
    loss = net.backward(st["target"])
    net.get_params(grads=st["grads"])
    return {"out": st["out"], "loss": loss, "grads": st["grads"]}


# ------------------------------------------------------------------- work --

def _krylov_work(n, cells, prec, p):
    """J.v reads U and v and writes w; one exact pressure solve (six dense transforms) and one correction."""
    flops = cells * (4.0 * sum(n) + 300)
    return {"bytes": cells * (72.0 + (8 if p else 0)), "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_krylov_work((n, n, n), n ** 3, "mixed", False) for n, _, _ in _instances(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    n = (case["nx"], case["ny"], case["nz"])
    cells = n[0] * n[1] * n[2]
    if kind == "krylov":
        return _krylov_work(n, cells, case["prec"], case["p"])
    if kind == "arnoldi":   # at the least one Krylov dimension of vectors, orthogonalised twice
        one = _krylov_work(n, cells, case["prec"], False)
        m = case["m"]
        return {"bytes": m * one["bytes"] + 24.0 * cells * m * m, "flops": m * one["flops"] + 12.0 * cells * m * m}
    if kind == "newton":    # at the least one vector per correction of a few
        one = _krylov_work(n, cells, case["prec"], False)
        return {k: 5 * one[k] for k in one}
    if kind == "mg":        # at the least one smoothing cycle (12 sweeps of 7-point rows) and the vectors of one step
        return {"bytes": cells * 16.0, "flops": cells * 200.0}
    if kind == "planes":
        a, c = {"xz": (0, 2), "yz": (1, 2), "xy": (0, 1)}[case["plane"]]
        return {"bytes": cells * 56.0, "flops": cells * (4.0 * (n[a] + n[c]) + 20)}
    flops = 0.0
    for lev, ci, co in _UNET:
        flops += 3 * 2 * 27.0 * ci * co * cells / 8 ** lev
    return {"bytes": 4.0 * (6 * cells + 3 * _N_PARAM), "flops": flops}


# ------------------------------------------------- float64 restatements ----

class _Ops:
    """Staggered finite-volume operators and exact Neumann solves in float64."""

    def __init__(self, shape, map):
        nz, ny, nx = shape
        self.n = (nx, ny, nz)
        self.shape = shape
        self.dx, self.dc, self.th, self.lam, self.E, self.Ei = [], [], [], [], [], []
        self.null = []
        for n in self.n:
            x = _faces(n, map)
            dx = np.diff(x)
            xc = 0.5 * (x[1:] + x[:-1])
            dc = np.concatenate([[0.5 * dx[0]], np.diff(xc), [0.5 * dx[-1]]])
            g = 1.0 / dc[1:-1]
            T = np.diag(g, 1) + np.diag(g, -1)
            T -= np.diag(T.sum(1))
            s = np.sqrt(dx)
            lam, Q = np.linalg.eigh(T / s[:, None] / s[None, :])
            self.null.append(int(np.argmax(lam)))
            to = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
            self.dx.append(to(dx))
            self.dc.append(to(dc))
            self.th.append(to(0.5 * dx[:-1] / dc[1:-1]))
            self.lam.append(to(lam))
            self.E.append(to(Q / s[:, None]))
            self.Ei.append(to(Q.T * s[None, :]))

    @staticmethod
    def last(a, d):
        return a.movedim(2 - d, -1)

    @staticmethod
    def back(a, d):
        return a.movedim(-1, 2 - d)

    def full(self, q):
        """[u | v | w] -> three arrays with both wall faces."""
        q = q.reshape(3, *self.shape)
        return [self.back(torch.nn.functional.pad(self.last(q[c], c), (0, 1)), c) for c in range(3)]

    def cut(self, q):
        return torch.stack([self.back(self.last(q[c], c)[..., :-1], c) for c in range(3)]).reshape(-1)

    def mid(self, a, d):
        """From centres along d to faces, distance-weighted; wall faces zero."""
        a = self.last(a, d)
        m = a[..., :-1] + self.th[d] * (a[..., 1:] - a[..., :-1])
        return self.back(torch.nn.functional.pad(m, (1, 1)), d)

    def jv(self, U, v, re):
        """(1/Re) Lap v - div(U v) - div(v U) with zero wall values."""
        out = []
        for c in range(3):
            acc = torch.zeros_like(v[c])
            for d in range(3):
                if d == c:
                    a, b = self.last(U[c], c), self.last(v[c], c)
                    f = (b[..., 1:] - b[..., :-1]) / self.dx[c] / re - 0.5 * (a[..., 1:] + a[..., :-1]) * (b[..., 1:] + b[..., :-1])
                    t = torch.nn.functional.pad((f[..., 1:] - f[..., :-1]) / self.dc[c][1:-1], (1, 1))
                else:
                    b = torch.nn.functional.pad(self.last(v[c], d), (1, 1))
                    g = (b[..., 1:] - b[..., :-1]) / self.dc[d] / re
                    f = self.mid(U[d], c) * self.mid(v[c], d) + self.mid(v[d], c) * self.mid(U[c], d)
                    t = g - self.last(f, d)
                    t = (t[..., 1:] - t[..., :-1]) / self.dx[d]
                acc += self.back(t, d)
            a = self.last(acc, c)
            a[..., 0] = 0.0
            a[..., -1] = 0.0
            out.append(acc)
        return out

    def div(self, q, axes=(0, 1, 2)):
        r = 0
        for c in axes:
            a = self.last(q[c], c)
            r = r + self.back((a[..., 1:] - a[..., :-1]) / self.dx[c], c)
        return r

    def grad(self, p, c):
        a = self.last(p, c)
        return self.back(torch.nn.functional.pad((a[..., 1:] - a[..., :-1]) / self.dc[c][1:-1], (1, 1)), c)

    def along(self, t, d):
        s = [1, 1, 1]
        s[2 - d] = -1
        return t.reshape(s)

    def solve(self, r, axes=(0, 1, 2)):
        """The sum of the 1-D Neumann operators along `axes`, inverted with the constants left out."""
        den, null = 0.0, True
        for d in axes:
            r = self.back(self.last(r, d) @ self.Ei[d].T, d)
            den = den + self.along(self.lam[d], d)
            null = null & self.along(torch.arange(self.n[d], device="cuda") == self.null[d], d)
        r = torch.where(null, 0.0, r / torch.where(null, 1.0, den))
        for d in axes:
            r = self.back(self.last(r, d) @ self.E[d].T, d)
        return r

    def krylov(self, U, v, re, sigma):
        U, v = self.full(U), self.full(v)
        w = [a + sigma * b for a, b in zip(self.jv(U, v, re), v)]
        p = self.solve(self.div(w))
        return self.cut([w[c] - self.grad(p, c) - sigma * v[c] for c in range(3)]), p.reshape(-1)

    def planes(self, v, plane):
        a, c = {"xz": (0, 2), "yz": (1, 2), "xy": (0, 1)}[plane]
        q = self.full(v)
        b = 3 - a - c
        q[b] = torch.zeros_like(q[b])
        phi = self.solve(self.div(q, (a, c)), (a, c))
        for d in (a, c):
            q[d] = q[d] - self.grad(phi, d)
        sign = 1.0 if plane == "xz" else -1.0
        body = sign * self.last(self.back(self.last(q[c], c)[..., :-1], c), a) * self.dx[a]
        psi = torch.nn.functional.pad(torch.cumsum(body, -1), (1, 0))
        psi = self.last(self.back(psi, a), c)
        psi = self.back(torch.nn.functional.pad(psi, (0, 1)), c)
        return self.cut(q), psi.reshape(-1)


# the learned guess: (level, channels in, channels out) of its 3^3 convolutions, in parameter order
_UNET = [(0, 16, 16), (0, 16, 16), (1, 16, 32), (1, 32, 32), (2, 32, 48), (2, 48, 48), (3, 48, 64), (3, 64, 64),
         (2, 112, 48), (2, 48, 48), (1, 80, 32), (1, 32, 32), (0, 48, 16), (0, 16, 16)]
_N_PARAM = sum(27 * ci * co + co for _, ci, co in _UNET) + 17


def _unet_params(gen):
    """He-normal weights and small biases in the network's flat layout."""
    parts = []
    for _, ci, co in _UNET:
        parts.append(torch.randn(27 * ci * co, device="cuda", generator=gen) * math.sqrt(2.0 / (27 * ci)))
        parts.append(0.05 * torch.randn(co, device="cuda", generator=gen))
    parts.append(torch.randn(17, device="cuda", generator=gen) * 0.25)
    return torch.cat(parts)


def _unet_exact(case, s):
    flat = s["params"].double().requires_grad_(True)
    o, convs = 0, []
    for _, ci, co in _UNET:
        w = flat[o:o + 27 * ci * co].reshape(3, 3, 3, co, ci).permute(3, 4, 0, 1, 2)
        o += 27 * ci * co
        convs.append((w, flat[o:o + co]))
        o += co
    head, bias = flat[o:o + 16], flat[o + 16]
    F = torch.nn.functional
    relu = lambda x, k: F.relu(F.conv3d(x, convs[k][0], convs[k][1], padding=1))  # noqa: E731
    x = s["planes"].double().reshape(1, 4, *_shape(case))
    x = F.pad(x, (0, 0, 0, 0, 0, 0, 0, 12))
    skips = []
    for lev in range(3):
        x = relu(relu(x, 2 * lev), 2 * lev + 1)
        skips.append(x)
        x = F.avg_pool3d(x, 2)
    x = relu(relu(x, 6), 7)
    for lev in (2, 1, 0):
        x = torch.cat([F.interpolate(x, scale_factor=2, mode="nearest"), skips[lev]], 1)
        k = 8 + 2 * (2 - lev)
        x = relu(relu(x, k), k + 1)
    out = (x[0] * head[:, None, None, None]).sum(0).reshape(-1) + bias
    e = out - s["target"].double()
    loss = (e - e.mean()).square().mean()
    (g,) = torch.autograd.grad(loss, flat)
    return {"out": out.detach(), "loss": float(loss), "grads": g}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("arnoldi", "newton"):
        return None
    s = _inputs(case, seed)
    if kind == "krylov":
        v, p = _Ops(_shape(case), case["map"]).krylov(s["U"], s["v"], case["re"], case["sigma"])
        return {"v": v, "p": p} if case["p"] else {"v": v}
    if kind == "batch":
        return [_Ops((n, n, n), case["map"]).krylov(U, v, re, case["sigma"])[0]
                for (n, re, _), U, v in zip(_instances(case), s["U"], s["v"])]
    if kind == "mg":
        return _Ops(_shape(case), case["map"]).solve(s["r"].reshape(_shape(case))).reshape(-1)
    if kind == "planes":
        v, psi = _Ops(_shape(case), case["map"]).planes(s["v"], case["plane"])
        return {"v": v, "psi": psi}
    return _unet_exact(case, s)
