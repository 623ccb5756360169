"""Performance cases: what a user of the library has it do, through its Python binding.

Four kinds of pass, each with inputs made from a seed:

* ``projection``  one pressure projection of a time step: assemble the operator for the current
                  volume fraction, form the right-hand side from the face velocities (with the
                  balanced radiation exit where every wall is free-slip), solve, project the
                  velocities.  Solved to 1e-12, where the pressure is settled in the digits it is
                  returned in.
* ``operator``    a new operator, its right-hand side and one product with it, as a caller does who
                  brings an iteration of his own.
* ``advect``      one volume-fraction step (flux-error correction and three split stages).
* ``network``     the learned preconditioner: one application, or one training step.

Bodies and waves are those of the library's workloads: a slender hull in waves on the stretched
3 x 1 x 1.5 domain, a half-immersed sphere, a wave on a uniform cube.
"""
import math
import os

import numpy as np
import torch

from paper_1410_1937_gb300 import inputs, vofp

NEUMANN, DIRICHLET = 0, 1
RHO_LIQUID, RHO_GAS, MERGE = 1000.0, 1.2, 0.1
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(vofp.__file__)), "weights", "unet_hull_256x128x64.npz")
DEV = "cuda"
F64 = torch.float64


# ---- the cases -------------------------------------------------------------------------------

def _projection(nx, ny, nz, body, mode, precond, smoothing=0, exit_flux=0):
    return {"kind": "projection", "nx": nx, "ny": ny, "nz": nz, "body": body, "mode": mode, "precond": precond,
            "smoothing": smoothing, "exit_flux": exit_flux}


def listed():
    return [
        # the small uniform cube: latency of a solve whose vectors fit in a few SMs' caches
        dict(_projection(32, 32, 32, "none", "fp64", "jacobi"), name="projection 32^3 fp64"),
        # a small grid in the time stepper's default mode (mixed precision, red-black)
        dict(_projection(64, 48, 40, "hull", "mixed", "rbsgs"), name="projection 64x48x40 mixed rb"),
        # the sphere with merged cells, plain FP64 conjugate gradients
        dict(_projection(128, 64, 64, "sphere", "fp64", "jacobi"), name="projection 128x64x64 fp64"),
        # odd sizes and the paper's boundary set: smoothed density, free-slip walls, radiation exit
        dict(_projection(125, 61, 47, "hull", "fp64", "rbsgs", 1, 1), name="projection 125x61x47 fp64 rb exit"),
        # rows that are not a multiple of 16 bytes, mixed precision with the diagonal preconditioner
        dict(_projection(250, 123, 62, "hull", "mixed", "jacobi"), name="projection 250x123x62 mixed"),
        # the grid the network is trained on: mixed precision, red-black
        dict(_projection(256, 128, 64, "hull", "mixed", "rbsgs"), name="projection 256x128x64 mixed rb"),
        # the ship-wave workload
        dict(_projection(512, 256, 128, "hull", "mixed", "rbsgs"), name="projection 512x256x128 mixed rb"),
        dict({"kind": "operator", "nx": 512, "ny": 256, "nz": 128, "body": "hull", "smoothing": 1},
             name="operator 512x256x128"),
        dict({"kind": "advect", "nx": 203, "ny": 101, "nz": 67, "body": "sphere", "order": 1},
             name="advect 203x101x67 zyx"),
        dict({"kind": "advect", "nx": 512, "ny": 256, "nz": 128, "body": "hull", "order": 0},
             name="advect 512x256x128"),
        dict({"kind": "network", "nx": 512, "ny": 256, "nz": 128, "body": "hull", "train": 0},
             name="network 512x256x128"),
        dict({"kind": "network", "nx": 256, "ny": 128, "nz": 64, "body": "hull", "train": 1},
             name="network training 256x128x64"),
    ]


def _grid(rng, lo, hi, step=1):
    """Sizes with lo .. hi cells (spread over the logarithm), x the longest axis."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ry, rz = rng.uniform(0.4, 1.0), rng.uniform(0.25, 0.8)
    nx = (cells / (ry * rz)) ** (1.0 / 3.0)
    dims = [max(8, step * int(n / step)) for n in (nx, ry * nx, rz * nx)]
    return {"nx": dims[0], "ny": dims[1], "nz": dims[2]}


def draw(rng):
    kind = rng.choice(["projection", "projection", "projection", "operator", "advect", "network"])
    if kind == "projection":
        mode = rng.choice(["fp64", "mixed", "mixed"])
        g = _grid(rng, 2e4, 6e5 if mode == "fp64" else 1.2e7, rng.choice([1, 2, 8, 16]))
        body = rng.choice(["none", "sphere", "hull", "hull"])
        c = _projection(g["nx"], g["ny"], g["nz"], body, mode, rng.choice(["jacobi", "rbsgs"]), rng.choice([0, 0, 1]),
                        rng.choice([0, 0, 1]))
    elif kind == "operator":
        c = {"kind": kind, **_grid(rng, 2e4, 1.6e7, rng.choice([1, 2, 8])), "body": rng.choice(["none", "sphere", "hull"]),
             "smoothing": rng.choice([0, 1])}
    elif kind == "advect":
        c = {"kind": kind, **_grid(rng, 2e4, 1.6e7, rng.choice([1, 2, 8])), "body": rng.choice(["none", "sphere", "hull"]),
             "order": rng.choice([0, 1])}
    else:
        train = rng.choice([0, 1])
        c = {"kind": kind, **_grid(rng, 3e4, 2e6 if train else 1.6e7, 4), "body": "hull", "train": train}
    return c


# ---- inputs ----------------------------------------------------------------------------------

def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=F64, device=DEV)


def _nodes(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["body"] == "none":
        return tuple(inputs.uniform_nodes(-0.5, 0.5, n) for n in (nx, ny, nz))
    if case["body"] == "sphere":
        return (inputs.tanh_nodes(-1.0, 1.0, nx, 0.0, 0.15), inputs.tanh_nodes(-0.5, 0.5, ny, 0.0, 0.15),
                inputs.tanh_nodes(-0.5, 0.5, nz, 0.0, 0.15))
    return inputs.hull_domain_nodes(nx, ny, nz)


def _half_width(body, x, z):
    """Half extent in y of the body at (x, z): the body is |y| < _half_width."""
    if body == "sphere":
        return torch.sqrt(torch.clamp(0.15 ** 2 - x * x - z * z, min=0.0))
    return 0.05 * torch.clamp(1 - (2 * x) ** 2, min=0.0) * torch.clamp(1 - (z / 0.0625) ** 2, min=0.0)


def _open_fractions(case, nodes, shift):
    """Open volume fractions and face apertures around the body moved by `shift` (by quadrature over
    the cells that can touch it; 1 elsewhere)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    vf = torch.ones(nz, ny, nx, dtype=F64, device=DEV)
    ax = torch.ones(nz, ny, nx + 1, dtype=F64, device=DEV)
    ay = torch.ones(nz, ny + 1, nx, dtype=F64, device=DEV)
    az = torch.ones(nz + 1, ny, nx, dtype=F64, device=DEV)
    if case["body"] == "none":
        return vf, ax, ay, az
    half = (0.15, 0.15, 0.15) if case["body"] == "sphere" else (0.5, 0.05, 0.0625)
    r, sub = [], []
    for n, s, h in zip(nodes, shift, half):
        n = n - s
        i0 = max(int(np.searchsorted(n, -h)) - 1, 0)
        i1 = min(int(np.searchsorted(n, h)) + 1, len(n) - 1)
        r.append((i0, max(i1, i0 + 1)))
        sub.append(_dev(n[i0:max(i1, i0 + 1) + 1]))
    (i0, i1), (j0, j1), (k0, k1) = r
    xn, yn, zn = sub
    t, wt = np.polynomial.legendre.leggauss(8)
    t, wt = 0.5 * (t + 1.0), 0.5 * wt

    def chord(x, z):
        """Blocked share of every y interval at (x, z): (z, y, x)."""
        h = _half_width(case["body"], x, z)
        a, b = yn[None, :-1, None], yn[None, 1:, None]
        return torch.clamp(torch.minimum(b, h) - torch.maximum(a, -h), min=0.0) / (b - a)

    def at(n, f):
        return n[:-1] + (n[1:] - n[:-1]) * f

    def snap(blocked):
        o = torch.clamp(1.0 - blocked, 0.0, 1.0)
        o[o < 1e-12] = 0.0
        o[o > 1 - 1e-12] = 1.0
        return o

    xs = [at(xn, f)[None, None, :] for f in t]
    zs = [at(zn, f)[:, None, None] for f in t]
    vf[k0:k1, j0:j1, i0:i1] = snap(sum(wa * wb * chord(x, z) for wa, x in zip(wt, xs) for wb, z in zip(wt, zs)))
    ax[k0:k1, j0:j1, i0:i1 + 1] = snap(sum(wb * chord(xn[None, None, :], z) for wb, z in zip(wt, zs)))
    az[k0:k1 + 1, j0:j1, i0:i1] = snap(sum(wa * chord(x, zn[:, None, None]) for wa, x in zip(wt, xs)))
    q = [(m + 0.5) / 12 for m in range(12)]
    ay[k0:k1, j0:j1 + 1, i0:i1] = snap(sum(
        (_half_width(case["body"], at(xn, f)[None, None, :], at(zn, g)[:, None, None]) > yn[None, :, None].abs()).to(F64)
        for f in q for g in q) / len(q) ** 2)
    return vf, ax, ay, az


def _fields(case, seed):
    """Grid, wave, body and face velocities of one time step."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(seed)
    amp, lam, theta = rng.uniform(0.005, 0.02), rng.uniform(0.2, 0.5), rng.uniform(0.0, 2 * math.pi)
    shift = (rng.uniform(-0.1, 0.1), rng.uniform(-0.05, 0.05), rng.uniform(-0.01, 0.01))
    xn, yn, zn = _nodes(case)
    if case["body"] == "none":
        amp, lam = 0.05, 1.0
    F = _dev(inputs.vof_cosine(xn, yn[:2], zn, amp, lam, theta)).expand(nz, ny, nx).contiguous()
    vf, ax, ay, az = _open_fractions(case, (xn, yn, zn), shift)
    g = torch.Generator(device=DEV).manual_seed(int(seed))

    def u(*shape):
        return torch.rand(*shape, generator=g, dtype=F64, device=DEV) * 2.0 - 1.0
    v = {"F": F, "vf": vf, "ax": ax, "ay": ay, "az": az, "u": u(nz, ny, nx + 1), "v": u(nz, ny + 1, nx),
         "w": u(nz + 1, ny, nx)}
    return np.diff(xn), np.diff(yn), np.diff(zn), {k: a.reshape(-1) for k, a in v.items()}


def _walls(case):
    """Free-slip walls; the exit has p = 0, or the radiation condition on a free-slip wall."""
    return (NEUMANN, NEUMANN if case.get("exit_flux") else DIRICHLET, NEUMANN, NEUMANN, NEUMANN, NEUMANN)


def _build(s):
    c, t = s["case"], s["t"]
    s["ctx"].vofp_build_operator(t["F"], t["ax"], t["ay"], t["az"], t["vf"], _walls(c), RHO_LIQUID, RHO_GAS, MERGE,
                                 c.get("smoothing", 0), 1.0)


def _network_state(s):
    """A network bound to the grid and a scaled residual for it: the committed weights, or for
    training the initial ones and the scaled solution they are to give."""
    c, t, ctx = s["case"], s["t"], s["ctx"]
    _build(s)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    x = torch.zeros_like(b)
    if c["train"]:
        x, _ = ctx.vofp_solve(b, mode=vofp.MODE_MIXED, precond=vofp.PRECOND_RBSGS, rtol=1e-6)
    r, target = ctx.vofp_scaled_pair(b, x)
    net = vofp.Network(seed=0)
    if not c["train"]:
        with np.load(WEIGHTS) as f:
            net.set_params(f["params"])
    net.bind(ctx, t["F"])
    geo, mask = net.export_geometry()
    s.update(net=net, r=r, target=target, geo=geo, mask=mask, params=net.get_params())
    ctx.close()
    del s["ctx"], s["t"]
    return s


def prepare(case, seed):
    dx, dy, dz, t = _fields(case, seed)
    s = {"case": case, "d": (dx, dy, dz), "t": t, "ctx": vofp.Context(dx, dy, dz)}
    kind = case["kind"]
    if kind == "network":
        return _network_state(s)
    if kind == "advect":
        # a projected velocity field, and the caller's Courant limit: 0.4 of a cell at its fastest
        _build(s)
        b = s["ctx"].vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
        p, _ = s["ctx"].vofp_solve(b, mode=vofp.MODE_MIXED, precond=vofp.PRECOND_RBSGS, rtol=1e-6)
        t["u"], t["v"], t["w"], _, _ = s["ctx"].vofp_project(p, t["u"], t["v"], t["w"], want_div=False, want_max=False)
        u = s["ctx"].vofp_vof_flux_correct(t["ax"], t["ay"], t["az"], t["u"], t["v"], t["w"])
        nz, ny, nx = len(dz), len(dy), len(dx)
        hx, hy, hz = _axis_widths((dx, dy, dz))
        ux, uy = u[0].reshape(nz, ny, nx + 1).abs(), u[1].reshape(nz, ny + 1, nx).abs()
        s["dt"] = 0.4 / max(float((a / h).max()) for a, h in (
            (ux[:, :, 1:], hx), (ux[:, :, :-1], hx), (uy[:, 1:], hy), (uy[:, :-1], hy),
            (u[2].reshape(nz, ny, nx).abs(), hz), (u[3].reshape(nz, ny, nx).abs(), hz)))
    if kind == "operator":
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
        s["x"] = torch.randn(t["F"].numel(), generator=g, dtype=F64, device=DEV)
    return s


# ---- one pass --------------------------------------------------------------------------------

def run(s):
    c = s["case"]
    if c["kind"] == "network":
        net = s["net"]
        if not c["train"]:
            return net.forward(s["r"])
        # a training set keeps each sample's geometry, and binds it for its step
        net.set_geometry((c["nz"], c["ny"], c["nx"]), s["geo"], s["mask"])
        loss = net.train_step(s["r"], s["target"], lr=1e-4)
        return {"loss": loss, "gradients": net.get_params(grads=True)}
    ctx, t = s["ctx"], s["t"]
    if c["kind"] == "advect":
        return ctx.vofp_vof_advect(t["F"], t["ax"], t["ay"], t["az"], t["vf"], t["u"], t["v"], t["w"], s["dt"],
                                   order=c["order"])
    _build(s)
    if c["kind"] == "operator":
        return {"b": ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"]), "y": ctx.vofp_apply(s["x"])}
    out = {}
    if c["exit_flux"]:
        out["g"], out["shift"] = ctx.vofp_exit_flux(t["u"], t["v"], t["w"], u_c=1.0, balance=True)
    b = ctx.vofp_rhs_from_face_velocity(t["u"], t["v"], t["w"])
    out["p"], _ = ctx.vofp_solve(b, mode=vofp.MODE_MIXED if c["mode"] == "mixed" else vofp.MODE_FP64,
                                 precond=vofp.PRECOND_RBSGS if c["precond"] == "rbsgs" else vofp.PRECOND_JACOBI,
                                 rtol=1e-12)
    out["u"], out["v"], out["w"], _, _ = ctx.vofp_project(out["p"], t["u"], t["v"], t["w"], want_div=False,
                                                          want_max=False)
    return out


def work(case):
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "network":
        # two operations per tap and pair of channels, at full, half and quarter resolution
        full, half, quarter = 8 * 16 + 16 * 16 + 48 * 16 + 16 * 16, 16 * 32 + 32 * 32 + 96 * 32 + 32 * 32, 32 * 64 + 64 * 64
        flops = 2.0 * 27 * n * (full + half / 8 + quarter / 64)
        # geometry channels (16 bytes), residual, mask, result (or target); training: three such passes
        return {"bytes": 28.0 * n, "flops": flops * (3 if case["train"] else 1)}
    # five input fields and three face velocities of 8 bytes; results: four fields, one or two
    out = {"projection": 4, "operator": 3, "advect": 1}[case["kind"]]
    flops = {"projection": 200, "operator": 60, "advect": 120}[case["kind"]]
    return {"bytes": 8.0 * n * (8 + out), "flops": float(flops * n)}


# ---- the same results in 64 bits by plain torch ------------------------------------------------

def _axis_widths(d):
    dx, dy, dz = (_dev(a) for a in d)
    return dx[None, None, :], dy[None, :, None], dz[:, None, None]


class _Operator:
    """The merged finite-volume operator, matrix-free on (nz, ny, nx) arrays."""

    def __init__(self, case, d, t):
        nz, ny, nx = self.shape = (case["nz"], case["ny"], case["nx"])
        self.h = dx, dy, dz = _axis_widths(d)
        g = {"F": (nz, ny, nx), "vf": (nz, ny, nx), "ax": (nz, ny, nx + 1), "ay": (nz, ny + 1, nx), "az": (nz + 1, ny, nx)}
        F, vf, ax, ay, az = (t[k].reshape(v).clone() for k, v in g.items())
        rho = RHO_GAS + (RHO_LIQUID - RHO_GAS) * F
        if case.get("smoothing"):
            for ax_ in (2, 1, 0):
                lo = torch.cat([rho.narrow(ax_, 0, 1), rho.narrow(ax_, 0, rho.shape[ax_] - 1)], ax_)
                hi = torch.cat([rho.narrow(ax_, 1, rho.shape[ax_] - 1), rho.narrow(ax_, rho.shape[ax_] - 1, 1)], ax_)
                rho = 0.25 * lo + 0.5 * rho + 0.25 * hi
        self.exit = _walls(case)[1] == DIRICHLET
        on = vf > 0
        while True:   # a cell without an open face that carries flux has no unknown
            o = torch.zeros_like(on)
            o[:, :, 1:] |= (ax[:, :, 1:-1] > 0) & on[:, :, :-1]
            o[:, :, :-1] |= (ax[:, :, 1:-1] > 0) & on[:, :, 1:]
            o[:, 1:] |= (ay[:, 1:-1] > 0) & on[:, :-1]
            o[:, :-1] |= (ay[:, 1:-1] > 0) & on[:, 1:]
            o[1:] |= (az[1:-1] > 0) & on[:-1]
            o[:-1] |= (az[1:-1] > 0) & on[1:]
            if self.exit:
                o[:, :, -1] |= ax[:, :, -1] > 0
            if bool((on & o).eq(on).all()):
                break
            on &= o
        self.on = on
        for a, dim in ((ax, 2), (ay, 1), (az, 0)):   # faces of a cell without an unknown are closed
            n = a.shape[dim]
            a.narrow(dim, 1, n - 1).mul_(on)
            a.narrow(dim, 0, n - 1).mul_(on)
        S = (dy * dz).expand(nz, ny, 1), (dx * dz).expand(nz, 1, nx), (dx * dy).expand(1, ny, nx)
        self.A = ax * S[0], ay * S[1], az * S[2]
        self.S = S
        self.inv, self.T = [], []
        for a, dim, h in zip(self.A, (2, 1, 0), (dx, dy, dz)):
            r = 0.5 * (h * rho)
            n = r.shape[dim]
            inv = 1.0 / (r.narrow(dim, 0, n - 1) + r.narrow(dim, 1, n - 1))
            self.inv.append(inv)
            self.T.append(a.narrow(dim, 1, n - 1) * inv)
        self.out = 1.0 / (0.5 * dx[:, :, -1:] * rho[:, :, -1:])          # towards the exit face
        diag = torch.zeros(self.shape, dtype=F64, device=DEV)
        for T, dim in zip(self.T, (2, 1, 0)):
            n = diag.shape[dim]
            diag.narrow(dim, 0, n - 1).add_(T)
            diag.narrow(dim, 1, n - 1).add_(T)
        if self.exit:
            diag[:, :, -1:] += self.A[0][:, :, -1:] * self.out
        self.diag = diag
        self.root = self._roots(vf)
        self.unknown = (self.root == torch.arange(self.root.numel(), device=DEV)) & on.reshape(-1)

    def _roots(self, vf):
        """Master cell of every cell's merge group (the cell itself where it is not merged)."""
        nz, ny, nx = self.shape
        n = nx * ny * nz
        Ax, Ay, Az = self.A
        root = torch.arange(n, device=DEV)
        small = (vf < MERGE) & self.on
        cells = small.reshape(-1).nonzero()[:, 0]
        if not cells.numel():
            return root
        k, j, i = cells // (nx * ny), cells // nx % ny, cells % nx
        f = torch.stack([Ax[k, j, i] * (i > 0), Ax[k, j, i + 1] * (i < nx - 1), Ay[k, j, i] * (j > 0),
                         Ay[k, j + 1, i] * (j < ny - 1), Az[k, j, i] * (k > 0), Az[k + 1, j, i] * (k < nz - 1)]).cpu().numpy()
        best = f.argmax(axis=0)
        off = np.array([-1, 1, -nx, nx, -nx * ny, nx * ny])
        cells = cells.cpu().numpy()
        vfs = dict(zip(cells.tolist(), vf.reshape(-1)[torch.as_tensor(cells, device=DEV)].tolist()))
        to = {int(a): int(a + off[b]) for a, b, m in zip(cells, best, f.max(axis=0)) if m > 0}
        end = {}
        for c0 in to:
            path, at, c = [], {}, c0
            while c in to and c not in end and c not in at:
                at[c] = len(path)
                path.append(c)
                c = to[c]
            if c in at:   # a cycle: its member of largest open volume
                ring = path[at[c]:]
                r = min(ring, key=lambda q: (-vfs[q], q))
                end.update({q: r for q in ring})
            r = end.get(c, c)
            for q in path:
                end.setdefault(q, r)
        if end:
            q = torch.tensor([list(end.keys()), list(end.values())], device=DEV)
            root[q[0]] = q[1]
        return root

    def fold(self, y):
        """Sum over each group at its master, 0 elsewhere."""
        y = y.reshape(-1) * self.on.reshape(-1)
        moved = ~self.unknown & self.on.reshape(-1)
        out = torch.where(self.unknown, y, torch.zeros_like(y))
        return out.index_add_(0, self.root[moved], y[moved])

    def spread(self, x):
        return (x.reshape(-1)[self.root] * self.on.reshape(-1)).reshape(self.shape)

    def apply(self, x):
        v = self.spread(x)
        y = self.diag * v
        for T, dim in zip(self.T, (2, 1, 0)):
            n = v.shape[dim]
            y.narrow(dim, 0, n - 1).addcmul_(T, v.narrow(dim, 1, n - 1), value=-1)
            y.narrow(dim, 1, n - 1).addcmul_(T, v.narrow(dim, 0, n - 1), value=-1)
        return self.fold(y)

    def rhs(self, t, g=None):
        """Per cell, not merged; the normal velocities of free-slip walls are not used."""
        nz, ny, nx = self.shape
        flux = []
        for a, q, shape, dim in zip(self.A, "uvw", ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)), (2, 1, 0)):
            f = a * t[q].reshape(shape)
            f.narrow(dim, 0, 1).zero_()
            if not (dim == 2 and self.exit):
                f.narrow(dim, f.shape[dim] - 1, 1).zero_()
            flux.append(f.narrow(dim, 1, f.shape[dim] - 1) - f.narrow(dim, 0, f.shape[dim] - 1))
        b = -(flux[0] + flux[1] + flux[2])
        if g is not None:
            b[:, :, -1] += self.A[0][:, :, -1] * g
        return (b * self.on).reshape(-1)

    def exit_flux(self, t):
        nz, ny, nx = self.shape
        u = t["u"].reshape(nz, ny, nx + 1)
        g = (u[:, :, -1] - u[:, :, -2]) / self.h[0][:, :, -1] - u[:, :, -1]
        area = self.A[0][:, :, -1]
        shift = float(self.rhs(t, g).sum() / area.sum())
        return torch.where(area > 0, g - shift, g), shift

    def solve(self, b):
        b = self.fold(b)
        if not self.exit:
            b = b - torch.where(self.unknown, b.sum() / self.unknown.sum(), torch.zeros_like(b))
        # diagonal of the merged operator: couplings inside a group drop out
        d = self.diag.clone()
        root = self.root.reshape(self.shape)
        for T, dim in zip(self.T, (2, 1, 0)):
            n = d.shape[dim]
            same = T * (root.narrow(dim, 0, n - 1) == root.narrow(dim, 1, n - 1))
            d.narrow(dim, 0, n - 1).sub_(same)
            d.narrow(dim, 1, n - 1).sub_(same)
        d = self.fold(d)
        w = torch.where(self.unknown, 1.0 / d, torch.zeros_like(d))
        x = torch.zeros_like(b)
        r, best = b.clone(), float(b.norm())
        for _ in range(3):   # restarted from the true residual
            z = w * r
            p, rz = z.clone(), (r * z).sum()
            for it in range(20000):
                q = self.apply(p)
                a = rz / (p * q).sum()
                x.addcmul_(p, a)
                r.addcmul_(q, a, value=-1)
                z = w * r
                new = (r * z).sum()
                p.mul_(new / rz).add_(z)
                rz = new
                if it % 20 == 19 and float(r.norm()) < 2e-15 * best:
                    break
            r = b - self.apply(x)
            if float(r.norm()) < 2e-14 * best:
                break
        if not self.exit:
            x = x - torch.where(self.unknown, x.sum() / self.unknown.sum(), torch.zeros_like(x))
        return self.spread(x).reshape(-1)

    def project(self, p, t, g=None):
        nz, ny, nx = self.shape
        p = p.reshape(self.shape)
        out = {}
        for q, a, inv, dim, shape in zip("uvw", self.A, self.inv, (2, 1, 0),
                                         ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))):
            u = t[q].reshape(shape).clone()
            n = p.shape[dim]
            u.narrow(dim, 1, n - 1).sub_((p.narrow(dim, 1, n - 1) - p.narrow(dim, 0, n - 1)) * inv
                                         * (a.narrow(dim, 1, n - 1) > 0))
            u.narrow(dim, 0, 1).zero_()
            last = u.narrow(dim, n, 1)
            if dim == 2 and self.exit:
                last.add_(p[:, :, -1:] * self.out * (a[:, :, -1:] > 0))
            elif dim == 2 and g is not None:
                last.copy_(-g[:, :, None])
            else:
                last.zero_()
            out[q] = u.reshape(-1)
        return out


def _cut_volume(m, alpha, h):
    """Volume of {0 <= x <= h, m.x <= alpha} (rows of m and h), by inclusion and exclusion of the
    corner tetrahedra, with the smallest normals' terms in closed form where they vanish."""
    alpha = alpha - (m.clamp(max=0.0) * h).sum(1)
    a = m.abs() * h
    s = a.sum(1)
    vol = h.prod(1)
    a, _ = torch.sort(a / s.clamp(min=1e-300)[:, None], dim=1)
    b = (alpha / s.clamp(min=1e-300)).clamp(0.0, 1.0)
    flip = b > 0.5
    b = torch.where(flip, 1.0 - b, b)
    c1, c2, c3 = a.unbind(1)
    safe1 = c1.clamp(min=1e-300)
    p = 3 * b * b - 3 * b * c1 + c1 * c1
    e2, e3 = b - c2, b - c3
    f1 = b * (b / safe1) * b / (6 * c2 * c3).clamp(min=1e-300)
    f2 = (b * (b - c1) + c1 * c1 / 3) / (2 * c2 * c3).clamp(min=1e-300)
    f3 = (p - e2 * (e2 / safe1) * e2) / (6 * c2 * c3).clamp(min=1e-300)
    f4 = f3 - e3 * (e3 / safe1) * e3 / (6 * c2 * c3).clamp(min=1e-300)
    f5 = (2 * b - c1 - c2) / (2 * c3)
    f = torch.where(b < c1, f1, torch.where(b < c2, f2, torch.where(b < torch.minimum(c1 + c2, c3), f3,
                    torch.where(c3 < c1 + c2, f4, f5))))
    f = torch.where(b <= 0, torch.zeros_like(f), f)
    return torch.where(flip, 1.0 - f, f) * vol


def _advect(case, d, t, dt):
    nz, ny, nx = shape = (case["nz"], case["ny"], case["nx"])
    h = _axis_widths(d)
    S = h[1] * h[2], h[0] * h[2], h[0] * h[1]
    ax, ay, az = t["ax"].reshape(nz, ny, nx + 1), t["ay"].reshape(nz, ny + 1, nx), t["az"].reshape(nz + 1, ny, nx)
    u, v, w = t["u"].reshape(ax.shape), t["v"].reshape(ay.shape), t["w"].reshape(az.shape)
    fx, fy, fz, A = ax * S[0] * u, ay * S[1] * v, az * S[2] * w, az * S[2]
    E = (fx[:, :, 1:] - fx[:, :, :-1]) + (fy[:, 1:] - fy[:, :-1]) + (fz[1:] - fz[:-1])
    tot = A[1:] + A[:-1]
    share = torch.where(tot > 0, E / tot.clamp(min=1e-300), torch.zeros_like(E))
    # corrected velocity of the uncut - and + face of every cell, per axis (x, y, z)
    faces = [(ax[:, :, :-1] * u[:, :, :-1], ax[:, :, 1:] * u[:, :, 1:]), (ay[:, :-1] * v[:, :-1], ay[:, 1:] * v[:, 1:]),
             ((fz[:-1] + share * A[:-1]) / S[2], (fz[1:] - share * A[1:]) / S[2])]
    vol = (h[0] * h[1] * h[2]).expand(shape)
    H = torch.stack([a.expand(shape) for a in h], -1).reshape(-1, 3)
    open_ = torch.nn.functional.pad(t["vf"].reshape(shape) > 0, (1,) * 6)
    phi = t["F"].reshape(shape)

    def spans(a):
        e = torch.cat([a[:1], a, a[-1:]])
        return 0.5 * e[:-2] + e[1:-1] + 0.5 * e[2:]

    span = [spans(_dev(a)) for a in d]
    for stage, axis in enumerate((0, 1, 2) if case["order"] == 0 else (2, 1, 0)):
        P = torch.nn.functional.pad(phi, (1,) * 6)
        grad = [torch.zeros_like(phi) for _ in range(3)]
        for k in range(3):
            for j in range(3):
                for i in range(3):
                    at = (slice(k, k + nz), slice(j, j + ny), slice(i, i + nx))
                    val = torch.where(open_[at], P[at], phi)
                    for g, (o, a, b) in zip(grad, ((i, j, k), (j, i, k), (k, i, j))):
                        if o != 1:
                            g.add_(val, alpha=(o - 1) * (2 - abs(a - 1)) * (2 - abs(b - 1)) / 16.0)
        m = torch.stack([-grad[0] / span[0][None, None, :], -grad[1] / span[1][None, :, None],
                         -grad[2] / span[2][:, None, None]], -1).reshape(-1, 3)
        del grad, P
        flat = phi.reshape(-1)
        cut = ((flat > 0) & (flat < 1) & (m.abs().sum(1) > 0)).nonzero()[:, 0]
        slot = torch.full((flat.numel(),), -1, dtype=torch.long, device=DEV)
        slot[cut] = torch.arange(cut.numel(), device=DEV)
        mc, hc, target = m[cut], H[cut], flat[cut] * vol.reshape(-1)[cut]
        del m
        lo, hi = (mc * hc).clamp(max=0.0).sum(1), (mc * hc).clamp(min=0.0).sum(1)
        for _ in range(70):
            mid = 0.5 * (lo + hi)
            below = _cut_volume(mc, mid, hc) < target
            lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
        alpha = 0.5 * (lo + hi)
        dim = 2 - axis
        n = phi.shape[dim]
        index = torch.arange(flat.numel(), device=DEV).reshape(shape)
        flow = []
        for side, vel in zip((0, 1), faces[axis]):      # - face, + face
            donor_self = vel <= 0 if side == 0 else vel > 0
            nb = index.index_select(dim, torch.arange(n, device=DEV).add(-1 if side == 0 else 1).clamp(0, n - 1))
            donor = torch.where(donor_self, index, nb).reshape(-1)
            plus = vel.reshape(-1) > 0                   # the slab lies at the donor's + face
            hd = H[donor]
            thick = torch.minimum(vel.abs().reshape(-1) * dt, hd[:, axis])
            moved = flat[donor] * (vol.reshape(-1)[donor] / hd[:, axis] * thick)
            sl = slot[donor]
            at = (sl >= 0).nonzero()[:, 0]
            sl, hs = sl[at], hd[at].clone()
            hs[:, axis] = thick[at]
            a = alpha[sl] - torch.where(plus[at], mc[sl, axis] * (hd[at, axis] - thick[at]), torch.zeros_like(alpha[sl]))
            moved[at] = torch.where(thick[at] > 0, _cut_volume(mc[sl], a, hs), torch.zeros_like(a))
            flow.append(torch.where(plus, moved, -moved).reshape(shape))
        adv = phi - (flow[1] - flow[0]) / vol
        div = dt * (faces[axis][1] - faces[axis][0]) / h[axis]
        phi = adv / (1.0 - div) if stage < 2 else adv + phi * div
    return phi.reshape(-1)


CHANNELS = [(16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (32, 32), (48, 16), (16, 16)]


def _network(case, s):
    flat = torch.as_tensor(s["params"], dtype=F64, device=DEV).requires_grad_(bool(case["train"]))
    shape = (case["nz"], case["ny"], case["nx"])
    layers, at = [], 0
    for cin, cout in CHANNELS:
        W = flat[at:at + 27 * cout * cin].reshape(27, cout, cin)
        layers.append((W, flat[at + 27 * cout * cin:at + 27 * cout * cin + cout]))
        at += 27 * cout * cin + cout
    head, bias = flat[at:at + 16], flat[at + 16]

    def conv(x, layer):
        W, b = layer
        c, (nz, ny, nx) = x.shape[0], x.shape[1:]
        xp = torch.nn.functional.pad(x, (1,) * 6)
        y = b[:, None].expand(-1, nz * ny * nx).clone()
        for tap in range(27):
            k, j, i = tap // 9, tap // 3 % 3, tap % 3
            y = y.addmm_(W[tap], xp[:, k:k + nz, j:j + ny, i:i + nx].reshape(c, -1)) if not case["train"] else \
                y + W[tap] @ xp[:, k:k + nz, j:j + ny, i:i + nx].reshape(c, -1)
        return torch.relu(y).reshape(-1, nz, ny, nx)

    def pool(x):
        return torch.nn.functional.avg_pool3d(x[None], 2)[0]

    def up(x):
        return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    r, mask = s["r"].to(F64).reshape(shape), s["mask"].to(F64).reshape(shape)
    rms = ((mask * r * r).sum() / mask.sum()).sqrt()
    geo = s["geo"].view(torch.bfloat16).to(F64).reshape(*shape, 8).permute(3, 0, 1, 2)
    x = torch.cat([geo[:7], (r / rms)[None], torch.zeros(8, *shape, dtype=F64, device=DEV)])
    s1 = conv(conv(x, layers[0]), layers[1])
    s2 = conv(conv(pool(s1), layers[2]), layers[3])
    b3 = conv(conv(pool(s2), layers[4]), layers[5])
    d2 = conv(conv(torch.cat([up(b3), s2]), layers[6]), layers[7])
    d1 = conv(conv(torch.cat([up(d2), s1]), layers[8]), layers[9])
    out = (head @ d1.reshape(16, -1) + bias).reshape(shape)
    if not case["train"]:
        return (mask * out * rms).reshape(-1)
    e = mask * (out - s["target"].to(F64).reshape(shape) / rms)
    loss = (e * e).sum() / mask.sum()
    loss.backward()
    return {"loss": float(loss), "gradients": flat.grad}


def exact(case, seed):
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "network":
        # 2 TFLOP at the card's FP64 rate, and a tape of FP64 activations in training
        return None if n > 3e6 else _network(case, prepare(case, seed))
    if case["kind"] == "advect":
        s = prepare(case, seed)
        return _advect(case, s["d"], s["t"], s["dt"])
    d, t = _fields(case, seed)[:3], _fields(case, seed)[3]
    if case["kind"] == "projection" and n > 3e6:
        return None   # thousands of unfused passes over the grid
    op = _Operator(case, d, t)
    if case["kind"] == "operator":
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
        return {"b": op.rhs(t), "y": op.apply(torch.randn(n, generator=g, dtype=F64, device=DEV))}
    out, g = {}, None
    if case["exit_flux"]:
        g, out["shift"] = op.exit_flux(t)
        out["g"] = g.reshape(-1)
    out["p"] = op.solve(op.rhs(t, g))
    return {**out, **op.project(out["p"], t, g)}
