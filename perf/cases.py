"""Timed workloads of the linear MHS solver: the calls a user's program makes, at the sizes and with the options in use.

A case is a dict of plain values.  ``listed()`` holds the fixed cases, ``draw(rng)`` gives further ones from the same
ranges, ``prepare`` builds what a program has in hand before the call (magnetogram, resident handle, output buffers),
``run`` is one pass through the public entry points, ``work`` the bytes and operations that pass cannot do without, and
``exact`` the exact discrete solution of the same inputs in plain FP64 tensor arithmetic (dense sine transforms, one
tridiagonal system along z per mode, finite differences).

Kinds of pass:

* ``solve``: a new magnetogram is prescribed, the lower-boundary and interior problems are solved to a relative residual
  of 1e-10, and Phi, B, p and rho are copied out (to device tensors, or to pinned host memory with ``host``);
* ``group``: new magnetograms for a resident batch of instances, one grouped solve, Phi of every instance;
* ``post``: B and the atmosphere are recovered from a resident solution and its current density formed, and field
  lines are traced through a field the caller holds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1307_6720_gb300 import mhs

TOL = 1e-10
FIELDS = ("Bx", "By", "Bz", "p", "rho")


def _solve(name, nx, ny, nz, mode, Lx=1.0, Ly=1.0, Lz=1.0, alpha=0.5, xi_kind=mhs.MHS_XI_EXP, a=0.5, kappa=1.0, b=0.0,
           omega=0.0, direct=False, host=False):
    return dict(name=name, kind="solve", nx=nx, ny=ny, nz=nz, Lx=Lx, Ly=Ly, Lz=Lz, alpha=alpha, xi_kind=xi_kind, a=a,
                kappa=kappa, b=b, omega=omega, mode=mode, direct=direct, host=host)


def listed():
    return [
        # the smallest solve in use, the potential-field limit (alpha = 0, xi = 0): launches and latency
        _solve("potential_33_fp64", 33, 33, 33, "fp64", alpha=0.0, xi_kind=mhs.MHS_XI_NONE, a=0.0),
        # the most frequent request of a served stream: host magnetogram in, host results out
        _solve("request_65_mixed_host", 65, 65, 65, "mixed", host=True),
        # the benchmark's workload: linear MHS on 129^3, FP64, all fields
        _solve("mhs_129_fp64", 129, 129, 129, "fp64"),
        # the same equilibrium in mixed precision
        _solve("mhs_129_mixed", 129, 129, 129, "mixed"),
        # the larger cubes: the FP64 comparison run and the mixed-precision production run
        _solve("mhs_257_fp64", 257, 257, 257, "fp64"),
        _solve("mhs_257_mixed", 257, 257, 257, "mixed", alpha=0.9),
        # the largest grid in use
        _solve("mhs_513x513x257_mixed", 513, 513, 257, "mixed", Lz=0.5),
        # a ragged box, no axis a power of two, anisotropic spacing, the second xi family
        _solve("ragged_193x161x97_fp64", 193, 161, 97, "fp64", Ly=0.8, Lz=0.6, alpha=0.3, xi_kind=mhs.MHS_XI_EXP_SIN,
               a=0.6, b=0.2, omega=3.0, kappa=0.8),
        # cross-field currents close to the ellipticity limit: the z-line smoother
        _solve("strong_129x129x65_mixed", 129, 129, 65, "mixed", Lz=0.5, a=0.999, kappa=0.5),
        # the separable direct solver, as a program takes it for many magnetograms of one atmosphere
        _solve("direct_257_fp64", 257, 257, 257, "fp64", direct=True),
        # an uneven batch (33^3 .. 129^3 and a flat box) as one grouped solve
        dict(name="group_32_mixed", kind="group", count=32, mode="mixed", shapes="33x33,65x65,129x129,129x65"),
        # what the figures of a solution are drawn from
        dict(name="post_129", kind="post", nx=129, ny=129, nz=129, Lx=1.0, Ly=1.0, Lz=1.0, alpha=0.5,
             xi_kind=mhs.MHS_XI_EXP, a=0.5, kappa=1.0, b=0.0, omega=0.0, lines=2048, steps=200),
    ]


def _axes(rng, nodes):
    """Odd node counts m 2^k + 1 per axis of about ``nodes`` nodes in all, and a box of nearly isotropic spacing."""
    base = nodes ** (1.0 / 3.0)
    want = [min(513.0, max(17.0, base * rng.uniform(0.7, 1.4))) for _ in range(3)]
    k = rng.choice([3, 4, 5])
    while k > 3 and min(want) / 2 ** k < 1.5:
        k -= 1
    while max(want) / 2 ** k > 16.5:
        k += 1
    n = [max(2, round(w / 2 ** k)) * 2 ** k + 1 for w in want]
    if rng.random() < 0.4:   # cubes and boxes of powers of two are the common choice
        n = [2 ** round(math.log2(v - 1)) + 1 for v in n]
    L = [1.0] + [(v - 1) / (n[0] - 1) * rng.uniform(0.9, 1.1) for v in n[1:]]
    return n, L


def draw(rng):
    t = rng.random()
    if t < 0.1:
        shapes = ["%dx%d" % (n, nz) for n, nz in rng.sample([(33, 33), (65, 65), (129, 129), (129, 65), (49, 25), (65, 33)],
                                                            4)]
        return dict(kind="group", count=rng.randint(8, 32), mode="mixed", shapes=",".join(shapes))
    n, L = _axes(rng, math.exp(rng.uniform(math.log(3.0e4), math.log(1.7e7))))
    xi = dict(xi_kind=mhs.MHS_XI_EXP, a=rng.uniform(0.0, 0.8), kappa=rng.uniform(0.5, 2.0), b=0.0, omega=0.0)
    if rng.random() < 0.25:
        xi = dict(xi_kind=mhs.MHS_XI_EXP_SIN, a=rng.uniform(0.3, 0.6), b=rng.uniform(0.0, 0.2), omega=rng.uniform(1.0, 4.0),
                  kappa=rng.uniform(0.5, 1.5))
    box = dict(nx=n[0], ny=n[1], nz=n[2], Lx=L[0], Ly=L[1], Lz=L[2], alpha=rng.uniform(0.0, 0.8), **xi)
    if t < 0.2:
        return dict(kind="post", lines=rng.randint(64, 4096), steps=rng.randint(50, 300), **box)
    if t < 0.3:   # close to the ellipticity limit
        box.update(xi_kind=mhs.MHS_XI_EXP, a=rng.uniform(0.97, 0.999), b=0.0, omega=0.0, kappa=rng.uniform(0.5, 1.0),
                   alpha=rng.uniform(0.0, 0.4))
    return dict(kind="solve", mode=rng.choice(["fp64", "mixed"]), direct=rng.random() < 0.2, host=rng.random() < 0.2, **box)


# ------------------------------------------------------------------ inputs


def _magnetogram(nx, ny, Lx, Ly, rs):
    """Eight Gaussian spots, amplitudes U[-1, 1], widths U[0.03, 0.1], centres U[0.15, 0.85], flux-balanced."""
    x = np.arange(nx) * (Lx / (nx - 1))
    y = np.arange(ny) * (Ly / (ny - 1))
    pos, neg = np.zeros((ny, nx)), np.zeros((ny, nx))
    for q in range(8):
        amp, width, cx, cy = rs.uniform(-1, 1), rs.uniform(0.03, 0.1) * min(Lx, Ly), rs.uniform(0.15, 0.85), rs.uniform(0.15, 0.85)
        amp = abs(amp) if q == 0 else -abs(amp) if q == 1 else amp   # both polarities
        spot = amp * np.exp(-((x[None, :] - cx * Lx) ** 2 + (y[:, None] - cy * Ly) ** 2) / width ** 2)
        if amp > 0:
            pos += spot
        else:
            neg += spot
    return pos + neg * (pos.sum() / -neg.sum())


def _xi_params(c):
    return mhs.xi_params(c["xi_kind"], c["a"], c["kappa"], c["b"], c["omega"])


def _solver(c):
    return mhs.Solver(c["nx"], c["ny"], c["nz"], c["Lx"], c["Ly"], c["Lz"], c["alpha"], _xi_params(c),
                      stream=torch.cuda.current_stream())


def _instances(c, seed):
    """The boxes of a batch (fixed per case) and one magnetogram each (from the seed)."""
    shapes = [tuple(int(v) for v in s.split("x")) for s in c["shapes"].split(",")]
    out = []
    for i in range(c["count"]):
        n, nz = shapes[i % len(shapes)]
        rs = np.random.RandomState(1000 + i)
        box = dict(nx=n, ny=n, nz=nz, Lx=1.0, Ly=1.0, Lz=(nz - 1) / (n - 1), alpha=rs.uniform(0.0, 0.8),
                   xi_kind=mhs.MHS_XI_EXP, a=rs.uniform(0.0, 0.9), kappa=rs.uniform(0.5, 2.0), b=0.0, omega=0.0)
        out.append((box, _magnetogram(n, n, 1.0, 1.0, np.random.RandomState((seed * 1009 + i) % (1 << 31)))))
    return out


def _arcade(c, seed):
    """A potential field on the box's nodes (sources below the lower boundary), the box and seeds of field lines."""
    rs = np.random.RandomState((seed * 7919 + 17) % (1 << 31))
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") * (L / (n - 1))
          for n, L in ((c["nx"], c["Lx"]), (c["ny"], c["Ly"]), (c["nz"], c["Lz"]))]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    B = [torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device="cuda") for _ in range(3)]
    for q in range(6):
        s = (1.0 if q % 2 else -1.0) * rs.uniform(0.5, 1.0)
        r = [x - rs.uniform(0.2, 0.8) * c["Lx"], y - rs.uniform(0.2, 0.8) * c["Ly"], z + rs.uniform(0.05, 0.15)]
        w = s * (r[0] ** 2 + r[1] ** 2 + r[2] ** 2) ** -1.5
        for a in range(3):
            B[a] += w * r[a]
    seeds = np.stack([rs.uniform(0.1, 0.9, c["lines"]) * c["Lx"], rs.uniform(0.1, 0.9, c["lines"]) * c["Ly"],
                      rs.uniform(0.02, 0.1, c["lines"]) * c["Lz"]], axis=1)
    return B, torch.from_numpy(seeds).cuda()


def _step(c):
    return 0.5 * min(c["Lx"] / (c["nx"] - 1), c["Ly"] / (c["ny"] - 1), c["Lz"] / (c["nz"] - 1))


# --------------------------------------------------------------- the passes


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "group":
        inst = _instances(c, seed)
        solvers = [_solver(b) for b, _ in inst]
        bz = [torch.from_numpy(m).cuda() for _, m in inst]
        g = _Group(solvers, mhs.MHS_MIXED)
        return dict(case=c, group=g, bz=bz, solvers=solvers)
    s = _solver(c)
    bz = torch.from_numpy(_magnetogram(c["nx"], c["ny"], c["Lx"], c["Ly"], np.random.RandomState(seed % (1 << 31))))
    if c["kind"] == "post":
        s.set_options(flags=mhs.MHS_FLAG_SEPARABLE, max_cycles=20)
        s.set_lower_bz(bz.cuda())
        try:
            s.solve(1e-13, mhs.MHS_FP64)
        except mhs.MhsError as e:   # the last iterate of a solve at its rounding floor is the solution
            if e.status != mhs.MHS_ERR_NO_CONVERGENCE:
                raise
        B, seeds = _arcade(c, seed)
        points = torch.zeros((c["lines"], c["steps"] + 1, 3), dtype=torch.float64, device="cuda")
        lengths = torch.zeros(c["lines"], dtype=torch.int32, device="cuda")
        return dict(case=c, solver=s, B=B, seeds=seeds, points=points, lengths=lengths)
    if c["direct"]:
        s.set_options(flags=mhs.MHS_FLAG_SEPARABLE)
    out = None
    if c["host"]:
        bz = bz.pin_memory()
        out = [torch.empty(s.shape, dtype=torch.float64, pin_memory=True) for _ in range(6)]
    else:
        bz = bz.cuda()
    return dict(case=c, solver=s, bz=bz, out=out)


class _Group:
    """A grouped solver that ends with its members."""

    def __init__(self, solvers, mode):
        self.solvers = solvers
        self.g = mhs.mhs_group_create([s.h for s in solvers], mode)

    def __del__(self):
        mhs.mhs_group_destroy(self.g)


def run(state):
    c = state["case"]
    if c["kind"] == "group":
        for s, bz in zip(state["solvers"], state["bz"]):
            s.set_lower_bz(bz)
        mhs.mhs_group_solve(state["group"].g, c["count"], TOL)
        return [s.phi() for s in state["solvers"]]
    s = state["solver"]
    if c["kind"] == "post":
        f = s.fields()
        j = [torch.empty(s.shape, dtype=torch.float64, device="cuda") for _ in range(5)]
        mhs.mhs_current(s.h, *j)
        mhs.mhs_trace_field(s.shape, (c["Lx"], c["Ly"], c["Lz"]), *state["B"], state["seeds"], _step(c), c["steps"], 1,
                            state["points"], state["lengths"], stream=torch.cuda.current_stream())
        return dict(fields=f, current=j, points=state["points"], lengths=state["lengths"])
    s.set_lower_bz(state["bz"])
    s.solve(TOL, mhs.MHS_FP64 if c["mode"] == "fp64" else mhs.MHS_MIXED)
    if c["host"]:
        out = state["out"]
        mhs.mhs_get_phi(s.h, out[0])
        mhs.mhs_fields(s.h, *out[1:])
        return dict(phi=out[0], fields=dict(zip(FIELDS, out[1:])))
    return dict(phi=s.phi(), fields=s.fields())


# ------------------------------------------------------------- minimal work


def _solve_flops(nx, ny, nz):
    """A multigrid solve to 1e-10 cannot do without about seven V(2,2) cycles of 46 operations per unknown of the finest
    level (four sweeps of 8, a residual of 10, transfers), 8/7 of that over all levels."""
    return 7 * 46 * (8.0 / 7.0) * (nx - 2.0) * (ny - 2.0) * (nz - 1.0)


def work(case):
    c = case
    if c["kind"] == "group":
        byt = flops = 0.0
        for i in range(c["count"]):
            n, nz = (int(v) for v in c["shapes"].split(",")[i % len(c["shapes"].split(","))].split("x"))
            byt += 8.0 * (n * n + n * n * nz)
            flops += _solve_flops(n, n, nz)
        return {"bytes": byt, "flops": flops}
    nodes = float(c["nx"]) * c["ny"] * c["nz"]
    if c["kind"] == "post":
        # P in, five fields and five current arrays out; the lines' points out
        return {"bytes": 8.0 * (11 * nodes + 3 * c["lines"] * (c["steps"] + 1)),
                "flops": 65.0 * nodes + 500.0 * c["lines"] * c["steps"]}
    if c["direct"]:
        # transforms of length 2 (n - 1) at 2.5 N log2 N along x and y, both ways, and one tridiagonal system per mode
        fl = nodes * (10.0 * (math.log2(2 * c["nx"]) + math.log2(2 * c["ny"])) + 5.0)
    else:
        fl = _solve_flops(c["nx"], c["ny"], c["nz"])
    return {"bytes": 8.0 * (float(c["nx"]) * c["ny"] + 6 * nodes), "flops": fl + 45.0 * nodes}


# ----------------------------------------------------------- exact solutions


def _xi(c, z):
    if c["xi_kind"] == mhs.MHS_XI_EXP:
        return c["a"] * torch.exp(-c["kappa"] * z), -c["kappa"] * c["a"] * torch.exp(-c["kappa"] * z)
    if c["xi_kind"] == mhs.MHS_XI_EXP_SIN:
        e, s = torch.exp(-c["kappa"] * z), c["a"] + c["b"] * torch.sin(c["omega"] * z)
        return s * e, (c["b"] * c["omega"] * torch.cos(c["omega"] * z) - c["kappa"] * s) * e
    return torch.zeros_like(z), torch.zeros_like(z)


def _sines(n):
    """sin(pi m i / (n - 1)) for interior i, m, the argument reduced exactly."""
    q = torch.arange(1, n - 1, dtype=torch.int64, device="cuda")
    return torch.sin(math.pi / (n - 1) * (q[:, None] * q[None, :] % (2 * (n - 1))).double())


def _exact_phi(c, bz):
    """The exact solution of eq. (lower_bound) and then of eq. (scalar_pot) on the nodes."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    hx, hy, hz = c["Lx"] / (nx - 1), c["Ly"] / (ny - 1), c["Lz"] / (nz - 1)
    Sx, Sy = _sines(nx), _sines(ny)
    m = [-(4 / h ** 2) * torch.sin(math.pi / (2 * (n - 1)) * torch.arange(1, n - 1, dtype=torch.float64, device="cuda")) ** 2
         for n, h in ((nx, hx), (ny, hy))]
    lam = m[1][:, None] + m[0][None, :]
    scale = 4.0 / ((nx - 1) * (ny - 1))
    hat = (Sy @ torch.as_tensor(bz, device="cuda")[1:-1, 1:-1] @ Sx) * -scale / lam   # lower boundary, mode space
    z = torch.arange(nz, dtype=torch.float64, device="cuda") * hz
    xi, _ = _xi(c, z)
    cz = 1.0 / hz ** 2
    rows = nz - 2
    P = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    xh = torch.empty((rows,) + lam.shape, dtype=torch.float64, device="cuda")
    cp = torch.empty_like(xh)
    for k in range(rows):
        den = (1.0 - xi[k + 1]) * lam + (c["alpha"] ** 2 - 2.0 * cz)
        if k:
            den = den - cz * cp[k - 1]
        cp[k] = cz / den
        xh[k] = -cz * (xh[k - 1] if k else hat) / den
    for k in range(rows - 2, -1, -1):
        xh[k] -= cp[k] * xh[k + 1]
    del cp
    P[0, 1:-1, 1:-1] = Sy @ hat @ Sx
    for k in range(rows):
        P[k + 1, 1:-1, 1:-1] = Sy @ xh[k] @ Sx
    return P


def _d1(f, h, ax):
    """Second-order first difference: central inside, one-sided on the first and last node."""
    f = f.movedim(ax, 0)
    out = torch.empty_like(f)
    out[1:-1] = (f[2:] - f[:-2]) / (2 * h)
    out[0] = (-3 * f[0] + 4 * f[1] - f[2]) / (2 * h)
    out[-1] = (3 * f[-1] - 4 * f[-2] + f[-3]) / (2 * h)
    return out.movedim(0, ax)


def _d2(f, h, ax):
    f = f.movedim(ax, 0)
    out = torch.empty_like(f)
    out[1:-1] = ((f[2:] - f[1:-1]) - (f[1:-1] - f[:-2])) / h ** 2
    out[0] = (2 * f[0] - 5 * f[1] + 4 * f[2] - f[3]) / h ** 2
    out[-1] = (2 * f[-1] - 5 * f[-2] + 4 * f[-3] - f[-4]) / h ** 2
    return out.movedim(0, ax)


def _exact_fields(c, P):
    hx, hy, hz = c["Lx"] / (c["nx"] - 1), c["Ly"] / (c["ny"] - 1), c["Lz"] / (c["nz"] - 1)
    Pz = _d1(P, hz, 0)
    Bx = c["alpha"] * _d1(P, hy, 1) + _d1(Pz, hx, 2)
    By = -c["alpha"] * _d1(P, hx, 2) + _d1(Pz, hy, 1)
    del Pz
    Bz = -(_d2(P, hx, 2) + _d2(P, hy, 1))
    z = (torch.arange(c["nz"], dtype=torch.float64, device="cuda") * hz)[:, None, None]   # below z1 = 5: T_b = 1
    xi, dxi = _xi(c, z)
    mu0, pb = 0.5, torch.exp(-z)
    p = pb - xi * Bz ** 2 / (2 * mu0)
    grad = Bx * _d1(Bz, hx, 2) + By * _d1(Bz, hy, 1) + Bz * _d1(Bz, hz, 0)
    return dict(Bx=Bx, By=By, Bz=Bz, p=p, rho=pb + dxi * Bz ** 2 / (2 * mu0) + xi * grad / mu0)


def _exact_lines(c, B, seeds):
    """The fixed-step RK4 field lines of the tracer: a step is taken when every stage and its end lie in the box."""
    n = torch.tensor([c["nx"], c["ny"], c["nz"]], device="cuda")
    L = torch.tensor([c["Lx"], c["Ly"], c["Lz"]], dtype=torch.float64, device="cuda")
    h = L / (n - 1)
    F = torch.stack([b.reshape(-1) for b in B], 1)
    ds = _step(c)

    def direction(r):
        ok = ((r >= 0) & (r <= L)).all(1)
        s = torch.minimum(torch.maximum(r, torch.zeros_like(r)), L) / h
        i = torch.minimum(s.floor().long(), n - 2)
        f = s - i
        b = 0.0
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    w = 1.0
                    for a, d in ((0, dx), (1, dy), (2, dz)):
                        w = w * (f[:, a] if d else 1 - f[:, a])
                    b = b + w[:, None] * F[(i[:, 0] + dx) + c["nx"] * ((i[:, 1] + dy) + c["ny"] * (i[:, 2] + dz))]
        m = b.norm(dim=1)
        return b / m[:, None], ok & (m > 0)

    pts = torch.zeros((c["lines"], c["steps"] + 1, 3), dtype=torch.float64, device="cuda")
    r = seeds.clone()
    alive = ((r >= 0) & (r <= L)).all(1)
    pts[alive, 0] = r[alive]
    for q in range(c["steps"]):
        k1, o1 = direction(r)
        k2, o2 = direction(r + 0.5 * ds * k1)
        k3, o3 = direction(r + 0.5 * ds * k2)
        k4, o4 = direction(r + ds * k3)
        e = r + ds / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
        alive = alive & o1 & o2 & o3 & o4 & ((e >= 0) & (e <= L)).all(1)
        r = torch.where(alive[:, None], e, r)
        pts[:, q + 1] = torch.where(alive[:, None], e, pts[:, q + 1])
    return pts


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "group":
        return [_exact_phi(b, m) for b, m in _instances(c, seed)]
    P = _exact_phi(c, _magnetogram(c["nx"], c["ny"], c["Lx"], c["Ly"], np.random.RandomState(seed % (1 << 31))))
    f = _exact_fields(c, P)
    if c["kind"] == "solve":
        return dict(phi=P, fields=f)
    del P
    h = [c["Lx"] / (c["nx"] - 1), c["Ly"] / (c["ny"] - 1), c["Lz"] / (c["nz"] - 1)]
    d = lambda q, a: _d1(f[q], h[a], 2 - a)   # noqa: E731
    j = [(d("Bz", 1) - d("By", 2)) / 0.5, (d("Bx", 2) - d("Bz", 0)) / 0.5, (d("By", 0) - d("Bx", 1)) / 0.5]
    j += [(j[0] ** 2 + j[1] ** 2 + j[2] ** 2).sqrt(), (f["Bx"] ** 2 + f["By"] ** 2 + f["Bz"] ** 2).sqrt()]
    # the lengths are whole numbers: a line that grazes a face may end a step apart under another rounding
    return dict(fields=f, current=j, points=_exact_lines(c, *_arcade(c, seed)), lengths=None)
