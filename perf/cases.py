"""The work that a user of the exchange engine has it do, case by case.

A program that runs hybrid-functional dynamics calls the engine once per
step: new occupied orbitals go in (``set_orbitals``, or ``scdm`` when they are
canonical), ``apply_vxx`` returns V_xx phi and E_xx, ``build_ace`` and
``apply_ace`` give the compressed operator to the outer solver.  The cases
below are those calls, alone and together, for water-like systems of 4 to 64
molecules at 0.4 to 1.1 g/cm^3, on grids of 0.18 to 0.4 bohr, in the plain
FP64 form (``precision = 0``, the default) and the mixed form (``precision =
1``), with device and pinned host buffers, one configuration and several, and
the Poisson solver on its own boxes.

A case is a dict of plain values: ``kind`` names the calls, the rest are sizes.

* ``poisson``: ``poisson_batch`` on ``n_box`` boxes of ``e_min``..``e_max`` points
  per axis (FP64).
* ``vxx``: ``set_orbitals`` and ``apply_vxx``.
* ``scdm``: ``scdm`` on a rotated (delocalized) orbital set, then ``apply_vxx``.
* ``ace``: ``build_ace`` and ``apply_ace`` on ``n_vec`` vectors, after an
  ``apply_vxx`` made in the preparation.
* ``ace_apply``: ``apply_ace`` alone, the operator built in the preparation.
* ``step``: all of ``set_orbitals``, ``apply_vxx``, ``build_ace``, ``apply_ace``;
  with ``host`` from and to pinned host arrays.
* ``batch``: ``set_orbitals`` on ``n_cfg`` contexts, then one ``apply_vxx_batch``.
"""
import math

import numpy as np
import torch

from paper_2208_06097_gb300 import sea, synth

BOHR = 0.529177210903  # angstrom per bohr
EPS = 10.0 ** -3.5  # the library's defaults of the orbital and pair thresholds
DELTA = 1e-3
P = 6  # half width of the order-12 stencil
LMAX = 6
DEV = "cuda"


def _mol(kind, n_mol, density, nx, ny=None, nz=None, precision=0, **more):
    """A case of n_mol waters at a density (g/cm^3) on an nx x ny x nz grid."""
    edge = (n_mol * 18.015 / (0.602214076 * density)) ** (1.0 / 3.0)  # angstrom
    return dict(kind=kind, n_mol=n_mol, edge=edge, nx=nx, ny=ny or nx, nz=nz or nx,
                precision=precision, **more)


def listed():
    return [
        # a few dozen boxes for the bare solver: the smallest call, launch and
        # latency bound
        dict(name="poisson_48_ragged", kind="poisson", n_box=48, e_min=9, e_max=16, h=0.245),
        # one (H2O)8 configuration, the smallest system that is run in earnest
        dict(_mol("vxx", 8, 1.0, 48), name="vxx_h2o8_48_fp64"),
        # (H2O)64 at ambient density, the paper-scale exchange application, in
        # the default FP64 form and in the mixed form
        dict(_mol("vxx", 64, 1.0, 96), name="vxx_h2o64_96_fp64"),
        dict(_mol("vxx", 64, 1.0, 96, precision=1), name="vxx_h2o64_96_mixed"),
        # a high plane-wave cutoff: few molecules on a fine grid, large pair boxes
        dict(_mol("vxx", 16, 1.0, 81, precision=1), name="vxx_h2o16_fine81_mixed"),
        # the compressed operator, built and applied to as many vectors as there
        # are orbitals (one outer iteration over all bands)
        dict(_mol("ace", 64, 1.0, 96, n_vec=256), name="ace_h2o64_96_fp64"),
        dict(_mol("ace", 64, 1.0, 96, precision=1, n_vec=256), name="ace_h2o64_96_mixed"),
        # the operator applied to a few vectors (band-by-band solvers), odd grid
        dict(_mol("ace_apply", 32, 1.0, 75, precision=1, n_vec=8), name="ace_few_h2o32_75_mixed"),
        # localization of canonical orbitals, then the exchange on them
        dict(_mol("scdm", 32, 1.0, 72, 75, 76, precision=1), name="scdm_h2o32_72_mixed"),
        # several small configurations in one batched call (data set generation)
        dict(_mol("batch", 8, 0.8, 52, precision=1, n_cfg=6), name="batch_6x_h2o8_52_mixed"),
        # a whole step for a CPU code that keeps its arrays in host memory
        dict(_mol("step", 32, 1.0, 76, precision=1, n_vec=128, host=True),
             name="step_host_h2o32_76_mixed"),
        # a whole step at low density: the largest grid of the stated workloads
        dict(_mol("step", 64, 0.4, 128, precision=1, n_vec=256, host=False),
             name="step_h2o64_d04_128_mixed"),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["poisson", "vxx", "vxx", "ace", "ace", "ace_apply", "scdm", "batch", "step"])
    if kind == "poisson":
        lo = rng.randint(6, 13)
        return dict(kind=kind, n_box=log_int(1, 600), e_min=lo, e_max=lo + rng.randint(0, 7),
                    h=round(rng.uniform(0.18, 0.4), 4))
    most = {"scdm": 40, "batch": 12}.get(kind, 64)
    n_mol = log_int(4, most)
    density = round(rng.uniform(0.4, 1.1), 3)
    edge = (n_mol * 18.015 / (0.602214076 * density)) ** (1.0 / 3.0) / BOHR  # bohr
    h = math.exp(rng.uniform(math.log(0.18), math.log(0.4)))
    top = {"scdm": 84, "batch": 64}.get(kind, 128)
    n = [min(top, max(24, int(edge / h) + d)) for d in (0, rng.randint(0, 2), rng.randint(0, 2))]
    more = {}
    if kind in ("ace", "ace_apply", "step"):
        more["n_vec"] = log_int(1, 4 * n_mol)
    if kind == "step":
        more["host"] = rng.random() < 0.3 and n_mol <= 32 and max(n) <= 96
    if kind == "batch":
        more["n_cfg"] = rng.randint(2, 8)
    return _mol(kind, n_mol, density, *n, precision=rng.randint(0, 1), **more)


def work(case):
    """Bytes: each input once, each output once.  Operations: the conjugate
    gradients (65 per unknown and iteration, about 70 iterations; about 2.5
    pairs per orbital, each on about 29 bohr^3) and the products with W, which
    is nonzero on about 290 bohr^3 per orbital."""
    if case["kind"] == "poisson":
        pts = case["n_box"] * (0.5 * (case["e_min"] + case["e_max"])) ** 3
        return {"bytes": 16.0 * pts, "flops": 65.0 * 70.0 * pts}
    ng = case["nx"] * case["ny"] * case["nz"]
    dv = (case["edge"] / BOHR) ** 3 / ng
    n = 4 * case["n_mol"]
    m = case.get("n_vec", 0)
    cfg = case.get("n_cfg", 1)
    nb = fl = 0.0
    if case["kind"] in ("vxx", "scdm", "batch", "step"):
        nb += 16.0 * n * ng * cfg  # orbitals in, V_xx phi out
        fl += 65.0 * 70.0 * 2.5 * n * min(29.0 / dv, ng) * cfg
    if case["kind"] == "scdm":
        fl += 2.0 * n * n * ng  # the rotation
    if case["kind"] == "ace":
        nb += 16.0 * n * ng  # orbitals and W
        fl += 2.0 * n * n * min(290.0 / dv, ng)
    if case["kind"] == "step":
        fl += 2.0 * n * n * min(290.0 / dv, ng)
    if m:
        nb += 16.0 * m * ng  # vectors in, V^ACE psi out
        fl += 4.0 * n * m * min(290.0 / dv, ng)
    return {"bytes": nb, "flops": fl}


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _orbitals(case, seed):
    """(orbitals, cell, grid) of one configuration, on the device."""
    grid = (case["nx"], case["ny"], case["nz"])
    return synth.make_waters_device(case["n_mol"], case["edge"], grid, seed, torch.device(DEV))


def _vectors(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn((case["n_vec"], case["nz"], case["ny"], case["nx"]), generator=g,
                       dtype=torch.float64, device=DEV)


def _canonical(case, seed):
    """A localized set mixed by a random rotation (an SCF's canonical orbitals)."""
    phi, cell, grid = _orbitals(case, seed)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 1)
    n = phi.shape[0]
    q, _ = torch.linalg.qr(torch.randn((n, n), generator=g, dtype=torch.float64, device=DEV))
    return (q @ phi.reshape(n, -1)).reshape(phi.shape), cell, grid


def _boxes(case, seed):
    """Box extents (the case's own) and right-hand sides 4 pi rho: per box an
    off-centre Gaussian pair density with a linear modulation."""
    n = case["n_box"]
    ext = np.random.default_rng(n).integers(case["e_min"], case["e_max"] + 1,
                                            size=(n, 3)).astype(np.int32)
    rng = np.random.default_rng(seed)
    cen = rng.uniform(-0.4, 0.4, size=(n, 3))  # bohr
    alpha = rng.uniform(3.0, 6.0, size=n)
    lin = rng.uniform(-0.5, 0.5, size=(n, 3))
    size = torch.as_tensor(ext.prod(axis=1).astype(np.int64), device=DEV)
    box = torch.repeat_interleave(torch.arange(n, device=DEV), size)
    t = torch.arange(int(size.sum()), device=DEV) - (torch.cumsum(size, 0) - size)[box]
    e = torch.as_tensor(ext.astype(np.int64), device=DEV)[box]
    u = torch.stack([t % e[:, 0], (t // e[:, 0]) % e[:, 1], t // (e[:, 0] * e[:, 1])], 1)
    d = (u - 0.5 * (e.double() - 1)) * case["h"] - torch.as_tensor(cen, device=DEV)[box]
    rho = torch.exp(-torch.as_tensor(alpha, device=DEV)[box] * (d * d).sum(1))
    rho = rho * (1.0 + (torch.as_tensor(lin, device=DEV)[box] * d).sum(1))
    return ext, 4.0 * math.pi * rho


def _pinned(t):
    """A numpy array in page-locked memory with t's values."""
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()


def prepare(case, seed):
    if case["kind"] == "poisson":
        ext, rhs = _boxes(case, seed)
        return dict(case=case, ext=ext, rhs=rhs, x=torch.empty_like(rhs),
                    h=(case["h"],) * 3)
    s = dict(case=case, stream=torch.cuda.Stream())
    if case["kind"] == "batch":
        s["ctx"], s["phi"], s["out"] = [], [], []
        for k in range(case["n_cfg"]):
            phi, cell, grid = _orbitals(case, 64 * seed + k)
            s["ctx"].append(sea.Context(cell, grid, stream=s["stream"].cuda_stream,
                                        precision=case["precision"]))
            s["phi"].append(phi)
            s["out"].append(torch.empty_like(phi))
        torch.cuda.synchronize()
        return s
    phi, cell, grid = (_canonical if case["kind"] == "scdm" else _orbitals)(case, seed)
    s["ctx"] = sea.Context(cell, grid, stream=s["stream"].cuda_stream, precision=case["precision"])
    s["phi"], s["vxx"] = phi, torch.empty_like(phi)
    if "n_vec" in case:
        s["psi"] = _vectors(case, seed)
        s["out"] = torch.empty_like(s["psi"])
    if case.get("host"):
        for k in ("phi", "vxx", "psi", "out"):
            s[k] = _pinned(s[k])
    torch.cuda.synchronize()
    if case["kind"] in ("ace", "ace_apply"):
        s["ctx"].set_orbitals(s["phi"])
        s["ctx"].apply_vxx(s["vxx"])
        if case["kind"] == "ace_apply":
            s["ctx"].build_ace()
        torch.cuda.synchronize()
    return s


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "poisson":
        iters, _ = sea.poisson_batch(state["h"], state["ext"], state["rhs"], state["x"])
        return {"x": state["x"], "iters": iters}
    if kind == "batch":
        for c, phi in zip(state["ctx"], state["phi"]):
            c.set_orbitals(phi)
        return {"exx": sea.apply_vxx_batch(state["ctx"], state["out"]), "vxx": state["out"]}
    ctx, res = state["ctx"], {}
    if kind == "scdm":
        res["U"], res["cols"] = ctx.scdm(state["phi"])
    elif kind in ("vxx", "step"):
        ctx.set_orbitals(state["phi"])
    if kind in ("vxx", "scdm", "step"):
        res["exx"] = ctx.apply_vxx(state["vxx"])
        res["vxx"] = state["vxx"]
    if kind in ("ace", "step"):
        ctx.build_ace()
    if "psi" in state:
        ctx.apply_ace(state["psi"], state["out"])
        res["out"] = state["out"]
    return res


# --------------------------------------------------------------------------
# The same results from the definitions, in torch and numpy float64
# --------------------------------------------------------------------------
def _fd(p=P):
    f = math.factorial
    c = [0.0] + [2.0 * (-1) ** (k + 1) * f(p) ** 2 / (k * k * f(p - k) * f(p + k))
                 for k in range(1, p + 1)]
    c[0] = -2.0 * sum(c)
    return c


class _Poisson:
    """-Lap_h x = b on a box with zeros outside, by the eigenvectors of the
    three one-dimensional operators."""

    def __init__(self, h):
        self.h, self.known, self.c = h, {}, _fd()

    def axis(self, a, e):
        if (a, e) not in self.known:
            A = torch.zeros((e, e), dtype=torch.float64)
            for k, ck in enumerate(self.c):
                for i in range(e - k):
                    A[i, i + k] = A[i + k, i] = -ck / self.h[a] ** 2
            lam, V = torch.linalg.eigh(A)
            self.known[a, e] = lam.to(DEV), V.to(DEV)
        return self.known[a, e]

    def solve(self, b):
        ez, ey, ex = b.shape
        (lx, vx), (ly, vy), (lz, vz) = self.axis(0, ex), self.axis(1, ey), self.axis(2, ez)
        t = torch.einsum("zyx,xa,yb,zc->cba", b, vx, vy, vz)
        t = t / (lz[:, None, None] + ly[None, :, None] + lx[None, None, :])
        return torch.einsum("cba,xa,yb,zc->zyx", t, vx, vy, vz)


def _solid(x, y, z):
    """Regular solid harmonics R_lm, 0 <= m <= l <= LMAX, as {(l, m): values},
    normalized so that 1/|r - r'| = (1/r) sum (l-m)!(l+m)! R_lm(r') conj
    R_lm(r / r^2) over -l <= m <= l."""
    r2, R = x * x + y * y + z * z, {(0, 0): torch.ones_like(x) + 0j}
    for l in range(LMAX):
        R[l + 1, l + 1] = -torch.complex(x, y) / (2 * l + 2) * R[l, l]
        for m in range(l + 1):
            t = (2 * l + 1) * z * R[l, m]
            if m < l:
                t = t - r2 * R[l - 1, m]
            R[l + 1, m] = t / ((l + 1) ** 2 - m * m)
    return R


_LM = [(l, m) for l in range(LMAX + 1) for m in range(l + 1)]


def _multipole(Q, x, y, z):
    r2 = x * x + y * y + z * z
    R = _solid(x / r2, y / r2, z / r2)
    v = 0.0
    for q, (l, m) in zip(Q, _LM):
        w = (1 if m == 0 else 2) * math.factorial(l - m) * math.factorial(l + m)
        v = v + w * (q * torch.conj(R[l, m])).real
    return v / torch.sqrt(r2)


def _fit(m, tail):
    """Shortest cyclic interval (start, length) whose outside mass is <= tail."""
    n = len(m)
    c = np.concatenate([[0.0], np.cumsum(np.concatenate([m, m]))])
    for length in range(1, n + 1):
        out = m.sum() - (c[length:length + n] - c[:n])
        if (out <= tail).any():
            return int(np.argmax(out <= tail)), length
    return 0, n


def _meet(s1, l1, s2, l2, n):
    """(start, length, shift of the second) of the overlap on a ring of n, or None."""
    if l1 >= n and l2 >= n:
        return s1, n, 0
    if l1 >= n:
        return s2, l2, 0
    if l2 >= n:
        return s1, l1, 0
    best = None
    for k in (-1, 0, 1):
        lo, hi = max(s1, s2 + k * n), min(s1 + l1, s2 + k * n + l2)
        if hi > lo and (best is None or hi - lo > best[1]):
            best = lo, hi - lo, k
    return best


def _window(s, length, k, n, lo, ext):
    return (lo - (n - ext) // 2, n) if length >= n else (s + k * n, length)


def _double(s, length, n):
    lo, ln = (s - length // 2, 2 * length) if length % 2 == 0 else (s + (length - 1) // 2 - length,
                                                                  2 * length + 1)
    return (lo + (ln - n) // 2, n) if ln >= n else (lo, ln)


def _exchange(phi, cell, grid):
    """(V_xx phi, E_xx) of localized orbitals: boxes, pairs, the pairs' Poisson
    problems with multipole boundary values, accumulation."""
    h = [cell[a] / grid[a] for a in range(3)]
    dv, n = h[0] * h[1] * h[2], phi.shape[0]
    dens = phi * phi
    marg = [(dens.sum((1, 2)) * dv).cpu().numpy(), (dens.sum((1, 3)) * dv).cpu().numpy(),
            (dens.sum((2, 3)) * dv).cpu().numpy()]
    del dens
    box = [[_fit(marg[a][i], EPS / 3.0) for a in range(3)] for i in range(n)]
    solver, c = _Poisson(h), _fd()

    def cut(f, lo, ext):
        ix = [(torch.arange(lo[a], lo[a] + ext[a], device=DEV)) % grid[a] for a in range(3)]
        return (ix[2][:, None, None], ix[1][None, :, None], ix[0][None, None, :])

    def offsets(lo, ext, pad=0):
        """Coordinates relative to the box centre on the box and `pad` points around."""
        t = [(torch.arange(-pad, ext[a] + pad, dtype=torch.float64, device=DEV)
              - 0.5 * (ext[a] - 1)) * h[a] for a in range(3)]
        zz, yy, xx = torch.meshgrid(t[2], t[1], t[0], indexing="ij")
        return xx, yy, zz

    out, exx = torch.zeros_like(phi), 0.0
    for i in range(n):
        for j in range(i, n):
            geo = []
            for a in range(3):
                g = _meet(*box[i][a], *box[j][a], grid[a])
                if g is None:
                    break
                geo.append(g)
            if len(geo) < 3:
                continue
            lo, ext, sh = zip(*geo)
            at = cut(phi, lo, ext)
            rho = phi[i][at] * phi[j][at]
            if i != j and float(rho.abs().sum()) * dv < DELTA:
                continue
            xx, yy, zz = offsets(lo, ext)
            R = _solid(xx, yy, zz)
            Q = [(rho * R[lm]).sum() * dv for lm in _LM]
            # values at the points outside the box that the stencil reaches
            xx, yy, zz = offsets(lo, ext, P)
            inside = torch.zeros_like(xx, dtype=torch.int64)
            for a, dim in ((0, 2), (1, 1), (2, 0)):
                u = torch.arange(-P, ext[a] + P, device=DEV)
                shape = [1, 1, 1]
                shape[dim] = -1
                inside += ((u < 0) | (u >= ext[a])).long().reshape(shape)
            shell = inside == 1
            G = torch.zeros_like(xx)
            G[shell] = _multipole(Q, xx[shell], yy[shell], zz[shell])
            b = 4.0 * math.pi * rho
            core = [slice(P, P + ext[2]), slice(P, P + ext[1]), slice(P, P + ext[0])]
            for a, dim in ((0, 2), (1, 1), (2, 0)):
                for k in range(1, P + 1):
                    for s in (-k, k):
                        sl = list(core)
                        sl[dim] = slice(P + s, P + s + ext[a])
                        b = b + c[k] / h[a] ** 2 * G[tuple(sl)]
            v = solver.solve(b)
            exx -= (1.0 if i == j else 2.0) * float((rho * v).sum()) * dv
            targets = [(i, j)] if i == j else [(i, j), (j, i)]
            for o, p in targets:
                win = []
                for a in range(3):
                    if i == j:
                        w = _double(*_window(*box[i][a], 0, grid[a], lo[a], ext[a]), grid[a])
                    elif o == i:
                        w = _window(*box[j][a], sh[a], grid[a], lo[a], ext[a])
                    else:
                        w = _window(*box[i][a], 0, grid[a], lo[a], ext[a])
                    win.append(w)
                t = [torch.arange(w[0] - lo[a], w[0] - lo[a] + w[1], device=DEV)  # box indices
                     for a, w in enumerate(win)]
                tz, ty, tx = torch.meshgrid(t[2], t[1], t[0], indexing="ij")
                val = torch.zeros(tx.shape, dtype=torch.float64, device=DEV)
                hit = ((tx >= 0) & (tx < ext[0]) & (ty >= 0) & (ty < ext[1])
                       & (tz >= 0) & (tz < ext[2]))
                val[hit] = v[tz[hit], ty[hit], tx[hit]]
                far = ~hit
                val[far] = _multipole(Q, *((u[far].double() - 0.5 * (ext[a] - 1)) * h[a]
                                           for a, u in enumerate((tx, ty, tz))))
                at = cut(phi, [w[0] for w in win], [w[1] for w in win])
                out[o][at] -= val * phi[p][at]
    return out, exx


def _ace(phi, W, psi, dv):
    """V^ACE psi = W (Mbar)^-1 W^T psi dV with Mbar = sym(Phi^T W dV)."""
    n, m = phi.shape[0], psi.shape[0]
    F, W, S = phi.reshape(n, -1), W.reshape(n, -1), psi.reshape(m, -1)
    M = (F @ W.T) * dv
    H = torch.cholesky_solve((W @ S.T) * dv, torch.linalg.cholesky(-0.5 * (M + M.T)))
    return -(H.T @ W).reshape(psi.shape)


def _localize(phi):
    """(U, pivots, Phi U): greedy column pivots of Phi^T, then the symmetric
    orthogonalization of the selected columns."""
    n = phi.shape[0]
    A = phi.reshape(n, -1)
    left, Q, cols = (A * A).sum(0), torch.zeros((0, n), dtype=torch.float64, device=DEV), []
    for _ in range(n):
        p = int(torch.argmax(left))
        cols.append(p)
        q = A[:, p].clone()
        for _ in range(2):
            q = q - Q.T @ (Q @ q)
        q = q / q.norm()
        Q = torch.cat([Q, q[None]])
        left = left - (q @ A) ** 2
        left[torch.as_tensor(cols, device=DEV)] = -1.0
    B = A[:, torch.as_tensor(cols, device=DEV)]
    lam, V = torch.linalg.eigh(B.T @ B)
    U = B @ ((V / torch.sqrt(lam)[None, :]) @ V.T)
    return U, np.array(cols, dtype=np.int32), (U.T @ A).reshape(phi.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        ext, rhs = _boxes(case, seed)
        solver, x, at = _Poisson((case["h"],) * 3), [], 0
        for e in ext.astype(int):
            m = int(e.prod())
            x.append(solver.solve(rhs[at:at + m].reshape(e[2], e[1], e[0])).reshape(-1))
            at += m
        return {"x": torch.cat(x), "iters": None}
    if kind == "batch":
        got = [_exchange(*_orbitals(case, 64 * seed + k)) for k in range(case["n_cfg"])]
        return {"exx": [e for _, e in got], "vxx": [v for v, _ in got]}
    phi, cell, grid = (_canonical if kind == "scdm" else _orbitals)(case, seed)
    res = {}
    if kind == "scdm":
        res["U"], res["cols"], phi = _localize(phi)
        res["cols"] = None
    W, exx = _exchange(phi, cell, grid)
    if kind in ("vxx", "scdm", "step"):
        res["exx"], res["vxx"] = exx, W
    if "n_vec" in case:
        dv = cell[0] * cell[1] * cell[2] / (grid[0] * grid[1] * grid[2])
        res["out"] = _ace(phi, W, _vectors(case, seed), dv)
    return res
