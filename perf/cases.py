"""Timed cases of the library: what a micromechanics program has it do.

A program holds one handle per periodic cell (or per batch of cells, or a
group of batches), loads it increment by increment and reads homogenised
stresses and tangents back (`step`, `group`, `fs_step`), or it runs its own
Krylov or fixed-point scheme on device tensors and calls the operators
(`project`, `matvec`, `constitutive`, `fs_project`, `fs_matvec`).
"""
import math

import numpy as np
import torch

from paper_1601_05970_gb300 import fftg
from paper_1601_05970_gb300 import inputs as I

GRIDS = (9, 15, 25, 27, 45, 75, 81, 125, 135, 225, 243)
GROUP_GRIDS = (15, 27, 45, 75)  # the grid sizes of the batched workload
IJ = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))  # components 11, 22, 33, 23, 13, 12
PRECISION = {"fp32": "mixed", "dd": "mixed", "mixed": "mixed", "fp64": "fp64"}


def listed():
    return [
        # one Gauss point of an FE^2 computation at the smallest grid of the
        # workloads: two increments and the 6x6 tangent, all latency
        dict(name="step-15", kind="step", N=15, precision="mixed", cells=1, increments=2, tangent=True),
        # a batch of equal cells that take their increments together
        dict(name="batch-27", kind="step", N=27, precision="mixed", cells=32, increments=2, tangent=False),
        # the plain FP64 path on an ordinary cell, with the tangent
        dict(name="step-45-fp64", kind="step", N=45, precision="fp64", cells=1, increments=1, tangent=True),
        # cells of four grid sizes, one graph launch per increment
        dict(name="group-15-75", kind="group", N=75, precision="mixed", cells=16, increments=2, tangent=False),
        # an ordinary large cell: increments and tangent, as in FE^2
        dict(name="step-135", kind="step", N=135, precision="mixed", cells=1, increments=2, tangent=True),
        # the benchmark's grid: increments of a load path
        dict(name="step-243", kind="step", N=243, precision="mixed", cells=1, increments=2, tangent=False),
        # the projection of a caller's field: large in FP32 and with double-float
        # transforms, and small, where the launches count
        dict(name="project-243", kind="project", N=243, precision="fp32"),
        dict(name="project-135-dd", kind="project", N=135, precision="dd"),
        dict(name="project-45", kind="project", N=45, precision="fp32"),
        # one matvec of a caller's own Krylov solver
        dict(name="matvec-225", kind="matvec", N=225, precision="fp32"),
        # the stress update alone, on a mostly plastic cell
        dict(name="constitutive-243", kind="constitutive", N=243, precision="mixed", exponent=1.0),
        # finite strain: a load cycle, an increment of a stretch-shear path and back
        dict(name="fs-step-125", kind="fs_step", N=125, precision="mixed", increments=1),
    ]


def draw(rng):
    kind = rng.choice(("step", "step", "group", "project", "project", "matvec", "matvec", "constitutive",
                       "fs_step", "fs_project", "fs_matvec"))
    if kind == "step":
        precision = rng.choice(("mixed", "mixed", "mixed", "fp64"))
        N = rng.choice([n for n in GRIDS if n <= (135 if precision == "mixed" else 45)])
        most = (1 << 21) if precision == "mixed" else (1 << 16)
        cells = max(1, min(64, int(most / N ** 3 * rng.random())))
        return dict(kind=kind, N=N, precision=precision, cells=cells, increments=rng.randint(1, 2),
                    tangent=rng.random() < 0.5)
    if kind == "group":
        return dict(kind=kind, N=75, precision="mixed", cells=rng.randint(1, 15), increments=rng.randint(1, 2),
                    tangent=False)
    if kind == "fs_step":
        return dict(kind=kind, N=rng.choice([n for n in GRIDS if n <= 81]), precision="mixed",
                    increments=rng.randint(1, 2))
    N = rng.choice(GRIDS)
    if kind == "constitutive":
        return dict(kind=kind, N=N, precision=rng.choice(("mixed", "fp64")), exponent=rng.choice((1.0, 1.0, 0.5)))
    if kind in ("project", "fs_project"):
        return dict(kind=kind, N=N, precision=rng.choice(("fp32", "dd", "fp64")))
    return dict(kind=kind, N=N, precision=rng.choice(("fp32", "fp32", "fp64")))


# ------------------------------------------------------------------- inputs
def _rng(seed, *more):
    return np.random.default_rng([int(seed), *more])


def _field(seed, ncomp, N, scale, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(ncomp * N ** 3, dtype=dtype, device="cuda", generator=g) * scale


def _spheres(N, seed, fraction=0.25):
    """Periodic random hard spheres in a soft matrix, about `fraction` of them
    hard (radii 3-8 voxels, as in the workloads; smaller in small cells)."""
    r_hi = min(8.0, N / 5)
    r_lo = 3.0 / 8.0 * r_hi
    mean = math.pi / 3.0 * (r_hi ** 4 - r_lo ** 4) / (r_hi - r_lo)
    n = max(1, round(-math.log(1.0 - fraction) * N ** 3 / mean))
    rng = _rng(seed, 11)
    centre = torch.tensor(rng.uniform(0, N, (n, 3)), device="cuda")
    radius = torch.tensor(rng.uniform(r_lo, r_hi, n), device="cuda")
    span = torch.arange(-math.floor(r_hi), math.ceil(r_hi) + 1, device="cuda")
    base = centre.floor().long()
    index = base[:, :, None] + span                      # [n, 3, span]
    d2 = (index - centre[:, :, None]) ** 2
    index = index % N
    inside = (d2[:, 0, :, None, None] + d2[:, 1, None, :, None] + d2[:, 2, None, None, :]
              <= radius[:, None, None, None] ** 2)
    flat = (index[:, 0, :, None, None] * N + index[:, 1, None, :, None]) * N + index[:, 2, None, None, :]
    phase = torch.zeros(N ** 3, dtype=torch.uint8, device="cuda")
    phase[flat[inside]] = 1
    return phase.reshape(N, N, N).cpu().numpy()


def _direction(seed, *more):
    """A random isochoric direction of unit Frobenius norm (six components)."""
    v = _rng(seed, 12, *more).standard_normal(6)
    v[:3] -= v[:3].mean()
    return v / I.frobenius6(v)


def _path(case, seed, *more):
    """A proportional path: to just below the soft phase's yield strain, then
    increments of norm 1e-3 through it (the batched workload's increment)."""
    return np.outer([2.9e-3] + [1e-3] * case["increments"], _direction(seed, *more))


def _materials(case):
    n = case.get("exponent", 1.0)
    return tuple(I.Phase(m.K, m.G, m.sigma_y, m.H, n) for m in I.TWO_PHASE)


def _fs_path(case, seed):
    """A stretch-shear path like the finite-strain workload's, turned at random:
    one increment and then the case's."""
    q, _ = np.linalg.qr(_rng(seed, 13).standard_normal((3, 3)))
    return [q @ dF @ q.T for dF in I.stretch_shear_path(1 + case["increments"])]


TOL_NEWTON, TOL_CG = 1e-8, 1e-8


def prepare(case, seed):
    kind, N = case["kind"], case["N"]
    s = dict(case=case, seed=seed)
    if kind == "step":
        cells = case["cells"]
        phase = np.stack([_spheres(N, seed + 1000 * c) for c in range(cells)])
        s["cell"] = fftg.Cell(N, phase if cells > 1 else phase[0], I.TWO_PHASE, precision=case["precision"],
                              nrhs_tangent=6 if case["tangent"] else 0)
        s["path"] = np.stack([_path(case, seed, c) for c in range(cells)], axis=1)  # [increments, cells, 6]
    elif kind == "group":
        s["cells"] = [fftg.Cell(n, np.stack([_spheres(n, seed + 1000 * c + n) for c in range(case["cells"])]),
                                I.TWO_PHASE, precision=case["precision"], nrhs_tangent=0) for n in GROUP_GRIDS]
        s["group"] = fftg.Group(s["cells"])
        s["path"] = [np.stack([_path(case, seed, c, n) for c in range(case["cells"])], axis=1) for n in GROUP_GRIDS]
    elif kind == "fs_step":
        s["cell"] = fftg.FsCell(N, _spheres(N, seed), I.SVK_TWO_PHASE, precision=case["precision"])
        first, *rest = _fs_path(case, seed)
        s["cell"].step(first, TOL_NEWTON, TOL_CG)
        s["path"] = rest + [-dF for dF in reversed(rest)]  # elastic: the cycle ends where it began
    elif kind in ("fs_project", "fs_matvec"):
        s["cell"] = fftg.FsCell(N, _spheres(N, seed), I.SVK_TWO_PHASE, precision=PRECISION[case["precision"]])
        if kind == "fs_matvec":
            state = _fs_state(case, seed)
            s["cell"].set_state(state)
        s["in"] = _operand(case, seed)
    else:
        s["cell"] = fftg.Cell(N, _spheres(N, seed), _materials(case), precision=PRECISION[case["precision"]],
                              nrhs_tangent=0)
        if kind != "project":
            s["eps"], s["dE"] = _strain(case, seed)
            s["sigma"] = torch.empty(6 * N ** 3, dtype=torch.float64, device="cuda")
        if kind == "matvec":
            s["cell"].constitutive(s["dE"], s["eps"])
        if kind != "constitutive":
            s["in"] = _operand(case, seed)
    return s


def _operand(case, seed):
    """Stresses to project, or a search direction (both of the path's sizes)."""
    ncomp = 9 if case["kind"].startswith("fs_") else 6
    dtype = torch.float32 if case["precision"] == "fp32" else torch.float64
    return _field(seed + 1, ncomp, case["N"], 3e-3, dtype)


def _strain(case, seed):
    """A fluctuating strain about a macroscopic one past the soft yield strain."""
    return _field(seed + 2, 6, case["N"], 4e-4), 4.5e-3 * _direction(seed)


def _fs_state(case, seed):
    F = np.eye(3) + I.stretch_shear_path(1)[0]
    Fs = _field(seed + 3, 9, case["N"], 5e-3).cpu().numpy()
    return np.concatenate([F.reshape(-1), Fs])


# ---------------------------------------------------------------- the calls
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        return _run_step(s, case)
    if kind == "group":
        for cell in s["cells"]:
            for b in range(cell.ncells):
                cell.select(b)
                cell.reset_state()
        out = []
        for k in range(case["increments"] + 1):
            out.append([sig for sig, _, _, _ in s["group"].step([p[k] for p in s["path"]], TOL_NEWTON, TOL_CG)])
        return {str(n): _hand_on(case, np.stack([o[i] for o in out])) for i, n in enumerate(GROUP_GRIDS)}
    if kind == "fs_step":
        return [_hand_on(case, s["cell"].step(dF, TOL_NEWTON, TOL_CG)[0]) for dF in s["path"]]
    if kind in ("project", "fs_project"):
        return s["cell"].project(s["in"], dd=case["precision"] == "dd")
    if kind in ("matvec", "fs_matvec"):
        q, pq = s["cell"].matvec(s["in"])
        # an FP32 handle sums <p, q> in FP32
        return q, (np.float32(pq) if case["precision"] == "fp32" else pq)
    return s["cell"].constitutive(s["dE"], s["eps"], s["sigma"])


def _run_step(s, case):
    cell, path = s["cell"], s["path"]
    for b in range(cell.ncells):
        cell.select(b)
        cell.reset_state()
    sig = []
    for dE in path:
        if cell.ncells == 1:
            sig.append(cell.step(dE[0], TOL_NEWTON, TOL_CG)[0][None])
        else:
            sig.append(cell.batch_step(dE, TOL_NEWTON, TOL_CG)[0])
    out = {"sigma": _hand_on(case, np.stack(sig))}
    cell.select(0)
    if case["tangent"]:
        out["tangent"] = _hand_on(case, cell.tangent(TOL_CG)[0])
    out["stress"] = _hand_on(case, cell.constitutive())  # the local stresses of the (first) cell
    return out


def _hand_on(case, values):
    """A program that has its systems solved in FP32 goes on in FP32."""
    if case["precision"] != "mixed":
        return values
    return values.float() if isinstance(values, torch.Tensor) else values.astype(np.float32)


# ------------------------------------------------------------------- work
def work(case):
    kind, N = case["kind"], case["N"]
    V = float(N ** 3)
    ncomp = 9 if kind.startswith("fs_") else 6
    # forward and inverse real transforms of every component: 2.5 log2(V)
    # flops a value and direction, as is usual for FFTs
    fft = 2 * ncomp * 2.5 * math.log2(V)
    el = 4 if case["precision"] in ("fp32", "mixed") else 8
    if kind in ("project", "fs_project"):
        return dict(bytes=V * 2 * ncomp * el, flops=V * (fft + 30))
    if kind == "matvec":
        return dict(bytes=V * (2 * 6 + 7) * el, flops=V * (fft + 70))
    if kind == "fs_matvec":
        return dict(bytes=V * (2 * 9 * el + 9 * 8 + 1), flops=V * (fft + 250))
    if kind == "constitutive":
        # strain, history and phase in; stress and compact tangent out
        return dict(bytes=V * (13 * 8 + 1 + 48 + 7 * el), flops=V * 120)
    # A solve of one increment: about 4 Newton and 80 inner iterations in a
    # plastic increment and 45 for a column of the tangent; an inner iteration
    # cannot do without the three vectors read and written and the tangent
    # read, a Newton iteration not without strain and history in, stress out.
    inc = case["increments"]
    cg, newton = 80.0 * inc, 4.0 * inc + 1
    if case.get("tangent"):
        cg += 6 * 45.0 / max(1, case.get("cells", 1))
    if kind == "fs_step":
        cg, newton = 60.0 * inc, 6.0 * inc
    vox = V * case.get("cells", 1)
    if kind == "group":
        vox = float(sum(n ** 3 for n in GROUP_GRIDS)) * case["cells"]
    it_bytes = (6 * ncomp + (7 if ncomp == 6 else 9)) * el
    return dict(bytes=vox * (cg * it_bytes + newton * (2 * ncomp + 7) * 8),
                flops=vox * (cg * (fft + 100) + newton * (fft + 250)))


# ----------------------------------------- the same in 64 bits, in plain torch
def exact(case, seed):
    kind, N = case["kind"], case["N"]
    if kind in ("project", "fs_project"):
        x = _operand(case, seed).double().view(-1, N, N, N)
        return _project(x).reshape(-1)
    if kind in ("constitutive", "matvec"):
        mats, phase = _materials(case), torch.tensor(_spheres(N, seed), device="cuda")
        eps, dE = _strain(case, seed)
        law = _J2(mats, phase)
        sig = law.update(eps.view(6, N, N, N) + _col(dE), torch.zeros(7, 1, 1, 1, dtype=torch.float64, device="cuda"))
        if kind == "constitutive":
            return sig.reshape(-1)
        p = _operand(case, seed).double().view(6, N, N, N)
        q = _project(law.tangent(p))
        return q.reshape(-1), _dot(p, q)
    if kind == "fs_matvec":
        state = _fs_state(case, seed)
        law = _Svk(torch.tensor(_spheres(N, seed), device="cuda"))
        F = torch.tensor(state[9:], device="cuda").view(9, N, N, N) + _col(state[:9])
        law.update(F)
        p = _operand(case, seed).double().view(9, N, N, N)
        q = _project(law.tangent(p))
        return q.reshape(-1), _dot(p, q)
    if N ** 3 * case.get("cells", 1) > 82 ** 3:
        return None  # an FP64 solve of these takes too long
    if kind == "fs_step":
        law = _Svk(torch.tensor(_spheres(N, seed), device="cuda"))
        Fs, Fbar, out = torch.zeros(9, N, N, N, dtype=torch.float64, device="cuda"), np.eye(3), []
        for dF in _fs_path(case, seed):
            Fbar = Fbar + dF
            Fs, P = _newton(law.update, law.tangent, Fs, _col(Fbar.reshape(-1)), np.linalg.norm(Fbar - np.eye(3)))
            out.append(P.mean(dim=(1, 2, 3)).cpu().numpy().reshape(3, 3))
        return out[1:] + out[-2::-1]
    if kind == "group" or N ** 3 * case.get("cells", 1) > 46 ** 3:
        return None
    sigma, tangent = [], None
    for c in range(case["cells"]):
        law = _J2(I.TWO_PHASE, torch.tensor(_spheres(N, seed + 1000 * c), device="cuda"))
        hist = torch.zeros(7, N, N, N, dtype=torch.float64, device="cuda")
        eps, E, out = torch.zeros(6, N, N, N, dtype=torch.float64, device="cuda"), np.zeros(6), []
        for dE in _path(case, seed, c):
            E = E + dE
            eps, sig = _newton(lambda e: law.update(e, hist), law.tangent, eps, _col(E), I.frobenius6(E))
            hist = law.history
            out.append(sig.mean(dim=(1, 2, 3)).cpu().numpy())
        sigma.append(np.stack(out))
        if c == 0:
            stress = sig.reshape(-1)
        if c == 0 and case["tangent"]:
            tangent = np.zeros((6, 6))
            for j in range(6):
                unit = _col(np.eye(6)[j]).expand_as(eps)
                x = _solve(law.tangent, -_project(law.tangent(unit)))
                tangent[:, j] = law.tangent(unit + x).mean(dim=(1, 2, 3)).cpu().numpy()
    out = {"sigma": np.stack(sigma, axis=1), "stress": stress}
    if case["tangent"]:
        out["tangent"] = tangent
    return out


def _col(v):
    return torch.tensor(np.asarray(v, dtype=np.float64), device="cuda").view(-1, 1, 1, 1)


def _weights(ncomp):
    return [1.0] * 9 if ncomp == 9 else [1.0, 1.0, 1.0, 2.0, 2.0, 2.0]


def _dot(a, b):
    return float(sum(w * (x * y).sum() for w, x, y in zip(_weights(a.shape[0]), a, b)))


def _project(x):
    """The projection of a field on the compatible ones, component by component."""
    N = x.shape[-1]
    f = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device=x.device)
    k = [f[:, None, None], f[None, :, None], f[None, None, : (N + 1) // 2].abs()]
    q = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    inv = torch.where(q > 0, 1.0 / q.clamp(min=1.0).sqrt(), torch.zeros_like(q))
    n = [c * inv for c in k]
    h = [torch.fft.rfftn(c) for c in x]
    back = lambda c: torch.fft.irfftn(c, s=(N, N, N))  # noqa: E731
    if len(h) == 9:
        t = [sum(n[j] * h[3 * i + j] for j in range(3)) for i in range(3)]
        return torch.stack([back(t[i] * n[j]) for i in range(3) for j in range(3)])
    full = {ij: h[c] for c, ij in enumerate(IJ)}
    full.update({(j, i): v for (i, j), v in list(full.items())})
    t = [sum(full[i, j] * n[j] for j in range(3)) for i in range(3)]
    nt = sum(n[i] * t[i] for i in range(3))
    return torch.stack([back(n[i] * t[j] + n[j] * t[i] - nt * n[i] * n[j]) for i, j in IJ])


class _J2:
    """J2 plasticity with hardening sigma_0 + H e^n: radial return and its tangent."""

    def __init__(self, mats, phase):
        pick = lambda name: torch.tensor([getattr(m, name) for m in mats], dtype=torch.float64,  # noqa: E731
                                         device="cuda")[phase.long()]
        self.K, self.G, self.sy, self.H = pick("K"), pick("G"), pick("sigma_y"), pick("H")
        self.n = float(mats[0].n)

    def update(self, strain, history):
        e = strain - history[:6]
        eb = history[6]
        tr = e[0] + e[1] + e[2]
        s = 2.0 * self.G * e
        s[:3] -= 2.0 * self.G * tr / 3.0
        seq = torch.sqrt(1.5 * (s[0] ** 2 + s[1] ** 2 + s[2] ** 2 + 2.0 * (s[3] ** 2 + s[4] ** 2 + s[5] ** 2)))
        phi = seq - (self.sy + self.H * eb ** self.n)
        plastic = phi > 1e-12 * self.sy
        if self.n == 1.0:
            dg = phi / (3.0 * self.G + self.H)
        else:  # the left side decreases: bisection on [0, phi / 3G]
            lo, hi = torch.zeros_like(phi), (phi / (3.0 * self.G)).clamp(min=0.0)
            for _ in range(80):
                dg = 0.5 * (lo + hi)
                over = seq - 3.0 * self.G * dg - self.sy - self.H * (eb + dg) ** self.n > 0
                lo, hi = torch.where(over, dg, lo), torch.where(over, hi, dg)
        dg = torch.where(plastic, dg, torch.zeros_like(dg))
        safe = torch.where(plastic, seq, torch.ones_like(seq))
        N = torch.where(plastic, 1.5 * s / safe, torch.zeros_like(s))
        slope = self.n * self.H * torch.where(plastic, eb + dg, torch.ones_like(dg)) ** (self.n - 1.0)
        ratio = dg / safe
        self.g2 = 2.0 * self.G - 6.0 * self.G ** 2 * ratio
        self.b = torch.where(plastic, 4.0 * self.G ** 2 * (ratio - 1.0 / (3.0 * self.G + slope)), torch.zeros_like(dg))
        self.N = N
        self.history = torch.cat([history[:6] + dg * N, (eb + dg)[None].expand(1, *dg.shape)])
        sig = s - 2.0 * self.G * dg * N
        sig[:3] += self.K * tr
        return sig

    def tangent(self, p):
        tr = p[0] + p[1] + p[2]
        out = self.g2 * p
        out[:3] += (self.K - self.g2 / 3.0) * tr
        Np = sum(w * a * b for w, a, b in zip(_weights(6), self.N, p))
        return out + self.b * Np * self.N


class _Svk:
    """St. Venant-Kirchhoff: P = F S and its derivative."""

    def __init__(self, phase):
        self.lam, self.mu = (torch.tensor([getattr(m, a) for m in I.SVK_TWO_PHASE], dtype=torch.float64,
                                          device="cuda")[phase.long()] for a in ("lam", "mu"))

    def _second(self, E2):
        """S for twice the strain E, as nine fields."""
        tr = E2[0] + E2[4] + E2[8]
        S = self.mu * E2
        for c in (0, 4, 8):
            S[c] += 0.5 * self.lam * tr
        return S

    def update(self, F):
        self.F = F
        H = F - _col(np.eye(3).reshape(-1))
        self.S = self._second(_t(H) + H + _mm(_t(H), H))
        return _mm(F, self.S)

    def tangent(self, d):
        M = _mm(_t(self.F), d)
        return _mm(d, self.S) + _mm(self.F, self._second(M + _t(M)))


def _t(a):
    return a[[0, 3, 6, 1, 4, 7, 2, 5, 8]]


def _mm(a, b):
    return torch.stack([sum(a[3 * i + k] * b[3 * k + j] for k in range(3)) for i in range(3) for j in range(3)])


def _newton(update, tangent, x, mean, norm):
    """Newton with conjugate gradients, to rounding; the fluctuation and the stress."""
    size = norm * math.sqrt(x[0].numel())
    for _ in range(30):
        sig = update(x + mean)
        d = _solve(tangent, -_project(sig), floor=1e-15 * math.sqrt(_dot(sig, sig)))
        x = x + d
        if math.sqrt(_dot(d, d)) <= 1e-12 * size:
            break
    return x, update(x + mean)


def _solve(tangent, r, floor=0.0):
    x, p = torch.zeros_like(r), r.clone()
    rr = _dot(r, r)
    stop = max(1e-24 * rr, floor ** 2)
    for _ in range(3000):
        if rr <= stop:
            break
        q = _project(tangent(p))
        a = rr / _dot(p, q)
        x += a * p
        r = r - a * q
        new = _dot(r, r)
        p = r + (new / rr) * p
        rr = new
    return x
