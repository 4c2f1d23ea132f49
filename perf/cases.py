"""The work that users of this library have it do, as cases to be timed.

Kinds of cases, each through the package's public entry points:

operator   one projected tangent product y = G*(K : x) (``Context.matvec``), what a Krylov solver of a user's own
           applies once per iteration;
outer      one evaluation of the outer level (``Context.stress`` and ``Context.residual``): P(F), its average and
           b = -G*(P - P-bar);
history    a load history from the undeformed cell in one call (``Context.set_F``, ``Context.solve``,
           ``Context.save_F``);
stepwise   the same history with one call per load step, as a program that looks at every step drives it;
batch      one history on several cells of uneven sizes at once (``solve_batch``);
adjoint    the differentiable homogenized response, forward and backward (``homogenized_response``) with FP32
           leaves for the phase parameters and the voxel stiffness scale.

Microstructures, load histories and fields are synthetic and depend on the seed; they are shaped like the
particle-reinforced cells and polycrystals of the repository's own configurations.
"""
import math

import numpy as np
import torch

from paper_1901_06531_gb300 import mixfft
from paper_1901_06531_gb300.adjoint import homogenized_response

DEV = "cuda"
# every control below prescribes, for each pair of off-diagonal components, at least one of F_ij and F_ji, so that no
# rigid rotation of the cell is left free and the converged state is unique
CUBIC = (168.0, 121.0, 75.0)


def listed():
    return [
        # the solver's inner loop at the size of the headline workload: FP32 operator, 200-grain polycrystal
        {"name": "operator-fp32-128", "kind": "operator", "nx": 128, "ny": 128, "nz": 128, "fp32": True,
         "law": "svk", "phases": 200},
        # the plain FP64 operator on a particle cell of the size the paper uses
        {"name": "operator-fp64-64", "kind": "operator", "nx": 64, "ny": 64, "nz": 64, "fp32": False,
         "law": "neo", "phases": 2},
        # a box with three different sides, as cut from an image: radix 3, odd factors, no square planes
        {"name": "operator-fp32-108x72x54", "kind": "operator", "nx": 108, "ny": 72, "nz": 54, "fp32": True,
         "law": "neo", "phases": 2},
        # the largest cell the library takes (the adjoint workload's size)
        {"name": "operator-fp32-256", "kind": "operator", "nx": 256, "ny": 256, "nz": 256, "fp32": True,
         "law": "neo", "phases": 2},
        # stress and residual at outer accuracy, FP32-inner context at the headline size
        {"name": "outer-fp32-128", "kind": "outer", "nx": 128, "ny": 128, "nz": 128, "fp32": True,
         "law": "svk", "phases": 200},
        # the same in plain FP64 on a small box with three different sides
        {"name": "outer-fp64-48x36x18", "kind": "outer", "nx": 48, "ny": 36, "nz": 18, "fp32": False,
         "law": "neo", "phases": 2},
        # the headline workload: cyclic stress on a polycrystal, 20 steps in one call, quadratic starts
        {"name": "history-fp32-128-polycrystal", "kind": "history", "n": 128, "fp32": True, "law": "svk",
         "phases": 200, "control": "cyclic", "steps": 20, "amplitude": 0.2, "predictor": 2},
        # particle-reinforced cell, uniaxial stretch in mixed control, 10 steps, starts extrapolated linearly
        {"name": "history-fp32-64-spheres", "kind": "history", "n": 64, "fp32": True, "law": "neo", "radius": 4.0,
         "vf": 0.25, "contrast": 10.0, "control": "stretch", "steps": 10, "amplitude": 0.05, "predictor": 1},
        # a small plain FP64 cell with everything at its default, stress ramp
        {"name": "history-fp64-16-sphere", "kind": "history", "n": 16, "fp32": False, "law": "neo", "radius": 4.0,
         "vf": 0.06, "contrast": 10.0, "control": "stress", "steps": 5, "amplitude": 0.1, "predictor": 0},
        # a small FP32-inner cell driven one step per call (a material point of a larger simulation)
        {"name": "stepwise-fp32-32-spheres", "kind": "stepwise", "n": 32, "fp32": True, "law": "neo", "radius": 4.0,
         "vf": 0.2, "contrast": 10.0, "control": "random", "steps": 6, "amplitude": 0.02, "predictor": 2},
        # many representative cells of uneven sizes at once
        {"name": "batch-12-cells", "kind": "batch", "cells": 12, "sizes": "32,48,64,96", "steps": 3,
         "amplitude": 0.02, "predictor": 2},
        # gradient of the response with respect to phase parameters and the voxel stiffness scale
        {"name": "adjoint-fp32-64", "kind": "adjoint", "n": 64, "fp32": True, "radius": 6.0, "vf": 0.2,
         "contrast": 10.0, "steps": 1, "amplitude": 0.05, "sigma": 0.3},
    ]


def _smooth(lo, hi, even):
    """Sizes 2^a 3^b in [lo, hi]; even ones only, or with a factor 3 where odd."""
    got = [2 ** a * 3 ** b for a in range(9) for b in range(6)]
    return sorted(n for n in got if lo <= n <= hi and (n % 2 == 0 or not even))


def _spread(rng, choices):
    """One of the sorted sizes, spread over their logarithm."""
    x = math.exp(rng.uniform(math.log(choices[0]), math.log(choices[-1])))
    return min(choices, key=lambda n: (abs(math.log(n / x)), n))


def draw(rng):
    kind = rng.choice(("operator", "operator", "operator", "outer", "outer", "history", "history", "stepwise",
                       "batch", "adjoint"))
    fp32 = rng.random() < 0.7
    neo = rng.random() < 0.6
    if kind in ("operator", "outer"):
        # half of them cubes of the sizes that cells usually have, half boxes of any admissible sides
        if rng.random() < 0.5:
            nx = ny = nz = rng.choice((16, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128))
        else:
            nx = _spread(rng, _smooth(8, 192, True))
            ny = _spread(rng, [n for n in _smooth(8, 192, True) if n * nx <= 12288])
            nz = _spread(rng, _smooth(4, 128, False))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "fp32": fp32, "law": "neo" if neo else "svk",
                "phases": 2 if neo else rng.randrange(20, 300)}
    if kind == "batch":
        sizes = rng.choice(("32,48,64,96", "32,48,64", "24,36,48,72", "16,32,64"))
        return {"kind": kind, "cells": rng.randrange(3, 9), "sizes": sizes, "steps": rng.randrange(1, 4),
                "amplitude": round(rng.uniform(0.005, 0.02), 4), "predictor": rng.randrange(3)}
    radius = round(rng.uniform(3.0, 6.0), 2)
    vf, contrast = round(rng.uniform(0.1, 0.3), 3), round(rng.uniform(5.0, 30.0), 2)
    if kind == "adjoint":
        return {"kind": kind, "n": rng.choice((24, 32, 36, 48, 54, 64)), "fp32": True, "radius": radius, "vf": vf,
                "contrast": contrast, "steps": 1, "amplitude": round(rng.uniform(0.02, 0.06), 4),
                "sigma": round(rng.uniform(0.1, 0.3), 3)}
    n = rng.choice((16, 24, 32, 36, 48, 54, 64, 72, 96) if fp32 else (16, 18, 24, 32, 36))
    steps = rng.randrange(1, 7) if n <= 64 else rng.randrange(1, 4)
    case = {"kind": kind, "n": n, "fp32": fp32, "law": "neo" if neo else "svk", "steps": steps,
            "predictor": rng.randrange(3)}
    if neo:
        control = rng.choice(("stretch", "stress", "random"))
        case.update(radius=radius, vf=vf, contrast=contrast, control=control,
                    amplitude=round(rng.uniform(0.01, 0.05) * (0.4 if control == "random" else 1.0), 5))
    else:
        case.update(phases=rng.randrange(20, 200), control="cyclic", amplitude=round(rng.uniform(0.05, 0.3), 4))
    return case


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _distance2(shape, centre, reach=None):
    """Squared periodic distance of the voxel centres [z, y, x] to a point (x, y, z)."""
    d2 = 0.0
    for axis, (n, c) in enumerate(zip(shape, centre[::-1])):
        d = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5 - float(c)).abs_()
        d = torch.minimum(d, n - d).square_()
        d2 = d2 + d.reshape([-1 if k == axis else 1 for k in range(3)])
    return d2


def _spheres(shape, radius, vf, rng):
    """Phase map of equal periodic spheres placed by random sequential addition up to a volume fraction."""
    lengths = np.array(shape[::-1], dtype=np.float64)
    want = max(1, int(round(vf * lengths.prod() / (4.0 / 3.0 * math.pi * radius ** 3))))
    centres = np.empty((0, 3))
    for _ in range(200000):
        c = rng.random(3) * lengths
        d = np.abs(centres - c)
        d = np.minimum(d, lengths - d)
        if not len(centres) or (d * d).sum(1).min() >= 4.0 * radius * radius:
            centres = np.vstack([centres, c])
            if len(centres) == want:
                break
    phase = torch.zeros(shape, dtype=torch.bool, device=DEV)
    for c in centres:
        phase |= _distance2(shape, c) <= radius * radius
    return phase.to(torch.int32)


def _grains(shape, count, rng):
    """Periodic Voronoi tessellation."""
    seeds = rng.random((count, 3)) * np.array(shape[::-1], dtype=np.float64)
    best = torch.full(shape, math.inf, dtype=torch.float64, device=DEV)
    grain = torch.zeros(shape, dtype=torch.int32, device=DEV)
    for g in range(count):
        d2 = _distance2(shape, seeds[g])
        closer = d2 < best
        best = torch.where(closer, d2, best)
        grain.masked_fill_(closer, g)
    return grain


def _rotations(count, rng):
    q = rng.standard_normal((count, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).reshape(count, 3, 3)


def _material(case, shape, rng):
    """(model, parameters per phase, rotations or None, phase map on the GPU)."""
    if case.get("law", "neo") == "svk":
        count = case["phases"]
        phase = _grains(shape, count, rng)
        return mixfft.MF_SVK_CUBIC, np.tile(np.array(CUBIC), (count, 1)), _rotations(count, rng), phase
    contrast = case.get("contrast", 10.0)
    phase = _spheres(shape, case.get("radius", min(shape) / 8.0), case.get("vf", 0.2), rng)
    return mixfft.MF_NEOHOOKE, np.array([[1.0, 2.0], [contrast, 2.0 * contrast]]), None, phase


IDENTITY = np.eye(3).reshape(9)


def _control(kind, steps, amplitude, rng):
    """(mask, target) of a load history; amplitudes vary a little with the seed."""
    amplitude = amplitude * rng.uniform(0.9, 1.0)
    t = np.arange(1, steps + 1) / steps
    mask = np.ones((steps, 9), dtype=np.uint8)
    target = np.zeros((steps, 9))
    if kind == "random":
        m = (rng.random(9) < 0.5).astype(np.uint8)
        m[rng.integers(0, 3) * 4] = 0
        target = IDENTITY + amplitude * rng.uniform(-1.0, 1.0, 9) * t[:, None]
        for up, low in ((1, 3), (2, 6), (5, 7)):
            if m[up] and m[low]:
                m[up] = 0
                target[:, up] = 0.0
        target[:, m == 1] = 0.0
        return np.tile(m, (steps, 1)), target
    mask[:, [1, 2, 5]] = 0
    if kind == "stretch":
        mask[:, 0] = 0
        target[:, 0] = 1.0 + amplitude * t
    elif kind == "stress":
        target[:, 0] = amplitude * t
    else:  # a triangle wave, one period in 20 steps
        s = np.arange(1, steps + 1) / 5.0
        target[:, 0] = amplitude * (1.0 - np.abs((s + 3.0) % 4.0 - 2.0))
    return mask, target


def _deformation(shape, phase, g):
    """A deformation gradient that differs from phase to phase and fluctuates within each, det F > 0 everywhere."""
    F = 0.02 * (2.0 * torch.rand((9,) + shape, dtype=torch.float64, device=DEV, generator=g) - 1.0)
    per = 0.02 * (2.0 * torch.rand((9, int(phase.max()) + 1), dtype=torch.float64, device=DEV, generator=g) - 1.0)
    F += per[:, phase.reshape(-1).long()].reshape(F.shape)
    F[0::4] += 1.0
    return F.contiguous()


def _inputs(case, seed):
    """Everything a case's answers depend on."""
    rng = np.random.default_rng(int(seed))
    kind = case["kind"]
    if kind in ("operator", "outer"):
        shape = (case["nz"], case["ny"], case["nx"])
        g = _generator(seed)
        model, params, rot, phase = _material(case, shape, rng)
        d = {"shape": shape, "model": model, "params": params, "rot": rot, "phase": phase,
             "F": _deformation(shape, phase, g), "mask": _control("random", 1, 0.02, rng)[0][0]}
        if kind == "operator":
            d["x"] = torch.randn((9,) + shape, device=DEV, generator=g,
                                 dtype=torch.float32 if case["fp32"] else torch.float64)
        else:
            d["pbar"] = 0.05 * rng.uniform(-1.0, 1.0, 9) * (10.0 if rot is not None else 1.0)
        return d
    if kind == "batch":
        sizes = [int(n) for n in case["sizes"].split(",")]
        cells = []
        for i in range(case["cells"]):
            n = sizes[i % len(sizes)]
            one = {"radius": n / 12.0 if n >= 32 else n / 8.0, "vf": rng.uniform(0.1, 0.3),
                   "contrast": rng.uniform(5.0, 50.0)}
            model, params, rot, phase = _material(one, (n, n, n), rng)
            mask, target = _control("random", case["steps"], case["amplitude"], rng)
            cells.append({"shape": (n, n, n), "model": model, "params": params, "rot": rot, "phase": phase,
                          "mask": mask, "target": target})
        return {"cells": cells}
    shape = (case["n"],) * 3
    model, params, rot, phase = _material(case, shape, rng)
    d = {"shape": shape, "model": model, "params": params, "rot": rot, "phase": phase}
    d["mask"], d["target"] = _control("stress" if kind == "adjoint" else case["control"], case["steps"],
                                      case["amplitude"], rng)
    if kind == "adjoint":
        s = case["sigma"]
        z = torch.randn(shape, device=DEV, generator=_generator(seed), dtype=torch.float64)
        d["scale"] = torch.exp(s * z - 0.5 * s * s).float()
        d["params"] = params.astype(np.float32)
        d["weights"] = torch.from_numpy(rng.standard_normal((case["steps"], 9)).astype(np.float32))
    return d


# ------------------------------------------------------------------ the calls

def _context(d, fp32, predictor=None):
    nz, ny, nx = d["shape"]
    c = mixfft.Context(nx, ny, nz, mixfft.MF_FP32_INNER if fp32 else mixfft.MF_FP64)
    c.set_material(d["model"], d["params"], d["phase"].cpu().numpy(), rot=d["rot"])
    if predictor is not None:
        c.set_predictor(predictor)
    return c


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        s["ctxs"] = [_context(x, True, case["predictor"]) for x in d["cells"]]
        s["masks"] = np.stack([x["mask"] for x in d["cells"]])
        s["targets"] = np.stack([x["target"] for x in d["cells"]])
        s["F"] = [torch.empty((9,) + x["shape"], dtype=torch.float64, device=DEV) for x in d["cells"]]
        return s
    if kind == "adjoint":
        nz, ny, nx = d["shape"]
        s["ctx"] = mixfft.Context(nx, ny, nz, mixfft.MF_FP32_INNER)
        s["phase"] = d["phase"].cpu().numpy()
        s["params"] = torch.from_numpy(d["params"]).requires_grad_()
        s["scale"] = d["scale"].requires_grad_()
        s.update(mask=d["mask"], target=d["target"], weights=d["weights"])
        return s
    c = s["ctx"] = _context(d, case["fp32"], case.get("predictor"))
    s["mask"] = d["mask"]
    if kind in ("operator", "outer"):
        c.load_F(d["F"])
        if kind == "operator":
            c.constitutive()
            s["x"] = d["x"]
            s["y"] = torch.empty_like(d["x"])
        else:
            s["pbar"] = d["pbar"]
            s["b"] = torch.empty_like(d["F"])
    else:
        s["target"] = d["target"]
        s["F"] = torch.empty((9,) + d["shape"], dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    return s


def run(s):
    kind = s["kind"]
    if kind == "operator":
        s["ctx"].matvec(s["x"], s["y"], s["mask"])
        return s["y"]
    if kind == "outer":
        mean = s["ctx"].stress()
        mean2 = s["ctx"].residual(s["mask"], s["pbar"], s["b"])
        return {"b": s["b"], "mean": mean, "mean_residual": mean2}
    if kind == "history":
        c = s["ctx"]
        c.set_F(None)
        out = c.solve(s["mask"], s["target"])
        c.save_F(s["F"])
        return {"F": s["F"], "Fbar": out["Fbar"], "Pbar": out["Pbar"]}
    if kind == "stepwise":
        c = s["ctx"]
        c.set_F(None)
        out = [c.solve(s["mask"][k:k + 1], s["target"][k:k + 1]) for k in range(len(s["mask"]))]
        c.save_F(s["F"])
        return {"F": s["F"], "Fbar": np.concatenate([o["Fbar"] for o in out]),
                "Pbar": np.concatenate([o["Pbar"] for o in out])}
    if kind == "batch":
        for c in s["ctxs"]:
            c.set_F(None)
        out = mixfft.solve_batch(s["ctxs"], s["masks"], s["targets"])
        for c, F in zip(s["ctxs"], s["F"]):
            c.save_F(F)
        return {"F": s["F"], "Fbar": out["Fbar"], "Pbar": out["Pbar"]}
    # an FP32 adjoint solve cannot reach the FP64 default of its forcing term
    resp = homogenized_response(s["ctx"], s["phase"], s["params"], s["mask"], s["target"], scale=s["scale"],
                                adj_tol_cg=1e-30, adj_cg_rel=1e-6)
    gp, gs = torch.autograd.grad((resp * s["weights"]).sum(), [s["params"], s["scale"]])
    return {"response": resp.detach(), "dparams": gp, "dscale": gs}


# ------------------------------------------------------------------ what a pass cannot do without

def _fft_flops(n):
    return 2.5 * math.log2(n) * n


def _operator_work(n, fp32, svk):
    """One G*(K : x): x and y once, the tangent from H and the phase (FP32) or 45 packed entries (FP64)."""
    b = 4 if fp32 else 8
    return {"bytes": n * (18 * b + (40 if fp32 else 45 * 8)), "flops": 18 * _fft_flops(n) + n * (200 if svk else 170)}


def _outer_work(n, svk):
    """P(F) and the residual: F and the phase in, b out, in 64-bit accuracy."""
    return {"bytes": n * (72 + 4 + 72), "flops": 18 * _fft_flops(n) + n * 250}


def _add(total, w, times=1.0):
    for k in total:
        total[k] += times * w[k]
    return total


def _history_work(n, steps, fp32, svk, predictor):
    """Iterations of the methods the library offers: per load step a first and a confirming residual, and the CG
    iterations that the contrast asks for; per CG iteration the operator and the four vectors' traffic."""
    newton, cg = (1, 6) if svk and predictor else (3, 25) if svk else (2, 50) if predictor else (4, 80)
    if not fp32:
        cg *= 2
    b = 4 if fp32 else 8
    one = _operator_work(n, fp32, svk)
    one["bytes"] += n * 36 * b
    total = {"bytes": 72.0 * n, "flops": 0.0}
    _add(total, _outer_work(n, svk), steps * newton)
    return _add(total, one, steps * cg)


def work(case):
    kind = case["kind"]
    if kind in ("operator", "outer"):
        n, svk = case["nx"] * case["ny"] * case["nz"], case["law"] == "svk"
        return _operator_work(n, case["fp32"], svk) if kind == "operator" else _outer_work(n, svk)
    if kind == "batch":
        sizes = [int(n) for n in case["sizes"].split(",")]
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["cells"]):
            _add(total, _history_work(sizes[i % len(sizes)] ** 3, case["steps"], True, False, case["predictor"]))
        return total
    n = case["n"] ** 3
    if kind == "adjoint":
        total = _history_work(n, case["steps"], True, False, 0)
        return _add(total, _operator_work(n, True, False), 60 * case["steps"])
    return _history_work(n, case["steps"], case["fp32"], case["law"] == "svk", case["predictor"])


# ------------------------------------------------------------------ 64-bit values by plain torch

def _mm(a, b):
    """Product of 3 x 3 matrices stored as [3, 3, voxels...]."""
    return torch.stack([torch.stack([a[i, 0] * b[0, j] + a[i, 1] * b[1, j] + a[i, 2] * b[2, j] for j in range(3)])
                        for i in range(3)])


def _inverse(F):
    c = torch.stack([torch.stack([F[(i + 1) % 3, (j + 1) % 3] * F[(i + 2) % 3, (j + 2) % 3]
                                  - F[(i + 1) % 3, (j + 2) % 3] * F[(i + 2) % 3, (j + 1) % 3] for i in range(3)])
                     for j in range(3)])
    J = F[0, 0] * c[0, 0] + F[0, 1] * c[1, 0] + F[0, 2] * c[2, 0]
    return c / J, J


class _Law:
    def __init__(self, d):
        phase = d["phase"].reshape(-1).long()
        params = torch.from_numpy(np.asarray(d["params"], dtype=np.float64)).to(DEV)
        self.p = [params[phase, k].reshape(d["shape"]) for k in range(params.shape[1])]
        self.scale = None if d.get("scale") is None else d["scale"].double()
        self.R = None
        if d["rot"] is not None:
            R = torch.from_numpy(d["rot"]).to(DEV)[phase]
            self.R = R.permute(1, 2, 0).reshape((3, 3) + d["shape"]).contiguous()

    def _times(self, P):
        return P if self.scale is None else P * self.scale

    def _cubic(self, E):
        c11, c12, c44 = self.p
        Rt = self.R.transpose(0, 1)
        e = _mm(_mm(Rt, E), self.R)
        s = 2.0 * c44 * e
        tr = e[0, 0] + e[1, 1] + e[2, 2]
        for a in range(3):
            s[a, a] += c12 * tr + (c11 - c12 - 2.0 * c44) * e[a, a]
        return _mm(_mm(self.R, s), Rt)

    def at(self, F):
        """P(F) without the voxel scale; keeps what the tangent needs."""
        self.F = F
        if self.R is None:
            mu, lam = self.p
            inv, J = _inverse(F)
            self.it, self.lnJ = inv.transpose(0, 1), torch.log(J)
            return mu * (F - self.it) + lam * self.lnJ * self.it
        E = 0.5 * _mm(F.transpose(0, 1), F)
        for a in range(3):
            E[a, a] -= 0.5
        self.S = self._cubic(E)
        return _mm(F, self.S)

    def stress(self, F):
        return self._times(self.at(F))

    def tangent(self, x):
        """K : x at the F of the last stress."""
        if self.R is None:
            mu, lam = self.p
            tr = (self.it * x).sum((0, 1))
            y = mu * x + (mu - lam * self.lnJ) * _mm(_mm(self.it, x.transpose(0, 1)), self.it) + lam * tr * self.it
            return self._times(y)
        E = _mm(self.F.transpose(0, 1), x)
        return self._times(_mm(x, self.S) + _mm(self.F, self._cubic(0.5 * (E + E.transpose(0, 1)))))


class _Projector:
    def __init__(self, shape):
        nz, ny, nx = shape
        f = [torch.fft.rfftfreq(nx, dtype=torch.float64, device=DEV)[None, None, :],
             torch.fft.fftfreq(ny, dtype=torch.float64, device=DEV)[None, :, None],
             torch.fft.fftfreq(nz, dtype=torch.float64, device=DEV)[:, None, None]]
        self.xi, self.shape = f, shape
        xi2 = f[0] ** 2 + f[1] ** 2 + f[2] ** 2
        xi2[0, 0, 0] = 1.0
        keep = torch.ones_like(xi2)
        for k, n in ((0, nz), (1, ny), (2, nx)):
            if n % 2 == 0:
                keep.select(k, n // 2).zero_()
        self.w = keep / xi2

    def __call__(self, A, mask, pbar=None):
        """G*(A - pbar) for a field [3, 3, z, y, x]."""
        N = A[0, 0].numel()
        out = torch.empty_like(A)
        for i in range(3):
            a = torch.fft.rfftn(A[i], dim=(1, 2, 3))
            q = (a[0] * self.xi[0] + a[1] * self.xi[1] + a[2] * self.xi[2]) * self.w
            mean = a[:, 0, 0, 0].clone()
            for j in range(3):
                a[j] = q * self.xi[j]
                m = float(mask[3 * i + j])
                a[j, 0, 0, 0] = m * (mean[j] - (0.0 if pbar is None else float(pbar[3 * i + j]) * N))
            out[i] = torch.fft.irfftn(a, s=self.shape, dim=(1, 2, 3))
        return out


def _cg(apply, b, rel, floor, most=2000):
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), (r * r).sum()
    stop = max(rel * rel * float(rr), floor * floor * b[0, 0].numel())
    for _ in range(most):
        if float(rr) <= stop:
            break
        t = apply(p)
        alpha = rr / (p * t).sum()
        x += alpha * p
        r -= alpha * t
        new = (r * r).sum()
        p = r + (new / rr) * p
        rr = new
    return x


def _mean(A):
    return A.mean((2, 3, 4)).reshape(9)


def _solve(d):
    """Converged F, averages per step, and the law at the last state."""
    law, G = _Law(d), _Projector(d["shape"])
    F = torch.eye(3, dtype=torch.float64, device=DEV)[:, :, None, None, None].expand((3, 3) + d["shape"]).clone()
    Fbar, Pbar, last = [], [], None
    for mask, target in zip(d["mask"], d["target"]):
        before = F.clone()
        if last is not None:
            F = 2.0 * F - last
        last = before
        mean, free = _mean(F), torch.from_numpy(mask == 0).to(DEV)
        want = torch.from_numpy(target).to(DEV)
        F = F + torch.where(free, want - mean, torch.zeros_like(mean)).reshape(3, 3, 1, 1, 1)
        for _ in range(12):
            P = law.stress(F)
            dF = _cg(lambda x: G(law.tangent(x), mask), -G(P, mask, target), 1e-5, 1e-15)
            F = F + dF
            if float((dF * dF).sum((0, 1)).max()) < 1e-22:
                break
        Fbar.append(_mean(F).cpu().numpy())
        Pbar.append(_mean(law.stress(F)).cpu().numpy())
    return {"F": F.reshape((9,) + d["shape"]), "Fbar": np.stack(Fbar), "Pbar": np.stack(Pbar)}, law, G


def exact(case, seed):
    kind = case["kind"]
    d = _inputs(case, seed)
    if kind == "operator":
        law, G = _Law(d), _Projector(d["shape"])
        law.stress(d["F"].reshape((3, 3) + d["shape"]))
        y = G(law.tangent(d["x"].double().reshape((3, 3) + d["shape"])), d["mask"])
        return y.reshape((9,) + d["shape"])
    if kind == "outer":
        P = _Law(d).stress(d["F"].reshape((3, 3) + d["shape"]))
        b = -_Projector(d["shape"])(P, d["mask"], d["pbar"])
        mean = _mean(P).cpu().numpy()
        return {"b": b.reshape((9,) + d["shape"]), "mean": mean, "mean_residual": mean}
    if kind == "batch":
        each = [_solve(x)[0] for x in d["cells"]]
        return {"F": [e["F"] for e in each], "Fbar": np.stack([e["Fbar"] for e in each]),
                "Pbar": np.stack([e["Pbar"] for e in each])}
    state, law, G = _solve(d)
    if kind != "adjoint":
        return state
    # adjoint of the free response of the (single) step at its converged state
    mask, N = d["mask"][-1], d["phase"].numel()
    g = d["weights"].double().numpy()[-1]
    response = np.where(mask == 1, state["Fbar"], state["Pbar"])
    field = lambda w: torch.from_numpy(w).to(DEV).reshape(3, 3, 1, 1, 1)  # noqa: E731
    wF, wP = field(np.where(mask == 1, g, 0.0)), field(np.where(mask == 1, 0.0, g))
    F = state["F"].reshape((3, 3) + d["shape"])
    P = law.at(F)
    rhs = G(wF + law.tangent(wP.expand_as(F)), mask)
    D = wP - _cg(lambda x: G(law.tangent(x), mask), rhs, 1e-11, 1e-15, 5000)
    dmu = (D * (F - law.it)).sum((0, 1)) * law.scale / N
    dlam = (D * law.it).sum((0, 1)) * law.lnJ * law.scale / N
    phase = d["phase"].reshape(-1).long()
    gp = torch.zeros((len(d["params"]), 2), dtype=torch.float64, device=DEV)
    gp[:, 0].index_add_(0, phase, dmu.reshape(-1))
    gp[:, 1].index_add_(0, phase, dlam.reshape(-1))
    return {"response": response, "dparams": gp, "dscale": (D * P).sum((0, 1)) / N}
