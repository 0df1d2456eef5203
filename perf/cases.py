"""The work that a user of this package has it do, as cases that can be timed.

The inputs are the package's own synthetic prostate phantoms (phantom.PhantomSpec): the tiny
5 mm one, the literal paper-shaped 2.5 mm grid, its mixed-resolution form, the 61M-nonzero
form of it that bench.py solves, and the jittered family of the batched workload. The geometry
of a case is fixed by its sizes; every seed scales each beamlet's column of D by its own output
factor (0.9 to 1.1) and draws the fluence, so each seed has other values of D and x.

Kinds of case:
  dose    plan_dose at a caller's fluence: the smallest call, made on every edit of a plan
  eval    plan_eval: objective, dose and gradient at a caller's fluence (a forward and a
          transposed pass), what a caller with an optimiser of its own asks for
  csr     imrt_eval_csr_noalloc: dose and objective straight from a device CSR
  solve   plan_solve of a resident plan (up to 200 Armijo iterations), then its x and its dose
  batch   plan_solve_batch of uneven plans in the persistent team solver, then every x
  replan  one request of the re-planning stream: plan_update from a new host CSR, a solve from
          the patient's last fluence, and x and the dose back on the host
  new     a new patient: plan_create from a pinned host CSR with the step-size rule, one
          evaluation at the first fluence, plan_destroy
"""
import ctypes
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_0908_4421_gb300 import Options, Plan, phantom, solve_batch
from paper_0908_4421_gb300 import _lib as L

PRECISIONS = {"fp32": (L.FP32, 4), "fp16": (L.FP16, 2), "bf16": (L.BF16, 2), "fp8": (L.FP8E4M3, 1)}
MAX_ITER = 200  # the package's default iteration cap, which these cases run into
TINY = dict(spacing=5.0, depth_mm=150.0, beams=5, beamlet_mm=5.0, sigma_mm=2.5, cutoff=1e-3, ptv=1.0, mixed=False)
PAPER = dict(spacing=2.5, depth_mm=240.0, beams=9, beamlet_mm=5.0, sigma_mm=2.5, cutoff=1e-3, ptv=1.0, mixed=False)
MIXED = dict(PAPER, mixed=True)
LARGE = dict(PAPER, beamlet_mm=2.5, sigma_mm=6.0, cutoff=1e-4)


def listed():
    return [
        # a planner drags one beamlet of a small plan: latency only
        dict(name="dose-tiny-fp32", kind="dose", precision="fp32", **TINY),
        # the objective and gradient of an ordinary plan for a caller's own optimiser; D fits L2
        dict(name="eval-paper-fp32", kind="eval", precision="fp32", **PAPER),
        # the same of the largest plan, in the two storage forms that are used in earnest
        dict(name="eval-large-fp32", kind="eval", precision="fp32", **LARGE),
        dict(name="eval-large-fp16", kind="eval", precision="fp16", **LARGE),
        # a delivery controller checks a dose with no device memory of its own to allocate:
        # the mixed-resolution plan, and the largest one
        dict(name="csr-mixed", kind="csr", **MIXED),
        dict(name="csr-large", kind="csr", **LARGE),
        # time-to-plan of a small plan (launches and latency count), and of the largest one:
        # bench.py's headline and its reduced-precision form with the FP32 polish
        dict(name="solve-tiny-fp32", kind="solve", precision="fp32", k_trials=1, **TINY),
        dict(name="solve-large-fp32", kind="solve", precision="fp32", k_trials=1, **LARGE),
        dict(name="solve-large-fp16", kind="solve", precision="fp16", k_trials=1, **LARGE),
        # the batched workload: 64 uneven plans, several Armijo steps a pass, one launch
        dict(name="batch-64-fp16", kind="batch", precision="fp16", plans=64),
        # one re-planning request as the server handles it
        dict(name="replan-tiny-fp16", kind="replan", precision="fp16", k_trials=1, **TINY),
        # admission of a new patient with the largest D in the mixed-precision form
        dict(name="new-large-fp16", kind="new", precision="fp16", **LARGE),
    ]


def draw(rng):
    kind = rng.choice(["dose", "eval", "eval", "csr", "solve", "solve", "batch", "replan", "new"])
    if kind == "batch":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp16", "bf16"]), plans=round(4 * 16 ** rng.random()))
    # nonzeros over the range's logarithm, shared out between voxel spacing and beamlet pitch
    top = 2e6 if kind == "replan" else 5e7
    nnz = 1e5 * (top / 1e5) ** rng.random()
    c = dict(TINY, depth_mm=rng.choice([150.0, 240.0]), beams=rng.choice([5, 7, 9]),
             sigma_mm=round(rng.uniform(2.5, 6.0), 1), cutoff=round(10 ** -rng.uniform(3, 4), 6),
             ptv=round(rng.uniform(0.8, 1.0), 2), mixed=rng.random() < 0.1)
    per = 126720 * (c["beams"] / 5) * c["sigma_mm"] ** 2 * math.log(1 / c["cutoff"]) / (2.5 ** 2 * math.log(1e3))
    if per > nnz:  # a wide kernel on few voxels would miss the target: take the narrow one
        c["sigma_mm"], c["cutoff"] = 2.5, 1e-3
        per = 126720 * c["beams"] / 5
    share = rng.uniform(0.4, 0.9)
    c["spacing"] = round(min(6.0, max(2.5, 5.0 * (per / nnz) ** (share / 3))), 2)
    left = nnz / (per * (5.0 / c["spacing"]) ** 3)
    c["beamlet_mm"] = round(min(10.0, max(2.5, 5.0 / math.sqrt(left))), 2)
    if kind != "csr":
        c["precision"] = rng.choice(["fp32", "fp32", "fp16", "fp16", "bf16"] + (["fp8"] if kind == "eval" else []))
    if kind in ("solve", "replan"):
        c["k_trials"] = rng.choice([1, 1, 1, 2, 4])
    return dict(kind=kind, **c)


# --- inputs ----------------------------------------------------------------------------------
def _spec(case):
    sp, wide = case["spacing"], case["depth_mm"] > 150.0
    extent = (480.0, 400.0, 240.0) if wide else (200.0, 200.0, 150.0)
    base = phantom.TINY_5MM_5BEAM
    return dataclasses.replace(
        base, shape=tuple(int(round(e / sp)) for e in extent), spacing=sp, n_beams=case["beams"],
        beamlet_mm=case["beamlet_mm"], sigma_mm=case["sigma_mm"], cutoff=case["cutoff"],
        ptv_radii=tuple(r * case["ptv"] for r in base.ptv_radii), coarse_unspecified=case["mixed"])


class _Geometry:
    """A phantom, and the fluence level that brings its PTV to 77 Gy on average."""

    def __init__(self, spec):
        self.case = c = phantom.make_case(spec)
        rows = np.flatnonzero(c.mask & 1)
        total = sum(float(c.val[c.row_ptr[j]:c.row_ptr[j + 1]].sum(dtype=np.float64)) for j in rows)
        self.level = 77.0 * max(1, rows.size) / max(total, 1e-9)


@functools.lru_cache(maxsize=3)
def _geometry(spec):
    return _Geometry(spec)


@functools.lru_cache(maxsize=2)
def _batch(plans):
    """The batched workload's phantoms (seeds 0, 1, ...) and each plan's step sizes per pass."""
    rng = np.random.Generator(np.random.PCG64(12345))
    return [(_Geometry(phantom.jittered_spec(i)), int(rng.choice((1, 4, 8)))) for i in range(plans)]


def _values(geo, seed):
    """This seed's D values and fluence (host arrays, FP32)."""
    c = geo.case
    rng = np.random.Generator(np.random.PCG64(seed))
    f = rng.uniform(0.9, 1.1, c.n).astype(np.float32)
    val = (torch.from_numpy(c.val).cuda() * torch.from_numpy(f).cuda()[torch.from_numpy(c.col).cuda()]).cpu().numpy()
    x = (geo.level * rng.uniform(0.5, 1.5, c.n)).astype(np.float32)
    return val, x


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _pinned(a):
    return torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()


def _make_plan(geo, val, options):
    c = geo.case
    return Plan(_dev(c.row_ptr), _dev(c.col), _dev(val), _dev(c.mask), c.thresholds, c.weights, m=c.m, n=c.n,
                options=options)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        s["plans"] = []
        for i, (geo, k) in enumerate(_batch(case["plans"])):
            val, _ = _values(geo, 1000 * seed + i)
            s["plans"].append(_make_plan(geo, val, Options(precision=PRECISIONS[case["precision"]][0], k_trials=k,
                                                           max_iter=MAX_ITER, solver=L.SOLVER_TEAM)))
        s["x"] = [torch.empty(p.n, device="cuda") for p in s["plans"]]
        return s
    geo = _geometry(_spec(case))
    c = geo.case
    val, x = _values(geo, seed)
    s["m"], s["n"], s["geo"] = c.m, c.n, geo
    if kind == "csr":
        s["keep"] = [_dev(c.row_ptr), _dev(c.col), _dev(val), _dev(c.mask), _dev(x)]
        rp, col, v, mask, xd = s["keep"]
        s["csr"] = L.imrt_csr(c.m, c.n, c.nnz, rp.data_ptr(), col.data_ptr(), v.data_ptr(), 1)
        s["z"] = torch.empty(c.m, device="cuda")
        return s
    options = Options(precision=PRECISIONS[case["precision"]][0], k_trials=case.get("k_trials", 1), max_iter=MAX_ITER)
    if kind == "new":
        s["host"] = [_pinned(a) for a in (c.row_ptr, c.col, val, c.mask)]
        s["options"], s["x"] = options, _dev(x)
    elif kind == "replan":
        # the patient's resident plan, the new fraction's D and the last fluence
        options = dataclasses.replace(options, solver=L.SOLVER_TEAM, x_init=2)
        s["plan"] = _make_plan(geo, _values(geo, seed + 7919)[0], options)
        s["host"], s["x0"] = [c.row_ptr, c.col, val, c.mask], x
    else:
        s["plan"] = _make_plan(geo, val, options)
        s["x"] = _dev(x)
        s["z"], s["g"] = torch.empty(c.m, device="cuda"), torch.empty(c.n, device="cuda")
    return s


# --- one pass --------------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "dose":
        return {"z": s["plan"].dose(s["x"], out=s["z"])}
    if kind == "eval":
        G, z, g = s["plan"].eval(s["x"], z_out=s["z"], g_out=s["g"])
        return {"G": G, "z": z, "g": g}
    if kind == "csr":
        _, _, _, mask, x = s["keep"]
        c, G = s["geo"].case, ctypes.c_double()
        L.check(L.load().imrt_eval_csr_noalloc(
            ctypes.byref(s["csr"]), mask.data_ptr(), c.n_structures, c.thresholds.ctypes.data, c.weights.ctypes.data,
            x.data_ptr(), s["z"].data_ptr(), ctypes.addressof(G), torch.cuda.current_stream().cuda_stream))
        return {"G": G.value, "z": s["z"]}
    if kind == "solve":
        r = s["plan"].solve()
        return {"objective": r.objective, "x": s["plan"].get_x(out=s["g"]), "z": s["plan"].dose(out=s["z"])}
    if kind == "batch":
        rs = solve_batch(s["plans"])
        return {"objective": np.array([r.objective for r in rs], np.float32),
                "x": torch.cat([p.get_x(out=x) for p, x in zip(s["plans"], s["x"])])}
    c = s["geo"].case
    if kind == "replan":
        p, (row_ptr, col, val, mask) = s["plan"], s["host"]
        p.update(row_ptr, col, val, mask, c.thresholds, c.weights, m=c.m, n=c.n)
        r = p.solve(x0=s["x0"])
        return {"objective": r.objective, "x": p.get_x(), "z": p.dose()}
    row_ptr, col, val, mask = s["host"]
    with Plan(row_ptr, col, val, mask, c.thresholds, c.weights, m=c.m, n=c.n, options=s["options"]) as p:
        info = p.info()
        G, z, g = p.eval(s["x"])
    return {"lambda0": info["lambda0_rule"], "x1_scale": info["x1_scale"], "G": G, "z": z, "g": g}


# --- what a pass cannot do without ------------------------------------------------------------
def _pass_bytes(case_, vb):
    """A forward and a transposed pass over a resident plan: D's values at their stored width with a
    16-bit index each, the row offsets, the mask, and x, z, r and g."""
    m, n, nnz = case_.m, case_.n, case_.nnz
    return nnz * (vb + 2) + 4 * m + 9 * m + 4 * n, nnz * (vb + 2) + 4 * n + 4 * m + 4 * n


def work(case):
    kind = case["kind"]
    vb = PRECISIONS[case.get("precision", "fp32")][1]
    if kind == "batch":
        b = f = 0
        for geo, k in _batch(case["plans"]):
            fw, bw = _pass_bytes(geo.case, vb)
            b += MAX_ITER * (fw + bw)
            f += MAX_ITER * 2 * geo.case.nnz * (k + 1)
        return {"bytes": b, "flops": f}
    c = _geometry(_spec(case)).case
    fw, bw = _pass_bytes(c, vb)
    csr = c.nnz * 8 + (c.m + 1) * 8 + c.m
    if kind == "dose":
        return {"bytes": c.nnz * 6 + 8 * c.m + 4 * c.n, "flops": 2 * c.nnz}
    if kind == "eval":
        return {"bytes": fw + bw, "flops": 4 * c.nnz}
    if kind == "csr":
        return {"bytes": csr + 4 * c.n + 4 * c.m, "flops": 2 * c.nnz}
    if kind == "new":  # the input once, the FP32 and the reduced layouts, 50 power steps over the FP32 ones
        f32 = sum(_pass_bytes(c, 4))
        return {"bytes": csr + (f32 if vb < 4 else 0) + fw + bw + 50 * f32, "flops": 2 * c.nnz * 102}
    k = case["k_trials"]
    solve = MAX_ITER * (fw + bw)
    return {"bytes": solve + (csr if kind == "replan" else 0), "flops": MAX_ITER * 2 * c.nnz * (k + 1)}


# --- the same in 64 bits -----------------------------------------------------------------------
class _Exact:
    """The method in FP64 torch: z = D x, G and r of the one-sided quadratic penalties, g = D^T r,
    the step-size rule and the projected-gradient Armijo loop."""

    def __init__(self, geo, val):
        c = geo.case
        row_ptr, col = _dev(c.row_ptr), _dev(c.col).long()
        v = _dev(val).double()
        self.D = torch.sparse_csr_tensor(row_ptr, col, v, size=(c.m, c.n))
        order = torch.sort(col, stable=True).indices
        t_ptr = torch.zeros(c.n + 1, dtype=torch.int64, device="cuda")
        t_ptr[1:] = torch.cumsum(torch.bincount(col, minlength=c.n), 0)
        rows = torch.repeat_interleave(torch.arange(c.m, device="cuda"), row_ptr[1:] - row_ptr[:-1])
        self.T = torch.sparse_csr_tensor(t_ptr, rows[order], v[order], size=(c.n, c.m))
        self.m, self.n = c.m, c.n
        self.terms = []  # (selected voxels as 0 / 1, threshold, coefficient, sign)
        mask = _dev(c.mask)
        for s in range(c.n_structures):
            sel = ((mask >> s) & 1).double()
            count = float(sel.sum())
            for k in range(2):
                t, w = float(c.thresholds[s, k]), float(c.weights[s, k])
                if not math.isnan(t) and w != 0.0 and count > 0:
                    self.terms.append((sel, t, w / count, -1.0 if k == 0 else 1.0))
        self.under = next(((sel, t) for sel, t, _, sign in self.terms if sign < 0), None)

    def dose(self, x):
        return (self.D @ x[:, None])[:, 0]

    def back(self, r):
        return (self.T @ r[:, None])[:, 0]

    def objective(self, z):
        G, r = 0.0, torch.zeros_like(z)
        for sel, t, c, sign in self.terms:
            e = torch.clamp(sign * (z - t), min=0.0) * sel
            G = G + c * (e * e).sum()
            r += 2.0 * c * sign * e
        return float(G), r

    def lambda0(self):
        diag = sum(c * sel for sel, _, c, _ in self.terms)
        v = torch.full((self.n,), 1.0 / math.sqrt(self.n), dtype=torch.float64, device="cuda")
        lam = 0.0
        for _ in range(50):
            w = self.back(diag * self.dose(v))
            lam = float(v @ w)
            norm = float(w.norm())
            if norm > 0:
                v = w / norm
        return 8.0 / (2.0 * lam) if lam > 0 else 1.0

    def x1_scale(self):
        if self.under is None:
            return 0.0
        sel, t = self.under
        z = self.dose(torch.ones(self.n, dtype=torch.float64, device="cuda"))
        return t / float((z * sel).sum() / sel.sum())

    def solve(self, x=None, eps=1e-4, alpha=2.0, delta=1e-6):
        lam0 = self.lambda0()
        if x is None:
            x = torch.full((self.n,), self.x1_scale(), dtype=torch.float64, device="cuda")
        z = self.dose(x)
        G, r = self.objective(z)
        for _ in range(MAX_ITER):
            g, lam = self.back(r), lam0
            for _ in range(51):
                xt = torch.clamp(x - lam * g, min=0.0)
                zt = self.dose(xt)
                Gt, rt = self.objective(zt)
                d2 = float(((xt - x) ** 2).sum())
                if d2 == 0.0 or Gt < G - eps / lam * d2:
                    break
                lam /= alpha
            if d2 == 0.0:
                break
            dG, x, z, r, G = abs(Gt - G), xt, zt, rt, Gt
            if G == 0.0 or dG < delta * G:
                break
        return x, z, G


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        xs, Gs = [], []
        for i, (geo, _) in enumerate(_batch(case["plans"])):
            x, _, G = _Exact(geo, _values(geo, 1000 * seed + i)[0]).solve()
            xs.append(x)
            Gs.append(G)
        return {"objective": np.array(Gs), "x": torch.cat(xs)}
    geo = _geometry(_spec(case))
    val, x = _values(geo, seed)
    E, x = _Exact(geo, val), _dev(x).double()
    if kind in ("solve", "replan"):
        x, z, G = E.solve(x if kind == "replan" else None)
        return {"objective": torch.tensor(G, dtype=torch.float64), "x": x, "z": z}
    z = E.dose(x)
    G, r = E.objective(z)
    G = torch.tensor(G, dtype=torch.float64)
    if kind == "dose":
        return {"z": z}
    if kind == "csr":
        return {"G": G, "z": z}
    if kind == "eval":
        return {"G": G, "z": z, "g": E.back(r)}
    wide = lambda v: torch.tensor(v, dtype=torch.float64)  # noqa: E731
    return {"lambda0": wide(E.lambda0()), "x1_scale": wide(E.x1_scale()), "G": G, "z": z, "g": E.back(r)}
