"""The measured workloads: building a factorization, applying it and its adjoint, differentiating
through it and applying batches of operators, through the public entry points of the package, over
the range of sizes, kernels, modes and numbers of right-hand sides that its tests, configurations
and benchmark use.

A case is a dict of plain values:
  op      "apply" (y = K x), "adjoint" (y = K^* x), "grad" (forward and backward of ||K x - b||^2),
          "batch" (many operators of uneven size), "build" (construct the plan, apply it once);
  kernel  "fio" (Example 1's 1D Fourier integral operator on the uniform grid), "dft" (Example 3's
          kernel on a jittered grid), "j0" (Example 2, the Schloemilch expansion), "nufft"
          (Example 3 on random points: coordinate-based trees with leaves of uneven size);
  N, leaf, eps, R (right-hand sides), mode ("fp64", "df64", "fp32", "tf32x3", "tf32x3_s64"), qr
  (arithmetic of the construction), tuned (Plan.autotune was called, as a serving program does).
"""
import math

import numpy as np
import torch

import paper_1809_10573_gb300 as P
from paper_1809_10573_gb300 import inputs

MODES = {"fp64": P.MODE_FP64, "df64": P.MODE_DF64, "fp32": P.MODE_FP32, "tf32x3": P.MODE_TF32X3,
         "tf32x3_s64": P.MODE_TF32X3_S64}
STORE = {"fp64": P.STORE_C128, "df64": P.STORE_DF64, "fp32": P.STORE_C64, "tf32x3": P.STORE_C64,
         "tf32x3_s64": P.STORE_C64}
QR = {"fp64": P.QR_FP64, "df64": P.QR_DF64}
# oversampling (inner steps, leaf step) that reaches eps for each kernel
OVERSAMPLE = {"fio": (2.0, 4.0), "dft": (2.0, 4.0), "j0": (2.0, 4.0), "nufft": (2.0, 4.0)}
EXACT_ENTRIES = 1 << 34  # dense entries up to which exact() stays within seconds


def _case(name, op, kernel, N, mode, R=1, leaf=64, eps=1e-6, qr="fp64", tuned=False):
    return dict(name=name, op=op, kernel=kernel, N=N, leaf=leaf, eps=eps, mode=mode, R=R, qr=qr, tuned=tuned)


def listed():
    return [
        # the smallest call: one vector through a small operator, everything at its default
        _case("apply-fp64-2e12", "apply", "fio", 1 << 12, "fp64", eps=1e-8),
        # an ordinary single-vector call of a program that tuned its plan
        _case("apply-df64-2e14", "apply", "fio", 1 << 14, "df64", tuned=True),
        # a large single-vector call: 12 GB of factors streamed once
        _case("apply-df64-2e18", "apply", "fio", 1 << 18, "df64", tuned=True),
        # short blocks in complex64: Example 2's operator
        _case("apply-fp32-j0-2e17", "apply", "j0", 1 << 17, "fp32", qr="df64", tuned=True),
        # a solver's adjoint product (least squares, power iterations)
        _case("adjoint-df64-2e16", "adjoint", "fio", 1 << 16, "df64"),
        # differentiation: forward and backward with 32 right-hand sides
        _case("grad-fp32-r32-2e16", "grad", "fio", 1 << 16, "fp32", R=32, qr="df64"),
        # many right-hand sides: the tensor-core mode
        _case("apply-tf32x3-r256-2e16", "apply", "fio", 1 << 16, "tf32x3", R=256, qr="df64"),
        # a few accurate right-hand sides on a size and leaf that fit no tile
        _case("apply-df64-r9-40960", "apply", "dft", 40960, "df64", R=9, leaf=40),
        # the non-uniform transform of a few signals: uneven leaves
        _case("nufft-fp32-r5-100003", "apply", "nufft", 100003, "fp32", R=5, qr="df64"),
        # uneven batch: 24 small operators, 1-32 right-hand sides each
        dict(name="batch-fp32-24ops", op="batch", ops=24, emin=10, emax=14, draw_seed=4, eps=1e-6, leaf=64,
             mode="fp32", qr="df64", tuned=True),
        # construction: a new operator, then its first product
        _case("build-fio-2e15", "build", "fio", 1 << 15, "fp32", qr="df64"),
        # construction on new random points, then the transform
        _case("build-nufft-50000", "build", "nufft", 50000, "fp32", qr="df64"),
    ]


def _spread(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "apply", "adjoint", "adjoint", "grad", "batch", "build"])
    if op == "batch":
        emin = rng.randint(9, 11)
        return dict(op=op, ops=rng.randint(8, 24), emin=emin, emax=rng.randint(emin + 1, 14), draw_seed=rng.randint(1, 999),
                    eps=1e-6, leaf=64, mode=rng.choice(["fp32", "fp32", "df64"]), qr="fp64", tuned=True)
    kernel = rng.choice(["fio", "fio", "dft", "j0", "nufft"])
    leaf = 64 if rng.random() < 0.5 else rng.randint(30, 90)
    if op == "grad":
        mode, R = "fp32", int(_spread(rng, 2, 33))
    elif op == "apply" and kernel != "nufft" and rng.random() < 0.2:
        mode, R = rng.choice(["tf32x3", "tf32x3", "tf32x3_s64"]), int(_spread(rng, 32, 256))
    else:
        mode = rng.choice(["fp64", "df64", "fp32"])
        R = 1 if op == "build" or rng.random() < 0.5 else int(_spread(rng, 2, 33))
    big = 15 if op == "build" else 17 if R == 1 else 16 if mode in ("fp32", "tf32x3") else 14
    N = int(_spread(rng, 1 << 10, 1 << big))
    if kernel != "nufft":
        N = leaf << max(2, round(math.log2(N / leaf)))
        while N > 1 << big:
            N //= 2
    eps = 1e-8 if mode in ("fp64", "df64") and N <= 1 << 14 and rng.random() < 0.4 else 1e-6
    qr = "df64" if mode in ("fp32", "tf32x3") else "fp64"
    tuned = op == "apply" and R == 1 and mode in MODES and rng.random() < 0.6
    return dict(op=op, kernel=kernel, N=N, leaf=leaf, eps=eps, mode=mode, R=R, qr=qr, tuned=tuned)


# ---- the operators ----------------------------------------------------------------------------
def _points(case, seed):
    N = case["N"]
    if case["kernel"] == "fio":
        return inputs.uniform_grid(N)
    if case["kernel"] == "dft":
        return inputs.jittered_grid(N, seed=seed)
    if case["kernel"] == "j0":
        return inputs.schlomilch_grid(N)
    return inputs.nufft_points(N, seed=seed)


def _build(case, points, trees=None):
    x, xi = points
    t, t_leaf = OVERSAMPLE[case["kernel"]]
    kw = dict(eps=case["eps"], oversample=t, oversample_leaf=t_leaf, qr_arith=QR[case["qr"]], storage=STORE[case["mode"]])
    if case["kernel"] == "nufft":
        L, rows, cols = trees or _trees(case, points)
        return P.Plan.build_leaves(x, xi, L, rows, cols, kernel="dft", sign=-1, **kw)
    return P.Plan.build(x, xi, leaf=case["leaf"], kernel=case["kernel"], c_profile=0, sign=-1, **kw)


def _trees(case, points):
    N = case["N"]
    L = P.tree_depth(N, case["leaf"])
    return L, P.dyadic_leaves(points[0], -N / 2, N / 2, L), P.dyadic_leaves(points[1], 0.0, 1.0, L)


def _ops(case):
    return inputs.uneven_batch(seed=case["draw_seed"], nops=case["ops"], emin=case["emin"], emax=case["emax"])


def _op_case(case, o):
    return dict(kernel=o["kind"], N=o["N"], leaf=case["leaf"], eps=case["eps"], mode=case["mode"], qr=case["qr"], R=o["nrhs"])


# A program builds a plan once and applies it to many inputs: the plans of one case at a time are
# kept here, with what a construction reads (points, trees) left to prepare().
_kept = {}


def _plans(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _kept:
        _kept.clear()
        if case["op"] == "batch":
            ops = [(_op_case(case, o), o["seed"]) for o in _ops(case)]
            made = [_build(c, _points(c, s)) for c, s in ops]
            b = P.Batch(made, [c["R"] for c, _ in ops], mode=MODES[case["mode"]])
            if case["tuned"]:
                b.autotune([_vectors(c["N"], c["R"], case["mode"], 1 + i) for i, (c, _) in enumerate(ops)], reps=5)
            _kept[key] = (made, b)
        else:
            p = _build(case if case["mode"] != "tf32x3_s64" else dict(case, mode="fp64"), _points(case, case["N"]))
            if case["mode"] == "tf32x3_s64":  # the middle factor in double-float, the others in complex64
                for l in range(p.L + 1):
                    p.set_level_storage(l, P.STORE_DF64 if l == p.L // 2 else P.STORE_C64)
            if case["tuned"]:
                p.autotune(MODES[case["mode"]], reps=10)
            _kept[key] = ([p], None)
    return _kept[key]


def _vectors(N, R, mode, seed):
    """Complex Gaussian right-hand sides on the GPU, column-major (N, R), or (N,) for one."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(R, N, dtype=torch.complex128, device="cuda", generator=g) * math.sqrt(2.0)
    if mode not in ("fp64", "df64"):
        v = v.to(torch.complex64)
    return v[0] if R == 1 else v.t()


# ---- one pass ---------------------------------------------------------------------------------
def prepare(case, seed):
    op, mode = case["op"], case["mode"]
    s = dict(op=op, mode=MODES[mode], case=case)
    if op == "batch":
        s["batch"] = _plans(case)[1]
        s["x"] = [_vectors(o["N"], o["nrhs"], mode, seed * 1000 + i) for i, o in enumerate(_ops(case))]
        return s
    s["x"] = _vectors(case["N"], case["R"], mode, seed)
    if op == "build":
        _kept.clear()
        s["points"] = _points(case, seed)
        s["trees"] = _trees(case, s["points"]) if case["kernel"] == "nufft" else None
        return s
    s["plan"] = _plans(case)[0][0]
    if op == "grad":
        s["b"] = _vectors(case["N"], case["R"], mode, seed + 7919)
    return s


def run(s):
    op = s["op"]
    if op == "apply":
        return s["plan"].apply(s["x"], mode=s["mode"])
    if op == "adjoint":
        return s["plan"].apply_adjoint(s["x"], mode=s["mode"])
    if op == "grad":
        x = s["x"].detach().requires_grad_(True)
        y = P.apply(s["plan"], x, s["mode"])
        loss = ((y - s["b"]).abs() ** 2).sum()
        loss.backward()
        return {"loss": loss.detach(), "y": y.detach(), "grad": x.grad}
    if op == "batch":
        return s["batch"].apply(s["x"])
    plan = _build(s["case"], s["points"], s["trees"])
    return plan.apply(s["x"], mode=s["mode"])


# ---- what a pass cannot do without ------------------------------------------------------------
def _apply_work(plan, R, mode):
    st = plan.stats()
    eb, vb = (8, 8) if mode not in ("fp64", "df64") else (16, 16)
    return (st["entries"] * eb + st["index_entries"] * 4 + 2 * plan.N * R * vb, 8 * st["entries"] * R)


def work(case):
    op, mode = case["op"], case["mode"]
    if op == "batch":
        ws = [_apply_work(p, o["nrhs"], mode) for p, o in zip(_plans(case)[0], _ops(case))]
        return {"bytes": sum(w[0] for w in ws), "flops": sum(w[1] for w in ws)}
    if op == "build":
        # the points read and the factors written once, then the apply; a pivoted QR of each ID's
        # samples (t b x b, mean sizes per step) to its rank k: 8 (2 m n k - k^2 (m + n) + 2 k^3 / 3) flops
        # complex, of which half are multiplications
        plan = _plans(case)[0][0]
        st = plan.stats()
        t, t_leaf = OVERSAMPLE[case["kernel"]]
        nids, L, hv = 2 << st["L"], st["L"], st["h_v"]
        k = [b / nids for b in st["boundary_entries"]]
        flops = 0.0
        for s in range(L):
            first = s == 0 or s == L - 1
            n = case["N"] / (1 << L) if first else 2 * (k[s - 1] if s < hv else k[s + 1])
            m = (t_leaf if first else t) * n
            flops += nids * 8 * (2 * m * n * k[s] - k[s] ** 2 * (m + n) + 2 * k[s] ** 3 / 3) / 2
        b, f = _apply_work(plan, case["R"], mode)
        return {"bytes": 2 * b + 16 * case["N"], "flops": flops + f}
    b, f = _apply_work(_plans(case)[0][0], case["R"], mode)
    return {"bytes": 2 * b, "flops": 2 * f} if op == "grad" else {"bytes": b, "flops": f}


# ---- the same in 64 bits, from the kernels' definitions ---------------------------------------
def _rows(kernel, x, xi):
    """K(x_i, xi_j) of a block of rows, complex128 (or float64 for the real kernel)."""
    if kernel == "j0":
        return torch.special.bessel_j0(x[:, None] * xi[None, :])
    if kernel == "fio":
        c = (2 + torch.sin(2 * math.pi * x) * torch.sin(4 * math.pi * x)) / 3
        ph = torch.frac(x[:, None] * xi[None, :]) + torch.frac(c[:, None] * xi.abs()[None, :])
    else:
        ph = -torch.frac(x[:, None] * xi[None, :])
    return torch.polar(torch.ones_like(ph), ph.mul_(2 * math.pi))


def _dense(case, points, v, adjoint=False):
    kernel = case["kernel"]
    x, xi = (torch.from_numpy(np.asarray(p)).cuda() for p in points)
    v = v.to(torch.complex128)
    v = v[:, None] if v.dim() == 1 else v
    step = max(1, (1 << 27) // xi.numel())
    out = torch.zeros_like(v)
    for i in range(0, x.numel(), step):
        K = _rows(kernel, x[i:i + step], xi).to(torch.complex128)
        if adjoint:
            out += K.mH @ v[i:i + step]
        else:
            out[i:i + step] = K @ v
    return out


def exact(case, seed):
    s = prepare(case, seed)
    if case["op"] == "batch":
        return [_dense(c, _points(c, o["seed"]), x).reshape(x.shape)
                for c, o, x in ((_op_case(case, o), o, x) for o, x in zip(_ops(case), s["x"]))]
    if case["N"] ** 2 > EXACT_ENTRIES or case["N"] ** 2 * case["R"] > 1 << 40:
        return None
    points = s["points"] if case["op"] == "build" else _points(case, case["N"])
    y = _dense(case, points, s["x"], adjoint=case["op"] == "adjoint").reshape(s["x"].shape)
    if case["op"] != "grad":
        return y
    d = y - s["b"]
    return {"loss": (d.abs() ** 2).sum(), "y": y, "grad": _dense(case, points, 2 * d, adjoint=True)}
