"""Rounding errors of the applies: no larger than those of kernels that cut every row and column into
short partial sums. The bars are those kernels' measured errors (one chain per row exceeds them by
15 to 60 %), with 5 % for the means over a few vectors; the FP64 bars are for the same vectors.
Relative errors against the FP64 apply of the same plan, or, for FP64, against the factors' product in
extended precision."""
import numpy as np
import pytest
import torch

import paper_1809_10573_gb300 as P
from paper_1809_10573_gb300 import inputs
from tests.cases import oracle_case

pytestmark = pytest.mark.gpu
MODES = {"fp32": (P.MODE_FP32, torch.complex64), "df64": (P.MODE_DF64, torch.complex128),
         "tf32x3": (P.MODE_TF32X3, torch.complex64), "tf32x3_s64": (P.MODE_TF32X3_S64, torch.complex64)}
# kernel, N, leaf: (mode, right-hand sides, adjoint, error)
BARS = [
    ("fio", 1 << 14, 64, [("fp32", 2, False, 4.14e-7), ("fp32", 4, False, 4.13e-7), ("fp32", 8, True, 4.03e-7),
                          ("df64", 1, True, 1.67e-14), ("df64", 4, True, 1.67e-14)]),
    ("fio", 1 << 12, 64, [("fp32", 2, True, 3.05e-7), ("fp32", 8, True, 3.26e-7), ("fp32", 32, True, 3.84e-7)]),
    ("dft", 40960, 40, [("fp32", 4, False, 3.37e-7), ("fp32", 8, False, 3.91e-7), ("fp32", 32, False, 4.91e-7),
                        ("df64", 4, True, 1.50e-14), ("tf32x3", 32, False, 5.80e-7), ("tf32x3_s64", 32, False, 4.90e-7)]),
]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("kernel,N,leaf,bars", BARS, ids=lambda v: str(v) if isinstance(v, (int, str)) else "")
def test_errors_against_fp64_are_those_of_short_partial_sums(kernel, N, leaf, bars):
    x, xi = inputs.uniform_grid(N) if kernel == "fio" else inputs.jittered_grid(N, 1)
    plan = P.Plan.build(x, xi, eps=1e-6, leaf=leaf, kernel=kernel, sign=-1, oversample=2, oversample_leaf=4)
    plan.set_storage(P.STORE_C128, P.STORE_DF64, P.STORE_C64)
    for name, R, adjoint, bar in bars:
        mode, dt = MODES[name]
        fn = plan.apply_adjoint if adjoint else plan.apply
        errors = []
        for seed in range(3):
            X = torch.from_numpy(inputs.complex_gaussian(N, R, seed=100 + seed)).cuda().to(dt)
            ref = fn(X.to(torch.complex128), mode=P.MODE_FP64)
            errors.append(float(torch.linalg.norm(fn(X, mode=mode).to(torch.complex128) - ref) / torch.linalg.norm(ref)))
        assert sum(errors) / 3 <= 1.05 * bar, (name, R, adjoint, errors)


def _extended(ex, X, adjoint):
    """The factors' product in extended precision, level by level over the exported blocks."""
    L, m = ex["L"], 1 << ex["L"]
    hv, n0, LD = L // 2, ex["n0"], np.clongdouble
    rows, cols, mo, io = (np.asarray(ex[k]).reshape(L + 1, m, 2) for k in ("blk_rows", "blk_cols", "blk_moff", "blk_ioff"))
    seg, mat, idx = np.asarray(ex["seg_len"]).reshape(L, 2 * m), np.asarray(ex["mat"]), np.asarray(ex["idx"])

    def out_seg(l, j, c):
        H = 1 << (L - l)
        return (j // H) * 2 * H + j % H + c * H

    def block(l, j, c):
        r, k = rows[l, j, c], cols[l, j, c]
        M = mat[mo[l, j, c]:mo[l, j, c] + r * k].reshape(r, k).astype(LD)
        nq, n = (r if l < hv else k), r + k
        ix = idx[io[l, j, c]:io[l, j, c] + n]
        return M, ix[:nq], ix[nq:]

    segs, Y = None, np.zeros(X.shape, LD)
    for l in range(L, -1, -1) if adjoint else range(L + 1):
        new = [None] * (2 * m)
        for j in range(m):
            leaf = slice(j * n0, (j + 1) * n0)
            ins = [2 * j, 2 * j + 1]
            outs = [out_seg(l, j, c) for c in (0, 1)]
            src, dst = (outs, ins) if adjoint else (ins, outs)
            v = [X[leaf].astype(LD)] if l == (L if adjoint else 0) else [segs[s] for s in src]
            u = np.concatenate(v)
            B = [block(l, j, c) for c in (0, 1)]
            if l == hv:      # S
                o = [sum(B[c][0].conj().T @ v[c] for c in (0, 1))] if adjoint else [B[c][0] @ u for c in (0, 1)]
            elif (l < hv) != adjoint:   # gathers: out_c = u[q_c] + M u[p_c]
                o = [u[q] + (M.conj().T if adjoint else M) @ u[p] for M, q, p in B]
            else:                        # scatters: t[q_c] += v_c, t[p_c] += M v_c
                t = np.zeros((B[0][1].size + B[0][2].size, X.shape[1]), LD)
                for (M, q, p), w in zip(B, v):
                    t[q] += w
                    t[p] += (M.conj().T if adjoint else M) @ w
                o = [t]
            if l == (0 if adjoint else L):
                Y[leaf] = o[0]
                continue
            if len(o) == 1:
                n = seg[l - 1 if adjoint else l, dst[0]]
                o = [o[0][:n], o[0][n:]]
            new[dst[0]], new[dst[1]] = o
        segs = new
    return Y


@pytest.mark.parametrize("case,bars", [
    ("dft_1024", [(2, False, 3.14e-16), (5, False, 3.06e-16), (8, False, 3.08e-16)]),
    ("fio_base_4096", [(1, True, 4.72e-16), (2, False, 6.04e-16), (2, True, 5.47e-16)])])
def test_fp64_errors_against_extended_precision(case, bars):
    c = oracle_case(case)
    plan = P.Plan.import_factors(c["ex"])
    X = inputs.complex_gaussian(c["N"], 8, seed=5)
    ref = {a: _extended(c["ex"], X, a) for a in {a for _, a, _ in bars}}
    for R, adjoint, bar in bars:
        fn = plan.apply_adjoint if adjoint else plan.apply
        r = ref[adjoint][:, :R]
        y = fn(torch.from_numpy(X[:, :R].copy()).cuda()).cpu().numpy().astype(np.clongdouble)
        err = np.linalg.norm((y - r).astype(complex)) / np.linalg.norm(r.astype(complex))
        assert err <= 1.05 * bar, (R, adjoint, err)
