"""The node kernels against the oracle at the edges of their work splits: few nodes (every node cut
into slices of rows, columns or positions), one, two or more right-hand-side blocks of every width,
ragged last blocks, even and uneven leaves, forward and adjoint, in every arithmetic.

Tolerances as in test_gpu_apply.py: 1e-12 for FP64 and double-float, 2e-5 for FP32 (unit roundoff
6e-8 through L + 1 levels of sums of up to a few hundred terms)."""
import numpy as np
import pytest
import torch

import paper_1809_10573_gb300 as P
from oracle import idbf
from paper_1809_10573_gb300 import inputs
from tests.cases import oracle_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


MODES = [(P.MODE_FP64, P.STORE_C128, np.complex128, 1e-12), (P.MODE_DF64, P.STORE_DF64, np.complex128, 1e-12),
         (P.MODE_FP32, P.STORE_C64, np.complex64, 2e-5)]


@pytest.mark.parametrize("case", ["dft_1024", "fio_base_4096", "fio_paper_2048"])
@pytest.mark.parametrize("mode,fmt,dt,tol", MODES)
def test_every_block_width_matches_the_oracle(case, mode, fmt, dt, tol):
    c = oracle_case(case)
    plan = P.Plan.import_factors(c["ex"], storage=fmt)
    for R in (1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 13, 16, 17, 33):
        X = inputs.complex_gaussian(c["N"], R, seed=R)
        xd = torch.from_numpy(X.astype(dt)).cuda()
        if R == 1:
            plan.set_level_variants(mode, [0] * (plan.L + 1))   # the node kernel on every level
        assert rel(plan.apply(xd, mode=mode).cpu().numpy(), idbf.apply(c["F"], X)) < tol, R
        assert rel(plan.apply_adjoint(xd, mode=mode).cpu().numpy(), idbf.apply_adjoint(c["F"], X)) < tol, R


@pytest.mark.parametrize("kind", ["V", "U"])
def test_unsorted_redundant_lists_are_reordered_with_their_blocks(kind):
    """An import whose lists p_c are reversed, with the rows or columns of the blocks in the same
    order, is the same operator: the slices of a cut node rely on ascending lists."""
    c = oracle_case("dft_1024")
    ex = {k: (v.copy() if isinstance(v, np.ndarray) else v) for k, v in c["ex"].items()}
    L, m, hv = ex["L"], 1 << ex["L"], ex["L"] // 2
    rows, cols = np.asarray(ex["blk_rows"]).reshape(-1), np.asarray(ex["blk_cols"]).reshape(-1)
    moff, ioff = np.asarray(ex["blk_moff"]).reshape(-1), np.asarray(ex["blk_ioff"]).reshape(-1)
    levels = range(hv) if kind == "V" else range(hv + 1, L + 1)
    for l in levels:
        for o in range(2 * m * l, 2 * m * (l + 1)):
            r, k, mo, io = int(rows[o]), int(cols[o]), int(moff[o]), int(ioff[o])
            M = ex["mat"][mo:mo + r * k].reshape(r, k)
            nq, npl = (r, k) if kind == "V" else (k, r)
            ex["idx"][io + nq:io + nq + npl] = ex["idx"][io + nq:io + nq + npl][::-1].copy()
            ex["mat"][mo:mo + r * k] = (M[:, ::-1] if kind == "V" else M[::-1, :]).copy().reshape(-1)
    plan = P.Plan.import_factors(ex)
    X = inputs.complex_gaussian(c["N"], 1, seed=3)
    xd = torch.from_numpy(X).cuda()
    assert rel(plan.apply(xd).cpu().numpy(), idbf.apply(c["F"], X)) < 1e-12
    assert rel(plan.apply_adjoint(xd).cpu().numpy(), idbf.apply_adjoint(c["F"], X)) < 1e-12


@pytest.mark.parametrize("case", ["dft_1024", "fio_base_4096", "fio_base_8192_oddL"])
def test_split_precision_widths_and_split_modes(case):
    """3xTF32: every width of the warp-level MMA kernel, ragged last tiles, and the two split modes that
    run the tcgen05 kernel. FP32-class results: the 2e-5 bar of the FP32 apply."""
    from paper_1809_10573_gb300 import _lib
    c = oracle_case(case)
    plan = P.Plan.import_factors(c["ex"], storage=P.STORE_C64)
    for R in (1, 7, 8, 9, 17, 33, 100):
        X = inputs.complex_gaussian(c["N"], R, seed=R)
        xd = torch.from_numpy(X.astype(np.complex64)).cuda()
        ref = idbf.apply(c["F"], X)
        for mode in (0, 1, 2) if R in (1, 33) else (0,):
            assert _lib.lib().idbf_set_tc_split(plan._h, mode) == _lib.OK
            assert rel(plan.apply(xd, mode=P.MODE_TF32X3).cpu().numpy(), ref) < 2e-5, (R, mode)
    plan.sync_status()
