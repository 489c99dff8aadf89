"""The node kernels on leaves of uneven size, some empty, and the wide middle factor of 3xTF32 over complex64
boundaries: every block width, ragged last blocks, forward and adjoint, against the oracle.
Tolerances as in test_gpu_node.py."""
import numpy as np
import pytest
import torch

import paper_1809_10573_gb300 as P
from oracle import idbf
from paper_1809_10573_gb300 import inputs
from tests.cases import oracle_case
from tests.test_gpu_nonuniform import case

pytestmark = pytest.mark.gpu
WIDTHS = (2, 3, 4, 6, 7, 8, 9, 12, 13, 16, 17, 33)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


@pytest.mark.parametrize("name", ["nufft_3000_oddL", "clustered_640"])
@pytest.mark.parametrize("mode,fmt,dt,tol", [(P.MODE_FP64, P.STORE_C128, np.complex128, 1e-12),
                                             (P.MODE_DF64, P.STORE_DF64, np.complex128, 1e-12),
                                             (P.MODE_FP32, P.STORE_C64, np.complex64, 2e-5)])
def test_every_block_width_on_uneven_leaves(name, mode, fmt, dt, tol):
    c = case(name)
    plan = P.Plan.import_factors(c["ex"], storage=fmt)
    for R in WIDTHS:
        X = inputs.complex_gaussian(c["N"], R, seed=R)
        xd = torch.from_numpy(X.astype(dt)).cuda()
        assert rel(plan.apply(xd, mode=mode).cpu().numpy(), idbf.apply(c["F"], X)) < tol, R
        assert rel(plan.apply_adjoint(xd, mode=mode).cpu().numpy(), idbf.apply_adjoint(c["F"], X)) < tol, R


@pytest.mark.parametrize("wide", [P.STORE_C128, P.STORE_DF64])
@pytest.mark.parametrize("name", ["dft_1024", "fio_base_8192_oddL"])
def test_wide_middle_factor_at_every_block_width(name, wide):
    c = oracle_case(name)
    plan = P.Plan.import_factors(c["ex"], storage=P.STORE_C128)
    plan.set_storage(P.STORE_C128, P.STORE_C64)
    plan.set_level_storage(plan.L // 2, wide, P.STORE_C64)
    for R in (1,) + WIDTHS:
        X = inputs.complex_gaussian(c["N"], R, seed=R)
        xd = torch.from_numpy(X.astype(np.complex64)).cuda()
        assert rel(plan.apply(xd, mode=P.MODE_TF32X3_S64).cpu().numpy(), idbf.apply(c["F"], X)) < 2e-5, R
