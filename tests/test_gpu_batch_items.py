"""The persistent batch launch with items of unequal length: an operator whose last item is shorter and
runs a wider body than its first ones (double-float, 9 right-hand sides: items of 5 and 4, passes of 3
and of 4), as the one that needs the most shared memory of its batch."""
import numpy as np
import pytest
import torch

import paper_1809_10573_gb300 as P
from oracle import idbf
from paper_1809_10573_gb300 import _lib, inputs
from tests.cases import oracle_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("mode,fmt,dt,tol", [(P.MODE_DF64, P.STORE_DF64, np.complex128, 1e-12),
                                             (P.MODE_FP32, P.STORE_C64, np.complex64, 2e-5),
                                             (P.MODE_FP64, P.STORE_C128, np.complex128, 1e-12)])
@pytest.mark.parametrize("R", [9, 17, 33])
def test_last_items_of_another_width_at_every_tiling(mode, fmt, dt, tol, R):
    # tolerances as in test_gpu_batch.py
    plans, xs, refs = [], [], []
    for k, (case, r) in enumerate([("dft_1024", 1), ("fio_base_4096", R)]):
        c = oracle_case(case)
        plans.append(P.Plan.import_factors(c["ex"], storage=fmt))
        X = inputs.complex_gaussian(c["N"], r, seed=30 + k)
        xs.append(torch.from_numpy(X.astype(dt)).cuda())
        refs.append(idbf.apply(c["F"], X))
    b = P.Batch(plans, [1, R], mode=mode)
    for tile in range(len(P.Batch.TILES)):
        try:
            b.set_tiling(tile)
        except P.IDBFError as e:
            assert e.status == _lib.EUNSUPPORTED
            continue
        ys = b.apply(xs)
        b.sync_status()
        for y, ref in zip(ys, refs):
            y = y.cpu().numpy()
            assert np.linalg.norm(y - ref) / np.linalg.norm(ref) < tol, (tile, b.info())
    b.close()
