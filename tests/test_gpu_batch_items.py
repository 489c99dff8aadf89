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


def _wide_middle(N0, k, k2, seed):
    """Host factors of a made-up operator (L = 2): leaves of N0 points, k skeletons per V block, k2 per U
    block, so that the middle nodes read 2 k elements and write few."""
    rng = np.random.default_rng(seed)
    m, L = 4, 2
    rows = np.array([[[k, k]] * m, [[k2, k2]] * m, [[N0 - k2] * 2] * m], dtype=np.int32)
    cols = np.array([[[N0 - k, N0 - k]] * m, [[2 * k] * 2] * m, [[k2, k2]] * m], dtype=np.int32)
    mat, idx, mo, io = [], [], np.zeros(rows.shape, np.int64), np.zeros(rows.shape, np.int64)
    nm = ni = 0
    for l in range(L + 1):
        for j in range(m):
            for c in range(2):
                r, q = int(rows[l, j, c]), int(cols[l, j, c])
                mat.append((rng.standard_normal(r * q) + 1j * rng.standard_normal(r * q)) / np.sqrt(q))
                mo[l, j, c], nm = nm, nm + r * q
                io[l, j, c] = ni
                if l != 1:
                    p = rng.permutation(N0)
                    nq = k if l == 0 else k2
                    idx.append(np.concatenate([np.sort(p[:nq]), np.sort(p[nq:])]))
                    ni += N0
    return dict(N=m * N0, n0=N0, L=L, seg_len=np.array([[k] * 2 * m, [k2] * 2 * m], np.int32), blk_rows=rows, blk_cols=cols,
                blk_moff=mo, blk_ioff=io, mat=np.concatenate(mat), idx=np.concatenate(idx).astype(np.int32))


def test_a_refused_fault_injection_leaves_the_batch_working():
    """Nine double-float vectors through middle nodes of 2400 inputs fit the level launches (three vectors
    per CTA), not the persistent launch that the fault injection needs (items of 5 and 4)."""
    plan = P.Plan.import_factors(_wide_middle(1204, 1200, 8, 1), storage=P.STORE_DF64)
    x = torch.from_numpy(inputs.complex_gaussian(plan.N, 9, seed=2)).cuda()
    b = P.Batch([plan], [9], mode=P.MODE_DF64)
    for _ in range(2):
        with pytest.raises(P.IDBFError) as e:
            b.debug_set_wait(20_000_000, 1)
        assert e.value.status == _lib.EUNSUPPORTED
        y = b.apply([x])[0].cpu().numpy()
        b.sync_status()
        ref = plan.apply(x, mode=P.MODE_DF64).cpu().numpy()
        assert np.linalg.norm(y - ref) / np.linalg.norm(ref) < 1e-13
    b.close()
