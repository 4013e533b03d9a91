"""Doses and corrections of the CQ step over row and column lengths around the
batches its kernels load ahead, against FP64: d = A_q x and, for a target whose
every dose is raised to d_ref, x + gamma A_q^T (d_ref - d).  The bound is the
suite's 1e-5 relative L2 (FP32 sums of up to 1600 positive terms).
"""
import numpy as np
import pytest

import paper_2606_27086_gb300 as pk
import synth
from tests.helpers import rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("mq,n,lens", [
    (1, 1, [1]),
    (40, 300, [0, 1, 31, 32, 33, 191, 192, 193, 224]),     # columns of about 16
    (1600, 33, [33, 32, 31, 0]),                            # columns of about 1200
    (700, 65, [65, 64, 40]),                                # columns of about 600
    (9000, 1200, [384, 385, 60]),                           # more rows than one wave of warps
])
@pytest.mark.parametrize("nrhs", [1, 2])
def test_dose_and_correction_shapes(mq, n, lens, nrhs):
    rng = np.random.default_rng(mq + n)
    ln = np.resize(lens, mq)
    rp = np.concatenate([[0], np.cumsum(ln)]).astype(np.int32)
    col = np.concatenate([np.sort(rng.permutation(n)[:k]) for k in ln]).astype(np.int32)
    A = synth.CSR(mq, n, rp, col, rng.uniform(0.1, 1.0, len(col)).astype(np.float32))
    l = np.full((mq, nrhs) if nrhs > 1 else mq, -np.inf, np.float32)   # no slab moves x after the step
    ctx = pk.Context(rp, col, A.val, mq, n, l, -l, np.full(1, -np.inf, np.float32),
                     np.full(1, np.inf, np.float32), nrhs=nrhs)
    M = A.to_scipy().astype(np.float64)
    x0 = rng.uniform(0.0, 1.0, (n, nrhs)).astype(np.float32)
    d = M @ x0
    ref = float(2 * d.max() + 1)
    ctx.suppy_set_dvc(rp, col, A.val, mq, np.array([0, mq], np.int32), [(1, 0, 1.0, ref)], 1.0)
    ctx.suppy_set_x(x0[:, 0].copy() if nrhs == 1 else x0)
    dose = ctx.suppy_dvc_dose().reshape(mq, nrhs)
    ctx.suppy_sweep(pk.suppy_params_default(), 1)
    x = ctx.suppy_get_x().reshape(n, nrhs)
    ctx.close()
    gamma = 1.0 / float((M.multiply(M)).sum())
    for b in range(nrhs):
        assert rel_l2(dose[:, b], d[:, b]) <= 1e-5
        assert rel_l2(x[:, b], x0[:, b] + gamma * (M.T @ (ref - d[:, b]))) <= 1e-5
