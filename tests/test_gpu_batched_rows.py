"""The row pass of several right-hand sides against the FP64 oracle, two-pass
sweeps.  One sweep's bound is the suite's 1e-5 relative L2 (FP32 sums of about a
hundred terms: 1e-7 relative each).

A warp reads a row in windows of 32 entries and the 8 warps of a CTA take its
rows in turn: rows of 0, 1, 31 .. 33 and 63 .. 65 entries, row counts around
multiples of 8, blocks smaller than a CTA's turn.
"""
import numpy as np
import pytest

import oracle as O
import paper_2606_27086_gb300 as pk
import synth
from tests.helpers import random_x, rel_l2, rounded_values

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nrhs,dtype", [(3, "f32"), (8, "bf16"), (16, "f32"), (16, "f16"), (32, "f32")])
@pytest.mark.parametrize("m,mode", [(1, O.CIMMINO), (7, O.CIMMINO), (41, O.BIP), (1601, O.CIMMINO)])
def test_rows_in_turn(nrhs, dtype, m, mode):
    n = 97
    rng = np.random.default_rng(m + nrhs)
    lens = rng.choice([0, 1, 31, 32, 33, 63, 64, 65, 97], m)
    lens[0] = 33
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    col = np.concatenate([rng.permutation(n)[:k] for k in lens]).astype(np.int32)
    A = synth.CSR(m, n, rp, col, rng.uniform(0.1, 1.0, len(col)).astype(np.float32))
    b = (A.to_scipy() @ rng.uniform(0.0, 1.0, (n, nrhs))) * (1 + 0.2 * rng.standard_normal((m, nrhs)))
    l, u = synth.slab_bounds(b, 0.03)
    prob = synth.Problem("turns", A, l, u, np.zeros(1, np.float32), np.ones(1, np.float32))
    if mode == O.BIP:
        prob.blocks = (np.arange(m) % 5).astype(np.int32)
    dt = {"f32": pk.SUPPY_F32, "bf16": pk.SUPPY_BF16, "f16": pk.SUPPY_F16}[dtype]
    ctx = pk.from_problem(prob, mode=mode, dtype=dt, strategy=pk.STRATEGY_TWO_PASS)
    x0 = random_x(n, nrhs, seed=3)
    ctx.suppy_set_x(x0)
    ctx.suppy_sweep(pk.suppy_params_default(lam=1.2), 1)
    xg = ctx.suppy_get_x()
    ctx.close()
    for k in range(nrhs):
        S, _, _, lo, hi = O.from_problem(prob, mode, values=rounded_values(prob.A.val, dtype))
        x = np.clip(x0[:, k].astype(np.float64), lo, hi)
        x, _ = O.sweep(S, mode, O.rhs(prob.l, k), O.rhs(prob.u, k), 1.2, lo, hi, x)
        assert rel_l2(xg[:, k], x) <= 1e-5
