"""The step length of EL and EMR multiplies the whole correction, so its rounding
would be an error in every unknown alike that changes from run to run.  What
is left without it is the rounding of the unknowns themselves, thousands of
independent ones: the distance of one right-hand side from the FP64 oracle is
then the same for every starting point.  Bound: largest to smallest over ten starts at most 1.25 (the
norm of N = 9216 independent roundings varies by about 1 / sqrt(2 N) < 1%; the
rest is room for the sums behind the step), against a factor of 1.5 to 2.5
with the step length held in one float."""
import numpy as np
import pytest

import oracle as O
import paper_2606_27086_gb300 as pk
import synth
from tests.helpers import random_x, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nrhs,kw", [(1, {}), (1, dict(stream_map=1)), (1, dict(tma=-1)), (3, {})])
@pytest.mark.parametrize("mode", [O.EL, O.EMR])
def test_step_length_is_not_rounded_to_a_float(mode, nrhs, kw):
    prob = synth.ct_problem(96, 120, 137, nrhs=nrhs)
    ctx = pk.from_problem(prob, mode=mode, strategy=pk.STRATEGY_TWO_PASS, **kw)
    S, l, u, lo, hi = O.from_problem(prob, mode)
    errs = [[] for _ in range(nrhs)]
    for seed in range(40, 50):
        x0 = random_x(prob.A.n, nrhs, seed=seed)
        ctx.suppy_set_x(x0)
        ctx.suppy_sweep(pk.suppy_params_default(lam=1.2), 1)
        xg = ctx.suppy_get_x().reshape(prob.A.n, nrhs)
        x0 = np.clip(x0.astype(np.float64), lo, hi).reshape(prob.A.n, nrhs)
        for b in range(nrhs):
            x, _ = O.sweep(S, mode, O.rhs(l, b), O.rhs(u, b), 1.2, lo, hi, x0[:, b])
            errs[b].append(rel_l2(xg[:, b], x))
    ctx.close()
    for e in errs:
        assert max(e) <= 1.25 * min(e)
