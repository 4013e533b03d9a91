"""The sums of the strip-ordered passes are at least as close to FP64 as those of
the passes they stand in for.  DROP's corrections are large enough beside x
for the distance from the oracle to show the sums and not only the rounding of
x; the two-pass sweep is bitwise reproducible, so the comparison is exact."""
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

STRIP_BLOCK = 800


def _error(prob, mode, strategy, sweeps, strips, **kw):
    ctx = pk.from_problem(prob, mode=mode, strategy=strategy, **kw)
    assert (ctx.suppy_info_get()["block"] == STRIP_BLOCK) == strips
    S, l, u, lo, hi = O.from_problem(prob, mode)
    errs = []
    for seed in range(20, 26):
        x0 = random_x(prob.A.n, 1, seed=seed)
        ctx.suppy_set_x(x0)
        ctx.suppy_sweep(pk.suppy_params_default(), sweeps)
        xg = ctx.suppy_get_x()
        x = np.clip(x0.astype(np.float64), lo, hi)
        for _ in range(sweeps):
            x, _ = O.sweep(S, mode, l, u, 1.0, lo, hi, x)
        errs.append(rel_l2(xg, x))
    ctx.close()
    return float(np.mean(errs))


@pytest.mark.parametrize("size", [(257, 181, 367), (128, 90, 183)])
def test_two_pass_strips_no_further_off_than_streamed_passes(size):
    prob = synth.ct_problem(*size)
    streamed = _error(prob, O.DROP, pk.STRATEGY_TWO_PASS, 2, False, stream_map=1)
    assert _error(prob, O.DROP, pk.STRATEGY_TWO_PASS, 2, True) <= streamed
