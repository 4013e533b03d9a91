"""The sums of the strip-ordered passes are at least as close to FP64 as those of
the passes they stand in for.  DROP's corrections are large enough beside x
for the distance from the oracle to show the sums and not only the rounding of
x; the two-pass sweep is bitwise reproducible, so the comparison is exact.
One pass on small images: the staged scatter's corrections are sums of the CTAs'
sums, and so are the strips'.  The order of the reductions varies, the means
below lie 9 and 39% apart.
"""
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


@pytest.mark.parametrize("size", [(64, 90, 91), (128, 90, 183)])
def test_one_pass_strips_no_further_off_than_the_staged_scatter(size):
    prob = synth.ct_problem(*size)
    staged = _error(prob, O.DROP, pk.STRATEGY_ONE_PASS, 2, False, tma=-1)
    assert _error(prob, O.DROP, pk.STRATEGY_ONE_PASS, 2, True) <= staged


@pytest.mark.parametrize("n", [1, 2, 3, 5, 63, 64, 257, 4095, 16381, 16384, 16385])
@pytest.mark.parametrize("m", [1, 600])
def test_copies_of_the_accumulator_at_the_edges(m, n):
    """Unknowns that are no multiple of four (the copies' distance is), fewer
    strips than copies, and one unknown beyond the form; DROP's iterates against
    the oracle at the suite's 1e-5;
    the copies are back at zero for the second sweep."""
    prob = synth.random_problem(m, n, seed=n + m, mean_len=min(n, 20))
    ctx = pk.from_problem(prob, mode=O.DROP, strategy=pk.STRATEGY_ONE_PASS)
    x0 = random_x(n, 1, seed=9)
    ctx.suppy_set_x(x0)
    ctx.suppy_sweep(pk.suppy_params_default(), 2)
    xg = ctx.suppy_get_x()
    ctx.close()
    S, l, u, lo, hi = O.from_problem(prob, O.DROP)
    x = np.clip(x0.astype(np.float64), lo, hi)
    for _ in range(2):
        x, _ = O.sweep(S, O.DROP, l, u, 1.0, lo, hi, x)
    assert rel_l2(xg, x) <= 1e-5
