"""A bounded device wait's budget covers that wait, not the kernel before: the
strip passes are launched while the perturbation phase still runs, and a phase
many times as long as the budget must not make them give up.  The host sees
only statuses; no wait here outlasts its limit by design."""
import numpy as np
import pytest

import paper_2606_27086_gb300 as pk
import synth
from tests.helpers import random_x, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

STRIP_BLOCK = 800


@pytest.mark.parametrize("strategy", [pk.STRATEGY_ONE_PASS, pk.STRATEGY_TWO_PASS])
@pytest.mark.parametrize("path", [1, 2])
def test_a_long_phase_does_not_use_up_the_strips_waits(strategy, path):
    """400 reduction steps of at least 5 us take millions of cycles; a ring
    that holds a third of the strips, and a wait in a pass or a barrier a few
    tens of thousands at most."""
    prob = synth.ct_problem(256, 180, 363)
    ctx = pk.from_problem(prob, obj=pk.SUPPY_OBJ_TV_ISO, strategy=strategy, perturb_path=path)
    assert ctx.suppy_info_get()["block"] == STRIP_BLOCK
    x0 = random_x(prob.A.n, 1, seed=3)
    P = pk.suppy_params_default(gamma=0.02, alpha=0.999, n_red=400, max_sweeps=2, use_graphs=0)
    out = []
    for limit in (0, 1_000_000):
        ctx.suppy_set_x(x0)
        ctx.suppy_set_wait_limit(limit)
        st = ctx.suppy_run(P)[0]
        assert st["accepted"] == 800
        out.append(ctx.suppy_get_x())
    ctx.close()
    assert np.all(np.isfinite(out[1]))
    assert rel_l2(out[1], out[0]) <= 1e-4   # the same iterations but for the order of the reductions
