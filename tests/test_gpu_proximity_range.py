"""The monitored proximity of the one-pass forms is an FP64 sum of FP64 terms (Eq.
(WeightedProximity)): squares of residuals far below the FP32 range are kept.
A problem scaled by 1e-15 .. 1e-21 has the proximity of the unscaled one times
the scale's square; the bound is the suite's 1e-5 (FP32 residuals)."""
import numpy as np
import pytest

import oracle as O
import paper_2606_27086_gb300 as pk
import synth
from tests.helpers import random_x, rel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _scaled(prob, scale):
    for name in ("l", "u", "box_lo", "box_hi"):
        setattr(prob, name, (getattr(prob, name).astype(np.float64) * scale).astype(np.float32))
    return prob


@pytest.mark.parametrize("scale", [1e-15, 1e-18, 1e-21])
@pytest.mark.parametrize("mode", [O.CIMMINO, O.BIP, O.DROP])
def test_small_units(mode, scale):
    prob = _scaled(synth.ct_problem(64, 90, 91), scale)
    if mode == O.BIP:
        prob.blocks = synth.angle_blocks(90, 91, 3)
    ctx = pk.from_problem(prob, mode=mode, strategy=pk.STRATEGY_ONE_PASS)
    x0 = (random_x(prob.A.n, 1, seed=6).astype(np.float64) * scale).astype(np.float32)
    ctx.suppy_set_x(x0)
    ctx.suppy_sweep(pk.suppy_params_default(prox_abs=0.0), 2)
    ph, _ = ctx.suppy_history()
    ctx.close()
    S, l, u, lo, hi = O.from_problem(prob, mode)
    x = np.clip(x0.astype(np.float64), lo, hi)
    for k in range(2):
        x, p = O.sweep(S, mode, l, u, 1.0, lo, hi, x)
        assert ph[k] > 0.0 and rel(ph[k], p) <= 1e-5
