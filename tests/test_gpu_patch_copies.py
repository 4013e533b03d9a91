"""Superiorized runs whose objective has no image of its own (L1, L2, linear) on
an image grid, with the one-pass sweep in the patch numbering: the row pass has
to gather the perturbed iterate, not an older copy of it (Algorithm 1's z is
the sweep's input).  Against the FP64 oracle at the suite's bound for a few
superiorized iterations (1e-4 relative L2; a stale copy is off by parts of 1).

Sizes on both sides of the automatic choice of the whole-GPU phase, in one
block (the box step writes no copies) and several, with an accepted step and
with none (every trial refused), and a range too large for the phase's shared
memory.
"""
import numpy as np
import pytest

import oracle as O
import paper_2606_27086_gb300 as pk
import synth
from tests.helpers import random_x, rel, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

KINDS = {"l1": (pk.SUPPY_OBJ_L1, O.OBJ_L1), "l2": (pk.SUPPY_OBJ_L2, O.OBJ_L2),
         "linear": (pk.SUPPY_OBJ_LINEAR, O.OBJ_LINEAR), "tv": (pk.SUPPY_OBJ_TV_ISO, O.OBJ_TV_ISO)}


def _run(prob, kind, mode=O.CIMMINO, iters=3, gamma=0.5, max_trials=100, **kw):
    H, W = prob.shape
    n = H * W
    if kind == "linear":
        prob.c_lin = np.random.default_rng(3).uniform(0.0, 1.0, n).astype(np.float32) / n
    obj, okind = KINDS[kind]
    ctx = pk.from_problem(prob, mode=mode, obj=obj, strategy=pk.STRATEGY_ONE_PASS, **kw)
    assert ctx.suppy_info_get()["scatter_patch"] == 1
    x0 = random_x(n, 1, seed=8, lo=0.1, hi=0.5)
    ctx.suppy_set_x(x0)
    P = dict(gamma=gamma, alpha=0.9, n_red=2, max_trials=max_trials, max_sweeps=iters)
    st = ctx.suppy_run(pk.suppy_params_default(**P))[0]
    xg = ctx.suppy_get_x()
    ph, _ = ctx.suppy_history()
    ctx.close()
    S, l, u, lo, hi = O.from_problem(prob, mode)
    ob = {"linear": lambda: O.Objective(okind, c=prob.c_lin), "tv": lambda: O.Objective(okind, prob.shape)}.get(
        kind, lambda: O.Objective(okind))()
    x0 = np.clip(x0.astype(np.float64), prob.box_lo, prob.box_hi)
    r = O.run(S, mode, l, u, lo, hi, ob, O.Params(**P), x0=x0)
    assert st["accepted"] == sum(r.accepted)
    for k in range(iters):
        assert rel(ph[k], r.prox_hist[k]) <= 1e-3
    assert rel_l2(xg, r.x) <= 1e-4
    return st


@pytest.mark.parametrize("mode", [O.CIMMINO, O.BIP, O.DROP])
@pytest.mark.parametrize("kind", ["l1", "l2", "linear", "tv"])
@pytest.mark.parametrize("shape", [(200, 333), (300, 260), (187, 201)])
def test_sweep_reads_the_perturbed_iterate(shape, kind, mode):
    prob = synth.seismic_problem(*shape, 24, 60, nrhs=1)
    if mode == O.BIP:
        prob.blocks = (np.arange(prob.A.m) % 3).astype(np.int32)
    _run(prob, kind, mode)


@pytest.mark.parametrize("form", [dict(perturb_path=1), dict(perturb_path=2),
                                  dict(perturb_path=2, scatter_transpose=2)])
@pytest.mark.parametrize("kind", ["l1", "l2"])
def test_both_phases_and_the_streamed_patch_form(kind, form):
    _run(synth.seismic_problem(139, 151, 24, 60, nrhs=1), kind, **form)


def test_every_trial_refused():
    """A step past the minimum of ||x||_2^2 raises it: y stays as it is."""
    st = _run(synth.seismic_problem(200, 333, 24, 60, nrhs=1), "l2", gamma=1e6, max_trials=3)
    assert st["accepted"] == 0


@pytest.mark.parametrize("kind", ["l1", "linear"])
def test_range_beyond_shared_memory(kind):
    """4.2 M unknowns: the whole-GPU phase that keeps y and g in L2."""
    H, W = 2050, 2052
    rng = np.random.default_rng(5)
    rows, k = 24, 2000
    along = (np.arange(12) * 83 + 7)[:, None] * W + 11 + np.arange(k)      # runs along image rows
    down = (np.arange(k) + 20)[None, :] * W + (np.arange(12) * 83 + 7)[:, None]   # and down columns
    col = np.concatenate([along, down]).astype(np.int32).ravel()
    A = synth.CSR(rows, H * W, np.arange(0, rows * k + 1, k, dtype=np.int32), col,
                  rng.uniform(0.1, 1.0, rows * k).astype(np.float32))
    b = A.to_scipy() @ np.full(H * W, 0.4)
    l, u = synth.slab_bounds(b, 0.03)
    prob = synth.Problem("range", A, l, u, np.zeros(1, np.float32), np.ones(1, np.float32), shape=(H, W))
    _run(prob, kind, iters=2)
