"""The tile-resident perturbation phase (Algorithm 1) on images whose sides
do not divide into its rectangles, against the FP64 oracle: single rows and
columns, rectangles of a pixel or two, images just above one CTA's share, the
largest the whole-GPU form keeps in shared memory and one beyond it.  Both
forms (whole GPU 2, cluster 1), several reduction steps (the halo is read anew
between them) and trials that are refused.  Accepted steps, trials and
exponent equal the oracle's; the point agrees as elsewhere in the suite
(1e-5 relative L2: FP32 steps along a unit vector)."""
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

KINDS = {"tv": (pk.SUPPY_OBJ_TV_ISO, O.OBJ_TV_ISO), "atv": (pk.SUPPY_OBJ_TV_ANISO, O.OBJ_TV_ANISO),
         "l1": (pk.SUPPY_OBJ_L1, O.OBJ_L1), "l2": (pk.SUPPY_OBJ_L2, O.OBJ_L2)}


def _phase(shape, kind, path, P, seed=7):
    H, W = shape
    n = H * W
    rng = np.random.default_rng(seed)
    m, k = 8, min(4, n)
    A = synth.CSR(m, n, np.arange(0, m * k + 1, k, dtype=np.int32),
                  np.tile(np.arange(k, dtype=np.int32), m), rng.uniform(0.1, 1, m * k).astype(np.float32))
    prob = synth.Problem("img", A, np.full(m, -9, np.float32), np.full(m, 9, np.float32),
                         np.zeros(1, np.float32), np.ones(1, np.float32), shape=shape)
    x0 = random_x(n, 1, seed=seed)
    obj, okind = KINDS[kind]
    ctx = pk.from_problem(prob, obj=obj, perturb_path=path)
    ctx.suppy_set_x(x0)
    acc = ctx.suppy_perturb(pk.suppy_params_default(**P))
    st = ctx.suppy_run(pk.suppy_params_default(max_sweeps=0))[0]
    xg = ctx.suppy_get_x()
    ctx.close()
    ost = O.PertState()
    ob = O.Objective(okind) if kind in ("l1", "l2") else O.Objective(okind, shape)
    y, a, t = O.perturbation_phase(ob, x0.astype(np.float64), ost, O.Params(**P))
    assert acc[0] == a and st["trials"] == t and st["ell"] == ost.ell
    assert rel_l2(xg, y) <= 1e-5


@pytest.mark.parametrize("path", [1, 2])
@pytest.mark.parametrize("kind", ["tv", "atv", "l1", "l2"])
@pytest.mark.parametrize("shape", [(1, 1), (1, 37), (41, 1), (2, 3), (3, 700), (700, 3), (17, 23), (151, 153),
                                   (257, 129)])
def test_shapes(shape, kind, path):
    _phase(shape, kind, path, dict(gamma=0.8, alpha=0.9, n_red=3, max_trials=30))


@pytest.mark.parametrize("path", [1, 2])
@pytest.mark.parametrize("gamma,alpha,max_trials", [(400.0, 0.9, 100), (400.0, 0.9, 5), (1e-6, 0.5, 20)])
def test_refused_and_vanishing_steps(gamma, alpha, max_trials, path):
    """Large steps pass after dozens of refusals (or not at all); steps below
    an ulp of y leave it unchanged and pass, f(z) being f(y) exactly."""
    _phase((61, 67), "tv", path, dict(gamma=gamma, alpha=alpha, n_red=4, max_trials=max_trials))


@pytest.mark.parametrize("shape", [(1500, 1700), (2100, 2300)])
def test_large_images(shape):
    """The whole-GPU form up to its shared-memory size, and beyond it (the
    form that keeps y and g in L2)."""
    _phase(shape, "tv", 0, dict(gamma=5.0, alpha=0.9, n_red=2, max_trials=20))
