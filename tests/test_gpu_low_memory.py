"""Device memory that runs short during suppy_create: strips are copies beside
the ones every form needs, so that a create which succeeds with the streamed
passes alone succeeds with default options or with tuning too.
Every allocation that fails is an ordinary status of cudaMalloc."""
import contextlib

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

MB = 1 << 20
STRIP_BLOCK = 800


@contextlib.contextmanager
def _left(mb):
    """About mb MB of free device memory."""
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(max(0, free - mb * MB), dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hog
        torch.cuda.empty_cache()


@pytest.fixture(scope="module")
def problem():
    prob = synth.ct_problem(256, 180, 363)
    x0 = random_x(prob.A.n, 1, seed=2)
    S, l, u, lo, hi = O.from_problem(prob)
    x, _ = O.sweep(S, O.CIMMINO, l, u, 1.0, lo, hi, x0.astype(np.float64))
    return prob, x0, x


def _create(problem, mb, **kw):
    """The form taken with mb MB left (threads per CTA of the row pass), or None
    when create ran out of memory; its sweep is checked."""
    prob, x0, x = problem
    with _left(mb):
        try:
            ctx = pk.from_problem(prob, **kw)
        except pk.SuppyError as e:
            assert "out of memory" in str(e), e
            return None
        block = ctx.suppy_info_get()["block"]
        ctx.suppy_set_x(x0)
        ctx.suppy_sweep(pk.suppy_params_default(use_graphs=0), 1)
        assert rel_l2(ctx.suppy_get_x(), x) <= 1e-5
        ctx.close()
    return block


@pytest.mark.parametrize("strategy", [pk.STRATEGY_ONE_PASS, pk.STRATEGY_TWO_PASS])
def test_strips_never_cost_a_create(problem, strategy):
    """One pass: against the patch numbering, which is the default without
    strips; two passes: against the streamed passes."""
    other = dict(scatter_transpose=2) if strategy == pk.STRATEGY_ONE_PASS else dict(stream_map=1)
    assert _create(problem, 4096, strategy=strategy, **other) != STRIP_BLOCK   # kernels loaded
    assert _create(problem, 4096, strategy=strategy) == STRIP_BLOCK
    forms = set()
    for mb in range(260, 680, 60):
        if _create(problem, mb, strategy=strategy, **other) is not None:
            form = _create(problem, mb, strategy=strategy)
            assert form is not None
            forms.add(form)
    assert len(forms) == 2   # the sizes lie on both sides


def test_tuned_create_keeps_a_form_that_fits(problem):
    """The tuner times the strips of one strategy, then the other's; what it
    chose has to fit again beside what it timed last.  The sizes lie around
    the sum of the matrix copies and both strategies' strips (about 770 MB)."""
    assert _create(problem, 8192, tune=1) is not None
    for mb in range(756, 788, 4):
        assert _create(problem, mb, tune=1) is not None
