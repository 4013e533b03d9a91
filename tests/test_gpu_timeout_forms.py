"""Bounded waits that run out in each form of the streaming sweep: the streamed
passes and the strips, one and two passes, and row strips beside streamed
columns.  As in test_gpu_timeout.py: a budget of one cycle makes a wait give up,
the next synchronizing call says SUPPY_ETIMEOUT, and with the default budget the
same context computes what the oracle computes."""
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

STRIP_BLOCK, STREAM_BLOCK = 800, 768
ONE, TWO = pk.STRATEGY_ONE_PASS, pk.STRATEGY_TWO_PASS


@pytest.mark.parametrize("mode,strategy,kw,block", [(O.CIMMINO, TWO, dict(stream_map=1), STREAM_BLOCK),
                                                    (O.CIMMINO, TWO, dict(stream_map=2), STREAM_BLOCK),
                                                    (O.CIMMINO, ONE, {}, STRIP_BLOCK),
                                                    (O.CIMMINO, TWO, {}, STRIP_BLOCK),
                                                    (O.BIP, ONE, {}, STRIP_BLOCK),
                                                    (O.BIP, TWO, {}, STRIP_BLOCK)])
def test_wait_runs_out_and_context_recovers(mode, strategy, kw, block):
    """BIP in two passes: the columns of a block are too ragged for strips and
    streamed, the rows are not."""
    prob = synth.ct_problem(160, 60, 227)
    prob.blocks = synth.angle_blocks(60, 227, 6)
    ctx = pk.from_problem(prob, mode=mode, strategy=strategy, **kw)
    info = ctx.suppy_info_get()
    assert info["block"] == block and info["tma"] == 1
    if mode == O.BIP and strategy == TWO:
        assert info["col_lanes"] == 4   # strips have eight
    ctx.suppy_set_x(random_x(prob.A.n, 1, seed=31))
    ctx.suppy_set_wait_limit(1)
    with pytest.raises(pk.SuppyError) as e:
        ctx.suppy_sweep(pk.suppy_params_default(use_graphs=0), 1)
        ctx.suppy_get_x()
    assert e.value.status == pk.SUPPY_ETIMEOUT
    ctx.suppy_set_wait_limit(0)
    S, l, u, lo, hi = O.from_problem(prob, mode)
    for seed in (32, 33):
        x = random_x(prob.A.n, 1, seed=seed)
        ctx.suppy_set_x(x)
        ctx.suppy_sweep(pk.suppy_params_default(use_graphs=0), 1)
        xo, _ = O.sweep(S, mode, l, u, 1.0, lo, hi, x.astype(np.float64))
        assert rel_l2(ctx.suppy_get_x(), xo) <= 1e-5
    ctx.close()
