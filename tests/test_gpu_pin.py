"""A tuned launch configuration rebuilt without timing from the pin that bench.py
reports for it, strips included: the same form, grid and numbering."""
import pytest

import bench
import paper_2606_27086_gb300 as pk
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

SAME = ("strategy", "block", "grid", "lanes_per_row", "col_grid", "col_lanes", "transposed_rows", "scatter_patch")


@pytest.mark.parametrize("kw", [{}, dict(strategy=pk.STRATEGY_ONE_PASS), dict(strategy=pk.STRATEGY_TWO_PASS)])
@pytest.mark.parametrize("size", [(64, 90, 91), (256, 120, 363)])
def test_pin_rebuilds_the_tuned_form(size, kw):
    prob = synth.ct_problem(*size)
    tuned = pk.from_problem(prob, tune=1, **kw)
    want = tuned.suppy_info_get()
    tuned.close()
    if want["strategy"] != pk.STRATEGY_TILED and want["block"] == 256:
        pytest.skip("register-fed: no streaming form to pin")
    ctx = pk.from_problem(prob, **bench.pinned_opts(pk, bench.pin_of(want)))
    got = ctx.suppy_info_get()
    ctx.close()
    assert {k: got[k] for k in SAME} == {k: want[k] for k in SAME}
