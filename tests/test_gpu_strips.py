"""The strip-ordered passes (rows and columns of A stored four at a time in
packets of 128 slots) against the FP64 oracle: Eq. (3)'s sweep, one per
strategy.  One sweep's bound is the suite's 1e-5 relative L2 (FP32 sums of a
few hundred terms: about 1e-7 relative each).

The sizes sit at the edges of the layout: rows of 1, 31 .. 33 and 127 .. 129
entries (a packet holds 32 of a row), blocks whose size is not a multiple of
four, empty rows and columns, unsorted column indices, rows whose entries lie
further apart than a 16-bit offset reaches, matrices too ragged for the form and
small ones of the same shape, which take it.
"""
import numpy as np
import pytest

import oracle as O
import paper_2606_27086_gb300 as pk
import synth
from tests.helpers import random_x, rel, rel_l2, rounded_values

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

STRIP_BLOCK = 800   # threads per CTA of the strip-ordered passes
STRATS = [pk.STRATEGY_ONE_PASS, pk.STRATEGY_TWO_PASS]


def _problem(lens, n, seed, spread=1):
    """Rows of the given lengths: runs of columns `spread` apart that start one
    column further from row to row, as rays and dose rows have them."""
    rng = np.random.default_rng(seed)
    cols = [(i % max(1, n - k * spread) + np.arange(k) * spread).astype(np.int32) for i, k in enumerate(lens)]
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    col = np.concatenate(cols)
    A = synth.CSR(len(lens), n, rp, col, rng.uniform(0.1, 1.0, len(col)).astype(np.float32))
    b = A.to_scipy() @ rng.uniform(0.0, 1.0, n) * (1 + 0.2 * rng.standard_normal(len(lens)))
    l, u = synth.slab_bounds(b, 0.03)
    return synth.Problem("strips", A, l, u, np.zeros(1, np.float32), np.ones(1, np.float32))


def _check(prob, strategy, mode=O.CIMMINO, dtype="f32", strips=True, sweeps=2, **kw):
    dt = {"f32": pk.SUPPY_F32, "bf16": pk.SUPPY_BF16, "f16": pk.SUPPY_F16}[dtype]
    ctx = pk.from_problem(prob, mode=mode, dtype=dt, strategy=strategy, **kw)
    info = ctx.suppy_info_get()
    assert info["strategy"] == strategy
    if strips is not None:
        assert (info["block"] == STRIP_BLOCK) == strips
    x0 = random_x(prob.A.n, 1, seed=5)
    ctx.suppy_set_x(x0)
    ctx.suppy_sweep(pk.suppy_params_default(lam=1.2), sweeps)
    xg = ctx.suppy_get_x()
    ph, _ = ctx.suppy_history()
    ctx.close()
    S, l, u, lo, hi = O.from_problem(prob, mode, values=rounded_values(prob.A.val, dtype))
    x = np.clip(x0.astype(np.float64), lo, hi)   # set_x projects onto the box
    for k in range(sweeps):
        x, p = O.sweep(S, mode, l, u, 1.2, lo, hi, x)
        assert rel(ph[k], p) <= 1e-5
    assert rel_l2(xg, x) <= 1e-5
    return xg


def _takes_strips(prob, strategy, **kw):
    ctx = pk.from_problem(prob, strategy=strategy, **kw)
    got = ctx.suppy_info_get()["block"] == STRIP_BLOCK
    ctx.close()
    return got


@pytest.mark.parametrize("strategy", STRATS)
@pytest.mark.parametrize("length", [1, 31, 32, 33, 64, 127, 129, 500])
@pytest.mark.parametrize("m,n", [(1, 700), (5, 3001), (601, 20011)])
def test_row_lengths_at_packet_edges(m, n, length, strategy):
    """One entry a row fills an eighth of its slots, and 33 take two packets;
    packets this few are taken all the same."""
    prob = _problem([length] * m, n, seed=length + m)
    got = _takes_strips(prob, strategy)
    assert got
    _check(prob, strategy, strips=got)


@pytest.mark.parametrize("strategy", STRATS)
@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("mode", [O.CIMMINO, O.BIP, O.DROP])
def test_image_grids(mode, dtype, strategy):
    """Rays on a grid whose sides are no multiples of eight, in blocks of a
    size that is no multiple of four."""
    prob = synth.ct_problem(133, 150, 189)
    if mode == O.BIP:
        prob.blocks = synth.angle_blocks(150, 189, 3)
    # a block's columns have a third of the entries: too ragged in BIP
    _check(prob, strategy, mode, dtype, strips=None if (mode, strategy) == (O.BIP, 2) else True)


@pytest.mark.parametrize("mode", [O.EL, O.EMR])
def test_extrapolated_steps(mode):
    _check(synth.ct_problem(131, 150, 187), pk.STRATEGY_TWO_PASS, mode, sweeps=1)


@pytest.mark.parametrize("strategy", STRATS)
def test_empty_rows_and_columns(strategy):
    """Rows without entries between full ones; columns no row touches still
    take the box."""
    lens = [200, 0, 200, 200, 0, 0, 0, 0, 200, 200, 200, 200] * 40
    prob = _problem(lens, 5000, seed=3)
    prob.box_lo = np.full(1, 0.3, np.float32)
    empty = np.asarray(lens) == 0
    prob.l[empty], prob.u[empty] = -1.0, 1.0
    strips = _takes_strips(prob, strategy)
    if strategy == pk.STRATEGY_ONE_PASS:
        assert strips
    x = _check(prob, strategy, strips=strips, sweeps=1)
    assert np.all(x >= np.float32(0.3))


@pytest.mark.parametrize("strategy", STRATS)
def test_unsorted_rows(strategy):
    prob = synth.ct_problem(130, 150, 185)
    rng = np.random.default_rng(9)
    rp = prob.A.row_ptr
    for i in range(prob.A.m):
        o = rng.permutation(np.arange(rp[i], rp[i + 1]))
        prob.A.col[rp[i]:rp[i + 1]], prob.A.val[rp[i]:rp[i + 1]] = prob.A.col[o], prob.A.val[o]
    _check(prob, strategy)


def test_offsets_beyond_sixteen_bits():
    """Entries 2100 columns apart: 31 of them fit a packet's offsets, so its
    windows are cut by the offsets, not by the slots; 4000 apart, 16 fit and
    the other forms take the matrix once its packets are more than 8 MB."""
    _check(_problem([310] * 64, 1 << 20, seed=12, spread=2100), pk.STRATEGY_ONE_PASS, strips=True)
    _check(_problem([200] * 64, 1 << 20, seed=11, spread=4000), pk.STRATEGY_ONE_PASS, strips=True)
    _check(_problem([200] * 4800, 1 << 20, seed=11, spread=4000), pk.STRATEGY_ONE_PASS, strips=False)


@pytest.mark.parametrize("m,n,strips", [(1, 3, True), (5, 40, True), (700, 20011, True), (80000, 20011, False)])
@pytest.mark.parametrize("strategy", STRATS)
def test_ragged_rows_take_the_other_forms_unless_small(m, n, strips, strategy):
    _check(synth.random_problem(m, n, seed=4, mean_len=3), strategy, strips=strips)


def test_fixed_forms_stay_fixed():
    """A caller-fixed streaming shape, lane map or pixel numbering, or the
    register-fed kernels, are taken as asked."""
    prob = synth.ct_problem(133, 150, 189)
    for kw in (dict(tma=-1), dict(stream_shape=(1024, 8, 32)), dict(stream_map=1),
               dict(scatter_transpose=2), dict(scatter_transpose=-1)):
        _check(prob, pk.STRATEGY_ONE_PASS, strips=False, **kw)


def test_two_pass_strips_are_bitwise_reproducible():
    prob = synth.ct_problem(133, 150, 189)
    a = _check(prob, pk.STRATEGY_TWO_PASS)
    assert np.array_equal(a, _check(prob, pk.STRATEGY_TWO_PASS))
