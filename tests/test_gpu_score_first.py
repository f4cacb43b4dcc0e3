"""Steps of many tokens that reuse attention outputs project the scoring head of every token first and the other queries of
the refresh set only: against the oracle's arithmetic on the stored operands (tests/rounding.py: over the 10^7 elements of the
O cache here the storage format alone passes the plain oracle's max-abs gate, 4.0e-2, by a tenth) on both sides of the gate between listed and dense projections, after steps
that left other queries behind, with scoring heads in either half of a column tile; steps given a reuse rate; layers of a stack.
Every step is checked to have taken the schedule that its case is about."""
import numpy as np
import pytest

from paper_2605_08134_b200 import workloads as wl
from tests import parity, rounding

pytestmark = pytest.mark.gpu

CASES = [
    # d_model, head_dim, batch, seq, window, score_head, modes that take the schedule
    (4096, 128, 1, 1153, 0, 31, (3,)),     # just past the smallest: ten row tiles, the last of one row
    (4096, 128, 2, 1201, 0, 1, (2, 3)),    # output reuse takes it too; tiles run on across sequences
    (2048, 64, 9, 520, 488, 3, (3,)),      # heads of 64, windows that are no multiple of 32 rows
    (2048, 64, 16, 288, 256, 16, (3,)),    # windows of whole row tiles
]


def _dare():
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    return dare


def _score_first(layer):
    return bool(layer.forms() & _dare().FORM_SCORE_FIRST)


@pytest.mark.parametrize("case", range(len(CASES)))
def test_score_first(case):
    dare = _dare()
    d_model, hd, batch, seq, window, head, modes = CASES[case]
    shape = wl.scaled(wl.LLADA_LAYER, d_model=d_model, n_heads=d_model // hd, head_dim=hd, batch=batch, seq=seq, prompt=seq // 2)
    w = wl.make_weights(shape, 1500 + case)
    hs = wl.HiddenStream(shape, 1500 + case)
    g = dare.Layer(shape, w, kernel_path=dare.PATH_TENSOR, score_head=head)
    o = rounding.rounded_layer(shape, w, score_head=head)
    parity.compare_step(g, o, hs.first(), 3, 0.1, shape, first=True)
    at = seq - window if window else 0
    for mode, frac in [(3, 0.1), (2, 0.4), (3, 0.72), (3, 0.78), (2, 0.95), (1, 0.1), (3, 0.0)]:
        x = hs.advance(wl.uniform_positions(hs.rng, shape, max(1, int(round(frac * seq)))))
        parity.compare_step(g, o, np.ascontiguousarray(x[:, at:]), mode, 0.1, shape, pos_begin=at)
        assert _score_first(g) == (mode in modes)
    g.close()


def test_output_reuse_with_heads_of_64_in_windows():
    """Output reuse alone: the queries in a launch of their own ahead of the dense K and V, over windows (75 row tiles)."""
    dare = _dare()
    shape = wl.scaled(wl.LLADA_LAYER, d_model=2048, n_heads=32, head_dim=64, batch=40, seq=256, prompt=16)
    w = wl.make_weights(shape, 1600)
    hs = wl.HiddenStream(shape, 1600)
    g = dare.Layer(shape, w, kernel_path=dare.PATH_TENSOR, score_head=5)
    o = rounding.rounded_layer(shape, w, score_head=5)
    parity.compare_step(g, o, hs.first(), 2, 0.1, shape, first=True)
    for frac in (0.1, 0.9):
        x = hs.advance(wl.uniform_positions(hs.rng, shape, int(round(frac * shape.seq))))
        parity.compare_step(g, o, np.ascontiguousarray(x[:, 16:]), 2, 0.1, shape, pos_begin=16)
        assert _score_first(g)
    g.close()


class _GivenRate:
    """A layer whose step reuses as many tokens as were left nearly unchanged, by count instead of by threshold."""

    def __init__(self, layer, reuse):
        self.layer, self.reuse = layer, reuse

    def __getattr__(self, name):
        return getattr(self.layer, name)

    def step(self, x, mode, tau, pos_begin=0):
        return self.layer.step_quantile(x, mode, self.reuse, pos_begin=pos_begin)


def test_steps_that_know_what_they_refresh():
    """A given reuse rate of more than a quarter takes the schedule; a lower one, or a threshold below every score, does not, as
    all queries but a few are projected then."""
    dare = _dare()
    shape = wl.scaled(wl.LLADA_LAYER, d_model=4096, n_heads=32, batch=2, seq=1201, prompt=600)
    w = wl.make_weights(shape, 1700)
    hs = wl.HiddenStream(shape, 1700)
    g = dare.Layer(shape, w, kernel_path=dare.PATH_TENSOR)
    o = rounding.rounded_layer(shape, w)
    parity.compare_step(g, o, hs.first(), 3, 0.1, shape, first=True)
    for mode, frac, taken in [(3, 0.15, True), (2, 0.74, True), (3, 0.76, False), (2, 0.9, False), (3, 0.3, True)]:
        n = int(round(frac * shape.seq))
        x = hs.advance(wl.uniform_positions(hs.rng, shape, n))
        parity.compare_step(_GivenRate(g, 2 * (shape.seq - n)), o, x, mode, 0.1, shape)
        assert _score_first(g) == taken
    x = hs.advance(wl.uniform_positions(hs.rng, shape, 100))
    parity.compare_step(g, o, x, 3, -1.0, shape)
    assert not _score_first(g)
    g.close()


@pytest.mark.parametrize("d_model,seq,taken", [(1024, 1024, True), (768, 1824, False)])
def test_narrow_layers(d_model, seq, taken):
    """Below a width of 1024 the scoring head's launch costs too much of what it saves, however many tokens there are."""
    import torch
    dare = _dare()
    shape = wl.scaled(wl.LLADA_LAYER, d_model=d_model, n_heads=d_model // 128, batch=16, seq=seq, prompt=seq // 2)
    assert 2.0 * 16 * seq * d_model ** 2 > 34e9
    g = dare.Layer(shape, wl.make_weights(shape, 5), kernel_path=dare.PATH_TENSOR)
    x = torch.randn(16, seq, d_model, device="cuda").bfloat16()
    g.step(x, 3, 0.1)
    x[:, ::7].normal_()
    g.step(x, 3, 0.1)
    assert g.status() == 0 and _score_first(g) == taken
    assert g.last_selection(16, seq)["count"] == 16 * len(range(0, seq, 7))
    g.close()


def test_layers_of_a_stack():
    """Residual blocks: the projection reads its input again, and the compact copies of the schedule must not lie over it.  As in
    tests/test_gpu_stack.py at full size: a layer's input and state are taken from the GPU, one step of the oracle is run from there."""
    import torch
    dare = _dare()
    lay = wl.scaled(wl.LLADA_LAYER, d_model=4096, n_heads=32, seq=288, prompt=32, batch=5, block=16, seed=3)
    shape = wl.StackShape("wide", 2, lay, 512, 1024, 256, seed=3)
    w = wl.make_stack_weights(shape)
    g = dare.Stack(shape, w, 5)
    rng = np.random.default_rng(9)
    toks = rng.integers(0, shape.vocab - 1, (5, 288)).astype(np.int32)
    g.forward(torch.from_numpy(toks).cuda(), 288, 0, 3, [0.1, 0.1])
    xbuf = torch.empty((5, 256, 4096), dtype=torch.bfloat16, device="cuda")
    hbuf = torch.empty_like(xbuf)
    for l, frac in [(0, 0.1), (1, 0.9), (1, 0.3)]:
        change = rng.random((5, 288)) < frac
        change[:, :32] = False
        toks = np.where(change, (toks + 1 + rng.integers(0, shape.vocab - 2, toks.shape)) % (shape.vocab - 1), toks).astype(np.int32)
        view = g.layer(l)
        pre = view.read_caches(5, 288)
        g.set_capture(l, xbuf, hbuf)
        g.forward(torch.from_numpy(toks).cuda(), 256, 32, 3, [0.1, 0.1])
        torch.cuda.synchronize()
        g.set_capture(-1)
        assert view.status() == 0 and _score_first(view)
        o = rounding.rounded_layer(lay, w["layers"][l])
        o.has_prev, o.batch, o.kv_len = True, 5, 288
        o.q_prev[:] = pre["q_prev"]; o.k_cache[:] = pre["k"]; o.v_cache[:] = pre["v"]; o.o_cache[:] = pre["o"]
        x = xbuf.float().cpu().numpy()
        y = o.step(x, 3, 0.1, pos_begin=32)
        parity.check_margin(o.last_scores, 0.1)
        sel = view.last_selection(5, 256)
        np.testing.assert_array_equal(sel["idx"], o.last_idx)
        np.testing.assert_allclose(sel["scores"], o.last_scores, rtol=0, atol=parity.SCORE_ATOL[wl.DTYPE_BF16])
        parity.assert_close("h", hbuf.float().cpu().numpy(), x + y, parity.TOL_BF16)
        post = view.read_caches(5, 288)
        for name, want in (("k", o.k_cache), ("v", o.v_cache), ("o", o.o_cache)):
            parity.assert_close(name, post[name], want, parity.TOL_BF16, max_factor=2.0)
    g.close()
