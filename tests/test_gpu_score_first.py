"""Steps of many tokens that reuse attention outputs project the scoring head of every token first and the other queries of
the refresh set only: against the oracle's arithmetic on the stored operands (tests/rounding.py: over the 10^7 elements of the
O cache here the storage format alone passes the plain oracle's max-abs gate, 4.0e-2, by a tenth) on both sides of the gate between listed and dense projections, after steps
that left other queries behind, with scoring heads in either half of a column tile."""
import numpy as np
import pytest

from paper_2605_08134_b200 import workloads as wl
from tests import parity, rounding

pytestmark = pytest.mark.gpu

CASES = [
    # d_model, head_dim, batch, seq, window, score_head
    (4096, 128, 1, 1153, 0, 31),      # just past the smallest: ten row tiles, the last of one row
    (4096, 128, 2, 1201, 0, 1),       # output reuse takes it too; tiles run on across sequences
    (2048, 64, 9, 520, 488, 3),       # heads of 64, windows that are no multiple of 32 rows
    (2048, 64, 16, 288, 256, 16),     # windows of whole row tiles
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_score_first(case):
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    d_model, hd, batch, seq, window, head = CASES[case]
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
    g.close()
