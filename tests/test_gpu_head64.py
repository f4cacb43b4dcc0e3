"""Heads of 64 on the tensor-core path against the fp64 oracle, at sizes that walk across the launch rules of its kernels
(narrow and wide MMA pairs, split reductions, the persistent projections dense and listed, key split, one and two query
tiles per attention CTA), with the scoring head in either half of a 128-column piece."""
import numpy as np
import pytest

from paper_2605_08134_b200 import workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu

CASES = [
    # d_model, batch, seq, prompt, scoring head
    (256, 1, 57, 20, 1),
    (256, 1, 2300, 252, 0),      # key split
    (512, 2, 128, 32, 3),        # narrow pair tiles
    (512, 5, 1031, 7, 7),        # gathered output projection, 256-wide gathered tiles
    (1024, 8, 1153, 129, 2),     # two query tiles per attention CTA
    (512, 16, 1153, 100, 5),     # persistent projections
    (1024, 3, 120, 20, 15),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_steps_with_heads_of_64(case):
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    d_model, batch, seq, prompt, head = CASES[case]
    shape = wl.scaled(wl.LLADA_LAYER, d_model=d_model, n_heads=d_model // 64, head_dim=64, batch=batch, seq=seq, prompt=prompt)
    w = wl.make_weights(shape, 700 + case)
    hs = wl.HiddenStream(shape, 700 + case)
    g = dare.Layer(shape, w, kernel_path=dare.PATH_TENSOR, score_head=head)
    o = parity.oracle_layer(shape, w, score_head=head)
    parity.compare_step(g, o, hs.first(), 3, 0.1, shape, first=True)
    for step, (mode, frac, window) in enumerate([(3, 0.13, False), (1, 0.4, True), (2, 0.05, False), (3, 1.0, True)]):
        n = max(1, int(round(frac * seq)))
        x = hs.advance(wl.uniform_positions(hs.rng, shape, n))
        pb = prompt if window else 0
        parity.compare_step(g, o, np.ascontiguousarray(x[:, pb:]), mode, 0.1, shape, pos_begin=pb)
    g.close()
