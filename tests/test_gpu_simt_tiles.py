"""CUDA-core kernels at the edges of their tiles against the fp64 oracle: every head width, widths that leave a partial
column tile or k-block, row counts just past a tile, all five tile heights of the projections, all four forms of the
attention kernel (row groups x key groups) at every head width, key counts around a key block."""
import numpy as np
import pytest

from paper_2605_08134_b200 import workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu

CASES = [
    # dtype, d_model, head_dim, batch, seq, prompt, scoring head
    (wl.DTYPE_F32, 96, 32, 1, 33, 16, 2),
    (wl.DTYPE_F32, 160, 32, 3, 65, 20, 4),
    (wl.DTYPE_F32, 192, 64, 2, 129, 1, 1),
    (wl.DTYPE_F32, 384, 128, 1, 31, 7, 2),
    (wl.DTYPE_F32, 256, 256, 2, 50, 17, 0),
    (wl.DTYPE_F32, 1024, 64, 3, 257, 100, 3),
    (wl.DTYPE_F32, 512, 128, 2, 300, 44, 1),
    (wl.DTYPE_BF16, 96, 32, 2, 47, 16, 1),
    (wl.DTYPE_BF16, 512, 256, 1, 161, 60, 1),
    (wl.DTYPE_BF16, 320, 64, 2, 97, 33, 4),
    # forms of the attention kernel's dense steps that the cases above do not reach
    (wl.DTYPE_F32, 64, 32, 25, 65, 20, 1),       # 2 x 2
    (wl.DTYPE_F32, 96, 32, 25, 33, 7, 2),        # 3 x 1
    (wl.DTYPE_F32, 32, 32, 38, 300, 50, 0),      # 4 x 1
    (wl.DTYPE_F32, 64, 64, 38, 300, 50, 0),
    (wl.DTYPE_F32, 128, 128, 1, 33, 16, 0),      # 2 x 2
    (wl.DTYPE_BF16, 256, 128, 32, 193, 60, 1),   # 4 x 1
    (wl.DTYPE_F32, 768, 256, 25, 33, 8, 2),      # 2 x 2
    (wl.DTYPE_BF16, 768, 256, 25, 65, 9, 1),     # 3 x 1
    (wl.DTYPE_F32, 1024, 256, 28, 97, 30, 3),    # 4 x 1
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_steps_at_tile_edges(case):
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    dtype, d_model, hd, batch, seq, prompt, head = CASES[case]
    shape = wl.scaled(wl.TINY_F32, dtype=dtype, d_model=d_model, n_heads=d_model // hd, head_dim=hd, batch=batch, seq=seq,
                      prompt=prompt)
    w = wl.make_weights(shape, 900 + case)
    hs = wl.HiddenStream(shape, 900 + case)
    g = dare.Layer(shape, w, kernel_path=dare.PATH_SIMT, score_head=head)
    o = parity.oracle_layer(shape, w, score_head=head)
    parity.compare_step(g, o, hs.first(), 3, 0.1, shape, first=True)
    for mode, frac, window in [(3, 0.1, False), (1, 0.5, True), (2, 0.03, True), (3, 1.0, False)]:
        x = hs.advance(wl.uniform_positions(hs.rng, shape, max(1, int(round(frac * seq)))))
        pb = prompt if window else 0
        parity.compare_step(g, o, np.ascontiguousarray(x[:, pb:]), mode, 0.1, shape, pos_begin=pb)
    g.close()
