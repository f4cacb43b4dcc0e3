"""Row tiles that run on across sequences, and the one-wave forms of the projections (narrow tiles, reduction split in
four, pairs or not), against the fp64 oracle: windows of a multiple of 32 rows, ragged windows, batches whose tiles end
inside a sequence."""
import numpy as np
import pytest

from paper_2605_08134_b200 import workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu

CASES = [
    # d_model, batch, seq, window
    (512, 4, 96, 32),        # one tile of four windows
    (1024, 5, 200, 32),      # two tiles
    (256, 3, 224, 160),      # windows of more than a tile
    (512, 3, 150, 70),       # ragged windows: the output projection's tiles end with their sequence
    (4096, 2, 70, 32),       # one row tile, reduction split in four
    (2048, 1, 130, 64),
    (1024, 7, 333, 0),       # whole sequences, tiles ending inside them
    (4096, 9, 256, 128),     # more than one wave: persistent, output rows in boxes of 32
    (512, 6, 1100, 1056),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_windows_across_sequences(case):
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    d_model, batch, seq, window = CASES[case]
    shape = wl.scaled(wl.LLADA_LAYER, d_model=d_model, n_heads=d_model // 128, batch=batch, seq=seq, prompt=seq // 2)
    w = wl.make_weights(shape, 1200 + case)
    hs = wl.HiddenStream(shape, 1200 + case)
    g = dare.Layer(shape, w, kernel_path=dare.PATH_TENSOR)
    o = parity.oracle_layer(shape, w)
    parity.compare_step(g, o, hs.first(), 3, 0.1, shape, first=True)
    pb = seq - window if window else 0
    for i, (mode, frac) in enumerate([(3, 0.2), (1, 0.05), (2, 0.5), (0, 0.1)]):
        x = hs.advance(wl.uniform_positions(hs.rng, shape, max(1, int(round(frac * seq)))))
        at = pb if i < 3 or not window else max(0, pb - 7)       # (the last one at an odd place)
        act = seq - pb
        parity.compare_step(g, o, np.ascontiguousarray(x[:, at:at + act]), mode, 0.1, shape, pos_begin=at)
    g.close()
