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
    (4096, 9, 256, 128),     # more than one wave
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


FORMS = [
    # d_model, head_dim, batch, seq, window: the form it is here for.  (Of a window of a multiple of 32 rows the output
    # projection fetches its rows in boxes of 32.)
    (768, 64, 41, 150, 0),       # K/V: persistent single-CTA tiles, across sequences
    (1024, 128, 37, 257, 128),   # ... inside them
    (768, 128, 16, 100, 0),      # K/V: wide tiles split in two
    (768, 64, 13, 129, 122),
    (3072, 128, 7, 129, 122),    # K/V: wide tiles
    (256, 64, 19, 257, 250),     # Q: narrow tiles
    (1536, 64, 1, 257, 0),       # Q: wide tiles split in two
    (1536, 128, 7, 129, 122),    # Q: wide pairs split in two
    (1280, 128, 9, 57, 50),      # output: wide tiles split in two
    (256, 128, 37, 200, 160),    # output, boxes of 32: narrow tiles
    (512, 64, 29, 100, 96),      # narrow pairs
    (1280, 64, 11, 100, 96),     # wide tiles split in two
    (1536, 64, 9, 100, 96),      # wide pairs split in two
    (768, 128, 37, 100, 96),     # wide pairs
    (768, 64, 41, 200, 160),     # persistent pairs
    (2048, 128, 29, 200, 160),   # persistent single-CTA tiles
    (2048, 64, 29, 200, 160),
]


@pytest.mark.parametrize("case", range(len(FORMS)))
def test_forms_of_the_projections(case):
    """Dense, K/V reuse and output reuse over the window: every form a projection takes (tile width, pairs, reduction split,
    persistent kernel) with row tiles that end with their sequence and with tiles that run on."""
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    d_model, hd, batch, seq, window = FORMS[case]
    shape = wl.scaled(wl.LLADA_LAYER, d_model=d_model, n_heads=d_model // hd, head_dim=hd, batch=batch, seq=seq, prompt=seq // 2)
    w = wl.make_weights(shape, 1300 + case)
    hs = wl.HiddenStream(shape, 1300 + case)
    g = dare.Layer(shape, w, kernel_path=dare.PATH_TENSOR, score_head=case % 3)
    o = parity.oracle_layer(shape, w, score_head=case % 3)
    parity.compare_step(g, o, hs.first(), 3, 0.1, shape, first=True)
    at = seq - window if window else 0
    for mode, frac in [(0, 0.1), (1, 0.2), (2, 0.5)]:
        x = hs.advance(wl.uniform_positions(hs.rng, shape, max(1, int(round(frac * seq)))))
        parity.compare_step(g, o, np.ascontiguousarray(x[:, at:]), mode, 0.1, shape, pos_begin=at)
    g.close()
