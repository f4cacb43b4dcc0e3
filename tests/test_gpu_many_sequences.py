"""Steps over more sequences than one dimension of a launch can count (65535), on both kernel paths: the refresh set of
every sequence against the plan, the outputs of sequences on both sides of that number against the fp64 oracle (sequences
are independent, so an oracle of the picked ones is the oracle of the step)."""
import numpy as np
import pytest

from paper_2605_08134_b200 import workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu

CASES = [
    # dtype, d_model, head_dim, batch, seq
    (wl.DTYPE_F32, 32, 32, 65_600, 3),
    (wl.DTYPE_BF16, 256, 64, 65_600, 3),
    (wl.DTYPE_BF16, 256, 128, 65_600, 3),
]


def steps_of_many_sequences(dtype, d_model, head_dim, batch, seq, plan):
    import torch
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    shape = wl.scaled(wl.TINY_F32, dtype=dtype, d_model=d_model, n_heads=d_model // head_dim, head_dim=head_dim, batch=batch,
                      seq=seq, prompt=1)
    w = wl.make_weights(shape, 31)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(31)
    normal = lambda: torch.empty((batch, seq, d_model), device="cuda").normal_(0, 1, generator=gen)
    pick = np.unique(np.r_[0:4, 255:258, 32_766:32_770, 65_533:min(batch, 65_542), batch - 4:batch])
    x = normal()
    g = dare.Layer(shape, w)
    o = parity.oracle_layer(shape, w, max_batch=len(pick))
    for i, (mode, begin) in enumerate([(3, 0)] + plan):
        if i > 0:
            changed = torch.rand((batch, seq), generator=gen, device="cuda") < 0.3
            x = torch.where(changed[:, :, None], normal(), x + 1e-3 * normal())
        xd = x[:, begin:].to(g.tdtype).contiguous()
        y = g.step(xd, mode, 0.1, pos_begin=begin)
        yo = o.step(xd[torch.from_numpy(pick).cuda()].float().cpu().numpy(), mode, 0.1, pos_begin=begin)
        assert g.status() == 0
        sel = g.last_selection(batch, seq - begin)
        mask = np.ones((batch, seq - begin), bool) if i == 0 else changed[:, begin:].cpu().numpy()
        np.testing.assert_array_equal(sel["idx"], np.nonzero(mask.reshape(-1))[0])
        np.testing.assert_array_equal(sel["batch_off"][pick + 1] - sel["batch_off"][pick], mask[pick].sum(1))
        tol = parity.tol_of(dtype)
        parity.assert_close("y", y[torch.from_numpy(pick).cuda()].float().cpu().numpy(), yo, tol, rel_rms=tol)
    g.close()


@pytest.mark.parametrize("case", range(len(CASES)))
def test_steps_of_many_short_sequences(case):
    steps_of_many_sequences(*CASES[case], plan=[(3, 0), (1, 0), (3, 1)])


def test_steps_of_more_row_tiles_than_one_grid_dimension():
    """65600 row tiles of 96 in the CUDA-core projections."""
    steps_of_many_sequences(wl.DTYPE_F32, 32, 32, 65_600, 96, plan=[(3, 0)])
