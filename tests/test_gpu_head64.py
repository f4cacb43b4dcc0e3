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
    (512, 2, 128, 32, 3),        # narrow tiles split in four, K/V of the dense step in wide pairs
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


PRECISION = [
    # d_model, batch, seq: one tile a CTA; the same with the keys split over a cluster; two tiles a CTA
    (256, 1, 57), (256, 1, 2300), (1024, 8, 1153),
]


@pytest.mark.parametrize("d_model,batch,seq", PRECISION)
def test_attention_is_as_exact_as_its_storage(d_model, batch, seq):
    """The stored attention output against fp64 attention on the stored operands (the GPU's own K and V, Q rounded to bf16):
    softmax weights and sums in more than 16 bits leave nothing but the output's own rounding to bf16, whose relative error
    is measured beside it.  Weights in one bf16 part would add an error of the same size, independent of it (a factor of
    1.4); 1.05 leaves room for elements of Q that fp32 and fp64 round to different sides.  Dense step, then row-sparse."""
    import torch
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    hd, heads = 64, d_model // 64
    shape = wl.scaled(wl.LLADA_LAYER, d_model=d_model, n_heads=heads, head_dim=hd, batch=batch, seq=seq, prompt=seq // 2)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(64 + seq)
    normal = lambda *s: torch.empty(s, device="cuda").normal_(0, 1, generator=gen)
    w = {k: (0.03 * normal(d_model, d_model)).to(torch.bfloat16) for k in ("w_q", "w_k", "w_v", "w_o")}
    w["rms_gain"] = torch.ones(d_model, device="cuda")
    layer = dare.Layer(shape, w, kernel_path=dare.PATH_TENSOR)
    bf = lambda v: v.to(torch.bfloat16).double()
    angle = torch.arange(seq, device="cuda").double()[:, None] * \
        shape.rope_theta ** (-2.0 * torch.arange(hd // 2, device="cuda").double() / hd)
    cos, sin = angle.cos()[None, :, None], angle.sin()[None, :, None]
    split = lambda v: v.view(batch, seq, heads, hd).transpose(1, 2)
    x = normal(batch, seq, d_model)
    rows = torch.ones((batch, seq), dtype=torch.bool, device="cuda")
    for step in range(2):
        if step == 1:
            rows = torch.rand((batch, seq), generator=gen, device="cuda") < 0.3
            x = torch.where(rows[:, :, None], normal(batch, seq, d_model), x + 1e-3 * normal(batch, seq, d_model))
        xd = x.to(torch.bfloat16)
        layer.step(xd, 3, 0.1)
        assert layer.status() == 0
        c = layer.read_caches(batch, seq)
        k, v, got = (torch.from_numpy(c[n]).cuda().double() for n in "kvo")
        x64 = xd.double()
        q = (bf(x64 * torch.rsqrt((x64 * x64).mean(-1, keepdim=True) + shape.rms_eps)) @ w["w_q"].double().T).view(batch, seq, heads, hd)
        a, b = q[..., :hd // 2], q[..., hd // 2:]
        q = bf(torch.cat([a * cos - b * sin, a * sin + b * cos], -1).view(batch, seq, d_model))
        want = torch.stack([(torch.softmax(split(q)[i] @ split(k)[i].transpose(-1, -2) / hd ** 0.5, -1) @ split(v)[i])
                            .transpose(0, 1).reshape(seq, d_model) for i in range(batch)])
        got, want = got[rows], want[rows]
        rel = ((got - want).norm() / want.norm()).item()
        storage = ((bf(want) - want).norm() / want.norm()).item()
        assert rel <= 1.05 * storage, (step, rel, storage)
    layer.close()
