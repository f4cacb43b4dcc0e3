"""The MLP half of a stack's block (RMSNorm, SwiGLU, down projection, residual, final norm) at row-tile and column-tile
counts on both sides of its launch rules, against a plain PyTorch fp32 evaluation from the captured attention output."""
import pytest

from paper_2605_08134_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [
    # d_model, d_ff, batch, seq
    (512, 4096, 3, 200),      # six row tiles: persistent SwiGLU, two-CTA tiles
    (512, 4096, 1, 600),      # five: a padding row tile
    (256, 12544, 3, 128),     # three row tiles of 98 column tiles: persistent SwiGLU, single-CTA tiles
    (512, 1024, 1, 129),      # two row tiles, one wave
    (256, 12544, 2, 77),      # ... one wave as well: 66 tiles of 192 outputs on 74 SM pairs
    (256, 19072, 2, 77),      # ... more than one wave: tiles of 256 (the widest), the 75th half full
    (256, 38016, 3, 40),      # one row tile, more than one wave: the 149th tile of 256 half full
    (4096, 12544, 3, 256),    # groups of column tiles of unequal width: 98 over nine groups of 11
    (4096, 2048, 2, 640),     # ten row tiles: persistent down projection
    (512, 2048, 2, 31),
]


@pytest.mark.parametrize("d,f,batch,seq", CASES)
def test_mlp_against_torch(d, f, batch, seq):
    import torch
    from paper_2605_08134_b200 import build
    build.build()
    from paper_2605_08134_b200 import dare
    g = torch.Generator(device="cuda")
    g.manual_seed(d + f + seq)
    draw = lambda *s: torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0, 0.02, generator=g)
    lay = wl.scaled(wl.LLADA_LAYER, d_model=d, n_heads=d // 128, batch=batch, seq=seq, prompt=seq // 2)
    shape = wl.StackShape("mlp", 1, lay, f, 512, seq - seq // 2)
    gain = torch.rand(d, generator=g, device="cuda") + 0.5
    lw = {k: draw(d, d) for k in ("w_q", "w_k", "w_v", "w_o")}
    lw.update(w_gate=draw(f, d), w_up=draw(f, d), w_down=draw(d, f), rms_gain=torch.ones(d, device="cuda"), gain2=gain)
    w = {"emb": draw(512, d) * 50, "head": draw(512, d), "final_gain": gain, "layers": [lw]}
    stack = dare.Stack(shape, w, batch)
    x, h = (torch.zeros((batch, seq, d), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    stack.set_capture(0, x, h)
    tokens = torch.randint(0, 512, (batch, seq), generator=g, device="cuda", dtype=torch.int32)
    out = stack.forward(tokens, seq, 0, 3, [0.1]).float()
    assert stack.layer(0).status() == 0

    def norm(v):
        return v * torch.rsqrt((v * v).mean(-1, keepdim=True) + lay.rms_eps) * gain
    hf = h.float()
    n = norm(hf).to(torch.bfloat16).float()
    act = torch.nn.functional.silu(n @ lw["w_gate"].float().T) * (n @ lw["w_up"].float().T)
    want = norm(hf + act.to(torch.bfloat16).float() @ lw["w_down"].float().T)
    err = (out - want).abs()
    assert err.max() < 0.06 and (out - want).norm() / want.norm() < 6e-3, (err.max(), (out - want).norm() / want.norm())
    stack.close()
