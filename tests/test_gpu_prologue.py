"""The forward's prologue at its edges: tokens that do not fill a block's share,
tokens of a whole block's share, condition rows of an odd length, feature and
embedding widths that leave 16-byte rows (the element-wise products) and widths
of several vectors per lane."""
import numpy as np
import pytest
import torch

from helpers import rel_l2, to_dev
from oracle import batch as ob
from oracle import dit
from oracle.params import DiTConfig
from paper_2608_01845_gb300 import synth, wdc

pytestmark = pytest.mark.gpu

BASE = dict(layers=1, hidden=128, heads=2, head_dim=64, mlp=128, dual_stream=0)


@pytest.mark.parametrize("dtype", [wdc.F32, wdc.BF16])
@pytest.mark.parametrize("in_ch,patch,frames,height,width,Lc,Dc,Fd,E", [
    (16, 2, 3, 10, 14, 5, 72, 256, 256),
    (16, 2, 1, 6, 10, 1, 8, 34, 70),
    (16, 8, 2, 24, 16, 3, 1032, 8, 36),        # 1024 values a token
    (32, 1, 2, 7, 9, 7, 200, 66, 1160),
])
def test_guided_forward(dtype, in_ch, patch, frames, height, width, Lc, Dc, Fd, E):
    """A guided forward (the null condition reads no tokens) against the
    oracle.  fp32: sums of up to 1160 terms, 1e-5.  bf16: weights and inputs
    are bf16 on both sides; activations are rounded 8 times on the way (2^-8
    each), and guidance 1.5 weighs two forwards by 1.5 and 0.5."""
    cfgd = dict(BASE, in_ch=in_ch, patch=patch, frames=frames, height=height, width=width, cond_tokens=Lc, cond_dim=Dc,
                freq_dim=Fd, temb_dim=E)
    shape = (in_ch, frames, height, width)
    W = synth.dit_weights(cfgd, 21, std=0.05, bias_std=0.05, bf16=dtype == wdc.BF16)
    z, ct = synth.latent(22, shape), synth.cond_tokens(23, Lc, Dc)
    if dtype == wdc.BF16:
        z, ct = synth.bf16_round(z), synth.bf16_round(ct)
    ctx = wdc.Context(wdc.make_config(dtype=dtype, max_batch=2, **cfgd), 2)
    ctx.set_weights(W)
    v = torch.empty(z.size, device="cuda")
    ctx.dit_forward_batch([to_dev(z.reshape(-1))], 412.5, [to_dev(ct)], [v], cfg=True, guidance=1.5)
    torch.cuda.synchronize()
    assert ctx.device_errors() == 0
    cfg = DiTConfig(**cfgd)
    want = ob.guided_velocity(dit.forward(W, cfg, z, 412.5, ct), dit.forward(W, cfg, z, 412.5, ob.null_tokens(cfg)), 1.5)
    assert rel_l2(v.cpu().numpy(), want) <= (1e-5 if dtype == wdc.F32 else 8 * 2.0 ** -8 * 1.6)
