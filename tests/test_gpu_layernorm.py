"""The bf16 LayerNorm kernels over the widths at which another one is chosen:
whole and partly used vector counts, the streamed width, and a width that is no
multiple of the 256 columns a warp loads at a time."""
import numpy as np
import pytest
import torch

from helpers import rel_l2
from oracle import dit
from oracle.params import DiTConfig
from paper_2608_01845_gb300 import synth, wdc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [256, 320, 512, 768, 1280, 2048, 2304, 3072, 4096])
def test_final_layernorm(D):
    """A model whose block adds nothing and whose final projection selects 64
    columns: its output is the modulated final LayerNorm.  Each of x, its
    position embedding and the result is rounded to bf16 once (at most 2^-8
    relative an element); normalising divides by the rows' deviation, which is
    their norm over sqrt(D) but for their mean, and |x| exceeds the embedding's
    norm here, so the three add up to at most 4 * 2^-8 of the result."""
    cfgd = dict(layers=1, hidden=D, heads=D // 64, head_dim=64, mlp=64, temb_dim=256, freq_dim=256, in_ch=16, frames=1,
                height=14, width=22, patch=2, cond_tokens=3, cond_dim=64, dual_stream=0)
    W = synth.dit_weights(cfgd, 11, std=0.25, bias_std=0.3, bf16=True)
    for name in W:
        if name.startswith("L0.") or name in ("final.mod.w", "final.w", "final.b"):
            W[name] = np.zeros_like(W[name])
    cols = np.linspace(0, D - 1, 64).astype(int)
    W["final.w"][np.arange(64), cols] = 1.0
    z, ct = synth.bf16_round(synth.latent(3, (16, 1, 14, 22))), synth.cond_tokens(4, 3, 64)
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, **cfgd), 2)
    ctx.set_weights(W)
    v = torch.empty(z.size, device="cuda")
    ctx.dit_forward(torch.from_numpy(z.reshape(-1)).cuda(), 600.0, torch.from_numpy(ct).cuda(), v)
    torch.cuda.synchronize()
    assert ctx.device_errors() == 0
    want = dit.forward(W, DiTConfig(**cfgd), z, 600.0, ct)
    assert rel_l2(v.cpu().numpy(), want) <= 4 * 2.0 ** -8
