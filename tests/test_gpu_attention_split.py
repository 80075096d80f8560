"""Attention on both sides of the rule that splits a partial round of units over
the key range."""
import numpy as np
import pytest
import torch

from helpers import rel_l2
from oracle import dit
from paper_2608_01845_gb300 import synth, wdc

pytestmark = pytest.mark.gpu

MODEL = dict(layers=1, hidden=256, heads=4, head_dim=64, mlp=512, temb_dim=256, freq_dim=256, in_ch=16, frames=1,
             height=4, width=4, patch=2, cond_tokens=4, cond_dim=64, dual_stream=0)


@pytest.mark.parametrize("H,L,d,split", [
    (2, 896, 64, False), (2, 897, 64, True),          # 7 and 8 steps in as many parts: 6 and 7 saved
    (1, 768, 128, False), (1, 769, 128, True),        # 12 and 13 steps in 8 parts: 10 and 11 saved
    (48, 900, 64, False), (24, 1600, 64, True),       # second round of 40 units in 3 parts (5 saved), 16 in 8 (11 saved)
])
def test_attention_around_the_split_rule(H, L, d, split):
    """Against fp64 on sampled rows: the probabilities are rounded to f16 (2^-11
    relative each, and they sum to one), the result to bf16 (at most 2^-8), and
    the scores are fp32 sums of d exact products."""
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, **MODEL), 2)
    q, k = (synth.bf16_round(synth.normal(s, (H, L, d))) for s in (31, 32))
    v = synth.normal(33, (H, L, d)).astype(np.float16)
    vt = torch.full((H, d, (L + 7) // 8 * 8), float("nan"), dtype=torch.float16)
    vt[:, :, :L] = torch.from_numpy(np.ascontiguousarray(v.transpose(0, 2, 1)))
    o = torch.empty(L, H * d, dtype=torch.bfloat16, device="cuda")
    dev = lambda a: torch.from_numpy(a).cuda().bfloat16()
    before = ctx.launches
    ctx.op_attention(dev(q), dev(k), vt.cuda(), o)
    torch.cuda.synchronize()
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert ctx.launches - before == (2 if split else 1)      # a split round is merged by a second kernel
    assert ctx.device_errors() == 0
    got = o.float().cpu().numpy()
    rows = np.unique(np.r_[np.linspace(0, L - 1, 40).astype(int), 255, 256, L - 1])
    for h in sorted({0, H // 2, H - 1}):
        want = dit.attention(q[h, rows].astype(np.float64), k[h].astype(np.float64), v[h].astype(np.float64), 1)
        assert rel_l2(got[rows, h * d:(h + 1) * d], want) <= 2.0 ** -8 + 2.0 ** -11 + d * 2.0 ** -22
