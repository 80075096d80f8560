"""The CTA-pair GEMM with 256-, 192- and 128-column tiles, at shapes for which
the launch rule takes them on 152 SMs, with remainders of rows, columns and K."""
import numpy as np
import pytest
import torch

from helpers import assert_gemms, rel_l2, to_dev
from oracle import dit
from oracle.params import DiTConfig
from paper_2608_01845_gb300 import synth, wdc

pytestmark = pytest.mark.gpu

MODEL = dict(layers=1, hidden=512, heads=8, head_dim=64, mlp=2048, temb_dim=256, freq_dim=256, in_ch=16, frames=4,
             height=40, width=40, patch=2, cond_tokens=13, cond_dim=64, dual_stream=0)


@pytest.mark.parametrize("M,N,K,width", [
    (257, 7328, 1032, 256), (2817, 3040, 1032, 256), (1999, 1504, 1544, 192), (2000, 1536, 1536, 192),
    (513, 4128, 520, 192), (1570, 1056, 4104, 128), (1600, 1024, 4096, 128)])     # (257 and 513: a last tile of one row)
@pytest.mark.parametrize("mode", ["store", "gelu", "resid"])
def test_gemm(M, N, K, width, mode):
    """Against fp64 on sampled rows: one rounding of the result to bf16 (at most
    2^-8 relative an element) and fp32 sums of K terms; nothing is written past
    the last row."""
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, **MODEL), 2)
    A, W = synth.bf16_round(synth.normal(1, (M, K))), synth.bf16_round(synth.normal(2, (N, K), 0.05))
    b = synth.normal(3, (N,), 0.5)
    rows = np.unique(np.r_[np.linspace(0, M - 1, 60).astype(int), 127, 128, 255, 256, M - 2])
    want = A[rows].astype(np.float64) @ W.astype(np.float64).T + b
    buf = torch.full((M + 40, N), 7.0, dtype=torch.bfloat16, device="cuda")
    C, kw = buf[:M], {}
    if mode == "gelu":
        kw["gelu"], want = True, dit.gelu_tanh(want)
    elif mode == "resid":
        R, g = synth.bf16_round(synth.normal(4, (M, N))), synth.normal(5, (N,))
        want = R[rows].astype(np.float64) + g * want
        kw.update(res=to_dev(R, torch.bfloat16), gate=to_dev(g))
    ctx.op_gemm(to_dev(A, torch.bfloat16), to_dev(W, torch.bfloat16), C, bias=to_dev(b), **kw)
    torch.cuda.synchronize()
    assert_gemms(ctx, f"pair{width}/{mode}")
    assert ctx.device_errors() == 0
    assert rel_l2(C.float().cpu().numpy()[rows], want) <= 2.0 ** -8 + K * 2.0 ** -22
    assert bool((buf[M:] == 7.0).all())


@pytest.mark.parametrize("dual", [0, 1])
def test_qkv_of_a_block(dual):
    """A block of 1613 tokens of width 512, whose QKV GEMM (1536 columns: three
    kinds in tiles of 192, and with both streams two problems in one launch)
    takes 192 columns, against fp64 on sampled rows: eight roundings to bf16."""
    cfgd = dict(MODEL, dual_stream=dual)
    L, D = 13 + 4 * 20 * 20, 512
    W = synth.dit_weights(cfgd, 7, std=0.05, bias_std=0.05, bf16=True)
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, **cfgd), 2)
    ctx.set_weights(W)
    x = synth.bf16_round(synth.normal(41, (L, D)))
    mod = synth.normal(42, (6 * (1 + dual), D), 0.3)
    xt = to_dev(x, torch.bfloat16)
    ctx.dit_block_forward(0, xt, to_dev(mod))
    torch.cuda.synchronize()
    assert_gemms(ctx, "pair192/qkv grouped" if dual else "pair192/qkv")
    assert ctx.device_errors() == 0
    rows = np.unique(np.r_[0, 5, 12, 13, np.linspace(14, L - 1, 60).astype(int)])
    mods = [mod[6 * s:6 * s + 6].astype(np.float64) for s in range(1 + dual)]
    want = dit.block_rows(x.astype(np.float64), W, DiTConfig(**cfgd), 0, mods, rows)
    assert rel_l2(xt.float().cpu().numpy()[rows], want) <= 8 * 2.0 ** -8
