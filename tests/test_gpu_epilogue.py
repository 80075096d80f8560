"""The GEMM epilogues where their 32-row x 64-column slabs can go wrong: row
and column remainders, V^T slabs that do not start on a 16-byte boundary, and
slabs that hold rows of two samples or of both streams."""
import numpy as np
import pytest
import torch

from helpers import assert_gemms, rel_l2, to_dev
from oracle import dit
from oracle.params import DiTConfig
from paper_2608_01845_gb300 import synth, wdc

pytestmark = pytest.mark.gpu

MODEL = dict(layers=1, hidden=256, heads=4, head_dim=64, mlp=512, temb_dim=256, freq_dim=256, in_ch=16, frames=3,
             height=14, width=22, patch=2, cond_tokens=16, cond_dim=64, dual_stream=0)


@pytest.mark.parametrize("M", [1, 31, 33, 127, 128, 255, 256, 257, 289])
@pytest.mark.parametrize("N", [32, 64, 96, 288])
@pytest.mark.parametrize("mode", ["store", "gelu", "resid"])
def test_gemm_rows_and_columns(M, N, mode):
    """Against fp64: one rounding of the result to bf16 (8 significant bits: at
    most 2^-8 relative an element, so at most that in the 2-norm) and fp32 sums
    of K terms; nothing is written past the last row."""
    K = 72
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, **MODEL), 2)
    A, W = synth.bf16_round(synth.normal(1, (M, K))), synth.bf16_round(synth.normal(2, (N, K), 0.1))
    b = synth.normal(3, (N,), 0.5)
    want = A.astype(np.float64) @ W.astype(np.float64).T + b
    buf = torch.full((M + 40, N), 7.0, dtype=torch.bfloat16, device="cuda")
    C, kw = buf[:M], {}
    if mode == "gelu":
        kw["gelu"], want = True, dit.gelu_tanh(want)
    elif mode == "resid":
        R, g = synth.bf16_round(synth.normal(4, (M, N))), synth.normal(5, (N,))
        want = R.astype(np.float64) + g * want
        kw.update(res=to_dev(R, torch.bfloat16), gate=to_dev(g))
    ctx.op_gemm(to_dev(A, torch.bfloat16), to_dev(W, torch.bfloat16), C, bias=to_dev(b), **kw)
    torch.cuda.synchronize()
    assert_gemms(ctx, f"one64/{mode}")
    assert ctx.device_errors() == 0
    assert rel_l2(C.float().cpu().numpy(), want) <= 2.0 ** -8 + K * 2.0 ** -22
    assert bool((buf[M:] == 7.0).all())


@pytest.mark.parametrize("Lc,dual,d", [(13, 0, 64), (13, 1, 64), (24, 1, 128), (37, 1, 128), (300, 1, 64), (1, 0, 128)])
def test_forward_slabs_across_samples_and_streams(Lc, dual, d):
    """A forward against the oracle, and a batch of three bitwise equal to its
    samples' own forwards, with condition-token counts that leave the video
    rows' V^T slabs unaligned and put two samples into one slab."""
    cfgd = dict(MODEL, cond_tokens=Lc, dual_stream=dual, head_dim=d, heads=256 // d)
    W = synth.dit_weights(cfgd, 7, std=0.06, bias_std=0.05, bf16=True)
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, max_batch=3, **cfgd), 2)
    ctx.set_weights(W)
    z = [synth.latent(20 + b, (16, 3, 14, 22)) for b in range(3)]
    ct = [synth.cond_tokens(30 + b, Lc, 64) for b in range(3)]
    zd, cd = [to_dev(a.reshape(-1)) for a in z], [to_dev(a) for a in ct]
    one = []
    for b in range(3):
        one.append(torch.empty_like(zd[b]))
        ctx.dit_forward(zd[b], 600.0, cd[b], one[b])
    many = [torch.empty_like(t) for t in zd]
    ctx.dit_forward_batch(zd, 600.0, cd, many)
    torch.cuda.synchronize()
    assert ctx.device_errors() == 0
    for b in range(3):
        assert torch.equal(one[b], many[b])
    want = dit.forward(W, DiTConfig(**cfgd), z[0], 600.0, ct[0])
    assert rel_l2(one[0].cpu().numpy(), want) <= 2e-2


@pytest.mark.parametrize("M,N,K,kernel", [
    (226, 3072, 3072, "split2"), (64, 1056, 8192, "split8"), (128, 512, 12288, "split8"), (1, 9216, 3072, "split2"),
    (257, 160, 4104, "split8"), (130, 32, 2056, "split8"), (64, 3072, 8192, "split4"), (200, 1056, 1544, "split4"),
    (700, 1024, 1024, {"store": "one64", "gelu": "split2", "resid": "one64"}), (129, 6176, 520, "one128"),
    (1600, 1024, 2048, "pair128")])
@pytest.mark.parametrize("mode", ["store", "gelu", "resid"])
def test_gemm_few_tiles(M, N, K, kernel, mode):
    """Shapes of the narrow-tile and split-K kernels (2, 4 and 8 CTAs a tile,
    shares past N, K blocks that do not divide evenly), bound as above."""
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, **MODEL), 2)
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)
    A, W, b = r(M, K).bfloat16(), (r(N, K) * K ** -0.5).bfloat16(), r(N)
    want, kw = A.double() @ W.double().T + b.double(), {}
    buf = torch.full((M + 40, N), 7.0, dtype=torch.bfloat16, device="cuda")
    if mode == "gelu":
        kw["gelu"] = True
        want = 0.5 * want * (1 + torch.tanh((2 / np.pi) ** 0.5 * (want + 0.044715 * want ** 3)))
    elif mode == "resid":
        R, gate = r(M, N).bfloat16(), r(N)
        want = R.double() + gate.double() * want
        kw.update(res=R, gate=gate)
    ctx.op_gemm(A, W, buf[:M], bias=b, **kw)
    torch.cuda.synchronize()
    assert_gemms(ctx, f"{kernel if isinstance(kernel, str) else kernel[mode]}/{mode}")
    assert ctx.device_errors() == 0
    assert float((buf[:M].double() - want).norm() / want.norm()) <= 2.0 ** -8 + K * 2.0 ** -22
    assert bool((buf[M:] == 7.0).all())


@pytest.mark.parametrize("Lc,dual,d,D,mlp,gemms", [
    (5, 0, 64, 2048, 4096, ["split4/store", "split2/qkv", "split4/gelu", "split4/resid"]),
    (5, 1, 128, 2048, 4096, ["split2/gelu grouped", "split4/resid grouped", "split8/unpatch"]),
    (100, 1, 128, 1536, 1024, ["split8/store", "split2/qkv grouped", "split4/gelu grouped", "split4/resid grouped",
                               "split4/unpatch"]),
    (140, 1, 64, 2048, 1024, ["split4/gelu grouped", "split2/resid grouped"])])
def test_forward_split_k(Lc, dual, d, D, mlp, gemms):
    """A wide model on few tokens, whose block's GEMMs split K (those named;
    two problems in one launch with both streams, of which the condition rows'
    have two row tiles at 140 tokens), against the oracle, and a batch of three
    bitwise equal to its samples' own forwards.  (QKV of more row tiles has too
    many tiles to be split.)"""
    cfgd = dict(MODEL, hidden=D, heads=D // d, head_dim=d, mlp=mlp, frames=1, height=8, width=10, cond_tokens=Lc,
                cond_dim=2048, dual_stream=dual)
    W = synth.dit_weights(cfgd, 9, std=0.02, bias_std=0.05, bf16=True)
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, max_batch=3, **cfgd), 2)
    ctx.set_weights(W)
    z = [synth.latent(20 + b, (16, 1, 8, 10)) for b in range(3)]
    ct = [synth.cond_tokens(30 + b, Lc, 2048) for b in range(3)]
    zd, cd = [to_dev(a.reshape(-1)) for a in z], [to_dev(a) for a in ct]
    one = []
    for b in range(3):
        one.append(torch.empty_like(zd[b]))
        ctx.dit_forward(zd[b], 600.0, cd[b], one[b])
    many = [torch.empty_like(t) for t in zd]
    ctx.dit_forward_batch(zd, 600.0, cd, many)
    torch.cuda.synchronize()
    assert_gemms(ctx, *gemms)
    assert ctx.device_errors() == 0
    for b in range(3):
        assert torch.equal(one[b], many[b])
    want = dit.forward(W, DiTConfig(**cfgd), z[0], 600.0, ct[0])
    assert rel_l2(one[0].cpu().numpy(), want) <= 2e-2


@pytest.mark.parametrize("M,N,K,kernel", [
    (257, 96, 72, "one64"), (129, 6176, 520, "one128"), (226, 3072, 3072, "split2"), (200, 1056, 1544, "split4"),
    (257, 160, 4104, "split8"), (1600, 1024, 2048, "pair128"), (513, 4128, 520, "pair192"), (257, 7328, 1032, "pair256")])
@pytest.mark.parametrize("dtype", [wdc.BF16, wdc.F32])
@pytest.mark.parametrize("in_place", [False, True])
def test_gemm_gelu_then_gated_residual(M, N, K, kernel, dtype, in_place):
    """C = res + gate * GELU(A W^T + bias), both options of one call, in every
    kernel of both dtypes.  bf16 as above; fp32: sums of K terms and the
    hardware exponential of GELU (2^-22 relative of a factor below one) against
    2^-24 a rounding."""
    ctx = wdc.Context(wdc.make_config(dtype=dtype, **MODEL), 2)
    td = torch.bfloat16 if dtype == wdc.BF16 else torch.float32
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)
    A, W, b, R, gate = r(M, K).to(td), (r(N, K) * K ** -0.5).to(td), r(N), r(M, N).to(td), r(N)
    x = A.double() @ W.double().T + b.double()
    want = R.double() + gate.double() * 0.5 * x * (1 + torch.tanh((2 / np.pi) ** 0.5 * (x + 0.044715 * x ** 3)))
    buf = torch.full((M + 40, N), 7.0, dtype=td, device="cuda")
    if in_place:
        buf[:M] = R
    ctx.op_gemm(A, W, buf[:M], bias=b, gelu=True, res=buf[:M] if in_place else R, gate=gate)
    torch.cuda.synchronize()
    if dtype == wdc.BF16:
        assert_gemms(ctx, f"{kernel}/resid_gelu")
    assert ctx.device_errors() == 0
    err = float((buf[:M].double() - want).norm() / want.norm())
    assert err <= (2.0 ** -8 if dtype == wdc.BF16 else 2.0 ** -20) + K * 2.0 ** -22
    assert bool((buf[M:] == 7.0).all())


@pytest.mark.parametrize("in_ch,p,frames,hp,wp,D,B,kernel", [
    (16, 2, 3, 7, 11, 256, 3, "one64"), (128, 2, 5, 14, 15, 512, 3, "one128"), (64, 4, 5, 14, 15, 1024, 3, "pair128"),
    (128, 2, 7, 10, 23, 768, 2, "pair192"), (48, 4, 7, 12, 20, 1536, 3, "pair256")])
def test_repeating_residual(in_ch, p, frames, hp, wp, D, B, kernel):
    """The position embedding of a batch (its rows repeat with each sample, and
    slabs of 32 rows hold two samples) in every kernel that takes it (with at
    most 1024 features a patch its K is never split): bitwise the samples' own
    forwards, whose residual does not repeat, and one of them against the oracle."""
    cfgd = dict(MODEL, hidden=D, heads=D // 64, mlp=D, in_ch=in_ch, frames=frames, height=hp * p, width=wp * p, patch=p,
                cond_tokens=5)
    shape = (in_ch, frames, hp * p, wp * p)
    W = synth.dit_weights(cfgd, 11, std=0.02, bias_std=0.05, bf16=True)
    ctx = wdc.Context(wdc.make_config(dtype=wdc.BF16, max_batch=B, **cfgd), 2)
    ctx.set_weights(W)
    z = [synth.latent(20 + b, shape) for b in range(B)]
    ct = [synth.cond_tokens(30 + b, 5, 64) for b in range(B)]
    zd, cd = [to_dev(a.reshape(-1)) for a in z], [to_dev(a) for a in ct]
    many = [torch.empty_like(t) for t in zd]
    ctx.dit_forward_batch(zd, 600.0, cd, many)
    torch.cuda.synchronize()
    assert_gemms(ctx, f"{kernel}/resid_repeat")
    for b in range(B):
        one = torch.empty_like(zd[b])
        ctx.dit_forward(zd[b], 600.0, cd[b], one)
        torch.cuda.synchronize()
        assert torch.equal(one, many[b])
    assert ctx.device_errors() == 0
    want = dit.forward(W, DiTConfig(**cfgd), z[0], 600.0, ct[0])
    assert rel_l2(many[0].cpu().numpy(), want) <= 2e-2
