"""The fp32 operators at the edges of their tiles, and where their operands are
not aligned for 16-byte copies."""
import numpy as np
import pytest
import torch

from paper_2608_01845_gb300 import wdc

pytestmark = pytest.mark.gpu

MODEL = dict(layers=1, hidden=256, heads=4, head_dim=64, mlp=512, temb_dim=256, freq_dim=256, in_ch=16, frames=1,
             height=4, width=4, patch=2, cond_tokens=1, cond_dim=64)


def _at(t, offset):
    """The same values at an address `offset` floats past a 16-byte boundary."""
    buf = torch.zeros(t.numel() + 4, device="cuda")
    buf[offset:offset + t.numel()] = t.reshape(-1)
    return buf[offset:offset + t.numel()].view(t.shape)


# The bound: an fp32 chain of K fused multiply-adds is off by at most K 2^-24 of
# the sum of the terms' magnitudes, and the epilogue adds a few roundings.
@pytest.mark.parametrize("M,N,K,offset", [(1, 1, 4, 0), (31, 15, 32, 0), (33, 17, 36, 0), (64, 64, 1024, 0),
                                          (272, 256, 1024, 0), (1300, 1024, 68, 0), (65, 63, 30, 0), (40, 48, 64, 1)])
@pytest.mark.parametrize("mode", ["store", "gelu", "resid"])
def test_gemm(M, N, K, offset, mode):
    ctx = wdc.Context(wdc.make_config(dtype=wdc.F32, **MODEL), 2)
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)
    A, W, b = _at(r(M, K), offset), r(N, K), r(N)
    terms = A.double().abs() @ W.double().abs().T + b.double().abs()
    want, kw = A.double() @ W.double().T + b.double(), {}
    buf = torch.full((M + 3, N), 7.0, device="cuda")
    if mode == "gelu":
        kw["gelu"] = True
        want = 0.5 * want * (1 + torch.tanh((2 / np.pi) ** 0.5 * (want + 0.044715 * want ** 3)))
    elif mode == "resid":
        R, gate = r(M, N), r(N)
        want = R.double() + gate.double() * want
        terms = R.double().abs() + gate.double().abs() * terms
        kw.update(res=R, gate=gate)
    ctx.op_gemm(A, W, buf[:M], bias=b, **kw)
    torch.cuda.synchronize()
    assert bool(((buf[:M].double() - want).abs() <= 2 * (K + 8) * 2.0 ** -24 * terms + 1e-6).all())
    assert bool((buf[M:] == 7.0).all())


@pytest.mark.parametrize("M,N,K", [(600, 768, 4), (600, 768, 16), (600, 768, 20), (2000, 1024, 32), (2000, 1024, 36),
                                   (2000, 1024, 48), (2000, 1024, 52), (2000, 1024, 176), (2000, 1024, 180)])
def test_gemm_of_short_k_has_the_bits_of_any_other_shape(M, N, K):
    """On both sides of the rule by which short K goes to the element-wise
    kernel: the rows of a large product are bit for bit those of a product of 16
    of them, which takes the small tiles."""
    ctx = wdc.Context(wdc.make_config(dtype=wdc.F32, **MODEL), 2)
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, W, b = (torch.randn(*s, device="cuda", generator=g) for s in ((M, K), (N, K), (N,)))
    C = torch.empty(M, N, device="cuda")
    ctx.op_gemm(A, W, C, bias=b)
    for m in (0, 336, M - 16):
        part = torch.empty(16, N, device="cuda")
        ctx.op_gemm(A[m:m + 16].clone(), W, part, bias=b)
        torch.cuda.synchronize()
        assert torch.equal(part, C[m:m + 16])


@pytest.mark.parametrize("H,L,d,offset", [(1, 1, 64, 0), (2, 15, 128, 0), (3, 16, 64, 0), (2, 63, 64, 0), (2, 65, 128, 0),
                                          (4, 272, 64, 0), (2, 129, 64, 1), (1, 130, 128, 3)])
def test_attention(H, L, d, offset):
    ctx = wdc.Context(wdc.make_config(dtype=wdc.F32, **MODEL), 2)
    g = torch.Generator(device="cuda").manual_seed(H + L + d)
    q, k, v = (torch.randn(H, L, d, device="cuda", generator=g) for _ in range(3))
    q = 3.0 * q                                   # peaked rows: the running maximum moves
    o = torch.full((L, H * d), float("nan"), device="cuda")
    ctx.op_attention(_at(q, offset), _at(k, offset), _at(v.transpose(1, 2).contiguous(), offset), o)
    torch.cuda.synchronize()
    p = torch.softmax(q.double() @ k.double().transpose(1, 2) * d ** -0.5, -1)
    want = (p @ v.double()).transpose(0, 1).reshape(L, H * d)
    assert float((o.double() - want).norm() / want.norm()) <= 1e-6 * max(1.0, d ** 0.5 / 4)
