"""The denoiser's kernels launched as programmatic dependents of one another
against the same calls launched plainly (as under the event profiler): the same
kernels on the same data, so the outputs are equal bit for bit.  Several
forwards on different inputs are queued back to back without a
synchronisation, so that a kernel that read or overwrote a buffer before its
predecessors were done would be seen; they are also captured into a graph, where
the launches are plain as well."""
import numpy as np
import pytest
import torch

from helpers import to_dev
from paper_2608_01845_gb300 import synth, wdc

pytestmark = pytest.mark.gpu
SMALL = dict(layers=2, hidden=256, heads=4, head_dim=64, mlp=1024, temb_dim=256, freq_dim=256, in_ch=16, frames=4,
             height=16, width=16, patch=2, cond_tokens=16, cond_dim=256, dual_stream=0)
DUAL = dict(SMALL, layers=1, hidden=512, heads=4, head_dim=128, cond_tokens=40, dual_stream=1)
MANY_TILES = dict(SMALL, layers=1, hidden=1024, heads=16, mlp=4096, frames=6, height=40, width=40)
REPEATS = 6


@pytest.mark.parametrize("dtype", [wdc.F32, wdc.BF16])
@pytest.mark.parametrize("model", ["small", "dual", "many_tiles"])
def test_chained_forwards_equal_plain_launches(dtype, model):
    cfgd = {"small": SMALL, "dual": DUAL, "many_tiles": MANY_TILES}[model]
    if model == "many_tiles" and dtype == wdc.F32:
        pytest.skip("a size for the tensor-core kernels")
    ctx = wdc.Context(wdc.make_config(dtype=dtype, max_batch=2, **cfgd), 10)
    ctx.set_weights(synth.dit_weights(cfgd, 5, std=0.02, bias_std=0.02))
    shape = (cfgd["in_ch"], cfgd["frames"], cfgd["height"], cfgd["width"])
    n = int(np.prod(shape))
    zs = [to_dev(synth.latent(70 + r, shape)) for r in range(REPEATS)]
    cts = [to_dev(synth.cond_tokens(80 + r, cfgd["cond_tokens"], 256)) for r in range(REPEATS)]

    def forwards():
        out = torch.full((REPEATS, n), float("nan"), device="cuda")
        for r in range(REPEATS - 1):
            ctx.dit_forward(zs[r], 90.0 * (r + 1), cts[r], out[r])
        ctx.dit_forward_batch([zs[-1]], 55.0, [cts[-1]], [out[-1]], cfg=True, guidance=1.5)
        return out

    chained = forwards()
    torch.cuda.synchronize()
    ctx.profile_enable(True)
    plain = forwards()
    torch.cuda.synchronize()
    ctx.profile_enable(False)
    assert torch.equal(chained, plain)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = forwards()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(captured, plain)
    assert ctx.device_errors() == 0
