"""What a call has written is there for the next one, whatever its stream.  A
parameter that wdc_set_tensor has returned from is on the device, whatever
stream uses it next: the timestep products read their weights before they wait
for the kernels ahead of them."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2608_01845_gb300 import synth, wdc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MODEL = dict(layers=1, hidden=1024, heads=16, head_dim=64, mlp=1024, temb_dim=512, freq_dim=256, in_ch=16, frames=1,
             height=8, width=8, patch=2, cond_tokens=4, cond_dim=64, dual_stream=0)


def test_the_upload_waits_for_its_copy():
    """A copy from pageable memory may return before its last part is on the
    device, so the upload has to wait for the copy's stream (read from the source:
    by timing the loss is rare)."""
    code = re.sub(r"//[^\n]*", "", open(os.path.join(ROOT, "paper_2608_01845_gb300", "csrc", "dit.cu")).read())
    body = re.search(r"static wdc_status upload\([^{]*\{(.*?)\n\}", code, re.S).group(1)
    assert "cudaMemcpy(" in body
    assert re.search(r"cudaMemcpy\(.*cuda(Stream|Device)Synchronize\([^\n]*\n\s*return WDC_OK;\s*$", body, re.S)
    assert body.count("return WDC_OK") == 1


def test_calls_that_zero_memory_wait_for_it():
    """A context's buffers and its cleared error word (read from the source)."""
    code = re.sub(r"//[^\n]*", "", open(os.path.join(ROOT, "paper_2608_01845_gb300", "csrc", "api.cu")).read())
    functions = re.findall(r"\nwdc_status (\w+)\([^{;]*\{(.*?)\n\}", code, re.S)
    zeroing = {name: body for name, body in functions if re.search(r"\bcudaMemset\(", body)}
    assert {"ensure_disp", "wdc_create", "wdc_device_errors"} <= set(zeroing)
    for name, body in zeroing.items():
        assert "zeros_written(c)" in body[body.rindex("cudaMemset("):], name


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [wdc.BF16, wdc.F32])
def test_a_forward_on_another_stream_right_after_an_upload(dtype):
    """Modulation vectors on a non-blocking stream right after new weights, 20
    times, equal those computed once the device is idle."""
    ctx = wdc.Context(wdc.make_config(dtype=dtype, **MODEL), 2)
    ctx.set_weights(synth.dit_weights(MODEL, 5, std=0.02, bias_std=0.02))
    rows, E = 6 * MODEL["hidden"], MODEL["temb_dim"]
    ws = [np.random.default_rng(s).standard_normal((rows, E), dtype=np.float32) for s in range(2)]
    new = lambda: torch.full((rows + 2 * MODEL["hidden"],), float("nan"), device="cuda")
    want = []
    for w in ws:
        ctx.set_tensor(wdc.LAYER_TENSORS["mod.w"], w)
        torch.cuda.synchronize()
        want.append(new())
        ctx.dit_modulation(300.0, want[-1])
        torch.cuda.synchronize()
    assert not torch.equal(want[0], want[1])
    side = torch.cuda.Stream()
    outs = [new() for _ in range(20)]
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        ctx.set_tensor(wdc.LAYER_TENSORS["mod.w"], ws[i % 2])
        ctx.dit_modulation(300.0, out, stream=side.cuda_stream)
        side.synchronize()
    for i, out in enumerate(outs):
        assert torch.equal(out, want[i % 2])
