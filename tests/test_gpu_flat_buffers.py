"""The buffers of a QuantizedQKV need not have the shapes or element types that alloc_qkv gives them: only their addresses
travel.  The output a call creates has the problem's shape all the same."""
import dataclasses

import pytest
import torch

from paper_2607_04302_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("view", [torch.uint8, torch.int32])
def test_output_shape_does_not_come_from_the_buffers(view):
    from paper_2607_04302_b200 import binding as hb
    cfg = synth.config("C3", B=2, Hq=4, Hkv=2, N=192)
    q, k, v = synth.make_qkv_device(cfg, DEV)
    qkv = hb.quantize_qkv(q, k, v)
    flat = dataclasses.replace(qkv, **{f.name: getattr(qkv, f.name).view(-1).view(view) for f in dataclasses.fields(qkv)
                                       if isinstance(getattr(qkv, f.name), torch.Tensor)})
    for out_dtype, dt in ((hb.F32, torch.float32), (hb.BF16, torch.bfloat16)):
        want = hb.attention_fwd(qkv, True, out_dtype=out_dtype)
        got = hb.attention_fwd(flat, True, out_dtype=out_dtype)
        assert got.shape == q.shape and got.dtype == dt and got.is_contiguous() and torch.equal(got, want)
