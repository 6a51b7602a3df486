"""The kernel on pairs of SMs (hifa4_attention_cta2.cu, d = 256) against the 64-key kernel, which the other tests hold
against the oracle.  The dump launch always runs the latter, so the two outputs must be equal bit for bit; the sizes are
large enough for the pairs to be chosen (more blocks than SMs) and cover what pairs and steps of two tiles can get wrong."""
import pytest
import torch

from paper_2607_04302_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = {
    # B, Hq, Hkv, N, causal, qmean, head map
    "even-group": (1, 16, 8, 1408, True, False, None),
    "odd-group-ragged-block": (2, 14, 2, 832, True, False, None),       # pairs straddle query blocks, last block half empty
    "odd-tile-count": (2, 12, 4, 1088, False, False, None),             # the last step's second tile lies past the last key
    "odd-block-count": (4, 4, 4, 1408, True, False, None),              # one head per KV head: a pair without a second block
    "one-tile": (64, 16, 8, 64, False, False, None),
    "two-tiles": (32, 16, 8, 128, True, False, None),
    "qmean": (2, 16, 8, 1024, True, True, None),
    "qmean-odd-tile-count": (2, 14, 2, 832, True, True, None),
    "head-map": (4, 8, 4, 1280, True, False, [3, 0, 0, 2, 1, 3, 3, 0]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_sm_pair_kernel_is_bit_identical(name):
    from paper_2607_04302_b200 import binding as hb
    B, Hq, Hkv, N, causal, qmean, head_map = CASES[name]
    cfg = synth.config("C2", d=256, B=B, Hq=Hq, Hkv=Hkv, N=N, causal=causal)
    q, k, v = synth.make_qkv_device(cfg, DEV)
    qkv = hb.quantize_qkv(q, k, v, q_to_kv=head_map, qmean=qmean)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    want, _ = hb.attention_fwd(qkv, causal, qmean=qmean, debug_blocks=[(0, 0, 0)], d_status=status)
    buf = torch.full((want.numel() + 4096,), 7.0, dtype=torch.float32, device=DEV)
    got = hb.attention_fwd(qkv, causal, qmean=qmean, out=buf[:want.numel()].view_as(want), d_status=status)
    assert torch.equal(got, want) and bool((buf[want.numel():] == 7.0).all())
    assert torch.equal(hb.attention_fwd(qkv, causal, qmean=qmean, out_dtype=hb.F16, d_status=status), want.half())
    assert torch.equal(hb.attention_fwd(qkv, causal, qmean=qmean, out_dtype=hb.BF16, d_status=status), want.bfloat16())
    assert torch.equal(hb.attention_fwd_raw(q, k, v, None, None, causal, q_to_kv=head_map, qmean=qmean, d_status=status), want)
    assert int(status.item()) == 0
    status.fill_(9)                                                     # a set status word makes the launch a no-op
    out = torch.full_like(want, 2.0)
    for _ in range(2):
        hb.attention_fwd(qkv, causal, qmean=qmean, out=out, d_status=status)
    assert bool((out == 2.0).all()) and int(status.item()) == 9
