"""The 64-key kernel with four groups of softmax warps (hifa4_attention_ws64.cu, few blocks, d = 64 and 128) against the same
kernel with two, which the dump launch always runs: the outputs must be equal bit for bit.  Sizes: fewer tiles than groups,
every remainder of tiles by groups, ragged query blocks, both sides of the line between the two."""
import pytest
import torch

from paper_2607_04302_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B, Hq, Hkv, N, causal, qmean, head_map", [
    (1, 1, 1, 64, True, False, None), (1, 2, 1, 128, False, True, None), (2, 3, 1, 192, False, False, None),
    (1, 4, 2, 256, True, False, None), (1, 4, 4, 320, True, True, None), (1, 2, 1, 384, False, False, None),
    (1, 6, 2, 448, False, True, [1, 0, 0, 1, 1, 0]), (1, 2, 2, 512, True, True, None), (2, 8, 4, 576, False, False, None),
    (1, 12, 4, 1984, True, False, None), (1, 16, 4, 1088, False, False, None), (1, 16, 4, 1152, True, True, None),
])
def test_four_groups_are_bit_identical_to_two(d, B, Hq, Hkv, N, causal, qmean, head_map):
    from paper_2607_04302_b200 import binding as hb
    cfg = synth.config("C2", d=d, B=B, Hq=Hq, Hkv=Hkv, N=N, causal=causal)
    q, k, v = synth.make_qkv_device(cfg, DEV)
    qkv = hb.quantize_qkv(q, k, v, q_to_kv=head_map, qmean=qmean)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    want, _ = hb.attention_fwd(qkv, causal, qmean=qmean, debug_blocks=[(0, 0, 0)], d_status=status)
    for dt, ref in ((hb.F32, want), (hb.F16, want.half()), (hb.BF16, want.bfloat16())):
        for _ in range(3):
            assert torch.equal(hb.attention_fwd(qkv, causal, qmean=qmean, out_dtype=dt, d_status=status), ref)
    assert int(status.item()) == 0
