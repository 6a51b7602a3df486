"""The kernel with two query blocks per CTA (hifa4_attention_pair.cu) against the 64-key kernel, which the other tests hold
against the oracle.  The dump launch always runs the latter, so the two outputs must be equal bit for bit; the sizes are
large enough for the two-block kernel to be chosen (hundreds of pairs) and cover what pairing can get wrong."""
import pytest
import torch

from paper_2607_04302_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = {
    # B, Hq, Hkv, N, causal, qmean, head map
    "even-group": (4, 32, 8, 1024, True, False, None),
    "odd-group-ragged-block": (4, 28, 4, 832, True, False, None),       # pairs straddle query blocks, last block half empty
    "odd-block-count": (8, 9, 9, 1152, True, False, None),              # one head per KV head: a pair without a second block
    "one-tile": (64, 16, 8, 64, False, False, None),
    "two-tiles": (32, 32, 8, 128, True, False, None),
    "non-causal-ragged": (4, 24, 4, 1344, False, False, None),
    "qmean": (4, 32, 8, 1024, True, True, None),
    "qmean-odd-group": (4, 28, 4, 832, True, True, None),               # halves of different length share the key-sum slots
    "qmean-odd-block-count": (7, 14, 14, 640, False, True, None),       # a half without a block, ten and 14 tiles, after a pair
    "qmean-odd-block-count-14-tiles": (2, 37, 37, 896, False, True, None),      # on the same SM: the key-sum slots go round
    "head-map": (8, 8, 4, 1088, True, False, [3, 0, 0, 2, 1, 3, 3, 0]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_two_block_kernel_is_bit_identical(name):
    from paper_2607_04302_b200 import binding as hb
    B, Hq, Hkv, N, causal, qmean, head_map = CASES[name]
    cfg = synth.config("C2", B=B, Hq=Hq, Hkv=Hkv, N=N, causal=causal)
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


@pytest.mark.parametrize("B, Hq, Hkv, N, causal, qmean, head_map", [
    (4, 32, 8, 1024, True, False, None), (4, 28, 4, 832, True, False, None),      # an odd number of 64-key tiles: N ends inside a tile
    (8, 9, 9, 1152, True, False, None), (64, 16, 8, 64, False, False, None), (4, 24, 4, 1344, False, False, None),
    (4, 32, 8, 1024, True, True, None), (8, 28, 4, 832, True, True, None), (7, 14, 14, 640, False, True, None), (8, 8, 4, 1088, True, False, [3, 0, 0, 2, 1, 3, 3, 0]),
])
def test_two_block_kernel_with_128_key_tiles(B, Hq, Hkv, N, causal, qmean, head_map):
    """Against the 128-key kernel (hifa4_attention_ws.cu), which the dump launch always runs."""
    from paper_2607_04302_b200 import binding as hb
    cfg = synth.config("C2", B=B, Hq=Hq, Hkv=Hkv, N=N, causal=causal)
    q, k, v = synth.make_qkv_device(cfg, DEV)
    qkv = hb.quantize_qkv(q, k, v, q_to_kv=head_map, qmean=qmean)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    want, _ = hb.attention_fwd(qkv, causal, Bc=128, qmean=qmean, debug_blocks=[(0, 0, 0)], d_status=status)
    for dt, ref in ((hb.F32, want), (hb.F16, want.half()), (hb.BF16, want.bfloat16())):
        assert torch.equal(hb.attention_fwd(qkv, causal, Bc=128, qmean=qmean, out_dtype=dt, d_status=status), ref)
    assert torch.equal(hb.attention_fwd_raw(q, k, v, None, None, causal, Bc=128, q_to_kv=head_map, qmean=qmean, d_status=status), want)
    assert int(status.item()) == 0


@pytest.mark.parametrize("name", ["even-group", "odd-group-ragged-block", "odd-block-count", "one-tile", "two-tiles", "head-map"])
def test_expired_wait_is_reported_and_leaves_the_device_usable(name):
    """The self-test instantiation of this kernel (hifa4_selftest_wait_timeout takes the kernel that a call would take): the arrivals
    that release P V are withheld, the issuer's wait runs out (site 7), the softmax warps' waits for P V see the abort flag, `out`
    stays untouched and the next call gives the right values."""
    from paper_2607_04302_b200 import binding as hb
    B, Hq, Hkv, N, causal, _, head_map = CASES[name]
    cfg = synth.config("C2", B=B, Hq=Hq, Hkv=Hkv, N=N, causal=causal)
    q, k, v = synth.make_qkv_device(cfg, DEV)
    qkv = hb.quantize_qkv(q, k, v, q_to_kv=head_map)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    want, _ = hb.attention_fwd(qkv, causal, debug_blocks=[(0, 0, 0)], d_status=status)
    assert int(status.item()) == 0
    out = torch.full_like(want, 3.0)
    hb.selftest_wait_timeout(qkv, causal, status, out=out)
    torch.cuda.synchronize()
    assert int(status.item()) == 6 + 16 * 7 and bool((out == 3.0).all())
    hb.attention_fwd(qkv, causal, out=out, d_status=status)             # a set status word: nothing happens
    assert bool((out == 3.0).all()) and int(status.item()) == 6 + 16 * 7
    status.zero_()
    hb.attention_fwd(qkv, causal, out=out, d_status=status)
    assert torch.equal(out, want) and int(status.item()) == 0
