"""The quantizer at the edges of its splits (one or two lane shares per thread, an odd number of V tiles, rows of 4, 8 and
16 lanes) and of its arithmetic (every scale code, saturation above the E6M2 range, FP16 subnormals, ties, empty groups),
bit for bit against the oracle."""
import pytest
import torch

from paper_2607_04302_b200 import synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("Hq,Hkv,N,d,dtype,qmean", [
    (1, 1, 64, 64, "bf16", False), (3, 1, 192, 64, "fp16", True), (1, 1, 64, 128, "bf16", True),
    (2, 1, 320, 128, "fp16", False), (1, 1, 64, 256, "bf16", True), (5, 5, 448, 64, "bf16", False)])
def test_sizes_match_the_oracle(Hq, Hkv, N, d, dtype, qmean):
    from paper_2607_04302_b200 import binding as hb
    cfg = synth.config("C2", N=N, Hq=Hq, Hkv=Hkv, d=d, dtype=dtype, cal_samples=2, cal_tokens=64)
    q, k, v = synth.make_qkv(cfg)
    s, inv_s = parity.calibrate(cfg, DEV)
    qkv = hb.quantize_qkv(q.to(DEV), k.to(DEV), v.to(DEV), s, inv_s, qmean=qmean)
    parity.check_quantized(cfg, q, k, v, s, inv_s, qkv, qmean=qmean)


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
def test_extreme_magnitudes_match_the_oracle(dtype):
    from paper_2607_04302_b200 import binding as hb
    gen = torch.Generator().manual_seed(7)
    cfg = synth.config("C3", N=512, Hq=1, Hkv=1, dtype=dtype)
    lo, hi = (-26.0, 15.9) if dtype == "fp16" else (-60.0, 30.0)       # past both ends of the E6M2 range in bf16
    e = torch.linspace(lo, hi, 512)[:, None]
    x = torch.randn((512, 128), generator=gen) * torch.exp2(e)
    ties = torch.exp2(torch.floor(e)) * torch.randint(-15, 16, (512, 128), generator=gen) / 2
    x = torch.where(torch.rand((512, 128), generator=gen) < 0.5, ties, x)
    x[17] = 0
    x[:, 5] = 0
    x = (x.clamp(-65504, 65504) if dtype == "fp16" else x).to(synth.torch_dtype(cfg))[None, None]
    qkv = hb.quantize_qkv(x.to(DEV), x.to(DEV), x.to(DEV))
    parity.check_quantized(cfg, x, x, x, None, None, qkv)


def test_fp16_overflow_saturates_like_the_oracle():
    """A smoothed FP16 product above 65504 rounds to infinity and saturates at the largest HIF4 magnitude (7 times the largest
    scale), as does an infinity of the input; the other elements of its group keep their values.  The query quantizer inside
    the attention kernel must agree with the stand-alone one bit for bit."""
    from paper_2607_04302_b200 import binding as hb
    gen = torch.Generator().manual_seed(3)
    cfg = synth.config("C3", N=128, Hq=2, Hkv=1, dtype="fp16", causal=False)
    q, k, v = (torch.randn((1, h, 128, 128), generator=gen) for h in (2, 1, 1))
    q *= torch.exp2(torch.linspace(-8, 13, 128))[:, None]
    k *= torch.exp2(torch.linspace(13, -8, 128))[:, None]
    v[..., 5, 3] = float("inf")
    v[..., 70:72, 9] = -float("inf")
    s = torch.exp2(torch.randint(-4, 5, (1, 128), generator=gen).float()) * 1.25
    inv_s = 1.0 / s
    q, k, v = (x.half() for x in (q, k, v))
    assert torch.isinf((q.float() * s).half()).any() and torch.isinf((k.float() * inv_s).half()).any()
    qd, kd, vd, sd, isd = (x.to(DEV) for x in (q, k, v, s, inv_s))
    qkv = hb.quantize_qkv(qd, kd, vd, sd, isd)
    parity.check_quantized(cfg, q, k, v, sd, isd, qkv)
    want = hb.attention_fwd(qkv, False)
    kv = hb.quantize_qkv(None, kd, vd, sd, isd, Hq=2)
    assert torch.equal(hb.attention_fwd_qraw(qd, sd, kv, False).view(torch.int32), want.view(torch.int32))


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
def test_nan_spoils_no_other_element(dtype):
    """A NaN in the input gives a NaN in the image and takes no part in the maxima; every other element of its group, its packed
    nibble included, is what it is with a zero in that place (infinities saturate beside it)."""
    from paper_2607_04302_b200 import binding as hb
    gen = torch.Generator().manual_seed(5)
    cfg = synth.config("C3", N=128, Hq=1, Hkv=1, dtype=dtype)
    x = torch.randn((1, 1, 128, 128), generator=gen)
    x[0, 0, 40, 70] = float("inf")
    bad = torch.rand(x.shape, generator=gen) < 0.05
    bad[0, 0, 40, 66] = True
    x = x.to(synth.torch_dtype(cfg))
    xd = torch.where(bad, torch.full_like(x, float("nan")), x).to(DEV)
    qkv = hb.quantize_qkv(xd, xd, xd)
    ref = hb.quantize_qkv(*(torch.where(bad, torch.zeros_like(x), x).to(DEV) for _ in range(3)))
    for n in "qkv":
        b = (bad.transpose(2, 3) if n == "v" else bad).to(DEV)
        assert torch.equal(getattr(qkv, n + "_meta"), getattr(ref, n + "_meta"))
        c, r = (torch.stack((t & 15, t >> 4), -1).flatten(-2) for t in (getattr(qkv, n + "_codes"), getattr(ref, n + "_codes")))
        assert torch.equal(c[~b], r[~b])
        c, r = getattr(qkv, n + "_mma"), getattr(ref, n + "_mma")
        assert torch.equal(c[~b], r[~b]) and bool(torch.isnan(c[b]).all())
