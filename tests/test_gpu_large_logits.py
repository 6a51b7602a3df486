"""Scaled scores of 16384 to 32768, where the running maximum, an FP16 value, is a multiple of 16: P = exp(S - m) then lies
anywhere up to e^8, far above 1, and so do the scales of its groups.  The first 64 channels carry an offset that is the same
for every key of a row, the others the differences between the keys; all products and their sums are exact in FP32, so P-hat
is held against the oracle at the usual bars.  Small grids run the 64-key kernel with four groups of softmax warps, 592
blocks (Bc = 128 and d = 256: 296) the two-block kernel and the one on pairs of SMs; the dump launch runs the 64-key (Bc = 128:
the 128-key) kernel."""
import pytest
import torch

from paper_2607_04302_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def inputs(cfg):
    gen = torch.Generator().manual_seed(11)
    q = torch.randint(-7, 8, (cfg.B, cfg.Hq, cfg.N, cfg.d), generator=gen) * 0.5
    k = torch.randint(-7, 8, (cfg.B, cfg.Hkv, cfg.N, cfg.d), generator=gen) * 0.5
    q[..., ::64] = 3.5                                             # every group holds 7 steps of 0.5: quantized exactly
    k[..., ::64] = 3.5
    q[..., :64] = 16.0 * torch.randint(4, 8, (cfg.B, cfg.Hq, cfg.N, 64), generator=gen)      # scores of about 20000 in all,
    k[..., :64] = 40.0 if cfg.d == 128 else 56.0                                             # 500 more or less from row to row
    if cfg.d == 256:                                               # two of the four groups carry the differences
        q[..., 192:] = 0
    v = torch.randn((cfg.B, cfg.Hkv, cfg.N, cfg.d), generator=gen)
    return tuple(x.to(synth.torch_dtype(cfg)) for x in (q, k, v))


@pytest.mark.parametrize("d,Bc,causal,B", [(128, 64, False, 1), (128, 64, True, 1), (128, 128, True, 1), (256, 64, False, 1),
                                           (128, 64, False, 74), (128, 128, False, 37), (256, 64, True, 37)])
def test_p_far_above_one_matches_the_oracle(d, Bc, causal, B):
    from tests import parity
    cfg = synth.config("C3", B=B, Hq=4, Hkv=2, N=256, d=d, Bc=Bc, causal=causal)
    res = parity.run_case(cfg, DEV, blocks=[(B - 1, h, t) for h in (0, 3) for t in (0, 1)], check_quant=B == 1,
                          qkv_host=inputs(cfg))
    print(parity.assert_within_bars(res, f"d={d} Bc={Bc} B={B}"))
    assert torch.isfinite(res["out"]).all()
