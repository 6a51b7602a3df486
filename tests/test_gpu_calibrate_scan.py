"""The one-pass calibration scan at the sizes where its splits can go wrong (shares of less than a row, segments that end
inside a share, remainders of the unrolled loads, interleaved head maps), against torch reductions and numpy float64."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("S,Hq,Hkv,N,d,dtype,head_map", [
    (1, 1, 1, 1, 64, torch.bfloat16, None),
    (1, 2, 1, 65, 256, torch.float16, None),
    (3, 14, 2, 257, 64, torch.bfloat16, None),
    (5, 6, 3, 1025, 128, torch.float16, [2, 0, 1, 1, 0, 2]),
    (2, 32, 8, 2047, 128, torch.bfloat16, None),
    (33, 8, 8, 129, 256, torch.bfloat16, None),
])
def test_scan_matches_torch(S, Hq, Hkv, N, d, dtype, head_map):
    from paper_2607_04302_b200 import binding as hb
    gen = torch.Generator(device=DEV).manual_seed(S * N + d)
    q = (torch.randn((S, Hq, N, d), generator=gen, device=DEV)).to(dtype)
    k = (torch.randn((S, Hkv, N, d), generator=gen, device=DEV) * 2).to(dtype)
    k[:, :, N // 2, 5] *= 30                                             # one dominant channel
    kv_of = torch.tensor(head_map or [h // (Hq // Hkv) for h in range(Hq)], device=DEV)
    kmax = k.float().abs().amax(2)                                       # [S,Hkv,d]
    qh = q.float().abs().amax(2)
    qmax = torch.stack([qh[:, kv_of == g].amax(1) for g in range(Hkv)], 1)
    kagg, qagg = (t.double().square().mean(0).sqrt() for t in (kmax, qmax))
    for mode, alpha in ((hb.MODE_STRONG, 0.5), (hb.MODE_MILD, 0.25)):
        s, inv_s = hb.smooth_calibrate(q, k, mode, q_to_kv=head_map)
        want = kagg.pow(alpha) / qagg.pow(1 - alpha)
        assert torch.allclose(s.double(), want, rtol=1e-6, atol=0)       # double pow on both sides, rounded once
        assert torch.equal(inv_s, 1.0 / s)
    _, _, stats = hb.smooth_calibrate_auto(q, k, q_to_kv=head_map)
    mag = np.sort(k.float().abs().flatten().cpu().numpy())
    p99 = float(mag[int(np.ceil(0.99 * mag.size)) - 1])
    top_k, top_q = float(mag[-1]), float(q.float().abs().max())
    assert stats[0].item() == np.float32(top_k / p99) and stats[1].item() == np.float32(top_k / top_q)


@pytest.mark.parametrize("S", [1, 2, 99, 100, 101, 200, 301])
def test_p99_aggregator_is_the_nearest_rank(S):
    """Around the sample counts where the rank leaves the maximum, with ties at the top (a magnitude out of five per sample)."""
    from paper_2607_04302_b200 import binding as hb
    gen = torch.Generator(device=DEV).manual_seed(S)
    q, k = (torch.randint(1, 6, (S, 2, 3, 64), generator=gen, device=DEV).bfloat16() for _ in range(2))
    k[:, :, :, 7] = 0                                                    # an aggregate of zero: s = 1
    rank = max(1, -(-99 * S // 100))
    kagg, qagg = (t.float().abs().amax(2).sort(0).values[rank - 1].double() for t in (k, q))
    s, _ = hb.smooth_calibrate(q, k, hb.MODE_STRONG | hb.AGG_P99)
    want = torch.where(kagg > 0, (kagg / qagg).sqrt(), torch.ones_like(kagg))
    assert torch.allclose(s.double(), want, rtol=1e-6, atol=0)           # double pow on both sides, rounded once
